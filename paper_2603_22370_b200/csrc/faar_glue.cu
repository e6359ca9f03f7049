// Element-wise pieces of a decoder block that sit between the linears: what the layer-wise driver needs
// to produce each linear's calibration input on the device (the MLP's SiLU-gated product feeds down_proj),
// and what full-model alignment (Eq. 6, Procedure steps 15-23) needs around the tensor-core GEMMs.
// All of them are HBM-bound: BF16 in and out as 16-byte vectors, FP32 arithmetic in registers.
#include <math.h>

#include "faar_internal.cuh"

namespace {

constexpr int GL_THREADS = 256;

__device__ __forceinline__ void unpack8(const uint4& raw, float (&x)[8]) {
  const uint32_t r[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(r[i] << 16);
    x[2 * i + 1] = __uint_as_float(r[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ uint4 pack8(const float (&x)[8]) {
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 p2 = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
    o[i] = *reinterpret_cast<uint32_t*>(&p2);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// Work split of the [rows, 8-element groups] kernels: threadIdx.x / blockIdx.x run over the groups of a row,
// threadIdx.y / blockIdx.y over rows (grid-stride), so no thread divides its index by the row length.
struct Split { dim3 grid, block; };
__device__ __forceinline__ int split_group() { return blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int split_row0() { return blockIdx.y * blockDim.y + threadIdx.y; }
__device__ __forceinline__ int split_row_step() { return gridDim.y * blockDim.y; }

// out = silu(gate) * up, silu(x) = x * sigmoid(x); two rows per thread in flight
__global__ void __launch_bounds__(GL_THREADS)
silu_mul_kernel(const __nv_bfloat16* gate, int64_t ldg, const __nv_bfloat16* up, int64_t ldu, __nv_bfloat16* out, int64_t ldo,
                int rows, int groups) {
  faar_pdl_sync();
  const int cg = split_group();
  if (cg >= groups) return;
  const int col = 8 * cg, step = split_row_step();
  for (int row = split_row0(); row < rows; row += 2 * step) {
    const int row1 = row + step;
    const bool two = row1 < rows;
    const uint4 ga = *reinterpret_cast<const uint4*>(gate + (int64_t)row * ldg + col);
    const uint4 ua = *reinterpret_cast<const uint4*>(up + (int64_t)row * ldu + col);
    uint4 gb = ga, ub = ua;
    if (two) {
      gb = *reinterpret_cast<const uint4*>(gate + (int64_t)row1 * ldg + col);
      ub = *reinterpret_cast<const uint4*>(up + (int64_t)row1 * ldu + col);
    }
    float a[8], b[8], y[8];
    unpack8(ga, a); unpack8(ua, b);
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = faar_silu_mul(a[i], b[i]);
    *reinterpret_cast<uint4*>(out + (int64_t)row * ldo + col) = pack8(y);
    if (two) {
      unpack8(gb, a); unpack8(ub, b);
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = faar_silu_mul(a[i], b[i]);
      *reinterpret_cast<uint4*>(out + (int64_t)row1 * ldo + col) = pack8(y);
    }
  }
}

// ---- RMSNorm: y = x / sqrt(mean(x^2) + eps) * g, one warp per row ---------------------------------
// Rows of up to 8 * 32 * NV elements stay in registers between the sum of squares and the scaled output (NV
// 16-byte vectors per lane); NV = 0 is the form for longer rows, which reads the row a second time (L1 / L2).
// With `b` the row is first formed as the BF16-rounded sum x + b and written to `sum_out` (a residual
// connection followed by the next norm): the same values as faar_add followed by faar_rmsnorm.
// EMBED: how a model's pass begins.  A row is a token's row of the embedding table `x` (zeros for a token outside it), stored to
// `sum_out`; the launch also leaves every row's rotary angles (an angle's rows side by side, as the rows' lanes will read them),
// one sine and cosine per token and angle for all blocks' products and attention kernels.  Two launches fewer than gathers and norms
// of their own, with both passes of a step sharing it: host time of the small model's step 203 -> 192 us with the loss's final sums.
struct EmbedArgs { const int* tokens; int vocab; const int* pos; int head_dim; float log2_theta; float2* rope; };
template <int NV, bool EMBED>
__global__ void __launch_bounds__(GL_THREADS)
rmsnorm_kernel(const __nv_bfloat16* x, int64_t ldx, const __nv_bfloat16* b, int64_t ldb, __nv_bfloat16* sum_out, int64_t lds,
               const float* __restrict__ g, float eps, __nv_bfloat16* y, int64_t ldy, float* __restrict__ rstd_out, int rows,
               int cols, const EmbedArgs em) {
  faar_pdl_sync();
  const int lane = threadIdx.x & 31;
  if (EMBED) {
    const int64_t all = (int64_t)rows * (em.head_dim / 2);
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < all; k += (int64_t)gridDim.x * blockDim.x) {
      const int i = (int)(k / rows), row = (int)(k - (int64_t)i * rows);
      float2 sc;
      sincosf((float)em.pos[row] * faar_rope_frequency(i, em.head_dim, em.log2_theta), &sc.x, &sc.y);
      em.rope[k] = sc;
    }
  }
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int n_groups = cols / 8;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < rows; row += warps) {
    const int token = EMBED ? em.tokens[row] : row;
    const bool known = !EMBED || (token >= 0 && token < em.vocab);
    const __nv_bfloat16* xr = x + (int64_t)(known ? token : 0) * ldx;
    const __nv_bfloat16* br = !EMBED && b ? b + (int64_t)row * ldb : nullptr;
    __nv_bfloat16* sr = EMBED || b ? sum_out + (int64_t)row * lds : nullptr;
    __nv_bfloat16* yr = y + (int64_t)row * ldy;
    float ss = 0.f;
    if constexpr (NV > 0) {
      uint4 v[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int c = lane + 32 * k;
        if (c < n_groups) {
          v[k] = *reinterpret_cast<const uint4*>(xr + 8 * c);
          if (EMBED) {
            if (!known) v[k] = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(sr + 8 * c) = v[k];
          }
        }
      }
      if (br) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          const int c = lane + 32 * k;
          if (c < n_groups) {
            float a[8], r[8];
            unpack8(v[k], a);
            unpack8(*reinterpret_cast<const uint4*>(br + 8 * c), r);
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] += r[i];
            v[k] = pack8(a);
            *reinterpret_cast<uint4*>(sr + 8 * c) = v[k];
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        if (lane + 32 * k < n_groups) {
          float a[8];
          unpack8(v[k], a);
#pragma unroll
          for (int i = 0; i < 8; ++i) ss = fmaf(a[i], a[i], ss);
        }
      }
      ss = faar_warp_sum(ss);
      const float rstd = 1.0f / sqrtf(ss / (float)cols + eps);
      if (lane == 0 && rstd_out) rstd_out[row] = rstd;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int c = lane + 32 * k;
        if (c < n_groups) {
          float a[8], o[8];
          unpack8(v[k], a);
          const float4 g0 = *reinterpret_cast<const float4*>(g + 8 * c), g1 = *reinterpret_cast<const float4*>(g + 8 * c + 4);
          const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i] = a[i] * rstd * gg[i];
          *reinterpret_cast<uint4*>(yr + 8 * c) = pack8(o);
        }
      }
    } else {
      for (int c = lane; c < n_groups; c += 32) {
        float a[8];
        uint4 raw = *reinterpret_cast<const uint4*>(xr + 8 * c);
        if (EMBED) {
          if (!known) raw = make_uint4(0u, 0u, 0u, 0u);
          *reinterpret_cast<uint4*>(sr + 8 * c) = raw;
        }
        unpack8(raw, a);
        if (br) {
          float r[8];
          unpack8(*reinterpret_cast<const uint4*>(br + 8 * c), r);
#pragma unroll
          for (int i = 0; i < 8; ++i) a[i] += r[i];
          const uint4 sum = pack8(a);
          *reinterpret_cast<uint4*>(sr + 8 * c) = sum;
          unpack8(sum, a);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) ss = fmaf(a[i], a[i], ss);
      }
      ss = faar_warp_sum(ss);
      const float rstd = 1.0f / sqrtf(ss / (float)cols + eps);
      if (lane == 0 && rstd_out) rstd_out[row] = rstd;
      const __nv_bfloat16* src = sr ? sr : xr;          // this lane wrote the groups it reads back
      for (int c = lane; c < n_groups; c += 32) {
        float a[8], o[8];
        unpack8(*reinterpret_cast<const uint4*>(src + 8 * c), a);
        const float4 g0 = *reinterpret_cast<const float4*>(g + 8 * c), g1 = *reinterpret_cast<const float4*>(g + 8 * c + 4);
        const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = a[i] * rstd * gg[i];
        *reinterpret_cast<uint4*>(yr + 8 * c) = pack8(o);
      }
    }
  }
}

// Backward of RMSNorm towards x (the norm weights are frozen): with xh = x * rstd and w = g * dy,
// dx = rstd * (w - xh * mean(w * xh)), optionally added to `add` (the residual branch's gradient).  dy is the
// FP32 sum of up to three BF16 tensors (the gradients of the linears that read the norm's output).  One warp
// per row; the row is read twice (the dot product, then the result), the second time from L1 / L2.  NG groups of a row are
// requested at a time: two for long rows and where few rows leave a warp alone with its loads' latency, else one, which
// leaves room for more warps.  Two gradients, one group -> two, us: 2000 x 2048 12.5 -> 10.5, 300 x 2048 8.1 -> 7.6,
// 8192 x 4096 81 -> 72; 4000 x 2048 15.5 -> 17.0, 8192 x 1024 12.5 -> 14.1, 20000 x 64 8.2 -> 10.3.
template <int NG>
__global__ void __launch_bounds__(GL_THREADS)
rmsnorm_bwd_kernel(const __nv_bfloat16* dy, const __nv_bfloat16* dy2, const __nv_bfloat16* dy3, int64_t lddy,
                   const __nv_bfloat16* x, int64_t ldx, const float* __restrict__ g, const float* __restrict__ rstd_in,
                   const __nv_bfloat16* add, int64_t ldadd, __nv_bfloat16* dx, int64_t lddx, int rows, int cols) {
  faar_pdl_sync();
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int n_groups = cols / 8;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < rows; row += warps) {
    const int64_t doff = (int64_t)row * lddy;
    const uint4* xr = reinterpret_cast<const uint4*>(x + (int64_t)row * ldx);
    const uint4* d1 = reinterpret_cast<const uint4*>(dy + doff);
    const uint4* d2 = reinterpret_cast<const uint4*>(dy2 ? dy2 + doff : nullptr);
    const uint4* d3 = reinterpret_cast<const uint4*>(dy3 ? dy3 + doff : nullptr);
    const uint4* ar = reinterpret_cast<const uint4*>(add ? add + (int64_t)row * ldadd : nullptr);
    uint4* out = reinterpret_cast<uint4*>(dx + (int64_t)row * lddx);
    const float rstd = rstd_in[row];
    uint4 xv[NG], v1[NG], v2[NG], v3[NG];
    auto request = [&](int c0) {
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int c = c0 + 32 * k;
        if (c < n_groups) {
          xv[k] = xr[c];
          v1[k] = d1[c];
          if (d2) v2[k] = d2[c];
          if (d3) v3[k] = d3[c];
        }
      }
    };
    // w = g * (dy + dy2 + dy3) of the k-th requested group
    auto weigh = [&](int k, int c, float (&w)[8]) {
      unpack8(v1[k], w);
      if (d2) {
        float t[8];
        unpack8(v2[k], t);
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] += t[i];
      }
      if (d3) {
        float t[8];
        unpack8(v3[k], t);
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] += t[i];
      }
      const float4 g0 = *reinterpret_cast<const float4*>(g + 8 * c), g1 = *reinterpret_cast<const float4*>(g + 8 * c + 4);
      const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] *= gg[i];
    };
    float dot = 0.f;
    for (int c0 = lane; c0 < n_groups; c0 += 32 * NG) {
      request(c0);
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int c = c0 + 32 * k;
        if (c < n_groups) {
          float a[8], w[8];
          unpack8(xv[k], a);
          weigh(k, c, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) dot = fmaf(w[i], a[i] * rstd, dot);
        }
      }
    }
    dot = faar_warp_sum(dot) / (float)cols;
    for (int c0 = lane; c0 < n_groups; c0 += 32 * NG) {
      request(c0);
      uint4 av[NG];
#pragma unroll
      for (int k = 0; k < NG; ++k)
        if (ar && c0 + 32 * k < n_groups) av[k] = ar[c0 + 32 * k];
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int c = c0 + 32 * k;
        if (c < n_groups) {
          float a[8], w[8], o[8];
          unpack8(xv[k], a);
          weigh(k, c, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i] = rstd * fmaf(-(a[i] * rstd), dot, w[i]);
          if (ar) {
            float r[8];
            unpack8(av[k], r);
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] += r[i];
          }
          out[c] = pack8(o);
        }
      }
    }
  }
}

// The same for one incoming gradient and rows of up to 8 * 32 * NV elements: x, dy and `add` stay in registers as they are
// in memory (BF16 pairs) between the passes, all requested at once (128 registers, 16 warps per SM): 8192 x 2048 with `add` 34.3 -> 27.0 us (134 MB),
// 2000 x 2048 17.4 -> 9.3.
template <int NV>
__global__ void __launch_bounds__(GL_THREADS, 2)
rmsnorm_bwd_row_kernel(const __nv_bfloat16* dy, int64_t lddy, const __nv_bfloat16* x, int64_t ldx, const float* __restrict__ g,
                       const float* __restrict__ rstd_in, const __nv_bfloat16* add, int64_t ldadd, __nv_bfloat16* dx, int64_t lddx,
                       int rows, int cols) {
  faar_pdl_sync();
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int n_groups = cols / 8;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < rows; row += warps) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + (int64_t)row * ldx);
    const uint4* dr = reinterpret_cast<const uint4*>(dy + (int64_t)row * lddy);
    const uint4* ar = reinterpret_cast<const uint4*>(add ? add + (int64_t)row * ldadd : nullptr);
    uint4* out = reinterpret_cast<uint4*>(dx + (int64_t)row * lddx);
    const float rstd = rstd_in[row];
    uint4 xv[NV], dv[NV], av[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = lane + 32 * k;
      if (c < n_groups) { xv[k] = xr[c]; dv[k] = dr[c]; }
    }
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (ar && lane + 32 * k < n_groups) av[k] = ar[lane + 32 * k];
    auto weigh = [&](int c, float (&w)[8]) {
      const float4 g0 = *reinterpret_cast<const float4*>(g + 8 * c), g1 = *reinterpret_cast<const float4*>(g + 8 * c + 4);
      const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] *= gg[i];
    };
    float dot = 0.f;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      if (lane + 32 * k < n_groups) {
        float a[8], w[8];
        unpack8(xv[k], a);
        unpack8(dv[k], w);
        weigh(lane + 32 * k, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) dot = fmaf(w[i], a[i] * rstd, dot);
      }
    }
    dot = faar_warp_sum(dot) / (float)cols;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = lane + 32 * k;
      if (c < n_groups) {
        float a[8], w[8], o[8];
        unpack8(xv[k], a);
        unpack8(dv[k], w);
        weigh(c, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = rstd * fmaf(-(a[i] * rstd), dot, w[i]);
        if (ar) {
          float r[8];
          unpack8(av[k], r);
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i] += r[i];
        }
        out[c] = pack8(o);
      }
    }
  }
}

// ---- rotary position embedding, half-split pairing ----------------------------------------------
// Inside every head, element i (i < head_dim / 2) pairs with element i + head_dim / 2; the pair of token t is
// rotated by pos[t] * theta^(-2 i / head_dim) (by the negative angle with inverse != 0: the backward pass of
// an orthogonal map).  One thread takes 8 consecutive i of HPT heads of one token (the angle does not depend
// on the head, so its sine and cosine serve all of them), for a stride of tokens.
template <int HPT>
__global__ void __launch_bounds__(GL_THREADS)
rope_kernel(const __nv_bfloat16* x, int64_t ldx, const int* __restrict__ pos, __nv_bfloat16* y, int64_t ldy, int rows,
            int groups, int head_dim, float log2_theta, int inverse) {
  faar_pdl_sync();
  const int cg = split_group();
  if (cg >= groups) return;
  const int half = head_dim / 2, gph = half / 8;                    // 8-element groups per half head
  const int chunk = cg / gph, gi = cg - chunk * gph;
  const int64_t off = (int64_t)chunk * HPT * head_dim + 8 * gi;
  float inv_freq[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) inv_freq[i] = faar_rope_frequency(8 * gi + i, head_dim, log2_theta);
  for (int row = split_row0(); row < rows; row += split_row_step()) {
    const __nv_bfloat16* xr = x + (int64_t)row * ldx + off;
    __nv_bfloat16* yr = y + (int64_t)row * ldy + off;
    uint4 ra[HPT], rb[HPT];
#pragma unroll
    for (int h = 0; h < HPT; ++h) {
      ra[h] = *reinterpret_cast<const uint4*>(xr + h * head_dim);
      rb[h] = *reinterpret_cast<const uint4*>(xr + h * head_dim + half);
    }
    const float p = (float)pos[row];
    float sn[8], cs[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      sincosf(p * inv_freq[i], &sn[i], &cs[i]);
      if (inverse) sn[i] = -sn[i];
    }
#pragma unroll
    for (int h = 0; h < HPT; ++h) {
      float a[8], b[8];
      unpack8(ra[h], a);
      unpack8(rb[h], b);
#pragma unroll
      for (int i = 0; i < 8; ++i) faar_rope_turn(a[i], b[i], sn[i], cs[i]);
      *reinterpret_cast<uint4*>(yr + h * head_dim) = pack8(a);
      *reinterpret_cast<uint4*>(yr + h * head_dim + half) = pack8(b);
    }
  }
}

// ---- backward of the gated product ----------------------------------------------------------------
__global__ void __launch_bounds__(GL_THREADS)
silu_mul_bwd_kernel(const __nv_bfloat16* dout, int64_t ldd, const __nv_bfloat16* gate, int64_t ldg, const __nv_bfloat16* up,
                    int64_t ldu, __nv_bfloat16* dgate, int64_t lddg, __nv_bfloat16* dup, int64_t lddu, int rows, int groups) {
  faar_pdl_sync();
  const int cg = split_group();
  if (cg >= groups) return;
  const int col = 8 * cg;
  for (int row = split_row0(); row < rows; row += split_row_step()) {
    float d[8], g[8], u[8], og[8], ou[8];
    unpack8(*reinterpret_cast<const uint4*>(dout + (int64_t)row * ldd + col), d);
    unpack8(*reinterpret_cast<const uint4*>(gate + (int64_t)row * ldg + col), g);
    unpack8(*reinterpret_cast<const uint4*>(up + (int64_t)row * ldu + col), u);
#pragma unroll
    for (int i = 0; i < 8; ++i) faar_silu_mul_bwd(d[i], g[i], u[i], og[i], ou[i]);
    *reinterpret_cast<uint4*>(dgate + (int64_t)row * lddg + col) = pack8(og);
    *reinterpret_cast<uint4*>(dup + (int64_t)row * lddu + col) = pack8(ou);
  }
}

// ---- embedding: out[t, :] = table[tokens[t], :]; a token outside [0, vocab) gives a row of zeros --------
__global__ void __launch_bounds__(GL_THREADS)
embedding_kernel(const __nv_bfloat16* __restrict__ table, int64_t ldt, const int* __restrict__ tokens, int vocab,
                 __nv_bfloat16* __restrict__ out, int64_t ldo, int rows, int groups) {
  faar_pdl_sync();
  const int cg = split_group();
  if (cg >= groups) return;
  const int col = 8 * cg;
  for (int row = split_row0(); row < rows; row += split_row_step()) {
    const int tok = tokens[row];
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (tok >= 0 && tok < vocab) v = *reinterpret_cast<const uint4*>(table + (int64_t)tok * ldt + col);
    *reinterpret_cast<uint4*>(out + (int64_t)row * ldo + col) = v;
  }
}

// ---- out = a + b (residual connections and the sums of gradients that meet at one tensor) -----------
__global__ void __launch_bounds__(GL_THREADS)
add_kernel(const __nv_bfloat16* a, int64_t lda, const __nv_bfloat16* b, int64_t ldb, __nv_bfloat16* out, int64_t ldo, int rows,
           int groups) {
  faar_pdl_sync();
  const int cg = split_group();
  if (cg >= groups) return;
  const int col = 8 * cg;
  for (int row = split_row0(); row < rows; row += split_row_step()) {
    float x[8], y[8], o[8];
    unpack8(*reinterpret_cast<const uint4*>(a + (int64_t)row * lda + col), x);
    unpack8(*reinterpret_cast<const uint4*>(b + (int64_t)row * ldb + col), y);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = x[i] + y[i];
    *reinterpret_cast<uint4*>(out + (int64_t)row * ldo + col) = pack8(o);
  }
}

// Launch shape for the kernels above: 256 threads as (groups of a row) x (rows), the row extent of the grid
// capped at eight blocks per SM.
Split glue_split(const faar_ctx* ctx, int rows, int groups) {
  int tx = 4;                                   // short rows: several rows per warp
  while (tx < GL_THREADS && tx < groups) tx *= 2;
  const int ty = GL_THREADS / tx;
  const int gx = (groups + tx - 1) / tx;
  int64_t gy = ((int64_t)rows + ty - 1) / ty;
  const int64_t cap = ((int64_t)ctx->num_sms * 8 + gx - 1) / gx;
  if (gy > cap) gy = cap;
  if (gy > 65535) gy = 65535;
  if (gy < 1) gy = 1;
  Split s;
  s.grid = dim3((unsigned)gx, (unsigned)gy, 1);
  s.block = dim3((unsigned)tx, (unsigned)ty, 1);
  return s;
}

int glue_grid(const faar_ctx* ctx, int64_t items) {
  int64_t blocks = (items + GL_THREADS - 1) / GL_THREADS;
  const int64_t cap = (int64_t)ctx->num_sms * 8;
  if (blocks > cap) blocks = cap;
  return (int)(blocks < 1 ? 1 : blocks);
}

}  // namespace

int faar_launch_silu_mul(faar_ctx* ctx, int rows, int cols, const void* gate, int64_t ldg, const void* up, int64_t ldu,
                         void* out, int64_t ldo) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const Split sp = glue_split(ctx, (rows + 1) / 2, cols / 8);
  faar_launch_pdl(ctx, silu_mul_kernel, sp.grid, sp.block, 0, 
      reinterpret_cast<const __nv_bfloat16*>(gate), ldg, reinterpret_cast<const __nv_bfloat16*>(up), ldu,
      reinterpret_cast<__nv_bfloat16*>(out), ldo, rows, cols / 8);
  return (int)cudaGetLastError();
}

// b / sum_out null: y = rmsnorm(x).  Otherwise sum_out = x + b (BF16) and y = rmsnorm(sum_out).
int faar_launch_rmsnorm(faar_ctx* ctx, int rows, int cols, const void* x, int64_t ldx, const void* b, int64_t ldb,
                        void* sum_out, int64_t lds, const float* g, float eps, void* y, int64_t ldy, float* rstd) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const int grid = glue_grid(ctx, (int64_t)rows * 32);
  auto* xp = reinterpret_cast<const __nv_bfloat16*>(x);
  auto* bp = reinterpret_cast<const __nv_bfloat16*>(b);
  auto* sp = reinterpret_cast<__nv_bfloat16*>(sum_out);
  auto* yp = reinterpret_cast<__nv_bfloat16*>(y);
  faar_launch_pdl(ctx, cols <= 8 * 32 * 8 ? rmsnorm_kernel<8, false> : rmsnorm_kernel<0, false>, dim3(grid), dim3(GL_THREADS), 0, xp, ldx, bp,
                  ldb, sp, lds, g, eps, yp, ldy, rstd, rows, cols, EmbedArgs{});
  return (int)cudaGetLastError();
}

int faar_launch_embed_rmsnorm(faar_ctx* ctx, int rows, int cols, int vocab, const void* table, const int* tokens, void* x, const float* g,
                              float eps, void* y, float* rstd, const int* pos, int head_dim, float theta, float2* rope) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const EmbedArgs em = {tokens, vocab, pos, head_dim, log2f(theta), rope};
  faar_launch_pdl(ctx, cols <= 8 * 32 * 8 ? rmsnorm_kernel<8, true> : rmsnorm_kernel<0, true>, dim3(glue_grid(ctx, (int64_t)rows * 32)),
                  dim3(GL_THREADS), 0, reinterpret_cast<const __nv_bfloat16*>(table), (int64_t)cols, (const __nv_bfloat16*)nullptr, (int64_t)0,
                  reinterpret_cast<__nv_bfloat16*>(x), (int64_t)cols, g, eps, reinterpret_cast<__nv_bfloat16*>(y), (int64_t)cols, rstd, rows, cols,
                  em);
  return (int)cudaGetLastError();
}

// dy2 / dy3 nullable: further gradients (same leading dimension as dy) summed with dy before the norm's backward.
int faar_launch_rmsnorm_bwd(faar_ctx* ctx, int rows, int cols, const void* dy, const void* dy2, const void* dy3, int64_t lddy,
                            const void* x, int64_t ldx, const float* g, const float* rstd, const void* add, int64_t ldadd,
                            void* dx, int64_t lddx) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const int grid = glue_grid(ctx, (int64_t)rows * 32);
  auto* d1 = reinterpret_cast<const __nv_bfloat16*>(dy);
  auto* d2 = reinterpret_cast<const __nv_bfloat16*>(dy2);
  auto* d3 = reinterpret_cast<const __nv_bfloat16*>(dy3);
  auto* xp = reinterpret_cast<const __nv_bfloat16*>(x);
  auto* ap = reinterpret_cast<const __nv_bfloat16*>(add);
  auto* op = reinterpret_cast<__nv_bfloat16*>(dx);
  if (!d2 && !d3 && cols <= 8 * 32 * 8)
    faar_launch_pdl(ctx, cols <= 8 * 32 * 2 ? rmsnorm_bwd_row_kernel<2> : rmsnorm_bwd_row_kernel<8>, dim3(grid), dim3(GL_THREADS), 0, d1, lddy,
                    xp, ldx, g, rstd, ap, ldadd, op, lddx, rows, cols);
  else
    faar_launch_pdl(ctx, cols > 8 * 32 * 8 || (cols > 8 * 32 * 4 && rows <= 16 * ctx->num_sms) ? rmsnorm_bwd_kernel<2> : rmsnorm_bwd_kernel<1>, dim3(grid), dim3(GL_THREADS), 0, d1, d2, d3, lddy, xp, ldx, g, rstd, ap, ldadd, op, lddx, rows, cols);
  return (int)cudaGetLastError();
}

int faar_launch_rope(faar_ctx* ctx, int rows, int n_heads, int head_dim, const void* x, int64_t ldx, const int* pos, float theta,
                     int inverse, void* y, int64_t ldy) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const bool four = n_heads % 4 == 0;                                 // four heads per thread share one sine / cosine
  const int groups = (four ? n_heads / 4 : n_heads) * (head_dim / 16);
  const Split sp = glue_split(ctx, rows, groups);
  auto* xp = reinterpret_cast<const __nv_bfloat16*>(x);
  auto* yp = reinterpret_cast<__nv_bfloat16*>(y);
  if (four)
    faar_launch_pdl(ctx, rope_kernel<4>, sp.grid, sp.block, 0, xp, ldx, pos, yp, ldy, rows, groups, head_dim, log2f(theta), inverse);
  else
    faar_launch_pdl(ctx, rope_kernel<1>, sp.grid, sp.block, 0, xp, ldx, pos, yp, ldy, rows, groups, head_dim, log2f(theta), inverse);
  return (int)cudaGetLastError();
}

int faar_launch_silu_mul_bwd(faar_ctx* ctx, int rows, int cols, const void* dout, int64_t ldd, const void* gate, int64_t ldg,
                             const void* up, int64_t ldu, void* dgate, int64_t lddg, void* dup, int64_t lddu) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const Split sp = glue_split(ctx, rows, cols / 8);
  faar_launch_pdl(ctx, silu_mul_bwd_kernel, sp.grid, sp.block, 0, 
      reinterpret_cast<const __nv_bfloat16*>(dout), ldd, reinterpret_cast<const __nv_bfloat16*>(gate), ldg,
      reinterpret_cast<const __nv_bfloat16*>(up), ldu, reinterpret_cast<__nv_bfloat16*>(dgate), lddg,
      reinterpret_cast<__nv_bfloat16*>(dup), lddu, rows, cols / 8);
  return (int)cudaGetLastError();
}

int faar_launch_embedding(faar_ctx* ctx, int rows, int cols, int vocab, const void* table, int64_t ldt, const int* tokens,
                          void* out, int64_t ldo) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const Split sp = glue_split(ctx, rows, cols / 8);
  faar_launch_pdl(ctx, embedding_kernel, sp.grid, sp.block, 0, 
      reinterpret_cast<const __nv_bfloat16*>(table), ldt, tokens, vocab, reinterpret_cast<__nv_bfloat16*>(out), ldo, rows,
      cols / 8);
  return (int)cudaGetLastError();
}

int faar_launch_add(faar_ctx* ctx, int rows, int cols, const void* a, int64_t lda, const void* b, int64_t ldb, void* out,
                    int64_t ldo) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const Split sp = glue_split(ctx, rows, cols / 8);
  faar_launch_pdl(ctx, add_kernel, sp.grid, sp.block, 0, 
      reinterpret_cast<const __nv_bfloat16*>(a), lda, reinterpret_cast<const __nv_bfloat16*>(b), ldb,
      reinterpret_cast<__nv_bfloat16*>(out), ldo, rows, cols / 8);
  return (int)cudaGetLastError();
}
