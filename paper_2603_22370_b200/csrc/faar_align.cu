// Full-model alignment loss (Eq. 6, Procedure steps 18-20): KL of the temperature softmaxes of the two
// models' logits, the squared error of their last hidden states, and both gradients towards the
// quantised model's outputs.
//
// Softmax needs a row's maximum and sum before any probability, and a token's two logit rows (2 x vocab BF16, 0.5 MB at a
// 128 K vocabulary) do not fit one SM's shared memory, so they are read twice: the first pass (from HBM) keeps a running
// maximum and sum of exponentials per thread, the second (from L2) forms P_fp, P_q, the KL terms and the gradient.  HBM
// sees each logit once and the gradient once; the four exponentials per vocabulary entry take the special-function units
// about as long as the traffic takes HBM.  To have both at work all the time, one loop does the second pass of a token
// together with the first pass of the next one.  Two tokens' rows per SM would be more than L2 holds at a 128 K vocabulary,
// so there two CTAs (a cluster on two SMs) share a token, half a row each, and exchange maxima and sums through
// distributed shared memory.
// Where the products that wrote the logits left the maxima and sums of the rows' parts as well, the first pass is over those.
// One token after the other, each pass for itself -> this, us: 2000 tokens, vocabulary 32000 144 -> 122; 512, 8000 23.7 ->
// 16.6; 3000, 50000 298 -> 251; 8192, 128256 1590 -> 1568 (6.3 GB).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "faar.h"
#include "faar_internal.cuh"

namespace {

constexpr int AL_THREADS = 1024, AL_STATS_THREADS = 256;      // one CTA per SM; with the products' statistics several

struct AlignParams {
  const __nv_bfloat16* Zfp; const __nv_bfloat16* Zq; long long ldz; int V;
  const __nv_bfloat16* Hfp; const __nv_bfloat16* Hq; long long ldh; int D;
  __nv_bfloat16* dZ; __nv_bfloat16* dH;
  float c;                 // log2(e) / tau: softmax(z / tau) in base 2
  float gscale;            // lambda_kl / (tau T)
  float* kl_partials;      // one per cluster (or CTA)
  float* mse_partials;
  float* loss_out2;        // {KL / T, MSE}: written by the cluster that finishes last
  uint32_t* finished;      // workspace: clusters that have, zero between launches
  float kl_scale;
  const float2* stats_fp; const float2* stats_q; int slots;      // STATS: [T, slots] (maximum, sum) of 128 columns each
  int T;                   // tokens; cluster k takes tokens k, k + the number of clusters, ...
};

__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint64_t l2_stream_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_keep_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint4 ldg128_policy(const uint4* ptr, uint64_t pol) {
  uint4 v;
  asm volatile("ld.global.L2::cache_hint.v4.b32 {%0,%1,%2,%3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(ptr), "l"(pol));
  return v;
}
// the gradient is written once and not read here: it should not push the rows out of L2
__device__ __forceinline__ void stg128_policy(void* ptr, uint4 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v4.b32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(ptr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w),
               "l"(pol)
               : "memory");
}

// (maximum m, sum s of 2^(y - m)) of two disjoint sets merged; an empty set is (-inf, 0)
__device__ __forceinline__ void merge(float& m, float& s, float m2, float s2) {
  const float M = fmaxf(m, m2);
  if (M == -INFINITY) { m = M; s = 0.f; return; }
  s = s * faar_ex2(m - M) + s2 * faar_ex2(m2 - M);
  m = M;
}

__device__ __forceinline__ void unpack8(const uint4& raw, float (&y)[8]) {      // eight BF16 -> FP32
  const uint32_t r[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    y[2 * i] = __uint_as_float(r[i] << 16);
    y[2 * i + 1] = __uint_as_float(r[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t w) { return *reinterpret_cast<__nv_bfloat162*>(&w); }
// elements n..7 of a group of eight BF16 replaced by -1e30 (BF16 0xF149)
__device__ __forceinline__ uint4 mask_tail(uint4 v, int n) {
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (2 * i >= n) w[i] = 0xF149F149u;
    else if (2 * i + 1 >= n) w[i] = (w[i] & 0xFFFFu) | 0xF1490000u;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&p);
}

// The two loss values, in a fixed order in double, by whichever cluster finishes last: a launch of its own for a few hundred
// sums cost a small model's step as much as any other.  One atomic that releases and acquires; fences around a relaxed one took
// 0.35 us more (192 tokens, vocabulary 512 7.45 -> 7.2, 4096 and 1024 58.7 -> 58.3).
__device__ __forceinline__ void final_sums(const AlignParams& p, int mine, int clusters, float kl, float mse) {
  const int lane = threadIdx.x & 31;
  uint32_t done = 0u;
  if (lane == 0) {
    p.kl_partials[mine] = kl;
    p.mse_partials[mine] = mse;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(done) : "l"(p.finished) : "memory");
    ++done;
  }
  if (__shfl_sync(0xffffffffu, done, 0) != (uint32_t)clusters) return;
  __syncwarp();                                                  // what lane 0 has acquired counts for all lanes
  double kl_sum = 0.0, mse_sum = 0.0;
  for (int c = lane; c < clusters; c += 32) { kl_sum += (double)__ldcg(p.kl_partials + c); mse_sum += (double)__ldcg(p.mse_partials + c); }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    kl_sum += __shfl_xor_sync(0xffffffffu, kl_sum, o);
    mse_sum += __shfl_xor_sync(0xffffffffu, mse_sum, o);
  }
  if (lane == 0) {
    p.loss_out2[0] = (float)(kl_sum * (double)p.kl_scale);
    p.loss_out2[1] = (float)mse_sum;
    *p.finished = 0u;                                            // ready for the next launch
  }
}

// CL CTAs per token.  STATS: maxima and sums of the rows' parts come from the products that wrote the logits, so the first pass is
// over those, a thirtieth of the bytes, and the logits are read once; half the exponentials, too.  Four CTAs of 256 threads an SM, because
// a token's pass ends in a reduction that one CTA alone would wait for.  Two passes -> this, us: 8192 tokens, vocabulary 128256 1597 ->
// 1103 (6.3 GB; 1140 with one CTA an SM, 1121 with two), 2000 tokens, vocabulary 32000 120 -> 76 (92, 78).
template <int CL, bool STATS>
__global__ void __launch_bounds__(STATS ? AL_STATS_THREADS : AL_THREADS, STATS ? AL_THREADS / AL_STATS_THREADS : 1)
align_loss_kernel(const AlignParams p) {
  constexpr int THREADS = STATS ? AL_STATS_THREADS : AL_THREADS, WARPS = THREADS / 32;
  if (CL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // with the wait below: both CTAs have started
  faar_pdl_sync();
  if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  __shared__ float4 wred[WARPS];
  __shared__ float4 xch[2][CL];                                    // by parity of the token: each CTA's maximum and sum, fp and q
  __shared__ alignas(8) float tot[CL][2];                          // rank 0: every CTA's sums
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = CL > 1 ? blockIdx.x % CL : 0, n_cl = gridDim.x / CL;
  const int ngroups = (p.V + 7) / 8;                               // 16-byte groups of a row (rows are padded: ldz >= ceil8(V))
  const int share = (ngroups + CL - 1) / CL, g_first = rank * share + threadIdx.x, g_end = min(ngroups, (rank + 1) * share);
  const int tail = p.V & 7;                                        // valid columns of a partial last group, 0 = none
  const uint64_t stream = l2_stream_policy(), keep = l2_keep_policy();   // first pass: keep the rows in L2; second: done with them
  float kl = 0.f, mse = 0.f;                                       // this thread's share over all of the CTA's tokens
  // running maximum and sum of 2^(c z - max) of this thread's part of a row, fp and q
  float mf, sf, mq, sq;
  auto online = [&](const uint4& v, float& m, float& s) {
    const __nv_bfloat162 x = __hmax2(__hmax2(as_bf162(v.x), as_bf162(v.y)), __hmax2(as_bf162(v.z), as_bf162(v.w)));
    const float m8 = fmaxf(__low2float(x), __high2float(x)) * p.c;          // tau > 0: scaling keeps the order
    if (m8 > m) { s *= faar_ex2(m - m8); m = m8; }                                // 2^-inf = 0 on the first group
    float z[8];
    unpack8(v, z);
#pragma unroll
    for (int i = 0; i < 8; ++i) s += faar_ex2(fmaf(z[i], p.c, -m));
  };
  // first pass of one group; columns beyond the vocabulary count as -1e30 (their exponentials are 0)
  auto first = [&](uint4 a, uint4 b, int g) {
    if (tail && g == ngroups - 1) { a = mask_tail(a, tail); b = mask_tail(b, tail); }
    online(a, mf, sf);
    online(b, mq, sq);
  };
  // log2-sum-exp of a token's rows from what the threads hold; `parity` alternates between tokens
  float lse_f = 0.f, lse_q = 0.f;
  auto combine = [&](int parity) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      merge(mf, sf, __shfl_xor_sync(0xffffffffu, mf, o), __shfl_xor_sync(0xffffffffu, sf, o));
      merge(mq, sq, __shfl_xor_sync(0xffffffffu, mq, o), __shfl_xor_sync(0xffffffffu, sq, o));
    }
    if (lane == 0) wred[warp] = make_float4(mf, sf, mq, sq);
    __syncthreads();
    if (warp == 0) {
      float4 r = lane < WARPS ? wred[lane] : make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        merge(r.x, r.y, __shfl_xor_sync(0xffffffffu, r.x, o), __shfl_xor_sync(0xffffffffu, r.y, o));
        merge(r.z, r.w, __shfl_xor_sync(0xffffffffu, r.z, o), __shfl_xor_sync(0xffffffffu, r.w, o));
      }
      if (lane < CL) {                                             // lane c: to CTA c of the cluster
        uint32_t dst = (uint32_t)__cvta_generic_to_shared(&xch[parity][rank]);
        if (CL > 1) asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(dst) : "r"(lane));
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(r.x), "f"(r.y), "f"(r.z), "f"(r.w) : "memory");
      }
    }
    if (CL > 1) {
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      __syncthreads();
    }
    float4 r = xch[parity][0];
#pragma unroll
    for (int c = 1; c < CL; ++c) {
      const float4 x = xch[parity][c];
      merge(r.x, r.y, x.x, x.y);
      merge(r.z, r.w, x.z, x.w);
    }
    lse_f = r.x + lg2f(r.y);
    lse_q = r.z + lg2f(r.w);
  };
  // STATS: this thread's part of a token's statistics instead of its first pass
  auto first_of_stats = [&](int t) {
    const float2 *f = p.stats_fp + (long long)t * p.slots, *q = p.stats_q + (long long)t * p.slots;
    for (int i = threadIdx.x; i < p.slots; i += THREADS) {
      const float2 a = f[i], b = q[i];
      merge(mf, sf, a.x, a.y);
      merge(mq, sq, b.x, b.y);
    }
  };
  auto row = [&](const __nv_bfloat16* z, int t) { return reinterpret_cast<const uint4*>(z + (long long)t * p.ldz); };

  int t = blockIdx.x / CL, parity = 0;
  mf = mq = -INFINITY;
  sf = sq = 0.f;
  if (t < p.T) {
    const uint4 *gf = row(p.Zfp, t), *gq = row(p.Zq, t);
    if (STATS) first_of_stats(t);
    else
      for (int g = g_first; g < g_end; g += THREADS) first(ldg128_policy(gf + g, keep), ldg128_policy(gq + g, keep), g);
    combine(parity);
  }
  for (; t < p.T; t += n_cl) {
    const int tn = t + n_cl;
    const bool more = tn < p.T;
    const uint4 *gf = row(p.Zfp, t), *gq = row(p.Zq, t), *nf = row(p.Zfp, more ? tn : t), *nq = row(p.Zq, more ? tn : t);
    // log2 P = c z - lse, so log2 P_fp - log2 P_q = c (z_fp - z_q) - (lse_fp - lse_q)
    const float dlse = lse_f - lse_q;
    __nv_bfloat16* const gd = p.dZ ? p.dZ + (long long)t * p.ldz : nullptr;
    mf = mq = -INFINITY;
    sf = sq = 0.f;
    uint4 a1 = make_uint4(0u, 0u, 0u, 0u), b1 = a1;
    if (STATS) {
      if (more) first_of_stats(tn);
      if (g_first < g_end) { a1 = ldg128_policy(gf + g_first, stream); b1 = ldg128_policy(gq + g_first, stream); }
    } else if (more && g_first < g_end) { a1 = ldg128_policy(nf + g_first, keep); b1 = ldg128_policy(nq + g_first, keep); }
    for (int g = g_first; g < g_end; g += THREADS) {
      uint4 va, vb;
      if (STATS) {                                                 // the row itself, its loads one group ahead
        va = a1; vb = b1;
        const int gn = g + THREADS;
        if (gn < g_end) { a1 = ldg128_policy(gf + gn, stream); b1 = ldg128_policy(gq + gn, stream); }
      } else {
        va = ldg128_policy(gf + g, stream); vb = ldg128_policy(gq + g, stream);
      }
      if (!STATS && more) {                                                  // the next token's first pass, its loads one group ahead
        const uint4 a = a1, b = b1;
        const int gn = g + THREADS;
        if (gn < g_end) { a1 = ldg128_policy(nf + gn, keep); b1 = ldg128_policy(nq + gn, keep); }
        first(a, b, g);
      }
      const bool last_partial = tail && g == ngroups - 1;
      if (last_partial) { va = mask_tail(va, tail); vb = mask_tail(vb, tail); }
      float a[8], b[8], gr[8];
      unpack8(va, a);
      unpack8(vb, b);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float pf = faar_ex2(fmaf(a[i], p.c, -lse_f)), pq = faar_ex2(fmaf(b[i], p.c, -lse_q));
        kl = fmaf(pf, fmaf(a[i] - b[i], p.c, -dlse), kl);
        gr[i] = p.gscale * (pq - pf);
      }
      if (gd) {
        if (!last_partial) {
          stg128_policy(gd + 8 * g, make_uint4(pack2(gr[0], gr[1]), pack2(gr[2], gr[3]), pack2(gr[4], gr[5]), pack2(gr[6], gr[7])),
                        stream);
        } else {
          for (int i = 0; i < tail; ++i) gd[8 * g + i] = __float2bfloat16_rn(gr[i]);
        }
      }
    }
    // ---- last hidden states
    {
      const __nv_bfloat16* hf = p.Hfp + (long long)t * p.ldh;
      const __nv_bfloat16* hq = p.Hq + (long long)t * p.ldh;
      __nv_bfloat16* dh = p.dH ? p.dH + (long long)t * p.ldh : nullptr;
      for (int g = rank * THREADS + threadIdx.x; 8 * g < p.D; g += CL * THREADS) {
        const int nv = min(8, p.D - 8 * g);
        float a[8], b[8], d[8];
        unpack8(reinterpret_cast<const uint4*>(hf)[g], a);         // rows are padded to 8 columns (ldh >= ceil8(D))
        unpack8(reinterpret_cast<const uint4*>(hq)[g], b);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          d[i] = b[i] - a[i];
          if (i < nv) mse = fmaf(d[i], d[i], mse);
          d[i] *= 2.0f;
        }
        if (dh) {
          if (nv == 8) {
            *reinterpret_cast<uint4*>(dh + 8 * g) = make_uint4(pack2(d[0], d[1]), pack2(d[2], d[3]), pack2(d[4], d[5]),
                                                                pack2(d[6], d[7]));
          } else {
            for (int i = 0; i < nv; ++i) dh[8 * g + i] = __float2bfloat16_rn(d[i]);
          }
        }
      }
    }
    if (more) {
      parity ^= 1;
      combine(parity);
    }
  }
  kl = faar_warp_sum(kl);
  mse = faar_warp_sum(mse);
  __syncthreads();                                                 // wred is reused
  if (lane == 0) wred[warp] = make_float4(kl, mse, 0.f, 0.f);
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.f, b = 0.f;
    for (int w = 0; w < WARPS; ++w) { a += wred[w].x; b += wred[w].y; }
    uint32_t dst = (uint32_t)__cvta_generic_to_shared(&tot[rank][0]);
    if (CL > 1) asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(dst));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(a), "f"(b) : "memory");
  }
  if (CL > 1) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (rank == 0 && warp == 0) {
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int c = 0; c < CL; ++c) { a += tot[c][0]; b += tot[c][1]; }
    final_sums(p, blockIdx.x / CL, n_cl, a * 0.6931471805599453f, b);          // log2 -> natural log
  }
}

// Statistics of logits whose product left none (a frozen model's outputs that a caller keeps): bit for bit those of the product.
// A lane takes 128 columns of a row in their order; the warp's 8 KB come in as whole lines and change lanes in shared memory: 40 us for
// 2000 tokens and a vocabulary of 32000, 280 for 4096 and 128256 (3.7 TB/s; each lane reading its own 256 bytes 304), which the loss in
// one pass gives back: step on given outputs 1494 -> 1484 and 5970 -> 5990 us.
constexpr int LS_THREADS = 128;
__global__ void __launch_bounds__(LS_THREADS)
logit_stats_kernel(const __nv_bfloat16* Z, long long ldz, int V, int T, int slots, float c, float2* stats) {
  __shared__ uint4 staged[LS_THREADS * 16];
  faar_pdl_sync();
  const int lane = threadIdx.x & 31, unit = lane & 15;
  uint4* const mine = staged + (threadIdx.x >> 5) * 512;
  const long long all = (long long)T * slots, step = (long long)gridDim.x * LS_THREADS;
  for (long long i0 = (long long)blockIdx.x * LS_THREADS + (threadIdx.x & ~31); i0 < all; i0 += step) {
    const long long first = i0 + (lane >> 4);             // this lane's 16 bytes are of every second of the warp's 32 slots
    long long row = first / slots;
    int slot = (int)(first - row * slots);
    uint4 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int col = 128 * slot + 8 * unit;
      v[k] = row < T && col < V ? __ldg(reinterpret_cast<const uint4*>(Z + row * ldz + col)) : make_uint4(0u, 0u, 0u, 0u);
      for (slot += 2; slot >= slots; slot -= slots) ++row;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int j = 2 * k + (lane >> 4);
      mine[16 * j + (unit ^ (j & 15))] = v[k];
    }
    __syncwarp();
    const long long i = i0 + lane;
    if (i < all) {
      const int n = min(128, V - 128 * (int)(i % slots));
      float m = -INFINITY, s = 0.f;
      for (int g = 0; g < n / 16; ++g) {
        float lo[8], hi[8], x[16];
        unpack8(mine[16 * lane + (2 * g ^ unit)], lo);
        unpack8(mine[16 * lane + ((2 * g + 1) ^ unit)], hi);
#pragma unroll
        for (int j = 0; j < 8; ++j) { x[j] = lo[j]; x[8 + j] = hi[j]; }
        faar_stats_update(x, c, m, s);
      }
      stats[i] = make_float2(m, s);
    }
    __syncwarp();
  }
}

}  // namespace

int faar_launch_logit_stats(faar_ctx* ctx, int T, int vocab, const void* Z, int64_t ldz, float tau, float2* stats) {
  faar_prof_scope ps(ctx, FAAR_K_GLUE);
  const int slots = (vocab + 127) / 128;
  long long blocks = ((long long)T * slots + LS_THREADS - 1) / LS_THREADS;
  if (blocks > 6ll * ctx->num_sms) blocks = 6ll * ctx->num_sms;
  faar_launch_pdl(ctx, logit_stats_kernel, dim3((unsigned)blocks), dim3(LS_THREADS), 0, reinterpret_cast<const __nv_bfloat16*>(Z),
                  (long long)ldz, vocab, T, slots, (float)(1.4426950408889634 / (double)tau), stats);
  return (int)cudaGetLastError();
}

int faar_launch_align_loss(faar_ctx* ctx, int T, int vocab, int hidden, const void* Z_fp, const void* Z_q, int64_t ldz,
                           const void* H_fp, const void* H_q, int64_t ldh, float tau, float lambda_kl, void* dZ_q,
                           void* dH_q, float* kl_partials, float* mse_partials, uint32_t* finished, float* loss_out2, const float2* stats_fp,
                           const float2* stats_q) {
  AlignParams p;
  p.Zfp = reinterpret_cast<const __nv_bfloat16*>(Z_fp); p.Zq = reinterpret_cast<const __nv_bfloat16*>(Z_q);
  p.ldz = ldz; p.V = vocab;
  p.Hfp = reinterpret_cast<const __nv_bfloat16*>(H_fp); p.Hq = reinterpret_cast<const __nv_bfloat16*>(H_q);
  p.ldh = ldh; p.D = hidden;
  p.dZ = reinterpret_cast<__nv_bfloat16*>(dZ_q); p.dH = reinterpret_cast<__nv_bfloat16*>(dH_q);
  p.c = (float)(1.4426950408889634 / (double)tau);
  p.gscale = (float)((double)lambda_kl / ((double)tau * (double)T));
  p.kl_partials = kl_partials; p.mse_partials = mse_partials;
  p.loss_out2 = loss_out2; p.finished = finished; p.kl_scale = (float)(1.0 / (double)T);
  p.T = T;
  // Persistent CTAs, one per SM.  Two tokens' rows (4 vocab bytes each) per CTA or cluster are in use at a time and are to
  // stay in L2: a CTA per token up to 130 MB, then two.  1500 tokens, one against two, us: vocabulary 88000 (99 MB) 214,
  // 239; 96000 230, 248; 104000 (117 MB) 258, 271.
  faar_prof_scope ps(ctx, FAAR_K_ALIGN_LOSS);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.stream = ctx->stream;
  cfg.attrs = attr;
  const int sms = ctx->num_sms;
  const bool given = stats_fp && stats_q;
  p.stats_fp = stats_fp; p.stats_q = stats_q; p.slots = (vocab + 127) / 128;
  cfg.blockDim = dim3(given ? AL_STATS_THREADS : AL_THREADS);
  const bool two = !given && T > sms / 2 && 2ll * (T < sms ? T : sms) * 4 * vocab > 130ll << 20;
  const int most = given ? sms * (AL_THREADS / AL_STATS_THREADS) : (two ? sms / 2 : sms), n = T < most ? T : most;
  cfg.gridDim = dim3(two ? 2 * n : n);
  cfg.numAttrs = two ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, given ? align_loss_kernel<1, true> : (two ? align_loss_kernel<2, false> : align_loss_kernel<1, false>), p);
  if (e != cudaSuccess) return (int)e;
  return (int)cudaGetLastError();
}
