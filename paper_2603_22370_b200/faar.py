"""Binding of libfaar.so (ctypes; the calls that enqueue work go through the native marshalling module
_faarbind, which is several microseconds a call faster).  Argument marshalling only: every function
below has the name and the arguments of the C entry point it calls; tensors
are torch CUDA tensors whose `data_ptr()` is handed through.  There is no
fallback: if the library is missing or a call fails, an exception is raised.
"""
from __future__ import annotations

import ctypes as C
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
#: the library this process binds: libfaar.so next to this file, or the file FAAR_LIB names (the debug build)
LIB_PATH = os.environ.get("FAAR_LIB") or os.path.join(_HERE, "libfaar.so")

OK, ERR_INVALID_ARG, ERR_SHAPE, ERR_ALIGN, ERR_DTYPE, ERR_WORKSPACE, ERR_ARCH, ERR_CUDA, ERR_TIMEOUT = range(9)
BF16, F32 = 0, 1

_P, _I, _L, _F, _Z, _U = C.c_void_p, C.c_int, C.c_int64, C.c_float, C.c_size_t, C.c_uint

#: every exported function: (result type, argument types), as declared in include/faar.h
SIGNATURES = {
    "faar_create": (_I, [_P, _I, _P]),
    "faar_destroy": (_I, [_P]),
    "faar_set_stream": (_I, [_P, _P]),
    "faar_status_string": (C.c_char_p, [_I]),
    "faar_last_cuda_error": (_I, [_P]),
    "faar_tune_tile_n": (_I, [_P, _I]),
    "faar_tune_tail_split": (_I, [_P, _I]),
    "faar_last_tail_split": (_I, [_P, _P]),
    "faar_last_gemm_config": (_I, [_P, _P, _P]),
    "faar_workspace_size": (_I, [_P, _P]),
    "faar_workspace_init": (_I, [_P, _P, _Z]),
    "faar_check_status": (_I, [_P, _P, _P]),
    "faar_selftest_wait_timeout": (_I, [_P, _P, _Z, _U]),
    "faar_profile_begin": (_I, [_P]),
    "faar_profile_end": (_I, [_P, _P, _I, _P]),
    "faar_kernel_name": (C.c_char_p, [_I]),
    "faar_softquant_init": (_I, [_P, _P, _P, _F, _P, _P, _P, _P, _P, _Z]),
    "faar_softquant_eval": (_I, [_P, _P, _P, _P, _P, _P, _F, _P, _P, _P]),
    "faar_softquant_operand_f32": (_I, [_P, _P, _P, _P, _P, _P, _F, _P]),
    "faar_transpose_bf16": (_I, [_P, _I, _I, _P, _L, _P, _L]),
    "faar_act_fakequant": (_I, [_P, _I, _I, _P, _L, _F, _P, _L, _P, _P, _P, _P, _Z]),
    "faar_layer_ref": (_I, [_P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_fwd": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_dx": (_I, [_P, _P, _F, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_dx_operand": (_I, [_P, _P, _P, _P, _P, _P, _Z]),
    "faar_round_loss": (_I, [_P, _P, _L, _P, _P, _Z]),
    "faar_round_loss_static": (_I, [_P, _P, _L, _P]),
    "faar_round_loss_static_max_n": (_L, []),
    "faar_layer_bwd": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_bwd_rowmajor": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_step": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_step_rowmajor": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_layer_step_host": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z]),
    "faar_nvfp4_expand": (_I, [_P, _I, _I, _P, _P, _P, _L]),
    "faar_layer_step_host_nvfp4": (_I, [_P] * 19 + [_Z]),
    "faar_harden_pack": (_I, [_P, _P, _P, _P, _P, _P, _P, _P, _P, _P, _I]),
    "faar_align_loss_workspace_size": (_I, [_I, _I, _P]),
    "faar_align_loss": (_I, [_P, _I, _I, _I, _P, _P, _L, _P, _P, _L, _F, _F, _P, _P, _P, _P, _Z]),
    "faar_logit_stats_size": (_I, [_P, _I, _I, _P]),
    "faar_logit_stats_pay": (_I, [_P, _I, _I, _P]),
    "faar_logit_stats": (_I, [_P, _I, _I, _P, _L, _F, _P, _Z]),
    "faar_align_loss_stats": (_I, [_P, _I, _I, _I, _P, _P, _L, _P, _P, _L, _F, _F, _P, _P, _Z, _P, _P, _P, _P, _Z]),
    "faar_swizzle_scales": (_I, [_P, _I, _I, _P, _P, _Z]),
    "faar_silu_mul": (_I, [_P, _I, _I, _P, _L, _P, _L, _P, _L]),
    "faar_rmsnorm": (_I, [_P, _I, _I, _P, _L, _P, _F, _P, _L, _P]),
    "faar_rmsnorm_bwd": (_I, [_P, _I, _I, _P, _L, _P, _L, _P, _P, _P, _L, _P, _L]),
    "faar_add_rmsnorm": (_I, [_P, _I, _I, _P, _L, _P, _L, _P, _L, _P, _F, _P, _L, _P]),
    "faar_rmsnorm_bwd_sum": (_I, [_P, _I, _I, _P, _P, _P, _L, _P, _L, _P, _P, _P, _L, _P, _L]),
    "faar_rope": (_I, [_P, _I, _I, _I, _P, _L, _P, _F, _I, _P, _L]),
    "faar_silu_mul_bwd": (_I, [_P, _I, _I, _P, _L, _P, _L, _P, _L, _P, _L, _P, _L]),
    "faar_embedding": (_I, [_P, _I, _I, _I, _P, _L, _P, _P, _L]),
    "faar_add": (_I, [_P, _I, _I, _P, _L, _P, _L, _P, _L]),
    "faar_tune_attention": (_I, [_P, _I]),
    "faar_attention_status": (_I, [_P, _P]),
    "faar_tune_wide_tiles": (_I, [_P, _I]),
    "faar_attention_fwd": (_I, [_P, _I, _I, _I, _I, _I, _P, _L, _P, _P, _L, _P, _L, _P]),
    "faar_attention_bwd": (_I, [_P, _I, _I, _I, _I, _I, _P, _L, _P, _P, _L, _P, _P, _L, _P, _P, _P, _P, _P]),
    "faar_model_sizes": (_I, [_P, _I, _I, _I, _P, _P]),
    "faar_model_forward": (_I, [_P, _P, _I, _I, _P, _P, _I, _F, _I, _P, _Z, _P, _P, _P, _Z]),
    "faar_model_overlap": (_I, [_P, _I, _I, _P]),
    "faar_model_forward_both": (_I, [_P, _P, _I, _I, _P, _P, _F, _P, _Z, _P, _P, _P, _Z, _P, _P, _P, _Z]),
    "faar_model_forward_stats": (_I, [_P, _P, _I, _I, _P, _P, _I, _F, _I, _P, _Z, _P, _P, _F, _P, _Z, _P, _Z]),
    "faar_model_forward_both_stats": (_I, [_P, _P, _I, _I, _P, _P, _F, _P, _Z, _P, _P, _P, _Z, _P, _P, _F, _P, _P, _Z, _P, _Z]),
    "faar_model_backward": (_I, [_P, _P, _I, _I, _P, _P, _P, _Z, _P, _L, _P, _P, _Z, _P, _Z]),
    "faar_nvfp4_gemm": (_I, [_P, _I, _I, _I, _P, _P, _P, _P, _P, _P, _P, _L, _P, _Z]),
}
EXPORTS = list(SIGNATURES)


class HParams(C.Structure):
    _fields_ = [("beta", C.c_float), ("lambda_round", C.c_float), ("mse_scale", C.c_float), ("opt", C.c_int),
                ("lr", C.c_float), ("beta1", C.c_float), ("beta2", C.c_float), ("eps", C.c_float),
                ("step", C.c_int), ("act_scale", C.c_float), ("beta_next", C.c_float), ("wsoft_ready", C.c_int)]


class Shape(C.Structure):
    _fields_ = [("O", C.c_int), ("K", C.c_int), ("T", C.c_int), ("ldw", C.c_int64), ("ldx", C.c_int64),
                ("ldxt", C.c_int64), ("ldy", C.c_int64), ("w_dtype", C.c_int), ("yref_dtype", C.c_int),
                ("yref_transposed", C.c_int)]


class Linear(C.Structure):
    _fields_ = [("rows", C.c_int), ("V", _P), ("code", _P), ("scales", _P), ("s_global", _P), ("adam_m", _P), ("adam_u", _P),
                ("dV", _P)]


class LinearGroup(C.Structure):
    _fields_ = [("n", C.c_int), ("W", _P), ("Wsoft", _P), ("lin", Linear * 3)]


class Block(C.Structure):
    _fields_ = [("qkv", LinearGroup), ("o", LinearGroup), ("gate_up", LinearGroup), ("down", LinearGroup), ("attn_norm", _P),
                ("mlp_norm", _P)]


class Model(C.Structure):
    _fields_ = [("vocab", C.c_int), ("hidden", C.c_int), ("n_layers", C.c_int), ("n_heads", C.c_int), ("n_kv_heads", C.c_int),
                ("head_dim", C.c_int), ("ffn", C.c_int), ("eps", C.c_float), ("theta", C.c_float), ("embed", _P), ("lm_head", _P),
                ("lm_head_t", _P), ("ld_lm_head_t", C.c_int64), ("final_norm", _P), ("blocks", _P)]


class FaarError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} (status {status})")


_lib = None


def lib() -> C.CDLL:
    """Loads libfaar.so (built in-tree by `paper_2603_22370_b200.build`)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise FileNotFoundError(f"{LIB_PATH} is missing; run `python -m paper_2603_22370_b200.build`")
        l = C.CDLL(LIB_PATH)
        for name, (res, args) in SIGNATURES.items():
            fn = getattr(l, name)
            fn.restype, fn.argtypes = res, args
        _lib = l
    return _lib


_native = None


def _fast():
    """The native marshalling module, bound to the same library as lib()."""
    global _native
    if _native is None:
        lib()
        try:
            from . import _faarbind
        except ImportError as e:
            raise ImportError(f"{e}; run `python -m paper_2603_22370_b200.build`") from e
        _faarbind.load(LIB_PATH)
        _native = _faarbind
    return _native


def status_string(status: int) -> str:
    return lib().faar_status_string(int(status)).decode()


def _p(t):
    if t is None:
        return C.c_void_p(0)
    if isinstance(t, int):
        return C.c_void_p(t)
    assert t.is_cuda, "device tensors only"
    return C.c_void_p(t.data_ptr())


def _check(status: int, where: str):
    if status != OK:
        raise FaarError(status, where)


def make_shape(O, K, T, ldw=None, ldx=None, ldxt=None, ldy=None, w_dtype=BF16, yref_dtype=BF16,
               yref_transposed=0) -> Shape:
    """yref_transposed: Y_ref (and the optional Y_q) are stored [O, ldy], ldy >= T rounded up to 16."""
    if ldy is None:
        ldy = (T + 15) // 16 * 16 if yref_transposed else O
    return Shape(O, K, T, ldw if ldw is not None else K, ldx if ldx is not None else K,
                 ldxt if ldxt is not None else (T + 7) // 8 * 8, ldy, w_dtype, yref_dtype, yref_transposed)


def make_hparams(beta=4.0, lambda_round=1.0, mse_scale=1.0, opt=1, lr=1e-2, beta1=0.9, beta2=0.999, eps=1e-8,
                 step=1, act_scale=0.0, beta_next=0.0, wsoft_ready=0) -> HParams:
    return HParams(beta, lambda_round, mse_scale, opt, lr, beta1, beta2, eps, step, act_scale, beta_next, wsoft_ready)


class Context:
    """Owns a faar_ctx bound to a device and a stream, plus (optionally) a workspace tensor."""

    def __init__(self, device: int = 0, stream: torch.cuda.Stream | None = None):
        self._h = C.c_void_p(0)
        self.device = device
        s = stream.cuda_stream if stream is not None else torch.cuda.current_stream(device).cuda_stream
        _check(lib().faar_create(C.byref(self._h), device, C.c_void_p(s)), "faar_create")
        self._n = self._h.value                     # the handle as the native marshalling takes it
        self.ws = None

    def close(self):
        if self._h:
            lib().faar_destroy(self._h)
            self._h = C.c_void_p(0)
            self._n = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    def set_stream(self, stream: torch.cuda.Stream):
        _check(lib().faar_set_stream(self._h, C.c_void_p(stream.cuda_stream)), "faar_set_stream")

    def last_cuda_error(self) -> int:
        return lib().faar_last_cuda_error(self._h)

    def workspace(self, shape: Shape) -> torch.Tensor:
        """Allocates (with torch) and initialises a workspace large enough for `shape`."""
        n = workspace_size(shape)
        if self.ws is None or self.ws.numel() < n:
            self.ws = torch.empty(n, dtype=torch.uint8, device=f"cuda:{self.device}")
            workspace_init(self, self.ws)
        return self.ws


def tune_tile_n(ctx: Context, bn: int):
    """Forces the GEMM tile width (multiple of 16 in [128, 256]); 0 restores the automatic choice."""
    _check(lib().faar_tune_tile_n(ctx._h, C.c_int(bn)), "faar_tune_tile_n")


def tune_tail_split(ctx: Context, columns: int):
    """Forces how many trailing tile columns are cut into half-width tiles (-1 = automatic, 0 = none)."""
    _check(lib().faar_tune_tail_split(ctx._h, C.c_int(columns)), "faar_tune_tail_split")


def last_tail_split(ctx: Context) -> int:
    n = C.c_int(0)
    _check(lib().faar_last_tail_split(ctx._h, C.byref(n)), "faar_last_tail_split")
    return n.value


def last_gemm_config(ctx: Context) -> tuple[int, int]:
    """(tile width, CTA pairs) of the most recent GEMM launch on this context."""
    bn, pairs = C.c_int(0), C.c_int(0)
    _check(lib().faar_last_gemm_config(ctx._h, C.byref(bn), C.byref(pairs)), "faar_last_gemm_config")
    return bn.value, pairs.value


def workspace_size(shape: Shape) -> int:
    n = C.c_size_t(0)
    _check(lib().faar_workspace_size(C.byref(shape), C.byref(n)), "faar_workspace_size")
    return n.value


def workspace_init(ctx: Context, ws: torch.Tensor):
    _check(_fast().faar_workspace_init(ctx._n, ws, ws.numel()), "faar_workspace_init")


def selftest_wait_timeout(ctx: Context, ws: torch.Tensor, limit_us: int = 1000):
    _check(lib().faar_selftest_wait_timeout(ctx._h, _p(ws), C.c_size_t(ws.numel()), C.c_uint(limit_us)),
           "faar_selftest_wait_timeout")


def check_status(ctx: Context, ws: torch.Tensor) -> int:
    d = C.c_uint32(0)
    st = lib().faar_check_status(ctx._h, _p(ws), C.byref(d))
    if st != OK:
        raise FaarError(st, f"faar_check_status (detail 0x{d.value:x})")
    return st


def softquant_init(ctx, shape, W, s_global_in, scales, s_global_out, code, V_init, ws):
    _check(_fast().faar_softquant_init(ctx._n, shape, W, s_global_in, scales, s_global_out, code, V_init, ws,
           ws.numel()), "faar_softquant_init")


def softquant_eval(ctx, shape, V, code, scales, s_global, beta, W_soft, h, W_soft_bf16=None):
    _check(_fast().faar_softquant_eval(ctx._n, shape, V, code, scales, s_global, beta, W_soft, h, W_soft_bf16),
           "faar_softquant_eval")


def softquant_operand_f32(ctx, shape, V, code, scales, s_global, beta, W_operand):
    _check(_fast().faar_softquant_operand_f32(ctx._n, shape, V, code, scales, s_global, beta, W_operand),
           "faar_softquant_operand_f32")


def act_fakequant(ctx, T, K, X, ldx, s_global_in, Xq_units, ldq, s_global_out, packed, scales, ws):
    _check(_fast().faar_act_fakequant(ctx._n, T, K, X, ldx, s_global_in, Xq_units, ldq, s_global_out, packed, scales,
           ws, ws.numel()), "faar_act_fakequant")


def align_loss_workspace_size(T, vocab) -> int:
    n = C.c_size_t(0)
    _check(lib().faar_align_loss_workspace_size(T, vocab, C.byref(n)), "faar_align_loss_workspace_size")
    return n.value


def align_loss(ctx, T, vocab, hidden, Z_fp, Z_q, ldz, H_fp, H_q, ldh, tau, lambda_kl, dZ_q, dH_q, loss_out2, ws):
    _check(_fast().faar_align_loss(ctx._n, T, vocab, hidden, Z_fp, Z_q, ldz, H_fp, H_q, ldh, tau, lambda_kl, dZ_q,
           dH_q, loss_out2, ws, ws.numel()), "faar_align_loss")


def logit_stats_size(ctx, T, vocab) -> int:
    n = C.c_size_t(0)
    _check(lib().faar_logit_stats_size(ctx._h, T, vocab, C.byref(n)), "faar_logit_stats_size")
    return n.value


def logit_stats_pay(ctx, T, vocab) -> bool:
    n = C.c_int(0)
    _check(lib().faar_logit_stats_pay(ctx._h, T, vocab, C.byref(n)), "faar_logit_stats_pay")
    return bool(n.value)


def _stats_bytes(*stats) -> int:
    """Bytes of the smallest of the buffers; none for one that is missing, which the call refuses."""
    return min(0 if s is None else s.nbytes for s in stats)


def logit_stats(ctx, T, vocab, Z, ldz, tau, stats):
    _check(_fast().faar_logit_stats(ctx._n, T, vocab, Z, ldz, tau, stats, _stats_bytes(stats)), "faar_logit_stats")


def align_loss_stats(ctx, T, vocab, hidden, Z_fp, Z_q, ldz, H_fp, H_q, ldh, tau, lambda_kl, stats_fp, stats_q, dZ_q, dH_q, loss_out2, ws):
    _check(_fast().faar_align_loss_stats(ctx._n, T, vocab, hidden, Z_fp, Z_q, ldz, H_fp, H_q, ldh, tau, lambda_kl, stats_fp, stats_q,
                                         _stats_bytes(stats_fp, stats_q), dZ_q, dH_q, loss_out2, ws, ws.numel()), "faar_align_loss_stats")


def swizzle_scales(ctx, rows, cols, scales, scales_tiled):
    _check(_fast().faar_swizzle_scales(ctx._n, rows, cols, scales, scales_tiled, scales_tiled.numel()),
           "faar_swizzle_scales")


def silu_mul(ctx, rows, cols, gate, ldg, up, ldu, out, ldo):
    _check(_fast().faar_silu_mul(ctx._n, rows, cols, gate, ldg, up, ldu, out, ldo), "faar_silu_mul")


def rmsnorm(ctx, rows, cols, x, ldx, g, eps, y, ldy, rstd=None):
    _check(_fast().faar_rmsnorm(ctx._n, rows, cols, x, ldx, g, eps, y, ldy, rstd), "faar_rmsnorm")


def rmsnorm_bwd(ctx, rows, cols, dy, lddy, x, ldx, g, rstd, add, ldadd, dx, lddx):
    _check(_fast().faar_rmsnorm_bwd(ctx._n, rows, cols, dy, lddy, x, ldx, g, rstd, add, ldadd, dx, lddx), "faar_rmsnorm_bwd")


def add_rmsnorm(ctx, rows, cols, a, lda, b, ldb, total, lds, g, eps, y, ldy, rstd=None):
    _check(_fast().faar_add_rmsnorm(ctx._n, rows, cols, a, lda, b, ldb, total, lds, g, eps, y, ldy, rstd),
           "faar_add_rmsnorm")


def rmsnorm_bwd_sum(ctx, rows, cols, dy, dy2, dy3, lddy, x, ldx, g, rstd, add, ldadd, dx, lddx):
    _check(_fast().faar_rmsnorm_bwd_sum(ctx._n, rows, cols, dy, dy2, dy3, lddy, x, ldx, g, rstd, add, ldadd, dx,
           lddx), "faar_rmsnorm_bwd_sum")


def rope(ctx, rows, n_heads, head_dim, x, ldx, positions, theta, inverse, y, ldy):
    _check(_fast().faar_rope(ctx._n, rows, n_heads, head_dim, x, ldx, positions, theta, int(inverse), y, ldy), "faar_rope")


def silu_mul_bwd(ctx, rows, cols, dout, ldd, gate, ldg, up, ldu, dgate, lddg, dup, lddu):
    _check(_fast().faar_silu_mul_bwd(ctx._n, rows, cols, dout, ldd, gate, ldg, up, ldu, dgate, lddg, dup, lddu),
           "faar_silu_mul_bwd")


def embedding(ctx, rows, cols, vocab, table, ldt, tokens, out, ldo):
    _check(_fast().faar_embedding(ctx._n, rows, cols, vocab, table, ldt, tokens, out, ldo), "faar_embedding")


def add(ctx, rows, cols, a, lda, b, ldb, out, ldo):
    _check(_fast().faar_add(ctx._n, rows, cols, a, lda, b, ldb, out, ldo), "faar_add")


def tune_wide_tiles(ctx, mode: int):
    """1: 256 x 512 GEMM tiles whenever the shape allows; 0: never; -1 (the default): for long forward products that
    tiles of 288 to 512 columns finish in one wave, of the least such width.  0 and 1 keep contractions whole."""
    _check(lib().faar_tune_wide_tiles(ctx._h, mode), "faar_tune_wide_tiles")


def attention_status(ctx):
    """Raises FaarError(TIMEOUT) if a wait of the tcgen05 attention kernel gave up (call after a synchronise)."""
    code = C.c_uint32(0)
    _check(lib().faar_attention_status(ctx._h, C.byref(code)), f"faar_attention_status (code {code.value:#x})")


def tune_attention(ctx, mode: int):
    """0 = tcgen05 kernels forward and backward (default), 2 = register-resident mma.sync kernels (head_dim 64),
    1 = the shared-memory fragment kernels."""
    _check(lib().faar_tune_attention(ctx._h, mode), "faar_tune_attention")


def attention_fwd(ctx, batch, seq, n_heads, n_kv_heads, head_dim, q, ldq, k, v, ldkv, out, ldo, lse):
    _check(_fast().faar_attention_fwd(ctx._n, batch, seq, n_heads, n_kv_heads, head_dim, q, ldq, k, v, ldkv, out, ldo,
           lse), "faar_attention_fwd")


def attention_bwd(ctx, batch, seq, n_heads, n_kv_heads, head_dim, q, ldq, k, v, ldkv, out, dout, ldo, lse, dsum, dq, dk, dv):
    _check(_fast().faar_attention_bwd(ctx._n, batch, seq, n_heads, n_kv_heads, head_dim, q, ldq, k, v, ldkv, out,
           dout, ldo, lse, dsum, dq, dk, dv), "faar_attention_bwd")


def nvfp4_gemm(ctx, M, N, K, A_packed, A_scales_tiled, A_s_global, B_packed, B_scales_tiled, B_s_global, C, ldc, ws):
    _check(_fast().faar_nvfp4_gemm(ctx._n, M, N, K, A_packed, A_scales_tiled, A_s_global, B_packed, B_scales_tiled,
           B_s_global, C, ldc, ws, ws.numel()), "faar_nvfp4_gemm")


def model_sizes(model: Model, batch: int, seq: int, keep: int) -> tuple[int, int]:
    """(arena bytes, scratch bytes) of a pass over the model."""
    a, b = C.c_size_t(0), C.c_size_t(0)
    _check(lib().faar_model_sizes(C.byref(model), batch, seq, keep, C.byref(a), C.byref(b)), "faar_model_sizes")
    return a.value, b.value


class Region(int):
    """Device memory by its address, `nbytes` long: stands for a tensor in the calls of a model's passes."""

    def __new__(cls, address: int, nbytes: int):
        r = int.__new__(cls, address)
        r.nbytes = nbytes
        return r

    def numel(self) -> int:
        return self.nbytes


def model_forward(ctx, model, batch, seq, tokens, positions, quantised, beta, keep, arena, Z, H, ws):
    _check(_fast().faar_model_forward(ctx._n, model, batch, seq, tokens, positions, int(quantised), beta, int(keep), arena,
                                      arena.numel(), Z, H, ws, ws.numel()), "faar_model_forward")


def model_overlap(model: Model, batch: int, seq: int) -> bool:
    """Whether the two forward passes of a step gain from running at once (model_forward_both)."""
    n = C.c_int(0)
    _check(lib().faar_model_overlap(C.byref(model), batch, seq, C.byref(n)), "faar_model_overlap")
    return bool(n.value)


def model_forward_both(ctx, model, batch, seq, tokens, positions, beta, arena_fp, Z_fp, H_fp, arena, Z, H, ws):
    _check(_fast().faar_model_forward_both(ctx._n, model, batch, seq, tokens, positions, beta, arena_fp, arena_fp.numel(), Z_fp, H_fp,
                                           arena, arena.numel(), Z, H, ws, ws.numel()), "faar_model_forward_both")


def model_forward_stats(ctx, model, batch, seq, tokens, positions, quantised, beta, keep, arena, Z, H, tau, stats, ws):
    _check(_fast().faar_model_forward_stats(ctx._n, model, batch, seq, tokens, positions, int(quantised), beta, int(keep), arena,
                                            arena.numel(), Z, H, tau, stats, _stats_bytes(stats), ws, ws.numel()),
           "faar_model_forward_stats")


def model_forward_both_stats(ctx, model, batch, seq, tokens, positions, beta, arena_fp, Z_fp, H_fp, arena, Z, H, tau, stats_fp, stats, ws):
    _check(_fast().faar_model_forward_both_stats(ctx._n, model, batch, seq, tokens, positions, beta, arena_fp, arena_fp.numel(), Z_fp, H_fp,
                                                 arena, arena.numel(), Z, H, tau, stats_fp, stats, _stats_bytes(stats_fp, stats), ws,
                                                 ws.numel()),
           "faar_model_forward_both_stats")


def model_backward(ctx, model, batch, seq, positions, hp, arena, dZ, ldz, dH, scratch, ws):
    _check(_fast().faar_model_backward(ctx._n, model, batch, seq, positions, hp, arena, arena.numel(), dZ, ldz, dH, scratch,
                                       scratch.numel(), ws, ws.numel()), "faar_model_backward")


def transpose_bf16(ctx, rows, cols, inp, ld_in, out, ld_out):
    _check(_fast().faar_transpose_bf16(ctx._n, rows, cols, inp, ld_in, out, ld_out), "faar_transpose_bf16")


def layer_ref(ctx, shape, X, W, Y_ref, ws):
    _check(_fast().faar_layer_ref(ctx._n, shape, X, W, Y_ref, ws, ws.numel()), "faar_layer_ref")


def layer_fwd(ctx, shape, hp, X, Y_ref, V, code, scales, s_global, dYt, loss_mse, Y_q, ws):
    _check(_fast().faar_layer_fwd(ctx._n, shape, hp, X, Y_ref, V, code, scales, s_global, dYt, loss_mse, Y_q, ws,
           ws.numel()), "faar_layer_fwd")


def layer_dx(ctx, shape, beta, dY, V, code, scales, s_global, WsoftT, dX, ws):
    _check(_fast().faar_layer_dx(ctx._n, shape, beta, dY, V, code, scales, s_global, WsoftT, dX, ws, ws.numel()),
           "faar_layer_dx")


def layer_dx_operand(ctx, shape, dY, Wsoft, dX, ws):
    _check(_fast().faar_layer_dx_operand(ctx._n, shape, dY, Wsoft, dX, ws, ws.numel()), "faar_layer_dx_operand")


def round_loss(ctx, V, N, loss_round, ws):
    _check(_fast().faar_round_loss(ctx._n, V, N, loss_round, ws, ws.numel()), "faar_round_loss")


def round_loss_static(ctx, V, N, loss_round):
    """Round Loss without a workspace: for callers that may not allocate device memory.  The scratch
    is a fixed array inside libfaar.so; N is limited to round_loss_static_max_n()."""
    _check(_fast().faar_round_loss_static(ctx._n, V, N, loss_round), "faar_round_loss_static")


def round_loss_static_max_n() -> int:
    return int(lib().faar_round_loss_static_max_n())


def layer_bwd(ctx, shape, hp, dYt, Xt, V, code, scales, s_global, adam_m, adam_u, dV, ws):
    _check(_fast().faar_layer_bwd(ctx._n, shape, hp, dYt, Xt, V, code, scales, s_global, adam_m, adam_u, dV, ws,
           ws.numel()), "faar_layer_bwd")


def layer_bwd_rowmajor(ctx, shape, hp, dY, X, V, code, scales, s_global, adam_m, adam_u, dV, ws):
    _check(_fast().faar_layer_bwd_rowmajor(ctx._n, shape, hp, dY, X, V, code, scales, s_global, adam_m, adam_u, dV,
           ws, ws.numel()), "faar_layer_bwd_rowmajor")


def layer_step(ctx, shape, hp, X, Xt, Y_ref, V, code, scales, s_global, adam_m, adam_u, loss_out2, ws):
    _check(_fast().faar_layer_step(ctx._n, shape, hp, X, Xt, Y_ref, V, code, scales, s_global, adam_m, adam_u,
           loss_out2, ws, ws.numel()), "faar_layer_step")


def layer_step_rowmajor(ctx, shape, hp, X, Y_ref, V, code, scales, s_global, adam_m, adam_u, loss_out2, ws):
    _check(_fast().faar_layer_step_rowmajor(ctx._n, shape, hp, X, Y_ref, V, code, scales, s_global, adam_m, adam_u,
           loss_out2, ws, ws.numel()), "faar_layer_step_rowmajor")


def harden_pack(ctx, shape, V, code, scales, s_global, packed, scales_out, decisions, W_final, wfinal_dtype=F32):
    _check(_fast().faar_harden_pack(ctx._n, shape, V, code, scales, s_global, packed, scales_out, decisions, W_final,
           wfinal_dtype), "faar_harden_pack")


def layer_step_host(ctx, shape, hp, X_host, Y_ref_host, W, X_dev, Xt_dev, Yref_dev, V, code, scales, s_global, adam_m,
                    adam_u, loss_dev2, loss_host2, ws):
    """X_host, Y_ref_host, loss_host2 are (pinned) CPU tensors; the rest are device tensors.  Y_ref_host None:
    the target is computed on the device from the copied X and W."""
    _check(_fast().faar_layer_step_host(ctx._n, shape, hp, X_host.data_ptr(),
           None if Y_ref_host is None else Y_ref_host.data_ptr(), W, X_dev, Xt_dev, Yref_dev, V, code, scales, s_global, adam_m, adam_u, loss_dev2,
           loss_host2.data_ptr(), ws, ws.numel()), "faar_layer_step_host")


def nvfp4_expand(ctx, rows, K, packed, scales, out, ld):
    _check(_fast().faar_nvfp4_expand(ctx._n, rows, K, packed, scales, out, ld), "faar_nvfp4_expand")


def layer_step_host_nvfp4(ctx, shape, hp, Xpacked_host, Xscales_host, Y_ref_host, Xpacked_dev, Xscales_dev, Xq_dev, Yref_dev,
                          V, code, scales, s_global, adam_m, adam_u, loss_dev2, loss_host2, ws):
    """Host tensors (pinned): packed codes, block scales, frozen target, the two-float loss."""
    _check(_fast().faar_layer_step_host_nvfp4(ctx._n, shape, hp, Xpacked_host.data_ptr(), Xscales_host.data_ptr(),
           Y_ref_host.data_ptr(), Xpacked_dev, Xscales_dev, Xq_dev, Yref_dev, V, code, scales, s_global, adam_m,
           adam_u, loss_dev2, loss_host2.data_ptr(), ws, ws.numel()), "faar_layer_step_host_nvfp4")


class KernelTime(C.Structure):
    _fields_ = [("kernel", C.c_int), ("launches", C.c_int), ("total_ms", C.c_float)]


def profile_begin(ctx):
    _check(lib().faar_profile_begin(ctx._h), "faar_profile_begin")


def profile_end(ctx) -> dict:
    """{kernel name: (launches, total_ms)} for the kernels launched since profile_begin."""
    arr = (KernelTime * 32)()
    n = C.c_int(0)
    _check(lib().faar_profile_end(ctx._h, arr, 32, C.byref(n)), "faar_profile_end")
    l = lib()
    return {l.faar_kernel_name(arr[i].kernel).decode(): (arr[i].launches, arr[i].total_ms) for i in range(n.value)}
