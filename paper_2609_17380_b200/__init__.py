"""paper_2609_17380_b200: bit-exact, replayable transformer training-step arithmetic on B200.

Binding of libdet.so (see include/det.h).  Every function here has the name and the argument
order of its C-ABI entry point and only marshals arguments: torch tensors (CUDA, contiguous) are passed as
device pointers, the current torch CUDA stream as the stream.  The stream-ordered entry points are called by
_binding.so (csrc/binding.cpp), the size queries, the calls with tables and the test hooks through ctypes.
Nothing is computed in Python and there is no CPU fallback: importing the binding without the built library
raises.
"""
import ctypes as C
import os

import torch

_DIR = os.path.dirname(os.path.abspath(__file__))
_SO = os.path.join(_DIR, "libdet.so")

DET_OK = 0
DET_F32, DET_BF16 = 0, 1
DET_DEV_TARGET, DET_DEV_TIMEOUT, DET_DEV_NONFINITE = 1, 2, 4   # bits of a device status word
DEV_TARGET, DEV_TIMEOUT, DEV_NONFINITE = 1, 2, 4
STATUS_NAMES = {0: "DET_OK", -1: "DET_ERR_ARG", -2: "DET_ERR_SHAPE", -3: "DET_ERR_ALIGN", -4: "DET_ERR_WORKSPACE",
                -5: "DET_ERR_RANGE", -6: "DET_ERR_CUDA"}


class DetError(RuntimeError):
    def __init__(self, fn, code):
        super().__init__("%s returned %s (%d)" % (fn, STATUS_NAMES.get(code, "?"), code))
        self.code = code


class det_accum(C.Structure):
    _fields_ = [("accum", C.c_int), ("dp_shard", C.c_int), ("dp_replicate", C.c_int), ("pushes", C.c_int),
                ("nstack", C.c_int), ("level", C.c_int * 34), ("slot", C.c_int * 34),
                ("free_mask", C.c_ulonglong), ("n", C.c_size_t), ("bufs", C.c_void_p), ("inner_slot", C.c_int),
                ("gr_slot", C.c_int)]


class det_adamw_desc(C.Structure):
    _fields_ = [("lr", C.c_double), ("beta1", C.c_double), ("beta2", C.c_double), ("eps", C.c_double),
                ("weight_decay", C.c_double), ("step", C.c_int)]


# Result and arguments of every entry point, one letter each (p pointer, i int, z size_t, f float, l long long, u unsigned long
# long): the types that ctypes converts by, also for the calls of the native binding with numbers that are no Python int or float.
_CTYPES = {"p": C.c_void_p, "i": C.c_int, "z": C.c_size_t, "f": C.c_float, "l": C.c_longlong, "u": C.c_ulonglong}
_SIGNATURES = {
    "det_device_sm_count": "i", "det_launch_count": "u", "det_sum_ws_bytes": "zz", "det_sum": "ipzippzp",
    "det_sum_static_max_n": "z", "det_sum_static": "ipzipp", "det_grad_norm_ws_bytes": "zpi",
    "det_grad_norm": "ippifpppzpp", "det_scale_inplace": "ipzpp", "det_lsq_weight_scale_ws_bytes": "zii",
    "det_lsq_weight_scale": "ipiiippzp", "det_lsq_act_scale_init_ws_bytes": "zz", "det_lsq_act_scale_init": "ipzppzp",
    "det_lsq_quantize_weight_ws_bytes": "zii", "det_lsq_quantize_weight": "ippiiippppzp",
    "det_linear_fwd": "ippppiiipppp", "det_linear_fwd_q": "ippppiiippp", "det_linear_bwd_ws_bytes": "ziii",
    "det_linear_bwd": "ippppppppiiiippppzpp", "det_rmsnorm_fwd": "iippiifppp", "det_rmsnorm_fwd_q": "ippiifppppp",
    "det_rmsnorm_bwd_ws_bytes": "zii", "det_rmsnorm_bwd": "iippppiipppzp", "det_headnorm_fwd": "ipiiifpipp",
    "det_headnorm_bwd": "ipipipiipip", "det_rope": "ipiiiippipip", "det_xent_ws_bytes": "zii",
    "det_xent_fwd": "ippiifpppppzpp", "det_xent_bwd": "ipppiiffp", "det_attn_fwd": "ipppiiiiiipipp",
    "det_attn_fwd_q": "ipppiiiiiipipppp", "det_attn_fwd_int8pv": "ipppiiiiiipippp", "det_attn_bwd_ws_bytes": "ziiii",
    "det_attn_bwd": "ippppppiiiiiiipppipzp", "det_attn_bwd_fixq_ws_bytes": "ziiii",
    "det_attn_bwd_fixq": "ippppppiiiiiiipppipzp", "det_swiglu_fwd": "ipiipp", "det_swiglu_fwd_q": "ipiipppp",
    "det_swiglu_bwd": "ippiipp", "det_residual_add": "ippzpp", "det_embed_fwd": "ipipiipp",
    "det_embed_bwd": "ipipiipp", "det_lmhead_fwd": "ippiiipp", "det_lmhead_bwd": "ipppiiippip",
    "det_lmhead_fwd_v2_ws_bytes": "ziii", "det_lmhead_fwd_v2": "ippiiippzpp", "det_lmhead_bwd_v2_ws_bytes": "ziii",
    "det_lmhead_bwd_v2": "ipppiiipppzpp", "det_attn_fwd_v2_ws_bytes": "ziii", "det_attn_fwd_v2": "ipppiiiipippzpp",
    "det_grad_accum_nbufs": "ii", "det_grad_accum_init": "ipiiizp", "det_grad_accum_push": "ippp",
    "det_grad_accum_result": "ippp", "det_adamw_step": "ipippppzp", "det_adamw_batch": "ipppppppipp",
    "det_tensor_hash_ws_bytes": "zz", "det_tensor_hash_async": "ipzppzp", "det_tensor_hash": "ipzppzp",
    "det_tensor_hash_batch_ws_bytes": "zpi", "det_tensor_hash_batch": "ippippzp", "det_test_prim": "iipppzp",
    "det_residual_rmsnorm_fwd": "ipppiifpppppp", "det_rmsnorm_bwd_residual": "ippppiippppzp", "det_test_igemm_tn": "ippiiipipp", "det_test_lmhead_tile": "iiippiiipip",
    "det_test_wait_timeout": "iplp", "det_test_wait_warp": "iplp", "det_test_attn_fwd": "iipppiiiiiipipppp",
    "det_test_attn_rows": "iiii", "det_test_lmhead_pick": "iiii",
}

# The entry points that csrc/binding.cpp calls directly: what it makes of each Python argument (letters as above; w: a workspace tensor or None,
# passed as address and size; s: the current stream, no argument of its own).
_PATTERNS = {
    "det_sum": "pzipws", "det_sum_static": "pzips", "det_scale_inplace": "pzps", "det_lsq_weight_scale": "piiipws",
    "det_lsq_act_scale_init": "pzpws", "det_lsq_quantize_weight": "ppiiipppws", "det_linear_fwd": "ppppiiippsp",
    "det_linear_fwd_q": "ppppiiipsp", "det_linear_bwd": "ppppppppiiiipppwsp", "det_rmsnorm_fwd": "ippiifpps",
    "det_rmsnorm_fwd_q": "ppiifpppps", "det_residual_rmsnorm_fwd": "pppiifppppps", "det_headnorm_fwd": "piiifpips",
    "det_headnorm_bwd": "pipipiipis", "det_rope": "piiiippipis", "det_rmsnorm_bwd": "ippppiippws",
    "det_rmsnorm_bwd_residual": "ppppiipppws", "det_xent_fwd": "ppiifppppwsp", "det_xent_bwd": "pppiiffs", "det_attn_fwd": "pppiiiiiipips",
    "det_attn_fwd_q": "pppiiiiiipippps", "det_attn_fwd_int8pv": "pppiiiiiipipsp", "det_attn_bwd": "ppppppiiiiiiipppiws",
    "det_attn_bwd_fixq": "ppppppiiiiiiipppiws", "det_swiglu_fwd": "piips", "det_swiglu_fwd_q": "piippps", "det_swiglu_bwd": "ppiips",
    "det_residual_add": "ppzps", "det_embed_fwd": "pipiips", "det_embed_bwd": "pipiips", "det_lmhead_fwd": "ppiiips",
    "det_lmhead_fwd_v2": "ppiiipwsp", "det_lmhead_bwd": "pppiiippis", "det_lmhead_bwd_v2": "pppiiippwsp",
    "det_attn_fwd_v2": "pppiiiipipwsp", "det_tensor_hash_async": "pzpws",
}


class _Calls:
    """The callables by name, there once the library is loaded."""

    def __getattr__(self, name):
        load()
        try:
            return self.__dict__[name]
        except KeyError:
            raise AttributeError(name) from None


_c = _Calls()
_lib = None


def load():
    """Load libdet.so; raises if it has not been built (python -m paper_2609_17380_b200.build)."""
    global _lib, _ptr, _stream
    if _lib is None:
        if not os.path.exists(_SO):
            raise ImportError("libdet.so is missing: build it with `python paper_2609_17380_b200/build.py` "
                              "(there is no fallback path)")
        lib = C.CDLL(_SO)
        for name, sig in _SIGNATURES.items():
            fn = getattr(lib, name)
            fn.restype = _CTYPES[sig[0]]
            fn.argtypes = [_CTYPES[c] for c in sig[1:]]
        from . import _binding
        _ptr, _stream = _binding.ptr, _binding.stream
        _c.__dict__.update(_binding.bind(_SO, _PATTERNS, _check, lib))
        _lib = lib
    return _lib


def _ptr(t):
    load()                       # replaces this function and _stream by the native ones
    return _ptr(t)


def _stream():
    load()
    return _stream()


def _check(fn, rc):
    if rc != DET_OK:
        raise DetError(fn, rc)


def _ws(ws):
    return (_ptr(ws), ws.numel() * ws.element_size()) if ws is not None else (None, 0)


# ---- information / primitives ------------------------------------------------------------------------
def det_device_sm_count():
    return load().det_device_sm_count()


def det_launch_count():
    return load().det_launch_count()


def det_test_prim(op, a, b, out):
    _check("det_test_prim", load().det_test_prim(op, _ptr(a), _ptr(b), _ptr(out), C.c_size_t(a.numel()), _stream()))


# ---- sums, norm, clip -----------------------------------------------------------------------------------
def det_sum_ws_bytes(n):
    return load().det_sum_ws_bytes(n)


def det_sum(x, n, squares, out, ws):
    _c.det_sum(x, n, squares, out, ws)


def det_sum_static_max_n():
    return load().det_sum_static_max_n()


def det_sum_static(x, n, squares, out):
    """det_sum without a workspace argument: scratch lives in a fixed array inside the library (see det.h)."""
    _c.det_sum_static(x, n, squares, out)


def _tensor_table(tensors):
    ptrs = (C.c_void_p * len(tensors))(*[t.data_ptr() for t in tensors])
    ns = (C.c_size_t * len(tensors))(*[t.numel() for t in tensors])
    return ptrs, ns


def det_grad_norm_ws_bytes(tensors):
    _, ns = _tensor_table(tensors)
    return load().det_grad_norm_ws_bytes(ns, len(tensors))


def det_grad_norm(tensors, max_norm, norm_out, coef_out, ws, status_dev=None):
    ptrs, ns = _tensor_table(tensors)
    _check("det_grad_norm", load().det_grad_norm(ptrs, ns, len(tensors), max_norm, _ptr(norm_out),
                                                 _ptr(coef_out), *_ws(ws), _stream(), _ptr(status_dev)))


def det_scale_inplace(g, n, coef_dev):
    _c.det_scale_inplace(g, n, coef_dev)


# ---- LSQ int8 linear -------------------------------------------------------------------------------------
def det_lsq_weight_scale_ws_bytes(N, K):
    return load().det_lsq_weight_scale_ws_bytes(N, K)


def det_lsq_weight_scale(W, N, K, per_tensor, s_w, ws):
    _c.det_lsq_weight_scale(W, N, K, per_tensor, s_w, ws)


def det_lsq_act_scale_init_ws_bytes(n):
    return load().det_lsq_act_scale_init_ws_bytes(n)


def det_lsq_act_scale_init(X, n, s_x, ws):
    _c.det_lsq_act_scale_init(X, n, s_x, ws)


def det_lsq_quantize_weight_ws_bytes(N, K):
    return load().det_lsq_quantize_weight_ws_bytes(N, K)


def det_lsq_quantize_weight(W, s_w, N, K, hadamard_block, qW, qWt_bwd, s_u, ws):
    _c.det_lsq_quantize_weight(W, s_w, N, K, hadamard_block, qW, qWt_bwd, s_u, ws)


def det_linear_fwd(X, qW, s_x, s_w, M, N, K, Y, qX_save, status_dev=None):
    _c.det_linear_fwd(X, qW, s_x, s_w, M, N, K, Y, qX_save, status_dev)


def det_linear_fwd_q(qX, qW, s_x, s_w, M, N, K, Y, status_dev=None):
    _c.det_linear_fwd_q(qX, qW, s_x, s_w, M, N, K, Y, status_dev)


def det_linear_bwd_ws_bytes(M, N, K):
    return load().det_linear_bwd_ws_bytes(M, N, K)


def det_linear_bwd(dY, X, qX, W, qWt_bwd, s_x, s_w, s_u, M, N, K, hadamard_block, dX, dW, ds_x, ws, status_dev=None):
    _c.det_linear_bwd(dY, X, qX, W, qWt_bwd, s_x, s_w, s_u, M, N, K, hadamard_block, dX, dW, ds_x, ws, status_dev)


def det_test_wait_timeout(status_dev, limit_cycles):
    _check("det_test_wait_timeout", load().det_test_wait_timeout(_ptr(status_dev), limit_cycles, _stream()))


def det_test_wait_warp(gone_on, limit_cycles):
    _check("det_test_wait_warp", load().det_test_wait_warp(_ptr(gone_on), limit_cycles, _stream()))


def det_test_igemm_tn(A, B, I, J, K, Cout, force_one_cta=0, status_dev=None):
    _check("det_test_igemm_tn", load().det_test_igemm_tn(_ptr(A), _ptr(B), I, J, K, _ptr(Cout),
                                                         force_one_cta, _stream(), _ptr(status_dev)))


# ---- RMSNorm, cross-entropy ---------------------------------------------------------------------------------
def det_rmsnorm_fwd(io, x, gamma, rows, D, eps, y, rstd):
    _c.det_rmsnorm_fwd(io, x, gamma, rows, D, eps, y, rstd)


def det_rmsnorm_fwd_q(x, gamma, rows, D, eps, y, rstd, s_q, qy):
    _c.det_rmsnorm_fwd_q(x, gamma, rows, D, eps, y, rstd, s_q, qy)


def det_residual_rmsnorm_fwd(a, b, gamma, rows, D, eps, sum_out, y, rstd, s_q=None, qy=None):
    _c.det_residual_rmsnorm_fwd(a, b, gamma, rows, D, eps, sum_out, y, rstd, s_q, qy)


def det_headnorm_fwd(x, ld, T, nh, eps, y, ld_y, rstd):
    _c.det_headnorm_fwd(x, ld, T, nh, eps, y, ld_y, rstd)


def det_headnorm_bwd(dy, ld_dy, x, ld, rstd, T, nh, dx, ld_dx):
    _c.det_headnorm_bwd(dy, ld_dy, x, ld, rstd, T, nh, dx, ld_dx)


def det_rope(x, ld, T, nh, S, cos_tab, sin_tab, inverse, y, ld_y):
    _c.det_rope(x, ld, T, nh, S, cos_tab, sin_tab, int(inverse), y, ld_y)


def det_rmsnorm_bwd_ws_bytes(rows, D):
    return load().det_rmsnorm_bwd_ws_bytes(rows, D)


def det_rmsnorm_bwd(io, dy, x, gamma, rstd, rows, D, dx, dgamma, ws):
    _c.det_rmsnorm_bwd(io, dy, x, gamma, rstd, rows, D, dx, dgamma, ws)


def det_rmsnorm_bwd_residual(dy, x, gamma, rstd, rows, D, res, dx, dgamma, ws):
    _c.det_rmsnorm_bwd_residual(dy, x, gamma, rstd, rows, D, res, dx, dgamma, ws)


def det_xent_ws_bytes(rows, V):
    return load().det_xent_ws_bytes(rows, V)


def det_xent_fwd(logits, target, rows, V, z_weight, loss_row, lse, loss_mean, z_mean, ws, status_dev=None):
    _c.det_xent_fwd(logits, target, rows, V, z_weight, loss_row, lse, loss_mean, z_mean, ws, status_dev)


def det_xent_bwd(logits_inout, target, lse, rows, V, z_weight, scale):
    _c.det_xent_bwd(logits_inout, target, lse, rows, V, z_weight, scale)


# ---- attention ------------------------------------------------------------------------------------------------
def det_attn_fwd(q, k, v, ld, B, H, S, out, ld_out, lse, Hkv=None, window=0):
    _c.det_attn_fwd(q, k, v, ld, B, H, H if Hkv is None else Hkv, S, window, out, ld_out, lse)


def det_attn_fwd_q(q, k, v, ld, B, H, S, out, ld_out, lse, s_q, qout, Hkv=None, window=0):
    _c.det_attn_fwd_q(q, k, v, ld, B, H, H if Hkv is None else Hkv, S, window, out, ld_out, lse, s_q, qout)


def det_attn_fwd_int8pv(q, k, v, ld, B, H, S, out, ld_out, lse, status_dev=None, Hkv=None, window=0):
    _c.det_attn_fwd_int8pv(q, k, v, ld, B, H, H if Hkv is None else Hkv, S, window, out, ld_out, lse, status_dev)


def det_attn_bwd_ws_bytes(B, H, S, Hkv=None):
    return load().det_attn_bwd_ws_bytes(B, H, H if Hkv is None else Hkv, S)


def det_attn_bwd(dout, q, k, v, out, lse, ld, ld_out, B, H, S, dq, dk, dv, ld_d, ws, Hkv=None, window=0):
    _c.det_attn_bwd(dout, q, k, v, out, lse, ld, ld_out, B, H, H if Hkv is None else Hkv, S, window, dq, dk, dv, ld_d, ws)


def det_attn_bwd_fixq_ws_bytes(B, H, S, Hkv=None):
    return load().det_attn_bwd_fixq_ws_bytes(B, H, H if Hkv is None else Hkv, S)


def det_attn_bwd_fixq(dout, q, k, v, out, lse, ld, ld_out, B, H, S, dq, dk, dv, ld_d, ws, Hkv=None, window=0):
    _c.det_attn_bwd_fixq(dout, q, k, v, out, lse, ld, ld_out, B, H, H if Hkv is None else Hkv, S, window, dq, dk, dv, ld_d, ws)


# ---- glue --------------------------------------------------------------------------------------------------------
def det_swiglu_fwd(gu, rows, F, h):
    _c.det_swiglu_fwd(gu, rows, F, h)


def det_swiglu_fwd_q(gu, rows, F, h, s_q, qh):
    _c.det_swiglu_fwd_q(gu, rows, F, h, s_q, qh)


def det_swiglu_bwd(dh, gu, rows, F, dgu):
    _c.det_swiglu_bwd(dh, gu, rows, F, dgu)


def det_residual_add(a, b, n, y):
    _c.det_residual_add(a, b, n, y)


def det_embed_fwd(tok, T, E, V, D, y):
    _c.det_embed_fwd(tok, T, E, V, D, y)


def det_embed_bwd(tok, T, dy, V, D, dE):
    _c.det_embed_bwd(tok, T, dy, V, D, dE)


def det_lmhead_fwd(H, W, M, V, K, logits):
    _c.det_lmhead_fwd(H, W, M, V, K, logits)


def det_lmhead_fwd_v2_ws_bytes(M, V, K):
    return load().det_lmhead_fwd_v2_ws_bytes(M, V, K)


def det_lmhead_fwd_v2(H, W, M, V, K, logits, ws, status_dev=None):
    _c.det_lmhead_fwd_v2(H, W, M, V, K, logits, ws, status_dev)


def det_lmhead_bwd_v2_ws_bytes(M, V, K):
    return load().det_lmhead_bwd_v2_ws_bytes(M, V, K)


def det_lmhead_bwd_v2(dlogits, H, W, M, V, K, dH, dW, ws, status_dev=None):
    _c.det_lmhead_bwd_v2(dlogits, H, W, M, V, K, dH, dW, ws, status_dev)


def det_attn_fwd_v2_ws_bytes(B, H, S):
    return load().det_attn_fwd_v2_ws_bytes(B, H, S)


def det_attn_fwd_v2(q, k, v, ld, B, H, S, out, ld_out, lse, ws, status_dev=None):
    _c.det_attn_fwd_v2(q, k, v, ld, B, H, S, out, ld_out, lse, ws, status_dev)


def det_lmhead_bwd(dlogits, H, W, M, V, K, dH, dW, first_chunk):
    _c.det_lmhead_bwd(dlogits, H, W, M, V, K, dH, dW, first_chunk)


def det_test_lmhead_tile(which, tile, A, B, M, V, K, out, first_chunk=1):
    _check("det_test_lmhead_tile", load().det_test_lmhead_tile(which, tile, _ptr(A), _ptr(B), M, V, K, _ptr(out), first_chunk, _stream()))


def det_test_attn_fwd(rows, q, k, v, ld, B, H, S, out, ld_out, lse, s_q, qout, Hkv=None, window=0):
    _check("det_test_attn_fwd", load().det_test_attn_fwd(rows, _ptr(q), _ptr(k), _ptr(v), ld, B, H, H if Hkv is None else Hkv, S, window,
                                                         _ptr(out), ld_out, _ptr(lse), _ptr(s_q), _ptr(qout), _stream()))


def det_test_attn_rows(heads, S, window=0):
    return load().det_test_attn_rows(heads, S, window)


def det_test_lmhead_pick(M, V, K):
    return load().det_test_lmhead_pick(M, V, K)


# ---- gradient accumulation, AdamW, hash ---------------------------------------------------------------------------
def det_grad_accum_nbufs(dp_replicate):
    return load().det_grad_accum_nbufs(dp_replicate)


def det_grad_accum_init(st, accum, dp_shard, dp_replicate, n, bufs):
    _check("det_grad_accum_init", load().det_grad_accum_init(C.byref(st), accum, dp_shard,
                                                             dp_replicate, n, _ptr(bufs)))


def det_grad_accum_push(st, g_microbatch):
    _check("det_grad_accum_push", load().det_grad_accum_push(C.byref(st), _ptr(g_microbatch), _stream()))


def det_grad_accum_result(st, g_out):
    _check("det_grad_accum_result", load().det_grad_accum_result(C.byref(st), _ptr(g_out), _stream()))


def det_adamw_step(desc, pdtype, p, g, m, v, n):
    _check("det_adamw_step", load().det_adamw_step(C.byref(desc), pdtype, _ptr(p), _ptr(g), _ptr(m), _ptr(v),
                                                   n, _stream()))


def det_adamw_batch(descs, pdtypes, ps, gs, ms, vs, coef_dev=None):
    """One launch for many tensors; coef_dev: device scalar every gradient is multiplied with first (in place)."""
    k, numel = len(ps), torch.Tensor.numel
    table = lambda ts: (C.c_void_p * k)(*map(_ptr, ts))
    counts = list(map(numel, ps))
    assert k == len(descs) == len(pdtypes) and all(list(map(numel, ts)) == counts for ts in (gs, ms, vs)) and \
        [2 if kind == DET_BF16 else 4 for kind in pdtypes] == list(map(torch.Tensor.element_size, ps)), \
        "one entry per tensor in every list; parameter, gradient and moments of a tensor have the same number of elements"
    _check("det_adamw_batch", load().det_adamw_batch((det_adamw_desc * k)(*descs), (C.c_int * k)(*pdtypes), table(ps), table(gs),
                                                     table(ms), table(vs), (C.c_size_t * k)(*counts), k, _ptr(coef_dev), _stream()))


def det_tensor_hash_ws_bytes(nbytes):
    return load().det_tensor_hash_ws_bytes(nbytes)


def det_tensor_hash_async(p, nbytes, out32_dev, ws):
    """Queues the hash; the 32-byte root lands in out32_dev (device) in stream order, nothing synchronises."""
    _c.det_tensor_hash_async(p, nbytes, out32_dev, ws)


def det_tensor_hash(p, nbytes, ws):
    """Returns the 32-byte root as a hex string (synchronises the current stream)."""
    out = (C.c_uint8 * 32)()
    _check("det_tensor_hash", load().det_tensor_hash(_ptr(p), nbytes, out, *_ws(ws), _stream()))
    return bytes(out).hex()


def det_tensor_hash_batch_ws_bytes(nbytes):
    """nbytes: byte counts of the tensors, or the tensors themselves."""
    counts = [n if isinstance(n, int) else n.numel() * n.element_size() for n in nbytes]
    return load().det_tensor_hash_batch_ws_bytes((C.c_size_t * len(counts))(*counts), len(counts))


def det_tensor_hash_batch(tensors, roots_dev, ws):
    """Queues the hashes of all tensors together; root t lands at roots_dev[32 t : 32 t + 32] in stream order."""
    k = len(tensors)
    ptrs = (C.c_void_p * k)(*map(_ptr, tensors))
    counts = (C.c_size_t * k)(*[t.numel() * t.element_size() for t in tensors])
    _check("det_tensor_hash_batch", load().det_tensor_hash_batch(ptrs, counts, k, _ptr(roots_dev), *_ws(ws), _stream()))
