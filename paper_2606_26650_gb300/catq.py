"""Python binding of libcatq (include/catq.h): argument marshalling only.

Every function here has the C name of the call it wraps, takes torch tensors that live on
the current CUDA device, passes their data pointers and the current torch stream to the
library, and raises CatqError on a non-zero status.  All arithmetic runs in the library's
CUDA kernels; there is no fallback.  PyTorch provides device memory and streams.
"""
from __future__ import annotations

import ctypes
import dataclasses
import os
import re
import struct

PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(PKG, "libcatq.so")
HEADER = os.path.join(os.path.dirname(PKG), "include", "catq.h")

F32, BF16 = 0, 1
PHASE_TEACHER, PHASE_SOFT, PHASE_HARD = 0, 1, 2
THR_HALF, THR_TWN07, THR_ABSMEAN, THR_TWN_STATIC = 0, 1, 2, 3
REDUCE_MEAN, REDUCE_SUM = 0, 1
RECON_ALPHA_T, RECON_ALPHA_T_MU = 0, 1

STATUS = {
    0: "CATQ_OK", 1: "CATQ_ERR_INVALID_ARG", 2: "CATQ_ERR_SHAPE", 3: "CATQ_ERR_DTYPE",
    4: "CATQ_ERR_ALIGN", 5: "CATQ_ERR_CUDA", 6: "CATQ_ERR_TIMEOUT", 7: "CATQ_ERR_NONFINITE",
    8: "CATQ_ERR_UNSUPPORTED", 9: "CATQ_ERR_WORKSPACE",
}


class CatqError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {STATUS.get(status, status)}")


class catq_layer(ctypes.Structure):
    _fields_ = [
        ("N", ctypes.c_int64), ("K", ctypes.c_int64), ("g", ctypes.c_int32), ("w_dtype", ctypes.c_int32),
        ("W", ctypes.c_void_p),
        ("mu0", ctypes.c_void_p), ("alpha0", ctypes.c_void_p), ("delta0", ctypes.c_void_p),
        ("d_mu", ctypes.c_void_p), ("d_alpha", ctypes.c_void_p), ("d_delta", ctypes.c_void_p),
        ("op_const", ctypes.c_void_p), ("recon", ctypes.c_int32), ("reserved", ctypes.c_int32),
    ]


class catq_grouped_layer(ctypes.Structure):
    _fields_ = [
        ("E", ctypes.c_int32), ("g", ctypes.c_int32), ("N", ctypes.c_int64), ("K", ctypes.c_int64),
        ("w_dtype", ctypes.c_int32), ("recon", ctypes.c_int32), ("W", ctypes.c_void_p),
        ("mu0", ctypes.c_void_p), ("alpha0", ctypes.c_void_p), ("delta0", ctypes.c_void_p),
        ("d_mu", ctypes.c_void_p), ("d_alpha", ctypes.c_void_p), ("d_delta", ctypes.c_void_p),
        ("op_const", ctypes.c_void_p),
    ]


class catq_schedule(ctypes.Structure):
    _fields_ = [("phase", ctypes.c_int32), ("s", ctypes.c_float)]


class catq_infer_layer(ctypes.Structure):
    _fields_ = [("codes", ctypes.c_void_p), ("alpha", ctypes.c_void_p), ("mu", ctypes.c_void_p),
                ("N", ctypes.c_int64), ("K", ctypes.c_int64), ("X", ctypes.c_void_p), ("Y", ctypes.c_void_p)]


class catq_adamw(ctypes.Structure):
    _fields_ = [("beta1", ctypes.c_float), ("beta2", ctypes.c_float), ("eps", ctypes.c_float),
                ("weight_decay", ctypes.c_float), ("margin", ctypes.c_float)]


_lib = None


def lib() -> ctypes.CDLL:
    """The loaded library; raises if it has not been built (there is no fallback)."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise RuntimeError(f"{LIB_PATH} is missing: build it with __graft_entry__.build()")
    L = ctypes.CDLL(LIB_PATH)
    P, I64, I32, F, S = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int32, ctypes.c_float, ctypes.c_size_t
    LP, GP, IP = (ctypes.POINTER(t) for t in (catq_layer, catq_grouped_layer, catq_infer_layer))
    sig = {
        "catq_abi_version": (I32, []),
        "catq_status_string": (ctypes.c_char_p, [I32]),
        "catq_group_stats": (I32, [LP, I32, P]),
        "catq_modulate_ternarize": (I32, [LP, catq_schedule, P, P, P, P]),
        "catq_soft_ternary_linear_fwd": (I32, [LP, catq_schedule, P, I64, I32, P, P]),
        "catq_bwd_workspace_bytes": (S, [LP, I64]),
        "catq_soft_ternary_linear_bwd": (I32, [LP, catq_schedule, P, P, I64, I32, P, P, P, P, P, S, P]),
        "catq_recon_loss_workspace_bytes": (S, [I64]),
        "catq_recon_loss": (I32, [P, P, I64, I32, I32, P, P, P, S, P]),
        "catq_hard_ternarize_pack": (I32, [LP, P, P, P, P]),
        "catq_device_status": (I32, [P, ctypes.POINTER(I32)]),
        "catq_selftest_wait_timeout": (I32, [ctypes.c_uint64, P]),
        "catq_ternary_infer": (I32, [P, P, P, I64, I64, I32, P, I64, I32, P, P]),
        "catq_soft_ternary_linear_bwd_noalloc": (I32, [LP, catq_schedule, P, P, I64, I32, P, P, P, P, P]),
        "catq_bwd_noalloc_max_scratch_bytes": (S, []),
        "catq_grouped_soft_ternary_linear_fwd": (I32, [GP, catq_schedule, P, P, I32, P, P]),
        "catq_grouped_bwd_workspace_bytes": (S, [GP, P]),
        "catq_schedule_at_epoch": (I32, [I32, I32, ctypes.c_double, ctypes.c_double, ctypes.POINTER(catq_schedule)]),
        "catq_linear_decay_lr": (I32, [ctypes.c_double, I64, I64, ctypes.POINTER(F)]),
        "catq_factor_adamw_step": (I32, [I64, P, P, P, P, P, P, P, ctypes.POINTER(catq_adamw), I64, F, P]),
        "catq_grouped_soft_ternary_linear_bwd": (I32, [GP, catq_schedule, P, P, P, I32, P, P, P, P, P, S, P]),
        "catq_soft_ternary_linear_fwd_ex": (I32, [LP, catq_schedule, P, I64, I32, P, P, I32, P]),
        "catq_fwd_loss_workspace_bytes": (S, [LP, I64]),
        "catq_soft_ternary_linear_fwd_loss": (I32, [LP, catq_schedule, P, I64, I32, P, P, I32, I32, P, P, P, P, S, P]),
        "catq_act_quant_a8": (I32, [P, I64, I64, I32, P, P, P, P]),
        "catq_direct_adamw_step": (I32, [I64, P, P, P, P, P, ctypes.POINTER(catq_adamw), I64, F, P]),
        "catq_ternary_infer_max_layers": (I32, []),
        "catq_ternary_infer_batched": (I32, [IP, I32, I32, I64, I32, P]),
        "catq_ternary_infer_max_stages": (I32, []),
        "catq_ternary_infer_sync_bytes": (S, []),
        "catq_ternary_infer_staged": (I32, [IP, I32, ctypes.POINTER(I32), I32, I64, I32, P, P]),
        "catq_group_recon_error": (I32, [LP, P, P]),
        "catq_linear_form": (I32, [I64, I64, I32, I32, catq_schedule, I64, I32, P, I32, I32, I32,
                                   ctypes.POINTER(I32)]),
        "catq_grouped_fwd_loss_workspace_bytes": (S, [GP, P]),
        "catq_rmsnorm_fwd": (I32, [P, I32, P, P, I64, I64, F, P, P, P, P]),
        "catq_rmsnorm_bwd": (I32, [P, I32, P, P, P, P, P, I64, I64, P, P]),
        "catq_rope": (I32, [P, I64, I64, I32, I32, F, I32, P]),
        "catq_swiglu_fwd": (I32, [P, P, I64, P, P]),
        "catq_swiglu_bwd": (I32, [P, P, P, I64, P, P, P]),
        "catq_block_output_loss": (I32, [P, P, I64, P, I32, P, P, P, P, S, P]),
        "catq_attention_fwd": (I32, [P, P, P, I32, I32, I32, I32, I32, P, P, P]),
        "catq_attention_bwd": (I32, [P, P, P, P, P, P, I32, I32, I32, I32, I32, P, P, P, P, P]),
        "catq_grouped_soft_ternary_linear_fwd_loss": (I32, [GP, catq_schedule, P, P, I32, P, I32, P, P, P, P, S, P]),
    }
    for name, (res, args) in sig.items():
        fn = getattr(L, name)
        fn.restype = res
        fn.argtypes = args
    _lib = L
    return L


def header_functions(path: str = HEADER):
    """Names of the functions include/catq.h declares."""
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(catq_[a-z0-9_]+)\s*\(", text)))


# ------------------------------------------------------------------ marshalling helpers
# A small call (a norm of a few rows, a decode step's layers) costs a few microseconds on the GPU,
# so these run on every argument of every call and keep to a handful of attribute reads each:
# addresses as ints, structs filled in one call, the stream without a Stream object.  Nothing is
# remembered from one call to the next.  On a Grace host, Python and launch together: forward of a
# layer 18.0 -> 9.6 us, its backward 27.3 -> 17.2, a row norm 9.7 -> 5.4, three decode layers
# 17.9 -> 10.7.

def _ptr(t):
    return None if t is None else t.data_ptr()


def _stream(stream=None):
    if stream is not None:
        return stream.cuda_stream
    import torch
    try:  # (not public: a PyTorch without them takes the public way, 1 us longer)
        return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())
    except AttributeError:
        return torch.cuda.current_stream().cuda_stream


_DTYPES: dict = {}


def _known_dtype(t):
    """The code of a tensor's dtype, None for one the library does not take."""
    if not _DTYPES:
        import torch
        _DTYPES.update({torch.bfloat16: BF16, torch.float32: F32})
    return _DTYPES.get(t.dtype)


def _dtype_code(t) -> int:
    code = _known_dtype(t)
    if code is None:
        raise TypeError(f"unsupported dtype {t.dtype}")
    return code


def _check(status: int, where: str):
    if status != 0:
        raise CatqError(status, where)


def _buf(t, name: str, nbytes: int, where: str):
    """The library reads and writes `nbytes` bytes at a tensor's address without seeing its
    size or device: refuse a host tensor or one too small before the call, so that a
    caller's mistake raises here instead of touching memory the tensor does not own.
    None passes (the call decides whether the argument is optional).  Returns the address."""
    if t is None:
        return None
    if t.is_cuda and t.is_contiguous() and t.numel() * t.element_size() >= nbytes:
        return t.data_ptr()
    if not t.is_cuda:
        raise ValueError(f"{where}: {name} must be a CUDA tensor")
    if not t.is_contiguous():
        raise ValueError(f"{where}: {name} must be contiguous")
    have = t.numel() * t.element_size()
    raise ValueError(f"{where}: {name} holds {have} bytes, the call needs {nbytes}")


def _ws(workspace, where: str):
    """(address, bytes) of a workspace; the call decides whether it is large enough."""
    if workspace is None:
        return None, 0
    return _buf(workspace, "workspace", 0, where), workspace.numel() * workspace.element_size()


# catq_layer, catq_grouped_layer and catq_infer_layer, to be filled in one call (native sizes and
# alignment): a ctypes structure sets its fields one by one.
_LAYER = struct.Struct("qqii8Qii")
_GROUPED = struct.Struct("iiqqii8Q")
_INFER = struct.Struct("QQQqqQQ")


@dataclasses.dataclass
class Layer:
    """One linear layer's device state: W [N, K], the per-group arrays ([G] fp32) and the
    operand-constant array the fused GEMMs read ([4 G] fp32, [5 G] with mu in the
    reconstruction).  `recon`: RECON_ALPHA_T (W ~ alpha T) or RECON_ALPHA_T_MU."""
    W: object
    g: int
    mu0: object
    alpha0: object
    delta0: object
    d_mu: object
    d_alpha: object
    d_delta: object
    op_const: object = None
    recon: int = RECON_ALPHA_T

    @classmethod
    def create(cls, W, g, d_mu=None, d_alpha=None, d_delta=None, recon=RECON_ALPHA_T):
        """Allocates the statistics, operand-constant and (identity, unless given) factor
        tensors."""
        import torch
        N, K = W.shape
        G = N * K // g
        kw = dict(device=W.device, dtype=torch.float32)
        return cls(W, g, torch.empty(G, **kw), torch.empty(G, **kw), torch.empty(G, **kw),
                   d_mu if d_mu is not None else torch.zeros(G, **kw),
                   d_alpha if d_alpha is not None else torch.ones(G, **kw),
                   d_delta if d_delta is not None else torch.ones(G, **kw),
                   torch.empty((5 if recon else 4) * G, **kw), int(recon))

    @property
    def N(self):
        return self.W.shape[0]

    @property
    def K(self):
        return self.W.shape[1]

    @property
    def G(self):
        return self.N * self.K // self.g

    def _addresses(self, N: int, K: int):
        """The checked addresses of W, the six per-group arrays and op_const (0: none)."""
        W, where, need = self.W, "Layer", 4 * (N * K // self.g)
        return (_buf(W, "W", N * K * W.element_size(), where), _buf(self.mu0, "mu0", need, where),
                _buf(self.alpha0, "alpha0", need, where), _buf(self.delta0, "delta0", need, where),
                _buf(self.d_mu, "d_mu", need, where), _buf(self.d_alpha, "d_alpha", need, where),
                _buf(self.d_delta, "d_delta", need, where),
                _buf(self.op_const, "op_const", (5 if self.recon else 4) * need, where) or 0)

    def struct(self) -> catq_layer:
        N, K = self.W.shape
        st = catq_layer()
        _LAYER.pack_into(st, 0, N, K, self.g, _dtype_code(self.W), *self._addresses(N, K), self.recon, 0)
        return st


def schedule(phase: int, s: float = 0.0) -> catq_schedule:
    return catq_schedule(int(phase), float(s))


# ------------------------------------------------------------------ the C calls

def catq_group_stats(layer: Layer, thr_init: int = THR_HALF, stream=None):
    _check(lib().catq_group_stats(layer.struct(), int(thr_init), _stream(stream)), "catq_group_stats")


def catq_modulate_ternarize(layer: Layer, sched: catq_schedule, Wq_out=None, T_out=None, alpha_out=None,
                            stream=None):
    st = layer.struct()
    w = "catq_modulate_ternarize"
    wq = _buf(Wq_out, "Wq_out", layer.N * layer.K * layer.W.element_size(), w)
    t = _buf(T_out, "T_out", layer.N * layer.K, w)
    al = _buf(alpha_out, "alpha_out", 4 * layer.G, w)
    _check(lib().catq_modulate_ternarize(st, sched, wq, t, al, _stream(stream)), w)


def catq_soft_ternary_linear_fwd(layer: Layer, sched: catq_schedule, X, Y, stream=None):
    w = "catq_soft_ternary_linear_fwd"
    st = layer.struct()
    N, K = layer.W.shape
    M, e = X.shape[0], X.element_size()
    _check(lib().catq_soft_ternary_linear_fwd(st, sched, _buf(X, "X", M * K * e, w), M, _dtype_code(X),
                                              _buf(Y, "Y", M * N * e, w), _stream(stream)), w)


def catq_soft_ternary_linear_fwd_ex(layer: Layer, sched: catq_schedule, X, Y, x_row_scale=None, stream=None):
    """Y = diag(x_row_scale) X Wq^T; Y may be fp32 for a bf16 layer."""
    w = "catq_soft_ternary_linear_fwd_ex"
    st = layer.struct()
    N, K = layer.W.shape
    M = X.shape[0]
    x = _buf(X, "X", M * K * X.element_size(), w)
    y = _buf(Y, "Y", M * N * (Y.element_size() if Y is not None else 0), w)
    rs = _buf(x_row_scale, "x_row_scale", 4 * M, w)
    _check(lib().catq_soft_ternary_linear_fwd_ex(st, sched, x, M, _dtype_code(X), rs, y, _dtype_code(Y),
                                                 _stream(stream)), w)


def catq_fwd_loss_workspace_bytes(layer: Layer, M: int) -> int:
    return int(lib().catq_fwd_loss_workspace_bytes(layer.struct(), int(M)))


def catq_soft_ternary_linear_fwd_loss(layer: Layer, sched: catq_schedule, X, Y_ref, loss_out, dY, Y=None,
                                      x_row_scale=None, workspace=None, reduction: int = REDUCE_MEAN, stream=None):
    """Forward, Eq. 7 loss and dY in one pass; Y_ref may be fp32 for a bf16 layer."""
    w = "catq_soft_ternary_linear_fwd_loss"
    st = layer.struct()
    N, K = layer.W.shape
    M, e = X.shape[0], X.element_size()
    x = _buf(X, "X", M * K * e, w)
    ref = _buf(Y_ref, "Y_ref", M * N * Y_ref.element_size(), w)
    dy = _buf(dY, "dY", M * N * e, w)
    y = _buf(Y, "Y", M * N * e, w)
    lo = _buf(loss_out, "loss_out", 4, w)
    rs = _buf(x_row_scale, "x_row_scale", 4 * M, w)
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_soft_ternary_linear_fwd_loss(st, sched, x, M, _dtype_code(X), rs, ref, _dtype_code(Y_ref),
                                                   int(reduction), lo, dy, y, ws, ws_bytes, _stream(stream)), w)


def catq_linear_form(N: int, K: int, g: int, sched: catq_schedule, M: int = 0, row_offsets=None, dx: bool = False,
                     fused_loss: bool = False, recon: int = RECON_ALPHA_T, sm_count: int = 152) -> tuple:
    """How a bf16 layer's forward or dX is cut: (CTA pairs per cluster, -1 for tiles of one CTA or 0 for the
    narrow kernel, and the narrow kernel's columns, accumulators, shares, A and W ring slots, table entries).
    Host only."""
    form = (ctypes.c_int32 * 7)()
    off = None if row_offsets is None else _offsets(row_offsets)
    E = 0 if row_offsets is None else len(row_offsets) - 1
    _check(lib().catq_linear_form(int(N), int(K), int(g), int(recon), sched, int(M), E, off, int(dx), int(fused_loss),
                                  int(sm_count), form), "catq_linear_form")
    return tuple(form)


def catq_act_quant_a8(X, codes, scale, X_deq=None, stream=None):
    """Per-token 8-bit codes (as exact values of X's dtype), scales [M] and (optionally) the
    dequantized activations."""
    M, K = X.shape
    n, w = M * K * X.element_size(), "catq_act_quant_a8"
    x, c, d = _buf(X, "X", n, w), _buf(codes, "codes", n, w), _buf(X_deq, "X_deq", n, w)
    sc = _buf(scale, "scale", 4 * M, w)
    _check(lib().catq_act_quant_a8(x, M, K, _dtype_code(X), c, sc, d, _stream(stream)), w)


def catq_bwd_workspace_bytes(layer: Layer, M: int) -> int:
    return int(lib().catq_bwd_workspace_bytes(layer.struct(), int(M)))


def catq_soft_ternary_linear_bwd(layer: Layer, sched: catq_schedule, X, dY, dX=None, g_dmu=None, g_dalpha=None,
                                 g_ddelta=None, workspace=None, stream=None):
    w = "catq_soft_ternary_linear_bwd"
    st = layer.struct()
    x, dy, dx, g0, g1, g2 = _bwd_bufs(layer, X, dY, dX, (g_dmu, g_dalpha, g_ddelta), w)
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_soft_ternary_linear_bwd(st, sched, x, dy, X.shape[0], _dtype_code(X), dx, g0, g1, g2, ws,
                                              ws_bytes, _stream(stream)), w)


def catq_soft_ternary_linear_bwd_noalloc(layer: Layer, sched: catq_schedule, X, dY, dX=None, g_dmu=None,
                                         g_dalpha=None, g_ddelta=None, stream=None):
    w = "catq_soft_ternary_linear_bwd_noalloc"
    st = layer.struct()
    x, dy, dx, g0, g1, g2 = _bwd_bufs(layer, X, dY, dX, (g_dmu, g_dalpha, g_ddelta), w)
    _check(lib().catq_soft_ternary_linear_bwd_noalloc(st, sched, x, dy, X.shape[0], _dtype_code(X), dx, g0, g1, g2,
                                                      _stream(stream)), w)


def _bwd_bufs(layer, X, dY, dX, grads, where):
    """The checked addresses of a backward's arrays."""
    N, K = layer.W.shape
    M, e, need = X.shape[0], X.element_size(), 4 * (N * K // layer.g)
    return (_buf(X, "X", M * K * e, where), _buf(dY, "dY", M * N * e, where), _buf(dX, "dX", M * K * e, where),
            _buf(grads[0], "g_dmu", need, where), _buf(grads[1], "g_dalpha", need, where),
            _buf(grads[2], "g_ddelta", need, where))


def catq_bwd_noalloc_max_scratch_bytes() -> int:
    return int(lib().catq_bwd_noalloc_max_scratch_bytes())


def catq_recon_loss_workspace_bytes(count: int) -> int:
    return int(lib().catq_recon_loss_workspace_bytes(int(count)))


def catq_recon_loss(Y, Y_ref, loss_out, dY=None, workspace=None, reduction: int = REDUCE_MEAN, stream=None):
    w, count = "catq_recon_loss", Y.numel()
    n = count * Y.element_size()
    y, ref, dy = _buf(Y, "Y", n, w), _buf(Y_ref, "Y_ref", n, w), _buf(dY, "dY", n, w)
    lo = _buf(loss_out, "loss_out", 4, w)
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_recon_loss(y, ref, count, _dtype_code(Y), int(reduction), lo, dy, ws, ws_bytes,
                                 _stream(stream)), w)


def catq_hard_ternarize_pack(layer: Layer, codes, alpha=None, mu=None, stream=None):
    st = layer.struct()
    w, G = "catq_hard_ternarize_pack", layer.G
    c = _buf(codes, "codes", layer.N * layer.K // 4, w)
    al, m = _buf(alpha, "alpha", 4 * G, w), _buf(mu, "mu", 4 * G, w)
    _check(lib().catq_hard_ternarize_pack(st, c, al, m, _stream(stream)), w)


def catq_device_status(stream=None) -> int:
    out = ctypes.c_int32(0)
    _check(lib().catq_device_status(_stream(stream), ctypes.byref(out)), "catq_device_status")
    return int(out.value)


def catq_ternary_infer(codes, alpha, N: int, K: int, g: int, X, Y, mu=None, stream=None):
    """Y [B, N] = X [B, K] (alpha T + mu)^T from the 2-bit codes, group scales and (for the
    W ~ alpha T + mu form) group offsets of catq_hard_ternarize_pack."""
    w, B, N, K = "catq_ternary_infer", X.shape[0], int(N), int(K)
    G, e = N * K // max(int(g), 1), X.element_size()
    c = _buf(codes, "codes", N * K // 4, w)
    al, m = _buf(alpha, "alpha", 4 * G, w), _buf(mu, "mu", 4 * G, w)
    x, y = _buf(X, "X", B * K * e, w), _buf(Y, "Y", B * N * e, w)
    _check(lib().catq_ternary_infer(c, al, m, N, K, int(g), x, B, _dtype_code(X), y, _stream(stream)), w)


def catq_ternary_infer_max_layers() -> int:
    return int(lib().catq_ternary_infer_max_layers())


def _infer_layer_array(layers, g, w):
    """The layers as an array of catq_infer_layer, and their token rows."""
    B, g = layers[0][4].shape[0] if layers else 0, max(int(g), 1)
    arr, size = (catq_infer_layer * max(1, len(layers)))(), _INFER.size
    for i, (codes, alpha, N, K, X, Y, mu) in enumerate(layers):
        N, K = int(N), int(K)
        n = N * K
        if X.shape[0] != B:
            raise ValueError(f"{w}: every layer needs the same token rows ({B})")
        e, need = X.element_size(), 4 * (n // g)
        _INFER.pack_into(arr, i * size, _buf(codes, "codes", n // 4, w), _buf(alpha, "alpha", need, w),
                         _buf(mu, "mu", need, w) or 0, N, K, _buf(X, "X", B * K * e, w), _buf(Y, "Y", B * N * e, w))
    return arr, B


def catq_ternary_infer_batched(layers, g: int, stream=None):
    """Several independent layers in one launch: `layers` is a list of tuples
    (codes, alpha, N, K, X, Y, mu) (mu may be None), all with the same token rows X.shape[0]."""
    w = "catq_ternary_infer_batched"
    arr, B = _infer_layer_array(layers, g, w)
    dt = _dtype_code(layers[0][4]) if layers else BF16
    _check(lib().catq_ternary_infer_batched(arr, len(layers), int(g), int(B), dt, _stream(stream)), w)


def catq_ternary_infer_sync_bytes() -> int:
    return int(lib().catq_ternary_infer_sync_bytes())


def catq_ternary_infer_max_stages() -> int:
    return int(lib().catq_ternary_infer_max_stages())


def catq_ternary_infer_staged(layers, stages, g: int, sync, stream=None):
    """Layers in dependency order in one cooperative launch: `layers` as in
    catq_ternary_infer_batched, `stages` the stage of each layer (0, then non-decreasing in steps
    of 1); a layer may read the Y of a layer of an earlier stage.  `sync`: a zeroed device buffer
    of catq_ternary_infer_sync_bytes() bytes (left zeroed)."""
    w = "catq_ternary_infer_staged"
    arr, B = _infer_layer_array(layers, g, w)
    sy = _buf(sync, "sync", catq_ternary_infer_sync_bytes(), w)
    if len(stages) != len(layers):
        raise ValueError(f"{w}: one stage per layer")
    st = (ctypes.c_int32 * max(1, len(stages)))(*[int(v) for v in stages])
    dt = _dtype_code(layers[0][4]) if layers else BF16
    _check(lib().catq_ternary_infer_staged(arr, len(layers), st, int(g), int(B), dt, sy, _stream(stream)), w)


def catq_schedule_at_epoch(e: int, m: int = 60, gamma: float = 0.8, s0: float = 30.0) -> catq_schedule:
    """Eq. 6's (phase, s) of calibration epoch e of m (host only)."""
    out = catq_schedule()
    _check(lib().catq_schedule_at_epoch(int(e), int(m), float(gamma), float(s0), ctypes.byref(out)),
           "catq_schedule_at_epoch")
    return out


def catq_linear_decay_lr(lr0: float, k: int, total: int) -> float:
    """Learning rate of update k of `total` under a linear decay to zero (host only)."""
    out = ctypes.c_float()
    _check(lib().catq_linear_decay_lr(float(lr0), int(k), int(total), ctypes.byref(out)), "catq_linear_decay_lr")
    return float(out.value)


def adamw(beta1: float = 0.9, beta2: float = 0.999, eps: float = 1e-8, weight_decay: float = 0.0,
          margin: float = 1e-4) -> catq_adamw:
    return catq_adamw(beta1, beta2, eps, weight_decay, margin)


def catq_factor_adamw_step(d_mu, d_alpha, d_delta, g_dmu, g_dalpha, g_ddelta, moments, hp: catq_adamw, t: int,
                           lr: float, stream=None):
    """One AdamW update of the factors [G] in place from their gradients; moments [6 * G]
    (zero before the first update) is the optimizer state."""
    G, w = d_mu.numel(), "catq_factor_adamw_step"
    n = 4 * G
    _check(lib().catq_factor_adamw_step(
        G, _buf(d_mu, "d_mu", n, w), _buf(d_alpha, "d_alpha", n, w), _buf(d_delta, "d_delta", n, w),
        _buf(g_dmu, "g_dmu", n, w), _buf(g_dalpha, "g_dalpha", n, w), _buf(g_ddelta, "g_ddelta", n, w),
        _buf(moments, "moments", 6 * n, w), ctypes.byref(hp), int(t), float(lr), _stream(stream)), w)


def catq_direct_adamw_step(d_alpha, d_delta, g_dalpha, g_ddelta, moments, hp: catq_adamw, t: int, lr: float,
                           stream=None):
    """Direct learning's update of (d_alpha, d_delta) [G] in place; moments [4 * G]."""
    G, w = d_alpha.numel(), "catq_direct_adamw_step"
    for name, arr in zip(("d_alpha", "d_delta", "g_dalpha", "g_ddelta"), (d_alpha, d_delta, g_dalpha, g_ddelta)):
        _buf(arr, name, 4 * G, w)
    _buf(moments, "moments", 4 * 4 * G, w)
    _check(lib().catq_direct_adamw_step(G, _ptr(d_alpha), _ptr(d_delta), _ptr(g_dalpha), _ptr(g_ddelta),
                                        _ptr(moments), ctypes.byref(hp), int(t), float(lr), _stream(stream)), w)


def catq_group_recon_error(layer: Layer, err, stream=None):
    """err [G] = per-group mean of (W - Wq)^2 for the hard reconstruction."""
    w = "catq_group_recon_error"
    _check(lib().catq_group_recon_error(layer.struct(), _buf(err, "err", 4 * layer.G, w), _stream(stream)), w)


def catq_selftest_wait_timeout(timeout_ns: int, stream=None):
    _check(lib().catq_selftest_wait_timeout(int(timeout_ns), _stream(stream)), "catq_selftest_wait_timeout")


def workspace(nbytes: int, device):
    """A byte tensor of at least nbytes (256-byte aligned by the caching allocator)."""
    import torch
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device=device)


# ------------------------------------------------------------------ grouped (MoE) layers

@dataclasses.dataclass
class GroupedLayer:
    """E experts stacked: W [E, N, K], per-group arrays [E * G] (expert-major).  `dense`
    views the stack as one [E * N, K] layer for catq_group_stats / pack."""
    W: object
    g: int
    dense: Layer

    @classmethod
    def create(cls, W, g, d_mu=None, d_alpha=None, d_delta=None, recon=RECON_ALPHA_T):
        E, N, K = W.shape
        return cls(W, g, Layer.create(W.reshape(E * N, K), g, d_mu, d_alpha, d_delta, recon))

    @property
    def E(self):
        return self.W.shape[0]

    def _fields(self):
        E, N, K = self.W.shape
        d = self.dense
        # the stacked weights and the [E * G] per-group arrays, checked as one dense layer
        ptrs = d._addresses(*d.W.shape)
        return (E, self.g, N, K, _dtype_code(self.W), d.recon, self.W.data_ptr()) + ptrs[1:]

    def struct(self) -> catq_grouped_layer:
        st = catq_grouped_layer()
        _GROUPED.pack_into(st, 0, *self._fields())
        return st


def _offsets(row_offsets):
    return struct.pack(f"{len(row_offsets)}q", *[int(v) for v in row_offsets])


def _grouped_bufs(layer, row_offsets, where, X=None, Y=None, dY=None, dX=None, grads=()):
    """The library reads E + 1 row offsets and rows 0 .. R-1 of the row-indexed arrays: the checked
    addresses of X, Y, dY, dX and the gradients."""
    E, N, K = layer.W.shape
    if len(row_offsets) != E + 1:
        raise ValueError(f"{where}: row_offsets has {len(row_offsets)} entries, the layer's {E} experts need {E + 1}")
    R = int(row_offsets[-1])
    e = X.element_size() if X is not None else 2
    return (_buf(X, "X", R * K * e, where), _buf(Y, "Y", R * N * e, where), _buf(dY, "dY", R * N * e, where),
            _buf(dX, "dX", R * K * e, where)) + tuple(
                _buf(arr, name, 4 * E * (N * K // layer.g), where)
                for name, arr in zip(("g_dmu", "g_dalpha", "g_ddelta"), grads))


def catq_grouped_soft_ternary_linear_fwd(layer: GroupedLayer, sched: catq_schedule, X, row_offsets, Y, stream=None):
    w = "catq_grouped_soft_ternary_linear_fwd"
    st = layer.struct()
    x, y, _, _ = _grouped_bufs(layer, row_offsets, w, X=X, Y=Y)
    _check(lib().catq_grouped_soft_ternary_linear_fwd(st, sched, x, _offsets(row_offsets), _dtype_code(X), y,
                                                      _stream(stream)), w)


def catq_grouped_bwd_workspace_bytes(layer: GroupedLayer, row_offsets) -> int:
    st = layer.struct()
    _grouped_bufs(layer, row_offsets, "catq_grouped_bwd_workspace_bytes")
    return int(lib().catq_grouped_bwd_workspace_bytes(st, _offsets(row_offsets)))


def catq_grouped_soft_ternary_linear_bwd(layer: GroupedLayer, sched: catq_schedule, X, dY, row_offsets, dX=None,
                                         g_dmu=None, g_dalpha=None, g_ddelta=None, workspace=None, stream=None):
    w = "catq_grouped_soft_ternary_linear_bwd"
    st = layer.struct()
    x, _, dy, dx, g0, g1, g2 = _grouped_bufs(layer, row_offsets, w, X=X, dY=dY, dX=dX,
                                             grads=(g_dmu, g_dalpha, g_ddelta))
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_grouped_soft_ternary_linear_bwd(st, sched, x, dy, _offsets(row_offsets), _dtype_code(X), dx, g0,
                                                      g1, g2, ws, ws_bytes, _stream(stream)), w)


def catq_grouped_fwd_loss_workspace_bytes(layer: GroupedLayer, row_offsets) -> int:
    st = layer.struct()
    _grouped_bufs(layer, row_offsets, "catq_grouped_fwd_loss_workspace_bytes")
    return int(lib().catq_grouped_fwd_loss_workspace_bytes(st, _offsets(row_offsets)))


def catq_grouped_soft_ternary_linear_fwd_loss(layer: GroupedLayer, sched: catq_schedule, X, row_offsets, Y_ref,
                                              loss_out, dY, Y=None, workspace=None, reduction: int = REDUCE_MEAN,
                                              stream=None):
    w = "catq_grouped_soft_ternary_linear_fwd_loss"
    st = layer.struct()
    x, y, dy, _ = _grouped_bufs(layer, row_offsets, w, X=X, Y=Y, dY=dY)
    ref = _grouped_bufs(layer, row_offsets, w, Y=Y_ref)[1]
    lo = _buf(loss_out, "loss_out", 4, w)
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_grouped_soft_ternary_linear_fwd_loss(st, sched, x, _offsets(row_offsets), _dtype_code(X), ref,
                                                           int(reduction), lo, dy, y, ws, ws_bytes,
                                                           _stream(stream)), w)


# ------------------------------------------------------------------ decoder-block layers
# bf16 activations [T, *] (tokens t = b S + s); fp32 gamma, r, lse, delta.

def _bf16(t, name: str, nbytes: int, where: str):
    if t is not None and _known_dtype(t) != BF16:
        raise ValueError(f"{where}: {name} must be bfloat16")
    return _buf(t, name, nbytes, where)


def _f32(t, name: str, nbytes: int, where: str):
    if t is not None and _known_dtype(t) != F32:
        raise ValueError(f"{where}: {name} must be float32")
    return _buf(t, name, nbytes, where)


def catq_rmsnorm_fwd(X, gamma, Z, r, eps, residual=None, h_out=None, stream=None):
    """Z = gamma * h / rms(h), h = X (+ residual, in fp32, stored into h_out); r [T] = 1 / rms(h).
    X bf16 or fp32; residual, Z bf16; h_out fp32."""
    T, H = X.shape
    n, w = T * H, "catq_rmsnorm_fwd"
    x = _buf(X, "X", n * X.element_size(), w)
    res, z = _bf16(residual, "residual", 2 * n, w), _bf16(Z, "Z", 2 * n, w)
    h = _f32(h_out, "h_out", 4 * n, w)
    ga, rr = _buf(gamma, "gamma", 4 * H, w), _buf(r, "r", 4 * T, w)
    _check(lib().catq_rmsnorm_fwd(x, _dtype_code(X), res, ga, T, H, float(eps), h, z, rr, _stream(stream)), w)


def catq_rmsnorm_bwd(h, gamma, r, dZ, dX, dZ2=None, d_residual=None, stream=None):
    """dX of catq_rmsnorm_fwd at h (bf16 or fp32); dZ, dZ2, d_residual, dX bf16."""
    T, H = h.shape
    n, w = T * H, "catq_rmsnorm_bwd"
    hp = _buf(h, "h", n * h.element_size(), w)
    dz, dz2 = _bf16(dZ, "dZ", 2 * n, w), _bf16(dZ2, "dZ2", 2 * n, w)
    dr, dx = _bf16(d_residual, "d_residual", 2 * n, w), _bf16(dX, "dX", 2 * n, w)
    ga, rr = _buf(gamma, "gamma", 4 * H, w), _buf(r, "r", 4 * T, w)
    _check(lib().catq_rmsnorm_bwd(hp, _dtype_code(h), ga, rr, dz, dz2, dr, T, H, dx, _stream(stream)), w)


def catq_rope(X, S, n_heads, d, base, inverse=False, stream=None):
    T = X.shape[0]
    w = "catq_rope"
    x = _bf16(X, "X", 2 * T * n_heads * d, w)
    _check(lib().catq_rope(x, T, int(S), int(n_heads), int(d), float(base), int(bool(inverse)), _stream(stream)), w)


def catq_swiglu_fwd(gate, up, M, stream=None):
    n, w = gate.numel(), "catq_swiglu_fwd"
    a, b, m = _bf16(gate, "gate", 2 * n, w), _bf16(up, "up", 2 * n, w), _bf16(M, "M", 2 * n, w)
    _check(lib().catq_swiglu_fwd(a, b, n, m, _stream(stream)), w)


def catq_swiglu_bwd(gate, up, dM, d_gate, d_up, stream=None):
    n, w = gate.numel(), "catq_swiglu_bwd"
    a, b, m = _bf16(gate, "gate", 2 * n, w), _bf16(up, "up", 2 * n, w), _bf16(dM, "dM", 2 * n, w)
    da, db = _bf16(d_gate, "d_gate", 2 * n, w), _bf16(d_up, "d_up", 2 * n, w)
    _check(lib().catq_swiglu_bwd(a, b, m, n, da, db, _stream(stream)), w)


def catq_block_output_loss(h, branch, out_ref=None, loss_out=None, d_out=None, out=None, workspace=None,
                           reduction: int = REDUCE_MEAN, stream=None):
    """out = h + branch in fp32; with out_ref, Eq. 7's loss into loss_out and d_out (bf16)."""
    n, w = h.numel(), "catq_block_output_loss"
    hp, ref, o = _f32(h, "h", 4 * n, w), _f32(out_ref, "out_ref", 4 * n, w), _f32(out, "out", 4 * n, w)
    br, do = _bf16(branch, "branch", 2 * n, w), _bf16(d_out, "d_out", 2 * n, w)
    lo = _buf(loss_out, "loss_out", 4, w)
    ws, ws_bytes = _ws(workspace, w)
    _check(lib().catq_block_output_loss(hp, br, n, ref, int(reduction), lo, do, o, ws, ws_bytes, _stream(stream)), w)


def catq_attention_fwd(Q, K, V, O, lse, B, S, n_heads, n_kv_heads, d, stream=None):
    w = "catq_attention_fwd"
    nq, nk = 2 * B * S * n_heads * d, 2 * B * S * n_kv_heads * d
    q, o = _bf16(Q, "Q", nq, w), _bf16(O, "O", nq, w)
    k, v = _bf16(K, "K", nk, w), _bf16(V, "V", nk, w)
    ls = _buf(lse, "lse", 4 * B * n_heads * S, w)
    _check(lib().catq_attention_fwd(q, k, v, int(B), int(S), int(n_heads), int(n_kv_heads), int(d), o, ls,
                                    _stream(stream)), w)


def catq_attention_bwd(Q, K, V, O, dO, lse, delta, dQ, dK, dV, B, S, n_heads, n_kv_heads, d, stream=None):
    w = "catq_attention_bwd"
    nq, nk, ns = 2 * B * S * n_heads * d, 2 * B * S * n_kv_heads * d, 4 * B * n_heads * S
    q, o = _bf16(Q, "Q", nq, w), _bf16(O, "O", nq, w)
    do, dq = _bf16(dO, "dO", nq, w), _bf16(dQ, "dQ", nq, w)
    k, v = _bf16(K, "K", nk, w), _bf16(V, "V", nk, w)
    dk, dv = _bf16(dK, "dK", nk, w), _bf16(dV, "dV", nk, w)
    ls, de = _buf(lse, "lse", ns, w), _buf(delta, "delta", ns, w)
    _check(lib().catq_attention_bwd(q, k, v, o, do, ls, int(B), int(S), int(n_heads), int(n_kv_heads), int(d), de, dq,
                                    dk, dv, _stream(stream)), w)
