"""ctypes binding of ``libnystra.so`` (C ABI in ``include/nystra.h``).

Argument marshalling, and for ``nystra_qkv`` the choice between two forms of the
same computation; every step of it runs in the CUDA kernels behind the C ABI.
torch is used for device memory and streams.
There is no CPU fallback: if the library is missing, every call raises.
"""
from __future__ import annotations

import contextlib
import ctypes
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libnystra.so")

NYSTRA_F32, NYSTRA_BF16, NYSTRA_F16 = 0, 1, 2
NYSTRA_OK, NYSTRA_EINVAL, NYSTRA_EDTYPE, NYSTRA_ELAUNCH, NYSTRA_ETIMEOUT, NYSTRA_EDEVICE = 0, -1, -2, -3, -4, -5
NYSTRA_LANDMARKS_SEGMENTS, NYSTRA_LANDMARKS_PATCHES = 0, 1
LANDMARKS = {"segments": NYSTRA_LANDMARKS_SEGMENTS, "patches": NYSTRA_LANDMARKS_PATCHES}
# Option flag OR-ed into the landmarks argument: derived factors rounded to
# the 16-bit I/O type (faster, accurate only for soft attention; nystra.h).
NYSTRA_FACTORS_16 = 16
FACTORS = {"pairs": 0, "16": NYSTRA_FACTORS_16}


def _lm(landmarks: str, factors: str = "pairs") -> int:
    return LANDMARKS[landmarks] | FACTORS[factors]
MAX_N, MAX_DH, MAX_M, MAX_ITERS = 1024, 64, 64, 100
QKV_MAX_C = 352
PROJ_MAX_C, PROJ_MAX_N = 384, 65536

_DTYPE_CODE = {torch.float32: NYSTRA_F32, torch.bfloat16: NYSTRA_BF16, torch.float16: NYSTRA_F16}

_lib = None


class NystraError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        msg = f"{where}: {strerror(status)} (status {status})"
        if status == NYSTRA_ELAUNCH:
            msg += f", cudaError {lib().nystra_last_cuda_error()}"
        super().__init__(msg)


def lib() -> ctypes.CDLL:
    """The loaded library; raises if it has not been built (no fallback)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(f"{LIB_PATH} is missing: build it with "
                               "`python -m paper_2506_08520_gb300.build` (no CPU fallback exists)")
        L = ctypes.CDLL(LIB_PATH)
        vp, i = ctypes.c_void_p, ctypes.c_int
        L.nystra_attention.argtypes = [vp, vp, vp, vp, i, i, i, i, i, i, i, vp]
        L.nystra_attention.restype = i
        L.exact_window_attention.argtypes = [vp, vp, vp, vp, i, i, i, i, i, vp]
        L.exact_window_attention.restype = i
        L.nystra_strerror.argtypes = [i]
        L.nystra_strerror.restype = ctypes.c_char_p
        L.nystra_version.restype = i
        L.nystra_last_cuda_error.restype = i
        L.nystra_status.argtypes = [vp]
        L.nystra_status.restype = i
        L.nystra_check.argtypes = [vp]
        L.nystra_check.restype = i
        L.nystra_debug_wait_timeout.argtypes = [ctypes.c_ulonglong, vp]
        L.nystra_debug_wait_timeout.restype = i
        L.nystra_debug_stages.argtypes = [vp, vp, vp, i, i, i, i, i, i, i, i, ctypes.c_longlong, vp, vp]
        L.nystra_attention_ex.argtypes = [vp, vp, vp, vp, i, i, i, i, i, i, i, i, vp]
        L.nystra_attention_ex.restype = i
        L.nystra_pool_bias.argtypes = [vp, i, i, i, i, vp, vp, vp, vp]
        L.nystra_pool_bias.restype = i
        L.nystra_attention_bias.argtypes = [vp, vp, vp, vp, i, i, i, i, i, i, i, vp, vp, vp, i, i, vp]
        L.nystra_attention_bias.restype = i
        L.nystra_attention_qkv.argtypes = [vp, vp, vp, vp, i, i, i, i, i, i, i, vp, vp, vp, i, i, vp]
        L.nystra_attention_qkv.restype = i
        L.nystra_project_qkv.argtypes = [vp, vp, vp, vp, vp, vp, i, i, i, i, i, vp]
        L.nystra_project_qkv.restype = i
        L.nystra_debug_stages.restype = i
        L.nystra_debug_stages_size.argtypes = [i, i, i]
        L.nystra_debug_stages_size.restype = ctypes.c_longlong
        _lib = L
    return _lib


# ---------------------------------------------------------------- raw C ABI
def nystra_attention(q, k, v, out, n_windows, heads, N, d_h, m, iters, dtype, stream) -> int:
    """Raw C-ABI call: pointers as ints, returns the status code."""
    return lib().nystra_attention(q, k, v, out, n_windows, heads, N, d_h, m, iters, dtype, stream)


def nystra_attention_ex(q, k, v, out, n_windows, heads, N, d_h, m, iters, landmarks, dtype, stream) -> int:
    """Raw C-ABI call with a landmark pooling (NYSTRA_LANDMARKS_*)."""
    return lib().nystra_attention_ex(q, k, v, out, n_windows, heads, N, d_h, m, iters, landmarks, dtype, stream)


def nystra_pool_bias(bias, n_bias, N, m, landmarks, bias_L, bias_U, bias_A, stream) -> int:
    return lib().nystra_pool_bias(bias, n_bias, N, m, landmarks, bias_L, bias_U, bias_A, stream)


def nystra_attention_bias(q, k, v, out, n_windows, heads, N, d_h, m, iters, landmarks, bias_L, bias_U, bias_A,
                          bias_windows, dtype, stream) -> int:
    return lib().nystra_attention_bias(q, k, v, out, n_windows, heads, N, d_h, m, iters, landmarks, bias_L, bias_U,
                                       bias_A, bias_windows, dtype, stream)


def nystra_attention_qkv(x, w_qkv, b_qkv, out, n_windows, heads, N, d_h, m, iters, landmarks, bias_L, bias_U,
                         bias_A, bias_windows, dtype, stream) -> int:
    return lib().nystra_attention_qkv(x, w_qkv, b_qkv, out, n_windows, heads, N, d_h, m, iters, landmarks, bias_L,
                                      bias_U, bias_A, bias_windows, dtype, stream)


def nystra_project_qkv(x, w_qkv, b_qkv, q, k, v, n_windows, heads, N, d_h, dtype, stream) -> int:
    return lib().nystra_project_qkv(x, w_qkv, b_qkv, q, k, v, n_windows, heads, N, d_h, dtype, stream)


def exact_window_attention(q, k, v, out, n_windows, heads, N, d_h, dtype, stream) -> int:
    return lib().exact_window_attention(q, k, v, out, n_windows, heads, N, d_h, dtype, stream)


def strerror(status: int) -> str:
    return lib().nystra_strerror(status).decode()


def version() -> int:
    return lib().nystra_version()


def status(stream=None) -> int:
    """Synchronise ``stream`` and return the device-side fault status."""
    return lib().nystra_status(_stream_ptr(stream))


def check(stream=None) -> int:
    """Same as ``status``."""
    return lib().nystra_check(_stream_ptr(stream))


def debug_wait_timeout(limit_ns: int, stream=None) -> int:
    """Test-only: launch a wait that can only time out (see the header)."""
    return lib().nystra_debug_wait_timeout(int(limit_ns), _stream_ptr(stream))


def nystra_debug_stages(q, k, v, n_windows, heads, N, d_h, m, iters, landmarks, dtype, unit, dump, stream) -> int:
    """Raw C-ABI call of the test-only stage dump (see the header)."""
    return lib().nystra_debug_stages(q, k, v, n_windows, heads, N, d_h, m, iters, landmarks, dtype, int(unit), dump,
                                     stream)


def nystra_debug_stages_size(N: int, d_h: int, m: int) -> int:
    return lib().nystra_debug_stages_size(N, d_h, m)


# Regions of the stage dump, in the order and with the shapes the header gives.
def _stage_shapes(N: int, d: int, m: int):
    return [("qbar", (m, d)), ("kbar", (m, d)), ("GLn", (N, m)), ("mU", (m,)), ("W", (m, d + 1)),
            ("GAn", (m, m)), ("Z", (m, m)), ("Y", (m, d + 1)), ("out", (N, d))]


# ------------------------------------------------------------ torch helpers
def _stream_ptr(stream) -> int | None:
    if stream is None:
        return torch.cuda.current_stream().cuda_stream
    if isinstance(stream, torch.cuda.Stream):
        return stream.cuda_stream
    return int(stream)


def _geometry(q: torch.Tensor):
    if q.dim() == 4:
        n_windows, heads, N, d = q.shape
    elif q.dim() == 3:
        (n_windows, N, d), heads = q.shape, 1
    else:
        raise ValueError("expected [n_windows, heads, N, d_h] or [units, N, d_h]")
    return n_windows, heads, N, d


def _check(q, k, v, out):
    for t in (q, k, v, out):
        if not t.is_cuda:
            raise ValueError("tensors must be on a CUDA device (no CPU path)")
        if not t.is_contiguous():
            raise ValueError("tensors must be contiguous")
        if t.shape != q.shape or t.dtype != q.dtype:
            raise ValueError("q, k, v and out must share shape and dtype")
    if q.dtype not in _DTYPE_CODE:
        raise ValueError(f"unsupported dtype {q.dtype}")


def nystra(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, m: int = 16, iters: int = 6,
           out: torch.Tensor | None = None, stream=None, landmarks: str = "segments",
           factors: str = "pairs") -> torch.Tensor:
    """PnP-Nystra attention of device tensors ``[n_windows, heads, N, d_h]``;
    ``landmarks`` is "segments" (default) or "patches" (square patches);
    ``factors`` "pairs" (default: derived factors as 16-bit hi + lo pairs) or
    "16" (rounded to the 16-bit I/O type, NYSTRA_FACTORS_16)."""
    out = torch.empty_like(q) if out is None else out
    _check(q, k, v, out)
    nw, h, N, d = _geometry(q)
    with torch.cuda.device(q.device):
        if landmarks == "segments" and factors == "pairs":
            rc = nystra_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), nw, h, N, d,
                                  m, iters, _DTYPE_CODE[q.dtype], _stream_ptr(stream))
        else:
            rc = nystra_attention_ex(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), nw, h, N, d,
                                     m, iters, _lm(landmarks, factors), _DTYPE_CODE[q.dtype], _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_attention")
    return out


def exact(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, out: torch.Tensor | None = None,
          stream=None) -> torch.Tensor:
    """Exact softmax window attention (the computation PnP-Nystra replaces)."""
    out = torch.empty_like(q) if out is None else out
    _check(q, k, v, out)
    nw, h, N, d = _geometry(q)
    with torch.cuda.device(q.device):
        rc = exact_window_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), nw, h, N, d,
                                    _DTYPE_CODE[q.dtype], _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "exact_window_attention")
    return out


def debug_stages(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, m: int, iters: int, unit: int,
                 stream=None, landmarks: str = "segments") -> dict:
    """Test-only: every intermediate of one unit (fp32 CPU tensors by name)."""
    _check(q, k, v, q)
    nw, h, N, d = _geometry(q)
    size = nystra_debug_stages_size(N, d, m)
    if size < 0:
        raise NystraError(int(size), "nystra_debug_stages_size")
    dump = torch.empty(size, dtype=torch.float32, device=q.device)
    with torch.cuda.device(q.device):
        rc = nystra_debug_stages(q.data_ptr(), k.data_ptr(), v.data_ptr(), nw, h, N, d, m, iters,
                                 LANDMARKS[landmarks], _DTYPE_CODE[q.dtype], unit, dump.data_ptr(),
                                 _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_debug_stages")
    torch.cuda.synchronize(q.device)
    host = dump.cpu()
    out, pos = {}, 0
    for name, shape in _stage_shapes(N, d, m):
        n = 1
        for x in shape:
            n *= x
        out[name] = host[pos:pos + n].reshape(shape)
        pos += n
    return out


def pool_bias(bias: torch.Tensor, m: int, landmarks: str = "segments", stream=None):
    """Landmark blocks (B_L, B_U, B_A) of an fp32 device bias ``[..., N, N]``."""
    if not bias.is_cuda or bias.dtype != torch.float32 or not bias.is_contiguous():
        raise ValueError("bias must be a contiguous fp32 CUDA tensor")
    N = bias.shape[-1]
    lead = bias.shape[:-2]
    n = bias.numel() // (N * N)
    bL = torch.empty(lead + (N, m), dtype=torch.float32, device=bias.device)
    bU = torch.empty(lead + (m, N), dtype=torch.float32, device=bias.device)
    bA = torch.empty(lead + (m, m), dtype=torch.float32, device=bias.device)
    with torch.cuda.device(bias.device):
        rc = nystra_pool_bias(bias.data_ptr(), n, N, m, LANDMARKS[landmarks], bL.data_ptr(), bU.data_ptr(),
                              bA.data_ptr(), _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_pool_bias")
    return bL, bU, bA


def nystra_biased(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, pooled, m: int = 16, iters: int = 6,
                  out: torch.Tensor | None = None, stream=None, landmarks: str = "segments",
                  factors: str = "pairs") -> torch.Tensor:
    """PnP-Nystra with a score bias already pooled by ``pool_bias``: blocks of
    shape ``[heads, ...]`` (shared by all windows) or ``[n_windows, heads, ...]``."""
    out = torch.empty_like(q) if out is None else out
    _check(q, k, v, out)
    nw, h, N, d = _geometry(q)
    bL, bU, bA = pooled
    bw = bL.numel() // (h * N * m)
    with torch.cuda.device(q.device):
        rc = nystra_attention_bias(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), nw, h, N, d, m, iters,
                                   _lm(landmarks, factors), bL.data_ptr(), bU.data_ptr(), bA.data_ptr(), bw,
                                   _DTYPE_CODE[q.dtype], _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_attention_bias")
    return out


def nystra_qkv(x: torch.Tensor, w_qkv: torch.Tensor, heads: int, m: int = 16, iters: int = 6,
               b_qkv: torch.Tensor | None = None, pooled=None, out: torch.Tensor | None = None, stream=None,
               landmarks: str = "segments", factors: str = "pairs") -> torch.Tensor:
    """Projection + PnP-Nystra: tokens ``x`` ``[n_windows, N, C]``, weights
    ``w_qkv`` ``[3C, C]`` (a linear layer's weight: Q rows, then K, then V),
    optional fp32 bias ``b_qkv`` ``[3C]`` and pooled score bias (as for
    ``nystra_biased``).  Returns ``[n_windows, heads, N, C / heads]``.  Runs as
    one fused kernel (nystra_attention_qkv) or, where that is faster, as the
    projection and the attention by turns over a workspace of up to
    ``QKV_WORKSPACE`` bytes from torch's allocator (`_two_pass`); without memory
    for it, and in a stream capture with ``out`` or ``stream`` given, as the fused
    kernel, which needs none."""
    if x.dim() != 3 or w_qkv.dim() != 2:
        raise ValueError("expected x [n_windows, N, C] and w_qkv [3C, C]")
    nw, N, C = x.shape
    if heads < 1 or C % heads:
        raise ValueError(f"C={C} does not split into {heads} heads")
    d = C // heads
    if tuple(w_qkv.shape) != (3 * C, C):
        raise ValueError(f"w_qkv must be [{3 * C}, {C}]")
    own = out is None
    out = torch.empty((nw, heads, N, d), dtype=x.dtype, device=x.device) if own else out
    for t in (x, w_qkv, out):
        if not t.is_cuda or not t.is_contiguous() or t.dtype != x.dtype:
            raise ValueError("x, w_qkv and out must be contiguous CUDA tensors of one dtype (no CPU path)")
    if x.dtype not in _DTYPE_CODE:
        raise ValueError(f"unsupported dtype {x.dtype}")
    if tuple(out.shape) != (nw, heads, N, d):
        raise ValueError(f"out must be [{nw}, {heads}, {N}, {d}]")
    bp = 0
    if b_qkv is not None:
        if not b_qkv.is_cuda or b_qkv.dtype != torch.float32 or not b_qkv.is_contiguous() or b_qkv.numel() != 3 * C:
            raise ValueError(f"b_qkv must be a contiguous fp32 CUDA tensor of {3 * C} values")
        bp = b_qkv.data_ptr()
    bL = bU = bA = 0
    bw = 0
    if pooled is not None:
        bL, bU, bA = (t.data_ptr() for t in pooled)
        bw = pooled[0].numel() // (heads * N * m)
    lm, dt = _lm(landmarks, factors), _DTYPE_CODE[x.dtype]
    with torch.cuda.device(x.device):
        two = _two_pass(nw, N, heads, d, m, iters, landmarks, x, w_qkv, b_qkv, pooled, bw, out, stream)
        rc = (_qkv_two_pass(x, w_qkv, bp, out, own, nw, heads, N, d, m, iters, lm, bL, bU, bA, bw, dt, stream)
              if two else None)
        if rc is None:
            rc = nystra_attention_qkv(x.data_ptr(), w_qkv.data_ptr(), bp, out.data_ptr(), nw, heads, N, d, m, iters,
                                      lm, bL, bU, bA, bw, dt, _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_attention_qkv")
    return out


# The two-pass form of nystra_qkv: the tcgen05 projection into a workspace of
# at most QKV_WORKSPACE bytes, then the attention on it, window chunk by window
# chunk.  Q, K and V are rounded to the I/O type in both forms.
QKV_WORKSPACE = 256 << 20


def _disjoint(out: torch.Tensor, t: torch.Tensor | None) -> bool:
    if t is None:
        return True
    a, b = out.data_ptr(), t.data_ptr()
    return a >= b + t.numel() * t.element_size() or b >= a + out.numel() * out.element_size()


def _two_pass(nw, N, heads, d, m, iters, landmarks, x, w_qkv, b_qkv, pooled, bw, out, stream) -> bool:
    """Whether nystra_qkv takes the two-pass form: where it is the faster one,
    for calls that nystra_attention_qkv accepts (it refuses the others) on a
    stream the workspace can be allocated for.

    The lines, from times of both forms (m = 16, bf16, fused / two-pass, us a call
    among others; a call that is waited for pays about 10 more for the second
    form's host work).  32x32 windows everywhere (1 x 16 features, 2048 tokens
    48/33; 6 x 30, 262144 tokens 706/240).  16x16 windows from 128 token features on
    (4 x 32, 2048 tokens 50/34; 6 x 30, 262144 tokens 586/248) or 64 and 65536 tokens
    (2 x 32: 62/52, 3 x 32: 70/71, the one tie; but 1 x 32: 27/33, and at 2048 tokens
    4 x 24: 33/29, waited for 42/48).  8x8 windows from 80 features and 65536 tokens
    on (4 x 20: 61/56, 4 x 30: 74/57, 8 x 30: 177/149, 11 x 30: 313/308; but 2 x 32:
    43/50, and at 32768 tokens 4 x 20: 33/40, 8 x 28: 92/99, 11 x 30: 158/169), up to
    180 features from 8e6 token features on (6 x 30, 45056 tokens 99/65, 5 x 30, 57344
    tokens 98/81; at 24576 tokens 62/44, waited for 71/64, and 42/48).  There heads of
    32 from 128 features and 98304 tokens on (4 x 32: 132/134 and, 131072 tokens,
    173/164, 8 x 32: 337/305; but 3 x 32: 100/108, 223/233 at 262144 tokens, and 9 x
    32, 65536 tokens: 264/274), and not 320 features (10 x 32, 65536 tokens: 322/405, 20
    x 16: 502/732): the projection's CTAs hold one head's weights there, so the tokens
    are read once a head, from rows that all start in one bank."""
    C, T = heads * d, nw * N
    if N == 64:
        faster = C >= 80 and (T >= 65536 or (C <= 180 and C * T >= 8e6)) and not (C > 256 and C % 64 == 0)
        faster = faster and (d < 32 or (C >= 128 and T >= 98304))
    else:
        faster = N == 1024 or (N == 256 and (C >= 128 or (C >= 64 and T >= 65536)))
    if not faster:
        return False
    inputs = (x, w_qkv, b_qkv) + (tuple(pooled) if pooled is not None else ())
    return (nw > 0 and x.dtype in (torch.bfloat16, torch.float16)
            and (stream is None or isinstance(stream, torch.cuda.Stream))
            and d % 2 == 0 and 2 <= d <= 32 and heads * d <= QKV_MAX_C and 0 <= iters <= 12
            and (m in (8, 16) or (m == 32 and N == 1024 and pooled is None)) and (landmarks == "segments" or m == 16)
            and (pooled is None or bw in (1, nw))
            and all(t is None or (t.data_ptr() % 16 == 0 and _disjoint(out, t)) for t in inputs)
            and out.data_ptr() % 16 == 0)


def _qkv_two_pass(x, w_qkv, bp, out, own, nw, heads, N, d, m, iters, lm, bL, bU, bA, bw, dt, stream):
    """The status code, or None if there is no memory to use as the workspace.

    A captured graph goes on using the workspace after this call has returned.  Only
    the allocator's own captures give such memory a pool of its own, and who began
    a capture cannot be told, so the workspace then lies behind ``out`` in the same
    storage and lives as long as the graph's result does.  Where ``out`` is the
    caller's (``own`` false), or lies in another stream's memory, there is no such
    place, and nothing is allocated."""
    win = heads * N * d * 2  # bytes of one window's Q (as of its tokens and its output)
    per = max(1, min(nw, QKV_WORKSPACE // (3 * win)))
    per = -(-nw // (-(-nw // per)))  # chunks of equal length
    try:
        # from the pool of the stream it is used on: safe to reuse in stream order once freed
        with contextlib.nullcontext() if stream is None else torch.cuda.stream(stream):
            if not torch.cuda.is_current_stream_capturing():
                ws, start = torch.empty(3 * per * win, dtype=torch.uint8, device=x.device), 0
            elif own and stream is None:
                start = -(-nw * win // 512) * 512
                ws = torch.empty(start + 3 * per * win, dtype=torch.uint8, device=x.device)
                out.set_(ws.untyped_storage(), 0, out.shape, out.stride())
            else:
                return None
    except RuntimeError:  # out of memory, or the allocator may not grow now
        return None
    q, k, v = (ws.data_ptr() + start + i * per * win for i in range(3))
    xp, op, wp, st = x.data_ptr(), out.data_ptr(), w_qkv.data_ptr(), _stream_ptr(stream)
    for i in range(0, nw, per):
        n = min(per, nw - i)
        rc = nystra_project_qkv(xp + i * win, wp, bp, q, k, v, n, heads, N, d, dt, st)
        if rc == NYSTRA_OK and bL == 0:
            rc = nystra_attention_ex(q, k, v, op + i * win, n, heads, N, d, m, iters, lm, dt, st)
        elif rc == NYSTRA_OK:
            u = i * heads * 4 if bw != 1 else 0  # per-window blocks: this chunk's first
            rc = nystra_attention_bias(q, k, v, op + i * win, n, heads, N, d, m, iters, lm, bL + u * N * m,
                                       bU + u * N * m, bA + u * m * m, n if bw != 1 else 1, dt, st)
        if rc != NYSTRA_OK:
            return rc
    return NYSTRA_OK


def project_qkv(x: torch.Tensor, w_qkv: torch.Tensor, heads: int, b_qkv: torch.Tensor | None = None,
                out=None, stream=None):
    """Q, K, V projections of tokens ``x`` ``[n_windows, N, C]`` by ``w_qkv``
    ``[3C, C]`` (+ optional fp32 ``b_qkv`` ``[3C]``), split into heads: returns
    ``(q, k, v)``, each ``[n_windows, heads, N, C / heads]`` in x's dtype,
    ready for ``nystra``/``exact``.  ``out`` may give the three tensors."""
    if x.dim() != 3 or w_qkv.dim() != 2:
        raise ValueError("expected x [n_windows, N, C] and w_qkv [3C, C]")
    nw, N, C = x.shape
    if heads < 1 or C % heads:
        raise ValueError(f"C={C} does not split into {heads} heads")
    d = C // heads
    if tuple(w_qkv.shape) != (3 * C, C):
        raise ValueError(f"w_qkv must be [{3 * C}, {C}]")
    if out is None:
        out = tuple(torch.empty((nw, heads, N, d), dtype=x.dtype, device=x.device) for _ in range(3))
    for t in (x, w_qkv, *out):
        if not t.is_cuda or not t.is_contiguous() or t.dtype != x.dtype:
            raise ValueError("x, w_qkv and the outputs must be contiguous CUDA tensors of one dtype (no CPU path)")
    if x.dtype not in _DTYPE_CODE:
        raise ValueError(f"unsupported dtype {x.dtype}")
    for t in out:
        if tuple(t.shape) != (nw, heads, N, d):
            raise ValueError(f"outputs must be [{nw}, {heads}, {N}, {d}]")
    bp = 0
    if b_qkv is not None:
        if not b_qkv.is_cuda or b_qkv.dtype != torch.float32 or not b_qkv.is_contiguous() or b_qkv.numel() != 3 * C:
            raise ValueError(f"b_qkv must be a contiguous fp32 CUDA tensor of {3 * C} values")
        bp = b_qkv.data_ptr()
    q, k, v = out
    with torch.cuda.device(x.device):
        rc = nystra_project_qkv(x.data_ptr(), w_qkv.data_ptr(), bp, q.data_ptr(), k.data_ptr(), v.data_ptr(), nw,
                                heads, N, d, _DTYPE_CODE[x.dtype], _stream_ptr(stream))
    if rc != NYSTRA_OK:
        raise NystraError(rc, "nystra_project_qkv")
    return q, k, v
