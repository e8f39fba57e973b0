"""Python binding of the C ABI in include/amq.h (same names, argument marshalling only).

PyTorch supplies device memory and the current stream; every step of the path runs in the CUDA
library.  Importing this module loads paper_1802_00150_b200/libamq_b200.so and raises if it is missing:
there is no CPU fallback.  The calls that enqueue work go through the native binding (csrc/amq_binding.cpp), which
checks tensors, takes their addresses and adds the current stream; size helpers and status calls go through ctypes.
"""
import ctypes
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
# the product library; AMQ_B200_LIBRARY names an instrumented build of the same sources instead (see build.py)
LIB_PATH = os.environ.get("AMQ_B200_LIBRARY") or os.path.join(_HERE, "libamq_b200.so")

if not os.path.exists(LIB_PATH):
    raise ImportError(
        "CUDA library %s is missing: build it with `python -m paper_1802_00150_b200.build` "
        "(there is no CPU fallback)" % LIB_PATH)

_lib = ctypes.CDLL(LIB_PATH)

from . import _amq_binding as _native  # noqa: E402  (built beside the library; raises if it is missing)

_native.open(LIB_PATH)

OK = 0
MAX_K = 4
MAX_N = 8192

_vp, _int, _sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t

EXPORTS = {
    "amq_status_string": (ctypes.c_char_p, [_int]),
    "amq_last_cuda_error": (_int, []),
    "amq_kernel_launches": (ctypes.c_ulonglong, []),
    "amq_words_per_row": (_int, [_int]),
    "amq_codes_bytes": (_sz, [_int, _int, _int]),
    "amq_quantize": (_int, [_vp, _int, _int, _int, _int, _int, _vp, _vp, _vp]),
    "amq_pack": (_int, [_vp, _int, _int, _int, _vp, _vp]),
    "amq_unpack": (_int, [_vp, _vp, _int, _int, _int, _vp, _vp]),
    "amq_binary_dots": (_int, [_vp, _int, _int, _int, _vp, _int, _int, _vp, _vp]),
    "amq_binary_gemm": (_int, [_vp, _vp, _int, _int, _int, _vp, _vp, _int, _int, _vp, _vp, _int, _vp]),
    "amq_quantized_gemv": (_int, [_vp, _vp, _int, _int, _int, _vp, _int, _int, _vp, _vp, _vp, _vp, _vp]),
    "amq_device_status": (_int, [_vp]),
    "amq_cell_workspace_bytes": (_sz, [_int, _int, _int, _int]),
    "amq_cell_host_staging_bytes": (_sz, [_int, _int, _int, _int]),
    "amq_lstm_step": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _vp, _vp, _int, _int, _int, _vp, _vp, _vp, _sz, _vp]),
    "amq_lstm_step_static_scratch_bytes": (_sz, [_int, _int, _int, _int]),
    "amq_lstm_step_static": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _vp, _vp, _int, _int, _int, _vp, _vp, _vp]),
    "amq_gru_step": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _vp, _int, _int, _int, _vp, _vp, _sz, _vp]),
    "amq_lstm_sequence": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _int, _vp, _vp, _int, _int, _int,
                                 _vp, _vp, _vp, _vp, _sz, _vp]),
    "amq_gru_sequence": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _int, _vp, _int, _int, _int,
                                _vp, _vp, _vp, _sz, _vp]),
    "amq_lstm_sequence_host": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _int, _vp, _vp, _int, _int, _int,
                                      _vp, _vp, _vp, _vp, _sz, _vp, _sz, _vp]),
    "amq_gru_sequence_host": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _int, _vp, _int, _int, _int,
                                     _vp, _vp, _vp, _sz, _vp, _sz, _vp]),
    "amq_workspace_status": (_int, [_vp, _vp]),
    "amq_selftest_sequence_give_up": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _int, _vp, _vp, _int, _int,
                                             _vp, _vp, _vp, _sz, ctypes.c_uint, _vp]),
    "amq_selftest_sequence_plan": (_int, [_int, _int, _int, _int, _int, _int, _int, ctypes.POINTER(_int), ctypes.POINTER(_int),
                                          ctypes.POINTER(ctypes.c_double)]),
    "amq_selftest_batched_sequence": (_int, [_vp, _vp, _vp, _int, _int, _int, _int, _vp, _int, _vp, _vp, _int, _int, _int,
                                             _vp, _vp, _vp, _vp, _sz, _int, _int, _int, _vp]),
    "amq_selftest_product_plan": (_int, [_int, _int, _int, _int, _int, _int, _int, ctypes.POINTER(_int), ctypes.POINTER(ctypes.c_double)]),
    "amq_selftest_binary_gemm": (_int, [_vp, _vp, _int, _int, _int, _vp, _vp, _int, _int, _vp, _vp, _int, _int, _vp]),
    "amq_selftest_decode_give_up": (_int, [_vp, _vp, _int, _int, _int, _vp, _vp, _vp, _vp, _vp, _int, _int, _vp, _vp, _vp, _int,
                                           _int, _int, _vp, _int, _vp, _vp, _vp, _sz, _int, _vp]),
    "amq_gru_original_workspace_bytes": (_sz, [_int, _int, _int, _int]),
    "amq_gru_step_original": (_int, [_vp, _vp, _vp, _int, _int, _int, _vp, _vp, _int, _int, _int, _vp, _vp, _sz, _vp]),
    "amq_quantize_variant": (_int, [_vp, _int, _int, _int, _int, _int, _int, _int, _vp, _vp, _vp]),
    "amq_lm_decode_workspace_bytes": (_sz, [_int, _int, _int, _int, _int]),
    "amq_lm_greedy_decode": (_int, [_vp, _vp, _int, _int, _int, _vp, _vp, _vp, _vp, _vp, _int, _int, _vp, _vp, _vp, _int,
                                    _int, _int, _vp, _int, _vp, _vp, _vp, _vp, _sz, _vp]),
    "amq_log_softmax_argmax": (_int, [_vp, _int, _int, _int, _vp, _int, _vp, _vp]),
    "amq_embedding_rows": (_int, [_vp, _vp, _int, _int, _int, _vp, _int, _vp, _vp, _vp]),
    "amq_lstm_paper_workspace_bytes": (_sz, [_int, _int, _int, _int]),
    "amq_lstm_step_paper": (_int, [_vp, _vp, _vp, _vp, _vp, _int, _int, _int, _vp, _vp, _int, _vp, _vp, _int, _int, _int,
                                   _vp, _vp, _vp, _sz, _vp]),
    "amq_lstm_sequence_paper": (_int, [_vp, _vp, _vp, _vp, _vp, _int, _int, _int, _vp, _vp, _int, _int, _vp, _vp, _int, _int,
                                       _int, _vp, _vp, _vp, _vp, _sz, _vp]),
}

for _name, (_res, _args) in EXPORTS.items():
    _fn = getattr(_lib, _name)
    _fn.restype = _res
    _fn.argtypes = _args


class AmqError(RuntimeError):
    def __init__(self, status):
        self.status = status
        msg = _lib.amq_status_string(status).decode()
        if status == -5:
            msg += " (cudaError %d)" % _lib.amq_last_cuda_error()
        super().__init__("amq status %d: %s" % (status, msg))


def _check(status):
    if status != OK:
        raise AmqError(status)


def _ptr(t):
    return None if t is None else t.data_ptr()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def status_string(status):
    return _lib.amq_status_string(status).decode()


def kernel_launches():
    return int(_lib.amq_kernel_launches())


def words_per_row(n):
    return _lib.amq_words_per_row(n)


def codes_bytes(rows, n, k):
    return _lib.amq_codes_bytes(rows, n, k)


def _new_codes(rows, k, n, like):
    return _native.empty(like, 1, rows, k, 4 * ((n + 127) // 128))


def quantize(x, k, T, codes=None, coeffs=None):
    """x (rows, n) fp32, possibly a row-strided view -> codes (rows, k, wpr) int32, coeffs (rows, k) fp32."""
    if not (x.is_cuda and x.dtype == torch.float32 and x.dim() == 2 and x.stride(1) == 1):
        raise TypeError("x must be a 2-D CUDA fp32 tensor with unit column stride")
    rows, n = x.shape
    ldx = x.stride(0) if rows > 1 else max(n, x.stride(0))
    codes = _new_codes(rows, k, n, x) if codes is None else codes
    coeffs = _native.empty(x, 0, rows, k) if coeffs is None else coeffs
    _check(_native.amq_quantize(x.data_ptr(), rows, n, ldx, k, T, codes, coeffs))
    return codes, coeffs


def pack(planes):
    """planes (rows, k, n) fp32 (>= 0 -> +1) -> codes (rows, k, wpr) int32."""
    rows, k, n = planes.shape
    codes = _new_codes(rows, k, n, planes)
    _check(_native.amq_pack(planes, rows, n, k, codes))
    return codes


def unpack(codes, coeffs, n):
    rows, k, _ = codes.shape
    xhat = _native.empty(codes, 0, rows, n)
    _check(_native.amq_unpack(codes, coeffs, rows, n, k, xhat))
    return xhat


def binary_dots(Wcodes, xcodes, n):
    """-> D (batch, m, k_w, k_a) int32."""
    m, k_w, _ = Wcodes.shape
    batch, k_a, _ = xcodes.shape
    D = _native.empty(Wcodes, 1, batch, m, k_w, k_a)
    _check(_native.amq_binary_dots(Wcodes, m, n, k_w, xcodes, batch, k_a, D))
    return D


def binary_gemm(Wcodes, Walpha, xcodes, xbeta, n, bias=None, y=None):
    """-> y (batch, m) fp32."""
    m, k_w, _ = Wcodes.shape
    batch, k_a, _ = xcodes.shape
    if y is None:
        y = _native.empty(Wcodes, 0, batch, m)
    _check(_native.amq_binary_gemm(Wcodes, Walpha, m, n, k_w, xcodes, xbeta, batch, k_a,
                                bias, y.data_ptr(), y.stride(0) if batch > 1 else max(m, y.stride(0))))
    return y


def quantized_gemv(Wcodes, Walpha, x, k_a, T, bias=None, y=None, want_codes=False):
    """Table 6's operation in one launch: x (n,) or (1, n) fp32 is quantized on-line (k_a bits, T cycles) inside the
    product kernel.  Returns y (m,), or (y, xcodes (k_a, wpr), xbeta (k_a,)) with want_codes."""
    m, k_w, wpr = Wcodes.shape
    n = x.numel()
    if y is None:
        y = _native.empty(x, 0, m)
    xc = _native.empty(x, 1, k_a, wpr) if want_codes else None
    xb = _native.empty(x, 0, k_a) if want_codes else None
    _check(_native.amq_quantized_gemv(Wcodes, Walpha, m, n, k_w, x, k_a, T, bias, y,
                                   xc, xb))
    return (y, xc, xb) if want_codes else y


def device_status():
    """0, or -6 when a bounded device-side wait of a product kernel ran out since the last call."""
    return _lib.amq_device_status(_stream())


def cell_workspace_bytes(I, H, batch, k_a):
    return _lib.amq_cell_workspace_bytes(I, H, batch, k_a)


def cell_host_staging_bytes(I, H, batch, steps):
    return _lib.amq_cell_host_staging_bytes(I, H, batch, steps)


def new_workspace(I, H, batch, k_a, device="cuda"):
    return torch.zeros(max(cell_workspace_bytes(I, H, batch, k_a), 16), dtype=torch.uint8, device=device)


def new_host_staging(I, H, batch, steps, device="cuda"):
    return torch.empty(max(cell_host_staging_bytes(I, H, batch, steps), 16), dtype=torch.uint8, device=device)


def lstm_step(Wcodes, Walpha, bias, I, H, x, h_in, c_in, k_a, T, workspace, h_out=None, c_out=None):
    batch, k_w = h_in.shape[0], Wcodes.shape[1]
    h_out = _native.empty(h_in, 0, *h_in.shape) if h_out is None else h_out
    c_out = _native.empty(c_in, 0, *c_in.shape) if c_out is None else c_out
    _check(_native.amq_lstm_step(Wcodes, Walpha, bias, I, H, k_w, x, h_in, c_in,
                              batch, k_a, T, h_out, c_out, workspace, workspace.numel()))
    return h_out, c_out


STATIC_SCRATCH_BYTES = 1 << 20


def lstm_step_static_scratch_bytes(I, H, batch, k_a):
    return _lib.amq_lstm_step_static_scratch_bytes(I, H, batch, k_a)


def lstm_step_static(Wcodes, Walpha, bias, I, H, x, h_in, c_in, k_a, T, h_out, c_out):
    """amq_lstm_step without a workspace: the library's built-in scratch array is used, and neither this
    wrapper nor the call allocates (the caller brings h_out and c_out).  Problems whose scratch exceeds
    STATIC_SCRATCH_BYTES raise AmqError(-4)."""
    batch, k_w = h_in.shape[0], Wcodes.shape[1]
    _check(_native.amq_lstm_step_static(Wcodes, Walpha, bias, I, H, k_w, x, h_in,
                                     c_in, batch, k_a, T, h_out, c_out))
    return h_out, c_out


def gru_step(Wcodes, Walpha, bias, I, H, x, h_in, k_a, T, workspace, h_out=None):
    batch, k_w = h_in.shape[0], Wcodes.shape[1]
    h_out = _native.empty(h_in, 0, *h_in.shape) if h_out is None else h_out
    _check(_native.amq_gru_step(Wcodes, Walpha, bias, I, H, k_w, x, h_in,
                             batch, k_a, T, h_out, workspace, workspace.numel()))
    return h_out


def lstm_sequence(Wcodes, Walpha, bias, I, H, x_seq, h0, c0, k_a, T, workspace, want_h_seq=False,
                  h_seq=None, h_last=None, c_last=None):
    steps, batch, k_w = x_seq.shape[0], h0.shape[0], Wcodes.shape[1]
    if want_h_seq and h_seq is None:
        h_seq = _native.empty(h0, 0, steps, batch, H)
    h_last = _native.empty(h0, 0, *h0.shape) if h_last is None else h_last
    c_last = _native.empty(c0, 0, *c0.shape) if c_last is None else c_last
    _check(_native.amq_lstm_sequence(Wcodes, Walpha, bias, I, H, k_w, x_seq, steps, h0,
                                  c0, batch, k_a, T, h_seq, h_last, c_last,
                                  workspace, workspace.numel()))
    return h_seq, h_last, c_last


def selftest_sequence_give_up(Wcodes, Walpha, bias, I, H, x_seq, h0, c0, k_a, T, workspace, poll_limit):
    """Test aid: the batch-1 LSTM sequence kernel with waits that run out (see amq.h).  Returns (h_last, c_last),
    which the kernel leaves unwritten; read the outcome with workspace_status."""
    h_last, c_last = torch.zeros_like(h0), torch.zeros_like(c0)
    _check(_native.amq_selftest_sequence_give_up(Wcodes, Walpha, bias, I, H, Wcodes.shape[1], x_seq,
                                              x_seq.shape[0], h0, c0, k_a, T, h_last, c_last,
                                              workspace, workspace.numel(), poll_limit))
    return h_last, c_last


FORM_CHAIN, FORM_STREAMING, FORM_RESIDENT = 0, 1, 2


def selftest_sequence_plan(gru, I, H, k_w, k_a, batch, sm_count=0, form=-1):
    """How a batched sequence would run (see amq.h): (form, (CTAs and vectors of a block, warps per quantized vector), estimated clocks of a
    timestep)."""
    f, split, clocks = _int(form), (_int * 3)(), ctypes.c_double(0.0)
    _check(_lib.amq_selftest_sequence_plan(int(gru), I, H, k_w, k_a, batch, sm_count, ctypes.byref(f), split, ctypes.byref(clocks)))
    return f.value, tuple(split), clocks.value


def selftest_product_plan(m, n, k_w, k_a, batch, sm_count=0, ldy=None):
    """Which kernel a product runs on (see amq.h): (form, (estimates of the streaming and of the resident form))."""
    f, clocks = _int(0), (ctypes.c_double * 2)()
    _check(_lib.amq_selftest_product_plan(m, n, k_w, k_a, batch, m if ldy is None else ldy, sm_count, ctypes.byref(f), clocks))
    return f.value, tuple(clocks)


PRODUCT_CUDA_CORES, PRODUCT_STREAMING, PRODUCT_RESIDENT = 0, 1, 2


def selftest_binary_gemm(Wcodes, Walpha, xcodes, xbeta, n, form, bias=None, y=None):
    """Test aid: binary_gemm on a given kernel (see amq.h)."""
    m, k_w, _ = Wcodes.shape
    batch, k_a, _ = xcodes.shape
    y = _native.empty(Wcodes, 0, batch, m) if y is None else y
    _check(_native.amq_selftest_binary_gemm(Wcodes, Walpha, m, n, k_w, xcodes, xbeta, batch, k_a, bias, y.data_ptr(),
                                            y.stride(0) if batch > 1 else max(m, y.stride(0)), form))
    return y


def selftest_batched_sequence(Wcodes, Walpha, bias, I, H, x_seq, h0, c0, k_a, T, workspace, form, counted=0, late=0):
    """Test aid: a batched sequence (LSTM, or GRU when c0 is None) in a given form, its progress counters starting as after `counted`
    timesteps, its waits running out with `late` (see amq.h).  Returns (h_seq, h_last, c_last or None)."""
    steps, batch, k_w, gru = x_seq.shape[0], h0.shape[0], Wcodes.shape[1], c0 is None
    h_seq = _native.empty(h0, 0, steps, batch, H)
    h_last, c_last = torch.zeros_like(h0), None if gru else torch.zeros_like(c0)
    _check(_native.amq_selftest_batched_sequence(Wcodes, Walpha, bias, I, H, k_w, int(gru), x_seq, steps, h0, c0, batch, k_a, T,
                                                 h_seq, h_last, c_last, workspace, workspace.numel(), form, counted, late))
    return h_seq, h_last, c_last


def gru_sequence(Wcodes, Walpha, bias, I, H, x_seq, h0, k_a, T, workspace, want_h_seq=False,
                 h_seq=None, h_last=None):
    steps, batch, k_w = x_seq.shape[0], h0.shape[0], Wcodes.shape[1]
    if want_h_seq and h_seq is None:
        h_seq = _native.empty(h0, 0, steps, batch, H)
    h_last = _native.empty(h0, 0, *h0.shape) if h_last is None else h_last
    _check(_native.amq_gru_sequence(Wcodes, Walpha, bias, I, H, k_w, x_seq, steps, h0,
                                 batch, k_a, T, h_seq, h_last, workspace, workspace.numel()))
    return h_seq, h_last


def _host(t, name):
    if t is None:
        return None
    if not (isinstance(t, torch.Tensor) and not t.is_cuda and t.dtype == torch.float32 and t.is_contiguous()):
        raise TypeError("%s must be a contiguous CPU fp32 tensor" % name)
    return t


def lstm_sequence_host(Wcodes, Walpha, bias, I, H, x_seq, h0, c0, k_a, T, workspace, staging,
                       h_last, c_last, h_seq=None):
    """x_seq, h0, c0, h_last, c_last, h_seq are HOST tensors (pinned for asynchronous copies)."""
    x_seq, h0, c0 = _host(x_seq, "x_seq"), _host(h0, "h0"), _host(c0, "c0")
    steps, batch, k_w = x_seq.shape[0], h0.shape[0], Wcodes.shape[1]
    _check(_native.amq_lstm_sequence_host(Wcodes, Walpha, bias, I, H, k_w, _ptr(x_seq), steps,
                                       _ptr(h0), _ptr(c0), batch, k_a, T, _ptr(_host(h_seq, "h_seq")),
                                       _ptr(_host(h_last, "h_last")), _ptr(_host(c_last, "c_last")),
                                       workspace, workspace.numel(), staging, staging.numel()))
    return h_seq, h_last, c_last


def gru_sequence_host(Wcodes, Walpha, bias, I, H, x_seq, h0, k_a, T, workspace, staging, h_last, h_seq=None):
    x_seq, h0 = _host(x_seq, "x_seq"), _host(h0, "h0")
    steps, batch, k_w = x_seq.shape[0], h0.shape[0], Wcodes.shape[1]
    _check(_native.amq_gru_sequence_host(Wcodes, Walpha, bias, I, H, k_w, _ptr(x_seq), steps,
                                      _ptr(h0), batch, k_a, T, _ptr(_host(h_seq, "h_seq")),
                                      _ptr(_host(h_last, "h_last")), workspace, workspace.numel(),
                                      staging, staging.numel()))
    return h_seq, h_last


def workspace_status(workspace):
    return _lib.amq_workspace_status(_ptr(workspace), _stream())


def embedding_rows(We_codes, We_alpha, n, tokens):
    """Rows of the quantized embedding matrix for int32 token ids of any shape -> codes (*shape, k, wpr), coeffs (*shape, k)."""
    vocab, k, wpr = We_codes.shape
    xcodes = torch.empty(tuple(tokens.shape) + (k, wpr), dtype=torch.int32, device=We_codes.device)
    xbeta = torch.empty(tuple(tokens.shape) + (k,), dtype=torch.float32, device=We_codes.device)
    _check(_native.amq_embedding_rows(We_codes, We_alpha, vocab, n, k, tokens, tokens.numel(),
                                   xcodes, xbeta))
    return xcodes, xbeta


def new_paper_workspace(H, batch, steps, k_a, device="cuda"):
    return torch.empty(max(_lib.amq_lstm_paper_workspace_bytes(H, batch, steps, k_a), 16), dtype=torch.uint8, device=device)


def lstm_step_paper(Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, I, H, xcodes, xbeta, h_in, c_in, k_a, T, workspace,
                    h_out=None, c_out=None):
    batch, k_w, k_e = h_in.shape[0], Wi_codes.shape[1], xcodes.shape[-2]
    h_out = _native.empty(h_in, 0, *h_in.shape) if h_out is None else h_out
    c_out = _native.empty(c_in, 0, *c_in.shape) if c_out is None else c_out
    _check(_native.amq_lstm_step_paper(Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, I, H, k_w,
                                    xcodes, xbeta, k_e, h_in, c_in, batch, k_a, T,
                                    h_out, c_out, workspace, workspace.numel()))
    return h_out, c_out


def lstm_sequence_paper(Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, I, H, xcodes_seq, xbeta_seq, h0, c0, k_a, T, workspace,
                        want_h_seq=False, h_last=None, c_last=None):
    steps, batch, k_e = xcodes_seq.shape[0], h0.shape[0], xcodes_seq.shape[-2]
    k_w = Wi_codes.shape[1]
    h_seq = _native.empty(h0, 0, steps, batch, H) if want_h_seq else None
    h_last = _native.empty(h0, 0, *h0.shape) if h_last is None else h_last
    c_last = _native.empty(c0, 0, *c0.shape) if c_last is None else c_last
    _check(_native.amq_lstm_sequence_paper(Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, I, H, k_w,
                                        xcodes_seq, xbeta_seq, k_e, steps, h0, c0, batch, k_a, T,
                                        h_seq, h_last, c_last, workspace, workspace.numel()))
    return h_seq, h_last, c_last


def log_softmax_argmax(logits, want_logp=True, argmax=None):
    """logits (rows, n) fp32, rows contiguous (any row stride) -> (log-probabilities (rows, n) or None, argmax (rows,) int32)."""
    if not (isinstance(logits, torch.Tensor) and logits.is_cuda and logits.dtype == torch.float32 and logits.dim() == 2
            and (logits.shape[1] == 1 or logits.stride(1) == 1)):
        raise TypeError("logits must be a 2-D CUDA float32 tensor with contiguous rows")
    rows, n = logits.shape
    ld = logits.stride(0) if rows > 1 else max(n, logits.stride(0))
    logp = _native.empty(logits, 0, rows, n) if want_logp else None
    argmax = _native.empty(logits, 1, rows) if argmax is None else argmax
    _check(_native.amq_log_softmax_argmax(logits.data_ptr(), rows, n, ld, logp, n, argmax))
    return logp, argmax


def new_decode_workspace(vocab, I, H, k_e, k_a, device="cuda"):
    return torch.empty((_lib.amq_lm_decode_workspace_bytes(vocab, I, H, k_e, k_a),), dtype=torch.uint8, device=device)


def lm_greedy_decode(We_codes, We_alpha, Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, Ws_codes, Ws_alpha, bias_s, I, H,
                     k_a, T, tokens, h, c, workspace, logp=None):
    """tokens: int32 (steps + 1,), tokens[0] given, the rest written; h, c: (H,) or (1, H) fp32, updated in place."""
    vocab, k_e = We_codes.shape[0], We_codes.shape[1]
    k_w, k_s = Wi_codes.shape[1], Ws_codes.shape[1]
    steps = tokens.numel() - 1
    _check(_native.amq_lm_greedy_decode(We_codes, We_alpha, vocab, I, k_e, Wi_codes, Wi_alpha,
                                     Wh_codes, Wh_alpha, bias, H, k_w, Ws_codes, Ws_alpha,
                                     bias_s, k_s, k_a, T, tokens, steps, h, c, logp,
                                     workspace, workspace.numel()))
    return tokens


def selftest_decode_give_up(We_codes, We_alpha, Wi_codes, Wi_alpha, Wh_codes, Wh_alpha, bias, Ws_codes, Ws_alpha, bias_s, I, H,
                            k_a, T, tokens, h, c, workspace, late):
    """Test aid: lm_greedy_decode in one launch with waits that run out (see amq.h); read the outcome with device_status."""
    _check(_native.amq_selftest_decode_give_up(We_codes, We_alpha, We_codes.shape[0], I, We_codes.shape[1], Wi_codes, Wi_alpha,
                                               Wh_codes, Wh_alpha, bias, H, Wi_codes.shape[1], Ws_codes, Ws_alpha, bias_s,
                                               Ws_codes.shape[1], k_a, T, tokens, tokens.numel() - 1, h, c, workspace,
                                               workspace.numel(), late))


METHOD_ALTERNATING, METHOD_REFINED_GREEDY = 0, 1


def quantize_variant(x, k, T, method=METHOD_ALTERNATING, final_refit=False):
    """As quantize, with the method (alternating / refined greedy) and an optional last coefficient refit."""
    if not (x.is_cuda and x.dtype == torch.float32 and x.dim() == 2 and x.stride(1) == 1):
        raise TypeError("x must be a 2-D CUDA fp32 tensor with unit column stride")
    rows, n = x.shape
    ldx = x.stride(0) if rows > 1 else max(n, x.stride(0))
    codes = _new_codes(rows, k, n, x)
    coeffs = _native.empty(x, 0, rows, k)
    _check(_native.amq_quantize_variant(x.data_ptr(), rows, n, ldx, k, T, method, int(final_refit), codes, coeffs))
    return codes, coeffs


def gru_step_original(Wcodes, Walpha, bias, I, H, x, h_in, k_a, T, workspace=None, h_out=None):
    """The GRU in its original form (reset gate applied to h before the candidate's product); bias (3H,) or None."""
    batch, k_w = h_in.shape[0], Wcodes.shape[1]
    if workspace is None:
        workspace = torch.empty((_lib.amq_gru_original_workspace_bytes(I, H, batch, k_a),), dtype=torch.uint8, device=h_in.device)
    h_out = _native.empty(h_in, 0, *h_in.shape) if h_out is None else h_out
    _check(_native.amq_gru_step_original(Wcodes, Walpha, bias, I, H, k_w, x, h_in, batch, k_a, T,
                                      h_out, workspace, workspace.numel()))
    return h_out
