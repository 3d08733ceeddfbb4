"""ctypes binding of the decoder's kernels (``libsplice_decoder.so``).

``model.py`` calls these in place of the torch expressions next to them
whenever nothing but the values is asked for (``plain``): eager CUDA tensors
of the decoder's own types, with no gradient, transform, mode or autocast that
would have to see the single operations.  Every launch goes to torch's current
stream, and every output is allocated here.
"""
from __future__ import annotations

import ctypes
import os
import threading

import torch
import torch.autograd.forward_ad as _fwad

_LIB = None
POSITIONS = {torch.int64: 0, torch.int32: 1, torch.float32: 2}
BF16, F32 = torch.bfloat16, torch.float32
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None) or (
    lambda device: torch.cuda.current_stream(device).cuda_stream)
_current_device = torch.cuda.current_device


def lib() -> ctypes.CDLL:
    global _LIB
    if _LIB is None:
        path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "libsplice_decoder.so")
        if not os.path.exists(path):
            raise RuntimeError(f"{path} is not built: run paper_2605_30574_gb300.build.build()")
        L = ctypes.CDLL(path)
        vp, i, l, f = ctypes.c_void_p, ctypes.c_int, ctypes.c_long, ctypes.c_float
        L.decoder_rms_norm.argtypes = [vp, vp, vp, l, i, f, vp]
        L.decoder_add_rms_norm.argtypes = [vp, vp, vp, vp, vp, l, i, f, vp]
        L.decoder_add.argtypes = [vp, vp, vp, l, vp]
        L.decoder_to_bf16.argtypes = [vp, vp, l, vp]
        L.decoder_silu_mul.argtypes = [vp, vp, l, vp, l, i, vp]
        L.decoder_qkv_post.argtypes = [vp, vp, vp, vp, vp, vp, ctypes.POINTER(l), vp, vp, vp, vp, i, l, i, i, i, f, vp]
        L.decoder_gemm.argtypes = [i, vp, vp, vp, vp, vp, i, i, i, vp]
        L.decoder_gemm_plan.argtypes = [i, i, i, i, ctypes.POINTER(i), ctypes.POINTER(l)]
        L.decoder_error.argtypes = [ctypes.POINTER(ctypes.c_uint)]
        L.decoder_scratch_bytes.argtypes = [i, l, i, i, i, i]
        L.decoder_scratch_bytes.restype = l
        L.decoder_qkv.argtypes = [vp] * 7 + [ctypes.POINTER(l), vp, vp, vp, vp, i, l, i, i, i, i, f, vp]
        L.decoder_block.argtypes = [vp, vp, i, vp, vp, vp, vp, vp, vp, vp, l, i, i, i, f, vp]
        L.decoder_causal.argtypes = [vp] * 4 + [l, i, i, i, f, vp]
        for fn in (L.decoder_qkv, L.decoder_block, L.decoder_causal, L.decoder_gemm, L.decoder_gemm_plan, L.decoder_error, L.decoder_rms_norm, L.decoder_add_rms_norm, L.decoder_add, L.decoder_to_bf16, L.decoder_silu_mul,
                   L.decoder_qkv_post):
            fn.restype = i
        _LIB = L
    return _LIB


def plain(acts, weights) -> bool:
    """Whether the kernels may stand in for the torch expressions on these
    activations and bf16 weights."""
    if torch.compiler.is_compiling():       # (first: a compiler cannot trace the rest)
        return False
    dev = acts[0].device
    if dev.type != "cuda" or dev.index != torch.cuda.current_device():
        return False
    if (torch._C._are_functorch_transforms_active() or torch._C._len_torch_dispatch_stack()
            or torch._C._len_torch_function_stack() or torch.is_autocast_enabled() or _fwad._current_level >= 0
            or torch.jit.is_tracing()):
        return False
    grad = torch.is_grad_enabled()
    for t in acts:
        if type(t) is not torch.Tensor or not _values(t, dev) or (grad and t.requires_grad):
            return False
    for t in weights:
        if t.dtype is not BF16 or type(t) not in (torch.Tensor, torch.nn.Parameter) or not _values(t, dev) \
                or (grad and t.requires_grad):
            return False
    return True


def _values(t, dev) -> bool:
    """Whether the tensor's values are what lies at its address: not those of a
    negated view, nor none (an empty tensor, one of zeros without memory)."""
    return t.device == dev and t.is_contiguous() and not t.is_neg() and t.numel() > 0 and t.data_ptr() != 0


def joined(*ws):
    """The matrices as one, when they are consecutive rows of one contiguous
    matrix (as the decoder lays them out), else None."""
    base = ws[0]._base
    if base is None or base.dim() != 2 or not base.is_contiguous() or base.dtype is not ws[0].dtype:
        return None
    at = base.data_ptr()
    for w in ws:
        if w._base is not base or w.data_ptr() != at or w.shape[1] != base.shape[1]:
            return None
        at += w.numel() * w.element_size()
    return base if sum(w.shape[0] for w in ws) == base.shape[0] else None


def _launch(name, *args):
    # (the raw handle of torch's current stream: a Stream object costs more
    # host time than the launch)
    rc = getattr(_LIB or lib(), name)(*args, _raw_stream(_current_device()))
    if rc != 0:
        raise RuntimeError(f"{name} failed with CUDA error {rc}")


def _rows(t):
    return t.numel() // t.shape[-1]


def _like(t, dtype):
    return torch.empty(t.shape, dtype=dtype, device=t.device)


def rms_norm(h, w, eps):
    """bf16(h / rms(h) * w) of fp32 rows."""
    x = _like(h, BF16)
    _launch("decoder_rms_norm", h.data_ptr(), w.data_ptr(), x.data_ptr(), _rows(h), h.shape[-1], eps)
    return x


def add_rms_norm(h, o, w, eps):
    """h + o and the bf16 norm of the sum."""
    h2, x = _like(h, F32), _like(h, BF16)
    _launch("decoder_add_rms_norm", h.data_ptr(), o.data_ptr(), w.data_ptr(), h2.data_ptr(), x.data_ptr(), _rows(h),
            h.shape[-1], eps)
    return h2, x


def add_(h, o):
    """h += o (o bf16)."""
    _launch("decoder_add", h.data_ptr(), o.data_ptr(), h.data_ptr(), h.numel())
    return h


def to_bf16(x):
    y = _like(x, BF16)
    _launch("decoder_to_bf16", x.data_ptr(), y.data_ptr(), x.numel())
    return y


def silu_mul(gate, up):
    """bf16(silu(gate) * up)."""
    f, y = gate.shape[-1], _like(gate, BF16)
    _launch("decoder_silu_mul", gate.data_ptr(), up.data_ptr(), f, y.data_ptr(), _rows(gate), f)
    return y


def silu_mul_joined(gate_up):
    """The same for rows that hold gate, then up."""
    f = gate_up.shape[-1] // 2
    y = torch.empty((*gate_up.shape[:-1], f), dtype=BF16, device=gate_up.device)
    p = gate_up.data_ptr()
    _launch("decoder_silu_mul", p, p + 2 * f, 2 * f, y.data_ptr(), _rows(y), f)
    return y


def qkv_post(q, k, v, strides, outs, out_strides, q_norm, k_norm, inv_freq, pos, hq, hkv, d, eps):
    """Per-head norm and RoPE of q and k, and v as it is.  q, k, v: pointers of
    the projections' rows, ``strides`` elements apart; outs: the three output
    pointers, with (row, head) strides each."""
    _launch("decoder_qkv_post", q, k, v, *outs, (ctypes.c_long * 9)(*strides, *out_strides), q_norm.data_ptr(),
            k_norm.data_ptr(), inv_freq.data_ptr(), pos.data_ptr(), POSITIONS[pos.dtype], pos.numel(), hq, hkv, d, eps)


# ---- a layer's halves in one call each ----

def _scratch(half, rows, D, nq, nqkv, f, device):
    """Device scratch of a half's call, None where the shape is not one for it."""
    n = (_LIB or lib()).decoder_scratch_bytes(half, rows, D, nq, nqkv, f)
    return torch.empty(n, dtype=torch.uint8, device=device) if n else None


def _aligned(*ts):
    for t in ts:
        if t.data_ptr() & 15:
            return False
    return True


def qkv(h, in_norm, wqkv, outs, out_strides, q_norm, k_norm, inv_freq, pos, hq, hkv, d, eps) -> bool:
    """Input norm, joined projection, per-head norm and RoPE, in one call.
    False, and nothing done, for the shapes it does not take."""
    rows, D = _rows(h), h.shape[-1]
    s = _scratch(0, rows, D, hq * d, wqkv.shape[0], 0, h.device) if _aligned(wqkv) else None
    if s is None:
        return False
    _launch("decoder_qkv", h.data_ptr(), in_norm.data_ptr(), wqkv.data_ptr(), s.data_ptr(), *outs,
            (ctypes.c_long * 6)(*out_strides), q_norm.data_ptr(), k_norm.data_ptr(), inv_freq.data_ptr(),
            pos.data_ptr(), POSITIONS[pos.dtype], rows, D, hq, hkv, d, eps)
    return True


def block(h, attn, wo, post_norm, w_gate, w_up, w_down, eps):
    """What follows a layer's attention, in one call: the residual stream after
    the layer, or None for the shapes it does not take."""
    rows, D, nq, f = _rows(h), h.shape[-1], wo.shape[1], w_gate.shape[0]
    s = _scratch(1, rows, D, nq, 0, f, h.device) if _aligned(attn, wo, w_gate, w_up, w_down) else None
    if s is None:
        return None
    out = torch.empty_like(h)
    _launch("decoder_block", h.data_ptr(), attn.data_ptr(), 1 if attn.dtype is BF16 else 0, wo.data_ptr(),
            post_norm.data_ptr(), w_gate.data_ptr(), w_up.data_ptr(), w_down.data_ptr(), s.data_ptr(), out.data_ptr(),
            rows, D, nq, f, eps)
    return out


def causal(q, k, v, scale):
    """Causal attention of q [T, Hq, d] over k, v [Hkv, T, d], bf16 and
    contiguous: [T, Hq, d] bf16; None for the shapes it does not take."""
    T, hq, d = q.shape
    hkv = k.shape[0]
    if T > 1 << 20 or d not in (64, 128, 256) or hq % hkv or not k.shape == v.shape == (hkv, T, d) or not _aligned(q, k, v):
        return None
    out = torch.empty_like(q)
    _launch("decoder_causal", q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), T, hq, hkv, d, scale)
    return out


# Up to this many rows the fused projections stream a large weight matrix faster
# than the library (151936 x 4096, fp32 out: 1 row 178 us against 205, 256 rows
# 224 against 237); with more, and two tiles of rows, they do not (320 rows 271
# against 257, 400 rows 320 against 298; of 151936 x 1024 108 against 97).  A
# small matrix is a question of host time, which the line does not look at: 4096
# x 1024 takes 27 us against 73 at any number of rows.
LOGITS_ROWS = 256


def logits(x, w):
    """x w^T in fp32, or None for the shapes it does not take."""
    rows, D = _rows(x), x.shape[-1]
    if rows > LOGITS_ROWS or D % 8 or w.shape[0] == 0 or not _aligned(x, w):
        return None
    y = torch.empty((*x.shape[:-1], w.shape[0]), dtype=torch.float32, device=x.device)
    _launch("decoder_gemm", 1, x.data_ptr(), w.data_ptr(), None, None, y.data_ptr(), rows, w.shape[0], D)
    return y


# The error word of a device is one for all its launches, and reading it clears
# it: what has been read is kept here, device by device, so that every reader
# sees it.
_records: dict = {}
_records_lock = threading.Lock()


class ErrorReader:
    """Whether a bounded wait of a launch on the current device ran out since the
    reader last asked (or was made, with ``fresh``; else ever): each reader is
    told once, whoever reads the word first, and also of others' launches,
    which the word does not tell apart."""

    def __init__(self, fresh: bool = True):
        self._seen = {}
        if fresh:
            self._take()

    def _take(self):
        """Synchronises the device, moves its word to the record and returns
        what this reader has not seen of it."""
        device, word = torch.cuda.current_device(), ctypes.c_uint()
        with _records_lock:
            record = _records.setdefault(device, [])
            rc = lib().decoder_error(ctypes.byref(word))
            if rc != 0:
                raise RuntimeError(f"decoder kernels: CUDA error {rc}")
            if word.value:
                record.append(word.value)
            at, self._seen[device] = self._seen.get(device, 0), len(record)
            return record[at:]

    def check(self):
        """Raises if one did; synchronises the device."""
        words = self._take()
        if words:
            raise RuntimeError("decoder kernels: error word " + ", ".join(f"0x{w:x}" for w in words))


_reader = ErrorReader(fresh=False)


def check_device_error():
    """The check of one reader that all callers of this function share."""
    _reader.check()
