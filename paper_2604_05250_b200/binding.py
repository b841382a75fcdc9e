"""Thin ctypes binding of ``include/dualdiff.h``: argument marshalling only.

Every function takes torch tensors (device memory for the plain calls, pinned
host memory for the ``*_host`` calls), passes their data pointers and sizes
through the C ABI, and raises ``DualDiffError`` on a non-zero status.  There is
no Python or CPU implementation behind these names: if ``libdualdiff.so`` is
missing the first call raises.
"""
from __future__ import annotations

import ctypes
import importlib.util
import os

import torch
from torch import Tensor

from .build import host_path

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libdualdiff.so")

DD_OK, DD_ERR_INVALID_ARG, DD_ERR_UNSUPPORTED, DD_ERR_CUDA, DD_ERR_TIMEOUT = 0, -1, -2, -3, -4
DD_MODE_TRUST, DD_MODE_KL, DD_MODE_CONF = 0, 1, 2
DD_FLAG_PROBABILISTIC, DD_FLAG_EMIT_DRAFTER = 0x100, 0x200
DD_LAYOUT_BHND, DD_LAYOUT_BNHD = 0, 1

# every symbol include/dualdiff.h declares
EXPORTS = (
    "dd_bidir_attention", "dd_block_attention", "dd_verify", "dd_unmask", "dd_bidir_attention_host", "dd_verify_host", "dd_verify_static",
    "dd_verify_workspace_bytes", "dd_attention_status", "dd_verify_status", "dd_launch_count", "dd_release",
    "dd_status_string", "dd_last_cuda_error", "dd_version", "dd_debug_set_max_ctas", "dd_clear_status", "dd_debug_expire_wait", "dd_lm_head_verify",
)


class DualDiffError(RuntimeError):
    def __init__(self, status: int, text: str):
        super().__init__(f"dualdiff status {status}: {text}")
        self.status = status


_lib = None


def lib() -> ctypes.CDLL:
    """Loads libdualdiff.so (once).  Raises if it has not been built."""
    global _lib
    if _lib is None:
        _lib = load(LIB_PATH)
    return _lib


class use_library:
    """Context manager: the wrappers below call the library at `path` (for instance the
    bounds-checked build) instead of libdualdiff.so until the block ends."""

    def __init__(self, path):
        self.path = path

    def __enter__(self):
        global _lib
        self.saved = _lib
        _lib = load(self.path)
        return _lib

    def __exit__(self, *exc):
        global _lib
        _lib = self.saved
        return False


def load(path) -> ctypes.CDLL:
    """Loads one build of the library and declares its entry points."""
    if True:
        if not os.path.exists(path):
            raise RuntimeError(
                f"{path} is missing: build it with `python -m paper_2604_05250_b200.build`; "
                "there is no fallback implementation")
        L = ctypes.CDLL(path)
        vp, i32, f32, u64 = ctypes.c_void_p, ctypes.c_int, ctypes.c_float, ctypes.c_uint64
        attn = [vp, vp, vp, vp, i32, i32, i32, i32, f32, vp]
        ver = [vp, vp, vp, vp, i32, f32, i32, u64, vp, vp, vp, i32, i32, i32, vp]
        L.dd_bidir_attention.argtypes = attn
        L.dd_bidir_attention_host.argtypes = attn
        L.dd_block_attention.argtypes = [vp, vp, vp, vp, i32, i32, i32, i32, i32, vp, i32, f32, vp]
        L.dd_block_attention.restype = i32
        L.dd_verify.argtypes = ver
        L.dd_verify_host.argtypes = ver
        L.dd_verify_static.argtypes = ver
        L.dd_unmask.argtypes = [vp, vp, vp, f32, i32, vp, vp, vp, i32, i32, i32, vp]
        L.dd_unmask.restype = i32
        L.dd_verify_static.restype = i32
        for name in ("dd_bidir_attention", "dd_bidir_attention_host", "dd_verify", "dd_verify_host",
                     "dd_attention_status", "dd_verify_status", "dd_release", "dd_version"):
            getattr(L, name).restype = i32
        L.dd_attention_status.argtypes = []
        L.dd_verify_status.argtypes = []
        L.dd_release.argtypes = []
        L.dd_version.argtypes = []
        L.dd_verify_workspace_bytes.argtypes = [i32, i32, i32]
        L.dd_verify_workspace_bytes.restype = ctypes.c_size_t
        L.dd_launch_count.argtypes = []
        L.dd_launch_count.restype = u64
        L.dd_lm_head_verify.argtypes = [vp, vp, vp, vp, vp, vp, i32, f32, i32, u64, vp, vp, vp, i32, i32, i32, i32, vp]
        L.dd_lm_head_verify.restype = i32
        L.dd_clear_status.argtypes = []
        L.dd_clear_status.restype = i32
        L.dd_debug_expire_wait.argtypes = [i32, vp]
        L.dd_debug_expire_wait.restype = i32
        L.dd_debug_set_max_ctas.argtypes = [i32]
        L.dd_debug_set_max_ctas.restype = i32
        L.dd_status_string.argtypes = [i32]
        L.dd_status_string.restype = ctypes.c_char_p
        L.dd_last_cuda_error.argtypes = []
        L.dd_last_cuda_error.restype = ctypes.c_char_p
    return L


_fast = None        # the native form of the wrappers below (csrc/host_call.cpp); None: the Python form serves every call


def load_native():
    """Loads the native form if it has been built for this Python and torch; build.build() calls it again."""
    global _fast
    path = host_path()
    if _fast is None and os.path.exists(path):
        name = __package__ + "._host_call"
        spec = importlib.util.spec_from_file_location(name, path)
        try:
            module = importlib.util.module_from_spec(spec)
            spec.loader.exec_module(module)
        except ImportError:
            return
        _fast = module


load_native()


def _addresses(L):
    """Addresses of the entry points that _fast calls, looked up once per library."""
    try:
        return L._dd_addresses
    except AttributeError:
        L._dd_addresses = {name: ctypes.cast(getattr(L, name), ctypes.c_void_p).value
                           for name in ("dd_bidir_attention", "dd_block_attention", "dd_verify", "dd_verify_static", "dd_unmask")}
        return L._dd_addresses


def _check(status: int):
    if status != DD_OK:
        L = lib()
        text = L.dd_status_string(status).decode()
        if status == DD_ERR_CUDA:
            text += ": " + L.dd_last_cuda_error().decode()
        raise DualDiffError(status, text)


# A call on small tensors is bound by what happens here, so the wrappers below check all tensors in one
# expression and only go through _require, which words the error, when something is wrong; addresses and
# the stream are passed as plain integers, and outputs are made like an input of the same shape.
# (dd_verify on the tiny workload, host side of a call: 23.2 us at first, 12.9 so; attention 14.9 and 8.3.)
# Calls on device tensors on the current stream go through _fast, which does the same natively (5.7 us, the
# launch itself included) and returns None for whatever it does not take, so that every error is worded here.

_BF16, _I32, _U8, _F32 = torch.bfloat16, torch.int32, torch.uint8, torch.float32
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)
_device = getattr(torch._C, "_cuda_getDevice", None)


def _stream_ptr(stream):
    """The given stream, or the current stream of the current device, as an integer."""
    if stream is not None:
        return stream.cuda_stream
    if _raw_stream is None or _device is None or not torch.cuda.is_initialized():
        return torch.cuda.current_stream().cuda_stream
    return _raw_stream(_device())


def _ptr(t):
    return None if t is None else t.data_ptr()


def _fits(t, dtype, shape, cuda):
    return isinstance(t, Tensor) and t.dtype is dtype and t.shape == shape and t.is_cuda is cuda and t.is_contiguous()


def _require(t, dtype, shape, cuda, name):
    if not isinstance(t, Tensor):
        raise TypeError(f"{name}: expected a torch.Tensor")
    if t.dtype != dtype or tuple(t.shape) != tuple(shape) or not t.is_contiguous():
        raise ValueError(f"{name}: expected contiguous {dtype} of shape {tuple(shape)}, "
                         f"got {t.dtype} {tuple(t.shape)}")
    if t.is_cuda != cuda:
        raise ValueError(f"{name}: expected a {'device' if cuda else 'host'} tensor")


def bidir_attention(q, k, v, out=None, scale=None, stream=None, host=False):
    """dd_bidir_attention (dd_bidir_attention_host if host=True).

    q, k, v: [B,H,N,D] torch.bfloat16.  Returns out (allocated if None)."""
    if _fast is not None and stream is None and not host:
        r = _fast.attention(_addresses(_lib or lib())["dd_bidir_attention"], q, k, v, out, scale)
        if r is not None:
            if type(r) is int:
                _check(r)
            return r
    shape = q.shape
    B, H, N, D = shape
    cuda = not host
    if not (_fits(q, _BF16, shape, cuda) and _fits(k, _BF16, shape, cuda) and _fits(v, _BF16, shape, cuda)):
        for name, t in (("q", q), ("k", k), ("v", v)):
            _require(t, _BF16, (B, H, N, D), cuda, name)
    if out is None:
        out = torch.empty_like(q)
    elif not _fits(out, _BF16, shape, cuda):
        _require(out, _BF16, (B, H, N, D), cuda, "out")
    if scale is None:
        scale = float(D) ** -0.5
    L = _lib or lib()
    fn = L.dd_bidir_attention_host if host else L.dd_bidir_attention
    status = fn(q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), B, H, N, D, float(scale), _stream_ptr(stream))
    if status:
        _check(status)
    return out


def block_attention(q, k, v, kv_len=None, layout="bhnd", out=None, scale=None, stream=None):
    """dd_block_attention: a block of Nq queries over Nkv stored keys and values.

    layout "bhnd": q [B,H,Nq,D], k, v [B,H,Nkv,D]; "bnhd": q [B,Nq,H,D], k, v [B,Nkv,H,D];
    torch.bfloat16 device tensors.  kv_len: int32 [B] device tensor (valid keys per sequence)
    or None.  Returns out (allocated if None), in the layout of q."""
    if _fast is not None and stream is None and (layout == "bhnd" or layout == "bnhd"):
        r = _fast.block(_addresses(_lib or lib())["dd_block_attention"], q, k, v, kv_len,
                        DD_LAYOUT_BHND if layout == "bhnd" else DD_LAYOUT_BNHD, out, scale)
        if r is not None:
            if type(r) is int:
                _check(r)
            return r
    shape = q.shape
    if layout == "bhnd":
        B, H, Nq, D = shape
        Nkv = k.shape[2]
        kshape = (B, H, Nkv, D)
    elif layout == "bnhd":
        B, Nq, H, D = shape
        Nkv = k.shape[1]
        kshape = (B, Nkv, H, D)
    else:
        raise ValueError("layout: 'bhnd' or 'bnhd'")
    if not (_fits(q, _BF16, shape, True) and _fits(k, _BF16, kshape, True) and _fits(v, _BF16, kshape, True)):
        _require(q, _BF16, tuple(shape), True, "q")
        _require(k, _BF16, kshape, True, "k")
        _require(v, _BF16, kshape, True, "v")
    if kv_len is not None and not _fits(kv_len, _I32, (B,), True):
        _require(kv_len, _I32, (B,), True, "kv_len")
    if out is None:
        out = torch.empty_like(q)
    elif not _fits(out, _BF16, shape, True):
        _require(out, _BF16, tuple(shape), True, "out")
    if scale is None:
        scale = float(D) ** -0.5
    status = (_lib or lib()).dd_block_attention(
        q.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), B, H, Nq, Nkv, D, _ptr(kv_len),
        DD_LAYOUT_BHND if layout == "bhnd" else DD_LAYOUT_BNHD, float(scale), _stream_ptr(stream))
    if status:
        _check(status)
    return out


def _decision_inputs(tokens, mask_flags, shape, cuda):
    if not (_fits(tokens, _I32, shape, cuda) and _fits(mask_flags, _U8, shape, cuda)):
        _require(tokens, _I32, shape, cuda, "tokens")
        _require(mask_flags, _U8, shape, cuda, "mask_flags")


def _decision_outputs(out_tokens, out_mask, out_score, want_score, tokens, mask_flags, like, shape, host, score_name):
    """The three outputs of shape [B,P]: made where they are None, checked where they are given."""
    cuda = not host
    near = cuda and tokens.device == like.device and mask_flags.device == like.device

    def make(source, dtype):
        return torch.empty_like(source, dtype=dtype) if near else torch.empty(shape, dtype=dtype, device=like.device, pin_memory=host)

    if out_tokens is None:
        out_tokens = torch.empty_like(tokens) if near else make(tokens, _I32)
    elif not _fits(out_tokens, _I32, shape, cuda):
        _require(out_tokens, _I32, shape, cuda, "out_tokens")
    if out_mask is None:
        out_mask = torch.empty_like(mask_flags) if near else make(mask_flags, _U8)
    elif not _fits(out_mask, _U8, shape, cuda):
        _require(out_mask, _U8, shape, cuda, "out_mask")
    if out_score is None:
        if want_score:
            out_score = make(tokens, _F32)
    elif not _fits(out_score, _F32, shape, cuda):
        _require(out_score, _F32, shape, cuda, score_name)
    return out_tokens, out_mask, out_score


def verify(drafter_logits, verifier_logits, tokens, mask_flags, mode, tau, k, seed,
           out_tokens=None, out_mask=None, out_score=None, want_score=True, stream=None, host=False,
           static_scratch=False):
    """dd_verify (dd_verify_host if host=True; dd_verify_static, the variant that allocates
    nothing, if static_scratch=True and every output tensor is passed in).

    Returns (out_tokens int32 [B,P], out_mask uint8 [B,P], out_score float32 [B,P] or None)."""
    if _fast is not None and stream is None and not host:
        r = _fast.verify(_addresses(_lib or lib())["dd_verify_static" if static_scratch else "dd_verify"], drafter_logits,
                         verifier_logits, tokens, mask_flags, mode, tau, k, seed, out_tokens, out_mask, out_score, want_score)
        if r is not None:
            if type(r) is int:
                _check(r)
            return r
    B, P, V = full = verifier_logits.shape
    cuda = not host
    if not _fits(verifier_logits, _BF16, full, cuda):
        _require(verifier_logits, _BF16, (B, P, V), cuda, "verifier_logits")
    if drafter_logits is not None and not _fits(drafter_logits, _BF16, full, cuda):
        _require(drafter_logits, _BF16, (B, P, V), cuda, "drafter_logits")
    shape = (B, P)
    _decision_inputs(tokens, mask_flags, shape, cuda)
    out_tokens, out_mask, out_score = _decision_outputs(out_tokens, out_mask, out_score, want_score, tokens, mask_flags,
                                                        verifier_logits, shape, host, "out_score")
    L = _lib or lib()
    fn = L.dd_verify_host if host else (L.dd_verify_static if static_scratch else L.dd_verify)
    status = fn(_ptr(drafter_logits), verifier_logits.data_ptr(), tokens.data_ptr(), mask_flags.data_ptr(),
                int(mode), float(tau), int(k), int(seed) & 0xFFFFFFFFFFFFFFFF,
                out_tokens.data_ptr(), out_mask.data_ptr(), _ptr(out_score), B, P, V, _stream_ptr(stream))
    if status:
        _check(status)
    return out_tokens, out_mask, out_score


def lm_head_verify(drafter_hidden, drafter_weight, verifier_hidden, verifier_weight, tokens, mask_flags,
                   mode, tau, k, seed, out_tokens=None, out_mask=None, out_score=None, stream=None):
    """dd_lm_head_verify: the language-model heads fused with the verification algorithm.

    verifier_hidden [B,P,K], verifier_weight [V,K]: torch.bfloat16 device tensors; drafter_hidden,
    drafter_weight: the same shapes, or None in the modes that need the verifier only.
    Returns (out_tokens int32 [B,P], out_mask uint8 [B,P], out_score float32 [B,P])."""
    B, P, K = verifier_hidden.shape
    V = verifier_weight.shape[0]
    if drafter_hidden is not None:
        _require(drafter_hidden, _BF16, (B, P, K), True, "drafter_hidden")
    if drafter_weight is not None:
        _require(drafter_weight, _BF16, (V, K), True, "drafter_weight")
    _require(verifier_hidden, _BF16, (B, P, K), True, "verifier_hidden")
    _require(verifier_weight, _BF16, (V, K), True, "verifier_weight")
    shape = (B, P)
    _decision_inputs(tokens, mask_flags, shape, True)
    out_tokens, out_mask, out_score = _decision_outputs(out_tokens, out_mask, out_score, True, tokens, mask_flags,
                                                        verifier_hidden, shape, False, "out_score")
    status = (_lib or lib()).dd_lm_head_verify(
        _ptr(drafter_hidden), _ptr(drafter_weight), verifier_hidden.data_ptr(), verifier_weight.data_ptr(),
        tokens.data_ptr(), mask_flags.data_ptr(), int(mode), float(tau), int(k), int(seed) & 0xFFFFFFFFFFFFFFFF,
        out_tokens.data_ptr(), out_mask.data_ptr(), out_score.data_ptr(), B, P, K, V, _stream_ptr(stream))
    if status:
        _check(status)
    return out_tokens, out_mask, out_score


def unmask(logits, tokens, mask_flags, tau, k, out_tokens=None, out_mask=None, out_conf=None, stream=None):
    """dd_unmask: one confidence-based unmasking step on logits [B,P,V] (device tensors).

    Returns (out_tokens int32 [B,P], out_mask uint8 [B,P] with 1 = still masked, out_conf float32 [B,P])."""
    if _fast is not None and stream is None:
        r = _fast.unmask(_addresses(_lib or lib())["dd_unmask"], logits, tokens, mask_flags, tau, k, out_tokens, out_mask, out_conf)
        if r is not None:
            if type(r) is int:
                _check(r)
            return r
    B, P, V = full = logits.shape
    if not _fits(logits, _BF16, full, True):
        _require(logits, _BF16, (B, P, V), True, "logits")
    shape = (B, P)
    _decision_inputs(tokens, mask_flags, shape, True)
    out_tokens, out_mask, out_conf = _decision_outputs(out_tokens, out_mask, out_conf, True, tokens, mask_flags,
                                                       logits, shape, False, "out_conf")
    status = (_lib or lib()).dd_unmask(logits.data_ptr(), tokens.data_ptr(), mask_flags.data_ptr(), float(tau), int(k),
                                       out_tokens.data_ptr(), out_mask.data_ptr(), out_conf.data_ptr(), B, P, V,
                                       _stream_ptr(stream))
    if status:
        _check(status)
    return out_tokens, out_mask, out_conf


def attention_status() -> int:
    return int(lib().dd_attention_status())


def verify_status() -> int:
    return int(lib().dd_verify_status())


def launch_count() -> int:
    return int(lib().dd_launch_count())


def debug_set_max_ctas(n: int):
    """Test hook: cap the grid of the streaming verify kernel (0 = no cap)."""
    _check(lib().dd_debug_set_max_ctas(int(n)))


def clear_status():
    """Re-arms the kernels' health words on the current device after a recorded timeout."""
    _check(lib().dd_clear_status())


def debug_expire_wait(which: int, stream=None):
    """Test hook: records an expired wait for the attention kernel (0) or dd_verify (1)."""
    _check(lib().dd_debug_expire_wait(int(which), _stream_ptr(stream)))


def release():
    _check(lib().dd_release())


def version() -> int:
    return int(lib().dd_version())


def verify_workspace_bytes(B, P, V) -> int:
    return int(lib().dd_verify_workspace_bytes(B, P, V))
