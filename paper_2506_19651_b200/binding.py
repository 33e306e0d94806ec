"""Thin binding over the C ABI of libpevlm.so (include/pevlm.h), same names: the calls that launch work go through the
_pevlm_call module (csrc/pycall.c), the others through ctypes.

Argument marshalling only: every step of the path runs in the library's CUDA kernels.
Tensors are torch CUDA tensors (torch is used for device memory and streams); a call
enqueues work on torch's current stream and returns.  There is no CPU fallback: if the
library has not been built, `lib()` raises.
"""
from __future__ import annotations

import ctypes as C
import os
from dataclasses import dataclass

_DIR = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_DIR, "libpevlm.so")

PEVLM_OK = 0
PEVLM_EINVAL, PEVLM_EALIGN, PEVLM_EUNSUPPORTED, PEVLM_EWORKSPACE, PEVLM_ECUDA, PEVLM_ETIMEOUT = -1, -2, -3, -4, -5, -6
MASK_PEVLM, MASK_FULL_CAUSAL = 0, 1
WS_PREFILL, WS_QUERY = 0, 1

NOALLOC_SCRATCH_BYTES = 32 << 20

EXPORTS = ["pevlm_rope_qk", "pevlm_rope_qkv", "pevlm_layer_forward", "pevlm_rope_qk_mrope", "pevlm_parallel_prefill_attn", "pevlm_block_attn", "pevlm_assemble_kv", "pevlm_query_attn",
           "pevlm_query_attn_noalloc",
           "pevlm_workspace_bytes", "pevlm_read_status", "pevlm_selftest_wait_expiry", "pevlm_tile_stats", "pevlm_strerror",
           "pevlm_last_cuda_error"]


class Shape(C.Structure):
    """pevlm_shape_t"""
    _fields_ = [("batch", C.c_int32), ("sink_len", C.c_int32), ("block_len", C.c_int32),
                ("num_blocks", C.c_int32), ("query_len", C.c_int32), ("num_q_heads", C.c_int32),
                ("num_kv_heads", C.c_int32), ("head_dim", C.c_int32), ("rope_theta", C.c_float),
                ("softmax_scale", C.c_float), ("mask_mode", C.c_int32)]

    @property
    def n_video(self):
        return self.sink_len + self.num_blocks * self.block_len

    @property
    def L(self):
        return self.n_video + self.query_len


def make_shape(S, B, N, Q, Hq, Hkv, d, theta=1e4, scale=0.0, mask_mode=MASK_PEVLM, batch=1) -> Shape:
    return Shape(batch, S, B, N, Q, Hq, Hkv, d, theta, scale, mask_mode)


class PevlmError(RuntimeError):
    def __init__(self, code, where):
        self.code = code
        text = lib().pevlm_strerror(code).decode()
        extra = lib().pevlm_last_cuda_error().decode() if code == PEVLM_ECUDA else ""
        super().__init__(f"{where}: {text} ({code}) {extra}".strip())


_lib = None


def lib():
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(f"{LIB_PATH} is missing: build it with `python -m paper_2506_19651_b200.build` "
                               "(there is no CPU fallback)")
        l = C.CDLL(LIB_PATH)
        vp, sp = C.c_void_p, C.POINTER(Shape)
        l.pevlm_rope_qk.argtypes = [sp, vp, vp, vp, vp, C.c_int64, C.c_int64, vp, vp]
        l.pevlm_rope_qkv.argtypes = [sp, vp, vp, vp, vp, vp, vp, C.c_int64, C.c_int64, vp, vp]
        l.pevlm_rope_qkv.restype = C.c_int
        l.pevlm_layer_forward.argtypes = [sp, C.c_int32] + [vp] * 11 + [vp, C.c_size_t, vp, C.c_size_t, vp]
        l.pevlm_layer_forward.restype = C.c_int
        l.pevlm_rope_qk_mrope.argtypes = [sp, vp, vp, vp, vp, C.c_int64, vp, C.POINTER(C.c_int32), vp]
        l.pevlm_rope_qk_mrope.restype = C.c_int
        l.pevlm_parallel_prefill_attn.argtypes = [sp, vp, vp, vp, vp, vp, vp, C.c_size_t, vp]
        l.pevlm_block_attn.argtypes = [sp, vp, vp, vp, C.c_int64, C.c_int64, vp, vp, vp, C.c_size_t, vp]
        l.pevlm_block_attn.restype = C.c_int
        l.pevlm_assemble_kv.argtypes = [sp, vp, vp, vp, vp, vp, vp, vp]
        l.pevlm_query_attn.argtypes = [sp, vp, vp, vp, vp, vp, vp, C.c_size_t, vp]
        l.pevlm_query_attn_noalloc.argtypes = [sp, vp, vp, vp, vp, vp, vp]
        l.pevlm_query_attn_noalloc.restype = C.c_int
        l.pevlm_workspace_bytes.argtypes = [sp, C.c_int]
        l.pevlm_workspace_bytes.restype = C.c_size_t
        l.pevlm_read_status.argtypes = [vp, vp, C.POINTER(C.c_int32), C.POINTER(C.c_int32)]
        l.pevlm_selftest_wait_expiry.argtypes = [vp, C.c_size_t, C.c_int64, vp]
        l.pevlm_selftest_wait_expiry.restype = C.c_int
        l.pevlm_tile_stats.argtypes = [sp, C.c_int, C.POINTER(C.c_int64), C.POINTER(C.c_double)]
        l.pevlm_strerror.argtypes = [C.c_int]
        l.pevlm_strerror.restype = C.c_char_p
        l.pevlm_last_cuda_error.restype = C.c_char_p
        for name in ("pevlm_rope_qk", "pevlm_parallel_prefill_attn", "pevlm_assemble_kv", "pevlm_query_attn",
                     "pevlm_read_status", "pevlm_tile_stats"):
            getattr(l, name).restype = C.c_int
        _lib = l
    return _lib


def _ptr(t):
    return None if t is None else t.data_ptr()


_calls = None


def _native():
    """The module with the library's calls.  A missing library raises as in lib()."""
    global _calls
    if _calls is None:
        lib()
        try:
            from . import _pevlm_call
        except ImportError as e:
            raise RuntimeError("_pevlm_call is missing: build it with `python -m paper_2506_19651_b200.build`") from e
        _calls = _pevlm_call
    return _calls


_raw_stream = None


def _stream():
    """Handle of torch's current stream on the current device (the raw accessor costs a third of building a Stream object)."""
    global _raw_stream
    if _raw_stream is None:
        import torch
        raw = getattr(torch._C, "_cuda_getCurrentRawStream", None)
        if raw is None:
            _raw_stream = lambda: torch.cuda.current_stream().cuda_stream
        else:
            device = torch.cuda.current_device   # also initialises CUDA where nothing has yet
            device()
            device = getattr(torch._C, "_cuda_getDevice", device)
            _raw_stream = lambda: raw(device())
    return _raw_stream()


def _address(shape):
    if not isinstance(shape, Shape):
        raise C.ArgumentError(f"expected a Shape, got {type(shape).__name__}")
    return C.addressof(shape)


def _check(rc, where):
    if rc != PEVLM_OK:
        raise PevlmError(rc, where)


def pevlm_workspace_bytes(shape: Shape, which: int) -> int:
    return int(lib().pevlm_workspace_bytes(C.byref(shape), which))


# A tensor argument may also be None where the C call takes NULL, or a device address.

def pevlm_rope_qk(shape: Shape, q_in, k_in, q_out, k_out, first_token: int, n_tokens: int, pos_ids=None):
    _check(_native().rope_qk(_address(shape), q_in, k_in, q_out, k_out, first_token, n_tokens, pos_ids, _stream()), "pevlm_rope_qk")


def pevlm_rope_qkv(shape: Shape, q_in, k_in, v_in, q_out, k_out, v_out, first_token: int, n_tokens: int, pos_ids=None):
    _check(_native().rope_qkv(_address(shape), q_in, k_in, v_in, q_out, k_out, v_out, first_token, n_tokens, pos_ids, _stream()),
           "pevlm_rope_qkv")


def pevlm_layer_forward(shape: Shape, q, k, v, q_video, q_question, k_cache, v_cache, o_video, lse_video, o_question,
                        lse_question, ws_prefill, ws_query, last_len: int = 0):
    _check(_native().layer_forward(_address(shape), last_len, q, k, v, q_video, q_question, k_cache, v_cache, o_video, lse_video,
                                   o_question, lse_question, ws_prefill, ws_prefill.nbytes, ws_query, ws_query.nbytes, _stream()),
           "pevlm_layer_forward")


def pevlm_rope_qk_mrope(shape: Shape, q_in, k_in, q_out, k_out, n_tokens: int, pos_ids3, sections):
    """sections: pairs per position component; components that are not given have none."""
    sections = tuple(sections)
    sections += (0,) * (3 - len(sections))
    _check(_native().rope_qk_mrope(_address(shape), q_in, k_in, q_out, k_out, n_tokens, pos_ids3, *sections, _stream()),
           "pevlm_rope_qk_mrope")


def pevlm_parallel_prefill_attn(shape: Shape, q, k, v, o, lse, workspace):
    _check(_native().parallel_prefill_attn(_address(shape), q, k, v, o, lse, workspace, workspace.nbytes, _stream()),
           "pevlm_parallel_prefill_attn")


def pevlm_block_attn(shape: Shape, q_blocks, k_cache, v_cache, first_key_row: int, cache_rows: int, o, lse, workspace):
    _check(_native().block_attn(_address(shape), q_blocks, k_cache, v_cache, first_key_row, cache_rows, o, lse, workspace,
                                workspace.nbytes, _stream()), "pevlm_block_attn")


def pevlm_assemble_kv(shape: Shape, k_video, v_video, k_question, v_question, k_cache, v_cache):
    _check(_native().assemble_kv(_address(shape), k_video, v_video, k_question, v_question, k_cache, v_cache, _stream()),
           "pevlm_assemble_kv")


def pevlm_query_attn(shape: Shape, q_question, k_cache, v_cache, o, lse, workspace):
    _check(_native().query_attn(_address(shape), q_question, k_cache, v_cache, o, lse, workspace, workspace.nbytes, _stream()),
           "pevlm_query_attn")


def pevlm_query_attn_noalloc(shape: Shape, q_question, k_cache, v_cache, o, lse):
    """Question attention for callers that cannot allocate device memory: no workspace argument,
    the partials go to the library's built-in scratch array (see include/pevlm.h for its limits)."""
    _check(_native().query_attn_noalloc(_address(shape), q_question, k_cache, v_cache, o, lse, _stream()), "pevlm_query_attn_noalloc")


def pevlm_selftest_wait_expiry(workspace, limit_ns: int):
    _check(lib().pevlm_selftest_wait_expiry(_ptr(workspace), workspace.nbytes,
                                            limit_ns, _stream()), "pevlm_selftest_wait_expiry")


def pevlm_read_status(workspace):
    """workspace = None reads the built-in array of pevlm_query_attn_noalloc on the current device."""
    st, det = C.c_int32(0), C.c_int32(0)
    _check(lib().pevlm_read_status(_ptr(workspace), _stream(), C.byref(st), C.byref(det)), "pevlm_read_status")
    return st.value, det.value


@dataclass
class TileStats:
    tiles: int
    flops: float


def pevlm_tile_stats(shape: Shape, which: int) -> TileStats:
    t, f = C.c_int64(0), C.c_double(0.0)
    _check(lib().pevlm_tile_stats(C.byref(shape), which, C.byref(t), C.byref(f)), "pevlm_tile_stats")
    return TileStats(t.value, f.value)
