"""ctypes binding of libkvq.so: argument marshalling only.

Every function here has the name of the C entry point it calls (include/kvq.h)
and does nothing but turn torch tensors into device pointers, strides and a
stream handle.  All of the method's arithmetic runs in the CUDA kernels behind
the C ABI; there is no CPU or PyTorch fallback: if the library cannot be loaded,
importing this module raises.
"""
from __future__ import annotations

import ctypes as C
import os

import torch

from .build import py_call_target

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "libkvq.so")

KVQ_OK = 0
KVQ_ERR_INVALID_ARG, KVQ_ERR_UNSUPPORTED, KVQ_ERR_ALIGNMENT = -1, -2, -3
KVQ_ERR_CAPACITY, KVQ_ERR_CUDA, KVQ_ERR_TIMEOUT, KVQ_ERR_WORKSPACE = -4, -5, -6, -7
KVQ_ROTATE_K = 1
KVQ_RING = 2
KVQ_ROTATE_V = 4
KVQ_K_PER_CHANNEL = 8
KVQ_CORRECTION_OFF, KVQ_CORRECTION_ON, KVQ_CORRECTION_EXACT = 0, 1, 2
KVQ_KERNEL_AUTO, KVQ_KERNEL_MMA_SYNC, KVQ_KERNEL_TCGEN05, KVQ_KERNEL_TCGEN05_PAIR = 0, 1 << 8, 2 << 8, 3 << 8


class kvq_cache_desc(C.Structure):
    _fields_ = [
        ("batch", C.c_int32), ("heads", C.c_int32), ("head_dim", C.c_int32),
        ("bits", C.c_int32), ("group", C.c_int32), ("flags", C.c_uint32),
        ("capacity", C.c_int64),
        ("k_codes", C.c_void_p), ("v_codes", C.c_void_p),
        ("k_scale", C.c_void_p), ("v_scale", C.c_void_p),
        ("k_zero", C.c_void_p), ("v_zero", C.c_void_p),
        ("signs", C.c_void_p),
    ]


class kvq_strides(C.Structure):
    _fields_ = [("b", C.c_int64), ("h", C.c_int64), ("t", C.c_int64)]


def _load():
    if not os.path.exists(LIB_PATH):
        raise ImportError(
            f"{LIB_PATH} is missing: build it with `python -m paper_2605_26266_b200.build` "
            "(there is no fallback path)")
    lib = C.CDLL(LIB_PATH)
    lib.kvq_version.restype = C.c_int
    lib.kvq_last_cuda_error.restype = C.c_int
    lib.kvq_status_string.restype = C.c_char_p
    lib.kvq_status_string.argtypes = [C.c_int]
    lib.kvq_cache_bytes.restype = C.c_int
    lib.kvq_cache_bytes.argtypes = [C.POINTER(kvq_cache_desc), C.POINTER(C.c_size_t)]
    lib.kvq_quantize_append.restype = C.c_int
    lib.kvq_quantize_append.argtypes = [C.POINTER(kvq_cache_desc), C.c_int64, C.c_void_p, C.c_void_p,
                                        kvq_strides, C.c_int64, C.c_void_p]
    lib.kvq_attn_workspace_bytes.restype = C.c_int
    lib.kvq_attn_workspace_bytes.argtypes = [C.POINTER(kvq_cache_desc), C.c_int64, C.c_int64, C.c_int64,
                                             C.c_uint32, C.POINTER(C.c_size_t)]
    lib.kvq_attn_kernel_launches.restype = C.c_int
    lib.kvq_attn_kernel_launches.argtypes = [C.POINTER(kvq_cache_desc), C.c_int64, C.c_int64, C.c_int64,
                                             C.c_uint32, C.POINTER(C.c_int)]
    lib.kvq_attn_corrected.restype = C.c_int
    lib.kvq_attn_corrected.argtypes = [
        C.POINTER(kvq_cache_desc), C.c_int64, C.c_int64,
        C.c_void_p, kvq_strides, C.c_void_p, C.c_void_p, kvq_strides,
        C.c_int64, C.c_int64, C.c_void_p, kvq_strides,
        C.c_float, C.c_uint32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p]
    lib.kvq_attn_corrected_static_scratch.restype = C.c_int
    lib.kvq_attn_corrected_static_scratch.argtypes = [
        C.POINTER(kvq_cache_desc), C.c_int64, C.c_int64,
        C.c_void_p, kvq_strides, C.c_void_p, C.c_void_p, kvq_strides,
        C.c_int64, C.c_int64, C.c_void_p, kvq_strides,
        C.c_float, C.c_uint32, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.kvq_status_word_result.restype = C.c_int
    lib.kvq_status_word_result.argtypes = [C.c_int32]
    lib.kvq_set_wait_budget_cycles.restype = C.c_int
    lib.kvq_set_wait_budget_cycles.argtypes = [C.c_uint64]
    lib.kvq_attn_weight_jsd.restype = C.c_int
    lib.kvq_attn_weight_jsd.argtypes = [
        C.POINTER(kvq_cache_desc), C.c_int64, C.c_int64, C.c_void_p, kvq_strides, C.c_void_p, kvq_strides,
        C.c_void_p, kvq_strides, C.c_int64, C.c_int64, C.c_float, C.c_uint32, C.c_void_p, C.c_void_p]
    lib.kvq_unpack_codes.restype = C.c_int
    lib.kvq_unpack_codes.argtypes = [C.POINTER(kvq_cache_desc), C.c_int, C.c_int64, C.c_int64,
                                     C.c_void_p, C.c_void_p]
    return lib


lib = _load()
_quantize_append, _attn_workspace_bytes, _attn_corrected = lib.kvq_quantize_append, lib.kvq_attn_workspace_bytes, lib.kvq_attn_corrected
_BF16 = torch.bfloat16

# The plain calls of the hot path go through a small CPython extension (csrc/py_call.cpp), which reads the tensors without the
# Python-level accessors: a small append is a few microseconds of Python around a kernel of two (5.7 us a call through ctypes).
# It answers _NOT_PLAIN to anything else (subclasses, other dtypes or layouts, whatever raises), and where it cannot be loaded or
# was built for another torch or Python every call takes the ctypes route below it.
_NOT_PLAIN = -1000
try:
    from . import _py_call
    if getattr(_py_call, "built_for", None) != py_call_target(torch.__version__):
        raise ImportError("_py_call is of another torch or Python")
    _py_call.bind(*(C.cast(f, C.c_void_p).value for f in (_quantize_append, _attn_workspace_bytes, _attn_corrected)))
    _append_call, _attn_call = _py_call.append, _py_call.attn
except ImportError:
    def _append_call(*_):
        return _NOT_PLAIN
    _attn_call = _append_call


class KvqError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        msg = lib.kvq_status_string(status).decode()
        if status == KVQ_ERR_CUDA:
            msg += f" (cudaError {lib.kvq_last_cuda_error()})"
        super().__init__(f"{where}: {msg} [{status}]")


def _check(status: int, where: str):
    if status != KVQ_OK:
        raise KvqError(status, where)


def _strides_of(st) -> kvq_strides:
    assert len(st) == 4 and st[3] == 1, "tensor must be [batch, heads, tokens, head_dim] with unit inner stride"
    return kvq_strides(st[0], st[1], st[2])


def _strides(t: torch.Tensor) -> kvq_strides:
    return _strides_of(t.stride())


# The current stream's handle without the Stream object around it: a small append is a few microseconds of Python around a
# kernel of two, and the object alone was two of them.  A torch that lacks the two functions gets the object.
_raw_stream, _current_device = (getattr(torch._C, f, None) for f in ("_cuda_getCurrentRawStream", "_cuda_getDevice"))


def _stream() -> int:
    if _raw_stream is None or _current_device is None:
        return torch.cuda.current_stream().cuda_stream
    return _raw_stream(_current_device())


_capturing = getattr(torch._C, "_cuda_isCurrentStreamCapturing", torch.cuda.is_current_stream_capturing)


def _ptr(t):
    return None if t is None else t.data_ptr()


class Cache:
    """Caller-side owner of the six device buffers of one quantized cache plus its descriptor."""

    def __init__(self, batch, heads, head_dim, bits, group, capacity, rotate_k=True, signs=None, device="cuda",
                 ring=False, rotate_v=False, k_per_channel=False):
        self.desc = kvq_cache_desc(batch, heads, head_dim, bits, group,
                                   (KVQ_ROTATE_K if rotate_k else 0) | (KVQ_RING if ring else 0)
                                   | (KVQ_ROTATE_V if rotate_v else 0) | (KVQ_K_PER_CHANNEL if k_per_channel else 0),
                                   capacity)
        sizes = kvq_cache_bytes(self.desc)
        self.buffers = [torch.zeros(n, dtype=torch.uint8, device=device) for n in sizes]
        (self.desc.k_codes, self.desc.v_codes, self.desc.k_scale, self.desc.v_scale,
         self.desc.k_zero, self.desc.v_zero) = [b.data_ptr() for b in self.buffers]
        self.signs = None
        if signs is not None:
            self.signs = torch.as_tensor(signs, dtype=torch.int8).to(device).contiguous()
            self.desc.signs = self.signs.data_ptr()
        self.length = 0
        self.workspace = None
        self._stream_workspaces = {}

    def _stream_workspace(self, need, stream, device):
        """Heads of 64 channels had no workspace once, so that calls which only read one cache could run on several streams
        and threads: a buffer for each stream (at most eight are kept), a fresh one for a call that is being captured."""
        capturing = _capturing()
        kept = self._stream_workspaces
        ws = None if capturing else kept.get(stream)
        if ws is None or ws.numel() < need:
            ws = torch.empty(need, dtype=torch.uint8, device=device)
            if not capturing:
                if stream not in kept and len(kept) >= 8:
                    kept.pop(list(kept)[0], None)
                kept[stream] = ws
        return ws

    @property
    def groups(self):
        return self.desc.head_dim // self.desc.group

    def views(self):
        """The six buffers shaped [batch, heads, capacity, ...] (codes u8, scale u8, zero as int16 bits)."""
        d = self.desc
        B, H, Cp, G = d.batch, d.heads, d.capacity, self.groups
        kc, vc, ks, vs, kz, vz = self.buffers
        # per-channel keys: one row of head_dim steps / zero-points per block of `group` tokens
        kshape = (B, H, Cp // d.group, d.head_dim) if d.flags & KVQ_K_PER_CHANNEL else (B, H, Cp, G)
        return {
            "k_codes": kc.view(B, H, Cp, -1), "v_codes": vc.view(B, H, Cp, -1),
            "k_scale": ks.view(*kshape), "v_scale": vs.view(B, H, Cp, G),
            "k_zero": kz.view(torch.int16).view(*kshape), "v_zero": vz.view(torch.int16).view(B, H, Cp, G),
        }


def _workspace(cache, need, stream, device):
    """A workspace of `need` bytes where the cache's own does not do."""
    if cache.desc.head_dim == 64:
        return cache._stream_workspace(need, stream, device)
    cache.workspace = torch.empty(need, dtype=torch.uint8, device=device)
    return cache.workspace


def kvq_version() -> int:
    return lib.kvq_version()


def kvq_cache_bytes(desc: kvq_cache_desc):
    out = (C.c_size_t * 6)()
    _check(lib.kvq_cache_bytes(C.byref(desc), out), "kvq_cache_bytes")
    return list(out)


def kvq_quantize_append(cache: Cache, k: torch.Tensor, v: torch.Tensor, cache_len: int | None = None) -> int:
    """Appends the chunk k, v ([batch, heads, n, head_dim] BF16, CUDA) at token `cache_len`
    (default: the cache's running length) and returns the new length."""
    pos = cache.length if cache_len is None else cache_len
    status = _append_call(C.addressof(cache.desc), pos, k, v, _stream()) if k.is_cuda else _NOT_PLAIN
    if status == _NOT_PLAIN:
        assert k.dtype is _BF16 and v.dtype is _BF16 and k.is_cuda and v.is_cuda
        st = k.stride()
        assert k.shape == v.shape and st == v.stride()
        status = _quantize_append(C.byref(cache.desc), pos, k.data_ptr(), v.data_ptr(), _strides_of(st), k.shape[2], _stream())
    if status:
        _check(status, "kvq_quantize_append")
    cache.length = pos + k.shape[2]
    return cache.length


def kvq_attn_workspace_bytes(cache: Cache, cache_len: int, m_tokens: int, n_cur: int, flags: int) -> int:
    out = C.c_size_t(0)
    _check(lib.kvq_attn_workspace_bytes(C.byref(cache.desc), cache_len, m_tokens, n_cur, flags, C.byref(out)),
           "kvq_attn_workspace_bytes")
    return out.value


def kvq_attn_kernel_launches(cache: Cache, cache_len: int, m_tokens: int, n_cur: int, flags: int) -> int:
    out = C.c_int(0)
    _check(lib.kvq_attn_kernel_launches(C.byref(cache.desc), cache_len, m_tokens, n_cur, flags, C.byref(out)),
           "kvq_attn_kernel_launches")
    return out.value


def kvq_attn_corrected(cache: Cache, q, k_cur, v_cur, softmax_scale, flags=KVQ_CORRECTION_ON,
                       cache_begin=0, cache_len=None, out=None, lse=None, cached_mass=None,
                       status_word=None):
    """out = corrected attention of q over [cache window ; current chunk].  Tensors are
    [batch, heads, tokens, head_dim] BF16 CUDA; returns `out` (allocated if not given)."""
    n_cache = cache.length - cache_begin if cache_len is None else cache_len
    if out is None and type(q) is torch.Tensor:
        out = torch.empty_like(q, memory_format=torch.contiguous_format)
    if out is not None and q.is_cuda:
        stream, ws = _stream(), cache.workspace
        if ws is None and cache._stream_workspaces and not _capturing():
            ws = cache._stream_workspaces.get(stream)
        for _ in range(2):
            status = _attn_call(C.addressof(cache.desc), cache_begin, n_cache, q, k_cur, v_cur, out, softmax_scale, flags, lse,
                                cached_mass, status_word, ws, stream)
            if status <= 0:
                break
            ws = _workspace(cache, status, stream, q.device)
        if status == KVQ_OK:
            return out
        if status != _NOT_PLAIN:      # refused or failed, and not issued again; the size query is host arithmetic and tells which call it was
            size = C.c_size_t(0)
            _check(_attn_workspace_bytes(C.byref(cache.desc), n_cache, q.shape[2], k_cur.shape[2], flags, C.byref(size)), "kvq_attn_workspace_bytes")
            _check(status, "kvq_attn_corrected")
    # not a plain call: checked and raised here
    for t in (q, k_cur, v_cur):
        assert t.dtype is _BF16 and t.is_cuda
    kv_shape, kv_st = k_cur.shape, k_cur.stride()
    assert kv_shape == v_cur.shape and kv_st == v_cur.stride()
    if out is None:
        out = torch.empty_like(q, memory_format=torch.contiguous_format)
    m, n_cur, desc, size = q.shape[2], kv_shape[2], C.byref(cache.desc), C.c_size_t(0)
    status = _attn_workspace_bytes(desc, n_cache, m, n_cur, flags, C.byref(size))
    if status:
        _check(status, "kvq_attn_workspace_bytes")
    need, ws, stream = size.value, None, _stream()
    if need:
        ws = cache.workspace
        if ws is None or ws.numel() < need:
            ws = _workspace(cache, need, stream, q.device)
    status = _attn_corrected(
        desc, cache_begin, n_cache, q.data_ptr(), _strides_of(q.stride()), k_cur.data_ptr(), v_cur.data_ptr(),
        _strides_of(kv_st), m, n_cur, out.data_ptr(), _strides_of(out.stride()), float(softmax_scale), flags, _ptr(lse),
        _ptr(cached_mass), _ptr(ws), ws.numel() if need else 0, _ptr(status_word), stream)
    if status:
        _check(status, "kvq_attn_corrected")
    return out


def kvq_attn_corrected_static_scratch(cache: Cache, q, k_cur, v_cur, softmax_scale, flags=KVQ_CORRECTION_ON,
                                      cache_begin=0, cache_len=None, out=None, lse=None, cached_mass=None,
                                      status_word=None):
    """kvq_attn_corrected without a workspace: split units keep their partial results in the scratch buffer
    built into the library.  `out` must be given by callers that may not allocate; it is allocated here only
    as a convenience when omitted."""
    for t in (q, k_cur, v_cur):
        assert t.dtype == torch.bfloat16 and t.is_cuda
    assert k_cur.shape == v_cur.shape and k_cur.stride() == v_cur.stride()
    n_cache = cache.length - cache_begin if cache_len is None else cache_len
    if out is None:
        out = torch.empty_like(q, memory_format=torch.contiguous_format)
    _check(lib.kvq_attn_corrected_static_scratch(
        C.byref(cache.desc), cache_begin, n_cache, q.data_ptr(), _strides(q), k_cur.data_ptr(), v_cur.data_ptr(),
        _strides(k_cur), q.shape[2], k_cur.shape[2], out.data_ptr(), _strides(out), float(softmax_scale), flags,
        _ptr(lse), _ptr(cached_mass), _ptr(status_word), _stream()), "kvq_attn_corrected_static_scratch")
    return out


def kvq_attn_weight_jsd(cache: Cache, q, k_cur, k_cached, softmax_scale, flags=KVQ_CORRECTION_ON, cache_begin=0,
                        cache_len=None, out=None):
    """Per-row JSD of the attention weights against those of the BF16 keys k_cached ([batch, heads, cache_len,
    head_dim], the keys the attended cache window was quantized from); returns float32 [batch, heads, rows]."""
    for t in (q, k_cur) + ((k_cached,) if k_cached is not None else ()):
        assert t.dtype == torch.bfloat16 and t.is_cuda
    n_cache = cache.length - cache_begin if cache_len is None else cache_len
    assert n_cache == 0 or k_cached.shape[2] == n_cache
    if out is None:
        out = torch.empty(q.shape[:3], dtype=torch.float32, device=q.device)
    kc_ptr, kc_str = (k_cached.data_ptr(), _strides(k_cached)) if n_cache else (None, kvq_strides(0, 0, 0))
    _check(lib.kvq_attn_weight_jsd(
        C.byref(cache.desc), cache_begin, n_cache, q.data_ptr(), _strides(q), k_cur.data_ptr(), _strides(k_cur),
        kc_ptr, kc_str, q.shape[2], k_cur.shape[2], float(softmax_scale), flags, out.data_ptr(), _stream()),
        "kvq_attn_weight_jsd")
    return out


def kvq_status_word_result(word: int) -> int:
    return lib.kvq_status_word_result(int(word))


def kvq_set_wait_budget_cycles(cycles: int) -> None:
    _check(lib.kvq_set_wait_budget_cycles(int(cycles)), "kvq_set_wait_budget_cycles")


def kvq_unpack_codes(cache: Cache, which: int, begin: int, n: int) -> torch.Tensor:
    d = cache.desc
    out = torch.empty((d.batch, d.heads, n, d.head_dim), dtype=torch.uint8, device=cache.buffers[0].device)
    _check(lib.kvq_unpack_codes(C.byref(d), which, begin, n, out.data_ptr(), _stream()), "kvq_unpack_codes")
    return out
