"""Thin binding of the C-ABI library (`include/gta.h`): argument marshalling only, by ctypes and, for the calls of a
serving loop, in the extension `_gta_binding` (csrc/gta_binding.cpp).

Every step of the operator runs inside the CUDA library; PyTorch is used for device memory,
streams and host<->device copies.  There is no CPU fallback: if `libgta_b200.so` has not been
built (``python -m paper_2506_17286_b200.build``) every entry point raises.
"""
from __future__ import annotations

import ctypes
import functools
import importlib.machinery
import importlib.util
import os

import torch

from .build import native_path

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libgta_b200.so")

GTA_OK, GTA_ERR_INVALID_ARG, GTA_ERR_UNSUPPORTED, GTA_ERR_WORKSPACE = 0, 1, 2, 3
GTA_ERR_CUDA, GTA_ERR_CACHE_FULL, GTA_ERR_TIMEOUT, GTA_ERR_STATIC_SCRATCH = 4, 5, 6, 7
GTA_ERR_BAD_PAGE = 8
STATIC_SCRATCH_BYTES = 16 << 20
GTA_F32, GTA_BF16 = 0, 1

EXPORTS = (
    "gta_prefill_workspace_bytes", "gta_prefill", "gta_decode_workspace_bytes", "gta_decode",
    "gta_cache_append", "gta_status_string", "gta_version", "gta_prefill_path", "gta_last_launch_count",
    "gta_prefill_stages", "gta_decode_stages", "gta_decode_static", "gta_prefill_chunk", "gta_prefill_chunk_workspace_bytes",
    "gta_decode_paged_workspace_bytes", "gta_decode_paged", "gta_cache_append_paged",
    "gta_layer_prefill_workspace_bytes", "gta_layer_prefill", "gta_layer_decode_workspace_bytes", "gta_layer_decode",
    "gta_layer_decode_paged_workspace_bytes", "gta_layer_decode_paged", "gta_debug_attention_wait",
    "gta_debug_decode_wait",
    "gta_ref_gqa_prefill", "gta_ref_gqa_decode_workspace_bytes", "gta_ref_gqa_decode",
    "gta_decode_fp8_workspace_bytes", "gta_cache_append_fp8", "gta_decode_fp8", "gta_decode_append",
    "gta_prefill_chunk_paged", "gta_layer_prefill_paged", "gta_decode_fp8_path",
    "gta_decode_hostcache_workspace_bytes", "gta_decode_hostcache",
)


class GtaShape(ctypes.Structure):
    """Mirror of gta_shape_t."""
    _fields_ = [
        ("batch", ctypes.c_int32), ("seq", ctypes.c_int32), ("d_model", ctypes.c_int32),
        ("n_heads", ctypes.c_int32), ("n_q_groups", ctypes.c_int32), ("n_k_groups", ctypes.c_int32),
        ("n_c_groups", ctypes.c_int32), ("head_dim", ctypes.c_int32), ("latent_dim", ctypes.c_int32),
        ("causal", ctypes.c_int32), ("dtype", ctypes.c_int32), ("softmax_scale", ctypes.c_float),
    ]


class GtaError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} (status {status})")


_lib = None
_native = None


def lib():
    """Load the shared library (once).  Raises if it is missing: there is no fallback."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(
                f"{LIB_PATH} not found: build it with `python -m paper_2506_17286_b200.build` "
                "(the GTA operator has no CPU or PyTorch fallback)")
        L = ctypes.CDLL(LIB_PATH)
        vp, i32, sz = ctypes.c_void_p, ctypes.c_int32, ctypes.c_size_t
        sp = ctypes.POINTER(GtaShape)
        L.gta_prefill_workspace_bytes.argtypes = [sp]
        L.gta_prefill_workspace_bytes.restype = sz
        L.gta_prefill_chunk_workspace_bytes.argtypes = [sp, i32]
        L.gta_prefill_chunk_workspace_bytes.restype = sz
        L.gta_prefill.argtypes = [sp, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_prefill.restype = i32
        L.gta_prefill_stages.argtypes = [sp, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp, vp, i32]
        L.gta_prefill_stages.restype = i32
        L.gta_prefill_chunk.argtypes = [sp, i32, i32, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_prefill_chunk.restype = i32
        L.gta_prefill_chunk_paged.argtypes = [sp, i32, vp, vp, vp, vp, i32, i32, i32, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_prefill_chunk_paged.restype = i32
        L.gta_layer_prefill_paged.argtypes = [sp, i32, ctypes.c_float, vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i32, vp,
                                              vp, sz, vp, vp]
        L.gta_layer_prefill_paged.restype = i32
        L.gta_decode_stages.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp, vp, i32]
        L.gta_decode_stages.restype = i32
        L.gta_decode_workspace_bytes.argtypes = [sp, i32]
        L.gta_decode_workspace_bytes.restype = sz
        L.gta_decode.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_decode.restype = i32
        L.gta_decode_hostcache_workspace_bytes.argtypes = [sp, i32]
        L.gta_decode_hostcache_workspace_bytes.restype = sz
        L.gta_decode_hostcache.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_decode_hostcache.restype = i32
        L.gta_decode_static.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, vp]
        L.gta_decode_static.restype = i32
        L.gta_cache_append.argtypes = [sp, vp, vp, i32, vp, vp, i32, vp, vp, vp]
        L.gta_cache_append.restype = i32
        L.gta_decode_paged_workspace_bytes.argtypes = [sp, i32, i32]
        L.gta_decode_paged_workspace_bytes.restype = sz
        L.gta_decode_paged.argtypes = [sp, vp, vp, vp, vp, i32, i32, i32, vp, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_decode_paged.restype = i32
        L.gta_cache_append_paged.argtypes = [sp, vp, vp, vp, i32, i32, i32, vp, vp, i32, vp, vp, vp]
        L.gta_cache_append_paged.restype = i32
        L.gta_layer_prefill_workspace_bytes.argtypes = [sp]
        L.gta_layer_prefill_workspace_bytes.restype = sz
        L.gta_layer_prefill.argtypes = [sp, i32, i32, ctypes.c_float, vp, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_layer_prefill.restype = i32
        L.gta_layer_decode_workspace_bytes.argtypes = [sp, i32]
        L.gta_layer_decode_workspace_bytes.restype = sz
        L.gta_layer_decode.argtypes = [sp, i32, ctypes.c_float, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_layer_decode.restype = i32
        L.gta_layer_decode_paged_workspace_bytes.argtypes = [sp, i32, i32]
        L.gta_layer_decode_paged_workspace_bytes.restype = sz
        L.gta_layer_decode_paged.argtypes = [sp, vp, i32, i32, i32, ctypes.c_float, vp, vp, vp, vp, vp, vp, vp, vp, vp,
                                             vp, sz, vp, vp]
        L.gta_layer_decode_paged.restype = i32
        L.gta_status_string.argtypes = [i32]
        L.gta_status_string.restype = ctypes.c_char_p
        L.gta_version.restype = i32
        L.gta_prefill_path.argtypes = [sp]
        L.gta_prefill_path.restype = i32
        L.gta_last_launch_count.restype = i32
        L.gta_ref_gqa_prefill.argtypes = [sp, vp, vp, vp, vp, vp, vp]
        L.gta_ref_gqa_prefill.restype = i32
        L.gta_ref_gqa_decode_workspace_bytes.argtypes = [sp]
        L.gta_ref_gqa_decode_workspace_bytes.restype = sz
        L.gta_ref_gqa_decode.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, sz, vp, vp]
        L.gta_ref_gqa_decode.restype = i32
        L.gta_decode_fp8_workspace_bytes.argtypes = [sp, i32]
        L.gta_decode_fp8_workspace_bytes.restype = sz
        L.gta_decode_fp8_path.argtypes = [sp, i32]
        L.gta_decode_fp8_path.restype = i32
        L.gta_cache_append_fp8.argtypes = [sp, vp, vp, vp, vp, i32, vp, vp, i32, vp, vp, vp]
        L.gta_cache_append_fp8.restype = i32
        L.gta_decode_fp8.argtypes = [sp, vp, vp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_decode_fp8.restype = i32
        L.gta_decode_append.argtypes = [sp, vp, vp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp, vp]
        L.gta_decode_append.restype = i32
        L.gta_debug_attention_wait.argtypes = [ctypes.c_uint64, i32]
        L.gta_debug_attention_wait.restype = i32
        L.gta_debug_decode_wait.argtypes = [ctypes.c_uint64, i32]
        L.gta_debug_decode_wait.restype = i32
        _lib = L
    return _lib


def native():
    """The extension, bound to the entry points of the loaded library (once)."""
    global _native
    if _native is None:
        L = lib()
        path = native_path()
        if not os.path.exists(path):
            raise RuntimeError(f"{path} not found: build it with `python -m paper_2506_17286_b200.build`")
        loader = importlib.machinery.ExtensionFileLoader("_gta_binding", path)
        mod = importlib.util.module_from_spec(importlib.util.spec_from_loader("_gta_binding", loader))
        loader.exec_module(mod)
        for name in EXPORTS:
            mod.bind(name, ctypes.cast(getattr(L, name), ctypes.c_void_p).value)
        _native = mod
    return _native


def status_string(status: int) -> str:
    return lib().gta_status_string(int(status)).decode()


def version() -> int:
    return int(lib().gta_version())


def debug_decode_wait(limit_ns: int = 0, withhold_first_arrive: bool = False) -> None:
    """Test hook of the tensor-memory decode stream kernels' bounded waits (see gta_debug_decode_wait in include/gta.h)."""
    st = lib().gta_debug_decode_wait(int(limit_ns), int(bool(withhold_first_arrive)))
    if st != GTA_OK:
        raise GtaError(st, "gta_debug_decode_wait")


def debug_attention_wait(limit_ns: int = 0, withhold_first_arrive: bool = False) -> None:
    """Test hook: time limit of the attention kernel's bounded waits (0 = built-in) and the switch that
    makes the first hand-over of the prefill kernels wait in vain (see gta_debug_attention_wait in include/gta.h)."""
    st = lib().gta_debug_attention_wait(int(limit_ns), int(bool(withhold_first_arrive)))
    if st != GTA_OK:
        raise GtaError(st, "gta_debug_attention_wait")


def last_launch_count() -> int:
    return int(lib().gta_last_launch_count())


def _dtype_code(t: torch.Tensor) -> int:
    if t.dtype == torch.float32:
        return GTA_F32
    if t.dtype == torch.bfloat16:
        return GTA_BF16
    raise TypeError(f"unsupported dtype {t.dtype}: the library takes float32 or bfloat16")


# The helpers of the ctypes calls stay with plain integers: addresses and streams go to ctypes as they are, device
# identity is an index, and the structs are kept by value.
def _ptr(t):
    return None if t is None else t.data_ptr()


def _stream(stream):
    # (looked up here: a torch without CUDA imports this module too)
    return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice()) if stream is None else stream.cuda_stream


def _check_tensors(*ts):
    dev, dt = ts[0].get_device(), ts[0].dtype
    for t in ts:
        if t.dtype is not dt or t.get_device() != dev:
            raise ValueError("all operator tensors must share one device and one dtype")
        if not t.is_contiguous():
            raise ValueError("operator tensors must be contiguous")
        if dev < 0:
            raise ValueError("operator tensors must live on a CUDA device")


@functools.lru_cache(maxsize=1024)
def _shape(batch, seq, d_model, n_heads, n_q, n_k, n_c, d_h, d_l, code, causal, softmax_scale):
    """The struct of a call, kept by its values (the library only reads it) and never handed out."""
    return GtaShape(batch, seq, d_model, n_heads, n_q, n_k, n_c, d_h, d_l, causal, code, softmax_scale)


def make_shape(*, batch, seq, d_model, n_heads, n_q, n_k, n_c, d_h, d_l, dtype, causal=True,
               softmax_scale=0.0) -> GtaShape:
    code = dtype if isinstance(dtype, int) else (GTA_F32 if dtype == torch.float32 else GTA_BF16)
    return GtaShape(batch, seq, d_model, n_heads, n_q, n_k, n_c, d_h, d_l, int(bool(causal)), code,
                    float(softmax_scale))


def prefill_workspace_bytes(shape: GtaShape) -> int:
    return int(lib().gta_prefill_workspace_bytes(ctypes.byref(shape)))


def prefill_chunk_workspace_bytes(shape: GtaShape, kv_len: int) -> int:
    return int(lib().gta_prefill_chunk_workspace_bytes(ctypes.byref(shape), int(kv_len)))


def decode_workspace_bytes(shape: GtaShape, s_cap: int) -> int:
    return int(lib().gta_decode_workspace_bytes(ctypes.byref(shape), int(s_cap)))


def prefill_path(shape: GtaShape) -> int:
    return int(lib().gta_prefill_path(ctypes.byref(shape)))


def _workspace(nbytes: int, device) -> torch.Tensor:
    return torch.empty(max(nbytes, 256), dtype=torch.uint8, device=device)


def gta_prefill(q, k, c, x, w_p, w_g, *, causal=True, softmax_scale=0.0, out=None, workspace=None,
                status_word=None, stream=None, stages=3):
    """out[B, N, n_h, d_h] = GTA prefill.  q [B,n_q,N,d_h], k [B,n_k,N,d_h], c [B,n_c,N,d_l],
    x [B,N,H], w_p [n_h,d_l,d_h], w_g [H,n_h*d_h]; all on one CUDA device, one dtype."""
    if stages == 3:
        r = (_native or native()).prefill(q, k, c, x, w_p, w_g, 1 if causal else 0, softmax_scale, out, workspace, status_word,
                                          stream)
        if type(r) is int:
            raise GtaError(r, "gta_prefill")
        return r
    _check_tensors(q, k, c, x, w_p, w_g)
    B, n_q, N, d_h = q.shape
    n_k, n_c, d_l = k.shape[1], c.shape[1], c.shape[3]
    n_h, H = w_p.shape[0], x.shape[2]
    if k.shape != (B, n_k, N, d_h) or c.shape != (B, n_c, N, d_l) or x.shape != (B, N, H) \
            or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h):
        raise ValueError("inconsistent operator tensor shapes")
    shape = _shape(B, N, H, n_h, n_q, n_k, n_c, d_h, d_l, _dtype_code(q), 1 if causal else 0, float(softmax_scale))
    if out is None:
        out = q.new_empty((B, N, n_h, d_h))
    if workspace is None:
        workspace = _workspace(prefill_workspace_bytes(shape), q.device)
    st = lib().gta_prefill_stages(ctypes.byref(shape), _ptr(q), _ptr(k), _ptr(c), _ptr(x), _ptr(w_p), _ptr(w_g), _ptr(out),
                                  _ptr(workspace), workspace.nbytes, _ptr(status_word), _stream(stream), stages)
    if st != GTA_OK:
        raise GtaError(st, "gta_prefill")
    return out


def gta_prefill_chunk(q, k, c, x, w_p, w_g, kv_len, *, causal=True, softmax_scale=0.0, out=None, workspace=None,
                      status_word=None, stream=None):
    """gta_prefill for the last N of kv_len positions.  q [B,n_q,N,d_h], x [B,N,H]; k [B,n_k,kv_cap,d_h],
    c [B,n_c,kv_cap,d_l] of which rows 0 .. kv_len-1 are attended."""
    _check_tensors(q, k, c, x, w_p, w_g)
    B, n_q, N, d_h = q.shape
    n_k, kv_cap, n_c, d_l = k.shape[1], k.shape[2], c.shape[1], c.shape[3]
    n_h, H = w_p.shape[0], x.shape[2]
    if k.shape != (B, n_k, kv_cap, d_h) or c.shape != (B, n_c, kv_cap, d_l) or x.shape != (B, N, H) \
            or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h):
        raise ValueError("inconsistent operator tensor shapes")
    shape = _shape(B, N, H, n_h, n_q, n_k, n_c, d_h, d_l, _dtype_code(q), 1 if causal else 0, float(softmax_scale))
    if out is None:
        out = q.new_empty((B, N, n_h, d_h))
    if workspace is None:
        workspace = _workspace(prefill_chunk_workspace_bytes(shape, kv_len), q.device)
    st = lib().gta_prefill_chunk(ctypes.byref(shape), int(kv_len), int(kv_cap), _ptr(q), _ptr(k), _ptr(c), _ptr(x),
                                 _ptr(w_p), _ptr(w_g), _ptr(out), _ptr(workspace),
                                 workspace.nbytes, _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_prefill_chunk")
    return out


def _check_pools(k_pool, c_pool, block_table):
    if block_table.dtype != torch.int32 or block_table.get_device() != k_pool.get_device() \
            or not block_table.is_contiguous() or block_table.dim() != 2:
        raise ValueError("block_table must be a contiguous int32 [B, max_pages] tensor on the pools' device")
    n_pages, n_k, page_size, d_h = k_pool.shape
    n_c, d_l = c_pool.shape[1], c_pool.shape[3]
    if c_pool.shape != (n_pages, n_c, page_size, d_l):
        raise ValueError("inconsistent pool tensor shapes")
    return n_pages, page_size, block_table.shape[1]


def gta_prefill_chunk_paged(q, k_pool, c_pool, block_table, x, w_p, w_g, kv_len, *, causal=True, softmax_scale=0.0,
                            out=None, workspace=None, status_word=None, stream=None):
    """gta_prefill_chunk over a paged cache: the N queries are the last N of kv_len positions, whose keys and
    latents are read from k_pool [n_pages,n_k,page_size,d_h], c_pool [n_pages,n_c,page_size,d_l] through
    block_table int32 [B,max_pages]."""
    _check_tensors(q, k_pool, c_pool, x, w_p, w_g)
    n_pages, page_size, max_pages = _check_pools(k_pool, c_pool, block_table)
    B, n_q, N, d_h = q.shape
    n_k, n_c, d_l = k_pool.shape[1], c_pool.shape[1], c_pool.shape[3]
    n_h, H = w_p.shape[0], x.shape[2]
    if k_pool.shape[3] != d_h or block_table.shape[0] != B or x.shape != (B, N, H) \
            or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h):
        raise ValueError("inconsistent operator tensor shapes")
    shape = _shape(B, N, H, n_h, n_q, n_k, n_c, d_h, d_l, _dtype_code(q), 1 if causal else 0, float(softmax_scale))
    if out is None:
        out = q.new_empty((B, N, n_h, d_h))
    if workspace is None:
        workspace = _workspace(prefill_workspace_bytes(shape), q.device)
    st = lib().gta_prefill_chunk_paged(ctypes.byref(shape), int(kv_len), _ptr(q), _ptr(k_pool), _ptr(c_pool),
                                       _ptr(block_table), page_size, n_pages, max_pages, _ptr(x), _ptr(w_p),
                                       _ptr(w_g), _ptr(out), _ptr(workspace),
                                       workspace.nbytes, _ptr(status_word),
                                       _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_prefill_chunk_paged")
    return out


def gta_layer_prefill_paged(x, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, *, pos0=0, rope_base=10000.0, n_q,
                            softmax_scale=0.0, out=None, workspace=None, status_word=None, stream=None):
    """gta_layer_prefill over a paged cache: the chunk's keys and latents are written to the pages that
    block_table assigns to positions pos0 .. pos0+N-1, and the chunk attends everything up to there."""
    r = (_native or native()).layer_prefill_paged(x, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, int(pos0), rope_base,
                                                  n_q, softmax_scale, out, workspace, status_word, stream)
    if type(r) is int:
        raise GtaError(r, "gta_layer_prefill_paged")
    return r


def layer_prefill_workspace_bytes(shape: GtaShape) -> int:
    return int(lib().gta_layer_prefill_workspace_bytes(ctypes.byref(shape)))


def gta_layer_prefill(x, w_qkc, w_p, w_g, w_o, k_cache, c_cache, *, pos0=0, rope_base=10000.0, n_q, softmax_scale=0.0,
                      out=None, workspace=None, status_word=None, stream=None):
    """u[B, N, H] = the whole attention layer for a chunk that starts at position pos0: projections + RoPE, keys
    and latents written to rows pos0 .. pos0+N-1 of the caches, the operator, the output projection.
    x [B,N,H], w_qkc [H,(n_q+n_k)d_h+n_c d_l], w_o [n_h d_h,H], k_cache [B,n_k,S_cap,d_h], c_cache [B,n_c,S_cap,d_l]."""
    _check_tensors(x, w_qkc, w_p, w_g, w_o, k_cache, c_cache)
    B, N, H = x.shape
    n_h, d_l, d_h = w_p.shape
    n_k, s_cap, n_c = k_cache.shape[1], k_cache.shape[2], c_cache.shape[1]
    if k_cache.shape != (B, n_k, s_cap, d_h) or c_cache.shape != (B, n_c, s_cap, d_l) \
            or w_qkc.shape != (H, (n_q + n_k) * d_h + n_c * d_l) or w_g.shape != (H, n_h * d_h) \
            or w_o.shape != (n_h * d_h, H):
        raise ValueError("inconsistent layer tensor shapes")
    shape = _shape(B, N, H, n_h, n_q, n_k, n_c, d_h, d_l, _dtype_code(x), 1, float(softmax_scale))
    if out is None:
        out = x.new_empty((B, N, H))
    if workspace is None:
        workspace = _workspace(layer_prefill_workspace_bytes(shape), x.device)
    st = lib().gta_layer_prefill(ctypes.byref(shape), int(pos0), int(s_cap), float(rope_base), _ptr(x), _ptr(w_qkc),
                                 _ptr(w_p), _ptr(w_g), _ptr(w_o), _ptr(k_cache), _ptr(c_cache), _ptr(out),
                                 _ptr(workspace), workspace.nbytes, _ptr(status_word),
                                 _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_layer_prefill")
    return out


def layer_decode_workspace_bytes(shape: GtaShape, s_cap: int) -> int:
    return int(lib().gta_layer_decode_workspace_bytes(ctypes.byref(shape), int(s_cap)))


def gta_layer_decode(x_t, w_qkc, w_p, w_g, w_o, k_cache, c_cache, seq_lens, *, rope_base=10000.0, n_q,
                     softmax_scale=0.0, out=None, workspace=None, status_word=None, stream=None):
    """u[B, H] = one decode step of the whole attention layer: the new token of every sequence is projected,
    rotated at position seq_lens[b], written to the caches (seq_lens advances), attended and projected by w_o."""
    _check_tensors(x_t, w_qkc, w_p, w_g, w_o, k_cache, c_cache)
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != x_t.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the operator's device")
    B, H = x_t.shape
    n_h, d_l, d_h = w_p.shape
    n_k, s_cap, n_c = k_cache.shape[1], k_cache.shape[2], c_cache.shape[1]
    if k_cache.shape != (B, n_k, s_cap, d_h) or c_cache.shape != (B, n_c, s_cap, d_l) \
            or w_qkc.shape != (H, (n_q + n_k) * d_h + n_c * d_l) or w_g.shape != (H, n_h * d_h) \
            or w_o.shape != (n_h * d_h, H) or seq_lens.shape != (B,):
        raise ValueError("inconsistent layer tensor shapes")
    shape = _shape(B, 0, H, n_h, n_q, n_k, n_c, d_h, d_l, _dtype_code(x_t), 1, float(softmax_scale))
    if out is None:
        out = x_t.new_empty((B, H))
    if workspace is None:
        workspace = _workspace(layer_decode_workspace_bytes(shape, s_cap), x_t.device)
    st = lib().gta_layer_decode(ctypes.byref(shape), int(s_cap), float(rope_base), _ptr(x_t), _ptr(w_qkc), _ptr(w_p),
                                _ptr(w_g), _ptr(w_o), _ptr(k_cache), _ptr(c_cache), _ptr(seq_lens), _ptr(out),
                                _ptr(workspace), workspace.nbytes, _ptr(status_word),
                                _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_layer_decode")
    return out


def layer_decode_paged_workspace_bytes(shape: GtaShape, page_size: int, max_pages: int) -> int:
    return int(lib().gta_layer_decode_paged_workspace_bytes(ctypes.byref(shape), int(page_size), int(max_pages)))


def gta_layer_decode_paged(x_t, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, seq_lens, *, rope_base=10000.0,
                           n_q, softmax_scale=0.0, out=None, workspace=None, status_word=None, stream=None):
    """gta_layer_decode over a paged cache (pools and block table as in gta_decode_paged)."""
    r = (_native or native()).layer_decode_paged(x_t, w_qkc, w_p, w_g, w_o, k_pool, c_pool, block_table, seq_lens, rope_base,
                                                 n_q, softmax_scale, out, workspace, status_word, stream)
    if type(r) is int:
        raise GtaError(r, "gta_layer_decode_paged")
    return r


def _decode_shape(q, k_cache, c_cache, x_t, w_p, softmax_scale) -> GtaShape:
    B, n_q, d_h = q.shape
    return _shape(B, 0, x_t.shape[1], w_p.shape[0], n_q, k_cache.shape[1], c_cache.shape[1], d_h, c_cache.shape[3],
                  _dtype_code(q), 1, float(softmax_scale))


def decode_shape(q, k_cache, c_cache, x_t, w_p, causal=True, softmax_scale=0.0) -> GtaShape:
    B, n_q, d_h = q.shape
    return make_shape(batch=B, seq=0, d_model=x_t.shape[1], n_heads=w_p.shape[0], n_q=n_q,
                      n_k=k_cache.shape[1], n_c=c_cache.shape[1], d_h=d_h, d_l=c_cache.shape[3],
                      dtype=_dtype_code(q), causal=causal, softmax_scale=softmax_scale)


def gta_decode(q, k_cache, c_cache, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None, workspace=None,
               status_word=None, stream=None, stages=7):
    """out[B, n_h, d_h] = one decode step.  q [B,n_q,d_h], k_cache [B,n_k,S_cap,d_h],
    c_cache [B,n_c,S_cap,d_l], seq_lens int32 [B] (new token included), x_t [B,H]."""
    _check_tensors(q, k_cache, c_cache, x_t, w_p, w_g)
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != q.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the operator's device")
    B, n_q, d_h = q.shape
    s_cap = k_cache.shape[2]
    shape = _decode_shape(q, k_cache, c_cache, x_t, w_p, softmax_scale)
    n_h, d_l, H = shape.n_heads, shape.latent_dim, shape.d_model
    if k_cache.shape != (B, shape.n_k_groups, s_cap, d_h) or c_cache.shape != (B, shape.n_c_groups, s_cap, d_l) \
            or x_t.shape != (B, H) or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h) \
            or seq_lens.shape != (B,):
        raise ValueError("inconsistent operator tensor shapes")
    if out is None:
        out = q.new_empty((B, n_h, d_h))
    if workspace is None:
        workspace = _workspace(decode_workspace_bytes(shape, s_cap), q.device)
    args = (ctypes.byref(shape), _ptr(q), _ptr(k_cache), _ptr(c_cache), _ptr(seq_lens), s_cap, _ptr(x_t),
            _ptr(w_p), _ptr(w_g), _ptr(out), _ptr(workspace), workspace.nbytes,
            _ptr(status_word), _stream(stream))
    st = lib().gta_decode(*args) if stages == 7 else lib().gta_decode_stages(*args, stages)
    if st != GTA_OK:
        raise GtaError(st, "gta_decode")
    return out


def decode_hostcache_workspace_bytes(shape: GtaShape, s_cap: int) -> int:
    return int(lib().gta_decode_hostcache_workspace_bytes(ctypes.byref(shape), int(s_cap)))


def gta_decode_hostcache(q, k_cache, c_cache, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None, workspace=None,
                         status_word=None, stream=None):
    """gta_decode with k_cache / c_cache in page-locked HOST memory (pinned CPU tensors, read in place over the
    host link; CUDA tensors are accepted too); everything else lives on the device."""
    _check_tensors(q, x_t, w_p, w_g)
    for t in (k_cache, c_cache):
        if t.dtype != q.dtype or not t.is_contiguous():
            raise ValueError("the caches must be contiguous and of the operator's dtype")
        if t.device.type == "cpu" and not t.is_pinned():
            raise ValueError("a cache in host memory must be page-locked (tensor.pin_memory())")
        if t.device.type == "cuda" and t.device != q.device:
            raise ValueError("a cache in device memory must live on the operator's device")
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != q.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the operator's device")
    B, n_q, d_h = q.shape
    s_cap = k_cache.shape[2]
    shape = _decode_shape(q, k_cache, c_cache, x_t, w_p, softmax_scale)
    n_h, d_l, H = shape.n_heads, shape.latent_dim, shape.d_model
    if k_cache.shape != (B, shape.n_k_groups, s_cap, d_h) or c_cache.shape != (B, shape.n_c_groups, s_cap, d_l) \
            or x_t.shape != (B, H) or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h) \
            or seq_lens.shape != (B,):
        raise ValueError("inconsistent operator tensor shapes")
    if out is None:
        out = q.new_empty((B, n_h, d_h))
    if workspace is None:
        workspace = _workspace(decode_hostcache_workspace_bytes(shape, s_cap), q.device)
    st = lib().gta_decode_hostcache(ctypes.byref(shape), _ptr(q), _ptr(k_cache), _ptr(c_cache), _ptr(seq_lens), s_cap,
                                    _ptr(x_t), _ptr(w_p), _ptr(w_g), _ptr(out), _ptr(workspace),
                                    workspace.nbytes, _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_decode_hostcache")
    return out


def gta_decode_append(q, k_cache, c_cache, k_new, c_new, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None,
                      workspace=None, status_word=None, stream=None):
    """One decode step including the append of its token: k_new [B, n_k, 1, d_h] / c_new [B, n_c, 1, d_l] join the
    caches at row seq_lens[b], seq_lens advances, the new token's queries attend over everything."""
    r = (_native or native()).decode_append(q, k_cache, c_cache, k_new, c_new, seq_lens, x_t, w_p, w_g, softmax_scale, out,
                                            workspace, status_word, stream)
    if type(r) is int:
        raise GtaError(r, "gta_decode_append")
    return r


def gta_decode_static(q, k_cache, c_cache, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None,
                      status_word=None, stream=None):
    """gta_decode for callers that cannot allocate device memory (a pool that owns the whole
    device, a plug-in barred from the allocator, a loop that cannot take an allocation's device
    synchronisation): the split-KV scratch is a fixed STATIC_SCRATCH_BYTES array inside the
    library instead of a workspace tensor.  Pass `out`, and nothing is allocated at all.
    Raises GtaError(GTA_ERR_STATIC_SCRATCH) when the problem needs more than the array holds.
    Calls on one device share the array: order them on one stream."""
    _check_tensors(q, k_cache, c_cache, x_t, w_p, w_g)
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != q.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the operator's device")
    B, n_q, d_h = q.shape
    s_cap = k_cache.shape[2]
    shape = _decode_shape(q, k_cache, c_cache, x_t, w_p, softmax_scale)
    n_h, d_l, H = shape.n_heads, shape.latent_dim, shape.d_model
    if k_cache.shape != (B, shape.n_k_groups, s_cap, d_h) or c_cache.shape != (B, shape.n_c_groups, s_cap, d_l) \
            or x_t.shape != (B, H) or w_p.shape != (n_h, d_l, d_h) or w_g.shape != (H, n_h * d_h) \
            or seq_lens.shape != (B,):
        raise ValueError("inconsistent operator tensor shapes")
    if out is None:
        out = q.new_empty((B, n_h, d_h))
    st = lib().gta_decode_static(ctypes.byref(shape), _ptr(q), _ptr(k_cache), _ptr(c_cache), _ptr(seq_lens), s_cap,
                                 _ptr(x_t), _ptr(w_p), _ptr(w_g), _ptr(out), _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_decode_static")
    return out


def gta_cache_append(k_cache, c_cache, k_new, c_new, seq_lens, *, status_word=None, stream=None):
    """In place: rows k_new [B,n_k,n_new,d_h] / c_new [B,n_c,n_new,d_l] go behind seq_lens[b] in the
    caches and seq_lens advances by n_new.  A full sequence is skipped and raises *status_word."""
    _check_tensors(k_cache, c_cache, k_new, c_new)
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != k_cache.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the caches' device")
    B, n_k, s_cap, d_h = k_cache.shape
    n_c, d_l = c_cache.shape[1], c_cache.shape[3]
    n_new = k_new.shape[2]
    if c_cache.shape != (B, n_c, s_cap, d_l) or k_new.shape != (B, n_k, n_new, d_h) \
            or c_new.shape != (B, n_c, n_new, d_l) or seq_lens.shape != (B,):
        raise ValueError("inconsistent cache tensor shapes")
    n_q = n_k * n_c // _gcd(n_k, n_c)   # any common multiple serves: append ignores the query groups
    shape = _shape(B, 0, 8, n_q, n_q, n_k, n_c, d_h, d_l, _dtype_code(k_cache), 1, 0.0)
    st = lib().gta_cache_append(ctypes.byref(shape), _ptr(k_cache), _ptr(c_cache), s_cap, _ptr(k_new),
                                _ptr(c_new), n_new, _ptr(seq_lens), _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_cache_append")
    return seq_lens


def _check_paged(k_pool, c_pool, block_table, seq_lens):
    if block_table.dtype != torch.int32 or block_table.get_device() != k_pool.get_device() \
            or not block_table.is_contiguous() or block_table.dim() != 2:
        raise ValueError("block_table must be a contiguous int32 [B, max_pages] tensor on the pools' device")
    if seq_lens.dtype != torch.int32 or seq_lens.get_device() != k_pool.get_device() or not seq_lens.is_contiguous():
        raise ValueError("seq_lens must be a contiguous int32 tensor on the pools' device")
    n_pages, n_k, page_size, d_h = k_pool.shape
    n_c, d_l = c_pool.shape[1], c_pool.shape[3]
    if c_pool.shape != (n_pages, n_c, page_size, d_l) or seq_lens.shape != (block_table.shape[0],):
        raise ValueError("inconsistent pool tensor shapes")
    return n_pages, page_size, block_table.shape[1]


def decode_paged_workspace_bytes(shape: GtaShape, page_size: int, max_pages: int) -> int:
    return int(lib().gta_decode_paged_workspace_bytes(ctypes.byref(shape), int(page_size), int(max_pages)))


def gta_decode_paged(q, k_pool, c_pool, block_table, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None,
                     workspace=None, status_word=None, stream=None):
    """gta_decode over a paged cache.  k_pool [n_pages,n_k,page_size,d_h], c_pool [n_pages,n_c,page_size,d_l],
    block_table int32 [B,max_pages]: token t of sequence b is row t % page_size of page block_table[b, t // page_size]."""
    _check_tensors(q, k_pool, c_pool, x_t, w_p, w_g)
    n_pages, page_size, max_pages = _check_paged(k_pool, c_pool, block_table, seq_lens)
    B, n_q, d_h = q.shape
    shape = _decode_shape(q, k_pool, c_pool, x_t, w_p, softmax_scale)
    n_h, d_l, H = shape.n_heads, shape.latent_dim, shape.d_model
    if k_pool.shape[3] != d_h or x_t.shape != (B, H) or w_p.shape != (n_h, d_l, d_h) \
            or w_g.shape != (H, n_h * d_h) or block_table.shape[0] != B:
        raise ValueError("inconsistent operator tensor shapes")
    if out is None:
        out = q.new_empty((B, n_h, d_h))
    if workspace is None:
        workspace = _workspace(decode_paged_workspace_bytes(shape, page_size, max_pages), q.device)
    st = lib().gta_decode_paged(ctypes.byref(shape), _ptr(q), _ptr(k_pool), _ptr(c_pool), _ptr(block_table),
                                page_size, n_pages, max_pages, _ptr(seq_lens), _ptr(x_t), _ptr(w_p), _ptr(w_g),
                                _ptr(out), _ptr(workspace), workspace.nbytes,
                                _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_decode_paged")
    return out


def gta_cache_append_paged(k_pool, c_pool, block_table, k_new, c_new, seq_lens, *, status_word=None, stream=None):
    """gta_cache_append over a paged cache: the new rows go to the pages the block table names for positions
    seq_lens[b] .. seq_lens[b] + n_new - 1, and seq_lens advances by n_new."""
    _check_tensors(k_pool, c_pool, k_new, c_new)
    n_pages, page_size, max_pages = _check_paged(k_pool, c_pool, block_table, seq_lens)
    B = block_table.shape[0]
    n_k, d_h, n_c, d_l = k_pool.shape[1], k_pool.shape[3], c_pool.shape[1], c_pool.shape[3]
    n_new = k_new.shape[2]
    if k_new.shape != (B, n_k, n_new, d_h) or c_new.shape != (B, n_c, n_new, d_l):
        raise ValueError("inconsistent cache tensor shapes")
    n_q = n_k * n_c // _gcd(n_k, n_c)
    shape = _shape(B, 0, 8, n_q, n_q, n_k, n_c, d_h, d_l, _dtype_code(k_pool), 1, 0.0)
    st = lib().gta_cache_append_paged(ctypes.byref(shape), _ptr(k_pool), _ptr(c_pool), _ptr(block_table), page_size,
                                      n_pages, max_pages, _ptr(k_new), _ptr(c_new), n_new, _ptr(seq_lens),
                                      _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_cache_append_paged")
    return seq_lens


def gta_cache_append_fp8(k_codes, c_codes, k_scales, c_scales, k_new, c_new, seq_lens, *, status_word=None, stream=None):
    """Quantises k_new [B, n_k, n_new, d_h] / c_new [B, n_c, n_new, d_l] to e4m3 codes + per-row scales behind the
    live rows of the 8-bit caches and advances seq_lens."""
    r = (_native or native()).cache_append_fp8(k_codes, c_codes, k_scales, c_scales, k_new, c_new, seq_lens, status_word, stream)
    if type(r) is int:
        raise GtaError(r, "gta_cache_append_fp8")
    return r


def decode_fp8_path(shape: GtaShape, s_cap: int) -> int:
    """0 unsupported, 1 plain-ALU kernels, 2 streaming kernels."""
    return int(lib().gta_decode_fp8_path(ctypes.byref(shape), int(s_cap)))


def decode_fp8_workspace_bytes(shape: GtaShape, s_cap: int) -> int:
    return int(lib().gta_decode_fp8_workspace_bytes(ctypes.byref(shape), int(s_cap)))


def gta_decode_fp8(q, k_codes, c_codes, k_scales, c_scales, seq_lens, x_t, w_p, w_g, *, softmax_scale=0.0, out=None,
                   workspace=None, status_word=None, stream=None):
    """gta_decode over 8-bit caches (e4m3 codes + one fp32 scale per cached row)."""
    r = (_native or native()).decode_fp8(q, k_codes, c_codes, k_scales, c_scales, seq_lens, x_t, w_p, w_g, softmax_scale, out,
                                         workspace, status_word, stream)
    if type(r) is int:
        raise GtaError(r, "gta_decode_fp8")
    return r


def gqa_shape(*, batch, seq, n_heads, n_kv, d_h, dtype, causal=True, softmax_scale=0.0) -> GtaShape:
    """Shape of the comparison operators: only batch, seq, n_heads, n_k (key / value heads), d_h are read."""
    return make_shape(batch=batch, seq=seq, d_model=8, n_heads=n_heads, n_q=n_heads, n_k=n_kv, n_c=n_kv, d_h=d_h,
                      d_l=d_h, dtype=dtype, causal=causal, softmax_scale=softmax_scale)


def gta_ref_gqa_prefill(q, k, v, *, causal=True, softmax_scale=0.0, out=None, status_word=None, stream=None):
    """Grouped-query attention (App. B.3 of the paper), the comparison operator: q [B, n_h, N, d_h],
    k, v [B, n_kv, N, d_h] -> out [B, n_h, N, d_h]."""
    _check_tensors(q, k, v)
    B, n_h, N, d_h = q.shape
    n_kv = k.shape[1]
    if k.shape != (B, n_kv, N, d_h) or v.shape != k.shape:
        raise ValueError("inconsistent tensor shapes")
    shape = gqa_shape(batch=B, seq=N, n_heads=n_h, n_kv=n_kv, d_h=d_h, dtype=_dtype_code(q), causal=causal,
                      softmax_scale=softmax_scale)
    if out is None:
        out = q.new_empty((B, n_h, N, d_h))
    st = lib().gta_ref_gqa_prefill(ctypes.byref(shape), _ptr(q), _ptr(k), _ptr(v), _ptr(out), _ptr(status_word),
                                   _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_ref_gqa_prefill")
    return out


def gqa_decode_workspace_bytes(shape: GtaShape) -> int:
    return int(lib().gta_ref_gqa_decode_workspace_bytes(ctypes.byref(shape)))


def gta_ref_gqa_decode(q, k_cache, v_cache, seq_lens, *, softmax_scale=0.0, out=None, workspace=None, status_word=None,
                       stream=None):
    """One decode step of grouped-query attention: q [B, n_h, d_h], caches [B, n_kv, S_cap, d_h], seq_lens int32 [B]
    (counting the new token) -> out [B, n_h, d_h]."""
    _check_tensors(q, k_cache, v_cache)
    B, n_h, d_h = q.shape
    n_kv, s_cap = k_cache.shape[1], k_cache.shape[2]
    if k_cache.shape != (B, n_kv, s_cap, d_h) or v_cache.shape != k_cache.shape or seq_lens.shape != (B,) \
            or seq_lens.dtype != torch.int32:
        raise ValueError("inconsistent tensor shapes")
    shape = gqa_shape(batch=B, seq=0, n_heads=n_h, n_kv=n_kv, d_h=d_h, dtype=_dtype_code(q), softmax_scale=softmax_scale)
    if out is None:
        out = q.new_empty((B, n_h, d_h))
    if workspace is None:
        workspace = _workspace(gqa_decode_workspace_bytes(shape), q.device)
    st = lib().gta_ref_gqa_decode(ctypes.byref(shape), _ptr(q), _ptr(k_cache), _ptr(v_cache), _ptr(seq_lens), int(s_cap),
                                  _ptr(out), _ptr(workspace), workspace.nbytes,
                                  _ptr(status_word), _stream(stream))
    if st != GTA_OK:
        raise GtaError(st, "gta_ref_gqa_decode")
    return out


def _gcd(a, b):
    while b:
        a, b = b, a % b
    return a
