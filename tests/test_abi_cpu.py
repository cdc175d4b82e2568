"""CPU-only checks of the C-ABI library: it loads, exports every declared symbol, and rejects
bad arguments on the host before anything could be launched (no GPU is touched)."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def B():
    from paper_2506_17286_b200 import build, binding
    build.build()
    binding.lib()
    return binding


def test_the_extension_of_another_torch_is_not_loaded(B, monkeypatch):
    """The extension is built against the C++ interfaces of one torch; after an upgrade it is missing, not stale."""
    assert B.native() is not None
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    monkeypatch.setattr(B, "_native", None)
    with pytest.raises(RuntimeError, match="not found"):
        B.native()


def test_the_binding_imports_on_a_torch_without_cuda():
    code = ("import torch\nfor n in ('_cuda_getCurrentRawStream', '_cuda_getDevice'):\n    delattr(torch._C, n)\n"
            "import paper_2506_17286_b200.binding")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "gta.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"GTA_API[^;(]*?\b(gta_\w+)\s*\(", text)))


def test_every_declared_symbol_is_exported(B):
    names = _declared_symbols()
    assert set(names) >= {"gta_prefill", "gta_decode", "gta_cache_append"}
    L = ctypes.CDLL(B.LIB_PATH)
    for n in names:
        assert hasattr(L, n), f"{n} declared in include/gta.h but not exported"
    assert set(names) == set(B.EXPORTS)


def test_version_and_status_strings(B):
    assert B.version() >= 100
    seen = {B.status_string(i) for i in range(9)}
    assert len(seen) == 9 and B.status_string(0) == "ok"
    assert B.status_string(99) == "unknown status"


def _shape(B, **kw):
    base = dict(batch=2, seq=64, d_model=64, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=32, d_l=64, dtype=B.GTA_BF16)
    base.update(kw)
    return B.make_shape(**base)


def test_workspace_sizes(B):
    s = _shape(B)
    assert B.prefill_workspace_bytes(s) >= 2 * 2 * 64 * 64 * 2
    assert B.prefill_workspace_bytes(s) % 256 == 0
    assert B.decode_workspace_bytes(s, 1000) > 0 and B.decode_workspace_bytes(s, 1000) % 256 == 0
    assert B.decode_workspace_bytes(s, 4000) > B.decode_workspace_bytes(s, 1000)
    assert B.prefill_workspace_bytes(_shape(B, n_q=3)) == 0       # n_q does not divide n_h
    assert B.decode_workspace_bytes(s, -1) == 0


@pytest.mark.parametrize("layer", [
    dict(n_heads=16, n_q=4, n_k=4, n_c=1, d_h=128, d_l=512, d_model=2048), dict(n_heads=20, n_q=5, n_k=1, n_c=1, d_h=64, d_l=128, d_model=1280),
    dict(n_heads=4, n_q=2, n_k=2, n_c=1, d_h=128, d_l=256, d_model=64), dict(),
    dict(n_heads=20, n_q=5, n_k=1, n_c=1, d_h=64, d_l=128, d_model=1280, dtype=0),
    dict(n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128, d_model=256, dtype=0)], ids=["h2048", "gta1b", "small", "plain_alu", "gta1b_f32", "tiny_f32"])
def test_prefill_workspace_never_falls_as_batch_or_length_grow(B, layer):
    """A buffer for the longest prompt of the largest batch serves every shorter one and every chunk."""
    sizes = [1, 2, 64, 128, 129, 255, 256, 257, 1000, 2048, 2304, 2305, 2560, 3500, 4096, 4097, 9000, 16384]
    for query in (B.prefill_workspace_bytes, B.layer_prefill_workspace_bytes):
        rows = [[query(_shape(B, batch=b, seq=n, **layer)) for n in sizes] for b in (1, 2, 3, 4, 7, 8, 32, 21845, 21846, 32767, 32768, 65535)]
        assert all(x > 0 for r in rows for x in r)
        for r in rows:
            assert r == sorted(r)
        for col in zip(*rows):
            assert list(col) == sorted(col)


def test_prefill_chunk_workspace(B):
    """Room for the fp32 attention's operands behind a longer cache; the plain query's size where there are none."""
    f32 = dict(n_heads=20, n_q=5, n_k=1, n_c=1, d_h=64, d_l=128, d_model=1280, dtype=0)
    for layer in (f32, dict(f32, dtype=1), dict(), dict(f32, d_l=72)):
        pieces = layer == f32
        for b in (1, 8, 40000):
            s = _shape(B, batch=b, seq=100, **layer)
            sizes = [B.prefill_chunk_workspace_bytes(s, kv) for kv in (100, 101, 128, 129, 1000, 100000)]
            assert sizes[0] == B.prefill_workspace_bytes(s) and sizes == sorted(sizes) and (sizes[-1] > sizes[0]) == pieces
            assert B.prefill_chunk_workspace_bytes(s, 99) == 0
            assert [B.prefill_chunk_workspace_bytes(_shape(B, batch=b, seq=n, **layer), 1000) for n in (1, 2, 100, 1000)] == \
                sorted(B.prefill_chunk_workspace_bytes(_shape(B, batch=b, seq=n, **layer), 1000) for n in (1, 2, 100, 1000))


GTA1B = dict(n_heads=20, n_q=5, n_k=1, n_c=1, d_h=64, d_l=128, d_model=1280)


@pytest.mark.parametrize("layer", [dict(GTA1B, dtype=0), dict(), dict(n_heads=6, n_q=6, n_k=3, d_h=40, d_l=200, d_model=96, dtype=0),
                                   dict(n_heads=32, n_q=8, n_k=8, d_h=128, d_l=1024, d_model=4096, dtype=0)])
def test_plain_decode_workspace_never_falls_as_batch_or_capacity_grow(B, layer):
    """A buffer for the largest batch serves what is left of it when sequences finish: contiguous caches, pages that the
    stream kernels do not take, caches in host memory, 8-bit caches."""
    caps = [1, 31, 32, 33, 64, 65, 200, 1000, 1024, 2999, 3000, 4096, 6000, 9473, 20000, 32768]
    fp8 = layer.get("d_h", 32) % 16 == 0 and layer.get("d_l", 64) % 16 == 0
    for query in (B.decode_workspace_bytes, lambda s, c: B.decode_paged_workspace_bytes(s, 8, -(-c // 8)),
                  B.decode_hostcache_workspace_bytes) + ((B.decode_fp8_workspace_bytes,) if fp8 else ()):
        rows = [[query(_shape(B, batch=b, **layer), c) for c in caps] for b in list(range(1, 41)) + [64, 75, 76, 96, 128, 300, 700]]
        assert all(x > 0 for r in rows for x in r)
        for r in rows:
            assert r == sorted(r)
        for col in zip(*rows):
            assert list(col) == sorted(col)


def test_plain_decode_runs_in_the_workspace_of_64_token_chunks(B):
    """Partial sums (fp32) and (maximum, sum) pairs of every chunk of 64 tokens, of 128 .. 256 where the batch has more than
    1184 chunks of fewer: that much, and a buffer for the largest batch, is never refused.  (Without a GPU the call ends at
    the device check, behind that of the workspace.)"""
    if torch.cuda.is_available():
        pytest.skip("the pointers are not device memory")
    L = B.lib()
    buf = (ctypes.c_char * 1024)()
    p = ctypes.c_void_p((ctypes.addressof(buf) + 255) & ~255)

    def status(batch, cap, ws):
        s = _shape(B, batch=batch, dtype=0, **GTA1B)
        return L.gta_decode(ctypes.byref(s), p, p, p, p, cap, p, p, p, p, p, ws, None, None)

    def least(batch, cap):
        chunk = min(256, max(64, -(-(batch * cap // 1184) // 64) * 64))
        n = batch * -(-cap // chunk) * 5
        return -(-n * 128 * 4 // 256) * 256 + -(-n * 8 // 256) * 256

    for cap in (1, 100, 3000, 4096, 9000):
        most = B.decode_workspace_bytes(_shape(B, batch=40, dtype=0, **GTA1B), cap)
        for batch in range(1, 41):
            assert status(batch, cap, most) != B.GTA_ERR_WORKSPACE
            assert status(batch, cap, least(batch, cap)) != B.GTA_ERR_WORKSPACE
            assert status(batch, cap, least(batch, cap) - 256) == B.GTA_ERR_WORKSPACE


def test_bad_arguments_are_rejected_on_the_host(B):
    L = B.lib()
    good = _shape(B)
    buf = (ctypes.c_char * 4096)()
    base = ctypes.addressof(buf)
    p = ctypes.c_void_p((base + 255) & ~255)          # an aligned (host) address: never dereferenced
    odd = ctypes.c_void_p(((base + 255) & ~255) + 2)
    args = [p] * 7

    def prefill(shape, a=args, ws=p, ws_bytes=1 << 40):
        return L.gta_prefill(ctypes.byref(shape), *a, ws, ws_bytes, None, None)

    assert L.gta_prefill(None, *args, p, 1 << 40, None, None) == B.GTA_ERR_INVALID_ARG
    assert prefill(good, [None] + args[1:]) == B.GTA_ERR_INVALID_ARG
    assert prefill(good, [odd] + args[1:]) == B.GTA_ERR_INVALID_ARG
    assert prefill(_shape(B, n_k=3)) == B.GTA_ERR_INVALID_ARG          # n_k must divide n_q
    assert prefill(_shape(B, n_c=4)) == B.GTA_ERR_INVALID_ARG          # n_c must divide n_q
    assert prefill(_shape(B, dtype=7)) == B.GTA_ERR_INVALID_ARG
    assert prefill(_shape(B, seq=-1)) == B.GTA_ERR_INVALID_ARG
    assert prefill(_shape(B, softmax_scale=-1.0)) == B.GTA_ERR_INVALID_ARG
    assert prefill(_shape(B, d_h=20)) == B.GTA_ERR_UNSUPPORTED         # rows must be 16-byte vectors
    assert prefill(_shape(B, d_h=512, d_l=512)) == B.GTA_ERR_UNSUPPORTED
    assert prefill(good, ws=None) == B.GTA_ERR_WORKSPACE
    assert prefill(good, ws_bytes=16) == B.GTA_ERR_WORKSPACE
    assert prefill(_shape(B, seq=0)) == B.GTA_OK                       # empty problem: no-op
    assert prefill(_shape(B, batch=0)) == B.GTA_OK

    def chunk(shape, kv_len, kv_cap):
        return L.gta_prefill_chunk(ctypes.byref(shape), kv_len, kv_cap, *args, p, 1 << 40, None, None)

    n = good.seq
    assert chunk(good, n - 1, n) == B.GTA_ERR_INVALID_ARG              # fewer keys than queries
    assert chunk(good, n + 8, n + 4) == B.GTA_ERR_INVALID_ARG          # more keys than the buffers hold
    assert L.gta_prefill_chunk(None, 8, 8, *args, p, 1 << 40, None, None) == B.GTA_ERR_INVALID_ARG
    assert chunk(_shape(B, seq=0), 16, 16) == B.GTA_OK                 # no queries: no-op

    def decode(shape, s_cap=128, ws=p, ws_bytes=1 << 40, lens=p):
        return L.gta_decode(ctypes.byref(shape), p, p, p, lens, s_cap, p, p, p, p, ws, ws_bytes, None, None)

    assert decode(good, s_cap=-1) == B.GTA_ERR_INVALID_ARG
    assert decode(good, lens=None) == B.GTA_ERR_INVALID_ARG
    assert decode(good, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert decode(_shape(B, d_l=4096)) == B.GTA_ERR_UNSUPPORTED
    assert decode(_shape(B, batch=0)) == B.GTA_OK

    def decode_host(shape, s_cap=128, ws=p, ws_bytes=1 << 40, lens=p):
        return L.gta_decode_hostcache(ctypes.byref(shape), p, p, p, lens, s_cap, p, p, p, p, ws, ws_bytes, None, None)

    assert decode_host(good, s_cap=-1) == B.GTA_ERR_INVALID_ARG
    assert decode_host(good, lens=None) == B.GTA_ERR_INVALID_ARG
    assert decode_host(good, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert decode_host(_shape(B, batch=0)) == B.GTA_OK
    assert B.decode_hostcache_workspace_bytes(good, 1000) > 0

    def append(shape, n_new=1, lens=p):
        return L.gta_cache_append(ctypes.byref(shape), p, p, 128, p, p, n_new, lens, None, None)

    assert append(good, n_new=-1) == B.GTA_ERR_INVALID_ARG
    assert append(good, lens=None) == B.GTA_ERR_INVALID_ARG
    assert append(good, n_new=0) == B.GTA_OK

    def decode_paged(shape, table=p, page_size=64, n_pages=10, max_pages=4, ws_bytes=1 << 40):
        return L.gta_decode_paged(ctypes.byref(shape), p, p, p, table, page_size, n_pages, max_pages, p, p, p, p, p,
                                  p, ws_bytes, None, None)

    assert decode_paged(good, table=None) == B.GTA_ERR_INVALID_ARG
    assert decode_paged(good, table=odd) == B.GTA_ERR_INVALID_ARG
    assert decode_paged(good, page_size=0) == B.GTA_ERR_INVALID_ARG
    assert decode_paged(good, n_pages=0) == B.GTA_ERR_INVALID_ARG
    assert decode_paged(good, max_pages=-3) == B.GTA_ERR_INVALID_ARG
    assert decode_paged(good, page_size=1 << 20, max_pages=1 << 12) == B.GTA_ERR_INVALID_ARG   # capacity over int32
    assert decode_paged(good, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert decode_paged(_shape(B, batch=0)) == B.GTA_OK
    assert B.decode_paged_workspace_bytes(good, 64, 4) == B.decode_workspace_bytes(good, 256)
    assert B.decode_paged_workspace_bytes(good, 0, 4) == 0

    def layer_prefill(shape, pos0=0, s_cap=128, base=10000.0, ws_bytes=1 << 40):
        return L.gta_layer_prefill(ctypes.byref(shape), pos0, s_cap, ctypes.c_float(base), p, p, p, p, p, p, p, p, p,
                                   ws_bytes, None, None)

    lay = _shape(B, d_model=128, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128)     # (2 + 2) 64 + 128 = 384 columns
    assert layer_prefill(lay, pos0=-1) == B.GTA_ERR_INVALID_ARG
    assert layer_prefill(lay, pos0=65) == B.GTA_ERR_INVALID_ARG           # 65 + 64 tokens do not fit 128 rows
    assert layer_prefill(lay, base=1.0) == B.GTA_ERR_INVALID_ARG
    assert layer_prefill(_shape(B, d_model=128, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128, causal=0)) \
        == B.GTA_ERR_INVALID_ARG
    assert layer_prefill(_shape(B, d_model=128, n_heads=4, n_q=2, n_k=1, n_c=1, d_h=64, d_l=128)) \
        == B.GTA_ERR_UNSUPPORTED                                          # 320 projection columns: no multiple of 128
    assert layer_prefill(_shape(B, d_model=128, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128, dtype=B.GTA_F32)) \
        == B.GTA_ERR_UNSUPPORTED
    assert layer_prefill(lay, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert layer_prefill(_shape(B, d_model=128, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128, seq=0)) == B.GTA_OK
    assert B.layer_prefill_workspace_bytes(lay) > B.prefill_workspace_bytes(lay)

    def layer_decode(shape, s_cap=128, base=10000.0, lens=p, ws_bytes=1 << 40):
        return L.gta_layer_decode(ctypes.byref(shape), s_cap, ctypes.c_float(base), p, p, p, p, p, p, p, lens, p, p,
                                  ws_bytes, None, None)

    assert layer_decode(lay, s_cap=0) == B.GTA_ERR_INVALID_ARG
    assert layer_decode(lay, base=0.5) == B.GTA_ERR_INVALID_ARG
    assert layer_decode(lay, lens=None) == B.GTA_ERR_INVALID_ARG
    assert layer_decode(lay, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert layer_decode(_shape(B, d_model=128, n_heads=4, n_q=2, n_k=2, n_c=1, d_h=64, d_l=128, batch=0)) == B.GTA_OK
    assert L.gta_layer_decode_paged(ctypes.byref(lay), None, 64, 10, 4, ctypes.c_float(1e4), p, p, p, p, p, p, p, p, p,
                                    p, 1 << 40, None, None) == B.GTA_ERR_INVALID_ARG
    assert L.gta_layer_decode_paged(ctypes.byref(lay), p, 0, 10, 4, ctypes.c_float(1e4), p, p, p, p, p, p, p, p, p,
                                    p, 1 << 40, None, None) == B.GTA_ERR_INVALID_ARG
    assert B.layer_decode_paged_workspace_bytes(lay, 64, 2) == B.layer_decode_workspace_bytes(lay, 128)

    def append_paged(shape, table=p, page_size=64, n_new=1):
        return L.gta_cache_append_paged(ctypes.byref(shape), p, p, table, page_size, 10, 4, p, p, n_new, p, None, None)

    assert append_paged(good, table=None) == B.GTA_ERR_INVALID_ARG
    assert append_paged(good, page_size=-1) == B.GTA_ERR_INVALID_ARG
    assert append_paged(good, n_new=-1) == B.GTA_ERR_INVALID_ARG
    assert append_paged(good, n_new=0) == B.GTA_OK

    def chunk_paged(shape, kv_len, table=p, page_size=64, n_pages=10, max_pages=4, ws_bytes=1 << 40):
        return L.gta_prefill_chunk_paged(ctypes.byref(shape), kv_len, p, p, p, table, page_size, n_pages, max_pages,
                                         p, p, p, p, p, ws_bytes, None, None)

    assert chunk_paged(good, n, table=None) == B.GTA_ERR_INVALID_ARG
    assert chunk_paged(good, n, table=odd) == B.GTA_ERR_INVALID_ARG
    assert chunk_paged(good, n, page_size=0) == B.GTA_ERR_INVALID_ARG
    assert chunk_paged(good, n - 1) == B.GTA_ERR_INVALID_ARG             # fewer keys than queries
    assert chunk_paged(good, 64 * 4 + 1) == B.GTA_ERR_INVALID_ARG        # more keys than the block table covers
    assert chunk_paged(good, n, ws_bytes=8) == B.GTA_ERR_WORKSPACE
    assert chunk_paged(_shape(B, seq=0), 16) == B.GTA_OK                 # no queries: no-op
    assert L.gta_prefill_chunk_paged(None, 8, p, p, p, p, 64, 10, 4, p, p, p, p, p, 1 << 40, None,
                                     None) == B.GTA_ERR_INVALID_ARG

    def layer_prefill_paged(shape, pos0=0, table=p, page_size=64, max_pages=2, base=10000.0, ws_bytes=1 << 40):
        return L.gta_layer_prefill_paged(ctypes.byref(shape), pos0, ctypes.c_float(base), p, p, p, p, p, p, p, table,
                                         page_size, 10, max_pages, p, p, ws_bytes, None, None)

    assert layer_prefill_paged(lay, table=None) == B.GTA_ERR_INVALID_ARG
    assert layer_prefill_paged(lay, page_size=-4) == B.GTA_ERR_INVALID_ARG
    assert layer_prefill_paged(lay, pos0=65) == B.GTA_ERR_INVALID_ARG     # 65 + 64 tokens do not fit two pages
    assert layer_prefill_paged(lay, base=1.0) == B.GTA_ERR_INVALID_ARG
    assert layer_prefill_paged(lay, ws_bytes=8) == B.GTA_ERR_WORKSPACE


def test_binding_rejects_cpu_tensors_and_missing_library(B, monkeypatch):
    import torch
    t = torch.zeros(1, 1, 8, 8)
    with pytest.raises(ValueError):
        B.gta_prefill(t, t, t, torch.zeros(1, 8, 8), torch.zeros(1, 8, 8), torch.zeros(8, 8))
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", os.path.join(ROOT, "does_not_exist.so"))
    with pytest.raises(RuntimeError, match="no CPU or PyTorch fallback"):
        B.lib()
