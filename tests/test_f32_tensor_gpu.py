"""fp32 prefill on the tensor cores (three bf16 pieces per operand): tile edges, remainders and splits against torch in 64 bits,
the plain-ALU attention (a smallest workspace selects it) on elements that the pieces cannot hold, guard bands."""
import numpy as np
import pytest
import torch

from tests.parity_utils import Guarded

pytestmark = pytest.mark.gpu

# Pieces are exact (from 2^-110 on) and the products left out below 2^-24 of a product, 2^-26.5 rms; a sum of 64 products is cut at 2^-23 of its value up to
# eight times, sums are rounded to 2^-24 from there, an exponential is good to 2 ulp: 2.1e-7 measured (3.9e-7 the FMA chain).
REL, MAX = 8e-7, 4e-5


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2506_17286_b200 import build, binding
    build.build()
    binding.lib()
    return binding


def _inputs(B, N, cap, H, n_h, n_q, n_k, n_c, d_h, d_l, seed=0):
    gen = torch.Generator("cuda").manual_seed(seed)

    def r(*s, std=1.0):
        return torch.randn(s, generator=gen, device="cuda") * std
    return dict(q=r(B, n_q, N, d_h), k=r(B, n_k, cap, d_h), c=r(B, n_c, cap, d_l), x=r(B, N, H),
                w_p=r(n_h, d_l, d_h, std=d_l ** -0.5), w_g=r(H, n_h * d_h, std=H ** -0.5))


def _exact(t, kv, causal):
    q, k, c, x, w_p, w_g = (t[n].double() for n in ("q", "k", "c", "x", "w_p", "w_g"))
    B, n_q, N, d_h = q.shape
    k, c, n_h = k[:, :, :kv], c[:, :, :kv], w_p.shape[0]
    s = torch.einsum("bgtd,bgsd->bgts", q, k.repeat_interleave(n_q // k.shape[1], 1)) * d_h ** -0.5
    if causal:
        s = s.masked_fill(torch.ones(N, kv, device="cuda", dtype=torch.bool).triu(kv - N + 1), -float("inf"))
    lat = torch.einsum("bgts,bgsl->bgtl", s.softmax(-1), c.repeat_interleave(n_q // c.shape[1], 1))
    y = torch.einsum("bhtl,hld->bthd", lat.repeat_interleave(n_h // n_q, 1), w_p)
    return y * torch.sigmoid(x @ w_g).reshape(B, N, n_h, -1)


def _run(G, t, kv, causal, least=False):
    B, n_q, N, d_h = t["q"].shape
    n_h, d_l = t["w_p"].shape[:2]
    shape = G.make_shape(batch=B, seq=N, d_model=t["x"].shape[2], n_heads=n_h, n_q=n_q, n_k=t["k"].shape[1],
                         n_c=t["c"].shape[1], d_h=d_h, d_l=d_l, dtype=torch.float32)
    plain = (4 * B * n_q * N * d_l + 255) // 256 * 256
    room = plain if least else G.prefill_chunk_workspace_bytes(shape, kv)
    ws, out = Guarded((room,), torch.uint8), Guarded((B, N, n_h, d_h), torch.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.gta_prefill_chunk(t["q"], t["k"], t["c"], t["x"], t["w_p"], t["w_g"], kv, causal=causal, workspace=ws.t, out=out.t,
                        status_word=status)
    torch.cuda.synchronize()
    ws.check("workspace"); out.check("out")
    assert int(status.item()) == 0
    return out.t


CASES = [  # B, N, kv, cap, H, n_h, n_q, n_k, n_c, d_h, d_l, causal
    (1, 192, 192, 192, 1280, 20, 5, 1, 1, 64, 128, True),       # plain decoder behind the tensor-core attention
    (2, 257, 257, 257, 200, 20, 5, 1, 1, 64, 128, True),        # a row past two row tiles; H not a multiple of 32; four CTAs a tile
    (1, 1000, 1000, 1000, 64, 16, 4, 2, 2, 64, 256, True),      # two latent groups, two slices; one key tile of 40 rows at the end
    (3, 1025, 1025, 1025, 96, 10, 5, 1, 1, 64, 128, True),      # a row past a pair's tile; 128 columns a map; 256 | 3075 does not hold
    (2, 1500, 1500, 1500, 1280, 20, 5, 1, 1, 64, 128, True),    # 256-column blocks, two CTAs a row tile
    (2, 700, 700, 700, 72, 18, 6, 3, 1, 64, 128, True),         # 192 columns a map: the second block is half empty
    (1, 300, 300, 320, 256, 20, 5, 1, 1, 64, 384, False),       # not causal, three slices, rows behind the keys in the cache
    (2, 130, 777, 800, 256, 20, 5, 1, 1, 64, 128, True),        # a chunk behind a longer cache
    (1, 5, 300, 300, 64, 2, 2, 1, 1, 64, 128, True),            # fewer rows than a warp
    (5, 333, 333, 333, 64, 8, 4, 4, 1, 128, 72, True),          # plain attention in front of the tensor-core decoder; d_l = 72
    (9, 1024, 1024, 1024, 32, 4, 2, 2, 1, 64, 128, True),       # more than one wave, one CTA a row tile
]


@pytest.mark.parametrize("case", CASES, ids=[f"B{c[0]}_N{c[1]}_kv{c[2]}_H{c[4]}_dh{c[9]}_dl{c[10]}" for c in CASES])
def test_against_64_bits(G, case):
    B, N, kv, cap, H, n_h, n_q, n_k, n_c, d_h, d_l, causal = case
    t = _inputs(B, N, cap, H, n_h, n_q, n_k, n_c, d_h, d_l)
    t["k"][:, :, kv:], t["c"][:, :, kv:] = float("nan"), float("inf")
    got, want = _run(G, t, kv, causal).double(), _exact(t, kv, causal)
    err = got - want
    rms = want.pow(2).mean().sqrt()
    assert torch.isfinite(got).all()
    assert float(err.norm() / want.norm()) <= REL and float((err.abs() / torch.maximum(want.abs(), rms)).max()) <= MAX


SHORT = [  # both stages in one plain-ALU kernel: row and key tile edges, k-blocks of the gate, a chunk, heads of a map
    (1, 1, 1, 1, 8, 2, 2, 1, 1, 64, 128, True), (2, 16, 16, 16, 72, 3, 1, 1, 1, 64, 128, True),
    (1, 17, 17, 17, 1280, 20, 5, 1, 1, 64, 128, True), (2, 128, 128, 128, 256, 4, 2, 2, 2, 64, 128, True),
    (1, 129, 129, 140, 256, 4, 2, 2, 1, 64, 128, False), (1, 191, 191, 191, 200, 4, 2, 1, 1, 64, 128, True),
    (3, 33, 190, 200, 136, 6, 2, 1, 1, 64, 128, True),
]


@pytest.mark.parametrize("case", SHORT, ids=[f"B{c[0]}_N{c[1]}_kv{c[2]}_H{c[4]}" for c in SHORT])
def test_short_prompts_against_64_bits(G, case):
    test_against_64_bits(G, case)


# (sequences, rows, keys) of a layer with four maps: which side of the rule, one launch fewer on the plain one (no pieces of K and C)
@pytest.mark.parametrize("case", [(256, 1, 1, 2), (40, 95, 95, 2), (40, 96, 96, 3), (100, 3, 300, 2), (100, 3, 640, 3), (40, 3, 300, 3), (100, 64, 300, 3)])
def test_few_rows_of_many_sequences_stay_on_the_plain_kernel(G, case):
    B, N, kv, launches = case
    test_against_64_bits(G, (B, N, kv, kv, 64, 4, 4, 1, 1, 64, 128, True))
    assert G.last_launch_count() == launches


def test_more_key_and_latent_groups_than_a_grid_dimension(G):
    """520 sequences x (128 key groups + 1): more than 65535 of them are cut into pieces, the last like the first."""
    t = _inputs(520, 96, 96, 8, 128, 128, 128, 1, 64, 128)
    for n in ("q", "k", "c", "x"):
        t[n][519] = t[n][0]
    got = _run(G, t, 96, True)
    assert G.last_launch_count() == 3 and torch.equal(got[519], got[0])
    few = {n: v[518:].contiguous() if n in ("q", "k", "c", "x") else v for n, v in t.items()}
    want = _exact(few, 96, True)
    assert float((got[518:].double() - want).norm() / want.norm()) <= REL


def test_short_prompt_rows_before_an_odd_element_keep_their_bits(G):
    t = _inputs(1, 100, 100, 256, 4, 2, 2, 1, 64, 128)
    want = _run(G, t, 100, True).clone()
    t["k"][:, :, 41:], t["c"][:, :, 41:] = float("nan"), float("inf")
    assert torch.equal(_run(G, t, 100, True)[:, :41], want[:, :41])


def _times_out(G, t, N):
    """With the first hand-over withheld and a limit of 2 ms the call comes back with GTA_ERR_TIMEOUT, and the next ordinary call gives
    bit for bit what the call before gave."""
    want = _run(G, t, N, True).clone()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.debug_attention_wait(limit_ns=2_000_000, withhold_first_arrive=True)
    try:
        G.gta_prefill(t["q"], t["k"], t["c"], t["x"], t["w_p"], t["w_g"], status_word=status)
        torch.cuda.synchronize()
        assert int(status.item()) == G.GTA_ERR_TIMEOUT
    finally:
        G.debug_attention_wait()
    assert torch.equal(_run(G, t, N, True).view(torch.int32), want.view(torch.int32))


@pytest.mark.parametrize("N", [100, 170])       # one key tile; two, the second of which must not be asked for any more
def test_a_wait_that_runs_out_unwinds_the_short_prompt_kernel(G, N):
    _times_out(G, _inputs(1, N, N, 256, 4, 2, 2, 1, 64, 128), N)


# one CTA a row tile and four, tiles in flight when the wait runs out; the tensor-core decoder behind plain attention (d_l = 72)
@pytest.mark.parametrize("case", [(9, 1024, 32, 4, 2, 2, 1, 64, 128), (1, 333, 64, 20, 5, 1, 1, 64, 128), (1, 192, 64, 4, 2, 2, 1, 64, 128),
                                  (5, 333, 64, 8, 4, 4, 1, 128, 72)])
def test_a_wait_that_runs_out_unwinds_the_tensor_core_kernels(G, case):
    B, N, H, n_h, n_q, n_k, n_c, d_h, d_l = case
    _times_out(G, _inputs(B, N, N, H, n_h, n_q, n_k, n_c, d_h, d_l), N)


def test_a_long_attention_kernel_does_not_run_out_the_decoders_waits(G):
    """700 rows behind 40000 keys take some 200 us, four CTAs a row tile; the decoder kernel starts beside them, and its waits may
    take 50 us here."""
    t = _inputs(1, 700, 40000, 64, 20, 5, 1, 1, 64, 128)
    want = _run(G, t, 40000, True).clone()
    G.debug_attention_wait(limit_ns=50_000)
    try:
        got = _run(G, t, 40000, True)
    finally:
        G.debug_attention_wait()
    assert torch.equal(got, want)


@pytest.mark.parametrize("size", [1e-30, 1e15])
def test_range_of_the_pieces(G, size):
    """Latents and decoder weights far from one: the pieces have fp32's exponents."""
    t = _inputs(1, 300, 300, 64, 20, 5, 1, 1, 64, 128)
    t["c"] *= size
    t["w_p"] *= size if size > 1 else 1e3
    got, want = _run(G, t, 300, True).double(), _exact(t, 300, True)
    assert float((got - want).norm() / want.norm()) <= REL


@pytest.mark.parametrize("small,large", [("c", "w_p"), ("w_p", "c"), ("x", "w_g"), ("w_g", "x"), ("q", "k"), ("k", "q")])
def test_operands_too_small_for_pieces(G, small, large):
    """At 1e-36 three pieces hold 15 bits of an element, and the other operand makes ordinary numbers of it: done again with FMAs, in
    one chain of up to 300 (2^-24 of the sum at each step, at random: 6e-8 x 17)."""
    t = _inputs(1, 300, 300, 64, 20, 5, 1, 1, 64, 128)
    t[small] *= 1e-36
    t[large] *= 1e36
    got, want = _run(G, t, 300, True).double(), _exact(t, 300, True)
    assert float((got - want).norm() / want.norm()) <= 2 * REL


def test_few_small_elements_and_rows(G):
    """Rows of the result that are made of small elements alone keep their precision; a few of them in ordinary rows and columns
    cost none."""
    t = _inputs(1, 300, 300, 64, 20, 5, 1, 1, 64, 128)
    t["c"][:, :, :3] *= 1e-36
    t["w_p"][3, :, 40:44] *= 1e-35              # (results of 1e-36: below 1.2e-38 a result, and every sum on the way, ends at 2^-149)
    t["x"][:, 50] *= 1e-36
    for n in ("q", "k", "c", "x", "w_p", "w_g"):
        t[n].view(-1)[::1009] *= 1e-37
    got, want = _run(G, t, 300, True).double(), _exact(t, 300, True)
    err = (got - want).norm(dim=-1) / want.norm(dim=-1)           # of each token and head
    tail = slice(3, None)                       # (1e-36 x 1e-35 is nothing)
    err[:, tail, 3] = (got - want)[:, tail, 3, 40:44].norm(dim=-1) / want[:, tail, 3, 40:44].norm(dim=-1)
    assert float(err.max()) <= 8 * REL          # (a head's 64 outputs, or four of them, against a row's latents)


def test_workspace_of_a_chunk_behind_a_longer_cache(G):
    """With the size that its query gives, or without a workspace, the chunk takes the tensor cores; a byte less and it takes the plain
    kernel, in place."""
    B, N, kv = 2, 130, 777
    t = _inputs(B, N, 800, 256, 20, 5, 1, 1, 64, 128)
    shape = G.make_shape(batch=B, seq=N, d_model=256, n_heads=20, n_q=5, n_k=1, n_c=1, d_h=64, d_l=128, dtype=torch.float32)
    args = (t["q"], t["k"], t["c"], t["x"], t["w_p"], t["w_g"], kv)
    want, plain = _run(G, t, kv, True).clone(), _run(G, t, kv, True, least=True).clone()
    assert G.last_launch_count() == 2 and not torch.equal(want, plain)
    assert torch.equal(G.gta_prefill_chunk(*args), want) and G.last_launch_count() == 3
    for room in (G.prefill_chunk_workspace_bytes(shape, kv) - 1, G.prefill_workspace_bytes(shape)):
        ws = Guarded((room,), torch.uint8)
        assert torch.equal(G.gta_prefill_chunk(*args, workspace=ws.t), plain) and G.last_launch_count() == 2
        ws.check("workspace")


@pytest.mark.parametrize("case", [(2, 500, 500, 64, 20, 5, 1, 1, True), (1, 300, 600, 64, 4, 2, 2, 1, False), (3, 1025, 1025, 96, 10, 5, 1, 1, True)])
@pytest.mark.parametrize("what,where,value", [("c", (slice(None), slice(None), 0, 1), float("inf")), ("k", (slice(None), slice(None), 2, 5), -float("inf")),
                                              ("x", (slice(None), slice(None), 3), float("inf")), ("w_g", (3, slice(None)), float("inf")),
                                              ("w_p", (1, slice(None), 7), float("inf"))], ids=["c", "k", "x", "w_g", "w_p"])
def test_infinities_that_every_row_or_column_sees(G, case, what, where, value):
    """All rows of all tiles are done again, in blocks of rows with remainders: against the plain-ALU attention, and torch for the rest."""
    B, N, kv, H, n_h, n_q, n_k, n_c, causal = case
    t = _inputs(B, N, kv, H, n_h, n_q, n_k, n_c, 64, 128)
    t[what][where] = value
    got = _run(G, t, kv, causal)
    if what in ("c", "k"):
        want = _run(G, t, kv, causal, least=True)
        assert torch.equal(torch.isnan(got), torch.isnan(want)) and torch.equal(torch.isinf(got), torch.isinf(want))
        ok = torch.isfinite(want)
        assert not ok.any() or float((got - want)[ok].double().norm() / want[ok].double().norm()) <= 2 * REL
    else:
        torch.testing.assert_close(got, _exact(t, kv, causal).float(), rtol=1e-4, atol=1e-5, equal_nan=True)


BAD = [("q", (0, 1, 40, 3), float("nan")), ("q", (0, 0, 299, 0), float("inf")), ("k", (0, 0, 130, 5), float("inf")),
       ("k", (0, 0, 299, 63), float("nan")), ("c", (0, 0, 70, 127), float("nan")), ("c", (0, 0, 290, 1), -float("inf")),
       ("c", (0, 0, 5, 1), 3.4e38), ("x", (0, 17, 9), float("inf")), ("x", (0, 299, 63), float("nan")),
       ("w_g", (3, 700), -float("inf")), ("w_p", (7, 11, 2), float("nan")), ("x", (0, 30, 0), 3.4e38)]


@pytest.mark.parametrize("what,where,value", BAD, ids=[f"{w}_{v}_{p[-2]}" for w, p, v in BAD])
def test_elements_that_the_pieces_cannot_hold(G, what, where, value):
    """They reach the rows and columns that see them, and no others."""
    t = _inputs(1, 300, 300, 64, 20, 5, 1, 1, 64, 128)
    t[what][where] = value
    got, plain, want = _run(G, t, 300, True), _run(G, t, 300, True, least=True), _exact(t, 300, True)
    if what in ("q", "k", "c"):         # the plain-ALU attention, whose masked rows do not see the element
        assert torch.equal(torch.isnan(got), torch.isnan(plain)) and torch.equal(torch.isinf(got), torch.isinf(plain))
        ok = torch.isfinite(got)
        assert float((got - plain)[ok].double().norm() / plain[ok].double().norm()) <= 2 * REL
    else:
        torch.testing.assert_close(got, want.float(), rtol=1e-4, atol=1e-5, equal_nan=True)
