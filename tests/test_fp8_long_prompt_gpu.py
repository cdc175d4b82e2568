"""The quantising append of a long prompt (more elements per lane): the codes, scales and lengths of the same rows appended piece by
piece, bit for bit, at widths around the lanes' pieces, with rows of zeros, of elements that are no numbers and full caches."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2506_17286_b200 import build, binding
    build.build()
    binding.lib()
    return binding


CASES = [("bf16", 4, 1, 128, 512, 4, 1700), ("bf16", 1, 1, 64, 128, 9, 2051), ("bf16", 8, 1, 128, 1024, 3, 777), ("f32", 4, 2, 128, 512, 3, 1333),
         ("bf16", 3, 1, 48, 80, 8, 2500), ("f32", 2, 1, 256, 272, 4, 1100), ("bf16", 1, 1, 16, 1008, 2, 1700), ("bf16", 1, 1, 16, 1024, 3, 1100)]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}_dh{c[3]}_dl{c[4]}_n{c[6]}" for c in CASES])
def test_a_long_prompt_is_its_pieces(B, case):
    dt, n_k, n_c, d_h, d_l, nb, n = case
    assert nb * n * (n_k * d_h + n_c * d_l) >= 3 << 20
    T = torch.bfloat16 if dt == "bf16" else torch.float32
    g = torch.Generator("cuda").manual_seed(n)
    k = (torch.randn(nb, n_k, n, d_h, generator=g, device="cuda") * 3).to(T)
    c = torch.randn(nb, n_c, n, d_l, generator=g, device="cuda").to(T)
    k[0, 0, 5], c[0, 0, n - 1], c[1, 0, 7, d_l - 1], k[1, 0, n - 2, 3] = 0, 0, float("nan"), float("inf")
    cap = n + 8
    lens = torch.tensor([i % 7 for i in range(nb)], dtype=torch.int32, device="cuda")
    lens[nb - 1] = 9                                        # does not fit

    def caches():
        return [torch.full((nb, n_k, cap, d_h), 0xA5, dtype=torch.uint8, device="cuda"),
                torch.full((nb, n_c, cap, d_l), 0xA5, dtype=torch.uint8, device="cuda"),
                torch.full((nb, n_k, cap), -1.0, device="cuda"), torch.full((nb, n_c, cap), -1.0, device="cuda"), lens.clone()]

    whole, pieces = caches(), caches()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.gta_cache_append_fp8(*whole[:4], k, c, whole[4], status_word=status)
    assert int(status.item()) == B.GTA_ERR_CACHE_FULL
    keep = pieces[4][nb - 1].clone()
    for i in range(0, n, 61):
        pieces[4][nb - 1] = cap                             # (the pieces of that sequence would fit)
        B.gta_cache_append_fp8(*pieces[:4], k[:, :, i:i + 61].contiguous(), c[:, :, i:i + 61].contiguous(), pieces[4])
    pieces[4][nb - 1] = keep
    torch.cuda.synchronize()
    for a, b in zip(whole, pieces):
        assert torch.equal(a.view(torch.int32) if a.dtype == torch.float32 else a, b.view(torch.int32) if b.dtype == torch.float32 else b)


@pytest.mark.parametrize("case", [("bf16", 4, 1, 128, 512, 4096, 1), ("f32", 1, 1, 64, 128, 20000, 1), ("bf16", 8, 1, 128, 1024, 900, 2)],
                         ids=lambda c: f"{c[0]}_dl{c[4]}_B{c[5]}_n{c[6]}")
def test_few_rows_of_many_sequences_are_one_launch(B, case):
    """As many elements as a long prompt, a row or two of each sequence: one launch, and what parts of the batch give."""
    dt, n_k, n_c, d_h, d_l, nb, n = case
    assert nb * n * (n_k * d_h + n_c * d_l) >= 3 << 20
    T = torch.bfloat16 if dt == "bf16" else torch.float32
    g = torch.Generator("cuda").manual_seed(nb)
    k, c = torch.randn(nb, n_k, n, d_h, generator=g, device="cuda").to(T), torch.randn(nb, n_c, n, d_l, generator=g, device="cuda").to(T)
    whole = [torch.zeros(nb, n_k, 5, d_h, dtype=torch.uint8, device="cuda"), torch.zeros(nb, n_c, 5, d_l, dtype=torch.uint8, device="cuda"),
             torch.zeros(nb, n_k, 5, device="cuda"), torch.zeros(nb, n_c, 5, device="cuda"),
             torch.arange(nb, dtype=torch.int32, device="cuda") % 4]
    parts = [t.clone() for t in whole]
    B.gta_cache_append_fp8(*whole[:4], k, c, whole[4])
    assert B.last_launch_count() == 1
    for i in range(0, nb, 100):
        B.gta_cache_append_fp8(*(t[i:i + 100] for t in parts[:4]), k[i:i + 100], c[i:i + 100], parts[4][i:i + 100])
    torch.cuda.synchronize()
    for a, b in zip(whole, parts):
        assert torch.equal(a, b)
