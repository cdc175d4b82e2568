"""The plain-ALU decode step with its append folded in, and its finish kernel's slabs: the same bits as append, then decode; full
caches are skipped and reported; lengths of the contractions around the slabs' edges, few and many sequences."""
import numpy as np
import pytest
import torch

from paper_2506_17286_b200 import inputs as I
from tests.parity_utils import assert_close, oracle_shape

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2506_17286_b200 import build, binding
    build.build()
    binding.lib()
    return binding


CASES = [  # dtype, batch, H, n_h, n_q, n_k, n_c, d_h, d_l, lengths, capacity
    ("f32", 4, 1280, 20, 5, 1, 1, 64, 128, [0, 31, 32, 64], 65),          # chunk edges, an empty sequence, a chunk's first token
    ("f32", 5, 1288, 6, 6, 3, 1, 40, 72, [9, 10, 3, 10, 0], 10),          # full caches; a slab of eight elements
    ("f32", 3, 2600, 4, 2, 1, 1, 256, 1024, [300, 1, 129], 301),          # three slabs of the gate
    ("f32", 20, 2600, 4, 2, 1, 1, 256, 1024, [(7 * i) % 90 for i in range(20)], 100),    # five, and two of the decoder
    ("f32", 33, 648, 20, 5, 1, 1, 64, 128, [(37 * i) % 200 for i in range(33)], 200),    # slabs of 640, a last CTA of one sequence
    ("bf16", 9, 1288, 6, 6, 3, 1, 40, 200, [(37 * i) % 90 for i in range(9)], 90),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}_B{c[1]}_H{c[2]}_dl{c[8]}" for c in CASES])
def test_fused_step_is_append_then_decode(B, oracle, case):
    dt, nb, H, n_h, n_q, n_k, n_c, d_h, d_l, lens, cap = case
    w = I.Workload("step", "decode", dt, nb, 0, H, n_h, n_q, n_k, n_c, d_h, d_l, seed=5)
    t = I.decode_inputs(w, device="cuda", s_cap=cap, seq_lens=lens)
    cap = t["k_cache"].shape[2]
    k_new = torch.randn(nb, n_k, 1, d_h, device="cuda").to(w.torch_dtype())
    c_new = torch.randn(nb, n_c, 1, d_l, device="cuda").to(w.torch_dtype())
    k1, c1, l1, s1 = t["k_cache"].clone(), t["c_cache"].clone(), t["seq_lens"].clone(), torch.zeros(1, dtype=torch.int32, device="cuda")
    k2, c2, l2, s2 = k1.clone(), c1.clone(), l1.clone(), s1.clone()
    B.gta_cache_append(k1, c1, k_new, c_new, l1, status_word=s1)
    want = B.gta_decode(t["q"], k1, c1, l1, t["x_t"], t["w_p"], t["w_g"], status_word=s1)
    got = B.gta_decode_append(t["q"], k2, c2, k_new, c_new, l2, t["x_t"], t["w_p"], t["w_g"], status_word=s2)
    torch.cuda.synchronize()
    for a, b in ((got, want), (k2, k1), (c2, c1), (l2, l1), (s2, s1)):
        assert torch.equal(a, b)
    assert int(s2.item() != 0) == int(any(n >= cap for n in lens))
    exact = oracle.decode(oracle_shape(w, seq=0), *(x.cpu() for x in (t["q"], k1, c1)), l1.cpu().numpy().astype(np.int32), cap,
                          *(t[n].cpu() for n in ("x_t", "w_p", "w_g")))
    assert_close(got, exact, w.torch_dtype(), "step")
