"""Contexts on a GPU whose memory is nearly taken: with room for a few workspace slots a
step and the entropies, which need two slots, run and agree with the same context on an
empty GPU, whatever the SVD's stages would need."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N, CHI = 8, 200
MAT = (4 * CHI) ** 2 * 8
# bytes of a slot without the SVD's stages: three matrices, the right vectors, norms
PLAIN = 3 * MAT + CHI * 4 * CHI * 8 + 2 * 4 * CHI * 8


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()
    return torch


def run(precision):
    from paper_2203_05871_gb300 import Solver
    wl = W.random_model(N, W.chain_bonds(N), 71, chi_max=CHI, cutoff=1e-12)
    s = Solver(N, batch=1, chi_cap=CHI, precision=precision)
    s.build_gates(wl)
    s.set_state(0, *W.random_mpo_state(N, CHI, seed=72, decay=0.03))
    out = [s.renyi2()[0], s.osee()[0]]
    s.step(1)
    out = np.concatenate([out, s.measure_1q(range(N), "Z")[0]])
    s.close()
    return out


@pytest.mark.parametrize("precision", ["FP64", "MIXED_BF16X3"])
@pytest.mark.parametrize("slots", [4, 9, 14])
def test_few_slots(torch, precision, slots):
    import paper_2203_05871_gb300 as M
    want = run(getattr(M, precision))   # every kernel is loaded now
    torch.cuda.empty_cache()
    per = PLAIN * (1 if precision == "FP64" else 4)   # (a mixed slot was three to four times that)
    room = N * CHI * 4 * CHI * 8 + slots * per + (64 << 20)   # the state, the slots, small buffers
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(max(0, free - room), dtype=torch.uint8, device="cuda")
    try:
        got = run(getattr(M, precision))
    finally:
        del fill
        torch.cuda.empty_cache()
    assert np.abs(got - want).max() <= (1e-9 if precision == "FP64" else 1e-5)
