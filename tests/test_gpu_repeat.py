"""The entropies of a state that is left alone, asked for several times: bit for bit the
same.  Their Gram matrices come from symmetric products, where a 128-row tile on the
diagonal holds entries of both triangles; each must have one writer (bond dimensions
around the tiles' edges of 16, 32, 64 and 128)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()


@pytest.mark.parametrize("chi", [17, 63, 100, 130, 200])
def test_entropies_repeat_themselves(chi):
    from paper_2203_05871_gb300 import Solver
    n = 9
    wl = W.random_model(n, W.chain_bonds(n), 61, chi_max=chi)
    dims, tens = W.random_mpo_state(n, chi, seed=62, decay=0.05)
    s = Solver(n, batch=1, chi_cap=chi)
    s.build_gates(wl)
    s.set_state(0, dims, tens)
    first = None
    for _ in range(8):
        got = np.array([s.renyi2()[0]] + [s.osee(bond)[0] for bond in (3, 4)])
        assert np.all(np.isfinite(got))
        first = got if first is None else first
        assert np.array_equal(got, first)
    s.close()


@pytest.mark.parametrize("precision", ["FP64", "MIXED_TF32"])
def test_step_repeats_itself(precision):
    """A step from one state, several times, bit for bit: many CTAs work on a bond of 384
    rows, most of them discarded, and every CTA has to find the same limit below which
    rows do not count from norms that others are about to change."""
    import paper_2203_05871_gb300 as M
    n, chi = 10, 96
    wl = W.random_model(n, W.chain_bonds(n), 63, chi_max=chi, cutoff=1e-12)
    dims, tens = W.random_mpo_state(n, chi, seed=64, decay=0.05)
    s = M.Solver(n, batch=1, chi_cap=chi, precision=getattr(M, precision))
    s.build_gates(wl)
    first = None
    for _ in range(6):
        s.set_state(0, dims, tens)
        s.step(1)
        got = s.get_state(0)
        first = got if first is None else first
        assert got[0] == first[0]
        assert all(np.array_equal(a, b) for a, b in zip(got[1], first[1]))
    s.close()
