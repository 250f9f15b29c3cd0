"""The operator space entanglement entropy of FP64 contexts against the oracle's QR
canonicalisation and SVD, on both sides of chi = 32 (the FP64 Jacobi pass alone, the
SVD's stages) and on flat, graded and rank-deficient spectra.  Bound: the Gram
matrices square the bond matrix, so each of up to 130 p_k carries 1e-16 of the
largest, times |ln p| < 40: 5e-13, and 1e-12 with the normalisation."""
import numpy as np
import pytest

import workloads as W
from oracle import tebd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()


@pytest.mark.parametrize("chi", [20, 31, 32, 50, 65, 130])
@pytest.mark.parametrize("decay,rank", [(0.0, 1.0), (0.08, 1.0), (0.02, 0.5)])
def test_osee(chi, decay, rank):
    from paper_2203_05871_gb300 import Solver
    n = 9
    wl = W.random_model(n, W.chain_bonds(n), 3, chi_max=chi)
    dims, tens = W.random_mpo_state(n, chi, seed=chi, decay=decay)
    if rank < 1.0:
        for t in tens:
            t[max(1, int(rank * t.shape[0])):] = 0.0
    s = Solver(n, batch=1, chi_cap=chi)
    s.build_gates(wl)
    s.set_state(0, dims, tens)
    st = tebd.MPOState(tens, [np.ones(d) for d in dims[1:-1]])
    bonds = range(2, 6)
    got = np.array([s.osee(b)[0] for b in bonds])
    want = np.array([st.osee(b) for b in bonds])
    assert s.status()["status"][0] == 0
    s.close()
    assert np.abs(got - want).max() <= 1e-12, (got, want)
