"""The operator space entanglement entropy through the staged SVDs (global.cu: chi
>= 32 on FP64 contexts) at sizes around the stages' groups of 4, 32 and 64 rows, on
graded, rank-deficient and equal spectra, against the oracle's QR canonicalisation
and against the FP64 Jacobi passes alone (a sweep limit under 16, where those
converge within it).

Bound: the entropies' 1e-9 of the oracle comparison at chi = 128, 1e-12 between the
two routes (each squares the bond matrix: errors of 1e-16 of the largest p_k in up
to 130 of them, times |ln p| < 40)."""
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


def random_state(n, chi, kind):
    rng = np.random.default_rng(chi)
    dims = [1] + [min(chi, 4 ** min(p + 1, n - p - 1)) for p in range(n - 1)] + [1]
    grade = {"flat": 0.0, "graded": 20.0, "deficient": 3.0}[kind]
    tens = []
    for a, b in zip(dims, dims[1:]):
        t = rng.standard_normal((a, 4, b)) * np.exp(-grade / chi * np.arange(b)) / np.sqrt(4 * a)
        if kind == "deficient":
            t[a // 2:] = 0.0
        t[0, :, 0] = [0.7, 0.2, -0.1, 0.3]
        tens.append(t)
    return dims, tens


@pytest.mark.parametrize("chi,kind", [(31, "graded"), (32, "flat"), (33, "graded"), (50, "deficient"),
                                      (65, "flat"), (130, "graded")])
def test_osee(chi, kind):
    from paper_2203_05871_gb300 import Solver
    n = 9
    wl = W.random_model(n, W.chain_bonds(n), 3, chi_max=chi)
    dims, tens = random_state(n, chi, kind)
    st = tebd.MPOState(tens, [np.ones(d) for d in dims[1:-1]])
    got = []
    for limit in (100, 15):
        s = Solver(n, batch=1, chi_cap=chi, jacobi_max_sweeps=limit)
        s.build_gates(wl)
        s.set_state(0, dims, tens)
        got.append([s.osee(bond)[0] for bond in (3, 4)])
        converged = s.status()["status"][0] == 0
        assert converged or limit == 15
        s.close()
    want = [st.osee(bond) for bond in (3, 4)]
    assert np.abs(np.array(got[0]) - want).max() <= 1e-9, (got, want)
    assert not converged or np.abs(np.array(got[0]) - got[1]).max() <= 1e-12, got
