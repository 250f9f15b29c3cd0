"""The SVD finish through the rows' Gram matrix (refine.cu) against the Jacobi
passes alone: a sweep limit under 16 leaves every SVD to the latter (FP64 path:
the FP64 Jacobi pass on the rows of R).  Sizes at the edges of the kernels'
tiles (rows of 4 to 4 chi elements, 64 and 128 wide product tiles, one row),
rank-deficient and exactly degenerate bond matrices (graph states), and spectra
graded over 14 decades.

Bounds: the parity tests' 1e-10 (FP64) and 1e-5 (mixed) on ratios of traces,
relative to their size.  Both sides run at the default side's ranks."""
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


def observables(s, n):
    pairs = [(i, j) for i in range(n) for j in range(i + 1, n)]
    return np.concatenate([s.measure_1q(range(n), c)[0] for c in "XYZ"] +
                          [s.measure_2q(pairs, "ZZ", connected=False)[0]])


def both(wl, chi, start, steps, **kw):
    from paper_2203_05871_gb300 import Solver
    out, ranks = [], None
    for limit in (100, 15):
        s = Solver(wl.n, batch=1, chi_cap=chi, jacobi_max_sweeps=limit, **kw)
        s.build_gates(wl)
        start(s)
        s.force_ranks(ranks)
        s.step(steps)
        if ranks is None:
            ranks = s.rank_log(steps)
        assert s.status()["status"][0] == 0
        out.append(observables(s, wl.n))
        s.close()
    return out


def precision_of(name):
    from paper_2203_05871_gb300 import FP64, MIXED_BF16X3, MIXED_TF32
    return {"fp64": (FP64, 1e-10), "tf32": (MIXED_TF32, 1e-5), "bf16": (MIXED_BF16X3, 1e-5)}[name]


@pytest.mark.parametrize("precision", ["fp64", "tf32", "bf16"])
@pytest.mark.parametrize("chi,grade", [(1, 0.0), (2, 1.0), (7, 2.0), (16, 4.0), (33, 32.0), (64, 5.0)])
def test_step_matches_the_jacobi_passes(chi, grade, precision):
    prec, tol = precision_of(precision)
    n = 7
    wl = W.random_model(n, W.ring_bonds(n), 900 + chi, chi_max=chi, cutoff=0.0, dt=0.05)
    rng = np.random.default_rng(chi)
    dims = [1] + [min(chi, 4 ** min(p + 1, n - p - 1)) for p in range(n - 1)] + [1]
    tens = [rng.standard_normal((a, 4, b)) * np.exp(-grade / chi * np.arange(b)) / np.sqrt(4 * a)
            for a, b in zip(dims, dims[1:])]
    for t in tens:   # a leading product state: traces are well conditioned
        t[0, :, 0] = [0.7, 0.2, -0.1, 0.3]
    a, b = both(wl, chi, lambda s: s.set_state(0, dims, tens), 1, precision=prec)
    assert np.all(np.isfinite(a))
    assert np.all(np.abs(a - b) <= tol * np.maximum(1.0, np.abs(b))), np.abs(a - b).max()


@pytest.mark.parametrize("precision", ["fp64", "tf32"])
def test_rank_deficient_and_degenerate(precision):
    """From a graph state (every kept Schmidt value equal, the rest exactly zero)
    and from a product state (one non-zero singular value)."""
    prec, tol = precision_of(precision)
    n = 6
    wl = W.random_model(n, W.chain_bonds(n), 77, chi_max=16, cutoff=1e-12, dt=0.05)
    for pairs in ([(0, 1), (1, 2), (2, 3), (3, 4), (4, 5)], []):
        a, b = both(wl, 16, lambda s: s.init_graph_state(pairs), 2, precision=prec)
        assert np.abs(a - b).max() <= tol


@pytest.mark.parametrize("chi", [96, 160])
@pytest.mark.parametrize("order", ["wide", "tall"])
def test_mixed_right_vectors_are_orthonormal(chi, order):
    """The right sites of a mixed step's last layer are the right singular vectors of their
    bonds.  The refinement leaves pairs of rows at a tenth of the mixed tolerance, 1e-11,
    at most, the rotations that become the vectors of a transposed bond are orthogonal to
    the third order of the FP32 pass's defect (1e-5: 1e-15), and the products add 2^-46 per
    term and sqrt(c) of them (4e-13): 2e-11 covers both."""
    from paper_2203_05871_gb300 import MIXED_TF32, Solver
    n = 9
    wl = W.random_model(n, W.chain_bonds(n), 91, chi_max=chi, cutoff=1e-14, dt=0.02)
    dims, tens = W.random_mpo_state(n, chi, seed=92, decay=0.04)
    if order == "tall":   # mirrored: the bonds that were wide are tall
        tens = [t.transpose(2, 1, 0) for t in tens[::-1]]
        tens = [np.ascontiguousarray(t) for t in tens]
        dims = [1] + [t.shape[2] for t in tens]
    s = Solver(n, batch=1, chi_cap=chi, precision=MIXED_TF32)
    s.build_gates(wl)
    s.set_state(0, dims, tens)
    s.step(1)
    _, out = s.get_state(0)
    worst = 0.0
    for p in (1, 3, 5, 7):
        v = out[p].reshape(out[p].shape[0], -1)
        worst = max(worst, np.abs(v @ v.T - np.eye(len(v))).max())
    assert worst <= 2e-11, worst
    s.close()
