"""An instance's results do not depend on the other instances of its batch, bit for bit:
small bonds next to large ones take the route that they take alone (FP64 contexts: bonds
of at most 20 rows leave the SVD's stages out, entropies below chi 32 too), also when
the instance with the large bonds fails and shrinks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N, STEPS = 7, 2


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()


def solver(chis, wl, states, which, precision=None):
    """A context of the instances `which` of the model wl."""
    from paper_2203_05871_gb300 import FP64, Solver
    pick = {f: getattr(wl, f)[which] for f in ("h_x", "h_y", "h_z", "g0", "g1", "g2", "J", "Jz", "cutoff")}
    m = wl.with_(chi_max=np.array([chis[b] for b in which]), **pick)
    s = Solver(N, batch=len(which), chi_cap=max(chis), precision=FP64 if precision is None else precision)
    s.build_gates(m)
    for k, b in enumerate(which):
        s.set_state(k, *states[b])
    return s


def same(a, b):
    return a[0] == b[0] and all(np.array_equal(x, y) for x, y in zip(a[1], b[1]))


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("poison", [False, True])
@pytest.mark.parametrize("precision", ["FP64", "MIXED_TF32"])
def test_step(graph, poison, precision):
    import paper_2203_05871_gb300 as M
    precision = getattr(M, precision)
    chis = [64, 4, 5, 24]
    wl = W.random_model(N, W.chain_bonds(N), 401, batch=4, chi_max=64, cutoff=1e-12)
    states = [W.random_mpo_state(N, c, seed=402 + b) for b, c in enumerate(chis)]
    if poison:
        states[0][1][3][0, 1, 0] = np.nan
    s = solver(chis, wl, states, [0, 1, 2, 3], precision)
    s.step(STEPS, graph=graph, check=False)
    for b in (1, 2, 3):
        alone = solver(chis, wl, states, [b], precision)
        alone.step(STEPS, graph=graph)
        assert same(s.get_state(b), alone.get_state(0)), b
        alone.close()
    s.close()


def test_entropies():
    chis = [20, 40, 33]
    wl = W.random_model(N, W.chain_bonds(N), 411, batch=3, chi_max=40, cutoff=1e-12)
    states = [W.random_mpo_state(N, c, seed=412 + b, decay=0.1) for b, c in enumerate(chis)]
    s = solver(chis, wl, states, [0, 1, 2])
    got = np.array([s.renyi2()] + [s.osee(bond) for bond in range(N - 1)])
    s.close()
    for b in range(3):
        alone = solver(chis, wl, states, [b])
        want = np.array([alone.renyi2()[0]] + [alone.osee(bond)[0] for bond in range(N - 1)])
        assert np.array_equal(got[:, b], want), (b, got[:, b] - want)
        alone.close()
