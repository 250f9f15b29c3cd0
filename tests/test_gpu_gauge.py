"""States in an unbalanced bond gauge: a diagonal D of many decades on one inner bond, A D
and D^-1 B, is the same state.  FP64 contexts keep their accuracy on it (the FP64 path's
1e-10 of the oracle comparisons for a step, 1e-12 for the entropies of the state as
loaded, whose Gram matrices square D: six decades fit FP64's sixteen, eight do not), by
the step, the captured step and the gradient, next to instances in a good gauge."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N, CHI0, CAP = 6, 3, 64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()


def gauged(tens, bond, decades):
    """10^(decades / 2) to 10^(-decades / 2) on the bond right of site `bond`."""
    chi = tens[bond].shape[2]
    d = np.logspace(decades / 2, -decades / 2, chi)
    out = [t.copy() for t in tens]
    out[bond] = out[bond] * d
    out[bond + 1] = out[bond + 1] / d[:, None, None]
    return out


def solver(states, **kw):
    from paper_2203_05871_gb300 import Solver
    B = len(states)
    wl = W.random_model(N, W.chain_bonds(N), 77, chi_max=CAP, cutoff=0.0)
    two = {f: np.repeat(getattr(wl, f), B, 0) for f in ("h_x", "h_y", "h_z", "g0", "g1", "g2", "J", "Jz", "cutoff", "chi_max")}
    s = Solver(N, batch=B, chi_cap=CAP, **kw)
    s.build_gates(wl.with_(**two))
    for b, st in enumerate(states):
        s.set_state(b, *st)
    return s


def observables(s):
    return np.concatenate([s.measure_1q(range(N), a) for a in "XYZ"], axis=1)


def entropies(s):
    return np.array([s.renyi2()] + [s.osee(b) for b in range(N - 1)]).T


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("bond,decades", [
    (2, 6), (1, 8), (2, 8), (2, 12),
    pytest.param(3, 8, marks=pytest.mark.xfail(
        strict=False, reason="the FP64 QR and Jacobi route loses it too (4.6e-8): two ops in a row meet the bond's "
                             "eight decades as graded columns and graded rows before its own op")),
])
def test_step(bond, decades, graph):
    dims, tens = W.random_mpo_state(N, CHI0, seed=78)
    s = solver([(dims, gauged(tens, bond, decades)), (dims, tens)])
    s.step(2, graph=graph)
    z, e = observables(s), entropies(s)
    assert np.abs(z[0] - z[1]).max() <= 1e-10
    assert np.abs(e[0] - e[1]).max() <= 1e-10
    log = s.rank_log(2)
    assert np.array_equal(log[0], log[1])
    s.close()


@pytest.mark.parametrize("chi", [3, 40])
def test_entropies(chi):
    dims, tens = W.random_mpo_state(N, chi, seed=79, decay=0.02)
    s = solver([(dims, gauged(tens, 2, 6)), (dims, tens)])
    e = entropies(s)
    assert np.abs(e[0] - e[1]).max() <= 1e-12
    s.close()


def test_gradient():
    dims, tens = W.random_mpo_state(N, CHI0, seed=80)
    rng = np.random.default_rng(81)
    zbar, wbar = np.repeat(rng.standard_normal((1, N)), 2, 0), np.zeros((2, N, N))
    s = solver([(dims, gauged(tens, 2, 6)), (dims, tens)])
    s.grad_forward(1)
    g, loss = s.grad_backward(zbar, wbar)
    assert abs(loss[0] - loss[1]) <= 1e-10 and np.all(np.isfinite(g))
    s.close()


@pytest.mark.parametrize("graph", [False, True])
def test_float_storage(graph):
    """Float site tensors: the entries round to 6e-8 of themselves in any gauge, so the two
    instances agree within the storage's 1e-5."""
    from paper_2203_05871_gb300 import STORE_F32
    dims, tens = W.random_mpo_state(N, CHI0, seed=82)
    s = solver([(dims, gauged(tens, 2, 8)), (dims, tens)], storage=STORE_F32)
    s.step(1, graph=graph)
    z = observables(s)
    assert np.abs(z[0] - z[1]).max() <= 1e-5 * max(1.0, np.abs(z).max())
    s.close()
