"""Traces, environments and all-pairs values (measure.cu) on set states whose
bonds are unequal and lie at the edges of the kernels' tiles: 1, below and above
the 8 CTAs of a cluster, 32 and 64 columns, 512 rows of a warp pass; three sites, an
odd and an even chain (the pairs meet at its middle), pairs listed in either order
and only some of them, instances with bonds of their own, both storages.

Reference: numpy in FP64 on the same tensors.  Bound: each value is a quotient of
two chain products, so its error is at most 4 n max(chi) 2^-53 of the same products
over absolute values, on both sides."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

COMP = {"X": 1, "Y": 2, "Z": 3}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    B.build()


def value(tens, at):
    v = np.ones(1)
    for p, t in enumerate(tens):
        v = v @ t[:, at.get(p, 0), :]
    return v[0]


def check(got, tens, at, n, chi):
    eps = 4 * n * chi * 2.0 ** -53
    ab = [np.abs(t) for t in tens]
    num, den = value(tens, at), value(tens, {})
    bound = eps * (value(ab, at) / abs(den) + abs(num) / den ** 2 * value(ab, {}))
    assert abs(got - num / den) <= 2 * bound, (at, got, num / den, bound)


@pytest.mark.parametrize("store", ["f64", "f32"])
@pytest.mark.parametrize("dims", [
    [1, 4, 1, 1], [1, 7, 9, 8, 1], [1, 4, 16, 33, 31, 4, 1], [1, 64, 65, 129, 40, 66, 64, 1],
    [1, 2, 512, 511, 3, 1]])
def test_values(dims, store):
    from paper_2203_05871_gb300 import STORE_F32, STORE_F64, Solver
    n, chi = len(dims) - 1, max(dims)
    wl = W.random_model(n, W.chain_bonds(n), 7, batch=2, chi_max=chi)
    s = Solver(n, batch=2, chi_cap=chi, storage=STORE_F32 if store == "f32" else STORE_F64)
    s.build_gates(wl)
    rng = np.random.default_rng(sum(dims))
    tens = []
    for b in range(2):
        d = dims if b == 0 else dims[::-1]
        t = [rng.standard_normal((x, 4, y)) * 0.3 / np.sqrt(x) for x, y in zip(d, d[1:])]
        for q in t:
            q[0, :, 0] = [1.0, 0.3, -0.2, 0.4]
        if store == "f32":
            t = [q.astype(np.float32).astype(np.float64) for q in t]
        s.set_state(b, d, t)
        tens.append(t)
    one = {c: s.measure_1q(range(n), c) for c in "XYZ"}
    some = s.measure_1q([n - 1, 0], "X")
    every = [(i, j) for i in range(n) for j in range(n) if i != j]
    few = [(n - 1, 0), (0, n // 2)]
    xz = s.measure_2q(every, "XZ", connected=False)
    yy = s.measure_2q(every, "YY", connected=True)
    part = s.measure_2q(few, "ZX", connected=False)
    for b in range(2):
        for c in "XYZ":
            for q in range(n):
                check(one[c][b][q], tens[b], {q: COMP[c]}, n, chi)
        assert some[b][0] == one["X"][b][n - 1] and some[b][1] == one["X"][b][0]
        for k, (i, j) in enumerate(every):
            check(xz[b][k], tens[b], {i: 1, j: 3}, n, chi)
            check(yy[b][k] + one["Y"][b][i] * one["Y"][b][j], tens[b], {i: 2, j: 2}, n, chi)
        for k, (i, j) in enumerate(few):
            check(part[b][k], tens[b], {i: 3, j: 1}, n, chi)
    s.close()
