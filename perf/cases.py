"""Performance cases of the MPO Lindblad solver: what a program that uses the
package calls, over the sizes it is used at.

Six kinds of work, each through the public entry points:

  evolve       a simulation from a Pauli product state: build_gates, step(n),
               then every observable (small systems, bonds grow from 1 and the
               cutoff picks the ranks);
  step         a prepared MPO is loaded, advanced by Trotter steps and measured
               (the production regime: every bond at chi_max);
  gradient     forward with checkpoints, observables, reverse sweep (noise-model
               fitting);
  observables  <X>, <Y>, <Z> of every qubit and the connected <ZZ> of every pair
               of a state that is already on the device;
  entropies    the second Renyi entropy and the operator space entanglement
               entropy at the central bond of such a state;
  gemm         the FP64-accurate tensor-core product on the caller's matrices.

The tensors of an MPO are only defined up to a gauge on every bond (the signs of
singular vectors at least), so an evolved state is returned as what is unique in
it: the Bloch vector of every qubit, the connected correlator of every pair and
the bond dimensions.

Prepared states are a product state plus correlations whose weight falls off
along every bond by a factor exp(-GRADE), the shape that evolved states have.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2203_05871_gb300 as mpdo
from paper_2203_05871_gb300.mpdo import gemm_tc

PRECISION = {"fp64": mpdo.FP64, "tf32": mpdo.MIXED_TF32, "bf16x3": mpdo.MIXED_BF16X3}
STORAGE = {"f64": mpdo.STORE_F64, "f32": mpdo.STORE_F32}


def listed():
    return [
        # the small validation run: 8 qubits, chi 32, cutoff 1e-12, dt 0.05 x 40 steps, FP64
        dict(name="evolve_chain8_fp64", kind="evolve", graph="chain", n=8, chi=32, cutoff=1e-12, dt=0.05, steps=40,
             precision="fp64"),
        # a two-dimensional patch on the snake path: swap gates, one op per layer
        dict(name="evolve_grid3x3_fp64", kind="evolve", graph="grid3", n=9, chi=32, cutoff=1e-10, dt=0.05, steps=4,
             precision="fp64"),
        # the precision study's chain in FP64: bond matrices of 512 x 512
        dict(name="step_chain20_chi128_fp64", kind="step", graph="chain", n=20, chi=128, batch=1, steps=1,
             precision="fp64", replay=False, uneven=False),
        # the headline workload: 20 qubits, every inner bond at 256, mixed path
        dict(name="step_chain20_chi256_tf32", kind="step", graph="chain", n=20, chi=256, batch=1, steps=1,
             precision="tf32", replay=False, uneven=False),
        # an odd bond dimension and the other tensor-core kind
        dict(name="step_chain11_chi173_bf16x3", kind="step", graph="chain", n=11, chi=173, batch=1, steps=1,
             precision="bf16x3", replay=False, uneven=False),
        # a parameter scan: independent chains, chi_max of each instance from {32, 64, 128, 256}
        dict(name="step_batch6_chain16_tf32", kind="step", graph="chain", n=16, chi=256, batch=6, steps=1,
             precision="tf32", replay=False, uneven=True),
        # many small instances replaying the captured step
        dict(name="step_graph_batch16_chi24", kind="step", graph="chain", n=10, chi=24, batch=16, steps=2,
             precision="tf32", replay=True, uneven=False),
        # one gradient of a fit: ring, closing bond through swaps, FP64
        dict(name="gradient_ring12_chi32", kind="gradient", graph="ring", n=12, chi=32, batch=1, steps=1,
             precision="fp64"),
        # all observables at the largest size: the 4 x 10 grid's path at chi 512
        dict(name="observables_n40_chi512", kind="observables", n=40, chi=512, batch=1, storage="f64"),
        # the smallest calls: read-out of a small batch in float storage between steps
        dict(name="observables_batch4_n8_f32", kind="observables", n=8, chi=32, batch=4, storage="f32"),
        # global characteristics of the headline state
        dict(name="entropies_chain20_chi256", kind="entropies", n=20, chi=256, batch=1),
        # the tensor-core product on a caller's ragged matrices
        dict(name="gemm_1000x1500x777_tf32", kind="gemm", m=1000, nn=1500, k=777, precision="tf32"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["evolve", "step", "step", "step", "gradient", "observables", "entropies", "gemm"])
    if kind == "evolve":
        graph = rng.choice(["chain", "ring", "grid3"])
        n = 9 if graph == "grid3" else rng.randint(5, 9)
        return dict(kind=kind, graph=graph, n=n, chi=rng.randint(12, 32), cutoff=10.0 ** -rng.randint(9, 12),
                    dt=rng.uniform(0.03, 0.06), steps=rng.randint(4, 20) if graph == "chain" else rng.randint(2, 4),
                    precision="fp64")
    if kind == "step":
        precision = rng.choice(["fp64", "tf32", "bf16x3"])
        small = rng.random() < 0.5
        n = rng.randint(6, 20)
        chi = log(12, 64) if small else log(64, 128 if precision == "fp64" else 256)
        return dict(kind=kind, graph="ring" if small and n <= 9 and rng.random() < 0.3 else "chain", n=n, chi=chi,
                    batch=log(1, 12) if small else rng.randint(1, 3) if chi <= 128 else 1,
                    steps=rng.randint(1, 2) if small else 1, precision=precision,
                    replay=small and rng.random() < 0.5, uneven=rng.random() < 0.3)
    if kind == "gradient":
        return dict(kind=kind, graph=rng.choice(["chain", "ring"]), n=rng.randint(6, 12), chi=rng.randint(8, 32),
                    batch=rng.randint(1, 2), steps=1, precision="fp64")
    if kind == "observables":
        return dict(kind=kind, n=rng.randint(6, 40), chi=log(16, 480), batch=rng.randint(1, 2),
                    storage=rng.choice(["f64", "f32"]))
    if kind == "entropies":
        return dict(kind=kind, n=rng.randint(6, 20), chi=log(16, 250), batch=1)
    return dict(kind=kind, m=log(32, 1024), nn=log(32, 1536), k=log(32, 1024),
                precision=rng.choice(["tf32", "bf16x3"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def bonds_of(graph, n):
    b = [(i, i + 1) for i in range(n - 1)]
    if graph == "ring":
        return b + [(0, n - 1)]
    if graph == "grid3":   # columns of three on a snake path
        pos = lambda x, y: 3 * x + (y if x % 2 == 0 else 2 - y)
        col = [(pos(x, y), pos(x, y + 1)) for x in range(n // 3) for y in range(2)]
        row = [(pos(x, y), pos(x + 1, y)) for x in range(n // 3 - 1) for y in range(3)]
        return [(min(p), max(p)) for p in col + row]
    return b


def chi_of(case):
    """chi_max of every instance."""
    B, chi = case.get("batch", 1), case["chi"]
    if not case.get("uneven"):
        return [chi] * B
    return [max(4, chi >> (b % 4)) for b in range(B)]


def model(case, rng):
    """A seeded model: detuned, driven, decaying and dephasing qubits with XY couplings."""
    n, B = case["n"], case.get("batch", 1)
    bonds = bonds_of(case.get("graph", "chain"), n)
    u = lambda lo, hi, k: rng.uniform(lo, hi, size=(B, k))
    init = [str(v) for v in rng.choice(["+x", "-x", "+y", "-y", "+z", "-z"], size=n)]
    return SimpleNamespace(
        n=n, batch=B, bonds=bonds, h_x=u(0.3, 0.7, n), h_y=np.zeros((B, n)),
        h_z=np.arange(n)[None, :] % 2 + u(-0.1, 0.1, n), g0=u(0.005, 0.02, n), g1=np.zeros((B, n)), g2=u(0.01, 0.03, n),
        J=u(0.05, 0.2, len(bonds)), Jz=np.zeros((B, len(bonds))), chi_max=np.array(chi_of(case)),
        cutoff=np.full(B, case.get("cutoff", 1e-12)), dt=case.get("dt", 0.02), init=init)


def dims_of(n, chi):
    return [1] + [min(chi, 4 ** min(p + 1, n - p - 1)) for p in range(n - 1)] + [1]


GRADE, CORRELATED = 4.0, 1.5


def state(n, chi, rng):
    """(dims, tensors) of one instance: product state plus graded correlations."""
    dims, out = dims_of(n, chi), []
    for p in range(n):
        cl, cr = dims[p], dims[p + 1]
        t = rng.standard_normal((cl, 4, cr))
        t *= (CORRELATED / math.sqrt(4.0 * cl)) * np.exp(-(GRADE / chi) * np.arange(cr))
        t[0, :, 0] = np.array([1.0, *rng.uniform(-0.5, 0.5, 3)]) / math.sqrt(2.0)
        out.append(t)
    return dims, out


def all_pairs(n):
    return [(i, j) for i in range(n) for j in range(i + 1, n)]


def inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "gemm":   # rows and columns of very different size, as bond matrices have
        a = rng.standard_normal((case["m"], case["k"])) * np.logspace(0, -4, case["m"])[:, None]
        b = rng.standard_normal((case["k"], case["nn"])) * np.logspace(0, -2, case["nn"])[None, :]
        return SimpleNamespace(a=a, b=b)
    wl = model(case, rng)
    x = SimpleNamespace(wl=wl, states=None)
    if case["kind"] != "evolve":
        x.states = [state(case["n"], c, rng) for c in chi_of(case)]
    if case["kind"] == "gradient":
        x.zbar = rng.standard_normal((wl.batch, wl.n))
        x.wbar = np.triu(rng.standard_normal((wl.batch, wl.n, wl.n)), 1)
    return x


def prepare(case, seed):
    x = inputs(case, seed)
    x.case = case
    if case["kind"] == "gemm":
        x.a, x.b = torch.tensor(x.a, device="cuda"), torch.tensor(x.b, device="cuda")
        return x
    x.solver = mpdo.Solver(case["n"], batch=x.wl.batch, chi_cap=case["chi"],
                           precision=PRECISION[case.get("precision", "fp64")],
                           storage=STORAGE[case.get("storage", "f64")])
    x.solver.build_gates(x.wl)
    if case["kind"] in ("observables", "entropies"):
        load(x)
    return x


def load(x):
    for b, (dims, tensors) in enumerate(x.states):
        x.solver.set_state(b, dims, tensors)


def read_out(s):
    qubits = range(s.n)
    return {"x": s.measure_1q(qubits, "X"), "y": s.measure_1q(qubits, "Y"), "z": s.measure_1q(qubits, "Z"),
            "zz": s.measure_2q(all_pairs(s.n), "ZZ", connected=True)}


def run(x):
    kind = x.case["kind"]
    if kind == "gemm":
        return gemm_tc(x.a, x.b, PRECISION[x.case["precision"]])
    s = x.solver
    if kind == "evolve":
        s.build_gates(x.wl)
        s.step(x.case["steps"])
        return read_out(s)
    if kind == "step":
        load(x)
        s.step(x.case["steps"], graph=x.case["replay"])
        out = read_out(s)
        return {**out, "chi": s.status()["chi"]}
    if kind == "gradient":
        load(x)
        s.grad_forward(x.case["steps"])
        out = read_out(s)
        grad, loss = s.grad_backward(x.zbar, x.wbar)
        return {**out, "grad": grad, "loss": loss}
    if kind == "observables":
        return read_out(s)
    return {"renyi2": s.renyi2(), "osee": s.osee()}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def schedule(n, bonds):
    """Ops (layer by layer, in order) of one second-order step: ("gate", p, qubit
    at p, qubit at p + 1, bond, fraction of dt) or ("swap", p)."""
    even = [("gate", i, k) for k, (i, j) in enumerate(bonds) if j == i + 1 and i % 2 == 0]
    odd = [("gate", i, k) for k, (i, j) in enumerate(bonds) if j == i + 1 and i % 2 == 1]
    half = [sorted(layer, key=lambda o: o[1]) for layer in (even, odd) if layer]
    for k, (i, j) in enumerate(bonds):
        if j > i + 1:
            there = [[("swap", p, -1)] for p in range(j - 1, i, -1)]
            half += there + [[("gate", i, k)]] + there[::-1]
    back = half[::-1]
    while half[-1][0][0] == "swap":   # the two halves meet: equal swaps cancel, the middle layer runs once
        half, back = half[:-1], back[1:]
    at, ops = list(range(n)), []
    for layer, frac in [(x, 0.5) for x in half[:-1]] + [(half[-1], 1.0)] + [(x, 0.5) for x in back[1:]]:
        for kind, p, k in layer:
            ops.append((kind, p, at[p], at[p + 1], k, frac))
            if kind == "swap":
                at[p], at[p + 1] = at[p + 1], at[p]
    return ops


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["nn"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    n, bytes_, flops = case["n"], 0.0, 0.0
    for chi in chi_of(case):
        d = dims_of(n, chi)
        elems = [d[p] * 4 * d[p + 1] for p in range(n)]
        esize = 4.0 if case.get("storage") == "f32" else 8.0
        if kind == "observables":   # the state once; environments and the stacked rows of all pairs
            bytes_ += esize * sum(elems)
            flops += sum(2.0 * d[p] * d[p + 1] * (5 + 2 * p) for p in range(n))
            continue
        if kind == "entropies":     # Gram sweeps over the state, three spectral decompositions of the centre
            bytes_ += esize * sum(elems)
            flops += sum(16.0 * d[p] * d[p + 1] * max(d[p], d[p + 1]) for p in range(n))
            flops += 3 * 9.0 * d[n // 2] ** 3
            continue
        ops = schedule(n, bonds_of(case["graph"], n))
        steps = case["steps"] * (3 if kind == "gradient" else 1)
        bytes_ += 2 * 8.0 * sum(elems)
        for _, p, *_ in ops:   # merge, gate, singular values and right vectors, new left site
            cl, cm, cr = d[p], d[p + 1], d[p + 2]
            small, large = 4.0 * min(cl, cr), 4.0 * max(cl, cr)
            flops += steps * (32.0 * cl * cm * cr + 512.0 * cl * cr + 4 * large * small ** 2 + 8 * small ** 3
                              + 32.0 * cl * cm * cr)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same results from plain torch in 64 bits
# ---------------------------------------------------------------------------
SX = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128)
SY = torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128)
SZ = torch.tensor([[1, 0], [0, -1]], dtype=torch.complex128)
PAULI = [torch.eye(2, dtype=torch.complex128), SX, SY, SZ]


def superop(f, basis):
    """Matrix of the map f in an orthonormal Hermitian operator basis (real for Hermitian-preserving f)."""
    cols = [f(b) for b in basis]
    return torch.stack([torch.stack([torch.trace(a @ c).real for c in cols]) for a in basis])


def generators():
    """Site generators of h_x, h_y, h_z, g0, g1, g2 (4 x 4) and bond generators of J, Jz (16 x 16)."""
    one = [p / math.sqrt(2) for p in PAULI]
    two = [torch.kron(a, b) for a in one for b in one]
    up, down = (SX + 1j * SY) / 2, (SX - 1j * SY) / 2
    com = lambda h: (lambda r: -1j * (h @ r - r @ h))
    jump = lambda c: (lambda r: c @ r @ c.mH - 0.5 * (c.mH @ c @ r + r @ c.mH @ c))
    site = [superop(f, one) for f in (com(0.5 * SX), com(0.5 * SY), com(0.5 * SZ), jump(up), jump(down), jump(SZ))]
    xy = 0.5 * (torch.kron(SX, SX) + torch.kron(SY, SY))
    return site, [superop(com(xy), two), superop(com(0.5 * torch.kron(SZ, SZ)), two)]


def step_gates(wl, params, ops):
    """16 x 16 gate of every op of one instance; params: h_x .. g2 of every qubit, J and Jz of every bond, in a row."""
    n, nb = wl.n, len(wl.bonds)
    site, bond = generators()
    deg = [sum(q in b for b in wl.bonds) for q in range(n)]
    eye = torch.eye(4, dtype=torch.float64)
    local = [sum(params[u * n + q] * site[u] for u in range(6)) / deg[q] for q in range(n)]
    out = []
    for kind, p, qa, qb, k, frac in ops:
        if kind == "swap":
            out.append(torch.eye(16, dtype=torch.float64).reshape(4, 4, 16).transpose(0, 1).reshape(16, 16))
            continue
        g = params[6 * n + k] * bond[0] + params[6 * n + nb + k] * bond[1]
        g = g + torch.kron(local[qa].contiguous(), eye) + torch.kron(eye, local[qb].contiguous())
        g = g * (frac * wl.dt / 16)
        e = term = torch.eye(16, dtype=torch.float64)
        for i in range(1, 16):
            term = term @ g / i
            e = e + term
        for _ in range(4):
            e = e @ e
        out.append(e)
    return out


def advance(tensors, wl, b, params, steps):
    """Trotter steps of instance b on a list of tensors."""
    ops = schedule(wl.n, wl.bonds)
    gates = step_gates(wl, params, ops)
    B, lam = list(tensors), [torch.ones(t.shape[2], dtype=torch.float64) for t in tensors]
    for _ in range(steps):
        for (_, p, *_), g in zip(ops, gates):
            cl, cr = B[p].shape[0], B[p + 1].shape[2]
            th = torch.einsum("lsm,mtr->stlr", B[p], B[p + 1]).reshape(16, cl * cr)
            th = (g @ th).reshape(4, 4, cl, cr).permute(2, 0, 1, 3).reshape(4 * cl, 4 * cr)
            left = lam[p - 1].repeat_interleave(4)[:, None] if p > 0 else 1.0
            _, s, vt = torch.linalg.svd(left * th, full_matrices=False)
            w = (s * s).detach()
            tail = torch.flip(torch.cumsum(torch.flip(w, [0]), 0), [0])   # tail[k]: weight from k on
            ok = (torch.cat([tail, torch.zeros(1, dtype=torch.float64)]) <= float(wl.cutoff[b]) * float(tail[0]))
            k = min(int(wl.chi_max[b]), max(1, int(torch.nonzero(ok)[0])))
            lam[p] = s[:k]
            B[p + 1] = vt[:k].reshape(k, 4, cr)
            B[p] = (th @ vt[:k].T).reshape(cl, 4, k)
        tr = torch.ones(1, dtype=torch.float64)
        for t in B:
            tr = tr @ t[:, 0]
        B[0] = B[0] / (2.0 ** (wl.n / 2) * tr)
    return B


def observables(B):
    """x, y, z of every qubit and the connected zz of every pair."""
    n = len(B)
    L, R = [torch.ones(1, dtype=torch.float64)], [torch.ones(1, dtype=torch.float64)]
    for t in B:
        L.append(L[-1] @ t[:, 0])
    for t in B[::-1]:
        R.append(t[:, 0] @ R[-1])
    R, e = R[::-1], L[-1][0]
    one = [torch.stack([L[q] @ B[q][:, a] @ R[q + 1] / e for q in range(n)]) for a in (1, 2, 3)]
    zz = []
    for i in range(n):
        w = L[i] @ B[i][:, 3]
        for j in range(i + 1, n):
            zz.append(w @ B[j][:, 3] @ R[j + 1] / e - one[2][i] * one[2][j])
            w = w @ B[j][:, 0]
    return one[0], one[1], one[2], torch.stack(zz)


def entropies(B):
    n = len(B)
    x, tr = torch.ones(1, 1, dtype=torch.float64), torch.ones(1, dtype=torch.float64)
    for t in B:
        x = torch.einsum("lk,lsr,ksq->rq", x, t, t)
        tr = tr @ t[:, 0]
    left = right = torch.ones(1, 1, dtype=torch.float64)
    for t in B[: n // 2]:
        m = torch.einsum("ij,jsr->isr", left, t)
        left = torch.linalg.qr(m.reshape(-1, m.shape[2]))[1]
    for t in B[n // 2:][::-1]:
        m = torch.einsum("lsr,rj->lsj", t, right)
        right = torch.linalg.qr(m.reshape(m.shape[0], -1).T)[1].T
    p = torch.linalg.svdvals(left @ right) ** 2
    p = p / p.sum()
    p = p[p > 0]
    return -torch.log(x[0, 0] / (2.0 ** n * tr[0] ** 2)), -(p * p.log()).sum()


def exact(case, seed):
    kind = case["kind"]
    if kind == "step" and sum(c ** 3 for c in chi_of(case)) * case["n"] > 4.5e8 * 1.5:
        return None
    x = inputs(case, seed)
    if kind == "gemm":
        return torch.tensor(x.a) @ torch.tensor(x.b)
    wl, rows = x.wl, []
    for b in range(wl.batch):
        if kind == "evolve":
            B = [torch.zeros(1, 4, 1, dtype=torch.float64) for _ in range(wl.n)]
            for t, (sign, axis) in zip(B, wl.init):
                t[0, 0, 0] = 1.0 / math.sqrt(2.0)
                t[0, "xyz".index(axis) + 1, 0] = float(sign + "1") / math.sqrt(2.0)
        else:
            B = [torch.tensor(t) for t in x.states[b][1]]
        if case.get("storage") == "f32":
            B = [t.float().double() for t in B]
        if kind == "entropies":
            rows.append(dict(zip(("renyi2", "osee"), entropies(B))))
            continue
        row = {}
        if kind != "observables":
            params = torch.tensor(np.concatenate([getattr(wl, f)[b] for f in ("h_x", "h_y", "h_z", "g0", "g1", "g2", "J", "Jz")]))
            params.requires_grad_(kind == "gradient")
            B = advance(B, wl, b, params, case["steps"])
            if kind == "step":
                row = {"chi": torch.tensor([t.shape[2] for t in B[:-1]], dtype=torch.int32)}
        row.update(zip(("x", "y", "z", "zz"), observables(B)))
        if kind == "gradient":
            w = torch.tensor([x.wbar[b][i][j] for i, j in all_pairs(wl.n)])
            row["loss"] = torch.tensor(x.zbar[b]) @ row["z"] + w @ row["zz"]
            row["grad"], = torch.autograd.grad(row["loss"], params)
        rows.append(row)
    return {k: torch.stack([r[k].detach().double() if r[k].is_floating_point() else r[k] for r in rows]).numpy()
            for k in rows[0]}
