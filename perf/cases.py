"""Performance cases: the work a user of the library has it do, over its real range.

A case is a dict of plain values. Its "kind" names the call that is timed:
  rhs       one semi-discrete right-hand side (Solver.rhs)
  step      `steps` LSERK4 steps of one mesh (Solver.step)
  ensemble  `steps` LSERK4 steps of many meshes in one call (Solver.ensemble_step)
  misfit    misfit and gradients of an inversion step (ReceiverMisfit, backward)
  traces    differentiable receiver traces (MaxwellSolve, a loss on them, backward)
Meshes are boxes of nx x ny x nz hexahedra cut into six tetrahedra each, with
jittered interior vertices, numbered x fastest or along a Hilbert curve, the
materials uniform in [1, 4) per element; fields are smooth pulses over the
cavity mode. The time step is 0.5 h / N^2 (0.2 h at N = 1, whose stability limit is lower).

exact() computes the same outputs in 64 bits with numpy and torch alone: its own
nodes, operators, geometry and connectivity, and torch's reverse mode for the
gradients.
"""
import itertools
import math

import numpy as np
import torch

import paper_1211_0582_gb300 as dg

LSERK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
           -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
LSERK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
           1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
           2277821191437.0 / 14882151754819.0)
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------ the cases
def _single(name, kind, N, n, precision, steps=1, order="hilbert", materials="none", alpha=1.0, receivers=0, ckpt=0):
    return dict(name=name, kind=kind, N=N, nx=n[0], ny=n[1], nz=n[2], precision=precision, steps=steps, order=order,
                materials=materials, alpha=alpha, receivers=receivers, ckpt=ckpt)


def _ensemble(name, N, members, lo, hi, precision, steps):
    return dict(name=name, kind="ensemble", N=N, members=members, lo=lo, hi=hi, precision=precision, steps=steps,
                order="lexicographic", materials="eps", alpha=1.0, receivers=0, ckpt=0)


def listed():
    return [
        # one operator application on a test-sized mesh: a Krylov or eigenvalue iteration's inner call
        _single("rhs_fp32_n3_small", "rhs", 3, (3, 3, 3), "fp32", order="lexicographic", materials="eps"),
        # a small cavity stepped in a long loop: launches and latency count
        _single("step_fp16x3_n4_small", "step", 4, (6, 6, 6), "fp16x3", steps=40, order="lexicographic",
                materials="eps"),
        # the default precision on the benchmark's mesh
        _single("step_fp32_n5", "step", 5, (24, 24, 24), "fp32", steps=5),
        # the benchmark's headline workload
        _single("step_fp16x3_n5", "step", 5, (24, 24, 24), "fp16x3", steps=10),
        # a box of uneven sides at a low order, the mesh generator's own numbering
        _single("step_fp16x3_n3_box", "step", 3, (31, 19, 23), "fp16x3", steps=10, order="lexicographic",
                materials="eps_mu"),
        # a resonator with materials at high order: the largest state
        _single("step_fp16x3_n7", "step", 7, (32, 32, 32), "fp16x3", steps=2, materials="eps"),
        # the fastest split at a streamed order, central flux
        _single("step_bf16x3_n6", "step", 6, (13, 12, 11), "bf16x3", steps=5, materials="eps", alpha=0.0),
        # highest orders: FP32 only
        _single("step_fp32_n8", "step", 8, (16, 16, 16), "fp32", steps=3, materials="eps"),
        # a parameter study: many meshes of uneven sizes advanced together
        _ensemble("ensemble_fp32_n4", 4, 16, 8, 16, "fp32", 10),
        _ensemble("ensemble_fp16x3_n4", 4, 16, 8, 16, "fp16x3", 10),
        # one iteration of a permittivity inversion on the adjoint benchmark's mesh
        _single("misfit_fp32_n4", "misfit", 4, (20, 20, 20), "fp32", steps=40, materials="eps", receivers=256,
                ckpt=20),
        # the solver inside a differentiable program, split precision, automatic segments
        _single("traces_fp16x3_n5", "traces", 5, (9, 8, 7), "fp16x3", steps=30, materials="eps", receivers=61,
                ckpt=0),
    ]


def draw(rng):
    kind = rng.choices(("rhs", "step", "ensemble", "misfit", "traces"), (1, 5, 2, 1.5, 1))[0]
    precision = rng.choice(("fp32", "fp16x3", "fp16x3", "bf16x3"))
    if kind == "ensemble":
        lo = rng.randint(2, 10)
        c = _ensemble("", rng.randint(2, 6), rng.randint(3, 24), lo, rng.randint(lo + 1, 14), precision, 1)
    else:
        N = rng.randint(1, 9 if precision == "fp32" and kind in ("rhs", "step") else 7 if kind in ("rhs", "step") else 6)
        # state sizes from a few thousand to some 10^8 values, over their logarithm
        values = math.exp(rng.uniform(math.log(2e4), math.log(1.2e8 if kind in ("rhs", "step") else 1e7)))
        side = max(2.0, (values / (36 * _np(N))) ** (1 / 3))
        n = [max(2, round(side * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(3)]
        while n[0] * n[1] * n[2] * 36 * _np(N) > 1.4e8:
            n[n.index(max(n))] -= 1
        c = _single("", kind, N, n, precision, order=rng.choice(("hilbert", "lexicographic")),
                    materials=rng.choice(("none", "eps", "eps", "eps_mu")) if kind in ("rhs", "step") else "eps",
                    alpha=rng.choice((1.0, 1.0, 1.0, 0.0)))
        if kind in ("misfit", "traces"):
            c["receivers"] = rng.randint(1, min(300, 6 * n[0] * n[1] * n[2]))
            c["ckpt"] = rng.choice((0, 5, 20))
    del c["name"]
    if kind != "rhs":
        most = 1.2e12 if precision == "fp32" else 8e11
        c["steps"] = max(1, min(rng.randint(1, 60), int(most / work(c)["flops"])))
    return c


def _np(N):
    return (N + 1) * (N + 2) * (N + 3) // 6


def _sizes(case):
    """Hexahedra per side of each mesh of the case."""
    if case["kind"] != "ensemble":
        return [(case["nx"], case["ny"], case["nz"])]
    sizes = np.random.default_rng(case["members"] * 1000 + case["N"]).integers(case["lo"], case["hi"] + 1,
                                                                               size=case["members"])
    return [(int(n),) * 3 for n in sizes]


def work(case):
    """Bytes: each stage of a step reads the state and the residual and writes both (the first reads no residual), with
    160 bytes of geometry per element; states that fit the 126 MB L2 cache twice over are read and written once. A
    gradient adds the reverse sweep: both multipliers read and written, the stage's state and half a right-hand side
    read. Flops: derivatives, lifting, chain rule and fluxes; the reverse sweep costs as much as the forward one."""
    N, Np, Nfp = case["N"], _np(case["N"]), (case["N"] + 1) * (case["N"] + 2) // 2
    K = sum(6 * a * b * c for a, b, c in _sizes(case))
    field = 24.0 * K * ((Np + 3) // 4 * 4)
    stage_flops = K * (36.0 * Np * Np + 48.0 * Np * Nfp + 78.0 * Np + 240.0 * Nfp)
    if case["kind"] == "rhs":
        return {"bytes": 2 * field + 160.0 * K, "flops": stage_flops}
    stages = 5 * case["steps"]
    resident = 2 * field < 126e6
    nbytes = 3 * field + 160.0 * K if resident else stages * (3.8 * field + 160.0 * K)
    flops = stages * stage_flops
    if case["kind"] in ("misfit", "traces"):
        flops *= 2
        nbytes += stages * 1.5 * 2 * field + (field if resident else stages * 4.0 * field)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ inputs
def _hilbert(n):
    """The hexahedra (x fastest indices) of a box along a 3D Hilbert curve (Skilling, AIP Conf. Proc. 707, 2004)."""
    bits = max(1, math.ceil(math.log2(max(n))))
    z, y, x = np.meshgrid(*(np.arange(m, dtype=np.int64) for m in n[::-1]), indexing="ij")
    X = [x.ravel().copy(), y.ravel().copy(), z.ravel().copy()]
    Q = 1 << (bits - 1)
    while Q > 1:
        for i in range(3):
            flip = (X[i] & Q) != 0
            t = np.where(flip, 0, (X[0] ^ X[i]) & (Q - 1))
            X[0] = np.where(flip, X[0] ^ (Q - 1), X[0]) ^ t
            X[i] = X[i] ^ t
        Q >>= 1
    X[1] = X[1] ^ X[0]
    X[2] = X[2] ^ X[1]
    t = np.zeros_like(X[0])
    Q = 1 << (bits - 1)
    while Q > 1:
        t = np.where((X[2] & Q) != 0, t ^ (Q - 1), t)
        Q >>= 1
    code = np.zeros_like(X[0])
    for b in range(bits - 1, -1, -1):
        for i in range(3):
            code = (code << 1) | (((X[i] ^ t) >> b) & 1)
    return np.argsort(code, kind="stable")


def _box(n, order, rng):
    """Vertices and tetrahedra of a jittered box of n[0] x n[1] x n[2] hexahedra in the unit cube."""
    nx, ny, nz = n
    g = [np.arange(m + 1) / m for m in n]
    VZ, VY, VX = (v.ravel().copy() for v in np.meshgrid(g[2], g[1], g[0], indexing="ij"))
    inner = (VX > 0) & (VX < 1) & (VY > 0) & (VY < 1) & (VZ > 0) & (VZ < 1)
    for V, m in ((VX, nx), (VY, ny), (VZ, nz)):
        V[inner] += rng.uniform(-0.1 / m, 0.1 / m, size=int(inner.sum()))
    k, j, i = (v.ravel() for v in np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"))
    if order == "hilbert":
        o = _hilbert(n)
        i, j, k = i[o], j[o], k[o]
    tets = []
    for perm in itertools.permutations((0, 1, 2)):
        corner = [0, 0, 0]
        walk = [tuple(corner)]
        for axis in perm:
            corner[axis] += 1
            walk.append(tuple(corner))
        if sum(perm[a] > perm[b] for a in range(3) for b in range(a + 1, 3)) % 2:
            walk[1], walk[2] = walk[2], walk[1]
        tets.append(np.stack([(i + a) + (nx + 1) * ((j + b) + (ny + 1) * (k + c)) for a, b, c in walk], axis=1))
    return VX, VY, VZ, np.stack(tets, axis=1).reshape(-1, 4).astype(np.int32)


def _inputs(case, seed):
    """Meshes, materials, time steps and starting fields of a case (64-bit values that are exact in 32 bits)."""
    rng = np.random.default_rng([seed, case["N"]])
    sizes = _sizes(case)
    meshes = [_box(n, case["order"], rng) for n in sizes]
    Ks = [m[3].shape[0] for m in meshes]
    eps = [np.ones(K, np.float32) if case["materials"] == "none" else rng.uniform(1, 4, K).astype(np.float32)
           for K in Ks]
    mu = rng.uniform(0.5, 2, Ks[0]).astype(np.float32) if case["materials"] == "eps_mu" else None
    dts = [0.5 / max(n) / max(case["N"] ** 2, 2.5) for n in sizes]
    verts = np.concatenate([np.stack(m[:3], axis=1) for m in meshes])
    base = np.cumsum([0] + [m[0].size for m in meshes])
    tets = np.concatenate([m[3].astype(np.int64) + b for m, b in zip(meshes, base)])
    X = torch.as_tensor(verts, device=DEV)[torch.as_tensor(tets, device=DEV)]  # [K, 4, 3]
    r, s, t = _nodes(case["N"])
    lam = torch.as_tensor(np.stack([-(1 + r + s + t) / 2, (1 + r) / 2, (1 + s) / 2, (1 + t) / 2], axis=1), device=DEV)
    u = torch.zeros(6, X.shape[0], (len(r) + 3) // 4 * 4, device=DEV)
    x, y, z = torch.einsum("iv,kvc->cki", lam, X)
    S, C = [torch.sin(math.pi * v) for v in (x, y, z)], [torch.cos(math.pi * v) for v in (x, y, z)]
    u[0, :, :len(r)], u[1, :, :len(r)], u[2, :, :len(r)] = C[0] * S[1] * S[2], -2 * S[0] * C[1] * S[2], S[0] * S[1] * C[2]
    for field in (0, 0, 3, 3):  # two electric and two magnetic pulses, each the curl of a Gaussian
        c, w, p = rng.uniform(0.3, 0.7, 3), rng.uniform(0.08, 0.2), rng.standard_normal(3)
        d = [x - c[0], y - c[1], z - c[2]]
        g = torch.exp(-(d[0] ** 2 + d[1] ** 2 + d[2] ** 2) / w ** 2) / w
        for a in range(3):
            b, e = (a + 1) % 3, (a + 2) % 3
            u[field + a, :, :len(r)] += (g * (p[b] * d[e] - p[e] * d[b])).float()
    state = dict(meshes=meshes, eps=eps, mu=mu, dts=dts, X=X, tets=tets, u0=u)
    if case["receivers"]:
        R, T = case["receivers"], case["steps"]
        state["recv"] = torch.as_tensor(rng.choice(Ks[0] * len(r), R, replace=False).astype(np.int64), device=DEV)
        # recorded signals: a few oscillations per receiver and component over the run
        f, ph, a = (torch.as_tensor(rng.uniform(lo, hi, (1, 3, R)), device=DEV) for lo, hi in
                    ((0.5, 3), (0, 6.28), (0.1, 1)))
        tt = torch.linspace(0, 1, T, dtype=torch.float64, device=DEV)[:, None, None]
        state["Eref"] = (a * torch.cos(6.28 * f * tt + ph)).float()
    return state


def prepare(case, seed):
    inp = _inputs(case, seed)
    s = dg.Solver(case["N"], precision=case["precision"])
    state = dict(case=case, solver=s)
    if case["kind"] == "ensemble":
        s.upload_ensemble(inp["meshes"], inp["eps"], inp["dts"])
        s.ensemble_tune()
    else:
        s.upload(*inp["meshes"][0], eps=inp["eps"][0], mu=inp["mu"])
        state["dt"] = inp["dts"][0]
    if case["kind"] in ("misfit", "traces"):
        state["u0"] = inp["u0"].requires_grad_()
        state["eps"] = torch.as_tensor(inp["eps"][0], device="cuda").requires_grad_()
        state["recv"], state["Eref"] = inp["recv"], inp["Eref"]
    else:
        state["u"], state["out"] = inp["u0"], s.zeros()
    return state


def run(state):
    c, s = state["case"], state["solver"]
    if c["kind"] == "rhs":
        return s.rhs(state["u"], out=state["out"], alpha=c["alpha"])
    # the state after the steps; the residual beside it is the scheme's scratch (no call reads its entry value)
    if c["kind"] == "step":
        return s.step(state["u"], state["out"], state["dt"], c["steps"], alpha=c["alpha"])[0]
    if c["kind"] == "ensemble":
        return s.ensemble_step(state["u"], state["out"], c["steps"], alpha=c["alpha"])[0]
    u0, eps = state["u0"], state["eps"]
    u0.grad = eps.grad = None
    if c["kind"] == "misfit":
        J = dg.ReceiverMisfit.apply(u0, eps, s, state["recv"], state["Eref"], state["dt"], c["steps"], c["ckpt"],
                                    c["alpha"])
        J.backward()
        # the misfit as a training loop logs it: the accuracy is that of the 32-bit fields it sums
        return {"J": J.detach().float(), "deps": eps.grad, "du0": u0.grad}
    traces = dg.MaxwellSolve.apply(u0, eps, s, state["recv"], state["dt"], c["steps"], c["ckpt"], c["alpha"])
    ((traces - state["Eref"]) ** 2).sum().backward()
    return {"traces": traces.detach(), "deps": eps.grad, "du0": u0.grad}


# ------------------------------------------------------------------ the same in 64 bits
def _lgl(N):
    """Legendre-Gauss-Lobatto points: the ends and the roots of P_N'."""
    c = np.zeros(N + 1)
    c[N] = 1
    inner = np.real(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c))) if N > 1 else np.zeros(0)
    return np.concatenate([[-1.0], np.sort(inner), [1.0]])


def _nodes(N):
    """Warp & blend nodes of the tetrahedron without a blend parameter (Warburton 2006), r fastest."""
    eq, lgl = np.linspace(-1, 1, N + 1), _lgl(N)

    def warp(r):
        w = np.zeros_like(r)
        for i in range(N + 1):
            li = np.ones_like(r)
            for j in range(N + 1):
                if j != i:
                    li = li * (r - eq[j]) / (eq[i] - eq[j])
            w += (lgl[i] - eq[i]) * li
        inside = np.abs(r) < 1 - 1e-10
        return np.where(inside, w / np.where(inside, 1 - r * r, 1.0), 0.0)

    ijk = np.array([(i, j, k) for k in range(N + 1) for j in range(N + 1 - k) for i in range(N + 1 - k - j)], float)
    L = np.concatenate([1 - ijk.sum(1, keepdims=True) / N, ijk / N], axis=1)
    V = np.array([[-1, -1 / math.sqrt(3), -1 / math.sqrt(6)], [1, -1 / math.sqrt(3), -1 / math.sqrt(6)],
                  [0, 2 / math.sqrt(3), -1 / math.sqrt(6)], [0, 0, 3 / math.sqrt(6)]])
    X = L @ V
    for o, a, b, c in ((3, 0, 1, 2), (2, 0, 1, 3), (0, 1, 2, 3), (1, 0, 2, 3)):
        t1, t2 = V[b] - V[a], V[c] - (V[a] + V[b]) / 2
        t1, t2 = t1 / np.linalg.norm(t1), t2 / np.linalg.norm(t2)
        La, Lb, Lc, Lo = L[:, a], L[:, b], L[:, c], L[:, o]
        e = [4 * p * q * warp(q - p) for p, q in ((La, Lb), (Lb, Lc), (Lc, La))]
        dx = e[0] + math.cos(2 * math.pi / 3) * e[1] + math.cos(4 * math.pi / 3) * e[2]
        dy = math.sin(2 * math.pi / 3) * e[1] + math.sin(4 * math.pi / 3) * e[2]
        den = (La + Lo / 2) * (Lb + Lo / 2) * (Lc + Lo / 2)
        shift = np.where(den > 1e-10, La * Lb * Lc / np.where(den > 1e-10, den, 1.0), La * Lb * Lc)[:, None] * (
            dx[:, None] * t1 + dy[:, None] * t2)
        edge = (Lo < 1e-10) & ((La > 1e-10).astype(int) + (Lb > 1e-10) + (Lc > 1e-10) < 3)
        # an edge belongs to two faces, whose shifts agree on it: it is set, not added
        X = np.where(edge[:, None], L @ V + dx[:, None] * t1 + dy[:, None] * t2, X + shift)
    lam = np.linalg.solve((V[1:] - V[0]).T, (X - V[0]).T)
    return tuple(2 * lam - 1)


def _legendre(N, *x):
    """Products of Legendre polynomials of total degree <= N at the points x, and their gradients."""
    P = np.polynomial.legendre
    one = [[P.legval(v, np.eye(N + 1)[k]) for k in range(N + 1)] for v in x]
    der = [[P.legval(v, P.legder(np.eye(N + 1)[k])) for k in range(N + 1)] for v in x]
    modes = [m for m in itertools.product(range(N + 1), repeat=len(x)) if sum(m) <= N]
    val = np.stack([np.prod([one[d][m[d]] for d in range(len(x))], axis=0) for m in modes], axis=1)
    grad = [np.stack([np.prod([(der if d == q else one)[d][m[d]] for d in range(len(x))], axis=0) for m in modes],
                     axis=1) for q in range(len(x))]
    return val, grad


def _simplex_rule(N, dim):
    """Collapsed Gauss rule, exact for degree 2N on the reference triangle or tetrahedron."""
    g, w = np.polynomial.legendre.leggauss(N + 3)
    if dim == 2:
        a, b = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))
        return ((1 + a) * (1 - b) / 2 - 1, b), np.outer(w, w).ravel() * (1 - b) / 2
    a, b, c = (v.ravel() for v in np.meshgrid(g, g, g, indexing="ij"))
    s = (1 + b) * (1 - c) / 2 - 1
    return ((1 + a) * (-s - c) / 2 - 1, s, c), np.einsum("i,j,k->ijk", w, w, w).ravel() * (1 - b) / 2 * (
        (1 - c) / 2) ** 2


FACES = ((0, 1, 2), (0, 1, 3), (1, 2, 3), (0, 2, 3))
OPPOSITE = (3, 2, 0, 1)


class _Exact:
    """The semi-discrete Maxwell operator in 64 bits (nodal DG, upwind flux with material jumps, PEC walls)."""

    def __init__(self, N, X, tets, nverts):
        r, s, t = _nodes(N)
        V, G = _legendre(N, r, s, t)
        Vi = np.linalg.inv(V)
        D = [g @ Vi for g in G]
        q, w = _simplex_rule(N, 3)
        B = _legendre(N, *q)[0] @ Vi
        M = B.T @ (w[:, None] * B)
        # face nodes listed by their lattice position about the face's vertices, once per order of the vertices, so
        # that two elements that list a face's vertices by global number list its nodes alike
        ijk = [(i, j, k) for k in range(N + 1) for j in range(N + 1 - k) for i in range(N + 1 - k - j)]
        where = {(N - sum(m),) + m: n for n, m in enumerate(ijk)}
        tri = [(a, b, N - a - b) for a in range(N + 1) for b in range(N + 1 - a)]
        vmap, lift = [], []
        for f in range(4):
            for perm in itertools.permutations(range(3)):
                v = [FACES[f][p] for p in perm]
                rows = []
                for m in tri:
                    bary = [0] * 4
                    for vert, n in zip(v, m):
                        bary[vert] = n
                    rows.append(where[tuple(bary)])
                lam = np.stack([-(1 + r + s + t) / 2, (1 + r) / 2, (1 + s) / 2, (1 + t) / 2])[:, rows]
                a, b = 2 * lam[v[1]] - 1, 2 * lam[v[2]] - 1
                qf, wf = _simplex_rule(N, 2)
                F = _legendre(N, *qf)[0] @ np.linalg.inv(_legendre(N, a, b)[0])
                E = np.zeros((len(r), len(tri)))
                E[rows] = F.T @ (wf[:, None] * F)
                vmap.append(rows)
                lift.append(np.linalg.solve(M, E))
        to = dict(dtype=torch.float64, device=DEV)
        self.Np, self.K, self.Nfp = len(r), X.shape[0], len(tri)
        self.D = torch.as_tensor(np.concatenate(D), **to)
        lift = torch.as_tensor(np.stack(lift), **to)
        vmap = torch.as_tensor(np.array(vmap), device=DEV)
        # geometry
        J = torch.stack([(X[:, v] - X[:, 0]) / 2 for v in (1, 2, 3)], dim=2)
        self.J = torch.linalg.det(J)
        self.G = torch.linalg.inv(J)  # [K, reference direction, physical direction]
        lam_grad = torch.cat([-self.G.sum(1, keepdim=True), self.G], dim=1) / 2  # barycentric gradients
        n = -lam_grad[:, list(OPPOSITE)]
        length = n.norm(dim=2)
        self.n = (n / length[..., None]).permute(2, 0, 1)[..., None]  # [3, K, 4, 1]
        # |face Jacobian| / J: the face's height is 1 / |grad lambda|, and area / volume = 3 / height, both over their
        # reference measures (2 and 4/3)
        self.fscale = (2 * length)[..., None]
        # connectivity
        T = torch.as_tensor(tets, device=DEV)
        fv = torch.stack([T[:, list(f)] for f in FACES], dim=1)  # [K, 4, 3]
        srt, arg = fv.sort(dim=2)
        code = {p: i for i, p in enumerate(itertools.permutations(range(3)))}
        table = torch.zeros(27, dtype=torch.long, device=DEV)
        for p, i in code.items():
            table[p[0] * 9 + p[1] * 3 + p[2]] = i
        kind = table[arg[..., 0] * 9 + arg[..., 1] * 3 + arg[..., 2]] + 6 * torch.arange(4, device=DEV)
        key = (srt[..., 0] * nverts + srt[..., 1]) * nverts + srt[..., 2]
        _, inv, cnt = torch.unique(key.reshape(-1), return_inverse=True, return_counts=True)
        o = torch.argsort(inv, stable=True)
        nbr = torch.arange(4 * self.K, device=DEV)
        pair = cnt[inv[o]] == 2
        po = o[pair].reshape(-1, 2)
        nbr[po[:, 0]], nbr[po[:, 1]] = po[:, 1], po[:, 0]
        self.nbr = nbr
        self.wall = (cnt[inv] == 1).reshape(self.K, 4)
        idx = (torch.arange(self.K, device=DEV)[:, None, None] * self.Np + vmap[kind]).reshape(4 * self.K, -1)
        self.mine, self.theirs = idx.reshape(-1), idx[nbr].reshape(-1)
        self.kind = [torch.nonzero(kind.reshape(-1) == i)[:, 0] for i in range(24)]
        self.lift = lift

    def rhs(self, u, eps, mu, alpha):
        K, Np = self.K, self.Np
        d = (u.reshape(6 * K, Np) @ self.D.T).reshape(6, K, 3, Np)
        dx = torch.einsum("kdl,ckdi->clki", self.G, d)
        curl = lambda f: torch.stack([dx[f + 2, 1] - dx[f + 1, 2], dx[f, 2] - dx[f + 2, 0],  # noqa: E731
                                      dx[f + 1, 0] - dx[f, 1]])
        E, H = curl(3), -curl(0)
        flat = u.reshape(6, K * Np)
        qm = flat[:, self.mine].reshape(6, K, 4, -1)
        qp = flat[:, self.theirs].reshape(6, K, 4, -1)
        sign = torch.ones(6, K, 4, 1, dtype=u.dtype, device=u.device)
        sign[:3, self.wall] = -1
        jump = sign * qp - qm
        dE, dH = jump[:3], jump[3:]
        Z = torch.sqrt(mu / eps)
        Zm = Z[:, None].expand(K, 4)
        Zp = Zm.reshape(-1)[self.nbr].reshape(K, 4)
        Zm, Zp = Zm[..., None], Zp[..., None]
        Ym, Yp = 1 / Zm, 1 / Zp
        n = self.n.expand(3, K, 4, qm.shape[3])
        cross = lambda a, b: torch.linalg.cross(a, b, dim=0)  # noqa: E731
        fE = cross(n, Zp * dH - alpha * cross(n, dE)) / (Zm + Zp) * self.fscale
        fH = -cross(n, Yp * dE + alpha * cross(n, dH)) / (Ym + Yp) * self.fscale
        f = torch.cat([fE, fH]).reshape(6, 4 * K, -1)
        lifted = torch.zeros(6, 4 * K, Np, dtype=u.dtype, device=u.device)
        for i, at in enumerate(self.kind):
            lifted = lifted.index_copy(1, at, f[:, at] @ self.lift[i].T)
        lifted = lifted.reshape(6, K, 4, Np).sum(2)
        return torch.cat([(E + lifted[:3]) / eps[:, None], (H + lifted[3:]) / mu[:, None]])

    def step(self, u, eps, mu, dt, alpha):
        res = torch.zeros_like(u)
        for a, b in zip(LSERK_A, LSERK_B):
            res = a * res + dt * self.rhs(u, eps, mu, alpha)
            u = u + b * res
        return u


def exact(case, seed):
    inp = _inputs(case, seed)
    Np, Npad = _np(case["N"]), inp["u0"].shape[2]
    op = _Exact(case["N"], inp["X"], inp["tets"], 1 + int(inp["tets"].max()))
    to64 = lambda a: torch.as_tensor(a, device=DEV).double()  # noqa: E731
    pad = lambda a: torch.nn.functional.pad(a, (0, Npad - Np))  # noqa: E731
    u, eps = to64(inp["u0"][:, :, :Np]), to64(np.concatenate(inp["eps"]))
    mu = torch.ones_like(eps) if inp["mu"] is None else to64(inp["mu"])
    alpha, steps = case["alpha"], case["steps"]
    dt = torch.cat([torch.full((m[3].shape[0],), d, dtype=torch.float64, device=DEV)
                    for m, d in zip(inp["meshes"], inp["dts"])])[:, None]
    if case["kind"] in ("rhs", "step", "ensemble"):
        with torch.no_grad():
            if case["kind"] == "rhs":
                return pad(op.rhs(u, eps, mu, alpha))
            for _ in range(steps):
                u = op.step(u, eps, mu, dt, alpha)
            return pad(u)
    # gradients: the states at the ends of the steps are kept, each step is differentiated on its own
    recv, Eref = inp["recv"], to64(inp["Eref"])
    at = lambda v: v[:3].reshape(3, -1)[:, recv]  # noqa: E731
    states = [u]
    with torch.no_grad():
        for _ in range(steps):
            states.append(op.step(states[-1], eps, mu, dt, alpha))
    traces = torch.stack([at(v) for v in states[1:]])
    lam, deps = torch.zeros_like(u), torch.zeros_like(eps)
    for n in range(steps - 1, -1, -1):
        lam[:3].reshape(3, -1)[:, recv] += 2 * (traces[n] - Eref[n])
        v, e = states[n].detach().requires_grad_(), eps.detach().requires_grad_()
        gu, ge = torch.autograd.grad(op.step(v, e, mu, dt, alpha), (v, e), lam)
        lam, deps = gu.contiguous(), deps + ge
    if case["kind"] == "misfit":
        return {"J": ((traces - Eref) ** 2).sum(), "deps": deps, "du0": pad(lam)}
    return {"traces": traces, "deps": deps, "du0": pad(lam)}
