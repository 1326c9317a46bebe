"""The measured cases: what a user of this framework has it compute.

Six families, each through the package's public entry points:

  acoustic   LSRK steps of the acoustic solver (``binding.Solver.step``) and the state read back on the device
  record     a run that records receiver traces (``binding.Solver.record``): one data run of the surrogate workload
  adjoint    the receiver-misfit gradient with respect to c^2 (``record`` + ``adjoint``)
  elastic    LSRK steps of the elastic solver (``binding.ElasticSolver.step``)
  batch      LSRK steps of many instances of uneven size and degree (``binding.Batch.step``)
  surrogate  one gradient evaluation (forward, loss, backward) of the neural operator, or its forward alone

Meshes are the Kuhn cube (n^3 hexes x 6 tets) of the package's workloads, jittered and with shuffled vertex orders
where a case says so (every face orientation then occurs). Media and states are seeded smooth random fields.
``exact`` is the same method in plain torch, FP64, with dense element matrices built from the closed-form Bernstein
moments; it shares no code with the package.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1808_08645_gb300 import binding as B
from paper_1808_08645_gb300 import surrogate as S

RK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
RK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0, 1720146321549.0 / 2090206949498.0,
        3134564353537.0 / 4481467310338.0, 2277821191437.0 / 14882151754819.0)
FACE_VERTS = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))
F64 = torch.float64


def np3(n):
    return (n + 1) * (n + 2) * (n + 3) // 6


def np2(n):
    return (n + 1) * (n + 2) // 2


# ---------------------------------------------------------------------------
# the cases


def listed():
    return [
        # the smallest call: the FP64-parity workload's mesh in FP32, where launches and latency count
        dict(name="acoustic_n3_384", kind="acoustic", N=3, M=1, hexes=4, steps=2, prec=32, jitter=True),
        # low degree on the throughput mesh (196,608 tets)
        dict(name="acoustic_n2_196608", kind="acoustic", N=2, M=2, hexes=32, steps=1, prec=32, jitter=False),
        # the middle degree on an odd, unstructured mesh (55,566 tets, ragged last groups, all face orientations)
        dict(name="acoustic_n5_55566", kind="acoustic", N=5, M=2, hexes=21, steps=1, prec=32, jitter=True),
        # a high degree, 48,000 tets
        dict(name="acoustic_n7_48000", kind="acoustic", N=7, M=2, hexes=20, steps=1, prec=32, jitter=False),
        # the highest degree, 82,944 tets: the largest state
        dict(name="acoustic_n9_82944", kind="acoustic", N=9, M=2, hexes=24, steps=1, prec=32, jitter=False),
        # double precision, the convergence study's use
        dict(name="acoustic_n4_f64_6000", kind="acoustic", N=4, M=1, hexes=10, steps=1, prec=64, jitter=True),
        # a data run of the surrogate workload: N = 4 on 24,576 tets, point source, 64 receivers, traces to the host
        dict(name="record_n4_24576", kind="record", N=4, M=2, hexes=16, steps=32, prec=32, jitter=False),
        # the gradient of the adjoint workload (shorter run), every pressure bracket kept
        dict(name="adjoint_n5_24576", kind="adjoint", N=5, M=2, hexes=16, steps=12, prec=32, jitter=False),
        # the elastic solver at a low and a high degree
        dict(name="elastic_n3_82944", kind="elastic", N=3, M=2, hexes=24, steps=1, prec=32, jitter=False),
        dict(name="elastic_n6_24576", kind="elastic", N=6, M=2, hexes=16, steps=1, prec=32, jitter=True),
        # many small instances, N = 3..7, advanced together by replayed graphs
        dict(name="batch_n3_n7", kind="batch", M=2, instances=10, lo=7, hi=9, steps=16, prec=32),
        # training of the neural operator: 64^3 grid, batch of 8
        dict(name="surrogate_train_64", kind="surrogate", grid=64, width=32, batch=8, train=True),
    ]


def _hexes(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["acoustic"] * 5 + ["elastic"] * 2 + ["record", "adjoint", "batch", "surrogate"])
    if kind == "acoustic":
        N = rng.randint(1, 9)
        prec = 64 if rng.random() < 0.15 else 32
        hi = 8 if prec == 64 else {1: 32, 2: 32, 3: 32, 4: 28, 5: 26, 6: 24, 7: 23, 8: 21, 9: 20}[N]
        return dict(kind=kind, N=N, M=rng.choice((0, 1, 2, 2, 2, 3)), hexes=_hexes(rng, 3, hi),
                    steps=rng.randint(1, 2), prec=prec, jitter=rng.random() < 0.5)
    if kind == "elastic":
        N = rng.randint(1, 9)
        hi = {1: 24, 2: 22, 3: 20, 4: 18, 5: 16, 6: 14, 7: 12, 8: 11, 9: 10}[N]
        return dict(kind=kind, N=N, M=rng.choice((1, 2, 2, 3)), hexes=_hexes(rng, 3, hi), steps=1, prec=32,
                    jitter=rng.random() < 0.5)
    if kind == "record":
        return dict(kind=kind, N=rng.randint(3, 6), M=rng.choice((1, 2)), hexes=_hexes(rng, 4, 12),
                    steps=rng.randint(5, 24), prec=32, jitter=rng.random() < 0.5)
    if kind == "adjoint":
        return dict(kind=kind, N=rng.randint(2, 6), M=rng.choice((1, 2)), hexes=_hexes(rng, 3, 12),
                    steps=rng.randint(2, 8), prec=32, jitter=rng.random() < 0.5)
    if kind == "batch":
        lo = rng.randint(3, 7)
        return dict(kind=kind, M=rng.choice((1, 2)), instances=rng.randint(3, 10), lo=lo, hi=lo + rng.randint(0, 2),
                    steps=rng.randint(4, 16), prec=32)
    return dict(kind=kind, grid=rng.choice((16, 24, 32, 48, 64)), width=32, batch=rng.randint(1, 6),
                train=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# meshes and fields


def cube(n, jitter, seed):
    """(vxyz, etov) of the unit cube cut into n^3 hexes x 6 tets, positively oriented."""
    rng = np.random.default_rng(seed)
    g = np.linspace(0.0, 1.0, n + 1)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    v = np.stack([x, y, z], -1).reshape(-1, 3)
    if jitter:
        inner = np.all((v > 1e-9) & (v < 1 - 1e-9), axis=1)
        v[inner] += rng.uniform(-0.1 / n, 0.1 / n, (int(inner.sum()), 3))
    k, j, i = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    base = (i + (n + 1) * (j + (n + 1) * k)).reshape(-1, 1)
    step = np.array([1, n + 1, (n + 1) ** 2])
    tets = np.array([np.concatenate([[0], np.cumsum(step[list(p)])]) for p in itertools.permutations(range(3))])
    e = (base[:, :, None] + tets[None]).reshape(-1, 4).astype(np.int64)
    if jitter:
        e = np.take_along_axis(e, np.argsort(rng.random(e.shape), axis=1), axis=1)
    p = v[e]
    neg = np.einsum("ki,ki->k", np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), p[:, 3] - p[:, 0]) < 0
    e[neg, 2], e[neg, 3] = e[neg, 3].copy(), e[neg, 2].copy()
    return np.ascontiguousarray(v), np.ascontiguousarray(e)


def lattice(n):
    """Multi-indices of degree n in the library's order."""
    return [(n - j - k - l, j, k, l) for l in range(n + 1) for k in range(n - l + 1) for j in range(n - l - k + 1)]


def domain_points(v, e, n):
    """[K, np3(n), 3] domain points on the GPU (the centroid for n = 0)."""
    w = torch.tensor(lattice(n) if n else [(1, 1, 1, 1)], dtype=F64, device="cuda") / (n if n else 4)
    x = torch.tensor(v, device="cuda")[torch.tensor(e, device="cuda")]
    return torch.einsum("pa,kad->kpd", w, x)


def smooth(x, seed, lo, hi):
    """A smooth random field in [lo, hi] at the points x [..., 3]."""
    g = np.random.default_rng(seed)
    out = torch.zeros(x.shape[:-1], dtype=F64, device=x.device)
    for _ in range(6):
        kv = g.integers(1, 4, 3) * math.pi
        out += torch.cos(x[..., 0] * kv[0] + x[..., 1] * kv[1] + x[..., 2] * kv[2] + g.uniform(0, 2 * math.pi)) / 6
    return lo + (hi - lo) * (out + 1) / 2


def rounded(x, prec):
    return x.float().double() if prec == 32 else x


def wave_state(v, e, N, fields, seed, prec):
    x = domain_points(v, e, N)
    return rounded(torch.stack([smooth(x, 100 * seed + f, -1.0, 1.0) for f in range(fields)]), prec)


def media(v, e, M, n, seed, prec):
    x = domain_points(v, e, M)
    return [rounded(smooth(x, 100 * seed + 50 + f, 0.5, 2.0), prec) for f in range(n)]


def source_point(seed):
    return np.random.default_rng(seed).uniform([0.3, 0.3, 0.6], [0.7, 0.7, 0.8])


def receivers():
    c = (np.arange(8) + 0.5) / 8
    x, y = np.meshgrid(c, c, indexing="ij")
    return np.stack([x.ravel(), y.ravel(), np.full(64, 0.9)], 1)


def cfl(v, e, N, c2max, factor=0.5):
    """The library's CFL rule; the cases hand their solver the same number that ``exact`` uses."""
    grad, _ = geometry(v, e)
    ratio = 3.0 * float(grad.square().sum(-1).sqrt().max())
    return factor / (math.sqrt(c2max) * (N + 1) * (N + 3) / 3.0 * ratio)


def instances(case, seed):
    """(mesh, N) of the instances of a batch: sizes and degrees do not depend on the seed."""
    out = []
    for i in range(case["instances"]):
        n = case["lo"] + i % (case["hi"] - case["lo"] + 1)
        out.append((cube(n, False, 0), 3 + (3 * i) % 5))
    return out


# ---------------------------------------------------------------------------
# prepare and run


def prepare(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        return prepare_surrogate(case, seed)
    if kind == "batch":
        return prepare_batch(case, seed)
    N, M, prec = case["N"], case["M"], case["prec"]
    v, e = cube(case["hexes"], case["jitter"], seed)
    dtype = torch.float32 if prec == 32 else F64
    nf = 9 if kind == "elastic" else 4
    if kind == "elastic":
        med = media(v, e, M, 3, seed, prec)
        s = B.ElasticSolver(v, e, N, M, prec)
        s.set_media(*(m.cpu().numpy() for m in med))
        dt = cfl(v, e, N, 2.0 * (2.0 + 2.0 * 2.0))
    else:
        c2 = media(v, e, M, 1, seed, prec)[0].cpu().numpy()
        s = B.Solver(v, e, N, M, prec)
        s.set_c2(c2)
        dt = cfl(v, e, N, 2.0)
    st = dict(case=case, s=s, dt=dt, q=torch.empty((nf, len(e), np3(N)), dtype=dtype, device="cuda"))
    q0 = wave_state(v, e, N, nf, seed, prec)
    if kind in ("acoustic", "elastic"):
        q0 = q0.to(dtype).contiguous()
        s.set_state_device(q0, None, prec)
        torch.cuda.synchronize()
        return st
    s.set_receivers(receivers())
    s.set_point_source(source_point(seed), B.ricker_samples(dt, case["steps"], f0=12.0, t0=4.0 * dt))
    st["q0"] = q0.cpu().numpy()
    if kind == "adjoint":
        st["g"] = np.random.default_rng(seed).standard_normal((case["steps"], 64))
    return st


def prepare_batch(case, seed):
    inst = instances(case, seed)
    b = B.Batch([m for m, _ in inst], [n for _, n in inst], case["M"], case["prec"])
    for i, ((v, e), N) in enumerate(inst):
        b.set_c2(i, media(v, e, case["M"], 1, seed + i, case["prec"])[0].cpu().numpy())
        b.set_state(i, wave_state(v, e, N, 4, seed + i, case["prec"]).cpu().numpy())
    return dict(case=case, s=b, dt=batch_dt(inst))


def batch_dt(inst):
    return min(cfl(v, e, N, 2.0) for (v, e), N in inst)


def surrogate_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    G, nb = case["grid"], case["batch"]
    c = (torch.arange(G, dtype=F64, device="cuda") + 0.5) / G
    pts = torch.stack(torch.meshgrid(c, c, c, indexing="ij"), -1)
    x = torch.empty((nb, G, G, G, 6), device="cuda")
    for b in range(nb):
        xs = torch.tensor(source_point(seed + b), device="cuda")
        d2 = (pts - xs).square().sum(-1)
        x[b, ..., 0] = ((smooth(pts, 100 * seed + b, 0.5, 2.0) - 1.25) / 0.75).float()
        x[b, ..., 1:4] = (2 * pts - 1).float()
        x[b, ..., 4] = torch.exp(-d2 / (2 * 0.05 ** 2)).float()
        x[b, ..., 5] = (2 * d2.sqrt()).float()
    return x, torch.randn((nb, 64, 512), generator=g, device="cuda")


def prepare_surrogate(case, seed):
    net = S.Net(S.default_config(grid=case["grid"], width=case["width"]), seed=seed)
    x, y = surrogate_inputs(case, seed)
    return dict(case=case, net=net, x=x, y=y)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("acoustic", "elastic"):
        state["s"].step(state["dt"], case["steps"])
        state["s"].get_state_device(state["q"], None, case["prec"])
        return state["q"]
    if kind == "record":  # the record of a new run starts from its initial state, as each data run does
        state["s"].set_state(state["q0"])
        traces = state["s"].record(state["dt"], case["steps"], case["steps"])
        state["s"].get_state_device(state["q"], None, case["prec"])
        return [traces, state["q"]]
    if kind == "adjoint":
        state["s"].set_state(state["q0"])
        traces = state["s"].record(state["dt"], case["steps"], 0)
        return [traces, state["s"].adjoint(state["g"])[0]]
    if kind == "batch":
        b = state["s"]
        b.step(state["dt"], case["steps"])
        return [b.get_state(i) for i in range(b.n)]
    net = state["net"]
    y, cache = net.forward(state["x"])
    if not case["train"]:
        return y
    loss, dy = net.loss(y, state["y"])
    g = net.backward(cache, dy)
    return [y, loss, {k: t for k, t in g.items()}]


# ---------------------------------------------------------------------------
# the work a pass cannot do without


def stage_flops(N, M, fields, projections, lifted):
    """Operations of one stage per element with the sparse Bernstein operators: derivatives and their elevation, the
    lift pyramids of `lifted` quantities per face, and `projections` weight-adjusted projections."""
    Np, v = np3(N), np3(N - 1)
    vol = 24 * v + 4 * fields * Np
    if fields == 9:
        vol = 2 * 18 * 4 * v // 2 + 4 * 9 * Np
    lift = 4 * lifted * (3 * np2(N - 1) + 4 * np2(N) + 3 * np3(N - 1)) + 4 * fields * Np
    proj = np3(M) * np3(N + M) + sum(4 * np3(n) for n in range(N, N + M)) + 2 * sum(4 * np3(n) for n in range(N))
    return 2 * (vol + lift + projections * proj + 2 * fields * Np + 16 * 4 * np2(N))


def stage_bytes(N, M, fields, med, size):
    return size * ((3 * fields + fields * 4 / 5) * np3(N) + med * np3(M) + 9) + 16


def work(case):
    kind = case["kind"]
    if kind == "surrogate":
        G, C, nb = case["grid"], case["width"], case["batch"]
        P, L, H, T, R = nb * G ** 3, 4, 128, 512, 64
        nm = 6 * 6 * 6
        spec = 2 * P * C * 6 * (1 + 6 / G + 36 / G ** 2) * 2 + 2 * nb * nm * C * C
        fwd = 2 * P * C * 6 + L * (2 * P * C * C + spec) + 2 * nb * R * (C * H + H * T)
        params = L * nm * C * C * 4
        if not case["train"]:
            return {"bytes": P * 24 + L * P * C * 4 * 2 + params, "flops": fwd}
        # forward: each layer reads its input and writes its output and pre-activation; backward: each layer reads its
        # input, its pre-activation and the output gradient and writes the input gradient
        return {"bytes": P * 24 * 2 + L * P * C * 4 * (3 + 4) + 3 * params, "flops": 3 * fwd}
    if kind == "batch":
        out = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["instances"]):
            n, N = case["lo"] + i % (case["hi"] - case["lo"] + 1), 3 + (3 * i) % 5
            K = 6 * n ** 3
            out["bytes"] += 5 * case["steps"] * K * stage_bytes(N, case["M"], 4, 1, 4) + K * np3(N) * 4 * 12
            out["flops"] += 5 * case["steps"] * K * stage_flops(N, case["M"], 4, 1, 2)
        return out
    N, M, K, size = case["N"], case["M"], 6 * case["hexes"] ** 3, case["prec"] // 8
    nst = 5 * case["steps"]
    if kind == "elastic":
        return {"bytes": nst * K * stage_bytes(N, M, 9, 3, size) + 2 * 9 * K * np3(N) * size,
                "flops": nst * K * stage_flops(N, M, 9, 10, 6)}
    by, fl = nst * K * stage_bytes(N, M, 4, 1, size), nst * K * stage_flops(N, M, 4, 1, 2)
    if kind == "adjoint":
        # per stage: the recorded bracket written and read, the two dual states read and written
        by += nst * K * size * (2 * np3(N) + 16 * np3(N) + 2 * np3(M) + 9) + 16 * nst * K
        pairs = np3(N) ** 2 + np3(M) * np3(2 * N)
        fl += fl + nst * K * 2 * pairs
    return {"bytes": by + 2 * 4 * K * np3(N) * size, "flops": fl}


# ---------------------------------------------------------------------------
# the same in plain torch, FP64


FACT = np.array([float(math.factorial(i)) for i in range(40)])


def fact(a):
    """Products of the factorials of multi-indices [..., d]."""
    return FACT[np.asarray(a)].prod(-1)


def moments(A, Bx):
    """[len(A), len(Bx)] integrals of B_a B_b over the unit-measure simplex of dimension len(a) - 1."""
    A, Bx = np.array(A), np.array(Bx)
    n, m, d = A[0].sum(), Bx[0].sum(), A.shape[1] - 1
    return FACT[n] * FACT[m] * FACT[d] / FACT[n + m + d] * fact(A[:, None] + Bx[None]) / (
        fact(A)[:, None] * fact(Bx)[None])


class Ops:
    """Dense element matrices of degree N (and the M-weighted masses)."""

    def __init__(self, N, M):
        A = lattice(N)
        at = {a: i for i, a in enumerate(A)}
        low = {a: i for i, a in enumerate(lattice(N - 1))}
        Minv = np.linalg.inv(moments(A, A))
        D = np.zeros((4, len(A), len(A)))
        for m in range(4):
            up = np.zeros((len(A), len(low)))
            dn = np.zeros((len(low), len(A)))
            for a, i in at.items():
                for d in range(4):
                    b = tuple(x - (d == y) for y, x in enumerate(a))
                    if a[d] > 0:
                        up[i, low[b]] += a[d] / N
                b = tuple(x - (m == y) for y, x in enumerate(a))
                if a[m] > 0:
                    dn[low[b], i] = N
            D[m] = up @ dn
        F2 = [(N - b1 - b2, b1, b2) for b2 in range(N + 1) for b1 in range(N - b2 + 1)]
        Mf = moments(F2, F2)
        lift = np.zeros((4, len(A), len(F2)))
        idx = np.zeros((4, 6, len(F2)), np.int64)  # volume index of face node b with its vertices in order perm
        self.perms = list(itertools.permutations(range(3)))
        for f in range(4):
            own = []
            for b in F2:
                a = [0, 0, 0, 0]
                for x in range(3):
                    a[FACE_VERTS[f][x]] = b[x]
                own.append(at[tuple(a)])
            lift[f] = Minv[:, own] @ Mf
            for p, perm in enumerate(self.perms):
                for q, b in enumerate(F2):
                    a = [0, 0, 0, 0]
                    for x in range(3):
                        a[FACE_VERTS[f][perm[x]]] = b[x]
                    idx[f, p, q] = at[tuple(a)]
        # lift of a flux in the order perm: columns permuted accordingly
        pos = [{int(i): q for q, i in enumerate(idx[f, 0])} for f in range(4)]
        lp = np.zeros((4, 6) + lift.shape[1:])
        for f in range(4):
            for p in range(6):
                lp[f, p] = lift[f][:, [pos[f][int(i)] for i in idx[f, p]]]
        W = []
        for b in lattice(M):
            c0 = FACT[N] ** 2 * FACT[M] * 6 / FACT[2 * N + M + 3]
            a = np.array(A)
            T = c0 * fact(a[:, None] + a[None] + np.array(b)) / (fact(a)[:, None] * fact(a)[None] * fact(b))
            W.append(Minv @ T)
        dev = dict(dtype=F64, device="cuda")
        self.D = torch.tensor(D, **dev)
        self.lift = torch.tensor(lp, **dev)
        self.idx = torch.tensor(idx, device="cuda")
        self.W = torch.tensor(np.array(W), **dev)
        self.Minv = torch.tensor(Minv, **dev)


def geometry(v, e):
    """(grad lambda [K, 4, 3], volume [K]) on the GPU."""
    x = torch.tensor(v, device="cuda")[torch.tensor(e, device="cuda")]
    J = (x[:, 1:] - x[:, :1]).transpose(1, 2)
    inv = torch.linalg.inv(J)
    return torch.cat([-inv.sum(1, keepdim=True), inv], 1), torch.linalg.det(J) / 6


class Ref:
    """Connectivity and geometry of a mesh, and traces in the order of the faces' sorted vertices."""

    def __init__(self, v, e, N, M):
        self.o = Ops(N, M)
        self.grad, self.vol = geometry(v, e)
        K = len(e)
        fv = np.stack([e[:, list(f)] for f in FACE_VERTS], 1)
        order = np.argsort(fv, axis=2)
        code = {p: i for i, p in enumerate(self.o.perms)}
        table = np.zeros((3, 3, 3), np.int64)
        for p, i in code.items():
            table[p] = i
        perm = table[order[..., 0], order[..., 1], order[..., 2]]
        key = np.sort(fv, axis=2).reshape(-1, 3)
        k = (key[:, 0] * len(v) + key[:, 1]) * len(v) + key[:, 2]
        o = np.argsort(k, kind="stable")
        nb = np.full(4 * K, -1, np.int64)
        same = k[o[1:]] == k[o[:-1]]
        nb[o[:-1][same]], nb[o[1:][same]] = o[1:][same], o[:-1][same]
        self.K = K
        self.perm = torch.tensor(perm, device="cuda")
        self.nb = torch.tensor(nb, device="cuda")
        self.nidx = self.o.idx[torch.arange(4, device="cuda")[None], self.perm]  # [K, 4, Nfp]
        gn = self.grad.square().sum(-1).sqrt()
        self.n = -self.grad / gn[..., None]
        self.fs = 3.0 * gn  # |f| / |D|
        self.wall = (self.nb < 0).reshape(K, 4)

    def trace(self, q):
        """Own and neighbour traces [K, 4, Nfp] of q [K, Np] (the neighbour's own value repeated on walls)."""
        own = torch.gather(q[:, None].expand(-1, 4, -1), 2, self.nidx)
        other = own.reshape(4 * self.K, -1)[self.nb.clamp(min=0)].reshape(own.shape)
        return own, torch.where(self.wall[..., None], own, other)

    def lifted(self, f, flux):
        """|f|/|D| L^f flux of face f, flux [K, Nfp] in the sorted order."""
        L = self.o.lift[f]
        out = torch.zeros((self.K, L.shape[1]), dtype=F64, device="cuda")
        for p in range(6):
            m = (self.perm[:, f] == p).to(F64)[:, None]
            out = out + (flux * m) @ L[p].T
        return out * self.fs[:, f:f + 1]

    def weight(self, c, r):
        """M^-1 M_c r, c [K, Mp]."""
        out = 0.0
        for b in range(c.shape[1]):
            out = out + c[:, b:b + 1] * (r @ self.o.W[b].T)
        return out


def acoustic_rhs(R, c2, q, src=None):
    p, vel = q[0], q[1:]
    D, g = R.o.D, R.grad
    ru = [0.0, 0.0, 0.0]
    rp = 0.0
    for m in range(4):
        dp = p @ D[m].T
        for d in range(3):
            ru[d] = ru[d] - g[:, m, d:d + 1] * dp
        rp = rp - (g[:, m, 0:1] * vel[0] + g[:, m, 1:2] * vel[1] + g[:, m, 2:3] * vel[2]) @ D[m].T
    pm, pp = R.trace(p)
    pp = torch.where(R.wall[..., None], -pm, pp)
    ndu = 0.0
    for d in range(3):
        um, up = R.trace(vel[d])
        ndu = ndu + R.n[..., d:d + 1] * (up - um)
    jp = pp - pm
    Fp, Fu = 0.5 * (jp - ndu), 0.5 * (ndu - jp)
    for f in range(4):
        rp = rp + R.lifted(f, Fp[:, f])
        lu = R.lifted(f, Fu[:, f])
        for d in range(3):
            ru[d] = ru[d] + R.n[:, f, d:d + 1] * lu
    if src is not None:
        rp = rp + src
    return torch.stack([R.weight(c2, rp), *ru])


# the nine fields: v_x v_y v_z, s_xx s_yy s_zz s_yz s_xz s_xy; A_i as index pairs (stress row, velocity row)
ELASTIC_A = (((0, 0), (5, 1), (4, 2)), ((5, 0), (1, 1), (3, 2)), ((4, 0), (3, 1), (2, 2)))


def elastic_rhs(R, med, q):
    rho_inv, lam, mu = med
    D, g = R.o.D, R.grad
    br = [0.0] * 9
    der = lambda a, i: sum(g[:, m, i:i + 1] * (a @ D[m].T) for m in range(4))  # noqa: E731
    jump = []
    for a in range(9):
        own, oth = R.trace(q[a])
        jump.append(torch.where(R.wall[..., None], -2 * own if a >= 3 else torch.zeros_like(own), oth - own))
    for i in range(3):
        for s, c in ELASTIC_A[i]:
            br[c] = br[c] + der(q[3 + s], i)
            br[3 + s] = br[3 + s] + der(q[c], i)
    At = [0.0] * 3  # A_n^T [sigma]
    Av = [0.0] * 6  # A_n [v]
    for i in range(3):
        for s, c in ELASTIC_A[i]:
            At[c] = At[c] + R.n[..., i:i + 1] * jump[3 + s]
            Av[s] = Av[s] + R.n[..., i:i + 1] * jump[c]
    Fv = [0.5 * t for t in At]
    Fs = [0.5 * t for t in Av]
    for i in range(3):
        for s, c in ELASTIC_A[i]:
            Fv[c] = Fv[c] + 0.5 * R.n[..., i:i + 1] * Av[s]
            Fs[s] = Fs[s] + 0.5 * R.n[..., i:i + 1] * At[c]
    for f in range(4):
        for a in range(9):
            br[a] = br[a] + R.lifted(f, (Fv + Fs)[a][:, f])
    out = [R.weight(rho_inv, br[c]) for c in range(3)]
    tr = R.weight(lam, br[3] + br[4] + br[5])
    out += [2 * R.weight(mu, br[3 + s]) + tr for s in range(3)]
    out += [R.weight(mu, br[3 + s]) for s in range(3, 6)]
    return torch.stack(out)


def lsrk(rhs, q, dt, steps, on_step=None):
    res = torch.zeros_like(q)
    for n in range(steps):
        for s in range(5):
            res = RK_A[s] * res + dt * rhs(q, 5 * n + s)
            q = q + RK_B[s] * res
        if on_step:
            on_step(q)
    return q


def locate(R, v, e, x):
    """(element, barycentric coordinates) of a point: the lowest element that holds it."""
    v0 = torch.tensor(v, device="cuda")[torch.tensor(e[:, 0], device="cuda")]
    lam = torch.einsum("kmd,kd->km", R.grad, torch.tensor(x, device="cuda")[None] - v0)
    lam[:, 0] += 1
    k = int(torch.nonzero((lam >= -1e-12).all(1))[0])
    return k, lam[k].clamp(min=0).cpu().numpy()


def basis_at(N, lam):
    return torch.tensor([FACT[N] / fact(a) * math.prod(float(lam[i]) ** a[i] for i in range(4))
                         for a in lattice(N)], dtype=F64, device="cuda")


def exact(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        return exact_surrogate(case, seed)
    if kind == "batch":
        inst = instances(case, seed)
        dt, out = batch_dt(inst), []
        for i, ((v, e), N) in enumerate(inst):
            R = Ref(v, e, N, case["M"])
            c2 = media(v, e, case["M"], 1, seed + i, case["prec"])[0]
            q = lsrk(lambda q, s: acoustic_rhs(R, c2, q), wave_state(v, e, N, 4, seed + i, case["prec"]), dt,
                     case["steps"])
            out.append(q.cpu().numpy())
        return out
    N, M, prec = case["N"], case["M"], case["prec"]
    v, e = cube(case["hexes"], case["jitter"], seed)
    R = Ref(v, e, N, M)
    if kind == "elastic":
        med = media(v, e, M, 3, seed, prec)
        return lsrk(lambda q, s: elastic_rhs(R, med, q), wave_state(v, e, N, 9, seed, prec),
                    cfl(v, e, N, 2.0 * (2.0 + 2.0 * 2.0)), case["steps"])
    c2, q0, dt = media(v, e, M, 1, seed, prec)[0], wave_state(v, e, N, 4, seed, prec), cfl(v, e, N, 2.0)
    if kind == "acoustic":
        return lsrk(lambda q, s: acoustic_rhs(R, c2, q), q0, dt, case["steps"])
    # stage times of the scheme: c_s of its Butcher form
    times, y, k = [], 0.0, 0.0
    for s in range(5):
        times.append(y)
        k = RK_A[s] * k + 1.0
        y += RK_B[s] * k
    ke, lam = locate(R, v, e, source_point(seed))
    vec = torch.linalg.solve(torch.linalg.inv(R.o.Minv), basis_at(N, lam)) / R.vol[ke]
    t = (np.arange(case["steps"])[:, None] + np.array(times)[None]) * dt
    a = (math.pi * 12.0 * (t - 4.0 * dt)) ** 2
    amp = ((1 - 2 * a) * np.exp(-a)).ravel()
    unit = torch.zeros((len(e), np3(N)), dtype=F64, device="cuda")
    unit[ke] = vec
    at = [locate(R, v, e, x) for x in receivers()]
    rk = torch.tensor([a[0] for a in at], device="cuda")
    rb = torch.stack([basis_at(N, a[1]) for a in at])
    traces = []

    def read(q):
        traces.append((q[0][rk] * rb).sum(1))

    if kind == "record":
        q = lsrk(lambda q, s: acoustic_rhs(R, c2, q, amp[s] * unit), q0, dt, case["steps"], read)
        return [torch.stack(traces).cpu().numpy(), q]
    if case["steps"] * 5 * len(e) * np3(N) * 8 * 160 > 150e9:  # autograd keeps every stage
        return None
    c2.requires_grad_()
    lsrk(lambda q, s: acoustic_rhs(R, c2, q, amp[s] * unit), q0, dt, case["steps"], read)
    tr = torch.stack(traces)
    g = torch.tensor(np.random.default_rng(seed).standard_normal((case["steps"], 64)), device="cuda")
    (gc,) = torch.autograd.grad((g * tr).sum(), [c2])
    return [tr.detach().cpu().numpy(), gc.cpu().numpy()]


def exact_surrogate(case, seed):
    """The network's forward (and autograd's gradients) in FP64."""
    cfg = S.default_config(grid=case["grid"], width=case["width"])
    net = S.Net(cfg, seed=seed)
    p = {k: t.double().requires_grad_(case["train"]) for k, t in net.p.items()}
    G, C = cfg["grid"], cfg["width"]
    i, k = torch.arange(G, dtype=F64, device="cuda")[:, None] + 0.5, torch.arange(6, dtype=F64, device="cuda")[None]
    phi = torch.cos(math.pi * k * i / G) * math.sqrt(2.0 / G)
    phi[:, 0] = math.sqrt(1.0 / G)
    phi = phi.float().double()  # the plan's bases are held in 32 bits
    x, target = surrogate_inputs(case, seed)
    u = x.double() @ p["W0"] + p["b0"]
    for l in range(cfg["layers"]):
        s = torch.einsum("bxyzc,zk->bxykc", u, phi)
        s = torch.einsum("bxykc,yj->bxjkc", s, phi)
        s = torch.einsum("bxjkc,xi->bijkc", s, phi)
        t = torch.einsum("bijkc,ijkcd->bijkd", s, p[f"W{l}_sp"].reshape(6, 6, 6, C, C))
        t = torch.einsum("bijkd,xi->bxjkd", t, phi)
        t = torch.einsum("bxjkd,yj->bxykd", t, phi)
        t = torch.einsum("bxykd,zk->bxyzd", t, phi)
        u = torch.nn.functional.gelu(u @ p[f"W{l}_pw"] + p[f"b{l}_pw"] + t)
    rx, ry, rz = (torch.tensor(cfg[n], device="cuda") for n in ("rx", "ry", "rz"))
    r = sum(u[:, rx + a, ry + b, rz + c] for a in (0, 1) for b in (0, 1) for c in (0, 1)) / 8
    y = torch.nn.functional.gelu(r @ p["W1"] + p["b1"]) @ p["W2"] + p["b2"]
    if not case["train"]:
        return y
    loss = (y - target.double()).square().mean()
    names = list(p)
    g = torch.autograd.grad(loss, [p[n] for n in names])
    return [y.detach(), loss.detach().reshape(1), dict(zip(names, g))]
