"""The work a user of this library has it do, as cases that can be timed and compared.

A case names one call (or the pair of calls a program makes together) of the public binding
`paper_2602_13841_gb300.stmg.Solver` with its sizes:

  apply     y = J_n(U) x on the finest level, FP64 (the operator of the outer FGMRES) or FP32
            (the level operator of the multigrid preconditioner)
  residual  R_n(U; V_prev), FP64 (every Newton step and line-search trial)
  sweep     two Vanka sweeps from zero on the finest level, as a V-cycle's pre-smoothing does
            (the second one computes the level residual first)
  build     the preconditioner rebuilt at a new state (level states, patch inverses of every
            level, coarse factorisation), then one sweep on every smoothed level
  solve     one whole slab: initial guess and Newton-FGMRES to the case's tolerance

Sizes come from the benchmark's workloads (2D 256^2 Q3/P2 DG(2); 3D 64^3 Q2/P1 DG(2); 3D 64^3
Q3/P2 DG(1); the 16^3 cavity), from the serving stream's shapes (2D 16..256, 3D 8..48, r = 1..3,
k = 0..2) and from the tests' small meshes.  `exact` restates the operator, the residual and the
Vanka sweep in plain torch FP64 from the assembled definition (no sum factorisation, dense
patch solves).
"""
import itertools
import math

import numpy as np
import torch
from numpy.polynomial import legendre as npleg

from paper_2602_13841_gb300 import inputs, stmg

DEV = "cuda"


def listed():
    return [
        # the outer Krylov operator of the 2D headline workload
        dict(name="apply64_2d_256_q3_dg2", op="apply", d=2, n=256, r=2, k=2, prec=64, amp=0.1),
        # the level operator of the same workload's preconditioner
        dict(name="apply32_2d_256_q3_dg2", op="apply", d=2, n=256, r=2, k=2, prec=32, amp=0.1),
        # the smallest problem that is run (8 x 8 cells): latency and launches
        dict(name="apply64_2d_8_q2_dg1", op="apply", d=2, n=8, r=1, k=1, prec=64, amp=0.0),
        # the outer Krylov operator of the 3D workload, mapped mesh
        dict(name="apply64_3d_64_q2_dg2", op="apply", d=3, n=64, r=1, k=2, prec=64, amp=0.1),
        # the 3D level operator at the higher order, an odd mesh (ragged colour classes)
        dict(name="apply32_3d_37_q3_dg1", op="apply", d=3, n=37, r=2, k=1, prec=32, amp=0.1),
        # a Newton residual of the lid-driven cavity's mesh
        dict(name="residual_3d_16_q3_dg2", op="residual", d=3, n=16, r=2, k=2, prec=64, amp=0.0, problem="CAV3D"),
        # the smoother of the 2D headline workload: the largest share of its solve
        dict(name="sweep32_2d_256_q3_dg2", op="sweep", d=2, n=256, r=2, k=2, prec=32, amp=0.1, fp16=0),
        # the smoother of the 3D workload (patches of 85 rows) ...
        dict(name="sweep32_3d_32_q2_dg2", op="sweep", d=3, n=32, r=1, k=2, prec=32, amp=0.1, fp16=0),
        # ... and of the 3D Q3/P2 workloads (patches of 202 rows)
        dict(name="sweep32_3d_16_q3_dg2", op="sweep", d=3, n=16, r=2, k=2, prec=32, amp=0.0, fp16=0),
        # rebuilding the preconditioner in 3D, the share of a slab that grows with the order
        dict(name="build32_3d_16_q3_dg1", op="build", d=3, n=16, r=2, k=1, prec=32, amp=0.0, fp16=0),
        # a small serving request: launches and host round trips
        dict(name="solve_2d_32_q2_dg1", op="solve", d=2, n=32, r=1, k=1, prec=32, amp=0.1, problem="MMS2D", re=400.0,
             sweeps=1, sweeps_tc=0),
        # the headline solve on a quarter of its cells
        dict(name="solve_2d_128_q3_dg2", op="solve", d=2, n=128, r=2, k=2, prec=32, amp=0.1, problem="TG2D", re=1000.0,
             sweeps=2, sweeps_tc=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "residual", "sweep", "sweep", "build", "solve"])
    d = rng.choice([2, 3])
    amp = rng.choice([0.0, 0.05, 0.1])
    k = rng.choice([0, 1, 2])
    if op in ("apply", "residual"):
        r = rng.choice([1, 2, 2, 3] if d == 2 else [1, 1, 2, 3])
        n = _log_int(rng, 4, 256) if d == 2 else _log_int(rng, 3, {1: 56, 2: 40, 3: 24}[r])
        case = dict(op=op, d=d, n=n, r=r, k=k, amp=amp, prec=64)
        if op == "apply":
            case["prec"] = rng.choice([32, 64])
        else:
            case["problem"] = rng.choice(["TG2D", "MMS2D"] if d == 2 else ["TG3D", "MMS3D", "CAV3D"])
        return case
    if op == "sweep":
        r = rng.choice([1, 2, 2, 3] if d == 2 else [1, 1, 2])
        # meshes that coarsen to at most 3 cells a side (5 in 2D)
        n = rng.choice([8, 12, 16, 20, 24, 32, 40, 48, 64, 80, 96, 128, 192] if d == 2 else [4, 6, 8, 12, 16, 24])
        if d == 3 and r == 2:
            n = min(n, 12)
        return dict(op=op, d=d, n=n, r=r, k=k, amp=amp, prec=rng.choice([32, 32, 32, 64]), fp16=rng.choice([0, 0, 0, 0, 1]))
    if op == "build":
        r = rng.choice([1, 2])
        n = rng.choice([8, 12, 16, 24, 32, 48, 64, 96, 128] if d == 2 else ([4, 8, 12, 16] if r == 1 else [4, 8]))
        return dict(op=op, d=d, n=n, r=r, k=k, amp=amp, prec=rng.choice([32, 32, 64]), fp16=0)
    return dict(op=op, d=2, n=rng.choice([16, 24, 32, 48, 64]), r=rng.choice([1, 2]), k=rng.choice([1, 2]), prec=32,
                amp=amp, problem=rng.choice(["MMS2D", "TG2D"]), re=float(rng.randrange(100, 400)),
                sweeps=rng.choice([1, 2]), sweeps_tc=rng.choice([0, 8]))


# ------------------------------------------------------------------------------------ inputs
NU = {2: 1e-3, 3: 1.0 / 400}
TAU = {2: 0.05, 3: 0.01}
T0 = 0.3


def _physics(case):
    nu = 1.0 / case["re"] if "re" in case else NU[case["d"]]
    return nu, TAU[case["d"]]


def _vertices(case, seed):
    return inputs.vertices(case["d"], case["n"], case["amp"], seed)


def _sizes(case):
    d, n, r, k = case["d"], case["n"], case["r"], case["k"]
    n1 = (r + 1) * n + 1
    nv = d * n1 ** d
    npc = math.comb(r + d, d)
    return n1, nv, n ** d * npc, npc, (k + 1) * (nv + n ** d * npc)


def _flow(case, gen, n1):
    """One velocity field on the node grid: a vortex with seeded phases plus 1 % noise."""
    d = case["d"]
    x = torch.linspace(0.0, 1.0, n1, dtype=torch.float64, device=DEV)
    ph = 2 * math.pi * torch.rand(d, d, generator=gen, dtype=torch.float64, device=DEV)
    out = []
    for c in range(d):
        f = torch.ones((), dtype=torch.float64, device=DEV)
        for l in range(d):                               # axis l is the l-th fastest index
            v = torch.sin(math.pi * (1 + (c == l)) * x + ph[c, l])
            f = f * v.reshape([-1 if m == d - 1 - l else 1 for m in range(d)])
        out.append(f.expand([n1] * d).reshape(-1))
    v = torch.cat(out)
    return v + 0.01 * torch.randn(v.numel(), generator=gen, dtype=torch.float64, device=DEV)


def _vectors(case, seed):
    """What the call reads, by name, in FP64: the state U (a flow that changes over the slab's time
    nodes), a Krylov vector or right-hand side x, and the velocity before the slab."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * (seed % 1000003) + 17)
    n1, nv, npr, _, nst = _sizes(case)
    k = case["k"]
    v0, v1 = _flow(case, gen, n1), _flow(case, gen, n1)
    U = torch.empty(nst, dtype=torch.float64, device=DEV)
    for a in range(k + 1):
        U[a * nv:(a + 1) * nv] = v0 + 0.1 * (a + 1) / (k + 1) * v1
    U[(k + 1) * nv:] = 0.1 * torch.randn((k + 1) * npr, generator=gen, dtype=torch.float64, device=DEV)
    return U, torch.randn(nst, generator=gen, dtype=torch.float64, device=DEV), v0


def _solver(case, seed, stream=None, **kw):
    nu, tau = _physics(case)
    p = stmg.default_params(dim=case["d"], n_cells_1d=case["n"], r=case["r"], k=case["k"], nu=nu, tau=tau,
                            problem=case.get("problem", "TG2D" if case["d"] == 2 else "MMS3D"),
                            precond_precision=stmg.STMG_FP32 if case["prec"] == 32 else stmg.STMG_FP64,
                            vanka_fp16=int(case.get("fp16", 0)), **kw)
    return stmg.Solver(p, _vertices(case, seed), stream=stream)


def prepare(case, seed):
    op = case["op"]
    st = {"op": op, "case": case}
    if op == "solve":
        # the program's stream (the V-cycle graph needs one of its own), the velocity at the start of
        # the slab: the problem's initial field plus 1 % seeded noise inside
        st["stream"] = torch.cuda.Stream()
        S = _solver(case, seed, st["stream"].cuda_stream, newton_rtol=1e-10, newton_atol=0.0, nu1=case["sweeps"],
                    nu2=case["sweeps"], nu_tc=case["sweeps_tc"])
        n1, nv, _, _, nst = _sizes(case)
        with torch.cuda.stream(st["stream"]):
            V0 = torch.empty(nv, dtype=torch.float64, device=DEV)
            S.initial_condition(V0)
            gen = torch.Generator(device=DEV)
            gen.manual_seed(seed)
            noise = 2.0 * torch.rand(nv, generator=gen, dtype=torch.float64, device=DEV) - 1.0
            inner = torch.ones([n1] * case["d"], dtype=torch.float64, device=DEV)
            for l in range(case["d"]):
                inner.select(l, 0).zero_()
                inner.select(l, n1 - 1).zero_()
            # (a field at rest, as the manufactured solution's, starts from noise of absolute size 1e-2)
            V0 += 0.01 * V0.abs().max().clamp(min=1.0) * noise * inner.reshape(-1).repeat(case["d"])
            st.update(S=S, V0=V0, U=torch.empty(nst, dtype=torch.float64, device=DEV))
        return st
    U, x, vprev = _vectors(case, seed)
    S = _solver(case, seed)
    st["S"] = S
    if op == "apply":
        dt = torch.float32 if case["prec"] == 32 else torch.float64
        st.update(U=U.to(dt), x=x.to(dt), y=torch.empty(x.numel(), dtype=dt, device=DEV),
                  prec=stmg.STMG_FP32 if case["prec"] == 32 else stmg.STMG_FP64)
    elif op == "residual":
        st.update(U=U, V=vprev, R=torch.empty_like(U))
    elif op == "sweep":
        S.smoother_build(U)
        st.update(rhs=x.to(S.pdtype), z=torch.empty(x.numel(), dtype=S.pdtype, device=DEV))
    else:
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 7)
        ls = S.levels[:-1]
        rhs = [x.to(S.pdtype)] + [torch.randn(L["Nst"], generator=gen, dtype=S.pdtype, device=DEV) for L in ls[1:]]
        st.update(U=U, rhs=rhs, z=[torch.empty(L["Nst"], dtype=S.pdtype, device=DEV) for L in ls])
    return st


def run(st):
    op, S = st["op"], st["S"]
    if op == "apply":
        S.apply(st["U"], st["x"], st["y"], 0, st["prec"])
        return st["y"]
    if op == "residual":
        S.residual(T0, st["U"], st["V"], st["R"])
        return st["R"]
    if op == "sweep":
        S.smoother_sweep(0, st["rhs"], st["z"], 2, zero_start=True)
        return st["z"]
    if op == "build":
        S.smoother_build(st["U"])
        for l, (b, z) in enumerate(zip(st["rhs"], st["z"])):
            S.smoother_sweep(l, b, z, 1, zero_start=True)
        return st["z"]
    with torch.cuda.stream(st["stream"]):
        S.initial_guess(st["V0"], st["U"])
        S.slab_solve(0.0, st["V0"], st["U"])
    return st["U"]


# ------------------------------------------------------------------------------------ least work
def _apply_work(d, n, r, k, es, residual=False):
    N = r + 2
    n1 = (r + 1) * n + 1
    nv, npr = d * n1 ** d, n ** d * math.comb(r + d, d)
    byts = es * (k + 1) * (3 * nv + 2 * npr) + 8 * d * (n + 1) ** d
    # per Gauss point and time node, multiply-adds: sum-factorised values of the increment and the
    # state (2 d^2 N), collocation gradient and its transpose (2 d^2 N), integration (d^2 N), time
    # mixing and the pointwise flux (about 3 d^3 + 4 d^2), pressure values and tests (2 d N)
    per = 5 * d * d * N + d * (k + 1) + 3 * d ** 3 + 4 * d * d + 2 * d * N
    if residual:
        byts = es * ((k + 1) * (2 * nv + 2 * npr) + nv) + 8 * d * (n + 1) ** d
        per -= d * d * N
    return byts, 2.0 * per * n ** d * N ** d * (k + 1)


def _levels(case):
    n, r, k = case["n"], case["r"], case["k"]
    h = lambda x: int(math.log2(x)) if x > 0 else 0  # noqa: E731
    out = [(n, r, k)]
    while h(r) > 0 or h(k) > 0:
        a, b = h(r), h(k)
        r, k = (r // 2 if a >= b else r), (k // 2 if b >= a else k)
        out.append((n, r, k))
    while n % 2 == 0 and n // 2 >= 2:
        n //= 2
        out.append((n, r, k))
    return out


def _sweep_work(d, n, r, k, es, store):
    ms = d * (r + 2) ** d + math.comb(r + d, d)
    byts = n ** d * ((k + 1) * ms * ms * store + 3 * (k + 1) * ms * es)
    fma = {0: 1, 1: 4, 2: 5}[k] * ms * ms
    return byts, 2.0 * fma * n ** d


def work(case):
    d, n, r, k, op = case["d"], case["n"], case["r"], case["k"], case["op"]
    es = 4 if case["prec"] == 32 else 8
    if op in ("apply", "residual"):
        b, f = _apply_work(d, n, r, k, es, op == "residual")
        return {"bytes": b, "flops": f}
    store = 2 if case.get("fp16") else es
    if op == "sweep":
        b, f = _sweep_work(d, n, r, k, es, store)
        ab, af = _apply_work(d, n, r, k, es)
        return {"bytes": 2 * b + ab, "flops": 2 * f + af}
    lev = _levels(case)[:-1]
    if op == "build":
        # patch inverses written and read once (the sweeps); per patch and eigenvalue an inversion
        # (2 m^3 real, 8 m^3 complex operations)
        b = f = 0.0
        for (ln, lr, lk) in lev:
            ms = d * (lr + 2) ** d + math.comb(lr + d, d)
            sb, sf = _sweep_work(d, ln, lr, lk, es, store)
            b += sb + ln ** d * (lk + 1) * ms * ms * store
            f += sf + {0: 2, 1: 8, 2: 10}[lk] * float(ms) ** 3 * ln ** d
        return {"bytes": b, "flops": f}
    # a slab solve: five Newton steps of five Krylov iterations, each one FP64 apply, one V-cycle
    # (sweeps, level residuals) and its share of the orthogonalisation
    b = f = 0.0
    for i, (ln, lr, lk) in enumerate(lev):
        tc = case["sweeps_tc"] > 0 and i == 0 and lk == 2
        m = 2 * (case["sweeps_tc"] if tc else case["sweeps"])
        sb, sf = _sweep_work(d, ln, lr, lk, es, store)
        ab, af = _apply_work(d, ln, lr, lk, es)
        b += m * (sb + ab)
        f += m * (sf + af)
    ab, af = _apply_work(d, n, r, k, 8)
    nst = _sizes(case)[4]
    its = 25
    return {"bytes": its * (b + ab + 4 * 3 * 8 * nst), "flops": its * (f + af)}


# ------------------------------------------------------------------------------------ 64-bit values
def _lobatto(n):
    c = np.zeros(n)
    c[n - 1] = 1.0
    inner = np.sort(np.real(npleg.legroots(npleg.legder(c)))) if n > 2 else np.zeros(0)
    return 0.5 * (np.concatenate([[-1.0], inner, [1.0]]) + 1.0)


def _radau(k):
    if k == 0:
        return np.array([1.0]), np.array([2.0])
    c = np.zeros(k + 2)
    c[k], c[k + 1] = 1.0, -1.0
    t = np.sort(np.real(npleg.legroots(c)))
    t[-1] = 1.0
    A = np.array([t ** p for p in range(k + 1)])
    return t, np.linalg.solve(A, np.array([(1.0 - (-1.0) ** (p + 1)) / (p + 1) for p in range(k + 1)]))


def _lagrange(nodes, x):
    """Values and derivatives [points, nodes] of the Lagrange polynomials on `nodes`."""
    n = len(nodes)
    V, D = np.ones((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        others = [j for j in range(n) if j != i]
        for j in others:
            V[:, i] *= (x - nodes[j]) / (nodes[i] - nodes[j])
        for m in others:
            t = np.full(len(x), 1.0 / (nodes[i] - nodes[m]))
            for j in others:
                if j != m:
                    t = t * (x - nodes[j]) / (nodes[i] - nodes[j])
            D[:, i] += t
    return V, D


class _Time:
    def __init__(self, k, tau):
        self.t, om = _radau(k)
        self.w = 0.5 * tau * om
        xg, wg = npleg.leggauss(k + 3)
        phi, dphi = _lagrange(self.t, xg)
        self.C = _lagrange(self.t, np.array([-1.0]))[0][0]
        self.K = np.einsum("q,qa,qb->ab", wg, phi, dphi) + np.outer(self.C, self.C)
        self.mid = _lagrange(self.t, np.array([0.0]))[0][0]
        self.tau = tau


class _Forms:
    """Dense element-wise evaluation of the discrete forms on the whole mesh, in chunks of cells."""

    def __init__(self, case, seed):
        self.d, self.n, self.r, self.k = d, n, r, k = case["d"], case["n"], case["r"], case["k"]
        self.nu, tau = _physics(case)
        self.time = _Time(k, tau)
        self.n1, self.nv, self.npr, self.npc, self.nst = _sizes(case)
        self.nn = self.n1 ** d
        self.N = N = r + 2
        gl = _lobatto(N)
        qx, qw = npleg.leggauss(N)
        qx, qw = 0.5 * (qx + 1.0), 0.5 * qw
        T = lambda a: torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
        idx = [t[::-1] for t in itertools.product(range(N), repeat=d)]            # x fastest
        self.modes = [m for s in range(r + 1) for m in
                      ([(s - j, j) for j in range(s + 1)] if d == 2 else
                       [(s - j - l, j, l) for l in range(s + 1) for j in range(s - l + 1)])]
        assert len(self.modes) == self.npc

        def tables(pts):
            L = [_lagrange(gl, pts[:, l]) for l in range(d)]
            phi = np.stack([np.prod([L[l][0][:, m[l]] for l in range(d)], axis=0) for m in idx], 1)
            dphi = np.stack([np.stack([np.prod([L[l][1 if g == l else 0][:, m[l]] for l in range(d)], axis=0)
                                       for g in range(d)], 1) for m in idx], 1)
            P = [np.stack([npleg.legval(2 * pts[:, l] - 1, np.eye(r + 1)[i]) for i in range(r + 1)], 1) for l in range(d)]
            psi = np.stack([np.prod([P[l][:, m[l]] for l in range(d)], axis=0) for m in self.modes], 1)
            dn = np.zeros((len(pts), 2 ** d, d))
            nn = np.zeros((len(pts), 2 ** d))
            for c in range(2 ** d):
                v = [pts[:, l] if (c >> l) & 1 else 1 - pts[:, l] for l in range(d)]
                s = [1.0 if (c >> l) & 1 else -1.0 for l in range(d)]
                nn[:, c] = np.prod(v, axis=0)
                for g in range(d):
                    dn[:, c, g] = np.prod([np.full(len(pts), s[l]) if l == g else v[l] for l in range(d)], axis=0)
            return dict(phi=T(phi), dphi=T(dphi), psi=T(psi), dn=T(dn), nn=T(nn))

        pts = np.array([[qx[i] for i in m] for m in idx])
        self.vol = tables(pts)
        self.qw = T(np.array([np.prod([qw[i] for i in m]) for m in idx]))
        self.face = {}
        for axis in range(d):
            for side in (0, 1):
                fp, fw = [], []
                for m in itertools.product(range(N), repeat=d - 1):
                    p, w, it = [0.0] * d, 1.0, iter(m)
                    for l in range(d):
                        if l == axis:
                            p[l] = float(side)
                        else:
                            i = next(it)
                            p[l], w = qx[i], w * qw[i]
                    fp.append(p)
                    fw.append(w)
                self.face[axis, side] = (tables(np.array(fp)), T(np.array(fw)))
        cm = torch.stack([torch.arange(n ** d, device=DEV) // n ** l % n for l in range(d)], 1)
        self.cm = cm
        verts = T(_vertices(case, seed).reshape(-1, d))
        bits = torch.tensor([[(c >> l) & 1 for l in range(d)] for c in range(2 ** d)], device=DEV)
        st = torch.tensor([(n + 1) ** l for l in range(d)], device=DEV)
        self.corner = verts[((cm[:, None, :] + bits) * st).sum(-1)]               # [cells, 2^d, d]
        st = torch.tensor([self.n1 ** l for l in range(d)], device=DEV)
        self.nodes = ((cm[:, None, :] * (r + 1) + torch.tensor(idx, device=DEV)) * st).sum(-1)
        self.h = 1.0 / ((r + 1) * (r + 2))
        self.idx = idx

    def chunks(self, size):
        nc = self.n ** self.d
        return [slice(o, min(nc, o + size)) for o in range(0, nc, size)]

    def geometry(self, cells, tab):
        J = torch.einsum("qcl,kci->kqil", tab["dn"], self.corner[cells])
        return torch.linalg.inv(J), torch.linalg.det(J)                           # G[m][i], det

    def on_face(self, cells, axis, side):
        tab, w = self.face[axis, side]
        G, det = self.geometry(cells, tab)
        cof = det[..., None] * G[:, :, axis, :] * (1.0 if side else -1.0)
        dS = cof.norm(dim=-1)
        _, dv = self.geometry(cells, self.vol)
        jw = dS * w
        return tab, G, cof / dS[..., None], jw, (dv * self.qw).sum(1) / jw.sum(1) * self.h

    def boundary(self, cells, axis, side):
        ids = torch.arange(self.n ** self.d, device=DEV)[cells] if isinstance(cells, slice) else cells
        return ids[self.cm[ids, axis] == (self.n - 1 if side else 0)]

    def local(self, v, cells):
        """[cells, d, nodes] of one component-major field."""
        return torch.stack([v[c * self.nn:(c + 1) * self.nn][self.nodes[cells]] for c in range(self.d)], 1)

    def modes_of(self, p, cells):
        return p.reshape(-1, self.npc)[cells]

    def slab(self, x, state, vprev=None, data=None):
        """J(state) x, or with vprev the residual at x (state unused)."""
        d, tm, nu = self.d, self.time, self.nu
        res = vprev is not None
        y = torch.zeros(self.nst, dtype=torch.float64, device=DEV)
        poff = (self.k + 1) * self.nv
        eye = torch.eye(d, dtype=torch.float64, device=DEV)

        def add(a, cells, rv, rp):
            for c in range(d):
                y[a * self.nv + c * self.nn:a * self.nv + (c + 1) * self.nn].index_add_(
                    0, self.nodes[cells].reshape(-1), rv[:, c].reshape(-1))
            y[poff + a * self.npr:poff + (a + 1) * self.npr].view(-1, self.npc)[cells] += rp

        for cells in self.chunks(1 << (15 if d == 2 else 13)):
            V, X = self.vol, [self.local(x[a * self.nv:(a + 1) * self.nv], cells) for a in range(self.k + 1)]
            G, det = self.geometry(cells, V)
            jw = det * self.qw
            xq = torch.einsum("qc,kci->kqi", V["nn"], self.corner[cells])
            val = [torch.einsum("qj,kcj->kqc", V["phi"], u) for u in X]
            vp = torch.einsum("qj,kcj->kqc", V["phi"], self.local(vprev, cells)) if res else None
            for a in range(self.k + 1):
                w, t = tm.w[a], T0 + 0.5 * tm.tau * (tm.t[a] + 1.0)
                u = val[a]
                gu = torch.einsum("kqcm,kqml->kqcl", torch.einsum("qjm,kcj->kqcm", V["dphi"], X[a]), G)
                pm = self.modes_of(x[poff + a * self.npr:poff + (a + 1) * self.npr], cells)
                p = pm @ V["psi"].T
                if res:
                    conv = u[..., :, None] * u[..., None, :]
                else:
                    s = torch.einsum("qj,kcj->kqc", V["phi"], self.local(state[a * self.nv:(a + 1) * self.nv], cells))
                    conv = u[..., :, None] * s[..., None, :] + s[..., :, None] * u[..., None, :]
                F = w * jw[..., None, None] * (nu * gu - conv - p[..., None, None] * eye)
                m = sum(tm.K[a][b] * val[b] for b in range(self.k + 1))
                if res:
                    m = m - tm.C[a] * vp - w * data.f(xq, t, nu)
                rv = torch.einsum("kqcm,qjm->kcj", torch.einsum("kqcl,kqml->kqcm", F, G), V["dphi"])
                rv += torch.einsum("kqc,qj->kcj", jw[..., None] * m, V["phi"])
                rp = -w * (jw * gu.diagonal(dim1=2, dim2=3).sum(-1)) @ V["psi"]
                add(a, cells, rv, rp)
        for axis in range(d):
            for side in (0, 1):
                cells = self.boundary(slice(None), axis, side)
                tab, G, nrm, jw, h = self.on_face(cells, axis, side)
                xf = torch.einsum("qc,kci->kqi", tab["nn"], self.corner[cells])
                dnphi = torch.einsum("pjm,kpml,kpl->kpj", tab["dphi"], G, nrm)
                for a in range(self.k + 1):
                    w, t = tm.w[a], T0 + 0.5 * tm.tau * (tm.t[a] + 1.0)
                    X = self.local(x[a * self.nv:(a + 1) * self.nv], cells)
                    u = torch.einsum("pj,kcj->kpc", tab["phi"], X)
                    dnu = torch.einsum("kpj,kcj->kpc", dnphi, X)
                    p = self.modes_of(x[poff + a * self.npr:poff + (a + 1) * self.npr], cells) @ tab["psi"].T
                    s = u if res else torch.einsum("pj,kcj->kpc", tab["phi"],
                                                   self.local(state[a * self.nv:(a + 1) * self.nv], cells))
                    g = data.g(xf, t, nu) if res else torch.zeros_like(u)
                    e = u - g
                    en, yn = (e * nrm).sum(-1), (s * nrm).sum(-1)
                    inflow = 0.5 * (yn.abs() + yn) - (yn.abs() - yn)
                    v = -nu * dnu + (nu * 10.0 / h)[:, None, None] * e + (10.0 / h)[:, None, None] * en[..., None] * nrm
                    v = v + p[..., None] * nrm + inflow[..., None] * u
                    if res:
                        gn = (g * nrm).sum(-1)
                        v = v + (0.5 * (gn.abs() - gn))[..., None] * g
                    else:
                        v = v + (0.5 * (3.0 - torch.sign(yn)) * en)[..., None] * s
                    rv = torch.einsum("kpc,pj->kcj", jw[..., None] * v, tab["phi"])
                    rv -= nu * torch.einsum("kpc,kpj->kcj", jw[..., None] * e, dnphi)
                    add(a, cells, w * rv, w * (jw * en) @ tab["psi"])
        return y

    def element_matrices(self, v):
        """A (velocity block at the velocity v), B (pressure rows) and the scalar mass of every cell."""
        d, nl, nu, nc = self.d, len(self.idx), self.nu, self.n ** self.d
        A = torch.zeros(nc, d, nl, d, nl, dtype=torch.float64, device=DEV)
        B = torch.zeros(nc, self.npc, d, nl, dtype=torch.float64, device=DEV)
        M = torch.zeros(nc, nl, nl, dtype=torch.float64, device=DEV)
        for cells in self.chunks(2048 if d == 2 else 512):
            tab = self.vol
            G, det = self.geometry(cells, tab)
            jw = det * self.qw
            gphi = torch.einsum("qjm,kqml->kqjl", tab["dphi"], G)
            s = torch.einsum("qj,kcj->kqc", tab["phi"], self.local(v, cells))
            wphi = jw[..., None] * tab["phi"]
            adv = torch.einsum("kqil,kql->kqi", gphi, s)
            same = nu * torch.einsum("kqil,kqjl->kij", gphi * jw[..., None, None], gphi) - torch.einsum("kqj,kqi->kij", wphi, adv)
            for c in range(d):
                for e in range(d):
                    A[cells, c, :, e, :] = -torch.einsum("kqj,kqi->kij", wphi, s[:, :, c, None] * gphi[..., e])
                A[cells, c, :, c, :] += same
            B[cells] = -torch.einsum("kqm,kqje->kmej", jw[..., None] * tab["psi"], gphi)
            M[cells] = torch.einsum("kqi,qj->kij", wphi, tab["phi"])
        for axis in range(d):
            for side in (0, 1):
                cells = self.boundary(slice(None), axis, side)
                tab, G, nrm, jw, h = self.on_face(cells, axis, side)
                dn = torch.einsum("pjm,kpml,kpl->kpj", tab["dphi"], G, nrm)
                s = torch.einsum("pj,kcj->kpc", tab["phi"], self.local(v, cells))
                yn = (s * nrm).sum(-1)
                wphi = jw[..., None] * tab["phi"]
                diag = -nu * torch.einsum("kpi,kpj->kij", wphi, dn)
                diag = diag + diag.transpose(1, 2)
                inflow = 0.5 * (yn.abs() + yn) - (yn.abs() - yn)
                diag = diag + torch.einsum("kpi,pj->kij", ((nu * 10.0 / h)[:, None] + inflow)[..., None] * wphi, tab["phi"])
                up = 0.5 * (3.0 - torch.sign(yn))
                for c in range(d):
                    for e in range(d):
                        f = (10.0 / h)[:, None] * nrm[..., c] * nrm[..., e] + up * nrm[..., e] * s[..., c]
                        blk = torch.einsum("kpi,pj->kij", f[..., None] * wphi, tab["phi"])
                        A[cells, c, :, e, :] += blk + (diag if c == e else 0)
                B[cells] += torch.einsum("kpm,kpej->kmej", jw[..., None] * tab["psi"],
                                         nrm[..., None] * tab["phi"][None, :, None, :])
        return A, B, M

    def shared(self, M, cells, comps):
        """Sum over the neighbour cells that share both nodes of an entry: M [cells, c, i, e, j] (or
        [cells, i, j] without components)."""
        d, N, n = self.d, self.N, self.n
        out = torch.zeros_like(M[cells])
        mi = torch.tensor(self.idx, device=DEV)
        stn = torch.tensor([N ** l for l in range(d)], device=DEV)
        stc = torch.tensor([n ** l for l in range(d)], device=DEV)
        ids = torch.arange(n ** d, device=DEV)[cells]
        for o in itertools.product((-1, 0, 1), repeat=d):
            ot = torch.tensor(o, device=DEV)
            other = mi - ot * (N - 1)
            ok = ((other >= 0) & (other < N)).all(1)
            here, there = ok.nonzero()[:, 0], (other[ok] * stn).sum(1)
            cn = self.cm[ids] + ot
            has = ((cn >= 0) & (cn < n)).all(1).nonzero()[:, 0]
            src = M[(cn[has] * stc).sum(1)]
            if comps:
                blk = src[:, :, there][:, :, :, :, there]
                out[has[:, None, None, None, None], torch.arange(d, device=DEV)[None, :, None, None, None],
                    here[None, None, :, None, None], torch.arange(d, device=DEV)[None, None, None, :, None],
                    here[None, None, None, None, :]] += blk
            else:
                out[has[:, None, None], here[None, :, None], here[None, None, :]] += src[:, there][:, :, there]
        return out

    def sweeps(self, U, rhs, count):
        """`count` damped additive sweeps from zero: velocity damping 1.2 / 2^d, pressure 1."""
        d, nl, k, tm = self.d, len(self.idx), self.k, self.time
        v = sum(tm.mid[a] * U[a * self.nv:(a + 1) * self.nv] for a in range(k + 1))
        A, B, M = self.element_matrices(v)
        mv = d * nl
        ms = mv + self.npc
        lam, Q = np.linalg.eig(tm.K / tm.w[:, None])
        Qi = np.linalg.inv(Q)
        C = lambda a: torch.tensor(a, dtype=torch.complex128, device=DEV)  # noqa: E731
        parts = self.chunks({2: 8192, 3: 1024 if ms < 100 else 256}[d])
        z = torch.zeros_like(rhs)
        for s in range(count):
            r = rhs if s == 0 else rhs - self.slab(z, U)
            up = torch.zeros_like(z)
            for ic, cells in enumerate(parts):
                loc = [torch.cat([self.local(r[a * self.nv:(a + 1) * self.nv], cells).reshape(-1, mv),
                                  self.modes_of(r[(k + 1) * self.nv + a * self.npr:(k + 1) * self.nv + (a + 1) * self.npr], cells)], 1)
                       for a in range(k + 1)]
                b = torch.stack(loc, 1) / torch.tensor(tm.w, device=DEV)[None, :, None]
                bh = torch.einsum("ea,kam->kem", C(Qi), b.to(torch.complex128))
                Ap = self.shared(A, cells, True).reshape(-1, mv, mv)
                Mp = self.shared(M, cells, False)
                yh = torch.empty_like(bh)
                for e in range(k + 1):
                    T = torch.zeros(Ap.shape[0], ms, ms, dtype=torch.complex128, device=DEV)
                    T[:, :mv, :mv] = Ap
                    for c in range(d):
                        T[:, c * nl:(c + 1) * nl, c * nl:(c + 1) * nl] += complex(lam[e]) * Mp
                    Bp = B[cells].reshape(-1, self.npc, mv)
                    T[:, mv:, :mv] = Bp
                    T[:, :mv, mv:] = Bp.transpose(1, 2)
                    yh[:, e] = torch.linalg.solve(T, bh[:, e, :, None])[..., 0]
                y = torch.einsum("ae,kem->kam", C(Q), yh).real
                for a in range(k + 1):
                    for c in range(d):
                        up[a * self.nv + c * self.nn:a * self.nv + (c + 1) * self.nn].index_add_(
                            0, self.nodes[cells].reshape(-1), y[:, a, c * nl:(c + 1) * nl].reshape(-1))
                    o = (k + 1) * self.nv + a * self.npr
                    up[o:o + self.npr].view(-1, self.npc)[cells] += y[:, a, mv:]
            pv = (k + 1) * self.nv
            z[:pv] += 1.2 / 2 ** d * up[:pv]
            z[pv:] += up[pv:]
        return z


class _Data:
    """f and g of the bundled problems at points x [.., d] (the library's analytic data)."""

    def __init__(self, problem):
        self.problem = problem

    def g(self, x, t, nu):
        pi, out = math.pi, torch.zeros_like(x)
        if self.problem == "TG2D":
            F = math.exp(-2 * pi * pi * nu * t)
            out[..., 0] = F * torch.sin(pi * x[..., 0]) * torch.cos(pi * x[..., 1])
            out[..., 1] = -F * torch.cos(pi * x[..., 0]) * torch.sin(pi * x[..., 1])
        elif self.problem == "TG3D":
            out[..., 0] = torch.sin(pi * x[..., 0]) * torch.cos(pi * x[..., 1]) * torch.cos(pi * x[..., 2])
            out[..., 1] = -torch.cos(pi * x[..., 0]) * torch.sin(pi * x[..., 1]) * torch.cos(pi * x[..., 2])
        elif self.problem == "CAV3D":
            out[..., 0] = (x[..., 2] > 1.0 - 1e-9).double() * math.sin(0.25 * pi * t)
        return out

    def f(self, x, t, nu):
        pi, out = math.pi, torch.zeros_like(x)
        if self.problem not in ("MMS2D", "MMS3D"):
            return out
        # f = v_t + (v . grad) v - nu lap v + grad p for v = sin t w(x), p = sin t q(x), by nested
        # forward-mode derivatives of w and q
        if self.problem == "MMS2D":
            w = lambda z: torch.stack([torch.sin(pi * z[0]) ** 2 * torch.sin(pi * z[1]) * torch.cos(pi * z[1]),  # noqa: E731
                                       -torch.sin(pi * z[0]) * torch.cos(pi * z[0]) * torch.sin(pi * z[1]) ** 2])
            q = lambda z: torch.sin(pi * z[0]) * torch.cos(pi * z[0]) * torch.sin(pi * z[1]) * torch.cos(pi * z[1])  # noqa: E731
        else:
            w = lambda z: torch.sin(pi * z[2]) * torch.stack([  # noqa: E731
                pi * torch.sin(pi * z[0]) ** 2 * torch.sin(2 * pi * z[1]),
                -pi * torch.sin(2 * pi * z[0]) * torch.sin(pi * z[1]) ** 2, 0 * z[2]])
            q = lambda z: (torch.sin(pi * z[0]) * torch.cos(pi * z[0]) * torch.sin(pi * z[1]) * torch.cos(pi * z[1])  # noqa: E731
                           * torch.sin(pi * z[2]) * torch.cos(pi * z[2]))
        jac, hes = torch.func.jacfwd(w), torch.func.jacfwd(torch.func.jacfwd(w))
        pts = x.reshape(-1, x.shape[-1])
        W, J = torch.vmap(w)(pts), torch.vmap(jac)(pts)
        L = torch.vmap(hes)(pts).diagonal(dim1=2, dim2=3).sum(-1)
        gq = torch.vmap(torch.func.jacfwd(q))(pts)
        st, ct = math.sin(t), math.cos(t)
        return (ct * W + st * st * torch.einsum("pcl,pl->pc", J, W) - nu * st * L + st * gq).reshape(x.shape)


def exact(case, seed):
    op = case["op"]
    if op == "solve":
        return None
    U, x, vprev = _vectors(case, seed)
    if case["prec"] == 32:
        x = x.float().double()
        if op == "apply":
            U = U.float().double()
    F = _Forms(case, seed)
    if op == "apply":
        return F.slab(x, U)
    if op == "residual":
        return F.slab(U, None, vprev, _Data(case["problem"]))
    if op == "sweep":
        return F.sweeps(U, x, 2)
    # the finest level alone: a coarse level's state is the library's own interpolation
    return [F.sweeps(U, x, 1)] + [None] * (len(_levels(case)) - 2)
