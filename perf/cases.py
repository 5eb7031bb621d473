"""Performance cases of the ESDG shallow-water library: the calls its users
make (whole solves, single right-hand sides, batched ensembles, diagnostics)
over the range of degrees, meshes, precisions, rules, inverse masses and
methods the library takes.

A case is a dict of plain values.  `prepare` builds the problem on the library
(operators, mesh, bathymetry, initial state) as a user's program does before
it calls it, `run` makes one pass through the public entry points, `work`
counts what the pass cannot do without, and `exact` computes the same outputs
in FP64 from the paper's formulas (arXiv 2005.02516), in plain torch.

Calls:
  step      set the state, advance `steps` LSRK45 steps at the CFL step, read the state
  rhs       du/dt of a caller's state (a caller with its own time integrator)
  ensemble  set the members' states, advance them together, read the states
  monitor   entropy, mass and entropy rate, and the L2 error against given values
"""

import math

import numpy as np
import torch

from paper_2005_02516_gb300 import esdg

SYMMETRIC_POINTS = {1: 3, 2: 6, 3: 12, 4: 16, 5: 25}
SBP_POINTS = {1: 6, 2: 10, 3: 18, 4: 22, 5: 34}


def _case(name=None, call="step", N=4, nx=16, ny=16, precision="fp32", rule="symmetric", mass="exact",
          method="modal", walls=False, problem="bump", warp=0.05, steps=1, members=0, pick=0):
    c = dict(call=call, N=N, nx=nx, ny=ny, precision=precision, rule=rule, mass=mass, method=method, walls=walls,
             problem=problem, warp=warp, steps=steps, members=members, pick=pick)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the plain FP64 solve of a small lake: a few launches a step, all latency
        _case("lake_fp64_k128_n2", N=2, nx=8, ny=8, precision="fp64", rule="collapsed", warp=0.0, steps=10),
        # the smallest served request (K = 512), solved alone in FP32
        _case("bump_fp32_k512_n4", N=4, nx=16, ny=16, steps=20),
        # the accuracy study: manufactured solution with forcing, N = 3, K = 8192, in both precisions
        _case("mms_fp32_k8192_n3", N=3, nx=64, ny=64, rule="collapsed", problem="mms", steps=10),
        _case("mms_fp64_k8192_n3", N=3, nx=64, ny=64, precision="fp64", rule="collapsed", problem="mms", steps=4),
        # the large dam break of the roofline study, FP32 right-hand side
        _case("dam_fp32_k131072_n4", N=4, nx=256, ny=256, problem="dam", steps=4),
        # the same flow on a quarter of the mesh in FP64, for an accurate reference run
        _case("dam_fp64_k32768_n4", N=4, nx=128, ny=128, precision="fp64", problem="dam", steps=2),
        # a closed basin without stored inverses, on a ragged mesh
        _case("basin_fp32_wadg_k31714_n3", N=3, nx=157, ny=101, mass="weight_adjusted", walls=True, steps=6),
        # the DG-SBP method on a ragged mesh
        _case("dam_fp32_sbp_k53938_n4", N=4, nx=181, ny=149, method="sbp", problem="dam", steps=4),
        # the highest degree in FP64 on an affine mesh (the degree study N = 1..5)
        _case("bump_fp64_k8192_n5", N=5, nx=64, ny=64, precision="fp64", warp=0.0, steps=2),
        # a parameter study: independent solves of mixed degree and mesh in one launch
        _case("ensemble_fp32_m24", call="ensemble", N=4, members=24, pick=1, steps=10),
        # one right-hand side for a caller's own integrator, odd mesh, highest degree
        _case("rhs_fp32_k3034_n5", call="rhs", N=5, nx=37, ny=41, problem="rough"),
        # monitoring a run: entropy, mass, entropy rate and L2 error
        _case("monitor_fp64_k32768_n2", call="monitor", N=2, nx=128, ny=128, precision="fp64", problem="rough"),
    ]


def draw(rng):
    """A case of the same ranges: K from 128 to 131072 triangles (to 32768 in
    FP64), every degree, rule, inverse mass, method, boundary and call."""
    call = rng.choice(["step"] * 6 + ["rhs", "rhs", "ensemble", "monitor"])
    if call == "ensemble":
        return _case(call=call, N=rng.choice([4, 4, 5]), rule=rng.choice(["symmetric", "symmetric", "collapsed"]),
                     members=rng.randint(3, 24), pick=rng.randint(2, 10**6), steps=rng.randint(3, 10))
    precision = rng.choice(["fp32", "fp32", "fp64"])
    N = rng.randint(1, 5)
    K = math.exp(rng.uniform(math.log(128), math.log(131072 if precision == "fp32" else 32768)))
    aspect = math.exp(rng.uniform(-0.4, 0.4))
    nx = max(8, round(math.sqrt(K / 2) * aspect))
    ny = max(8, round(K / 2 / nx))
    method = rng.choice(["modal", "modal", "modal", "sbp"])
    modal = method == "modal"
    problem = "rough" if call != "step" else rng.choice(["dam", "bump", "mms"])
    mass = "weight_adjusted" if modal and rng.random() < 0.2 else "exact"
    walls = modal and problem != "mms" and rng.random() < 0.25
    # at most the work of the largest listed case of this precision
    most = (131072 * 4 if precision == "fp32" else 32768) * 15 / (2 * nx * ny * (N + 1) * (N + 2) / 2)
    steps = max(1, min(rng.randint(2, 20), int(most))) if call == "step" else 1
    return _case(call=call, N=N, nx=nx, ny=ny, precision=precision, rule=rng.choice(["symmetric", "collapsed"]),
                 mass=mass, method=method, walls=walls, problem=problem, warp=rng.choice([0.05, 0.05, 0.0]),
                 steps=steps)


# ---- problems ---------------------------------------------------------------------

class _Problem:
    """Bathymetry and initial data of a case, drawn from the seed: functions of
    (x, y) numpy arrays, and (rough) a random part of the state itself."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([20050251, seed])
        self.kind, self.seed = case["problem"], seed
        self.surface = self.kind in ("bump", "rough")
        self.t0 = float(rng.uniform(0.0, 2.0)) if self.kind == "mms" else 0.0
        self.amp = float(rng.uniform(0.02, 0.2))
        self.cx, self.cy = (float(v) for v in rng.uniform(-0.3, 0.3, 2))
        self.radius = float(rng.uniform(0.25, 0.35))

    def bathymetry(self, x, y):
        if self.kind == "mms":
            return 0.1 * np.cos(np.pi * x) * np.cos(np.pi * y)
        if self.kind == "dam":
            return 0.05 * np.exp(-10.0 * ((x - 0.4) ** 2 + y * y))
        return self.amp * np.sin(np.pi * x) * np.sin(np.pi * y)

    def initial(self, x, y):
        r2 = (x - self.cx) ** 2 + (y - self.cy) ** 2
        if self.kind == "mms":
            h = 2.0 + 0.1 * np.sin(np.pi * (x + y - self.t0))
            return np.stack([h, 0.5 * h, 0.5 * h])
        if self.kind == "dam":
            return np.stack([1.0 + 0.5 * np.tanh(40.0 * (self.radius - np.sqrt(r2))), 0 * x, 0 * x])
        return np.stack([2.0 + 0.01 * np.exp(-25.0 * r2), 0 * x, 0 * x])

    def roughness(self, K, ndof, modal):
        """Random part of the state (rough): modal amplitudes falling with the
        mode, or nodal noise."""
        g = torch.Generator().manual_seed(self.seed + 7)
        d = 0.03 * torch.randn(3, K, ndof, dtype=torch.float64, generator=g)
        return d / (1.0 + torch.arange(ndof, dtype=torch.float64)) if modal else d


def _members(case):
    """The ensemble's members as step cases: degrees 2..N, K from 512 to 32768,
    the mesh sizes of the batched workload and odd ones."""
    rng = np.random.default_rng([20050251, case["pick"]])
    out = []
    for _ in range(case["members"]):
        n = int(round(math.exp(rng.uniform(math.log(16), math.log(128)))))
        nx = int(rng.choice([16, 32, 64, 128])) if rng.random() < 0.5 else n
        out.append(_case(N=int(rng.integers(2, case["N"] + 1)), nx=nx, ny=nx, rule=case["rule"], steps=case["steps"]))
    return out


# ---- preparation and one pass ---------------------------------------------------------

def _solver(case, seed):
    p = _Problem(case, seed)
    s = esdg.Solver(case["N"], case["nx"], case["ny"], precision=case["precision"], warp=case["warp"],
                    rule=case["rule"], walls=case["walls"], mass=case["mass"], method=case["method"],
                    forcing="mms_sine" if p.kind == "mms" else "none")
    xb, yb = s.points(esdg.ESDG_POINTS_NODAL)
    xq, yq = s.points(esdg.ESDG_POINTS_VOLQ)
    s.init_state(p.bathymetry(xb, yb), p.initial(xq, yq), surface=p.surface)
    u0 = torch.empty((3, s.K, s.ndof), dtype=torch.float64, device="cuda")
    s.get_state(u0)
    if p.kind == "rough":
        u0 += p.roughness(s.K, s.ndof, case["method"] == "modal").to("cuda")
        s.set_state(u0)
    return s, u0, p


def prepare(case, seed):
    if case["call"] == "ensemble":
        built = [_solver(m, seed * 64 + i) for i, m in enumerate(_members(case))]
        return dict(call="ensemble", steps=case["steps"], solvers=[b[0] for b in built], u0=[b[1] for b in built],
                    out=[torch.empty_like(b[1]) for b in built], ensemble=esdg.Ensemble([b[0] for b in built]))
    s, u0, p = _solver(case, seed)
    state = dict(call=case["call"], steps=case["steps"], solver=s, u0=u0, t0=p.t0, out=torch.empty_like(u0))
    if case["call"] == "monitor":
        xq, yq = s.points(esdg.ESDG_POINTS_VOLQ)
        state["given"] = torch.from_numpy(p.initial(xq, yq)).to("cuda")
    return state


def run(state):
    if state["call"] == "ensemble":
        for s, u0 in zip(state["solvers"], state["u0"]):
            s.set_state(u0)
        state["ensemble"].step(state["steps"])
        return [s.get_state(out) for s, out in zip(state["solvers"], state["out"])]
    s = state["solver"]
    if state["call"] == "rhs":
        return s.rhs(state["t0"], u_in=state["u0"], out=state["out"])
    if state["call"] == "monitor":
        entropy, mass, rate = s.entropy(state["t0"])
        return dict(entropy=entropy, mass=mass, rate=rate, error=s.l2_error(state["given"]))
    s.set_state(state["u0"])
    s.step(state["steps"], t=state["t0"])
    return s.get_state(state["out"])


# ---- the work of a pass -----------------------------------------------------------------

def _sizes(case):
    N = case["N"]
    Np, Nfq = (N + 1) * (N + 2) // 2, 3 * (N + 1)
    sbp = case["method"] == "sbp"
    Nq = SBP_POINTS[N] if sbp else SYMMETRIC_POINTS[N] if case["rule"] == "symmetric" else (N + 1) ** 2
    return 2 * case["nx"] * case["ny"], Np, Nq, Nfq, Nq if sbp else Np


def _stage(case, rk):
    """Bytes and operations of one element's stage: the state (and RK residual)
    read and written in FP64, the element's metrics, mass data, normals and
    bathymetry read in the right-hand side's precision, its face traces written
    and its neighbours' read; the contractions, one flux a pair, the interface."""
    K, Np, Nq, Nfq, ndof = _sizes(case)
    r = 4 if case["precision"] == "fp32" else 8
    sbp, wadg = case["method"] == "sbp", case["mass"] == "weight_adjusted"
    nodes = Nq if sbp else Nq + Nfq
    nbytes = (4 if rk else 2) * 3 * ndof * 8 + r * (5 * nodes + Nq + 9 * Nfq) + 4 * Nfq
    nbytes += 0 if sbp or wadg else r * Np * (Np + 1) // 2
    pairs = Nq * (Nq - 1) // 2 if sbp else Nq * (Nq - 1) // 2 + Nq * Nfq
    flops = 35 * pairs + 40 * Nfq + (12 * ndof if rk else 0)
    if sbp:
        flops += 9 * Nq
    else:
        dense = 2 * Nq * Np + 2 * (Nq + Nfq) * Np + (2 * Nq * Np if wadg else Np * Np) * 2
        flops += 6 * dense + 13 * Nq + 6 * (Nq + Nfq)
    return K * nbytes, K * flops


def work(case):
    if case["call"] == "ensemble":
        parts = [work(m) for m in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    K, Np, Nq, Nfq, ndof = _sizes(case)
    rk = case["call"] == "step"
    nbytes, flops = _stage(case, rk)
    if rk:
        n = 5 * case["steps"]
        return {"bytes": n * nbytes + 4 * 3 * K * ndof * 8, "flops": n * flops}
    if case["call"] == "monitor":
        # the right-hand side, then each sum over the volume points once
        return {"bytes": nbytes + K * (3 * 3 * ndof * 8 + 6 * Nq * 8), "flops": flops + K * Nq * (18 * Np + 40)}
    return {"bytes": nbytes, "flops": flops}


# ---- the same outputs in FP64, from the formulas of the paper ----------------------------

def _jacobi(x, a, b, n):
    """Orthonormal Jacobi polynomials P_0..P_n^(a,b) at x, by the three-term recurrence."""
    lg = math.lgamma
    p = [np.full_like(x, math.exp(0.5 * (lg(a + b + 2) - (a + b + 1) * math.log(2) - lg(a + 1) - lg(b + 1))))]
    if n > 0:
        p.append(p[0] * 0.5 * ((a + b + 2) * x + a - b) * math.sqrt((a + b + 3) / ((a + 1) * (b + 1))))
    old = 2 / (2 + a + b) * math.sqrt((a + 1) * (b + 1) / (a + b + 3)) if n > 0 else 0.0
    for i in range(1, n):
        h = 2 * i + a + b
        new = 2 / (h + 2) * math.sqrt((i + 1) * (i + 1 + a + b) * (i + 1 + a) * (i + 1 + b) / ((h + 1) * (h + 3)))
        mid = -(a * a - b * b) / (h * (h + 2))
        p.append(((x - mid) * p[i] - old * p[i - 1]) / new)
        old = new
    return p


def _djacobi(x, a, b, n):
    return np.zeros_like(x) if n == 0 else math.sqrt(n * (n + a + b + 1)) * _jacobi(x, a + 1, b + 1, n - 1)[n - 1]


def _basis(N, r, s):
    """Orthonormal Dubiner basis (modes i = 0..N, j = 0..N-i) and its r and s derivatives."""
    top = np.abs(1 - s) < 1e-14
    a = np.where(top, -1.0, 2 * (1 + r) / np.where(top, 1.0, 1 - s) - 1)
    d = np.where(top, 1.0, 1 - s)  # no derivative is asked for at the top vertex
    V, Vr, Vs = [], [], []
    for i in range(N + 1):
        f, df = _jacobi(a, 0, 0, i)[i], _djacobi(a, 0, 0, i)
        for j in range(N + 1 - i):
            g, dg = _jacobi(s, 2 * i + 1, 0, j)[j], _djacobi(s, 2 * i + 1, 0, j)
            w = (1 - s) ** i
            w1 = i * (1 - s) ** (i - 1) if i else 0 * s
            V.append(math.sqrt(2) * f * g * w)
            pa = math.sqrt(2) * df * g * w
            Vr.append(2 * pa / d)
            Vs.append(pa * (1 + a) / d + math.sqrt(2) * f * (dg * w - g * w1))
    return np.stack(V, 1), np.stack(Vr, 1), np.stack(Vs, 1)


def _collapsed_rule(n):
    x, w = np.polynomial.legendre.leggauss(n)
    # Gauss-Jacobi (1, 0): Golub-Welsch, polished by Newton on the polynomial
    k = np.arange(1, n)
    diag = -1.0 / ((2 * np.arange(n) + 1.0) * (2 * np.arange(n) + 3.0))
    off = np.sqrt(k * k * (k + 1.0) ** 2 / ((2 * k + 1.0) ** 2 * k * (k + 1.0)))
    y = np.linalg.eigvalsh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    for _ in range(3):
        y = y - _jacobi(y, 1, 0, n)[n] / _djacobi(y, 1, 0, n)
    wy = 1.0 / sum(p * p for p in _jacobi(y, 1, 0, n - 1))
    A, B = np.meshgrid(x, y, indexing="ij")
    return (0.5 * (1 + A) * (1 - B) - 1).ravel(), B.ravel(), (0.5 * np.outer(w, wy)).ravel()


# Orbits (centroid, points (a, a, 1 - 2a), points (a, b, 1 - a - b)) of the fully
# symmetric rules exact to degree 2N, and of the SBP rules exact to 2N - 1 with
# the face Gauss points on the edges: parameters to four digits (weights last in
# each orbit), refined below to the moment equations' solution.
_SYM = {1: ((0, 1, 0), [.1667, .6667]),
        2: ((0, 2, 0), [.0916, .2199, .4459, .4468]),
        3: ((0, 2, 1), [.0631, .1017, .2493, .2336, .0531, .3104, .1657]),
        4: ((1, 3, 1), [.2886, .0505, .0649, .1706, .2064, .4593, .1902, .0084, .2631, .0545]),
        5: ((1, 2, 3), [.1635, .0321, .0267, .1422, .0919, .0284, .1637, .0506, .0296, .3691, .0684, .1481, .3218,
                        .1278])}
_SBP = {1: ((0, 0, 0), [.3333]),
        2: ((1, 0, 0), [.2, .0833, .9]),
        3: ((0, 0, 1), [.0809, .0302, .1871, .2288, .2222]),
        4: ((1, 2, 0), [.0371, .0411, .0132, .1822, .1394, .2109, .4384, .2495]),
        5: ((1, 1, 2), [.0252, .0163, .0067, .2091, .2245, .0952, .0668, .1276, .0604, .0934, .3296, .1424])}


def _orbits(N, orbits, th, edges):
    """Points and weights of a symmetric rule with parameters th."""
    bary, w, th = [], [], list(th)
    if edges:
        t = np.polynomial.legendre.leggauss(N + 1)[0]
        for a in [0.5] * ((N + 1) % 2) + [0.5 * (1 - v) for v in sorted(t) if v > 1e-12]:
            wt = th.pop(0)
            pts = [(a, 1 - a, 0), (1 - a, a, 0), (0, a, 1 - a), (0, 1 - a, a), (a, 0, 1 - a), (1 - a, 0, a)]
            pts = pts[::2] if a == 0.5 else pts
            bary += pts
            w += [wt] * len(pts)
    n3, n21, n111 = orbits
    for _ in range(n3):
        bary.append((1 / 3, 1 / 3, 1 / 3))
        w.append(th.pop(0))
    for _ in range(n21):
        a, wt = th.pop(0), th.pop(0)
        bary += [(a, a, 1 - 2 * a), (a, 1 - 2 * a, a), (1 - 2 * a, a, a)]
        w += [wt] * 3
    for _ in range(n111):
        v = (th.pop(0), th.pop(0))
        v += (1 - v[0] - v[1],)
        bary += [tuple(v[i] for i in p) for p in
                 [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]]
        w += [th.pop(0)] * 6
    b = np.array(bary)
    return b[:, 1] - b[:, 0] - b[:, 2], b[:, 2] - b[:, 0] - b[:, 1], np.array(w)


def _symmetric_rule(N, sbp):
    orbits, th = (_SBP if sbp else _SYM)[N]
    th, deg = np.array(th, dtype=np.float64), 2 * N - 1 if sbp else 2 * N

    def off(p):
        r, s, w = _orbits(N, orbits, p, sbp)
        m = _basis(deg, r, s)[0].T @ w
        m[0] -= math.sqrt(2)
        return m
    for _ in range(40):  # Gauss-Newton with central differences
        J = np.stack([(off(th + e) - off(th - e)) / 2e-5 for e in 1e-5 * np.eye(th.size)], 1)
        d = np.linalg.lstsq(J, -off(th), rcond=None)[0]
        th = th + d
        if np.abs(d).max() < 1e-16:
            break
    return _orbits(N, orbits, th, sbp)


_RK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
         -1275806237668 / 842570457699)
_RK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
         3134564353537 / 4481467310338, 2277821191437 / 14882151754819)
_RK_C = (0.0, 1432997174477 / 9575080441755, 2526269341429 / 6820363962896, 2006345519317 / 3224310063776,
         2802321613138 / 2924317926251)


class _Exact:
    """The scheme of Secs. 2 and 3 in FP64 (g = 1, Lax-Friedrichs on, CFL 0.25)."""

    def __init__(self, case):
        N, nx, ny = case["N"], case["nx"], case["ny"]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.sbp, self.walls = case["method"] == "sbp", case["walls"]
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)  # noqa: E731
        # reference element
        if self.sbp or case["rule"] == "symmetric":
            r, s, w = _symmetric_rule(N, self.sbp)
        else:
            r, s, w = _collapsed_rule(N + 1)
        t, wt = np.polynomial.legendre.leggauss(N + 1)
        one = np.ones_like(t)
        rf, sf, wf = np.concatenate([t, -t, -one]), np.concatenate([-one, t, -t]), np.tile(wt, 3)
        nr, ns = np.concatenate([0 * t, one, -one]), np.concatenate([-one, one, 0 * t])
        Vq, Vqr, Vqs = _basis(N, r, s)
        Vf, Vfr, Vfs = _basis(N, rf, sf)
        M = Vq.T @ (w[:, None] * Vq)
        Pq = np.linalg.solve(M, Vq.T * w)
        self.Nq, self.Nf, self.Np = r.size, rf.size, Vq.shape[1]
        skew = []  # Q_h - Q_h^T of Sec. 2.3 in r and s
        for D, n in ((Vqr, nr), (Vqs, ns)):
            Q, EB = Pq.T @ M @ (Pq @ D) @ Pq, (Vf @ Pq).T * (wf * n)
            skew.append(T(np.block([[Q - Q.T, EB], [-EB.T, np.zeros((self.Nf, self.Nf))]])))
        self.skew, self.w, self.wf, self.Vq, self.Vh = skew, T(w), T(wf), T(Vq), T(np.vstack([Vq, Vf]))
        face = np.argmin(np.hypot(rf[:, None] - r, sf[:, None] - s), axis=1)
        self.node = torch.as_tensor(np.concatenate([np.arange(r.size), face]), device=self.dev)  # SBP: [I; I_f]
        # mesh: quads split along the diagonal, warped degree-N equispaced nodes
        jj, ii = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
        ij = [(0, 0), (1, 0), (1, 1)], [(0, 0), (1, 1), (0, 1)]
        vx = np.stack([np.stack([(ii + a).ravel() for a, _ in tri], 1) for tri in ij], 1).reshape(-1, 3)
        vy = np.stack([np.stack([(jj + b).ravel() for _, b in tri], 1) for tri in ij], 1).reshape(-1, 3)
        self.K = vx.shape[0]
        re = np.array([2 * i / N - 1 for j in range(N + 1) for i in range(N + 1 - j)])
        se = np.array([2 * j / N - 1 for j in range(N + 1) for i in range(N + 1 - j)])
        shape = np.stack([-(re + se) / 2, (1 + re) / 2, (1 + se) / 2])
        x, y = (2.0 * vx / nx - 1) @ shape, (2.0 * vy / ny - 1) @ shape
        a = case["warp"]
        self.xe = x + a * np.cos(0.5 * np.pi * x) * np.cos(1.5 * np.pi * y)
        self.ye = y + a * np.sin(2 * np.pi * x) * np.cos(0.5 * np.pi * y)
        self.Vei = np.linalg.inv(_basis(N, re, se)[0])
        X, Y = T(self.xe @ self.Vei.T), T(self.ye @ self.Vei.T)
        Dr, Ds = T(np.vstack([Vqr, Vfr])).T, T(np.vstack([Vqs, Vfs])).T
        xr, xs, yr, ys = X @ Dr, X @ Ds, Y @ Dr, Y @ Ds
        self.G = (ys, -yr), (-xs, xr)  # (rxJ, sxJ), (ryJ, syJ)
        self.J = (xr * ys - xs * yr)[:, :self.Nq].contiguous()
        n = [T(v) for v in (nr, ns)]
        self.nx, self.ny = (g[0][:, self.Nq:] * n[0] + g[1][:, self.Nq:] * n[1] for g in self.G)
        self.xq, self.yq = X @ self.Vq.T, Y @ self.Vq.T
        if case["mass"] == "weight_adjusted":
            Mi = T(np.linalg.inv(M))
            self.Mi = Mi @ torch.einsum("qn,kq,qm->knm", self.w[:, None] * self.Vq, 1 / self.J, self.Vq) @ Mi
        elif not self.sbp:
            self.Mi = torch.linalg.inv(torch.einsum("qn,kq,qm->knm", self.w[:, None] * self.Vq, self.J, self.Vq))
            Mt = torch.einsum("qn,kq,qm->knm", self.w[:, None] * self.Vq, self.J, self.Vq)
            self.Mi = self.Mi @ (2 * torch.eye(self.Np, dtype=torch.float64, device=self.dev) - Mt @ self.Mi)
        self.Mx = None
        if case["mass"] == "weight_adjusted":  # initial data are projected with the exact inverse
            self.Mx = torch.linalg.inv(torch.einsum("qn,kq,qm->knm", self.w[:, None] * self.Vq, self.J, self.Vq))
        self._faces(vx, vy, nx, ny, N + 1)
        self.dt = 0.25 * (2.0 / nx) / self.Np

    def _faces(self, vx, vy, nx, ny, Nfp):
        """Exterior node of every face node: faces matched by their vertices, nodes reversed."""
        if self.walls:
            v = vy.astype(np.int64) * (nx + 1) + vx
        else:
            v = (vy % ny).astype(np.int64) * nx + vx % nx
        ends = np.stack([v[:, [0, 1, 2]], v[:, [1, 2, 0]]], -1).reshape(-1, 2)
        key = ends.min(1) * (v.max() + 1) + ends.max(1)
        order = np.argsort(key, kind="stable")
        same = key[order][1:] == key[order][:-1]
        partner = np.arange(key.size)
        first, second = order[:-1][same], order[1:][same]
        partner[first], partner[second] = second, first
        alone = partner == np.arange(key.size)
        ext = partner[:, None] * Nfp + np.arange(Nfp - 1, -1, -1)
        self.ext = torch.as_tensor(ext.ravel(), device=self.dev)
        self.wall = torch.as_tensor(np.repeat(alone.reshape(-1, 3), Nfp, axis=1), device=self.dev)

    def data(self, p):
        """Bathymetry and initial state of problem p."""
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)  # noqa: E731
        bm = T(p.bathymetry(self.xe, self.ye) @ self.Vei.T)
        self.b, self.mms = bm @ self.Vh.T, p.kind == "mms"
        q = T(p.initial(self.xq.cpu().numpy(), self.yq.cpu().numpy()))
        if self.sbp:
            u = q.clone()
            if p.surface:
                u[0] -= self.b[:, :self.Nq]
        else:
            u = self._project(q, self.Mi if self.Mx is None else self.Mx)
            if p.surface:
                u[0] -= bm
        if p.kind == "rough":
            u += p.roughness(self.K, u.shape[2], not self.sbp).to(self.dev)
        return u, q

    def _project(self, q, Mi):
        return torch.einsum("knm,ckm->ckn", Mi, ((self.w * self.J) * q) @ self.Vq)

    def rhs(self, u, t):
        if self.sbp:
            ut = u[:, :, self.node]
            h, uu, vv = ut[0], ut[1] / ut[0], ut[2] / ut[0]
        else:
            q = u @ self.Vq.T
            uq, vq = q[1] / q[0], q[2] / q[0]
            ent = torch.stack([q[0] + self.b[:, :self.Nq] - 0.5 * (uq * uq + vq * vq), uq, vq])
            v = self._project(ent, self.Mi) @ self.Vh.T
            uu, vv = v[1], v[2]
            h = v[0] + 0.5 * (uu * uu + vv * vv) - self.b
        state = torch.stack([h, h * uu, h * vv, uu, vv])
        trace = state[:, :, self.Nq:].reshape(5, -1)[:, self.ext].reshape(5, self.K, -1)
        out = torch.empty_like(u)
        for k in range(0, self.K, 8192):
            out[:, k:k + 8192] = self._rows(state[:, k:k + 8192], trace[:, k:k + 8192], slice(k, k + 8192), t)
        return out

    def _rows(self, state, trace, ks, t):
        h, hu, hv, u, v = state
        b = self.b[ks]
        avg = lambda a: 0.5 * (a[:, :, None] + a[:, None, :])  # noqa: E731
        Qx, Qy = (self.skew[0] * avg(g[0][ks]) + self.skew[1] * avg(g[1][ks]) for g in self.G)
        hum, hvm, um, vm = avg(hu), avg(hv), avg(u), avg(v)
        P = 0.5 * h[:, :, None] * (h + b)[:, None, :]  # g {h}^2 - g {h^2} / 2 and the source's share
        flux = Qx * hum + Qy * hvm
        r = torch.stack([flux.sum(2), (flux * um + Qx * P).sum(2), (flux * vm + Qy * P).sum(2)])
        # interface: EC flux, the source's boundary share, Lax-Friedrichs
        h, hu, hv, u, v = (a[:, self.Nq:] for a in state)
        hP, huP, hvP, uP, vP = trace
        nx, ny = self.nx[ks], self.ny[ks]
        sJ = torch.sqrt(nx * nx + ny * ny)
        if self.walls:
            wall, un = self.wall[ks], (u * nx + v * ny) / sJ
            hP = torch.where(wall, h, hP)
            uP, vP = torch.where(wall, u - 2 * un * nx / sJ, uP), torch.where(wall, v - 2 * un * ny / sJ, vP)
            huP, hvP = hP * uP, hP * vP
        mass = 0.5 * (nx * (hu + huP) + ny * (hv + hvP))
        P = 0.5 * h * (hP + b[:, self.Nq:])
        f = torch.stack([mass, 0.5 * mass * (u + uP) + nx * P, 0.5 * mass * (v + vP) + ny * P])
        lam = torch.maximum(torch.abs(u * nx + v * ny) + sJ * torch.sqrt(h),
                            torch.abs(uP * nx + vP * ny) + sJ * torch.sqrt(hP))
        f -= 0.5 * lam * torch.stack([hP - h, huP - hu, hvP - hv])
        r[:, :, self.Nq:] += self.wf * f
        force = self._force(ks, t) if self.mms else None
        if self.sbp:
            s = torch.zeros_like(r[:, :, :self.Nq]).index_add_(2, self.node, r)
            du = -s / (self.w * self.J[ks])
            return du if force is None else du + force
        s = r @ self.Vh
        if force is not None:
            s = s - ((self.w * self.J[ks]) * force) @ self.Vq
        return -torch.einsum("knm,ckm->ckn", self.Mi[ks], s)

    def _force(self, ks, t):
        """q_t + div F + source of h = 2 + 0.1 sin pi (x + y - t), u = v = 1/2."""
        x, y = self.xq[ks], self.yq[ks]
        h = 2 + 0.1 * torch.sin(np.pi * (x + y - t))
        c = 0.1 * np.pi * torch.cos(np.pi * (x + y - t))
        bx = -0.1 * np.pi * torch.sin(np.pi * x) * torch.cos(np.pi * y)
        by = -0.1 * np.pi * torch.cos(np.pi * x) * torch.sin(np.pi * y)
        return torch.stack([0 * c, (h + 0 * c) * (c + bx), (h + 0 * c) * (c + by)])

    def steps(self, u, n, t):
        u, res = u.clone(), torch.zeros_like(u)
        for k in range(n):
            for a, b, c in zip(_RK_A, _RK_B, _RK_C):
                res = a * res + self.dt * self.rhs(u, t + k * self.dt + c * self.dt)
                u += b * res
        return u

    def monitor(self, u, q, t):
        du = self.rhs(u, t)
        a, d = (u, du) if self.sbp else (u @ self.Vq.T, du @ self.Vq.T)
        w, b = self.w * self.J, self.b[:, :self.Nq]
        uu, vv = a[1] / a[0], a[2] / a[0]
        entropy = (w * (0.5 * (a[1] * uu + a[2] * vv) + 0.5 * a[0] ** 2 + a[0] * b)).sum()
        rate = (w * ((a[0] + b - 0.5 * (uu * uu + vv * vv)) * d[0] + uu * d[1] + vv * d[2])).sum()
        error = (w * (a - q) ** 2).sum((1, 2)).sqrt()
        return dict(entropy=float(entropy), mass=float((w * a[0]).sum()), rate=float(rate),
                    error=error.cpu().numpy())


def exact(case, seed):
    if case["call"] == "ensemble":
        return [exact(m, seed * 64 + i) for i, m in enumerate(_members(case))]
    p, e = _Problem(case, seed), _Exact(case)
    u, q = e.data(p)
    if case["call"] == "rhs":
        return e.rhs(u, p.t0)
    if case["call"] == "monitor":
        return e.monitor(u, q, p.t0)
    return e.steps(u, case["steps"], p.t0)
