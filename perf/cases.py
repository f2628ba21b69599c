"""The work that users of this library have it do, as cases that can be timed and checked.

Almost every case is one pass of a parameter study: restore a saved state (lbcad_set_state),
advance it by a few hybrid steps, read the conserved sums and the centroid moments
(lbcad_observables) and save the new state (lbcad_get_state or lbcad_get_fields).  The passes
differ in what such studies differ in: the box (from a few thousand sites, where launches count,
to 256^3; cubes, uneven and odd edges), one droplet or a batch of them, FP32 or FP64, the
integrator and the coupling, the velocity set and the LB form, steps launched one by one or
replayed from a CUDA graph.  One family runs the adjoint instead: the gradient of the droplet's
drift.

The states are droplets in motion: a tanh droplet with a noisy cholesteric helix, carried by a
smooth flow of the size that active droplets make (|u| of a few 1e-3), populations at
equilibrium with it.  Sums and gradients of an FP32 run are returned in float32, the precision
its state has.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2011_00287_gb300 as L

DEV = "cuda:0"

# kinds of step: (precision, Simulation parameters).  The stress-in-equilibrium form and D3Q15
# run at relaxation times where the schemes are stable on a droplet.
KINDS = {
    "fp32": dict(precision=L.FP32),
    "fp64": dict(precision=L.FP64),
    "sync": dict(precision=L.FP32, coupling=L.SYNC),
    "heun": dict(precision=L.FP32, integrator=L.HEUN, coupling=L.LAGGED),
    "heun_sync": dict(precision=L.FP32, integrator=L.HEUN, coupling=L.SYNC),
    "d3q15": dict(precision=L.FP32, lattice=L.D3Q15),
    "stress": dict(precision=L.FP32, lb_form=L.LB_STRESS_EQ, tau=1.5),
    "d3q15_stress": dict(precision=L.FP32, lattice=L.D3Q15, lb_form=L.LB_STRESS_EQ, tau=2.5),
    "adjoint": dict(precision=L.FP32),
}
MAX_SITES = 256 ** 3
MAX_WORK = 6 * MAX_SITES  # site updates of the largest case


def listed():
    return [
        # a quick look at a very small droplet in an odd box: launches and latency decide
        dict(name="small_odd", kind="fp32", nx=21, ny=13, nz=10, steps=20, graph=0, count=1, zeta=0.01, pitch=8.0),
        # the small droplet of parameter scans and convergence checks
        dict(name="droplet_32", kind="fp32", nx=32, ny=32, nz=32, steps=20, graph=0, count=1, zeta=0.005, pitch=16.0),
        # a long swim: the 64^3 droplet whose steps are replayed from a CUDA graph
        dict(name="droplet_64_graph", kind="fp32", nx=64, ny=64, nz=64, steps=20, graph=10, count=1, zeta=0.005,
             pitch=32.0),
        # an elongated box with odd edges, as a channel or a film is
        dict(name="channel_odd", kind="fp32", nx=101, ny=47, nz=73, steps=12, graph=0, count=1, zeta=0.005, pitch=16.0),
        # the benchmark's droplet
        dict(name="droplet_128", kind="fp32", nx=128, ny=128, nz=128, steps=20, graph=0, count=1, zeta=0.005,
             pitch=32.0),
        # the largest droplet that is run in earnest
        dict(name="droplet_256", kind="fp32", nx=256, ny=256, nz=256, steps=6, graph=0, count=1, zeta=0.005,
             pitch=48.0),
        # a scan over activity and pitch: uneven boxes advanced by the same launches
        dict(name="batch_12", kind="fp32", nx=96, ny=96, nz=96, steps=10, graph=2, count=12, zeta=0.005, pitch=24.0),
        # the FP64 run that an FP32 one is checked against
        dict(name="fp64_32", kind="fp64", nx=32, ny=32, nz=32, steps=10, graph=0, count=1, zeta=0.005, pitch=16.0),
        # advection with the velocity of the same step
        dict(name="sync_96", kind="sync", nx=96, ny=80, nz=64, steps=10, graph=0, count=1, zeta=0.005, pitch=20.0),
        # the predictor-corrector
        dict(name="heun_sync_128", kind="heun_sync", nx=128, ny=128, nz=128, steps=8, graph=0, count=1, zeta=0.005,
             pitch=32.0),
        # the 15-velocity set with the stress in the equilibrium
        dict(name="d3q15_stress", kind="d3q15_stress", nx=72, ny=50, nz=61, steps=10, graph=0, count=1, zeta=0.005,
             pitch=16.0),
        # the gradient of the drift with respect to activity, chirality and the initial order
        dict(name="adjoint_64", kind="adjoint", nx=64, ny=64, nz=64, steps=40, graph=0, count=1, zeta=0.005,
             pitch=16.0),
    ]


def _edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp32"] * 6 + ["batch"] * 2 + ["fp64", "sync", "heun", "heun_sync", "d3q15", "stress",
                                                       "d3q15_stress", "adjoint"])
    hi = {"fp32": 256, "batch": 96, "fp64": 48, "adjoint": 80}.get(kind, 144)
    lo = 48 if kind == "batch" else 8
    while True:
        nx, ny, nz = (_edge(rng, lo, hi) for _ in range(3))
        if rng.random() < 0.3:
            ny = nz = nx
        if nx * ny * nz >= 1000:
            break
    count = rng.randint(4, 12) if kind == "batch" else 1
    most = min(20, MAX_WORK // (2 * nx * ny * nz * count))
    steps = rng.randint(min(4, most), most)
    graph = rng.choice([0, 2]) if kind in ("fp32", "batch") else 0
    if kind == "adjoint":
        steps = rng.randint(10, 30)
    return dict(kind="fp32" if kind == "batch" else kind, nx=nx, ny=ny, nz=nz, steps=steps, graph=graph, count=count,
                zeta=round(rng.uniform(0.001, 0.01), 5), pitch=round(rng.uniform(8.0, 40.0), 3))


def _instances(case):
    """The grid, the activity and the pitch of each instance: for a batch, boxes of edges from half of the
    case's upwards, and a spread of activities and pitches, the same for every seed."""
    base = (case["nx"], case["ny"], case["nz"])
    if case["count"] == 1:
        return [(base, case["zeta"], case["pitch"])]
    rng = np.random.default_rng(case["count"])
    out = []
    for _ in range(case["count"]):
        g = tuple(int(v) for v in np.round(np.asarray(base) * rng.choice([0.5, 0.66, 0.83, 1.0], size=3)))
        out.append((g, case["zeta"] * float(rng.uniform(0.2, 2.0)), case["pitch"] * float(rng.uniform(0.5, 1.6))))
    return out


def _params(case, grid, zeta, pitch):
    return L.default_params(grid, R=min(grid) / 4.0, p0=pitch, zeta=zeta, **KINDS[case["kind"]])


_C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
        (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
        (0, -1, 1)]
_C15 = _C19[:7] + [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]
_W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_W15 = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8


def _velocities(case):
    return (_C15, _W15) if KINDS[case["kind"]].get("lattice") == L.D3Q15 else (_C19, _W19)


def _start(case, inst, grid, zeta, pitch, seed):
    """The saved state of one instance, as lbcad_get_state lays it out: the stored populations, Q, psi and u."""
    nx, ny, nz = grid
    prm = _params(case, grid, zeta, pitch)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * int(seed) + inst)
    rng = np.random.default_rng([int(seed), inst])
    f64 = dict(dtype=torch.float64, device=DEV)
    z = torch.arange(nz, **f64).reshape(nz, 1, 1)
    y = torch.arange(ny, **f64).reshape(1, ny, 1)
    x = torch.arange(nx, **f64).reshape(1, 1, nx)
    centre = [c + float(rng.uniform(-1.0, 1.0)) for c in prm["centre"]]
    r = torch.sqrt((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2)
    psi = torch.tanh((prm["R"] - r) / 2.0)
    dz = z - centre[2] + 0.0 * r
    n0, n1 = torch.cos(prm["q0"] * dz), torch.sin(prm["q0"] * dz)
    S0, inside = prm["S0"], (r < prm["R"]).to(torch.float64)
    q = torch.stack([S0 * (n0 * n0 - 1 / 3), S0 * n0 * n1, 0 * n0, S0 * (n1 * n1 - 1 / 3), 0 * n0])
    q += prm["noise"] * (2.0 * torch.rand(q.shape, generator=gen, **f64) - 1.0)
    q *= inside
    # a steady stream and one long shear wave along each axis
    k = [2 * math.pi / n for n in (nx, ny, nz)]
    ph = rng.uniform(0, 2 * math.pi, size=6)
    am = rng.uniform(1e-3, 3e-3, size=6)
    drift = rng.uniform(2e-3, 5e-3, size=3)
    u = torch.stack([drift[0] + am[0] * torch.sin(k[1] * y + ph[0]) + am[1] * torch.sin(k[2] * z + ph[1]) + 0.0 * r,
                     drift[1] + am[2] * torch.sin(k[0] * x + ph[2]) + am[3] * torch.sin(k[2] * z + ph[3]) + 0.0 * r,
                     drift[2] + am[4] * torch.sin(k[0] * x + ph[4]) + am[5] * torch.sin(k[1] * y + ph[5]) + 0.0 * r])
    u2 = (u * u).sum(0)
    C, W = _velocities(case)
    dt = torch.float64 if prm["precision"] == L.FP64 else torch.float32
    n = nx * ny * nz
    out = torch.empty((len(C) + 9) * n, dtype=dt, device=DEV)
    for i, (c, w) in enumerate(zip(C, W)):
        cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
        f = w * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2)  # f_eq - w rho0 at rho0 = 1
        out[i * n:(i + 1) * n] = ((f if dt == torch.float32 else f + w)).reshape(-1)
    m = len(C) * n
    out[m:m + 5 * n] = q.reshape(-1)
    out[m + 5 * n:m + 6 * n] = psi.reshape(-1)
    out[m + 6 * n:] = u.reshape(-1)
    return out


def prepare(case, seed):
    insts = _instances(case)
    sim = L.Simulation([g for g, _, _ in insts], [_params(case, *i) for i in insts], seed=int(seed) % (1 << 31))
    if case["graph"]:
        sim.set_graph(case["graph"])
    start = [_start(case, k, *i, seed) for k, i in enumerate(insts)]
    out = [torch.empty_like(s) for s in start]
    return dict(case=case, sim=sim, start=start, out=out, q=len(_velocities(case)[0]))


def _split(buf, grid, q):
    nx, ny, nz = grid
    n = nx * ny * nz
    at = [0, q * n, (q + 5) * n, (q + 6) * n, (q + 9) * n]
    return {k: buf[at[j]:at[j + 1]].reshape(-1, nz, ny, nx) for j, k in enumerate(("g", "q", "psi", "u"))}


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "adjoint":
        sim.set_state(0, state["start"][0])
        J, dz, dq, dQ0 = sim.adjoint(case["steps"], max(1, case["steps"] // 4))
        return {"J_dzeta_dq0": np.array([J, dz, dq], dtype=np.float32), "dQ0": dQ0.astype(np.float32)}
    for i, s in enumerate(state["start"]):
        sim.set_state(i, s)
    sim.step(case["steps"])
    res = {}
    for i, g in enumerate(sim.grids):
        obs = sim.observables(i)
        if case["kind"] == "fp64":
            res["i%d" % i] = dict(sim.get_fields(i, on_device=True), obs=obs)
        else:
            sim.get_state(i, out=state["out"][i])
            res["i%d" % i] = dict(_split(state["out"][i], g, state["q"]), obs=obs.astype(np.float32))
    # a batch returns the state of each instance as one tensor
    if case["count"] > 1:
        res = {"i%d" % i: dict(state=state["out"][i], obs=res["i%d" % i]["obs"]) for i in range(case["count"])}
    return res


def work(case):
    """Each step reads and writes the state once (populations, Q, psi, u); a pass also restores and saves it.
    The adjoint runs every step forward twice and reverses it once, with a cotangent of the state's size.
    Operations: about 1,300 for the fields, the stresses, the update and the collision of a site."""
    sites = sum(g[0] * g[1] * g[2] for g, _, _ in _instances(case))
    es = 8 if case["kind"] == "fp64" else 4
    state = (len(_velocities(case)[0]) + 9) * es * sites
    if case["kind"] == "adjoint":
        return dict(bytes=state * 2 * case["steps"] * 3.5, flops=1300.0 * 5 * sites * case["steps"])
    heun = 1.6 if "heun" in case["kind"] else 1.0
    return dict(bytes=2.0 * state * (case["steps"] + 2), flops=1300.0 * heun * sites * case["steps"])


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

def _sh(f, c):
    """f(x + c) on the periodic box."""
    return f if c == (0, 0, 0) else torch.roll(f, shifts=(-c[2], -c[1], -c[0]), dims=(-3, -2, -1))


def _grad(f):
    """Isotropic gradient and the sum of w-weighted differences: (d_x, d_y, d_z, lap)."""
    g, lap = [0.0, 0.0, 0.0], 0.0
    for c, w in zip(_C19[1:], _W19[1:]):
        v = _sh(f, c)
        for a in range(3):
            if c[a]:
                g[a] = g[a] + 3.0 * w * c[a] * v
        lap = lap + 6.0 * w * (v - f)
    return g[0], g[1], g[2], lap


def _full(q):
    return [[q[0], q[1], q[2]], [q[1], q[3], q[4]], [q[2], q[4], -q[0] - q[3]]]


def _fields(p, q, psi):
    """H (3x3), mu and sigma (3x3) of Eqs. 1-5."""
    R3 = range(3)
    dq = [_grad(q[k]) for k in range(5)]
    dpx, dpy, dpz, lapp = _grad(psi)
    dp = [dpx, dpy, dpz]
    Q = _full(q)
    dQ = [_full([dq[k][a] for k in range(5)]) for a in R3]
    lapQ = _full([dq[k][3] for k in range(5)])
    e = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    neg = lambda c: tuple(-v for v in c)  # noqa: E731
    add = lambda c, d: tuple(u + v for u, v in zip(c, d))  # noqa: E731
    hess = [[None] * 3 for _ in R3]
    for a in R3:
        hess[a][a] = _sh(psi, e[a]) + _sh(psi, neg(e[a])) - 2.0 * psi
        for b in range(a + 1, 3):
            hess[a][b] = hess[b][a] = 0.25 * (_sh(psi, add(e[a], e[b])) + _sh(psi, add(neg(e[a]), neg(e[b])))
                                              - _sh(psi, add(e[a], neg(e[b]))) - _sh(psi, add(neg(e[a]), e[b])))
    chi = p["chi0"] + p["chis"] * (1.0 + psi)
    QQ = [[sum(Q[i][m] * Q[m][j] for m in R3) for j in R3] for i in R3]
    t2 = QQ[0][0] + QQ[1][1] + QQ[2][2]
    t3 = sum(QQ[i][j] * Q[i][j] for i in R3 for j in R3)
    C = [[dQ[(a + 1) % 3][(a + 2) % 3][b] - dQ[(a + 2) % 3][(a + 1) % 3][b] for b in R3] for a in R3]
    g2 = dp[0] ** 2 + dp[1] ** 2 + dp[2] ** 2
    A0, K, q0, W = p["A0"], p["K"], p["q0"], p["W"]
    H = [[None] * 3 for _ in R3]
    for i in R3:
        for j in R3:
            H[i][j] = (-A0 * (1 - chi / 3) * Q[i][j] + A0 * chi * (QQ[i][j] - t2 * Q[i][j]) + K * lapQ[i][j]
                       - 2 * K * q0 * (C[i][j] + C[j][i]) - 4 * K * q0 * q0 * Q[i][j] - W * dp[i] * dp[j])
            if i == j:
                H[i][j] = H[i][j] - (A0 * chi * t2 - W * g2) / 3
    mu = (-p["a"] * psi + p["b"] * psi ** 3 - p["kphi"] * lapp
          + A0 * p["chis"] * (-t2 / 6 - t3 / 3 + t2 * t2 / 4)
          - 2 * W * (sum(dQ[a][a][b] * dp[b] for a in R3 for b in R3)
                     + sum(Q[a][b] * hess[a][b] for a in R3 for b in R3)))
    G = [[sum(dQ[a][m][n] * dQ[b][m][n] for m in R3 for n in R3) for b in R3] for a in R3]
    Qdp = [sum(Q[i][m] * dp[m] for m in R3) for i in R3]
    f = (-0.5 * p["a"] * psi ** 2 + 0.25 * p["b"] * psi ** 4 + 0.5 * p["kphi"] * g2
         + A0 * (0.5 * (1 - chi / 3) * t2 - chi / 3 * t3 + chi / 4 * t2 * t2) + 0.5 * K * (G[0][0] + G[1][1] + G[2][2])
         + 2 * K * q0 * sum(Q[i][j] * C[i][j] for i in R3 for j in R3) + 2 * K * q0 * q0 * t2
         + W * sum(dp[i] * Qdp[i] for i in R3))
    P0 = psi * mu - f
    QH = [[sum(Q[i][m] * H[m][j] for m in R3) for j in R3] for i in R3]
    tQH = QH[0][0] + QH[1][1] + QH[2][2]
    xi, phic = p["xi"], 0.5 * (1.0 + psi)
    sig = [[None] * 3 for _ in R3]
    for a in R3:
        for b in R3:
            i, j = (b + 1) % 3, (b + 2) % 3
            v = sum(dQ[a][i][m] * Q[m][j] - dQ[a][j][m] * Q[m][i] for m in R3)
            d = 1.0 if a == b else 0.0
            sig[a][b] = (-P0 * d - xi * (QH[b][a] + QH[a][b] + 2 * H[a][b] / 3) + 2 * xi * tQH * (Q[a][b] + d / 3)
                         + QH[a][b] - QH[b][a] - p["zeta"] * phic * Q[a][b]
                         - K * G[a][b] - 2 * K * q0 * v - dp[a] * (p["kphi"] * dp[b] + 2 * W * Qdp[b]))
    return H, mu, sig


def _rhs(p, q, psi, H, mu, u):
    """Right-hand sides of Eqs. 1-2 with the advecting velocity u."""
    R3 = range(3)
    Q = _full(q)
    Wg = [_grad(u[a])[:3] for a in R3]
    e = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    xi = p["xi"]
    D = [[0.5 * (Wg[i][j] + Wg[j][i]) for j in R3] for i in R3]
    O = [[0.5 * (Wg[i][j] - Wg[j][i]) for j in R3] for i in R3]
    Qt = [[Q[i][j] + (1 / 3 if i == j else 0.0) for j in R3] for i in R3]
    tqw = sum(Q[i][j] * Wg[j][i] for i in R3 for j in R3)
    trd = D[0][0] + D[1][1] + D[2][2]
    rq = []
    for k, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2))):
        S = sum((xi * D[i][m] + O[i][m]) * Qt[m][j] + Qt[i][m] * (xi * D[m][j] - O[m][j]) for m in R3)
        S = S - 2 * xi * tqw * Qt[i][j]
        if i == j:
            S = S - 2 * xi / 9 * trd
        adv = 0.0
        for a in R3:
            m = tuple(-v for v in e[a])
            adv = adv + torch.clamp(u[a], min=0) * (q[k] - _sh(q[k], m)) + torch.clamp(u[a], max=0) * (_sh(q[k], e[a]) - q[k])
        rq.append(S - adv + p["gammaQ"] * H[i][j])
    div = 0.0
    for a in R3:
        ub = 0.5 * (u[a] + _sh(u[a], e[a]))
        J = ub * torch.where(ub > 0, psi, _sh(psi, e[a]))
        div = div + J - _sh(J, tuple(-v for v in e[a]))
    return torch.stack(rq), p["M"] * _grad(mu)[3] - div


def _step(p, C, W, g, q, psi, u):
    """One hybrid step on the stored state (g: post-collision populations of the previous step, unshifted)."""
    R3 = range(3)
    H, mu, sig = _fields(p, q, psi)
    f = [_sh(g[i], tuple(-v for v in c)) for i, c in enumerate(C)]
    stress = p["lb_form"] == L.LB_STRESS_EQ
    T = [[0.5 * (sig[a][b] - sig[b][a]) for b in R3] for a in R3] if stress else sig
    F = [sum(_grad(T[a][b])[b] for b in R3 if not (stress and a == b)) for a in R3]
    rho = sum(f)
    j = [sum(c[a] * f[i] for i, c in enumerate(C) if c[a]) for a in R3]
    un = [(j[a] if stress else j[a] + 0.5 * F[a]) / rho for a in R3]
    u2 = un[0] ** 2 + un[1] ** 2 + un[2] ** 2
    uF = sum(un[a] * F[a] for a in R3)
    gn = []
    if stress:
        P = [[rho * un[a] * un[b] - 0.5 * (sig[a][b] + sig[b][a]) for b in R3] for a in R3]
        trP = P[0][0] + P[1][1] + P[2][2]
    for i, (c, w) in enumerate(zip(C, W)):
        cu = sum(c[a] * un[a] for a in R3)
        cF = sum(c[a] * F[a] for a in R3)
        if stress:
            cPc = sum(c[a] * c[b] * P[a][b] for a in R3 for b in R3 if c[a] and c[b])
            feq = w * (rho + 3 * rho * cu + 4.5 * (cPc - trP / 3))
            src = 3 * w * cF
        else:
            feq = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * u2)
            src = (1 - 0.5 / p["tau"]) * w * (3 * (cF - uF) + 9 * cu * cF)
        gn.append(f[i] - (f[i] - feq) / p["tau"] + src)
    ua = un if p["coupling"] == L.SYNC else u
    rq, rp = _rhs(p, q, psi, H, mu, ua)
    if p["integrator"] == L.HEUN:
        q1, p1 = q + rq, psi + rp
        H1, mu1, _ = _fields(p, q1, p1)
        rq1, rp1 = _rhs(p, q1, p1, H1, mu1, ua)
        rq, rp = 0.5 * (rq + rq1), 0.5 * (rp + rp1)
    return torch.stack(gn), q + rq, psi + rp, torch.stack(list(un)), rho, [j[a] + F[a] for a in R3]


def _moments(psi):
    nz, ny, nx = psi.shape
    h = 0.5 * (1.0 + psi)
    cs, sn = [], []
    for n, dims in ((nx, (0, 1)), (ny, (0, 2)), (nz, (1, 2))):
        th = 2 * math.pi * torch.arange(n, dtype=torch.float64, device=psi.device) / n
        line = h.sum(dim=dims)
        cs.append((line * torch.cos(th)).sum())
        sn.append((line * torch.sin(th)).sum())
    return cs, sn, h.sum()


def _centroid(psi):
    cs, sn, _ = _moments(psi)
    return [torch.atan2(s, c) * n / (2 * math.pi) for s, c, n in zip(sn, cs, reversed(psi.shape))]


def _load(case, k, inst, seed):
    grid, zeta, pitch = inst
    C, W = _velocities(case)
    st = _split(_start(case, k, grid, zeta, pitch, seed).to(torch.float64), grid, len(C))
    p = _params(case, grid, zeta, pitch)
    g = st["g"] if case["kind"] == "fp64" else st["g"] + torch.tensor(W, dtype=torch.float64, device=DEV).reshape(-1, 1, 1, 1)
    return p, C, W, g, st["q"], st["psi"][0], st["u"]


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    p, C, W, g, q, psi, u = _load(case, 0, _instances(case)[0], seed)
    zeta, q0 = (torch.tensor(p[k], dtype=torch.float64, device=DEV, requires_grad=True) for k in ("zeta", "q0"))
    start = q.clone().requires_grad_(True)
    X0 = [v.detach() for v in _centroid(psi)]

    def one(g, q, psi, u, zeta, q0):
        return _step(dict(p, zeta=zeta, q0=q0), C, W, g, q, psi, u)[:4]

    q = start
    for _ in range(case["steps"]):
        g, q, psi, u = checkpoint(one, g, q, psi, u, zeta, q0, use_reentrant=False)
    J = 0.0
    for a, b, n in zip(_centroid(psi), X0, reversed(psi.shape)):
        d = a - b
        d = d - n * torch.round(d.detach() / n)
        J = J + 0.5 * d * d
    J.backward()
    return {"J_dzeta_dq0": torch.stack([J.detach(), zeta.grad, q0.grad]), "dQ0": start.grad}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    res = {}
    with torch.no_grad():
        for k, inst in enumerate(_instances(case)):
            p, C, W, g, q, psi, u = _load(case, k, inst, seed)
            for _ in range(case["steps"]):
                g, q, psi, u, rho, mom = _step(p, C, W, g, q, psi, u)
            cs, sn, sh = _moments(psi)
            obs = torch.stack([rho.sum(), psi.sum(), *(m.sum() for m in mom), *cs, *sn, sh])
            if case["kind"] == "fp64":  # get_fields gives the populations as they arrive at each site
                f = torch.stack([_sh(g[i], tuple(-v for v in c)) for i, c in enumerate(C)])
                res["i%d" % k] = dict(g=f, u=u, q=q, psi=psi, obs=obs)
                continue
            g = g - torch.tensor(W, dtype=torch.float64, device=DEV).reshape(-1, 1, 1, 1)
            if case["count"] > 1:
                res["i%d" % k] = dict(state=torch.cat([v.reshape(-1) for v in (g, q, psi, u)]), obs=obs)
            else:
                res["i%d" % k] = dict(g=g, q=q, psi=psi.unsqueeze(0), u=u, obs=obs)
    return res
