"""The adjoint on uneven and odd boxes: edges that are no multiple of a tile, fewer rows than a tile has, a last block
of sites that is partly empty, odd site numbers, and the three axes unlike each other, so that an exchange of two of
them shows.  The state is noisy everywhere, with a flow that moves the centroid.

References: FP64 against the oracle's forward-mode derivative, which differentiates the same arithmetic, so that
gradients agree to rounding (1e-5 relative, as on the cubes; a derivative along a random direction v is compared on the
scale of the gradient's norm, its standard deviation).  FP32 against FP64 on the same state: over nine steps the FP32
states are within 1e-6 of the FP64 ones, the displacement of the centroid (0.01 to 0.06 sites) within 1e-5, and at the few
sites (one in 1e4) whose velocity is below that error an upwind difference takes the other side; 1e-2 of the norm.
"""
import numpy as np
import pytest

import paper_2011_00287_gb300 as L
from paper_2011_00287_gb300 import observables as OB
from oracle import oracle as O

pytestmark = pytest.mark.gpu

BOXES = [(21, 13, 10), (33, 7, 5), (4, 5, 6), (37, 9, 35), (5, 34, 7)]
KW = dict(p0=8.0, zeta=0.02, W=0.05)
NSTEPS, CKPT = 9, 4  # segments of four, four and one


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2011_00287_gb300 import build as B
    B.build()
    O.build()


def _kw(shape):
    return dict(KW, R=min(shape) / 3.0)


def _state(shape):
    """Oracle state: the droplet, off the box's centre, under noise, in a flow."""
    s = O.State(shape, O.default_params(shape, **_kw(shape)), seed=3)
    rng = np.random.default_rng(shape[0])
    c, w = O.lattice()
    flow = 2e-3 * np.array([0.7, -0.4, 1.0])
    s.f *= (1.0 + 3.0 * (c @ flow)).reshape(19, 1, 1, 1)
    s.f += 1e-4 * w.reshape(19, 1, 1, 1) * rng.standard_normal(s.f.shape)
    s.q += 0.02 * rng.standard_normal(s.q.shape)
    s.psi = np.roll(s.psi, (1, 1, 1), axis=(0, 1, 2)) + 0.1 * rng.standard_normal(s.psi.shape)
    s.u += flow.reshape(3, 1, 1, 1) + 1e-3 * rng.standard_normal(s.u.shape)
    return s


def _centroid_tangent(psi, dpsi):
    nz, ny, nx = psi.shape
    out = np.zeros(3)
    for a, n, axis in ((0, nx, 2), (1, ny, 1), (2, nz, 0)):
        shp = [1, 1, 1]
        shp[axis] = n
        th = (2 * np.pi * np.arange(n) / n).reshape(shp)
        pc = 0.5 * (1 + psi)
        S, C = np.sum(pc * np.sin(th)), np.sum(pc * np.cos(th))
        dS, dC = np.sum(0.5 * dpsi * np.sin(th)), np.sum(0.5 * dpsi * np.cos(th))
        out[a] = n / (2 * np.pi) * (C * dS - S * dC) / (C * C + S * S)
    return out


def _oracle(shape, start, tangent=None, **par):
    """J and its derivative along a direction of the state or of a parameter (X(t0) held fixed)."""
    s = start.copy()
    x0 = OB.centroid(s.observables(), shape)
    t = s.step_tangent(NSTEPS, tangent or {}, **par)
    d = OB.centroid(s.observables(), shape) - x0
    d -= np.array(shape) * np.round(d / np.array(shape))
    return 0.5 * float(d @ d), float(d @ _centroid_tangent(s.psi, t["psi"]))


def _perm():
    cl, _ = L.lattice()
    co, _ = O.lattice()
    return np.array([int(np.where((co == v).all(1))[0][0]) for v in cl])


def _adjoint(shape, start, prec):
    sim = L.Simulation([shape], [L.default_params(shape, precision=prec, **_kw(shape))], seed=3)
    sim.set_fields(0, dict(g=start.f[_perm()], q=start.q, psi=start.psi, u=start.u))
    J, dz, dq, dQ0 = sim.adjoint(NSTEPS, CKPT)
    lam = sim.adjoint_fields()
    sim.close()
    assert np.array_equal(dQ0, lam["q"])
    return J, dz, dq, lam


@pytest.mark.parametrize("shape", BOXES, ids=["x".join(map(str, b)) for b in BOXES])
def test_gradients_on_uneven_boxes(shape):
    start = _state(shape)
    J, dz, dq, lam = _adjoint(shape, start, L.FP64)
    Jo, rz = _oracle(shape, start, dzeta=1.0)
    _, rq = _oracle(shape, start, dq0=1.0)
    assert J > 0 and abs(J - Jo) <= 1e-9 * Jo, (J, Jo)
    assert abs(dz - rz) <= 1e-5 * abs(rz) and abs(dq - rq) <= 1e-5 * abs(rq), (dz, rz, dq, rq)
    perm, rng = _perm(), np.random.default_rng(5)
    for name, okey in (("g", "f"), ("u", "u"), ("q", "q"), ("psi", "psi")):
        for _ in range(2):
            v = rng.standard_normal(lam[name].shape)
            tv = v[np.argsort(perm)] if name == "g" else v
            _, ref = _oracle(shape, start, {okey: tv})
            ad = float(np.sum(lam[name] * v))
            assert abs(ad - ref) <= 1e-5 * np.linalg.norm(lam[name]), (name, ad, ref)
    J32, dz32, dq32, lam32 = _adjoint(shape, start, L.FP32)
    assert abs(dz32 - dz) <= 1e-2 * abs(dz) and abs(dq32 - dq) <= 1e-2 * abs(dq), (dz32, dz, dq32, dq)
    for name in lam:
        assert np.linalg.norm(lam32[name] - lam[name]) <= 1e-2 * np.linalg.norm(lam[name]), name
