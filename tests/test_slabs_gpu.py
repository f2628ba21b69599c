"""The step in slabs: boxes above 2^26 sites, and batches that hold one.

The arithmetic of a site does not depend on how the step is divided, so every comparison is bit for bit.  The
states vary everywhere (small noise on every field), so that a plane that is missing, stale or taken from the wrong
place shows at each seam, the periodic one included.
"""
import numpy as np
import pytest

import paper_2011_00287_gb300 as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2011_00287_gb300 import build as B
    B.build()


def _noise(shape, prec, seed, q=19):
    """A state as lbcad_set_state takes it: populations, Q, psi and u, each with noise of its own size."""
    import torch
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(seed)
    n = shape[0] * shape[1] * shape[2]
    dt = torch.float64 if prec == L.FP64 else torch.float32
    s = torch.empty((q + 9) * n, dtype=dt, device="cuda:0")
    at = 0
    _, w = L.lattice()
    for comps, amp in ((q, 1e-4), (5, 0.02), (1, 0.3), (3, 1e-3)):
        s[at:at + comps * n].uniform_(-amp, amp, generator=gen)
        at += comps * n
    if prec == L.FP64:  # FP32 stores f_i - w_i rho0
        s[:q * n] += torch.tensor(w, dtype=dt, device="cuda:0").repeat_interleave(n)
    return s


def _run(shapes, states, prec, steps, **kw):
    """The states after the steps, and the sums, of one context with these boxes."""
    import torch
    prms = [L.default_params(s, R=min(s) / 4.0, p0=16.0, precision=prec, **kw) for s in shapes]
    sim = L.Simulation(list(shapes), prms, seed=1)
    for i, s in enumerate(states):
        sim.set_state(i, s)
    sim.step(steps)
    out = []
    for i, s in enumerate(states):
        o = torch.empty_like(s)
        sim.get_state(i, out=o)
        out.append((o, sim.observables(i)))
    sim.close()
    return out


@pytest.mark.parametrize("order", [(0, 1, 2), (1, 0, 2)], ids=["large-first", "large-second"])
def test_batch_with_a_box_in_slabs_steps_each_box_as_alone(order):
    import torch
    shapes = [(1000, 1000, 68), (32, 32, 32), (9, 7, 6)]  # 6.8e7 sites: slabs of 65 and 3 planes
    assert np.prod(shapes[0]) > 2 ** 26
    states = [_noise(s, L.FP32, 11 + i) for i, s in enumerate(shapes)]
    got = _run([shapes[i] for i in order], [states[i] for i in order], L.FP32, 3)
    for k, i in enumerate(order):
        (ref, sums), = _run([shapes[i]], [states[i]], L.FP32, 3)
        assert torch.isfinite(ref).all()
        assert torch.equal(got[k][0], ref), shapes[i]
        # the same FP64 sums of the same state, in another order: rounding of n terms of order one
        assert np.abs(got[k][1] - sums).max() <= 1e-12 * np.prod(shapes[i]), shapes[i]
