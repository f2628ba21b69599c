"""The step in slabs: boxes above 2^26 sites, batches that hold one, and boxes whose whole scratch finds no memory.

The arithmetic of a site does not depend on how the step is divided, so every comparison is bit for bit.  The
states vary everywhere (small noise on every field), so that a plane that is missing, stale or taken from the wrong
place shows at each seam, the periodic one included.
"""
import numpy as np
import pytest

import paper_2011_00287_gb300 as L
from paper_2011_00287_gb300 import lbcad as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2011_00287_gb300 import build
    build.build()


def _noise(shape, prec, seed, q=19):
    """A state as lbcad_set_state takes it: populations, Q, psi and u, each with noise of its own size."""
    import torch
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(seed)
    n = shape[0] * shape[1] * shape[2]
    dt = torch.float64 if prec == L.FP64 else torch.float32
    s = torch.empty((q + 9) * n, dtype=dt, device="cuda:0")
    at = 0
    _, w = L.lattice(L.D3Q15 if q == 15 else L.D3Q19)
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


class _Bounded(B._TorchAllocator):
    """Refuses every request above `most` bytes that is not a buffer of a state."""
    most, keep, refused = 0, (), 0

    def _alloc(self, nbytes, user):
        if self.most and nbytes > self.most and nbytes not in self.keep:
            type(self).refused += 1
            return None
        return super()._alloc(nbytes, user)


def _bound(monkeypatch, shapes, prec, q, planes):
    """No scratch of more than `planes` planes of the first box; buffers of the state as they are."""
    es = 8 if prec == L.FP64 else 4
    keep = set()
    for s in shapes:
        n = s[0] * s[1] * s[2]
        keep |= {(c * n * es + 255) // 256 * 256 for c in (q, 5, 1, 3)}
    monkeypatch.setattr(_Bounded, "keep", keep)
    # (requests come in multiples of 256 bytes)
    monkeypatch.setattr(_Bounded, "most", (planes * 12 * es * shapes[0][0] * shapes[0][1] + 255) // 256 * 256)
    monkeypatch.setattr(_Bounded, "refused", 0)
    monkeypatch.setattr(B, "_TorchAllocator", _Bounded)


@pytest.mark.parametrize("prec", [L.FP64, L.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("planes", [3, 8, 25])
@pytest.mark.parametrize("shapes,kw", [
    ([(64, 52, 40)], {}), ([(67, 49, 41), (9, 7, 6), (33, 31, 30)], {}), ([(64, 52, 40)], dict(lattice=L.D3Q15)),
], ids=["box", "batch", "d3q15"])
def test_step_with_less_scratch_is_the_same_step(monkeypatch, shapes, kw, planes, prec):
    """Where the scratch of whole boxes finds no memory, smaller slabs step them; so a box that fitted before there was
    a scratch still fits.  The seams lie anywhere in the noise of the state."""
    import torch
    q = 15 if kw else 19
    kw = dict(kw, tau=1.5)
    states = [_noise(s, prec, 21 + i, q) for i, s in enumerate(shapes)]
    ref = _run(shapes, states, prec, 4, **kw)
    _bound(monkeypatch, shapes, prec, q, planes)
    got = _run(shapes, states, prec, 4, **kw)
    assert _Bounded.refused > 0
    for s, (a, sums_a), (b, sums_b) in zip(shapes, got, ref):
        assert torch.isfinite(b).all() and torch.equal(a, b), s
        assert np.abs(sums_a - sums_b).max() <= 1e-12 * np.prod(s), s


def test_adjoint_with_less_scratch_is_the_same(monkeypatch):
    """The replay of the adjoint steps in the same slabs."""
    shape = (40, 36, 33)

    def grad():
        sim = L.Simulation([shape], [L.default_params(shape, R=9.0, p0=12.0, zeta=0.02)], seed=3)
        out = sim.adjoint(7, 3)
        sim.close()
        return out

    ref = grad()
    n = int(np.prod(shape))
    _bound(monkeypatch, [shape], L.FP32, 19, 8)
    # and the adjoint's own: checkpoints, segment, cotangents, work, forces
    sizes = {(v * n * 4 + 255) // 256 * 256 for v in (3 * 28, 4 * 28, 2 * 28, 56, 9)}
    monkeypatch.setattr(_Bounded, "keep", _Bounded.keep | sizes)
    got = grad()
    assert _Bounded.refused > 0
    assert np.array_equal(got[3], ref[3])
    np.testing.assert_allclose(got[:3], ref[:3], rtol=1e-9)


class _Budget(B._TorchAllocator):
    """Gives out at most `total` bytes at a time."""
    total, asked = None, 0

    def _alloc(self, nbytes, user):
        held = sum(t.numel() for t in self.live.values())
        if self.total is not None and held + nbytes > self.total:
            return None
        type(self).asked = max(self.asked, held + nbytes)
        return super()._alloc(nbytes, user)


@pytest.mark.parametrize("prec", [L.FP64, L.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("shapes", [[(64, 52, 40)], [(67, 49, 41), (9, 7, 6), (33, 31, 30)]], ids=["box", "batch"])
def test_create_wherever_the_scratch_meets_the_end_of_the_memory(monkeypatch, shapes, prec):
    """The scratch leaves room for what is allocated besides it: a context is created in every budget between the one
    with the whole scratch and one with three planes of it, the one that only the last work list exceeds included."""
    import torch
    monkeypatch.setattr(B, "_TorchAllocator", _Budget)
    monkeypatch.setattr(_Budget, "asked", 0)
    states = [_noise(s, prec, 31 + i) for i, s in enumerate(shapes)]
    ref = _run(shapes, states, prec, 3)
    whole, es = _Budget.asked, 8 if prec == L.FP64 else 4
    scratch = 12 * es * sum(int(np.prod(s)) for s in shapes)
    # (three planes of the largest box, and lists of one-plane slabs: at most 20 bytes an item, 96 a slot)
    least = whole - scratch + 3 * 12 * es * shapes[0][0] * shapes[0][1] + (1 << 20)
    assert least < whole
    for total in (whole - 1, whole - 256, whole - 4096, whole - scratch // 8, (whole + least) // 2, least):
        monkeypatch.setattr(_Budget, "total", total)
        got = _run(shapes, states, prec, 3)
        for s, (a, _), (b, _) in zip(shapes, got, ref):
            assert torch.equal(a, b), (s, total)
    monkeypatch.setattr(_Budget, "total", whole - scratch)
    with pytest.raises(B.LbcadError) as e:
        _run(shapes, states, prec, 3)
    assert e.value.code == B.LBCAD_E_OOM


@pytest.mark.parametrize("graph", [0, 2])
@pytest.mark.parametrize("prec", [L.FP64, L.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("shapes", [[(64, 52, 40)], [(67, 49, 41), (9, 7, 6), (33, 31, 30)]], ids=["box", "batch"])
def test_calls_that_need_the_memory_of_the_scratch(monkeypatch, shapes, prec, graph):
    """Buffers that later calls need (fields on their way to and from the host, the scratch of another path) may take the
    memory of the step's scratch; the steps after that, in smaller slabs, are the same steps."""
    import torch
    monkeypatch.setattr(B, "_TorchAllocator", _Budget)
    monkeypatch.setattr(_Budget, "total", None)
    monkeypatch.setattr(_Budget, "asked", 0)
    states = [_noise(s, prec, 41 + i) for i, s in enumerate(shapes)]
    ref = _run(shapes, states, prec, 7)
    whole, es, n0 = _Budget.asked, 8 if prec == L.FP64 else 4, int(np.prod(shapes[0]))

    def sim_in(total):
        monkeypatch.setattr(_Budget, "total", total)
        sim = L.Simulation(list(shapes), [L.default_params(s, R=min(s) / 4.0, p0=16.0, precision=prec) for s in shapes],
                           seed=1)
        sim.set_graph(graph)
        for i, s in enumerate(states):
            sim.set_state(i, s)
        return sim

    def check(sim):
        for i, (r, sums) in enumerate(ref):
            o = torch.empty_like(r)
            sim.get_state(i, out=o)
            assert torch.equal(o, r), shapes[i]
            assert np.abs(sim.observables(i) - sums).max() <= 1e-12 * r.numel()
        sim.close()

    # psi of the first box on its way to the host: 8 bytes a site where 1 is left
    sim = sim_in(whole + n0)
    sim.step(4)
    psi = sim.get_fields(0, L.FIELD_PSI)
    sim.step(2)
    sim.set_fields(0, {"psi": sim.get_fields(0, L.FIELD_PSI)["psi"]})
    sim.step(1)
    assert np.isfinite(psi["psi"]).all()
    check(sim)
    # the scratch of the two-kernel path: 15 values a site where as much is left but for half the step's scratch
    sites = sum(int(np.prod(s)) for s in shapes)
    sim = sim_in(whole + 15 * es * sites - 6 * es * sites)
    sim.step(4)
    sim.set_path(B.PATH_TWO_KERNEL)
    sim.set_path(B.PATH_FUSED)
    sim.step(3)
    check(sim)
    # more than the scratch can give: refused, and the context steps on
    sim = sim_in(whole)
    sim.step(4)
    with pytest.raises(B.LbcadError) as e:
        sim.set_path(B.PATH_TWO_KERNEL)
    assert e.value.code == B.LBCAD_E_OOM
    sim.step(3)
    check(sim)


def test_adjoint_after_the_scratch_gave_up_memory(monkeypatch):
    monkeypatch.setattr(B, "_TorchAllocator", _Budget)
    monkeypatch.setattr(_Budget, "total", None)
    shape = (40, 36, 33)

    def grad(bounded):
        sim = L.Simulation([shape], [L.default_params(shape, R=9.0, p0=12.0, zeta=0.02)], seed=3)
        if bounded:
            monkeypatch.setattr(_Budget, "total", sum(t.numel() for t in sim._alloc.live.values()) + 1024)
            sim.get_fields(0, L.FIELD_PSI)
            monkeypatch.setattr(_Budget, "total", None)
        out = sim.adjoint(7, 3)
        sim.close()
        return out

    ref, got = grad(False), grad(True)
    assert np.array_equal(got[3], ref[3])
    np.testing.assert_allclose(got[:3], ref[:3], rtol=1e-9)
