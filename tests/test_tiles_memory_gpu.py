"""A change of tile shape for which there is no memory left leaves the context as it was: the work lists and the slots
of the sums are replaced only when all of the new ones could be allocated, and a captured graph does not outlive the
lists that it reads."""
import numpy as np
import pytest

import paper_2011_00287_gb300 as L
from paper_2011_00287_gb300 import lbcad as B

pytestmark = pytest.mark.gpu

SHAPE = (64, 48, 40)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2011_00287_gb300 import build
    build.build()


class _Refusing(B._TorchAllocator):
    """Gives out memory until `full` is set."""
    full = False

    def _alloc(self, nbytes, user):
        return None if self.full else super()._alloc(nbytes, user)


def _sim(monkeypatch, prec):
    monkeypatch.setattr(B, "_TorchAllocator", _Refusing)
    sim = L.Simulation([SHAPE], [L.default_params(SHAPE, R=10.0, p0=16.0, precision=prec)], seed=5)
    return sim


def _state(sim):
    return sim.get_state(0).tobytes(), sim.observables(0)


@pytest.mark.parametrize("graph", [0, 2])
def test_autotune_without_memory_for_other_shapes(monkeypatch, graph):
    ref = _sim(monkeypatch, L.FP32)
    ref.step(7)
    state, sums = _state(ref)
    sim = _sim(monkeypatch, L.FP32)
    sim.set_graph(graph)
    sim.step(2)
    sim._alloc.full = True
    chosen, ms = sim.autotune(1)
    assert ms[0] > 0 and ms[chosen] > 0 and min(ms) < 0, ms  # some shape needed more memory
    sim.step(5)
    got, got_sums = _state(sim)
    assert got == state
    np.testing.assert_allclose(got_sums, sums, rtol=1e-12, atol=1e-12 * np.prod(SHAPE))


def test_set_tiles_without_memory(monkeypatch):
    ref = _sim(monkeypatch, L.FP32)
    ref.step(7)
    state, sums = _state(ref)
    sim = _sim(monkeypatch, L.FP32)
    sim.set_graph(2)
    sim.step(2)
    sim._alloc.full = True
    with pytest.raises(B.LbcadError) as e:
        sim.set_tiles(6)
    assert e.value.code == B.LBCAD_E_OOM
    sim.step(5)
    got, got_sums = _state(sim)
    assert got == state
    np.testing.assert_allclose(got_sums, sums, rtol=0, atol=0)
