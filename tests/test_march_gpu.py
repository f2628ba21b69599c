"""Edges of the z-marching kernels: boxes at and around the tile widths (32 and 16) and heights, slabs of one
and of many planes, batches at and beyond the 28 instances of one launch, and a box cut into slabs of
its own scratch.

Tolerances, as for the other parity tests: FP64 within 1e-12 max abs per field of the FP64 oracle after 5
steps (rounding of O(1) values over about 1e3 operations a site and step), FP32 within 1e-5 relative L2 (the
FP32 path's bound over 100 steps); FP64 sums within 1e-12 relative plus 1e-10.
"""
import numpy as np
import pytest

import paper_2011_00287_gb300 as L
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2011_00287_gb300 import build as B
    B.build()
    O.build()


def _perm():
    cl, _ = L.lattice()
    co, _ = O.lattice()
    return np.array([int(np.where((co == v).all(1))[0][0]) for v in cl])


def _check(got, ref, prec):
    _, w = O.lattice()
    w = w.reshape(19, 1, 1, 1)
    exp = {"g": (ref.f - w)[_perm()], "q": ref.q, "psi": ref.psi, "u": ref.u}
    for k, e in exp.items():
        g = got[k] - w[_perm()] if k == "g" else got[k]
        if prec == L.FP64:
            assert np.abs(g - e).max() <= 1e-12, k
        else:
            assert np.linalg.norm(g - e) <= 1e-5 * np.linalg.norm(e), k


@pytest.mark.parametrize("prec", [L.FP64, L.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("var", [dict(), dict(integrator=L.HEUN, coupling=L.SYNC)], ids=["euler", "heun-sync"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (16, 16, 5), (17, 15, 6), (31, 9, 7), (33, 8, 37), (64, 4, 5), (5, 34, 66)])
def test_tile_edges_match_oracle(shape, var, prec):
    kw = dict(R=1.8, p0=6.0, zeta=0.01, W=0.05, **var)
    ref = O.State(shape, O.default_params(shape, **kw), seed=2).step(5)
    for tiles in ([0, 3] if prec == L.FP32 and not var else [None]):  # Heun keeps the shape it was created with
        sim = L.Simulation([shape], [L.default_params(shape, precision=prec, **kw)], seed=2)
        if tiles is not None:
            sim.set_tiles(tiles)
        sim.step(5)
        _check(sim.get_fields(0), ref, prec)
        if prec == L.FP64:
            np.testing.assert_allclose(sim.observables(0), ref.observables(), rtol=1e-12, atol=1e-10)


@pytest.mark.parametrize("count", [28, 29, 57])
def test_batches_around_one_launch(count):
    """28 instances go in one launch; a 29th has a launch of its own, after which all share the scratch."""
    shapes = [(6 + i % 5, 5 + i % 3, 4 + i % 7) for i in range(count)]
    kws = [dict(R=1.5, p0=6.0, zeta=0.002 * (1 + i % 4)) for i in range(count)]
    sim = L.Simulation(shapes, [L.default_params(s, precision=L.FP64, **k) for s, k in zip(shapes, kws)], seed=9)
    sim.step(4)
    for i in sorted({0, 1, 27, 28 % count, count - 1}):
        ref = O.State(shapes[i], O.default_params(shapes[i], **kws[i]), seed=9, inst=i).step(4)
        _check(sim.get_fields(i), ref, L.FP64)
        np.testing.assert_allclose(sim.observables(i), ref.observables(), rtol=1e-12, atol=1e-10)


def test_slabs_of_a_large_box_match_the_two_kernel_path():
    """Above 2^26 sites the step runs slab by slab; the same step by the two-kernel path, which has no slabs, is
    the reference (FP32, 1e-6 relative L2 as between the paths at other sizes)."""
    shape = (1024, 520, 127)
    assert shape[0] * shape[1] * shape[2] > 2 ** 26
    kw = dict(R=40.0, p0=24.0)
    out = []
    for path in (L.lbcad.PATH_FUSED, L.lbcad.PATH_TWO_KERNEL):
        sim = L.Simulation([shape], [L.default_params(shape, precision=L.FP32, **kw)], seed=4)
        sim.set_path(path)
        sim.step(2)
        out.append((sim.get_fields(0, L.FIELD_U | L.FIELD_PSI), np.array(sim.observables(0))))
        sim.close()
    (a, oa), (b, ob) = out
    for k in a:
        assert np.linalg.norm(a[k] - b[k]) <= 1e-6 * np.linalg.norm(b[k]), k
    n = float(np.prod(shape))
    assert np.abs(oa - ob).max() <= 1e-10 * n
