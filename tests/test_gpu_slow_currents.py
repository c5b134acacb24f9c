"""Currents of slow particles at one point in the tiled pushes: a step moves
such a particle by a few units of its FP32 offset, rounded up to more than v dt,
and all of an item's current lies on a few nodes of the shared fixed-point box."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests.helpers import oracle_from_workload, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,order,k,tol", [
    (2, (32, 32), 2, 0, 1e-4), (2, (32, 32), 2, 3, 1e-4), (2, (32, 32), 2, 20, 1e-4),
    # W_4's polynomials round at about 2^-22 near an edge's middle, on a move of 2^-18.6
    (2, (32, 32), 4, 20, 0.2),
    (3, (16, 12, 8), 2, 0, 1e-4), (3, (16, 12, 8), 2, 3, 1e-4), (3, (13, 10, 9), 2, 3, 1e-4)])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("count", [1, 2, 400])
def test_current_of_a_rounded_up_move(dim, n, order, k, tol, axis, count):
    """each half drift of k + 3/4 units of 2^-24 cells rounds to k + 1 (offset
    1/2, where W_2 is exact to that unit): the current is the oracle's times
    (k + 1) / (k + 3/4)"""
    if axis >= dim:
        pytest.skip("inactive axis")
    dx = (0.1,) * dim
    dt = 0.95 * 0.1 / np.sqrt(dim)
    w, _ = random_state(dim, n, dx, dt, 1, seed=1, fields=False)
    s = w.species[0]
    u = (k + 0.75) * 2.0 ** -24 / (0.5 * dt / dx[0])
    at = [5.0, 3.0, 4.0]
    at[axis] += 0.5
    for d, key in enumerate(("x", "y", "z")):
        setattr(s, key, np.full(count, at[d] * 0.1) if d < dim else np.zeros(count))
    for d, key in enumerate(("ux", "uy", "uz")):
        setattr(s, key, np.full(count, u if d == axis else 0.0))
    s.capacity = count
    tile = (4, 4, 4) if dim == 3 else (16, 16, 1)
    sim = pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=1, tile=tile, order=order)
    o = oracle_from_workload(w, sort_interval=1, tile=tile)
    o.set_order(order)
    sim.pic_step(1)
    o.step(1)
    c = (pic.JX, pic.JY, pic.JZ)[axis]
    want = o.field(c) * ((k + 1.0) / (k + 0.75))
    assert np.max(np.abs(want)) > 0.0
    assert np.max(np.abs(sim.pic_fields(c) - want)) <= tol * np.max(np.abs(want))
    sim.close()


@pytest.mark.parametrize("dim,n,order", [(2, (32, 32), 2), (2, (32, 32), 4), (3, (16, 12, 8), 2), (3, (13, 10, 9), 2)])
@pytest.mark.parametrize("power", [-70, 108])
def test_current_scales_with_the_weight(dim, n, order, power):
    """a weight times a power of two: the same fixed-point values, in units that
    many times larger"""
    w, _ = random_state(dim, n, (0.1,) * dim, 0.05, 8, seed=5, fields=False)
    J = []
    for p in (0, power):
        w.species[0].w = 0.125 * 2.0 ** p
        sim = pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=1, tile=(4, 4, 4) if dim == 3 else (16, 16, 1),
                                order=order)
        try:
            sim.pic_step(1)
        except pic.PicError:
            pass  # (fields of 1e30 may be reported; the current is there)
        J.append([sim.pic_fields(c) * 2.0 ** -p for c in (pic.JX, pic.JY, pic.JZ)])
        sim.close()
    for a, b in zip(*J):
        assert np.max(np.abs(a)) > 0.0
        # (the items' sums meet in FP32, in any order)
        assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(a))
