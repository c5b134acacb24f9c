"""Rounding of the tiled pushes that stand in for the one-thread push (shape
order 4 in 2D, 3D grids of any size): no further from FP64 than it."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests.helpers import oracle_from_workload, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,order,tile", [(2, (96, 80), 4, (16, 16, 1)), (2, (96, 80), 4, (8, 8, 1)),
                                              (3, (21, 22, 19), 2, (4, 4, 4))])
@pytest.mark.parametrize("umax,strength", [(0.2, 0.3), (2.0, 10.0)])
def test_no_further_from_fp64_than_the_one_thread_push(dim, n, order, tile, umax, strength):
    """one step from a state that FP32 holds exactly: the two pushes take the
    same operations in the same precision, so the root mean squares of some
    50,000 errors agree within a few percent (10 % allowed)"""
    dx = (0.125,) * dim
    dt = 0.0625
    w, F = random_state(dim, n, dx, dt, 8, seed=81, umax=umax)
    s = w.species[0]
    for d, k in enumerate(("x", "y", "z")[:dim]):
        setattr(s, k, np.floor(getattr(s, k) / dx[d] * 2.0 ** 16) * (2.0 ** -16 * dx[d]))
    for k in ("ux", "uy", "uz"):
        setattr(s, k, getattr(s, k).astype(np.float32).astype(np.float64))
    F = [(f * (strength if c < 6 else 0.0)).astype(np.float32).astype(np.float64) for c, f in enumerate(F)]
    o = oracle_from_workload(w, sort_interval=1, tile=tile)
    o.set_order(order)
    for c in range(9):
        o.set_field(c, F[c])
    o.step(1)
    po, rms = o.particles(0), {}
    for v in (pic.PUSH_SIMPLE, pic.PUSH_AUTO):
        sim = pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=1, tile=tile, order=order, push_variant=v)
        for c in range(9):
            sim.pic_set_field(c, F[c])
        sim.pic_step(1)
        p = sim.pic_get_particles(0)
        err = {k: p[k] - po[k] for k in ("x", "y", "z")[:dim] + ("ux", "uy", "uz")}
        for d, k in enumerate(("x", "y", "z")[:dim]):
            err[k] -= n[d] * dx[d] * np.round(err[k] / (n[d] * dx[d]))  # (a periodic image)
        err.update({k: sim.pic_fields(c) - o.field(c) for k, c in (("jx", pic.JX), ("jy", pic.JY), ("jz", pic.JZ))})
        rms[v] = {k: float(np.sqrt(np.mean(e ** 2))) for k, e in err.items()}
        sim.close()
    for k in rms[pic.PUSH_AUTO]:
        assert rms[pic.PUSH_AUTO][k] <= 1.1 * rms[pic.PUSH_SIMPLE][k], (k, rms)
