"""The tiled pushes of order 4 in 2D and of ragged 3D grids when particles leave
their tile's box between two sorts (gather and deposit in device memory; in 3D
the deferred list), across periodic and absorbing faces of partial tiles: the
one-thread push and the FP64 oracle, to the tolerances of the same comparison at
order 2 on whole tiles."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic, workloads as W
from tests.helpers import oracle_from_workload, random_state

pytestmark = pytest.mark.gpu
A, P = W.ABSORB, W.PERIODIC


@pytest.mark.parametrize("n,order,tile,bc", [((45, 37), 4, (8, 8, 1), (P, P)), ((45, 37), 4, (16, 16, 1), (A, P)),
                                             ((13, 10, 9), 2, (4, 4, 4), (P, P, P)),
                                             ((13, 10, 9), 2, (4, 4, 4), (A, P, A)),
                                             ((18, 15, 12), 2, (4, 4, 4), (P, A, P))])
def test_off_box_particles_match_simple_kernel_and_oracle(n, order, tile, bc):
    dim = len(n)
    dx = (0.1, 0.12, 0.11)[:dim]
    dt = 0.9 / np.sqrt(sum(1.0 / d ** 2 for d in dx))
    w, F = random_state(dim, n, dx, dt, 3, seed=860 + n[0] + order, umax=3.0, bc=bc)
    sims = [pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=50, tile=tile, push_variant=v, order=order)
            for v in (pic.PUSH_AUTO, pic.PUSH_SIMPLE)]
    o = oracle_from_workload(w, sort_interval=50, tile=tile)
    o.set_order(order)
    for c in range(9):
        for s in sims:
            s.pic_set_field(c, F[c])
        o.set_field(c, F[c])
    for s in sims:
        s.pic_step(10)
    o.step(10)
    pa, pb, po = sims[0].pic_get_particles(0), sims[1].pic_get_particles(0), o.particles(0)
    # (a particle within the tolerance of an absorbing face may end on either side of it)
    assert (pa["alive"] != po["alive"]).sum() <= 2 and (pb["alive"] != po["alive"]).sum() <= 2
    live = (pa["alive"] != 0) & (pb["alive"] != 0) & (po["alive"] != 0)
    assert live.sum() > 0.3 * live.size
    umag = np.sqrt(po["ux"] ** 2 + po["uy"] ** 2 + po["uz"] ** 2)
    for d, k in enumerate(("x", "y", "z")[:dim]):
        for other in (pb, po):
            e = pa[k] - other[k]
            e -= n[d] * dx[d] * np.round(e / (n[d] * dx[d]))
            assert np.max(np.abs(e[live])) <= 1e-4, k
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(pa[k] - pb[k])[live]) < 1e-4, k
        assert np.all((np.abs(pa[k] - po[k]) <= 1e-4 * (umag + 1.0))[live]), k
    da, db, do = sims[0].pic_diagnostics(), sims[1].pic_diagnostics(), o.diagnostics()
    for k in ("U_E", "U_B"):
        assert abs(da[k] - db[k]) <= 1e-4 * max(db["U_E"], db["U_B"])
        assert abs(da[k] - do[k]) <= 1e-4 * max(do["U_E"], do["U_B"])
    if not (pa["alive"] != po["alive"]).any():
        assert abs(da["U_kin"][0] / do["U_kin"][0] - 1.0) <= 1e-4
    for s in sims:
        s.close()
