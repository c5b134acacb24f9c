"""Field half steps and the current fold where their launches change: 1D grids
on both sides of the one-block line, fold blocks leading the B update with
periodic, absorbing and mixed axes, the smallest periodic axis (all shell), a
laser entering on ragged rows.  Each against the FP64 oracle."""
import math

import numpy as np
import pytest

from paper_2104_00642_gb300 import pic, workloads as W
from tests.helpers import oracle_from_workload, random_state, window_scale

pytestmark = pytest.mark.gpu

TOL = {pic.FP32_CELLOFF: 1e-5, pic.FP64_PLAIN: 1e-10}
A, P = W.ABSORB, W.PERIODIC


@pytest.mark.parametrize("prec", list(TOL))
@pytest.mark.parametrize("n,bc,laser", [((8,), (P,), False), ((512,), (A,), True), ((513,), (P,), False),
                                        ((2048,), (P,), False), ((2049,), (A,), True),
                                        ((4096,), (A,), True), ((4097,), (A,), False),
                                        ((8, 21), (P, A), False), ((30, 8), (A, P), True), ((264, 9), (P, P), False),
                                        ((8, 8, 8), (P, P, P), False), ((9, 8, 11), (P, A, P), False),
                                        ((12, 9, 8), (A, P, A), False),
                                        # the laser's transverse profile covers n rows of an absorbing
                                        # axis; on the last node's row the oracle has the wave, too
                                        pytest.param((12, 9, 8), (A, P, A), True,
                                                     marks=pytest.mark.xfail(strict=True))])
def test_fields_and_fold_match_oracle(n, bc, laser, prec):
    dim = len(n)
    dx = (0.1, 0.12, 0.11)[:dim]
    dt = 0.9 / math.sqrt(sum(1.0 / d ** 2 for d in dx))
    w, F = random_state(dim, n, dx, dt, 2, seed=700 + n[0], bc=bc)
    if laser:
        w.laser = W.Laser(a0=2.0, waist=0.5 if dim > 1 else 0.0, fwhm=0.5, t_peak=0.2, x_focus=0.4,
                          yc=0.5 * w.n[1] * w.dx[1], zc=0.5 * w.n[2] * w.dx[2], pol=1)
    sim = pic.from_workload(w, precision=prec)
    o = oracle_from_workload(w)
    for c in range(9):
        sim.pic_set_field(c, F[c])
        o.set_field(c, F[c])
    # a call's first and last half steps, then those between two steps; a step
    # adds the rounding of its fields and currents, and from the second on of
    # currents whose particles are up to 10 tol cells off
    tol = TOL[prec]
    for steps, total in ((1, 1), (2, 3)):
        sim.pic_step(steps)
        o.step(steps)
        po = o.particles(0)
        jmax = max(window_scale(po, w, dim, a).max() for a in range(3))
        fmax = max(max(np.abs(o.field(c)).max(), 1.0) for c in range(6))
        bound = total * tol * (2 * fmax + w.dt * jmax) + (total - 1) * 20 * tol * w.dt * jmax
        for c in range(6):
            assert np.max(np.abs(sim.pic_fields(c) - o.field(c))) <= bound, (steps, c)
        for c, ax in ((pic.JX, 0), (pic.JY, 1), (pic.JZ, 2)):
            scale = window_scale(po, w, dim, ax, reach=3 + total).max()
            assert np.max(np.abs(sim.pic_fields(c) - o.field(c))) <= (1 + 20 * (total - 1)) * tol * scale, (steps, c)
    sim.close()
