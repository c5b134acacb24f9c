"""The FP64 push where its roundings decide: positions on cell faces, nodes and
half nodes, particles that stay, cross a node or cross a face."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests.helpers import oracle_from_workload, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dx", [0.1, 0.07, 1.0 / 3.0, 0.25])
def test_positions_on_faces_and_nodes(dx, order):
    """every k dx / 2 at rest and with small momenta of both signs: cells and
    currents as the oracle's (cells exactly: floor(x / dx); FP64 tolerance
    1e-10 of |q w| dx / dt times the five particles of a window)"""
    n = 24
    w, F = random_state(1, (n,), (dx,), 0.9 * dx, 1, seed=3, fields=False)
    s = w.species[0]
    x = np.repeat(np.arange(2 * n) * (0.5 * dx), 3)
    x = x[x < n * dx]
    s.x = x
    for k in ("y", "z", "uy", "uz"):
        setattr(s, k, np.zeros(x.size))
    s.ux = np.tile([0.0, 1e-9, -0.3], x.size // 3)
    s.capacity = x.size
    sim = pic.from_workload(w, precision=pic.FP64_PLAIN, order=order)
    o = oracle_from_workload(w)
    o.set_order(order)
    sim.pic_step(1)
    o.step(1)
    pg, po = sim.pic_get_particles(0), o.particles(0)
    assert np.max(np.abs(pg["x"] - po["x"])) <= 1e-13
    cells, _ = sim.pic_get_cells(0)
    assert np.array_equal(cells, np.clip(np.floor(pg["x"] / dx), 0, n - 1).astype(np.uint32))
    scale = 0.1 * dx / w.dt * 30
    for c in (pic.JX, pic.JY, pic.JZ):
        assert np.max(np.abs(sim.pic_fields(c) - o.field(c))) <= 1e-10 * scale
    sim.close()
