"""Cells of the FP64 push for positions on the faces of the longest axes."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dx", [0.1, 1.0 / 3.0])
@pytest.mark.parametrize("n", [4_000_000, 1 << 24])
def test_cells_on_faces_of_long_axes(n, dx):
    """positions within two units in the last place of k dx, at rest: the cell
    is floor(x / dx)"""
    rng = np.random.default_rng(n)
    x = rng.integers(n // 2, n - 1, 20_000) * dx
    for step in (0.0, np.inf, -np.inf):
        y = np.nextafter(x, step) if step else x
        x = np.concatenate([x, y, np.nextafter(y, step) if step else y])
    z = np.zeros(x.size)
    with pic.pic_create(1, (n,), (dx,), 0.5 * dx, [(-1.0, 1.0, 1e-6, x.size)], precision=pic.FP64_PLAIN) as s:
        s.pic_load_particles(0, x, None, None, z, z, z)
        s.pic_step(1)
        p, (cells, _) = s.pic_get_particles(0), s.pic_get_cells(0)
    assert np.array_equal(p["x"], x)
    assert np.array_equal(cells, np.floor(x / dx).astype(np.uint32))
