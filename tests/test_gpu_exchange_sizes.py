"""Field components to and from the host on the longest grids that pic_create takes."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu
PRECS = [pic.FP32_CELLOFF, pic.FP64_PLAIN]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [(8, 262_200), (8, 8, 65_600)])
def test_round_trip_on_many_rows_and_planes(n, prec):
    """more rows, and more planes, than 65535 blocks of a launch's y or z hold"""
    rng = np.random.default_rng(8)
    with pic.pic_create(len(n), n, (0.1,) * len(n), 0.05, [(-1.0, 1.0, 0.1, 4)], precision=prec) as s:
        a = rng.standard_normal(s.box()).astype(np.float32).astype(np.float64)
        for c in (pic.EX, pic.JZ):
            s.pic_set_field(c, a)
            assert np.array_equal(s.pic_fields(c), a), c
        top = n[-1] - 1  # (a particle at rest on the last row's node)
        x = [[0.3] if d < len(n) - 1 else [top * 0.1] for d in range(len(n))] + [None] * (3 - len(n))
        s.pic_load_particles(0, *x, [0.0], [0.0], [0.0])
        rho = s.pic_fields(pic.RHO)
        assert abs(rho.sum() + 0.1) <= 1e-12 and np.argmin(rho.reshape(n[-1], -1).sum(1)) == top
