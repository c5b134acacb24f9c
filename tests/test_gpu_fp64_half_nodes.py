"""The FP64 push of particles at the speed of light on a step of almost dx, from
half node to half node."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_light_speed_from_half_node_to_half_node(order, sign):
    """dt one unit below dx: positions k, k + 1/2 after the half drift and
    k + 3/2 after the step, which is one node further, not two; the summed
    current is q w times the speed of light"""
    n, w = 16, 0.1
    x = np.arange(2.0, 14.0)
    u = np.full(x.size, sign * 1e9)
    z = np.zeros(x.size)
    with pic.pic_create(1, (n,), (1.0,), np.nextafter(1.0, 0.0), [(-1.0, 1.0, w, x.size)], precision=pic.FP64_PLAIN,
                        order=order) as s:
        s.pic_load_particles(0, x, None, None, u, z, z)
        s.pic_step(1)
        assert abs(s.pic_fields(pic.JX).sum() + sign * w * x.size) <= 1e-12
