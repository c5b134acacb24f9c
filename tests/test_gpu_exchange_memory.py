"""Field components to and from the host without device memory to spare."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu
PRECS = [pic.FP32_CELLOFF, pic.FP64_PLAIN]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n,bc", [((19,), (1,)), ((20, 13), (1, 0)), ((9, 8, 11), (0, 1, 1))])
def test_read_backs_take_no_device_memory(n, bc, prec):
    """an allocator that has nothing left after pic_create"""
    class Spent(pic.TorchAllocator):
        spent = False

        def _do_alloc(self, ctx, nbytes, stream):
            return None if self.spent else super()._do_alloc(ctx, nbytes, stream)

    rng = np.random.default_rng(9)
    A = Spent()
    s = pic.pic_create(len(n), n, (0.1,) * len(n), 0.05, [(-1.0, 1.0, 0.1, 200)], bc=bc, precision=prec, allocator=A)
    x = [rng.uniform(0.0, n[d] * 0.1, 200) if d < len(n) else None for d in range(3)]
    s.pic_load_particles(0, *x, np.zeros(200), np.zeros(200), np.zeros(200))
    rho = s.pic_fields(pic.RHO)
    a = rng.standard_normal(s.box()).astype(np.float32).astype(np.float64)
    A.spent = True
    for c in range(9):
        s.pic_set_field(c, a + c)
        assert np.array_equal(s.pic_fields(c), (a + c).astype(np.float32 if prec == pic.FP32_CELLOFF else np.float64)), c
    # (the deposits' order is free: the same sums but for their rounding)
    assert np.max(np.abs(s.pic_fields(pic.RHO) - rho)) <= 1e-13
    s.close()
