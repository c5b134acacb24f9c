"""Weights round alike at the start and at the end of a particle's move: two
particles that change places in a step leave no current at all, to the bit.
(What an end point rounds off the next step's start point takes back; unlike
roundings would add up over the steps.)"""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,order,variant", [(1, (2048,), 2, pic.PUSH_AUTO), (1, (2048,), 4, pic.PUSH_AUTO),
                                                 (2, (256, 208), 2, pic.PUSH_SIMPLE), (2, (256, 208), 4, pic.PUSH_SIMPLE),
                                                 (2, (256, 208), 4, pic.PUSH_AUTO),
                                                 (3, (64, 56, 48), 2, pic.PUSH_SIMPLE), (3, (64, 56, 48), 4, pic.PUSH_SIMPLE),
                                                 (3, (66, 57, 51), 2, pic.PUSH_AUTO)])
def test_particles_that_change_places_leave_no_current(dim, n, order, variant):
    """one pair per block of 8 cells an axis; offsets and moves are multiples of
    2^-20 cells, which FP32 adds exactly, and 1/gamma is 1 (u < 2^-13)"""
    rng = np.random.default_rng(31 + dim)
    dx, unit = 0.125, 2.0 ** -20
    blocks = np.stack(np.meshgrid(*[np.arange(m // 8) for m in n], indexing="ij")).reshape(dim, -1)
    count = blocks.shape[1]
    a = 8.0 * blocks + 4.0 + rng.integers(0, 1 << 20, (dim, count)) * unit  # (cells)
    k = rng.integers(-31, 32, (dim, count))
    half = k * unit  # a half drift: dt / (2 dx) u = u / 4
    x = np.concatenate([a - half, a + 3.0 * half], axis=1) * dx
    u = np.concatenate([4.0 * half, -4.0 * half], axis=1)
    xs = [x[d] if d < dim else None for d in range(3)]
    us = [u[d] if d < dim else np.zeros(2 * count) for d in range(3)]
    with pic.pic_create(dim, n, (dx,) * dim, 0.0625, [(-1.0, 1.0, 0.1, 2 * count)], sort_interval=1, order=order,
                        push_variant=variant, tile=(4, 4, 4) if dim == 3 else (16, 16, 1)) as s:
        s.pic_load_particles(0, *xs, *us)
        s.pic_step(1)
        p = s.pic_get_particles(0)
        assert np.array_equal(np.sort(p["x"]), np.sort(((a[0] + half[0]) * dx).repeat(2)))  # (they meet half way)
        for c in (pic.JX, pic.JY, pic.JZ):
            assert not np.any(s.pic_fields(c)), c


@pytest.mark.parametrize("order", [2, 4])
def test_currents_of_many_steps_sum_to_one_move(order):
    """slow particles, one in 8 cells: the currents of 2048 steps add up to the
    difference of the weights at the two ends of the whole way (prefix sums along
    x), to the weights' rounding at the ends (2^-22) and that of a current in a
    step (2^-23 of it, 2048 moves of 2e-4 cells).  A step's start that is off its
    predecessor's end by a rounding of the offset (2^-25 and more) would add up
    to 1e-6."""
    rng = np.random.default_rng(12)
    n, dx, dt, steps, w = 1024, 0.125, 0.0625, 2048, 1e-9
    count = n // 8
    x = (8.0 * np.arange(count) + 3.0 + rng.random(count)) * dx
    u = rng.uniform(-4e-4, 4e-4, count)
    f = np.float32

    def end(p):  # offsets from cell 0 of the particles half a step on, in FP32
        c = np.floor(p["x"] / dx)
        o, un = (p["x"] / dx - c).astype(f), p["ux"].astype(f)
        ig = (f(1.0) / np.sqrt(f(1.0) + un * un, dtype=f)).astype(f)
        return c + (o.astype(float) + (f(0.25) * un).astype(f).astype(float) * ig.astype(float)).astype(f)

    def weights(X):  # W of the nodes i0 - 3 .. i0 + 4 of each particle, i0 the lower end of its way
        d = np.abs(np.arange(-3, 5)[:, None] + i0 - X)
        if order == 2:
            return np.where(d < 0.5, 0.75 - d * d, np.where(d < 1.5, 0.5 * (1.5 - d) ** 2, 0.0))
        inner = 115 / 192 - 0.625 * d ** 2 + 0.25 * d ** 4
        mid = (55 + 20 * d - 120 * d ** 2 + 80 * d ** 3 - 16 * d ** 4) / 96
        return np.where(d < 0.5, inner, np.where(d < 1.5, mid, np.where(d < 2.5, (5 - 2 * d) ** 4 / 384, 0.0)))

    with pic.pic_create(1, (n,), (dx,), dt, [(-1.0, 1.0, w, count)], order=order) as s:
        s.pic_load_particles(0, x, None, None, u, np.zeros(count), np.zeros(count))
        first, total = end(s.pic_get_particles(0)), np.zeros(n)
        for _ in range(steps):
            s.pic_step(1)
            total += s.pic_fields(pic.JX).ravel()
        last = end(s.pic_get_particles(0))
    i0 = np.floor(np.minimum(first, last))
    want = np.cumsum(weights(last) - weights(first), axis=0) * (w * dx / dt)
    got = total[(np.arange(-3, 5)[:, None] + i0).astype(int) % n]
    assert np.max(np.abs(got - want)) <= (2.0 ** -22 + steps * 2e-4 * 2.0 ** -23) * (w * dx / dt)
