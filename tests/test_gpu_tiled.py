"""Tiled pushes (shared-memory field and current boxes) where their items,
windows and boxes end: shape orders 2 and 4 in 2D, grids whose sizes are not
multiples of the tile, tiles with more particles than one work item holds,
one-particle items, absorbing faces.  Each against the FP64 oracle."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic, workloads as W
from tests.helpers import oracle_from_workload, random_state, window_scale

pytestmark = pytest.mark.gpu

# FP32 form: relative to |u| for momenta, to the sum of |contributions| of a
# node for currents, to 10 of these in cells for positions
TOL = 1e-5
A, P = W.ABSORB, W.PERIODIC


def _crowd(w, frac, cells, seed):
    """a share of the particles moved into the lowest `cells` cells per axis"""
    rng = np.random.default_rng(seed)
    s = w.species[0]
    m = rng.random(s.n) < frac
    for d, x in enumerate((s.x, s.y, s.z)[: w.dim]):
        x[m] = rng.random(int(m.sum())) * (cells * w.dx[d])


def _one_step(w, F, order, tile):
    sim = pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=1, tile=tile, order=order)
    o = oracle_from_workload(w, sort_interval=1, tile=tile)
    o.set_order(order)
    for c in range(9):
        sim.pic_set_field(c, F[c])
        o.set_field(c, F[c])
    sim.pic_step(1)
    o.step(1)
    pg, po = sim.pic_get_particles(0), o.particles(0)
    assert np.array_equal(pg["alive"], po["alive"])
    live = po["alive"] != 0
    for d, k in enumerate(("x", "y", "z")[: w.dim]):
        assert np.max(np.abs(pg[k] - po[k])[live]) <= 10 * TOL * w.dx[d]
    umag = np.sqrt(po["ux"] ** 2 + po["uy"] ** 2 + po["uz"] ** 2)
    for k in ("ux", "uy", "uz"):
        assert np.all((np.abs(pg[k] - po[k]) <= TOL * umag + 1e-7)[live])
    for c, ax in ((pic.JX, 0), (pic.JY, 1), (pic.JZ, 2)):
        scale = window_scale(po, w, w.dim, ax, reach=3 if order == 2 else 4)
        assert np.all(np.abs(sim.pic_fields(c) - o.field(c)) <= TOL * scale + 1e-30), c
    sim.close()


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n,nppc,crowd,bc", [((40, 21), 4, 0.7, (P, P)),   # a tile of more than 2 x 1024 particles
                                             ((37, 33), 1, 0.0, (A, P)),   # odd sizes, an absorbing axis, few per item
                                             ((16, 16), 0, 0.0, (P, P))])  # one particle
def test_tile2d_order4_one_step_matches_oracle(tile, n, nppc, crowd, bc):
    dx = (0.1, 0.12)
    dt = 0.9 / np.sqrt(sum(1.0 / d ** 2 for d in dx))
    w, F = random_state(2, n, dx, dt, max(nppc, 1), seed=640 + tile, umax=0.9, bc=bc)
    if nppc == 0:
        s = w.species[0]
        for k in ("x", "y", "z", "ux", "uy", "uz"):
            setattr(s, k, getattr(s, k)[:1].copy())
    _crowd(w, crowd, 3, 7)
    _one_step(w, F, 4, (tile, tile, 1))


@pytest.mark.parametrize("n,nppc,crowd,bc", [((13, 10, 9), 3, 0.0, (P, P, P)),    # ragged in every axis
                                             ((16, 12, 8), 2, 0.6, (P, P, P)),    # a tile of more than 640 particles
                                             ((11, 14, 17), 1, 0.0, (A, P, A)),   # absorbing faces on ragged tiles
                                             ((28, 9, 8), 0, 0.0, (P, P, P))])    # one particle (pitch = padded row)
def test_tile3d_ragged_one_step_matches_oracle(n, nppc, crowd, bc):
    dx = (0.1, 0.12, 0.11)
    dt = 0.9 / np.sqrt(sum(1.0 / d ** 2 for d in dx))
    w, F = random_state(3, n, dx, dt, max(nppc, 1), seed=650 + n[0], umax=0.9, bc=bc)
    if nppc == 0:
        s = w.species[0]
        for k in ("x", "y", "z", "ux", "uy", "uz"):
            setattr(s, k, getattr(s, k)[-1:].copy())
    _crowd(w, crowd, 3, 9)
    _one_step(w, F, 2, (4, 4, 4))


@pytest.mark.parametrize("n", [1, 31, 33, 4095, 4096, 4097, 9001])
def test_sort_is_numpys_stable_sort(n):
    """particles at rest on a ragged 2D grid, sorted at step 0 (blocks of 4096
    keys, 512 a warp): numpy's stable argsort by (tile, cell in the tile)"""
    rng = np.random.default_rng(n)
    nx, ny = 37, 22
    x, y = rng.random(n) * nx, rng.random(n) * ny
    z, tag = np.zeros(n), np.arange(n) * 1e-9
    with pic.pic_create(2, (nx, ny), (1.0, 1.0), 0.5, [(-1.0, 1.0, 1e-20, n + 5)], sort_interval=1, tile=(8, 8)) as s:
        s.pic_load_particles(0, x, y, None, z, z, tag)
        s.pic_step(1)
        p = s.pic_get_particles(0)
    cx, cy = x.astype(int), y.astype(int)
    key = ((cy // 8) * ((nx + 7) // 8) + cx // 8) * 64 + (cy % 8) * 8 + cx % 8
    assert np.array_equal(p["uz"], tag.astype(np.float32).astype(np.float64)[np.argsort(key, kind="stable")])
