"""Where a species has few particles an item the one-thread push takes the step
instead of the tiled one: on both sides of that line, with all particles in a few
tiles of a large grid, with tiles as full as they get, and across a save and a
restore between two sorts.  Against the FP64 oracle."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic, workloads as W
from tests.helpers import oracle_from_workload, random_state, window_scale

pytestmark = pytest.mark.gpu
TOL = 1e-5
A, P = W.ABSORB, W.PERIODIC
# per tile: the line, its neighbours, next to nothing, and far beyond
# (and a grid of too few tiles to ask)
GRIDS = [((32, 32, 32), 2, (4, 4, 4), 34), ((33, 31, 30), 2, (4, 4, 4), 34), ((640, 624), 2, (16, 16, 1), 64),
         ((320, 312), 2, (8, 8, 1), 46), ((640, 624), 4, (16, 16, 1), 60),
         ((320, 312), 4, (8, 8, 1), 50), ((16, 16, 12), 2, (4, 4, 4), 34)]


def _workload(n, per_tile, tile, lie, bc, seed):
    dim = len(n)
    dx = (0.1, 0.12, 0.11)[:dim]
    dt = 0.9 / np.sqrt(sum(1.0 / d ** 2 for d in dx))
    tiles = int(np.prod([-(-m // t) for m, t in zip(n, tile)]))
    w, F = random_state(dim, n, dx, dt, 1, seed=seed, umax=0.9, bc=bc)
    rng = np.random.default_rng(seed)
    s = w.species[0]
    count = max(1, per_tile * tiles)
    for d, k in enumerate(("x", "y", "z")):
        if d >= dim:
            setattr(s, k, np.zeros(count))
        elif lie == "even":  # as many in every tile
            t = np.arange(count) % tiles
            for a in range(d):
                t = t // -(-n[a] // tile[a])
            lo = (t % -(-n[d] // tile[d])) * tile[d]
            setattr(s, k, (lo + rng.random(count) * np.minimum(tile[d], n[d] - lo)) * dx[d])
        else:  # in one cell
            setattr(s, k, (n[d] // 2 + rng.random(count)) * dx[d])
    for k in ("ux", "uy", "uz"):
        setattr(s, k, rng.uniform(-0.5, 0.5, count))
    s.capacity = count
    return w, F


def _compare(sim, o, w, order, steps):
    pg, po = sim.pic_get_particles(0), o.particles(0)
    assert (pg["alive"] != po["alive"]).sum() == 0
    live = po["alive"] != 0
    umag = np.sqrt(po["ux"] ** 2 + po["uy"] ** 2 + po["uz"] ** 2)
    for d, k in enumerate(("x", "y", "z")[: w.dim]):
        L = w.n[d] * w.dx[d]
        e = pg[k] - po[k]
        assert np.max(np.abs(e - L * np.round(e / L))[live]) <= 10 * steps * TOL * w.dx[d]
    for k in ("ux", "uy", "uz"):
        assert np.all((np.abs(pg[k] - po[k]) <= steps * (TOL * umag + 1e-6))[live])
    for c, ax in ((pic.JX, 0), (pic.JY, 1), (pic.JZ, 2)):
        scale = window_scale(po, w, w.dim, ax, reach=(3 if order == 2 else 4) + steps)
        assert np.all(np.abs(sim.pic_fields(c) - o.field(c)) <= (20 * steps - 19) * TOL * scale.max() + 1e-30), c


@pytest.mark.parametrize("n,order,tile,line", GRIDS)
@pytest.mark.parametrize("lie,per_tile", [("even", 0), ("even", 3), ("even", -1), ("even", 1), ("heap", 3), ("heap", -1)])
def test_both_sides_of_the_line(n, order, tile, line, lie, per_tile):
    """per_tile 0: one particle; -1: the line itself; 1: one more a tile"""
    many = {0: 0, 3: 3, -1: line, 1: line + 1}[per_tile]
    w, F = _workload(n, many, tile, lie, (P,) * len(n), 870 + many)
    sim = pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=4, tile=tile, order=order)
    o = oracle_from_workload(w, sort_interval=4, tile=tile)
    o.set_order(order)
    for c in range(9):
        sim.pic_set_field(c, F[c])
        o.set_field(c, F[c])
    for steps in (1, 2):
        sim.pic_step(1)
        o.step(1)
        _compare(sim, o, w, order, steps)
    sim.close()


@pytest.mark.parametrize("lie", ["even", "heap"])
def test_restore_between_sorts(tmp_path, lie):
    """a sparse and a dense species saved after a sort: the restored run pushes
    every particle, as the one that went on"""
    n, tile = (32, 32, 32), (4, 4, 4)
    w, F = _workload(n, 12, tile, lie, (P,) * 3, 881)
    sims = [pic.from_workload(w, precision=pic.FP32_CELLOFF, sort_interval=50, tile=tile) for _ in range(2)]
    for c in range(9):
        sims[0].pic_set_field(c, F[c])
    sims[0].pic_step(2)
    sims[0].pic_save(str(tmp_path / "s"))
    sims[1].pic_restore(str(tmp_path / "s"))
    for s in sims:
        s.pic_step(3)
    a, b = sims[0].pic_get_particles(0), sims[1].pic_get_particles(0)
    for k in a:
        assert np.max(np.abs(a[k].astype(float) - b[k].astype(float))) <= 1e-4, k
    for s in sims:
        s.close()
