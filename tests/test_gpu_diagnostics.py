"""FP64 diagnostics against plain FP64 (numpy, long double where it cancels):
kinetic energies over the whole range of momenta, photon energies, the charge
density of single particles, and the exchange of field components on odd
grids."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic

pytestmark = pytest.mark.gpu
PRECS = [pic.FP32_CELLOFF, pic.FP64_PLAIN]


def _w2(d):
    return np.array([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2])


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [1, 255, 4097])
def test_kinetic_energy_over_all_magnitudes(prec, n):
    """momenta from 1e-12 to 1e17 (beyond 2^48.5 the FP32-seeded roots hand
    over), zeros among them.  Every term is good to a few units in the last
    place and the terms are positive, so the sum is good to 1e-13"""
    rng = np.random.default_rng(11)
    u = 10.0 ** rng.uniform(-12, 17, (3, n)) * rng.choice([-1.0, 1.0], (3, n))
    u[:, ::7] = 0.0
    r = np.float32 if prec == pic.FP32_CELLOFF else np.float64
    spec = [(-1.0, 2.0, 0.25, n), (0.0, 0.0, 0.5, n, pic.KIND_PHOTON, 0)]
    with pic.pic_create(1, (16,), (1.0,), 0.5, spec, precision=prec) as s:
        for i in range(2):
            s.pic_load_particles(i, rng.random(n) * 16.0, None, None, *u)
        d = s.pic_diagnostics()
    ul = u.astype(r).astype(np.longdouble)
    uu = (ul ** 2).sum(0)
    ref = 0.25 * 2.0 * (uu / (np.sqrt(1.0 + uu) + 1.0)).sum(), 0.5 * np.sqrt(uu).sum()
    for got, want in zip(d["U_kin"], ref):
        assert abs(got - float(want)) <= 1e-13 * float(want) + 1e-300
    assert d["n_alive"] == [n, n]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("u", [0.0, 1e-9, 0.3, 50.0, 1e16])
def test_charge_density_of_one_particle(prec, u):
    """W_2 at x -/+ (dt/2) v, half each, in 1D; at the node, the half node and
    near a cell face"""
    n, dx, dt, w = 16, 0.1, 0.09, 0.7
    r = np.float32 if prec == pic.FP32_CELLOFF else np.float64
    for X in (3.0, 7.25, 5.5, 9.999, 15.6):
        with pic.pic_create(1, (n,), (dx,), dt, [(-1.0, 1.0, w, 1)], precision=prec) as s:
            s.pic_load_particles(0, [X * dx], None, None, [u], [0.0], [0.0])
            rho = s.pic_fields(pic.RHO).ravel()
        ul = float(r(u))
        c = np.floor(X * dx / dx)
        x0 = c + float(r(X * dx / dx - c)) if prec == pic.FP32_CELLOFF else X * dx / dx
        ref = np.zeros(n)
        for side in (-0.5, 0.5):
            x = x0 + side * dt * ul / np.sqrt(1.0 + ul * ul) / dx
            ic = int(np.floor(x + 0.5))
            for a, v in zip((-1, 0, 1), _w2(x - ic)):
                ref[(ic + a) % n] += -0.5 * w * v
        # cell positions round at 16 units of 2^-53; W_2 has slope at most 1
        assert np.max(np.abs(rho - ref)) <= 1e-14


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n,bc", [((37,), (0,)), ((41,), (1,)), ((20, 13), (1, 0)), ((9, 8, 11), (0, 1, 1)), ((64, 33, 8), (0, 0, 0))])
def test_field_exchange_round_trip(prec, n, bc):
    dim = len(n)
    rng = np.random.default_rng(5)
    with pic.pic_create(dim, n, (0.1,) * dim, 0.05, [], bc=bc, precision=prec) as s:
        for c in range(9):
            a = rng.standard_normal(s.box())
            s.pic_set_field(c, a)
            want = a.astype(np.float32).astype(np.float64) if prec == pic.FP32_CELLOFF else a
            assert np.array_equal(s.pic_fields(c), want), c
