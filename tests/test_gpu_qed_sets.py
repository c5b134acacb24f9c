"""The QED species of a step side by side: pushes of several species in one
launch, their flags summed in one launch and their children made in one, with
more lepton species than a launch of pushes has places.  The same run with
per-phase timing on launches every species' push on its own: same bits.  The
weight is too small for self-fields to change a bit."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests import qed_setup as Q

pytestmark = pytest.mark.gpu

COUNTS = (300, 1, 0, 5000, 257)  # leptons per emitting species
N = (16, 12, 9)


def _sim(dim, prec, sort_interval):
    # electrons and positrons (the pairs' species) first, then other emitters, photons last
    spec = [(-1.0 if i != 1 else 1.0, 1.0, 1e-40, 30000, 0, 1) for i in range(len(COUNTS))]
    spec.append((0.0, 0.0, 1e-40, 200000, 1, 0))
    s = pic.pic_create(dim, N[:dim], (1.0,) * dim, Q.DT, spec, seed=Q.SEED, sort_interval=sort_interval, precision=prec,
                       tile=(8, 8, 8)[:dim])
    s.pic_set_qed(photon_sp=len(COUNTS), electron_sp=0, positron_sp=1, lambda_r_m=Q.LAMBDA)
    s.pic_set_field(pic.BZ, np.full(s.box(), Q.B0))
    rng = np.random.default_rng(11 + dim)
    for i, n in enumerate(COUNTS):
        if n == 0:
            continue
        x = [rng.uniform(0.0, N[d], n) if d < dim else None for d in range(3)]
        u = np.sqrt(Q.GAMMA0 ** 2 - 1.0) * (1.0 + 0.1 * i)  # a species' photons are told by their energies
        ang = rng.uniform(0.0, 2.0 * np.pi, n)
        s.pic_load_particles(i, *x, u * np.cos(ang), u * np.sin(ang), np.zeros(n))
    return s


def _state(s):
    out = []
    for i in range(len(COUNTS) + 1):
        p = s.pic_get_particles(i)
        ids, tau = s.pic_get_qed_state(i)
        out.append({**p, "ids": ids, "tau": tau})
    return out


@pytest.mark.parametrize("dim,prec,sort", [(1, pic.FP32_CELLOFF, 0), (2, pic.FP32_CELLOFF, 0), (3, pic.FP32_CELLOFF, 0),
                                           (2, pic.FP32_CELLOFF, 4), (1, pic.FP64_PLAIN, 0)])
def test_species_side_by_side_give_the_same_bits(dim, prec, sort):
    a, b = _sim(dim, prec, sort), _sim(dim, prec, sort)
    b.pic_profile(True)
    for _ in range(12):
        a.pic_step(1)
        b.pic_step(1)
    sa, sb = _state(a), _state(b)
    assert len(sa[-1]["ids"]) > 500 and len(sa[1]["ids"]) > 1  # photons, pairs
    for i, (p, q) in enumerate(zip(sa, sb)):
        for k in p:
            assert np.array_equal(p[k], q[k]), (i, k)
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [pic.FP32_CELLOFF, pic.FP64_PLAIN])
def test_children_follow_species_and_parents(prec):
    """one step: the photons are in species order, within one in the parents'
    order (each at its parent's position)"""
    s = _sim(1, prec, 0)
    s.pic_step(1)
    ph, x = s.pic_get_particles(len(COUNTS))["x"], []
    for i in range(len(COUNTS)):
        p = s.pic_get_particles(i)
        g0 = np.sqrt(Q.GAMMA0 ** 2 - 1.0) * (1.0 + 0.1 * i)
        emitted = np.sqrt(p["ux"] ** 2 + p["uy"] ** 2 + p["uz"] ** 2) < g0 * (1.0 - 1e-5)  # recoiled
        x.append(p["x"][emitted])
    x = np.concatenate(x)
    assert len(x) > 50
    # (an emission of less than 1e-5 of the energy may be missing from the list: a subsequence)
    at = 0
    for v in x:
        while at < len(ph) and ph[at] != v:
            at += 1
        assert at < len(ph), v
        at += 1
    assert len(ph) - len(x) <= 0.05 * len(ph) + 2
    s.close()
