"""The places of a step's children where a pair species has no particle on the
device yet while the host's bound on its count is already positive."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests import qed_setup as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [pic.FP32_CELLOFF, pic.FP64_PLAIN])
def test_first_pairs_of_an_empty_positron_species(prec):
    """electrons as many as there are pairs and as they were loaded, one
    positron for each photon gone, step by step; the same bits in every run"""
    rng = np.random.default_rng(4)
    n_ph, x, k = 9000, rng.uniform(0.0, 16.0, 9000), np.full(9000, 20.0)
    runs = []
    for _ in range(10):
        s = pic.pic_create(1, (16,), (1.0,), Q.DT, Q.species_spec(cap=20_000), seed=Q.SEED, precision=prec)
        s.pic_set_qed(photon_sp=2, electron_sp=0, positron_sp=1, lambda_r_m=Q.LAMBDA)
        s.pic_set_field(pic.BZ, np.full(s.box(), Q.B0))
        s.pic_load_particles(0, *Q.electrons())
        s.pic_load_particles(2, x, None, None, np.zeros(n_ph), k, np.zeros(n_ph))
        counts = []
        for _ in range(40):
            s.pic_step(1)
            e, p, g = (s.pic_get_particles(i) for i in range(3))
            counts.append(len(p["x"]))
            assert len(e["x"]) == Q.N_E + counts[-1] == Q.N_E + int((g["alive"] == 0).sum())
        runs.append((counts, e, p, g))
        s.close()
    assert runs[0][0][0] == 0 and runs[0][0][-1] > 0, runs[0][0]  # (the host's bound is positive from the first step on)
    for r in runs[1:]:
        assert r[0] == runs[0][0]
        for a, b in zip(r[1:], runs[0][1:]):
            for key in a:
                assert np.array_equal(a[key], b[key]), key
