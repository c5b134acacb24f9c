"""Training with one batch after work on a larger one in the same simulation:
the network is that of a fresh simulation, bit for bit."""
import numpy as np
import pytest

from paper_2104_00642_gb300 import pic
from tests import qed_setup as Q

pytestmark = pytest.mark.gpu


def _sim():
    s = pic.pic_create(1, (16,), (1.0,), Q.DT, Q.species_spec(cap=64), seed=Q.SEED)
    s.pic_set_qed(photon_sp=2, electron_sp=0, positron_sp=1, lambda_r_m=Q.LAMBDA, mode=pic.QED_TABLE)
    return s


@pytest.mark.parametrize("process", [pic.QED_EMISSION, pic.QED_PAIR])
@pytest.mark.parametrize("batch", [128, 2048, 4224])
def test_batch_after_a_larger_one_trains_as_in_a_fresh_simulation(process, batch):
    a, b = _sim(), _sim()
    a.pic_mlp_train(process, iterations=3, batch=8192, seed=5)
    x = np.zeros((32 * 300, 2), dtype=np.float32)
    a.pic_mlp_grad(process, x, x)
    ra = a.pic_mlp_train(process, iterations=7, batch=batch, seed=9)
    rb = b.pic_mlp_train(process, iterations=7, batch=batch, seed=9)
    assert np.array_equal(a.pic_mlp_get(process)[0], b.pic_mlp_get(process)[0])
    assert ra["loss"] == rb["loss"]
    a.close()
    b.close()
