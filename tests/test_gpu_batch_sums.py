"""Loss and dJ/dtheta of a batch equal those of its instances run alone, bit for bit, where an
instance is more blocks of particles than the batch leaves it in one wave (64^3 particles)."""
import numpy as np
import pytest

from paper_2211_09815_gb300 import inputs
from test_gpu_pm import _gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nm", [64, 128])
@pytest.mark.parametrize("precision", [0, 1])
def test_batch_sums_equal_single_runs(nm, precision):
    cfg = dict(box=100.0, n_mesh=nm, n_ptcl=64, n_steps=1)
    theta = np.array([inputs.THETA_FIDUCIAL, (2.3e-9, 0.95, 0.28, 0.049, 0.68), (1.9e-9, 0.98, 0.33, 0.049, 0.68)])
    tgt = np.zeros((3, nm ** 3))
    both = _gpu_run(cfg, precision, batch=3, theta=theta, target=tgt)
    for b in range(3):
        one = _gpu_run(cfg, precision, seed=1 + b, theta=theta[b], target=tgt[b:b + 1])
        for key in ("delta", "loss", "grad_omega", "grad_theta"):
            assert np.array_equal(one[key][0], both[key][b]), key
