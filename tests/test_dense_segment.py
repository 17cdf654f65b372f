"""FP32 segments of small dense instances in one launch (k_dense_seg): the same
bits as one launch per step, at the edges of its sizes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gda():
    import torch

    import __graft_entry__
    assert torch.cuda.is_available()
    __graft_entry__.ensure_built()
    from paper_1807_00699_gb300 import gda as mod
    return mod


@pytest.mark.parametrize("integ", ["euler", "rk4"])
@pytest.mark.parametrize("model,n,R,kw", [
    ("ising", 1, 1, {}),
    ("xy", 2, 3, dict(noise_D=0.2, noise_decay=1)),
    ("ising", 20, 64, dict(noise_D=0.2, noise_decay=1)),
    ("xy", 33, 65, dict(q=3, hq=0.05)),
    ("ising", 64, 611, dict(noise_D=0.1)),          # four columns per CTA
    ("xy", 65, 300, dict(noise_D=0.2, noise_decay=1)),
    ("ising", 130, 7, {}),
    ("xy", 200, 256, dict(noise_D=0.2, noise_decay=1)),
    ("ising", 233, 33, dict(noise_D=0.2, noise_decay=1)),  # the largest J0 in shared memory
    ("ising", 236, 33, {}),                                # no longer fits: a launch per step
])
def test_segment_equals_per_step(gda, integ, model, n, R, kw):
    J, g = synth.xy_gaussian(n, n + 1)
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    p = dict(integ=gda.RK4 if integ == "rk4" else gda.EULER, dt=0.02, eps=0.1, beta0=0.5, eps_hat=0.2, init_amp=0.1,
             seed=5, **kw)
    s.run(gda.default_params(energy_every=1, **p), R, 30)  # segments of one step: a launch per step
    a = s.get_state()
    s.run(gda.default_params(energy_every=13, **p), R, 30)  # 13 + 13 + 4
    b = s.get_state()
    s.run(gda.default_params(**p), R, 17)
    s.run(gda.default_params(**{**p, "init_mode": 2}), R, 13)
    c = s.get_state()
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
    s.close()
