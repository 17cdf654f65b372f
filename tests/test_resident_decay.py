"""Resident kernel under noise decay: every form waits for the density sums of
all row blocks of its column block (a lane per flag, more row blocks than lanes
included), with the bits of one launch per step."""
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


@pytest.mark.parametrize("model,n,R", [
    ("ising", 130, 8000), ("xy", 256, 3100), ("ising", 256, 9700),  # one block of 128 columns up to N = 256
    ("ising", 257, 6300), ("xy", 576, 1900),                        # two blocks of 64
    ("xy", 1500, 300), ("ising", 4200, 70),                         # 12 and 33 row blocks
])
def test_decay_matches_per_step(gda, model, n, R):
    J, g = synth.xy_gaussian(n, n)
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    p = dict(dt=0.02, eps=0.1, beta0=0.4, eps_hat=0.2, init_amp=0.1, seed=7, noise_D=0.3, noise_decay=1, prec=gda.BF16)
    out = []
    for sched in (gda.PER_STEP, gda.RESIDENT):
        s.run(gda.default_params(schedule=sched, **p), R, 12)
        out.append(s.get_state())
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    s.close()
