"""The resident kernel's forms (one 128-column block, one or two 64-column
blocks per CTA, kept and streamed coupling tiles): bits of per-step launches."""
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


@pytest.mark.parametrize("model,n,R,kw", [
    ("ising", 1, 1, {}),
    ("xy", 576, 33, dict(noise_D=0.2, noise_decay=1)),     # one 64-column block, tiles kept (9 K-blocks)
    ("ising", 577, 65, dict(noise_D=0.1)),                 # the same, streamed tiles
    ("ising", 300, 3300, dict(noise_D=0.2, noise_decay=1)),  # two blocks per CTA, the last CTA with one
    ("xy", 257, 1650, {}),                                 # two blocks per CTA, ragged
    ("ising", 1000, 1300, dict(noise_D=0.2, noise_decay=1)),  # one 128-column block
    ("xy", 2000, 450, {}),
])
def test_resident_equals_per_step(gda, model, n, R, kw):
    J, g = synth.xy_gaussian(n, n)
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    p = dict(prec=gda.BF16, dt=0.05, eps=0.1, beta0=0.5, eps_hat=0.2, init_amp=0.1, seed=3, energy_every=11, **kw)
    s.run(gda.default_params(schedule=gda.RESIDENT, **p), R, 25)
    a, ta = s.get_state(), s.trace()
    s.run(gda.default_params(schedule=gda.PER_STEP, **p), R, 25)
    for x, y in zip(a, s.get_state()):
        assert np.array_equal(x, y)
    for x, y in zip(ta, s.trace()):
        assert np.array_equal(x, y)
    s.close()
