"""gda_run with init_mode 2 recorded into a CUDA graph: replays of an even number
of noise-free steps continue the state, whatever the tracking segments, in
every kernel that runs many steps per launch."""
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


@pytest.mark.parametrize("every", [0, 5, 20])
@pytest.mark.parametrize("model,n,R,kw", [
    ("ising", 40, 9, dict(prec="FP32")),                      # dense segments
    ("xy", 40, 9, dict(prec="FP32", integ="RK4")),
    ("xy", 500, 9, dict(prec="FP32")),                        # a launch per step
    ("ising", 500, 9, dict(prec="SPARSE")),                   # sparse segments
    ("xy", 500, 9, dict(prec="SPARSE", integ="RK4")),
    ("xy", 300, 9, dict(prec="BF16", schedule="RESIDENT")),
    ("ising", 300, 9, dict(prec="BF16", schedule="STREAM")),
])
def test_replays_continue_the_state(gda, model, n, R, kw, every):
    import torch
    J = synth.sparse_3regular(n, 3)[0]
    kw = {k: getattr(gda, v) for k, v in kw.items()}
    p = dict(dt=0.005, eps=0.2, beta0=0.4, eps_hat=0.3, seed=3, init_amp=0.2, energy_every=every, **kw)
    st = torch.cuda.Stream()
    out = []
    for recorded in (False, True):
        s = gda.Solver(J, None, gda.XY if model == "xy" else gda.ISING, stream=st)
        s.run(gda.default_params(**p), R, 20)  # every buffer exists
        s.sync()
        q = gda.default_params(**{**p, "init_mode": 2})
        if recorded:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.stream(st):
                g.capture_begin()
                s.run(q, R, 20)
                g.capture_end()
        for _ in range(3):
            if recorded:
                with torch.cuda.stream(st):
                    g.replay()
            else:
                s.run(q, R, 20)
        s.sync()
        out.append([*s.get_state()[:3], s.energy()])
        s.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
