"""AUTO's choice between a segment in one launch and a launch per step (FP32 and
sparse paths): few columns of a large sparse instance and many columns of a
dense one keep a launch per step; either way the bits are PER_STEP's, in every
form of the sparse segment kernel (one to four tiles per group)."""
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


def ring(n, deg):
    J, i = np.zeros((n, n)), np.arange(n)
    for k in range(1, deg // 2 + 1):
        w = synth.normal(n + k, n)
        J[i, (i + 7 * k) % n] = w
        J[(i + 7 * k) % n, i] = w
    return J


@pytest.mark.parametrize("model,n,R,deg,segment", [
    ("ising", 4100, 300, 3, True), ("xy", 4100, 150, 8, True),      # two tiles per group
    ("ising", 7200, 300, 3, True), ("xy", 8210, 150, 8, True),      # two and three, two columns per CTA
    ("ising", 12418, 300, 8, True), ("xy", 12418, 150, 8, True),    # four
    ("xy", 13000, 150, 3, True),
    ("ising", 12418, 4, 8, False), ("xy", 8210, 4, 8, False), ("ising", 14000, 32, 3, False),
    ("xy", 233, 1024, 0, False), ("xy", 233, 256, 0, True),         # dense
])
def test_auto_picks_the_faster_form(gda, model, n, R, deg, segment):
    J = synth.xy_gaussian(n, n)[0] if deg == 0 else synth.sparse_3regular(n, n)[0] if deg == 3 else ring(n, deg)
    s = gda.Solver(J, 0.1 * synth.normal(n + 5, n), gda.XY if model == "xy" else gda.ISING)
    out, launches = [], []
    for sched in (gda.PER_STEP, gda.AUTO):
        p = gda.default_params(dt=0.01, eps=0.1, beta0=0.5, eps_hat=0.2, init_amp=0.1, seed=5, noise_D=0.2, noise_decay=1,
                               prec=gda.SPARSE if deg else gda.FP32, schedule=sched)
        before = s.kernel_launches()
        s.run(p, R, 60)
        launches.append(s.kernel_launches() - before)
        out.append(s.get_state())
    assert launches[0] >= 60 and (launches[1] < 60) == segment
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    s.close()
