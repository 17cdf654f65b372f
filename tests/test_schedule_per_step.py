"""GDA_SCHEDULE_PER_STEP launches every step by itself in the FP32 and sparse
paths too, and gives the bits of AUTO's segments."""
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


@pytest.mark.parametrize("every", [0, 7])
@pytest.mark.parametrize("model,n,prec,integ", [("ising", 20, "FP32", "EULER"), ("xy", 130, "FP32", "RK4"),
                                                ("ising", 800, "SPARSE", "EULER"), ("xy", 130, "SPARSE", "EULER")])
def test_per_step_is_honoured(gda, model, n, prec, integ, every):
    J = synth.sparse_3regular(n, 3)[0]
    steps, out = 50, {}
    for sched in (gda.PER_STEP, gda.AUTO):
        s = gda.Solver(J, None, gda.XY if model == "xy" else gda.ISING)
        p = gda.default_params(dt=0.005, eps=0.1, noise_D=0.1, noise_decay=1, seed=2, init_amp=0.1, energy_every=every,
                               prec=getattr(gda, prec), integ=getattr(gda, integ), schedule=sched)
        s.run(p, 9, steps)
        s.sync()
        before = s.kernel_launches()
        s.run(p, 9, steps)
        s.sync()
        out[sched] = (s.kernel_launches() - before, *s.get_state(), *s.trace())
        s.close()
    a, b = out[gda.PER_STEP], out[gda.AUTO]
    assert a[0] >= steps * (4 if integ == "RK4" else 1) > b[0]
    for x, y in zip(a[1:], b[1:]):
        assert np.array_equal(x, y)
