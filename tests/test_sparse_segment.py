"""Sparse Euler segments in one launch (k_sparse_euler_seg): the same bits as
one launch per step, at the edges of its tile and column counts."""
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


def graph(n, deg):
    if deg == 3:
        return synth.sparse_3regular(n, n)[0]
    J = np.zeros((n, n))
    for k in range(1, deg // 2 + 1):  # a ring of `deg` neighbours, and a hub-free remainder
        w = synth.normal(n + k, n)
        i = np.arange(n)
        J[i, (i + 7 * k) % n] = w
        J[(i + 7 * k) % n, i] = w
    np.fill_diagonal(J, 0.0)
    return J


@pytest.mark.parametrize("model,n,R,deg,kw", [
    ("ising", 46, 3, 3, {}),
    ("xy", 64, 5, 3, dict(noise_D=0.2, noise_decay=1)),
    ("ising", 1030, 611, 3, dict(noise_D=0.1)),
    ("xy", 1030, 77, 8, dict(q=3, hq=0.05)),
    ("ising", 4100, 150, 3, dict(noise_D=0.2, noise_decay=1)),   # two tiles per group, two columns
    ("ising", 6000, 611, 3, dict(noise_D=0.2, noise_decay=1)),   # two tiles per group, four columns
    ("xy", 6000, 130, 8, {}),
    ("ising", 7200, 5, 3, dict(noise_D=0.1)),                    # four columns no longer fit
    ("xy", 8210, 3, 3, dict(noise_D=0.2, noise_decay=1)),        # three tiles per group
    ("ising", 12418, 7, 8, {}),                                  # four tiles per group
])
def test_segment_equals_per_step(gda, model, n, R, deg, kw):
    J = graph(n, deg)
    g = 0.1 * synth.normal(n + 5, n)
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    p = dict(prec=gda.SPARSE, dt=0.01, eps=0.1, beta0=0.5, eps_hat=0.2, init_amp=0.1, seed=5, **kw)
    s.run(gda.default_params(energy_every=1, **p), R, 12)  # segments of one step: a launch per step
    a = s.get_state()
    s.run(gda.default_params(energy_every=5, **p), R, 12)  # 5 + 5 + 2
    b = s.get_state()
    s.run(gda.default_params(**p), R, 7)
    s.run(gda.default_params(**{**p, "init_mode": 2}), R, 5)
    c = s.get_state()
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
    s.close()
