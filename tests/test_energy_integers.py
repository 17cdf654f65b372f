"""Energies of integer couplings are exact integers in the kernel for small
instances (its size, magnitude and restart limits, and just past them) and in
the digit products, fields included where the sum can hold them."""
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


@pytest.mark.parametrize("n,R,scale", [(1, 1, 1), (2, 3, 1), (31, 5, 17), (32, 600, 1), (100, 256, 100), (200, 839, 1),
                                       (200, 838, 1), (256, 4, 256), (256, 4, 257), (256, 1, 1), (257, 9, 1),
                                       (500, 130, 40000), (1100, 5, 2 ** 31)])
@pytest.mark.parametrize("field", [False, True])
def test_integer_energies_are_exact(gda, n, R, scale, field):
    # magnitudes up to `scale`, one entry at it; multiples of 1/4 as fields
    u = synth.uniform01(n, n * n).reshape(n, n)
    J = np.rint((2.0 * u - 1.0) * scale)
    J = np.triu(J) + np.triu(J, 1).T
    J[0, 0] = scale
    g = np.rint(8.0 * synth.uniform01(n + 1, n) - 4.0) / 4.0 if field else None
    psi = synth.initial_amplitudes(n, R, n + R, 1.0, False).astype(np.float32)
    s = gda.Solver(J, g, gda.ISING)
    s.set_state(psi)
    E = s.energy()
    sp = np.where(psi >= 0, 1, -1).astype(np.int64)
    ref = -((sp @ J.astype(np.int64)) * sp).sum(1)
    ref = ref + (sp * g).sum(1) if field else ref.astype(np.float64)
    assert np.array_equal(E, ref)
    Eb, rb, _ = s.best()
    assert rb == int(np.argmin(ref)) and Eb == ref[rb]
    s.close()
