"""A J that gda_load_dev refuses has replaced the instance's couplings: energies
of the kept state are those of that J (NaN where it is not finite), not of
digits made before."""
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


@pytest.mark.parametrize("kind", ["gauss", "int"])
@pytest.mark.parametrize("model,n", [("xy", 130), ("ising", 40), ("ising", 300)])
def test_energies_after_a_refused_load(gda, model, n, kind):
    import torch
    J = (synth.sk_gaussian if kind == "gauss" else synth.ising_pm1)(n, n)[0]
    s = gda.Solver(J, None, gda.XY if model == "xy" else gda.ISING)
    psi = synth.initial_amplitudes(n, 5, n, 1.0, model == "xy")
    s.set_state(psi)
    before = s.energy()
    bad = torch.tensor(2.0 * J, device="cuda")
    bad[1, 0] = 5.0  # asymmetric, finite
    with pytest.raises(gda.GdaError):
        s.load_dev(bad.data_ptr())
    x = psi.astype(np.complex128 if model == "xy" else np.float64)
    sp = x / np.abs(x) if model == "xy" else np.where(x >= 0, 1.0, -1.0)
    want = -np.real(np.einsum("ri,ij,rj->r", sp.conj(), bad.cpu().numpy(), sp))
    assert np.allclose(s.energy(), want, rtol=1e-6) and not np.allclose(want, before, rtol=1e-3)
    for v in (float("nan"), float("inf")):
        bad[1, 0] = bad[0, 1] = v
        with pytest.raises(gda.GdaError):
            s.load_dev(bad.data_ptr())
        assert not np.isfinite(s.energy()).any()
    s.load(J)
    s.set_state(psi)
    assert np.array_equal(s.energy(), before)
    s.close()
