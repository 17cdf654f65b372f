"""Final energies of couplings whose rows sum far below N times their largest
entry (sparse rows; integer couplings of complex spins) and of dense ones: the
error is no larger than that of the FP64 product (gda_energy_noalloc)."""
import ctypes as ct

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


def noalloc(gda, J, psi):
    import torch
    R, n = psi.shape
    Jd = torch.tensor(J, device="cuda")
    pd = torch.tensor(np.ascontiguousarray(psi).view(np.float32).ravel(), device="cuda")
    E = torch.empty(R, dtype=torch.float64, device="cuda")
    st = gda.load_library().gda_energy_noalloc(
        ct.c_void_p(Jd.data_ptr()), None, n, gda.XY if np.iscomplexobj(psi) else gda.ISING, ct.c_void_p(pd.data_ptr()),
        R, ct.c_void_p(E.data_ptr()), None)
    assert st == 0
    torch.cuda.synchronize()
    return E.cpu().numpy()


@pytest.mark.parametrize("kind,model,n", [("graph3", "ising", 4096), ("graph3", "xy", 1000), ("pm1", "xy", 512),
                                          ("gauss", "xy", 512), ("gauss", "ising", 1000)])
def test_error_no_larger_than_the_fp64_product(gda, kind, model, n):
    R = 48
    J = {"graph3": synth.sparse_3regular, "pm1": synth.ising_pm1, "gauss": synth.sk_gaussian}[kind](n, n)[0]
    psi = synth.initial_amplitudes(n, R, n, 1.0, model == "xy").astype(np.complex64 if model == "xy" else np.float32)
    if model == "xy":
        x, y = psi.real.astype(np.float64), psi.imag.astype(np.float64)
        m = np.sqrt(x * x + y * y)
        parts = [x / m, y / m]
    else:
        parts = [np.where(psi >= 0, 1.0, -1.0)]
    ref = np.zeros(R, dtype=np.longdouble)
    cols = [np.nonzero(row)[0] for row in J]
    for p in parts:
        p = p.astype(np.longdouble)
        for k in range(n):
            ref -= p[:, k] * (p[:, cols[k]] * J[k, cols[k]].astype(np.longdouble)).sum(1)
    s = gda.Solver(J, None, gda.XY if model == "xy" else gda.ISING)
    s.set_state(psi)
    err = [np.sqrt(np.mean(((E.astype(np.longdouble) - ref) ** 2).astype(np.float64)))
           for E in (s.energy(), noalloc(gda, J, psi))]
    # 1.5: the sampling error of two root mean squares over 48 restarts
    assert err[0] <= 1.5 * err[1], err
    s.close()
