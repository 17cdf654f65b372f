"""gda_energy_dev on one stream, then calls on another without a wait by the
caller: state calls that share its scratch memory come after it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kept", [True, False])
def test_other_streams_come_after_the_energies(kept):
    import torch

    import __graft_entry__
    __graft_entry__.ensure_built()
    from paper_1807_00699_gb300 import gda
    n, R = 2000, 600
    J = synth.sk_gaussian(n, 1)[0]
    psi = synth.initial_amplitudes(n, R, 4, 1.0, True)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    s = gda.Solver(J, None, gda.XY, stream=a)
    if not kept:
        s.set_energy_workspace(0)
    s.set_state(psi)
    ref = s.energy()
    E = torch.zeros(R, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        s.set_stream(a)
        s.energy_dev(E.data_ptr())
        s.set_stream(b)
        got = s.get_state()[0]
        s.set_stream(a)
        s.energy_dev(E.data_ptr())
        s.set_stream(b)
        s.set_state(psi)
        Eb = s.energy()
        torch.cuda.synchronize()
        assert np.array_equal(got, psi.astype(np.complex64))
        assert np.array_equal(E.cpu().numpy(), ref) and np.array_equal(Eb, ref)
    s.close()
