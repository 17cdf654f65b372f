"""gda_energy_dev recorded into a CUDA graph: replays and direct calls between
them give the energies of the instance loaded at the time, whatever the digits
its couplings take, and after states of other restart counts."""
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


def couplings(kind, n, seed):
    if kind == "gauss":
        return synth.sk_gaussian(n, seed)[0]
    J = synth.ising_pm1(n, seed)[0]  # one digit
    return J if kind == "int" else np.rint(1e5 * synth.sk_gaussian(n, seed)[0])  # "bigint": three


def fresh(gda, J, model, psi):
    s = gda.Solver(J, None, model)
    s.set_state(psi)
    E = s.energy()
    s.close()
    return E


@pytest.mark.parametrize("direct_first", [False, True])
@pytest.mark.parametrize("recorded,later", [("gauss", ("int", "bigint", "gauss")), ("int", ("gauss", "int", "bigint")),
                                            ("bigint", ("gauss", "int"))])
@pytest.mark.parametrize("model,n", [("xy", 200), ("ising", 300), ("xy", 129)])
def test_replays_follow_the_loaded_instance(gda, model, n, recorded, later, direct_first):
    import torch
    R = 40
    m = gda.XY if model == "xy" else gda.ISING
    st = torch.cuda.Stream()
    psi = synth.initial_amplitudes(n, R, 4, 1.0, model == "xy")
    many = synth.initial_amplitudes(n, 100, 5, 1.0, model == "xy")  # same state buffers, another column block
    s = gda.Solver(couplings(recorded, n, 1), None, m, stream=st)
    s.set_state(psi)
    if direct_first:
        s.energy()
    E = torch.zeros(R, dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.capture_begin()
        s.energy_dev(E.data_ptr())
        g.capture_end()

    def replay():
        E.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            g.replay()
        torch.cuda.synchronize()
        return E.cpu().numpy()

    for k, kind in enumerate(later):
        J = couplings(kind, n, 10 + k)
        ref, ref_many = fresh(gda, J, m, psi), fresh(gda, J, m, many)
        s.load(J)
        s.set_state(psi)
        if k % 2 == 0:
            assert np.array_equal(s.energy(), ref)
        assert np.array_equal(replay(), ref)
        assert np.array_equal(s.energy(), ref)
        s.set_state(many)
        assert np.array_equal(s.energy(), ref_many)
        s.set_state(psi)
        assert np.array_equal(replay(), ref)
        assert np.array_equal(s.energy(), ref)
    s.close()
