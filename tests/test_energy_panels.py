"""Final energies where the digits of J are not kept whole: panels of kept
digits, and panels of J and of spins sharing the state's scratch memory, give
the bits of the unbounded workspace; the scratch they use disturbs no run."""
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


def block(n):  # bytes of one 128-row block of J's digits
    return 7 * ((n + 63) // 64) * 16384


# XY N = 300, R = 120: one block of J and one of spins at a time in scratch
@pytest.mark.parametrize("model,n,R", [("xy", 300, 120), ("ising", 300, 250), ("xy", 257, 3), ("ising", 129, 1),
                                       ("xy", 130, 300), ("ising", 1000, 40)])
@pytest.mark.parametrize("kind", ["gauss", "int"])
def test_panels_give_the_same_bits(gda, model, n, R, kind):
    J = (synth.sk_gaussian if kind == "gauss" else synth.ising_pm1)(n, n)[0]
    g = 0.3 * synth.normal(n + 3, n)
    psi = synth.initial_amplitudes(n, R, n + R, 1.0, model == "xy")
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    s.set_state(psi)
    E, best = s.energy(), s.best()
    for bytes in (0, block(n), 2 * block(n), 10 * block(n)):
        s.set_energy_workspace(bytes)
        for _ in range(2):
            assert np.array_equal(s.energy(), E)
        Eb, rb, cfg = s.best()
        assert (Eb, rb) == best[:2] and np.array_equal(cfg, best[2])
    s.set_energy_workspace(0)
    s.load(J)  # a state made under the bound
    s.set_state(np.concatenate([psi] * 3))
    three = s.energy()
    s.set_energy_workspace(1 << 31)
    assert np.array_equal(s.energy(), three)
    s.close()


@pytest.mark.parametrize("kw", [dict(integ="rk4"), dict(integ="rk4", prec="SPARSE"), dict(integ="rk4", prec="BF16"),
                                dict(integ="euler", energy_every=3)])
@pytest.mark.parametrize("model,n", [("xy", 300), ("ising", 250), ("xy", 97)])
def test_energies_between_runs_change_nothing(gda, model, n, kw):
    J = synth.sparse_3regular(n + n % 2, 3)[0][:n, :n]
    R = 9
    p = dict(dt=0.01, eps=0.2, beta0=0.4, eps_hat=0.3, noise_D=0.05, noise_decay=1, seed=3, init_amp=0.2,
             prec=getattr(gda, kw.get("prec", "FP32")), integ=gda.RK4 if kw["integ"] == "rk4" else gda.EULER,
             energy_every=kw.get("energy_every", 0))
    out = []
    for look in (False, True):
        s = gda.Solver(J, None, gda.XY if model == "xy" else gda.ISING)
        if look:
            s.set_energy_workspace(0)
        s.run(gda.default_params(**p), R, 7)
        for _ in range(3):
            if look:
                s.energy()
                s.best()
            s.run(gda.default_params(**{**p, "init_mode": 2}), R, 6)
        out.append([*s.get_state(), s.energy(), *s.trace()])
        s.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def test_recorded_energies_in_scratch(gda):
    import torch
    n, R = 300, 120
    st = torch.cuda.Stream()
    psi = synth.initial_amplitudes(n, R, 4, 1.0, True)
    s = gda.Solver(synth.ising_pm1(n, 1)[0], None, gda.XY, stream=st)
    s.set_energy_workspace(0)
    s.set_state(psi)
    E = torch.zeros(R, dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.capture_begin()
        s.energy_dev(E.data_ptr())
        g.capture_end()
    s.set_energy_workspace(1 << 30)
    for J in (synth.sk_gaussian(n, 2)[0], synth.ising_pm1(n, 3)[0]):
        s.load(J)
        s.set_state(psi)
        ref = s.energy()
        with torch.cuda.stream(st):
            g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(E.cpu().numpy(), ref) and np.array_equal(s.energy(), ref)
    s.close()
    s = gda.Solver(synth.sk_gaussian(n, 2)[0], None, gda.XY)
    with pytest.raises(gda.GdaError):
        s.set_energy_workspace(-1)
    s.close()


def test_batch_groups_give_the_same_bits(gda):
    # instances in one group, in several, and cut into panels of rows and columns down to single blocks
    inst = []
    for k, (n, R, xy) in enumerate([(129, 40, True), (300, 300, False), (50, 130, True), (700, 70, True),
                                    (257, 129, False)]):
        J = (synth.ising_pm1 if k % 2 else synth.sk_gaussian)(n, n)[0]
        inst.append((J / np.sqrt(n) if k % 2 == 0 else J, 0.1 * synth.normal(k, n), gda.XY if xy else gda.ISING, R))
    b = gda.Batch(inst, seed=3)
    p = dict(dt=0.002, init_amp=0.1, prec=gda.BF16)
    b.run(gda.default_params(**p), 20)
    for bytes in (0, 1 << 20, 3 << 20, 8 << 20, 1 << 40):
        ref = [b.best() for _ in range(2)]
        b.set_energy_workspace(bytes)
        for E, r in [b.best(), b.best(), *ref]:
            assert np.array_equal(E, ref[0][0]) and np.array_equal(r, ref[0][1])
        b.run(gda.default_params(**p, init_mode=2), 10)
    for k, (J, g, model, R) in enumerate(inst):
        s = gda.Solver(J, g, model)
        s.set_state(b.get_state(k)[0])
        E = s.energy()
        assert b.best()[0][k] == E.min() and b.best()[1][k] == np.argmin(E)
        s.close()
    with pytest.raises(gda.GdaError):
        b.set_energy_workspace(-1)
    b.close()
