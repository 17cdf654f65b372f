"""Final energies through exact digit products (csrc/energy_tc.cu): tile edges,
digit counts, panels of one row or column, wide coupling scales and symmetry,
against sums of the same spins in extended precision."""
import math

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


def couplings(kind, n):
    J = synth.sk_gaussian(n, n + 1)[0] if kind != "int" else synth.ising_pm1(n, n)[0]
    J = J + np.diag(synth.normal(n + 7, n) if kind != "int" else np.arange(n) % 5 - 2.0)
    if kind == "bigint":  # three digits
        J = np.rint(J * 1e6)
    if kind == "scales":  # rows of very different magnitude, and an isolated spin
        d = np.exp2(np.round(40 * synth.uniform01(n, n) - 20))
        J = J * d[:, None] * d[None, :]
        J[:, 0] = J[0, :] = 0.0
    if kind == "tiny":
        J = J * 2.0 ** -1015
    return J


def spins(psi):
    if not np.iscomplexobj(psi):
        return np.where(psi >= 0, 1.0, -1.0), None
    x, y = psi.real.astype(np.float64), psi.imag.astype(np.float64)
    m = np.sqrt(x * x + y * y)
    return x / m, y / m


@pytest.mark.parametrize("kind", ["gauss", "int", "bigint", "scales", "tiny"])
@pytest.mark.parametrize("model,n,R", [("ising", 1, 1), ("xy", 1, 2), ("ising", 20, 64), ("xy", 63, 65),
                                       ("ising", 129, 127), ("xy", 128, 64), ("xy", 513, 3), ("ising", 700, 130)])
def test_energies_against_extended_sums(gda, kind, model, n, R):
    J = couplings(kind, n)
    g = 0.3 * synth.normal(n + 3, n) * (2.0 ** -1015 if kind == "tiny" else 1.0) if R % 2 else None
    psi = synth.initial_amplitudes(n, R, n + R, 1.0, model == "xy")
    s = gda.Solver(J, g, gda.XY if model == "xy" else gda.ISING)
    s.set_state(psi)
    E = s.energy()
    sr, si = spins(psi.astype(np.complex64 if model == "xy" else np.float32))
    rowmax = np.abs(J).max(axis=1)
    for r in range(0, R, max(1, R // 4)):
        terms = [-sr[r, i] * J[i] * sr[r] for i in range(n)]
        if si is not None:
            terms += [-si[r, i] * J[i] * si[r] for i in range(n)]
        if g is not None:
            terms.append(g * sr[r])
        ref = math.fsum(np.concatenate(terms))
        # digits: 2^-52 rowmax_i per term of row i; the sums of s_i T_i in double
        T = np.abs(J) @ np.ones(n)
        # (the reference's own products round as well: 2^-52 per term)
        tol = 2.0 ** -52 * ((3 * n + 3) * rowmax.sum() + (n + 3) * (T.sum() + (np.abs(g).sum() if g is not None else 0)))
        assert abs(E[r] - ref) <= tol
        if kind in ("int", "bigint") and model == "ising" and g is None:
            assert E[r] == ref
    Eb, rb, _ = s.best()
    assert rb == int(np.argmin(E)) and Eb == E[rb]
    if g is None:  # global sign: the same bits
        s.set_state(-psi)
        Em = s.energy()
        zero = (psi.real == 0).any() if model == "ising" else False
        assert zero or np.array_equal(E, Em)
    s.close()


def test_extreme_digits_are_summed_exactly(gda):
    # every digit of J and s at its largest magnitude and one sign: the FP32
    # accumulators reach their bound over a full chunk
    n = 1024
    v = float(2 ** 55 - 1) / 2 ** 55  # digits 128, 0, 0, ..., -1
    w = sum(127 * 2.0 ** (8 * k) for k in range(7)) / 2 ** 55  # seven digits of 127
    for x in (v, w):
        J = np.full((n, n), x)
        s = gda.Solver(J, None, gda.XY)
        th = np.full((2, n), 0.25)
        s.set_state(np.exp(1j * th))
        sr, si = spins(np.exp(1j * th).astype(np.complex64))
        # all spins equal: E = -n^2 x (sr^2 + si^2), to the rounding of the double sums over n rows
        ref = -n * n * x * (sr[:, 0] ** 2 + si[:, 0] ** 2)
        assert np.abs(s.energy() - ref).max() <= 2.0 ** -52 * n * n * x * 8
        s.close()


def test_batch_energies_equal_single_instances(gda):
    inst, ref = [], []
    for k, (n, R, xy) in enumerate([(129, 40, True), (300, 17, False), (50, 130, True), (64, 9, False)]):
        J = couplings("int" if k == 3 else "gauss", n) / (1 if k == 3 else math.sqrt(n))
        inst.append((J, None, gda.XY if xy else gda.ISING, R))
    b = gda.Batch(inst, seed=3)
    b.run(gda.default_params(dt=0.01, prec=gda.BF16), 33)
    for _ in range(2):  # the second call reuses the coupling digits
        E, r = b.best()
        for k, (J, g, model, R) in enumerate(inst):
            s = gda.Solver(J, g, model)
            s.set_state(b.get_state(k)[0])
            Es = s.energy()
            assert r[k] == int(np.argmin(Es)) and E[k] == Es[r[k]]
            s.close()
        b.run(gda.default_params(dt=0.01, prec=gda.BF16, init_mode=2), 12)
    b.close()


def test_energies_recorded_into_a_graph(gda):
    # a recorded gda_energy_dev follows the instance loaded when it is replayed
    import torch
    n, R = 200, 40
    st = torch.cuda.Stream()
    J1, J2 = synth.sk_gaussian(n, 1)[0], synth.sk_gaussian(n, 2)[0]
    psi = synth.initial_amplitudes(n, R, 4, 1.0, True)
    s = gda.Solver(J1, None, gda.XY, stream=st)
    s.set_state(psi)
    E = torch.zeros(R, dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.capture_begin()
        s.energy_dev(E.data_ptr())  # the first energy call of this context
        g.capture_end()
    for J in (J1, J2, J1):
        s.load(J)
        s.set_state(psi)
        with torch.cuda.stream(st):
            g.replay()
        torch.cuda.synchronize()
        got = E.cpu().numpy()
        assert np.array_equal(got, s.energy())
    s.close()
