"""Edges of the instance check (mirrored 32 x 32 tiles) and of the proposal
network's kernels (64-row blocks, 16-byte reductions)."""
import ctypes as ct

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import __graft_entry__
    assert torch.cuda.is_available()
    __graft_entry__.ensure_built()
    from paper_1807_00699_gb300 import gda
    return torch, gda, gda.load_library()


@pytest.mark.parametrize("n,i,j", [(2, 0, 1), (33, 32, 0), (64, 31, 32), (65, 64, 64), (130, 5, 129), (130, 97, 98)])
def test_load_finds_one_bad_entry(env, n, i, j):
    torch, gda, _ = env
    J, g = synth.sk_gaussian(n, n)
    s = gda.Solver(J, g, gda.ISING)
    bad = []
    if i != j:
        a = J.copy()
        a[i, j] += 1e-9
        b = J.copy()
        b[j, i] += 1e-9
        bad += [a, b]
    for v in (np.nan, np.inf):
        a = J.copy()
        a[i, j] = a[j, i] = v
        bad.append(a)
        b = J.copy()
        b[j, i] = v
        bad.append(b)
    for a in bad:
        with pytest.raises(gda.GdaError) as e:
            s.load(a, g)
        assert e.value.status == 1
    J[i, i] = 0.25
    s.load(J, g)
    s.run(gda.default_params(dt=0.005), 3, 4)
    psi = np.where(s.get_state()[0] >= 0, 1.0, -1.0)
    E = -np.einsum("ri,ij,rj->r", psi, J, psi)
    assert np.allclose(s.energy(), E, rtol=1e-12, atol=1e-12 * np.abs(J).sum())
    s.close()


@pytest.mark.parametrize("M,shift", [(1, 0), (63, 1), (64, 0), (65, 3), (200, 0)])
def test_mlp_row_blocks(env, M, shift):
    torch, gda, lib = env
    from paper_1807_00699_gb300 import proposal
    rng = np.random.default_rng(M)
    p = proposal.init_params(M) + 0.05 * rng.normal(size=proposal.NPARAM).astype(np.float32)
    X = rng.normal(size=(M, 8)).astype(np.float32)
    dO = rng.normal(size=(M, 5)).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    pd, Xd, dOd = dev(p), dev(X), dev(dO)
    O = torch.empty((M, 5), device="cuda")
    H = torch.empty((M, 256), device="cuda")
    Gb = torch.zeros(proposal.NPARAM + 4, device="cuda")
    vp = lambda x: ct.c_void_p(x.data_ptr())  # noqa: E731
    G = Gb[shift:shift + proposal.NPARAM]  # also off a 16-byte boundary
    st = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.gda_mlp_forward(vp(pd), vp(Xd), M, vp(O), vp(H), st) == 0
    O2 = torch.empty_like(O)
    assert lib.gda_mlp_forward(vp(pd), vp(Xd), M, vp(O2), None, st) == 0
    assert lib.gda_mlp_backward(vp(pd), vp(Xd), vp(H), vp(dOd), M, vp(G), st) == 0
    torch.cuda.synchronize()
    o = np.cumsum([0, 1024, 128, 16384, 128, 640, 5])
    W = [p[o[k]:o[k + 1]].astype(np.float64) for k in range(6)]
    W1, W2, W3 = W[0].reshape(128, 8), W[2].reshape(128, 128), W[4].reshape(5, 128)

    def net(f, X, dO, h1, h2):
        """Outputs and gradient with every term through f (identity, or abs for the bound)."""
        a1 = f(X) @ f(W1).T + f(W[1])
        r1 = np.where(h1 > 0, a1, 0.0)
        a2 = r1 @ f(W2).T + f(W[3])
        r2 = np.where(h2 > 0, a2, 0.0)
        out = r2 @ f(W3).T + f(W[5])
        d2 = np.where(h2 > 0, f(dO) @ f(W3), 0.0)
        d1 = np.where(h1 > 0, d2 @ f(W2), 0.0)
        g = [d1.T @ f(X), d1.sum(0), d2.T @ r1, d2.sum(0), f(dO).T @ r2, f(dO).sum(0)]
        return out, np.concatenate([x.ravel() for x in g])

    h = H.cpu().numpy()
    same, size = net(lambda a: a, X, dO, h[:, :128], h[:, 128:]), net(np.abs, X, dO, h[:, :128], h[:, 128:])
    u = 2.0 ** -24  # every FP32 sum: at most as many roundings as terms, twice over two layers and the rows
    assert (np.abs(O.cpu().numpy() - same[0]) <= 300 * u * size[0] + 1e-30).all()
    assert torch.equal(O, O2)
    assert (np.abs(G.cpu().numpy() - same[1]) <= (600 + 2 * M) * u * size[1] + 1e-30).all()
    assert Gb[:shift].abs().sum() == 0 and Gb[shift + proposal.NPARAM:].abs().sum() == 0
