"""Workloads of the gain-dissipative solver: what its users have it do, through
the package's public entry points (gda.Solver, gda.Batch, proposal), over the
sizes, precisions, integrators and options in use.

listed() are the named workloads, draw(rng) gives another one of the same
ranges, prepare(case, seed) makes what a program holds before the call (an
instance, its solver, a batch, a network), run(state) is one pass with whole
outputs, work(case) the bytes and operations a pass cannot do without, and
exact(case, seed) the outputs in 64-bit arithmetic where that is defined.
"""
from __future__ import annotations

import ctypes as ct
import math

import numpy as np
import torch

from paper_1807_00699_gb300 import gda, proposal

PREC = {"fp32": gda.FP32, "bf16": gda.BF16, "fp8": gda.FP8, "sparse": gda.SPARSE}
INTEG = {"euler": gda.EULER, "rk4": gda.RK4}


def listed() -> list[dict]:
    return [
        # The paper's small Ising instance (N = 20, +-1 couplings, default parameters): 64 restarts
        # to the ground state and everything read back.  The smallest call: launches and latency.
        {"name": "ising20_fp32", "kind": "small", "model": "ising", "n": 20, "r": 64, "steps": 2000,
         "integ": "euler"},
        # The paper's XY integrator in the default precision, resumed from a checkpoint and
        # checkpointed again.
        {"name": "xy1000_rk4_fp32", "kind": "resume", "model": "xy", "n": 1000, "r": 256, "steps": 100,
         "integ": "rk4"},
        # The benchmark's XY solve: field, energy tracking every 100 steps, best configuration, final state.
        {"name": "xy1000_bf16", "kind": "solve", "model": "xy", "couplings": "gauss", "n": 1000, "r": 1024,
         "steps": 5000, "every": 100, "prec": "bf16", "integ": "euler", "noise": 0.0, "state": True},
        # The headline: SK N = R = 4096 with the coupling ramp (a tenth of its 10 000 steps).
        {"name": "sk4096_bf16", "kind": "solve", "model": "ising", "couplings": "sk", "n": 4096, "r": 4096,
         "steps": 1000, "every": 100, "prec": "bf16", "integ": "euler", "noise": 0.0, "state": False},
        # SK in FP8 at a ragged size.
        {"name": "sk3001_fp8", "kind": "solve", "model": "ising", "couplings": "sk", "n": 3001, "r": 2100,
         "steps": 1000, "every": 100, "prec": "fp8", "integ": "euler", "noise": 0.0, "state": False},
        # The paper's XY form with noise that fades at the threshold, RK4, on tensor cores.
        {"name": "xy1000_rk4_bf16", "kind": "solve", "model": "xy", "couplings": "gauss", "n": 1000, "r": 1024,
         "steps": 500, "every": 50, "prec": "bf16", "integ": "rk4", "noise": 0.05, "state": True},
        # The paper's 3-regular graphs over their nonzeros.
        {"name": "graph6000_sparse", "kind": "solve", "model": "ising", "couplings": "graph3", "n": 6000, "r": 512,
         "steps": 1000, "every": 100, "prec": "sparse", "integ": "euler", "noise": 0.0, "state": True},
        # The paper's second algorithm: a coupling matrix per restart.
        {"name": "xy1000_gdmod", "kind": "gdmod", "model": "xy", "n": 1000, "r": 256, "steps": 100},
        # The serving mix: 96 instances of both models stepped together.
        {"name": "mix96", "kind": "mix", "count": 96, "n_lo": 50, "n_hi": 2000, "r_lo": 16, "r_hi": 256,
         "steps": 300},
        # A request of the learned-proposal service: a new instance from the host, its proposal, a run, the answer.
        {"name": "request2000", "kind": "request", "model": "xy", "n": 2000, "r": 256, "steps": 500},
        # Judging a run: the Eq. (1) energies of every restart in FP64.
        {"name": "energies_xy1000", "kind": "energies", "model": "xy", "n": 1000, "r": 1024},
        # One optimiser step of the proposal network (a batch of 16 training instances).
        {"name": "train16", "kind": "train", "count": 16, "n_lo": 256, "n_hi": 1024},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["small", "resume", "solve", "solve", "solve", "graph", "gdmod", "mix", "request", "energies",
                       "train"])
    model = rng.choice(["ising", "xy"])
    if kind == "small":
        return {"kind": kind, "model": model, "n": _log_int(rng, 10, 200), "r": _log_int(rng, 16, 256),
                "steps": _log_int(rng, 200, 2000), "integ": rng.choice(["euler", "rk4"])}
    if kind == "resume":
        return {"kind": kind, "model": model, "n": _log_int(rng, 129, 1024), "r": _log_int(rng, 16, 512),
                "steps": rng.randint(40, 100), "integ": rng.choice(["euler", "rk4"])}
    if kind == "solve":
        c = {"kind": kind, "model": model, "couplings": "gauss" if model == "xy" else "sk",
             "n": _log_int(rng, 100, 4096), "r": _log_int(rng, 32, 4096 if model == "ising" else 2048),
             "steps": 0, "every": 100, "prec": rng.choice(["bf16", "bf16", "fp8"]),
             "integ": rng.choice(["euler", "euler", "rk4"]), "noise": rng.choice([0.0, 0.05])}
        cost = (4 if c["integ"] == "rk4" else 1) * c["n"] ** 2 * c["r"] * (2 if model == "xy" else 1)
        c["state"] = c["n"] * c["r"] <= 1 << 21
        c["steps"] = int(min(1000, max(100, rng.uniform(0.2, 0.6) * 1000 * 4096 ** 3 / cost)))
        return c
    if kind == "graph":
        return {"kind": "solve", "model": "ising", "couplings": "graph3", "n": 2 * _log_int(rng, 400, 4000),
                "r": _log_int(rng, 32, 1024), "steps": rng.randint(200, 600), "every": 100, "prec": "sparse",
                "integ": rng.choice(["euler", "euler", "rk4"]), "noise": rng.choice([0.0, 0.05]), "state": True}
    if kind == "gdmod":
        return {"kind": kind, "model": model, "n": _log_int(rng, 45, 1000), "r": _log_int(rng, 16, 256),
                "steps": rng.randint(30, 100)}
    if kind == "mix":
        return {"kind": kind, "count": _log_int(rng, 8, 96), "n_lo": 50, "n_hi": _log_int(rng, 300, 2000),
                "r_lo": 16, "r_hi": _log_int(rng, 32, 256), "steps": rng.randint(100, 400)}
    if kind == "request":
        return {"kind": kind, "model": model, "n": _log_int(rng, 256, 2048), "r": _log_int(rng, 32, 256),
                "steps": rng.randint(200, 800)}
    if kind == "energies":
        return {"kind": kind, "model": model, "n": _log_int(rng, 100, 2000), "r": _log_int(rng, 32, 1024)}
    return {"kind": "train", "count": _log_int(rng, 4, 16), "n_lo": 256, "n_hi": 1024}


# ---------------------------------------------------------------- inputs
def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed & 0x7FFFFFFFFFFF)


def _symmetric(upper: torch.Tensor) -> torch.Tensor:
    u = torch.triu(upper, 1)
    return u + u.T


def _couplings(kind: str, n: int, gen) -> torch.Tensor:
    """Symmetric FP64 couplings on the device, zero diagonal."""
    if kind == "gauss":  # N(0, 1/n)
        return _symmetric(torch.randn((n, n), generator=gen, device="cuda", dtype=torch.float64) / math.sqrt(n))
    if kind == "sk":  # N(0, 1)
        return _symmetric(torch.randn((n, n), generator=gen, device="cuda", dtype=torch.float64))
    if kind == "pm1":
        return _symmetric(torch.randint(0, 2, (n, n), generator=gen, device="cuda").double() * 2.0 - 1.0)
    if kind == "ternary":
        sign = 2 * torch.randint(0, 2, (n, n), generator=gen, device="cuda") - 1
        return _symmetric((sign * torch.randint(0, 2, (n, n), generator=gen, device="cuda")).double())
    # graph3: three random perfect matchings, weights U[-10, 10] (coinciding edges keep one weight)
    J = torch.zeros((n, n), device="cuda", dtype=torch.float64)
    for _ in range(3):
        p = torch.randperm(n, generator=gen, device="cuda")
        a, b = p[: n // 2], p[n // 2: 2 * (n // 2)]
        w = 20.0 * torch.rand(n // 2, generator=gen, device="cuda", dtype=torch.float64) - 10.0
        J[a, b] = w
        J[b, a] = w
    return J


def _field(n: int, gen) -> torch.Tensor:
    return 0.1 * (2.0 * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) - 1.0)


def _model(name: str) -> int:
    return gda.XY if name == "xy" else gda.ISING


def _amplitudes(model: str, r: int, n: int, scale: float, gen) -> np.ndarray:
    w = 2 if model == "xy" else 1
    x = scale * (2.0 * torch.rand((r, n, w), generator=gen, device="cuda", dtype=torch.float32) - 1.0)
    x = x.cpu().numpy()
    return x[..., 0] + 1j * x[..., 1] if w == 2 else x[..., 0]


def _instance(case: dict, seed: int):
    """(J, g or None) on the device for the single-instance workloads."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "small":
        J = _couplings("pm1" if case["model"] == "ising" else "gauss", case["n"], gen)
    elif kind == "solve":
        J = _couplings(case["couplings"], case["n"], gen)
    else:
        J = _couplings("gauss", case["n"], gen)
    g = _field(case["n"], gen) if case["model"] == "xy" else None
    return J, g, gen


def _mix_instances(case: dict, seed: int):
    rng = np.random.default_rng(case["count"])  # the sizes belong to the case, the values to the seed
    gen = _generator(seed)
    out = []
    for k in range(case["count"]):
        n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        r = int(rng.integers(case["r_lo"], case["r_hi"] + 1))
        J = _couplings("ternary" if k % 2 == 0 else "gauss", n, gen)
        out.append((J.cpu().numpy(), None, gda.ISING if k % 2 == 0 else gda.XY, r))
    return out


def _train_inputs(case: dict, seed: int) -> dict:
    """What a training loop holds: features, target spins and settings, network and optimiser state."""
    rng = np.random.default_rng(case["count"])  # the sizes belong to the case, the values to the seed
    gen = _generator(seed)
    sizes = [int(rng.integers(case["n_lo"], case["n_hi"] + 1)) for _ in range(case["count"])]
    cplx = [k % 2 for k in range(case["count"])]
    m = sum(sizes)
    phase = 2 * math.pi * torch.rand(m, generator=gen, device="cuda")
    S = torch.stack([torch.cos(phase), torch.sin(phase)], dim=1)
    for k, o in enumerate(np.concatenate([[0], np.cumsum(sizes)[:-1]])):
        if not cplx[k]:
            S[o:o + sizes[k], 0] = torch.where(S[o:o + sizes[k], 0] >= 0, 1.0, -1.0)
            S[o:o + sizes[k], 1] = 0.0
    p = torch.tensor(proposal.init_params(seed), device="cuda")
    return {"sizes": sizes, "cplx": cplx, "m": m, "S": S.contiguous(), "p0": p,
            "X": torch.randn((m, 8), generator=gen, device="cuda"),
            "T": torch.tensor([proposal.outputs_from_settings(*proposal.GRID[int(rng.integers(len(proposal.GRID)))])
                               for _ in sizes], dtype=torch.float32, device="cuda"),
            "m1": 0.01 * torch.randn(p.shape, generator=gen, device="cuda"),
            "m2": 1e-4 * torch.rand(p.shape, generator=gen, device="cuda"),
            "step": 20, "lr": 2e-3, "wset": 0.5}


def _params(case: dict, seed: int) -> gda.Params:
    kind = case["kind"]
    if kind == "small":
        return gda.default_params(integ=INTEG[case["integ"]], dt=0.01, init_amp=0.1, seed=seed & 0xFFFFFFFF)
    if kind == "resume":
        return gda.default_params(integ=INTEG[case["integ"]], dt=0.02, eps=0.2, beta0=0.5, eps_hat=0.2, init_mode=2)
    if kind == "gdmod":
        return gda.default_params(dt=0.05, eps=0.1, beta0=0.1, eps_hat=0.1, gamma_c=5.0, coupling=gda.GDMOD,
                                  init_amp=0.1, seed=seed & 0xFFFFFFFF)
    if kind == "mix":
        return gda.default_params(dt=0.005, eps=0.1, prec=gda.BF16)
    kw = dict(prec=PREC[case["prec"]], integ=INTEG[case["integ"]], energy_every=case["every"],
              noise_D=case["noise"], noise_decay=1, seed=seed & 0xFFFFFFFF)
    if case["couplings"] == "sk":  # the coupling ramp of the SK benchmark
        return gda.default_params(dt=0.1 / math.sqrt(case["n"]), eps=0.03, beta0=0.5, eps_hat=0.05, **kw)
    if case["couplings"] == "graph3":
        return gda.default_params(dt=0.005, eps=0.1, **kw)
    return gda.default_params(dt=0.05, eps=0.1, **kw)


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    st = {"case": case}
    if kind == "train":
        return {**st, **_train_inputs(case, seed)}
    if kind == "mix":
        st["batch"] = gda.Batch(_mix_instances(case, seed), seed=seed & 0xFFFFFFFF)
        st["params"] = _params(case, seed)
        return st
    J, g, gen = _instance(case, seed)
    Jh, gh = J.cpu().numpy(), None if g is None else g.cpu().numpy()
    if kind == "request":
        # the service's solver, created with an earlier instance of the same size
        st["solver"] = gda.Solver(np.zeros_like(Jh), None, _model(case["model"]))
        st["proposal"] = proposal.Proposal()
        return {**st, "J": Jh, "g": gh, "seed": seed & 0xFFFFFFFF}
    st["solver"] = gda.Solver(Jh, gh, _model(case["model"]))
    if kind == "energies":
        st["solver"].set_state(_amplitudes(case["model"], case["r"], case["n"], 1.0, gen))
        return st
    if kind == "resume":
        st["psi"] = _amplitudes(case["model"], case["r"], case["n"], 0.3, gen)
        st["gamma"] = np.zeros((case["r"], case["n"]), dtype=np.float32)
        st["beta"] = np.full(case["r"], 0.5, dtype=np.float32)
    st["params"] = _params(case, seed)
    return st


# ---------------------------------------------------------------- one pass
def _read_state(s: gda.Solver) -> dict:
    psi, gamma, beta, step = s.get_state()
    return {"psi": psi, "gamma": gamma, "beta": beta, "step": step}


def _read_best(s: gda.Solver) -> dict:
    E, r, cfg = s.best()
    return {"best_E": E, "best_r": r, "best_cfg": cfg}


def _train_step(st: dict) -> dict:
    """One step as the training loop takes it: forward, loss, gradient, Adam."""
    lib = gda.load_library()
    vp = lambda x: ct.c_void_p(x.data_ptr())  # noqa: E731
    cs = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
    p, m1, m2 = st["p0"].clone(), st["m1"].clone(), st["m2"].clone()
    offs = torch.tensor(np.concatenate([[0], np.cumsum(st["sizes"])]), dtype=torch.int32, device="cuda")
    cx = torch.tensor(st["cplx"], dtype=torch.int32, device="cuda")
    M, n_inst = st["m"], len(st["sizes"])
    O = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    H = torch.empty((M, 256), dtype=torch.float32, device="cuda")
    dO = torch.empty_like(O)
    L = torch.empty(n_inst, dtype=torch.float32, device="cuda")
    G = torch.zeros_like(p)
    for r in (lib.gda_mlp_forward(vp(p), vp(st["X"]), M, vp(O), vp(H), cs),
              lib.gda_proposal_loss(vp(O), vp(st["S"]), vp(st["T"]), vp(offs), vp(cx), n_inst, st["wset"], vp(dO),
                                    vp(L), cs),
              lib.gda_mlp_backward(vp(p), vp(st["X"]), vp(H), vp(dO), M, vp(G), cs),
              lib.gda_adam_step(vp(p), vp(G), vp(m1), vp(m2), proposal.NPARAM, st["lr"], 0.9, 0.999, 1e-8,
                                st["step"], cs)):
        if r != 0:
            raise gda.GdaError(r, "proposal training kernel failed")
    return {"O": O, "loss": L, "grad": G, "params": p, "m1": m1, "m2": m2}


def run(st: dict) -> dict:
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        return _train_step(st)
    if kind == "mix":
        st["batch"].run(st["params"], case["steps"])
        E, r = st["batch"].best()
        return {"E": E, "r": r}
    s = st["solver"]
    if kind == "energies":
        return {"E": s.energy()}
    if kind == "small":
        s.run(st["params"], case["r"], case["steps"])
        return {**_read_best(s), "E": s.energy(), **_read_state(s)}
    if kind == "resume":
        s.set_state(st["psi"], st["gamma"], st["beta"], 0)
        s.run(st["params"], case["r"], case["steps"])
        return _read_state(s)
    if kind == "gdmod":
        s.run(st["params"], case["r"], case["steps"])
        return {**_read_best(s), **_read_state(s)}
    if kind == "request":
        s.load(st["J"], st["g"])
        settings = st["proposal"].propose(s)
        s.run(proposal.proposed_params(settings, st["seed"], dt=0.05, prec=gda.BF16), case["r"], case["steps"])
        return {**settings, **_read_best(s)}
    s.run(st["params"], case["r"], case["steps"])
    steps, E, r = s.trace()
    out = {**_read_best(s), "trace_steps": steps, "trace_E": E, "trace_r": r}
    return {**out, **_read_state(s)} if case["state"] else out


# ---------------------------------------------------------------- the work a pass needs
def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "train":
        m = case["count"] * (case["n_lo"] + case["n_hi"]) // 2
        per_row = 2 * (8 * 128 + 128 * 128 + 128 * 5)
        return {"bytes": m * 4 * (8 + 2 + 5) + 18309 * 4 * 7, "flops": 3 * m * per_row}
    if kind == "mix":
        # log-uniform N: E[N^2], E[N] over [lo, hi], half the instances complex
        lo, hi = case["n_lo"], case["n_hi"]
        lg = math.log(hi / lo)
        n1, n2 = (hi - lo) / lg, (hi * hi - lo * lo) / (2 * lg)
        c = 1.5 * (case["r_lo"] + case["r_hi"]) / 2
        return {"bytes": int(case["count"] * (2 * n2 + 8 * n1 * c)),
                "flops": int(case["count"] * 2 * n2 * c * (case["steps"] + 1))}
    n, r = case["n"], case["r"]
    c = (2 if case["model"] == "xy" else 1) * r
    gemm = 2 * n * n * c
    state = 4 * n * c + 4 * n * r
    if kind == "energies":
        return {"bytes": 8 * n * n + 4 * n * c + 8 * r, "flops": gemm}
    stages = 4 if case.get("integ") == "rk4" else 1
    if kind == "small":
        return {"bytes": 4 * n * n + state + 8 * r, "flops": gemm * (stages * case["steps"] + 1)}
    if kind == "resume":
        return {"bytes": 4 * n * n + 2 * state, "flops": gemm * stages * case["steps"]}
    if kind == "gdmod":  # the per-restart matrices, rewritten every step, are larger than any on-chip memory
        return {"bytes": 8 * r * n * n * case["steps"], "flops": r * n * n * (5 + 2 * c // r) * case["steps"]}
    if kind == "request":
        return {"bytes": 8 * n * n + 8 * n, "flops": gemm * (case["steps"] + 1)}
    evals = case["steps"] // case["every"]
    if case["couplings"] == "graph3":
        nnz = 3 * n
        return {"bytes": 8 * nnz + state, "flops": 2 * nnz * c * (stages * case["steps"] + evals + 1)}
    width = 1 if case["prec"] == "fp8" else 2
    return {"bytes": width * n * n + state, "flops": gemm * (stages * case["steps"] + evals + 1)}


# ---------------------------------------------------------------- 64-bit values
def _philox_start(n: int, r: int, amp: float, seed: int, xy: bool) -> torch.Tensor:
    """Initial amplitudes U(-amp, amp) from Philox4x32-10 (Salmon et al., SC'11), counter (spin, restart, 0, 1)."""
    u32 = np.uint64(0xFFFFFFFF)
    x = [np.broadcast_to(np.arange(n, dtype=np.uint64)[None, :], (r, n)).copy(),
         np.broadcast_to(np.arange(r, dtype=np.uint64)[:, None], (r, n)).copy(),
         np.zeros((r, n), np.uint64), np.ones((r, n), np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(b >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), b & u32, (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), a & u32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [amp * (2.0 * ((v >> np.uint64(9)).astype(np.float64) + 0.5) / 8388608.0 - 1.0) for v in x[:2]]
    return torch.tensor(u[0] + 1j * u[1] if xy else u[0], device="cuda")


def _integrate(J, g, psi, gamma, beta, p: gda.Params, steps: int):
    """Eqs. (2), (5), (6) in 64 bits, psi [R][N] on the device."""
    J0 = J - torch.diag(torch.diagonal(J))
    h = 0.0 if g is None else -g * math.sqrt(p.rho_th)
    Jc = J0.to(psi.dtype)

    def rhs(x, ga, be):
        rho = (x * x.conj()).real
        return (x * (ga - rho) + be[:, None] * (x @ Jc) + h, p.eps * (p.rho_th - rho), p.eps_hat * (1.0 - be))

    for _ in range(steps):
        y = (psi, gamma, beta)
        k1 = rhs(*y)
        if p.integ == gda.EULER:
            psi, gamma, beta = (a + p.dt * k for a, k in zip(y, k1))
            continue
        k2 = rhs(*(a + 0.5 * p.dt * k for a, k in zip(y, k1)))
        k3 = rhs(*(a + 0.5 * p.dt * k for a, k in zip(y, k2)))
        k4 = rhs(*(a + p.dt * k for a, k in zip(y, k3)))
        psi, gamma, beta = (a + p.dt / 6.0 * (u + 2 * v + 2 * w + z) for a, u, v, w, z in zip(y, k1, k2, k3, k4))
    return psi, gamma, beta


def _energy64(J, g, psi) -> torch.Tensor:
    if psi.is_complex():
        m = psi.abs()
        s = torch.where(m > 0, psi / torch.where(m > 0, m, 1.0), torch.ones_like(psi))
        E = -((s.real @ J) * s.real + (s.imag @ J) * s.imag).sum(1)
        re = s.real
    else:
        re = torch.where(psi >= 0, 1.0, -1.0).double()
        E = -((re @ J) * re).sum(1)
    return E if g is None else E + re @ g


def _exact_train(case: dict, seed: int) -> dict:
    t = _train_inputs(case, seed)
    p = t["p0"].double().requires_grad_(True)
    o = np.cumsum([0, 128 * 8, 128, 128 * 128, 128, 5 * 128, 5])
    W1, b1, W2, b2, W3, b3 = (p[o[k]:o[k + 1]] for k in range(6))
    h = torch.relu(t["X"].double() @ W1.view(128, 8).T + b1)
    O = torch.relu(h @ W2.view(128, 128).T + b2) @ W3.view(5, 128).T + b3
    losses, i0 = [], 0
    for k, n in enumerate(t["sizes"]):
        Ok, S = O[i0:i0 + n], t["S"][i0:i0 + n].double()
        i0 += n
        if t["cplx"][k]:
            a, s = torch.complex(Ok[:, 0], Ok[:, 1]), torch.complex(S[:, 0], S[:, 1])
            c = (s.conj() * a).sum().detach()
            u = c / c.abs()
            amp = ((a - u * s).abs() ** 2).mean()
        else:
            u = 1.0 if float((S[:, 0] * Ok[:, 0]).sum()) >= 0 else -1.0
            amp = ((Ok[:, 0] - u * S[:, 0]) ** 2).mean()
        losses.append(amp + t["wset"] * ((Ok[:, 2:].mean(0) - t["T"][k].double()) ** 2).sum())
    L = torch.stack(losses)
    G, = torch.autograd.grad(L.sum(), p)
    m1 = 0.9 * t["m1"].double() + 0.1 * G
    m2 = 0.999 * t["m2"].double() + 0.001 * G * G
    q = p.detach() - t["lr"] * (m1 / (1 - 0.9 ** t["step"])) / ((m2 / (1 - 0.999 ** t["step"])).sqrt() + 1e-8)
    return {"O": O.detach(), "loss": L.detach(), "grad": G, "params": q, "m1": m1, "m2": m2}


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind not in ("small", "resume", "gdmod", "energies"):
        return None  # low-precision or long runs: no 64-bit value
    J, g, gen = _instance(case, seed)
    n, r, xy = case["n"], case["r"], case["model"] == "xy"
    if kind == "energies":
        psi = torch.tensor(_amplitudes(case["model"], r, n, 1.0, gen), device="cuda")
        return {"E": _energy64(J, g, psi.to(torch.complex128 if xy else torch.float64))}
    p = _params(case, seed)
    if kind == "resume":
        psi = torch.tensor(_amplitudes(case["model"], r, n, 0.3, gen), device="cuda")
        psi = psi.to(torch.complex128 if xy else torch.float64)
        beta = torch.full((r,), 0.5, device="cuda", dtype=torch.float64)
        psi, gamma, beta = _integrate(J, g, psi, torch.zeros((r, n), device="cuda", dtype=torch.float64), beta, p,
                                      case["steps"])
        return {"psi": psi, "gamma": gamma, "beta": beta, "step": None}
    psi = _philox_start(n, r, p.init_amp, seed & 0xFFFFFFFF, xy)
    gamma = torch.zeros((r, n), device="cuda", dtype=torch.float64)
    if kind == "small":
        if xy and case["steps"] > 400:
            return None  # soft modes: FP32 and 64-bit trajectories part
        beta = torch.ones(r, device="cuda", dtype=torch.float64)
        psi, gamma, beta = _integrate(J, g, psi, gamma, beta, p, case["steps"])
        E = _energy64(J, g, psi)
        return {"best_E": E.min(), "best_r": None, "best_cfg": None, "E": E, "psi": psi, "gamma": gamma, "beta": beta,
                "step": None}
    # GD-mod: one coupling matrix per restart, a few restarts at a time
    J0 = J - torch.diag(torch.diagonal(J))
    h = 0.0 if g is None else -g * math.sqrt(p.rho_th)
    outs = []
    for r0 in range(0, r, 64):
        x, ga = psi[r0:r0 + 64], gamma[r0:r0 + 64]
        K = (p.beta0 * J0).expand(x.shape[0], n, n).clone()
        for _ in range(case["steps"]):
            gi = ga + p.gamma_c
            DK = (gi[:, :, None] + gi[:, None, :]) * K
            if xy:
                y = torch.complex(torch.bmm(DK, x.real[:, :, None])[..., 0], torch.bmm(DK, x.imag[:, :, None])[..., 0])
            else:
                y = torch.bmm(DK, x[:, :, None])[..., 0]
            K += p.dt * p.eps_hat * (J0 - DK)
            rho = (x * x.conj()).real
            x, ga = x + p.dt * (x * (ga - rho) + y + h), ga + p.dt * p.eps * (p.rho_th - rho)
        outs.append((x, ga))
    psi, gamma = torch.cat([o[0] for o in outs]), torch.cat([o[1] for o in outs])
    E = _energy64(J, g, psi)
    return {"best_E": E.min(), "best_r": None, "best_cfg": None, "psi": psi, "gamma": gamma,
            "beta": None, "step": None}
