"""What the speed of this simulator is measured on: evolutions, measurements,
gradients and batches as a user's program runs them, from chains whose passes
are shorter than a launch to the 8 GiB state of the throughput workload.

Every pass starts from the same inputs (the initial state is written first, as
a run of the program does), so it can be repeated.  Couplings, product states,
bond terms and drives are drawn from the seed alone.  `exact` repeats each pass
in 64 bits with plain torch operations.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2111_08044_gb300 import capi, inputs
from paper_2111_08044_gb300.sim import FloquetBatch, FloquetSimulator, chain_params

# the tensor-core block form, as the accuracy study and the paper's experiment build it
BLOCK = dict(mode=capi.SV_MODE_BLOCK, block_n=6, split=capi.SV_SPLIT_BF16X3)


def listed():
    return [
        # the plain form at its smallest in earnest: the 12-site preset over its
        # 100 periods, energies recorded (launch latency decides)
        dict(name="plain_L12_100", kind="plain", L=12, periods=100, K=4, first=0, ew=0.5, drive=False),
        # the plain form on a state larger than the L2 cache, odd L, the other
        # layer order and whole edge fields
        dict(name="plain_L27", kind="plain", L=27, periods=2, K=4, first=1, ew=1.0, drive=False),
        # the block form on a single short chain: few tiles in a pass
        dict(name="block_L14_32", kind="block", L=14, periods=32, K=4, first=0, ew=0.5),
        # the 26-site preset in the block form, a stretch of its 1000 periods
        dict(name="block_L26_8", kind="block", L=26, periods=8, K=4, first=0, ew=0.5),
        # the throughput workload: an 8 GiB state in the block form
        dict(name="block_L30_2", kind="block", L=30, periods=2, K=4, first=0, ew=0.5),
        # check runs beside a complex64 study: double-float, then complex128 on
        # a short chain
        dict(name="df64_L20_4", kind="check", precision="df64", L=20, periods=4, K=4, first=0, ew=0.5),
        dict(name="c128_L13_25", kind="check", precision="c128", L=13, periods=25, K=4, first=1, ew=0.5),
        # one step of fitting a drive: the final energy and its gradient through
        # autograd (the 20-site adjoint preset over fewer periods)
        dict(name="gradient_L20_8", kind="gradient", precision="c64", L=20, periods=8, K=4, first=0, ew=0.5),
        # the paper's experiment: the random circuit from its dimer state, one
        # stretch of periods between two samples of E and sigma_E
        dict(name="circuit_L24_4", kind="circuit", L=24, periods=4, omega=6.0),
        # what an echo study reads off a state: energy density, E and sigma_E,
        # overlap with the product state it started from
        dict(name="measure_L25", kind="measure", L=25, ew=0.5),
        # a parameter scan over short chains, each resident in shared memory
        dict(name="scan_resident_64", kind="batch", form="resident", chains=64, lo=9, hi=13, periods=32),
        # the same over longer chains: groups of tensor-core passes
        dict(name="scan_groups_48", kind="batch", form="tc", chains=48, lo=15, hi=19, periods=32),
    ]


def _periods(L, most, full):
    """Periods of a run: `most`, fewer where 2^L amplitudes make a period long
    (`full` is the L at which one period is left)."""
    return max(1, min(most, 1 << max(0, full - L)))


def draw(rng):
    kind = rng.choice(["plain", "plain", "block", "block", "check", "gradient", "circuit",
                       "measure", "batch", "batch"])
    circuit = dict(K=rng.choice([2, 3, 4]), first=rng.choice([0, 1]), ew=rng.choice([0.5, 1.0]))
    if kind == "plain":
        L = rng.randint(6, 26)
        most = rng.randint(20, 100)
        return dict(kind=kind, L=L, periods=_periods(L, most, 27), drive=rng.random() < 0.3, **circuit)
    if kind == "block":
        L = rng.randint(13, 29)
        return dict(kind=kind, L=L, periods=_periods(L, rng.randint(8, 48), 29), **circuit)
    if kind == "check":
        precision = rng.choice(["df64", "c128"])
        L = rng.randint(8, 23 if precision == "df64" else 20)
        full = 23 if precision == "df64" else 22
        return dict(kind=kind, precision=precision, L=L,
                    periods=_periods(L, rng.randint(4, 32), full), **circuit)
    if kind == "gradient":
        L = rng.randint(8, 21)
        return dict(kind=kind, precision=rng.choice(["c64", "c64", "c128"]) if L <= 16 else "c64",
                    L=L, periods=rng.randint(2, 10), **circuit)
    if kind == "circuit":
        L = 2 * rng.randint(7, 13)
        return dict(kind=kind, L=L, periods=rng.randint(1, 12), omega=rng.choice([5.0, 6.0, 7.0, 8.0]))
    if kind == "measure":
        return dict(kind=kind, L=rng.randint(13, 27), ew=circuit["ew"])
    if rng.random() < 0.5:
        lo = rng.randint(6, 12)
        return dict(kind=kind, form="resident", chains=rng.randint(16, 160), lo=lo,
                    hi=min(14, lo + rng.randint(1, 5)), periods=rng.randint(8, 48))
    lo = rng.randint(14, 18)
    return dict(kind=kind, form="tc", chains=rng.randint(12, 48), lo=lo, hi=min(20, lo + rng.randint(1, 4)),
                periods=rng.randint(8, 48))


# ------------------------------------------------------------------ inputs

def _chain(case, seed):
    """A chain with couplings around the default circuit's and a random
    product state."""
    r = inputs.SplitMix64(seed * 2654435761 + 17)
    cfg = inputs.ChainConfig(
        L=case["L"], J=r.uniform_range(0.8, 1.2), hx=r.uniform_range(0.6, 1.0),
        hz=r.uniform_range(0.2, 0.6), theta=r.uniform_range(0.1, 0.5), K=case.get("K", 4),
        first_layer=case.get("first", 0), edge_field_weight=case["ew"], seed=seed + 1)
    if case.get("drive") or case["kind"] == "gradient":
        P = case["periods"]
        cfg.theta_p = np.array([r.uniform_range(0.1, 0.5) for _ in range(P)])
        cfg.hx_p = np.array([r.uniform_range(0.6, 1.0) for _ in range(P)])
    return cfg


def _chains(case, seed):
    """A scan's chains: every length of the range in turn."""
    got = inputs.batch_preset(case["chains"], seed=seed + 3, Lmin=case["lo"], Lmax=case["hi"])
    for k, c in enumerate(got):
        c.L = case["lo"] + k % (case["hi"] - case["lo"] + 1)
    return got


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        cfg = _chain(case, seed)
        return dict(kind=kind, cfg=cfg, precision=case["precision"],
                    theta=torch.tensor(cfg.theta_p), hx=torch.tensor(cfg.hx_p))
    if kind == "batch":
        form = capi.SV_BATCH_RESIDENT if case["form"] == "resident" else capi.SV_BATCH_BLOCK_TC
        b = FloquetBatch(_chains(case, seed), form=form)
        return dict(kind=kind, batch=b, start=b.state.clone(), periods=case["periods"])
    if kind == "circuit":
        cfg = inputs.CircuitConfig(L=case["L"], omega=case["omega"], seed=seed + 1)
        pairs = cfg.pair_states()
        sim = FloquetSimulator(cfg.L)
        sim.init_pairs(pairs)
        sim.build(**dict(cfg.build_kwargs(), **BLOCK))
        return dict(kind=kind, sim=sim, pairs=pairs, periods=case["periods"])
    cfg = _chain(case, seed)
    sim = FloquetSimulator(cfg.L, precision=case.get("precision", "c64"))
    spinors = cfg.spinors()
    sim.init_product_state(spinors)
    sim.build(**chain_params(cfg, **(BLOCK if kind in ("block", "measure") else {})))
    if kind == "measure":
        sim.evolve(1, record=False)
    return dict(kind=kind, sim=sim, spinors=spinors, periods=case.get("periods"))


def run(state):
    kind = state["kind"]
    if kind == "gradient":
        from paper_2111_08044_gb300.autograd import final_energy
        theta = state["theta"].clone().requires_grad_(True)
        hx = state["hx"].clone().requires_grad_(True)
        f = final_energy(theta, hx, state["cfg"], precision=state["precision"])
        f.backward()
        return dict(energy=f.detach(), grad_theta=theta.grad, grad_hx=hx.grad)
    if kind == "batch":
        b = state["batch"]
        b.state.copy_(state["start"])
        e, n = b.evolve(state["periods"])
        return dict(energy=e, norm=n, state=b.state.view(torch.complex64))
    sim = state["sim"]
    if kind == "measure":
        density, norm = sim.energy()
        e, sigma, norm2 = sim.energy_moments()
        overlap = sim.overlap_product(state["spinors"])
        return dict(density=density, norm=norm, energy=e, sigma=sigma, norm2=norm2,
                    overlap=[overlap.real, overlap.imag])
    if kind == "circuit":
        sim.init_pairs(state["pairs"])
        sim.evolve(state["periods"], record=False)
        e, sigma, norm = sim.energy_moments()
        return dict(energy=e, sigma=sigma, norm=norm, state=sim.state)
    sim.init_product_state(state["spinors"])
    e, n = sim.evolve(state["periods"])
    return dict(energy=e, norm=n, state=sim.state_c128() if kind == "check" else sim.state)


# -------------------------------------------------------------------- work

def _chain_work(L, periods, gates, amp):
    """The initial state written (or read) once and the last one written; 16
    complex products and sums for each four amplitudes of a gate."""
    n = float(1 << L)
    return dict(bytes=2 * amp * n, flops=32.0 * n * gates * periods)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        tot = dict(bytes=0.0, flops=0.0)
        for c in _chains(case, 0):
            w = _chain_work(c.L, case["periods"], 4 * (c.L - 1), 8)
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    L = case["L"]
    n = float(1 << L)
    if kind == "measure":
        # the state read once; H0 psi (L + 1 terms), three squared norms, one overlap
        return dict(bytes=8 * n, flops=n * (4 * (L + 1) + 20))
    if kind == "circuit":
        w = _chain_work(L, case["periods"], L - 1, 8)
        return dict(bytes=w["bytes"], flops=w["flops"] + n * 32 * (L - 1))
    amp = 16 if case.get("precision", "c64") != "c64" else 8
    w = _chain_work(L, case["periods"], case["K"] * (L - 1), amp)
    if kind == "gradient":
        # forward, then both states walked back with one derivative product a gate
        return dict(bytes=2 * w["bytes"], flops=4 * w["flops"])
    return w


# ------------------------------------------------------------------- exact

_X = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128)
_Z = torch.tensor([[1, 0], [0, -1]], dtype=torch.complex128)
_I = torch.eye(2, dtype=torch.complex128)
# the local index r = 2 b_i + b_{i+1} against the memory order 2 b_{i+1} + b_i
_SWAP = [0, 2, 1, 3]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _terms(L, J, hx, hz, ew):
    """Bond terms h_b (4x4); hx may carry a gradient."""
    XI, IX = torch.kron(_X, _I), torch.kron(_I, _X)
    ZI, IZ = torch.kron(_Z, _I), torch.kron(_I, _Z)
    out = []
    for b in range(L - 1):
        a = ew if b == 0 else 0.5
        c = ew if b == L - 2 else 0.5
        out.append(J * (ZI @ IZ) + hx * (a * XI + c * IX) + hz * (a * ZI + c * IZ))
    return out


def _apply(psi, g, b):
    """A gate on sites (b, b + 1); psi: (..., 2^L)."""
    g = g[_SWAP][:, _SWAP].to(psi.device)
    lo = 1 << b
    if b < 3:
        v = psi.reshape(-1, 4 * lo)
        return (v @ torch.kron(g, torch.eye(lo, dtype=g.dtype, device=g.device)).T.contiguous()).reshape(psi.shape)
    v = psi.reshape(-1, 4, lo)
    return torch.stack([sum(g[r, c] * v[:, c] for c in range(4)) for r in range(4)], 1).reshape(psi.shape)


def _period(psi, L, terms, theta, tau, K, first):
    seen, gates = {}, []
    for h in terms:  # interior bonds share their term
        key = h.detach().numpy().tobytes()
        if key not in seen:
            seen[key] = torch.linalg.matrix_exp(-1j * tau * h)
        gates.append(seen[key])
    for _ in range(K):
        for parity in (first, 1 - first):
            for b in range(parity, L - 1, 2):
                psi = _apply(psi, gates[b], b)
    if theta is None:
        return psi
    kick = torch.linalg.matrix_exp(-1j * theta * _X)
    two = torch.kron(kick, kick)
    for b in range(0, L - 1, 2):
        psi = _apply(psi, two, b)
    return _apply(psi, torch.kron(_I, kick), L - 2) if L % 2 else psi


def _grow(factors, device):
    psi = torch.ones(1, dtype=torch.complex128, device=device)
    for f in factors:
        f = torch.as_tensor(np.asarray(f), dtype=torch.complex128).to(device)
        psi = (f[:, None] * psi[None, :]).reshape(-1)
    return psi


def _spin(spinors):
    return [np.array([s[0] + 1j * s[1], s[2] + 1j * s[3]]) / np.linalg.norm(s) for s in spinors]


def _hpsi(psi, L, terms):
    out = torch.zeros_like(psi)
    for b, h in enumerate(terms):
        out += _apply(psi, h, b)
    return out


def _energy(psi, L, terms):
    """(E, sigma, norm) of a state that need not be normalised."""
    h = _hpsi(psi, L, terms)
    n = torch.vdot(psi, psi).real
    e = torch.vdot(psi, h).real / n
    return e, torch.sqrt(torch.clamp(torch.vdot(h, h).real / n - e * e, min=0)), n


def _chain_exact(cfg, periods, device):
    obs = _terms(cfg.L, cfg.J, cfg.hx, cfg.hz, cfg.edge_field_weight)
    psi = _grow(_spin(cfg.spinors()), device)
    e, n = np.zeros(periods), np.zeros(periods)
    for p in range(periods):
        theta = cfg.theta if cfg.theta_p is None else float(cfg.theta_p[p])
        hx = cfg.hx if cfg.hx_p is None else float(cfg.hx_p[p])
        psi = _period(psi, cfg.L, _terms(cfg.L, cfg.J, hx, cfg.hz, cfg.edge_field_weight), theta,
                      cfg.tau, cfg.K, cfg.first_layer)
        nn = torch.vdot(psi, psi).real
        h = sum(torch.vdot(psi, _apply(psi, t, b)).real for b, t in enumerate(obs))
        e[p], n[p] = float(h / nn) / cfg.L, float(nn)
    return dict(energy=e, norm=n, state=psi)


def exact(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "batch":
        chains = _chains(case, seed)
        if case["chains"] * case["periods"] > 2500:
            return None  # a chain at a time: too long
        got = [_chain_exact(c, case["periods"], dev) for c in chains]
        return dict(energy=np.stack([g["energy"] for g in got]), norm=np.stack([g["norm"] for g in got]),
                    state=torch.cat([g["state"] for g in got]))
    if kind == "circuit":
        cfg = inputs.CircuitConfig(L=case["L"], omega=case["omega"], seed=seed + 1)
        terms = [torch.as_tensor(h) for h in cfg.h_bonds()]
        psi = _grow([p[_SWAP] / np.linalg.norm(p) for p in cfg.pair_states()], dev)
        for _ in range(case["periods"]):
            psi = _period(psi, cfg.L, terms, None, cfg.T, 1, 1)
        e, sigma, n = _energy(psi, cfg.L, terms)
        return dict(energy=float(e), sigma=float(sigma), norm=float(n), state=psi)
    if (1 << case["L"]) * case.get("periods", 1) * case.get("K", 4) > 1 << 31:
        return None  # over 20 seconds
    cfg = _chain(case, seed)
    if kind == "measure":
        terms = _terms(cfg.L, cfg.J, cfg.hx, cfg.hz, cfg.edge_field_weight)
        start = _grow(_spin(cfg.spinors()), dev)
        psi = _period(start, cfg.L, terms, cfg.theta, cfg.tau, cfg.K, cfg.first_layer)
        e, sigma, n = _energy(psi, cfg.L, terms)
        o = complex(torch.vdot(start, psi))
        return dict(density=float(e) / cfg.L, norm=float(n), energy=float(e), sigma=float(sigma),
                    norm2=float(n), overlap=[o.real, o.imag])
    if kind == "gradient":
        from torch.utils.checkpoint import checkpoint
        theta = torch.tensor(cfg.theta_p).requires_grad_(True)
        hx = torch.tensor(cfg.hx_p).requires_grad_(True)

        def step(v, t, h):
            drive = _terms(cfg.L, cfg.J, h, cfg.hz, cfg.edge_field_weight)
            return _period(v, cfg.L, drive, t, cfg.tau, cfg.K, cfg.first_layer)

        psi = _grow(_spin(cfg.spinors()), dev)
        for p in range(case["periods"]):
            psi = checkpoint(step, psi, theta[p], hx[p], use_reentrant=False)
        obs = _terms(cfg.L, cfg.J, cfg.hx, cfg.hz, cfg.edge_field_weight)
        f = torch.vdot(psi, _hpsi(psi, cfg.L, obs)).real / cfg.L
        f.backward()
        return dict(energy=f.detach().cpu(), grad_theta=theta.grad, grad_hx=hx.grad)
    return _chain_exact(cfg, case["periods"], dev)
