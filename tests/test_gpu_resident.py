"""GPU parity of the chains held in shared memory for a run of periods (single
chains of 5 to 15 sites in the plain form, batch chains of 2 to 14) against the
FP64 oracle: one block and clusters of blocks, periods of more gates than the
tables held at a time, drives, mixed lengths, and runs of any length."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu

# the plain form's tolerance on a state after a few periods (test_gpu_plain.py)
TOL = 8e-6


@pytest.mark.parametrize("L,K,first,drive", [
    (5, 25, 1, False), (8, 14, 0, True), (11, 10, 0, False), (12, 9, 1, False),
    (13, 8, 0, False), (14, 4, 1, True), (15, 7, 0, True)])
def test_single_chain_matches_oracle(svlib, L, K, first, drive):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 2
    rng = np.random.default_rng(L)
    cfg = inputs.ChainConfig(L=L, K=K, first_layer=first, periods=P, seed=30 + L, T=0.6)
    if drive:
        cfg.theta_p, cfg.hx_p = rng.uniform(0.1, 0.5, P), rng.uniform(0.6, 1.0, P)
    psi_o, _, e_o, n_o = orc.run_chain(cfg)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg))
        e, n = sim.evolve(P)
        psi = sim.host_state().astype(np.complex128)
    # up to 200 gates in two periods; test_gpu_plain.py's tolerance is for 80 and
    # the tables' rounding can add up over them
    tol = TOL * max(1.0, P * K * (L - 1) / 80)
    assert np.linalg.norm(psi - psi_o) < tol
    # |H0|/L is below 3 and each energy is of a state within tol: 2 * 3 * tol
    np.testing.assert_allclose(e, e_o, atol=6 * tol, rtol=0)
    np.testing.assert_allclose(n, n_o, atol=2 * tol, rtol=0)


def _chains(Ls, K):
    cs = inputs.batch_preset(n_chains=len(Ls), seed=3, Lmin=2, Lmax=2, periods=8)
    return [inputs.ChainConfig(L=L, K=k, J=c.J, hx=c.hx, hz=c.hz, theta=c.theta, periods=8,
                               seed=c.seed) for L, k, c in zip(Ls, K, cs)]


@pytest.mark.parametrize("Ls,K", [
    # every length, alone on the device: clusters of up to eight blocks
    ([2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14], [4] * 13),
    # more gates than the tables held (64, 96 above ten sites), with shorter periods
    # of the same length beside them
    ([9, 9, 2, 12, 12, 14], [9, 2, 70, 9, 3, 8]),
    ([10, 9, 10, 11], [8, 8, 3, 10]),
    # as many chains as SMs and more: one block a chain
    ([10] * 90 + [13] * 80 + [5, 14], [2] * 172)])
def test_batch_matches_oracle(svlib, Ls, K):
    from paper_2111_08044_gb300.sim import FloquetBatch
    chains = _chains(Ls, K)
    runs = [3, 1]
    P = sum(runs)
    with FloquetBatch(chains, form=capi.SV_BATCH_RESIDENT) as b:
        assert list(b.forms()) == [capi.SV_BATCH_RESIDENT] * len(Ls)
        parts = [b.evolve(r) for r in runs]
        e = np.concatenate([p[0] for p in parts], axis=1)
        n = np.concatenate([p[1] for p in parts], axis=1)
        states = [b.chain_state(c) for c in range(len(chains))]
    for c in sorted({Ls.index(L) for L in Ls} | set(range(min(len(Ls), 13))) | {len(Ls) - 3}):
        cfg = chains[c]
        psi_o, _, e_o, n_o = orc.run_chain(cfg, periods=P)
        # test_gpu_batch.py's tolerance: 2e-7 a gate on the state; energies as above
        tol = 2e-7 * P * cfg.K * (cfg.L - 1) + 1e-5
        assert np.linalg.norm(states[c].astype(np.complex128) - psi_o) < tol, (c, cfg.L)
        np.testing.assert_allclose(e[c], e_o, atol=6 * tol, rtol=0, err_msg=f"chain {c} L={cfg.L}")
        np.testing.assert_allclose(n[c], n_o, atol=2 * tol, rtol=0)


def test_batch_runs_of_any_length(svlib):
    """A run is split into launches without a trace: 300 periods at once, and in
    runs of 1, 129, 128 and 42, give the same bits."""
    from paper_2111_08044_gb300.sim import FloquetBatch
    chains = _chains([3, 8, 10, 13], [1, 2, 2, 1])
    out = []
    for runs in ([300], [1, 129, 128, 42]):
        with FloquetBatch(chains, form=capi.SV_BATCH_RESIDENT) as b:
            parts = [b.evolve(r) for r in runs]
            out.append([np.concatenate([p[k] for p in parts], axis=1) for k in (0, 1)]
                       + [b.chain_state(c) for c in range(4)])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
