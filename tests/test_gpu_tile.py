"""GPU parity of the plain form's tile passes (consecutive gates of a period
on one tile of the state) against the FP64 oracle: chains that one tile holds,
the first sizes that need several tiles, tiles whose sites wrap from the end of
one gate layer to the start of the next, long periods that need more than one
pass on a single tile, per-period drives and inverse periods."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu

# the plain form's tolerance on a state after a few periods (test_gpu_plain.py)
TOL = {"c64": 8e-6, "df64": 2e-12, "c128": 4e-13}


@pytest.mark.parametrize("precision", ["c64", "df64", "c128"])
@pytest.mark.parametrize("L,K,first,drive", [
    (5, 1, 0, False), (6, 4, 1, True), (8, 2, 0, False), (9, 9, 1, False), (12, 4, 0, True),
    (10, 3, 1, False), (11, 2, 0, True), (13, 6, 1, False), (15, 2, 1, False), (16, 1, 0, False),
    (17, 2, 0, True), (18, 1, 1, False), (19, 1, 1, True)])
def test_tile_passes_match_oracle(svlib, precision, L, K, first, drive):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 3
    rng = np.random.default_rng(L)
    cfg = inputs.ChainConfig(L=L, K=K, first_layer=first, periods=P, seed=70 + L, T=0.6,
                             edge_field_weight=1.0 if drive else 0.5)
    if drive:
        cfg.theta_p, cfg.hx_p = rng.uniform(0.1, 0.5, P), rng.uniform(0.6, 1.0, P)
    psi_o, _, e_o, n_o = orc.run_chain(cfg)
    with FloquetSimulator(L, precision=precision) as sim:
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg))
        e, n = sim.evolve(P)
        psi = sim.host_state().astype(np.complex128)
    tol = TOL[precision]
    assert np.linalg.norm(psi - psi_o) < tol
    # |H0|/L is below 3 and each energy is of a state within tol: 2 * 3 * tol
    np.testing.assert_allclose(e, e_o, atol=6 * tol, rtol=0)
    np.testing.assert_allclose(n, n_o, atol=2 * tol, rtol=0)


@pytest.mark.parametrize("L", [11, 16])
def test_tile_passes_inverse_and_renormalised(svlib, L):
    """P periods forward and P inverse periods back return the start; a folded
    renormalisation holds the norm at 1."""
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, seed=5)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(cfg.spinors())
        psi0 = sim.host_state().astype(np.complex128)
        sim.build(**chain_params(cfg, renorm_every=2))
        _, n = sim.evolve(4)
        sim.build(**chain_params(cfg, inverse=1))
        sim.evolve(4)
        psi = sim.host_state().astype(np.complex128)
    tol = TOL["c64"]
    assert np.max(np.abs(n - 1)) < 2 * tol
    assert np.linalg.norm(psi - psi0) < tol
