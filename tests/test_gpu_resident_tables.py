"""Chains in shared memory whose periods need several loads of the gate tables:
the last round of one load and the round that takes its place in the next differ
in whether sums are taken from the finished round."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu


# Periods of 189 to 288 gates, 96 gates a load: where the last round of one load was
# held, the next puts a round with such sums (one block; four and sixteen blocks).
@pytest.mark.parametrize("L,K,first", [(8, 27, 0), (8, 41, 1), (9, 24, 0), (9, 36, 1),
                                       (13, 16, 1), (15, 14, 0)])
def test_several_table_loads_match_oracle(svlib, L, K, first):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 4
    cfg = inputs.ChainConfig(L=L, K=K, first_layer=first, periods=P, seed=30 + L, T=0.6)
    psi_o, _, e_o, n_o = orc.run_chain(cfg)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg))
        runs = []
        for _ in range(20):
            sim.init_product_state(cfg.spinors())
            e, n = sim.evolve(P)
            runs.append((e, n, sim.host_state()))
    for r in runs[1:]:
        for x, y in zip(r, runs[0]):
            assert np.array_equal(x, y)
    e, n, psi = runs[0]
    # the plain form's tolerance, 8e-6 for 80 gates (test_gpu_plain.py)
    tol = 8e-6 * P * K * (L - 1) / 80
    assert np.linalg.norm(psi.astype(np.complex128) - psi_o) < tol
    # |H0|/L is below 3 and each energy is of a state within tol: 2 * 3 * tol
    np.testing.assert_allclose(e, e_o, atol=6 * tol, rtol=0)
    np.testing.assert_allclose(n, n_o, atol=2 * tol, rtol=0)
