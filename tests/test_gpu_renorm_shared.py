"""Folded renormalisation of chains that stay in shared memory for a run of periods
(the norm of a period is read back by every block of the chain in the same launch),
against one launch per period and against the oracle."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {"c64": 8e-6, "df64": 2e-12, "c128": 4e-13}


@pytest.mark.parametrize("every", [1, 2])
@pytest.mark.parametrize("precision,L,drive", [
    # clusters of 2 to 16 blocks, one block; single tiles of the wider types
    ("c64", 12, False), ("c64", 13, True), ("c64", 14, False), ("c64", 15, True), ("c64", 9, False),
    ("c128", 8, False), ("c128", 6, True), ("df64", 10, False), ("df64", 7, True)])
def test_renormalised_run_in_one_launch(svlib, precision, L, drive, every):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 6
    cfg = inputs.ChainConfig(L=L, periods=P, seed=50 + L)
    if drive:
        cfg.theta_p, cfg.hx_p = np.linspace(0.2, 0.4, P), np.linspace(0.7, 0.9, P)
    psi_o, _, e_o, _ = orc.run_chain(cfg)
    scale = 1.7  # a norm that a missing or stale factor would show
    out = []
    for runs in ([P], [1] * P, [2, 4]):
        with FloquetSimulator(L, precision=precision) as sim:
            sim.init_product_state(cfg.spinors())
            sim.build(**chain_params(cfg, renorm_every=every))
            sim.set_host_state(sim.host_state() * scale)
            parts = [sim.evolve(r) for r in runs]
            out.append([np.concatenate([p[k] for p in parts]) for k in (0, 1)] + [sim.host_state()])
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert np.array_equal(x, y)
    e, n, psi = out[0]
    tol = TOL[precision]
    # the factor is folded into a period's first gate: from period `every` on
    assert np.max(np.abs(n[:every] / scale ** 2 - 1)) < 2 * tol
    assert np.max(np.abs(n[every:] - 1)) < 2 * tol
    assert np.linalg.norm(psi.astype(np.complex128) - psi_o) < 2 * tol
    np.testing.assert_allclose(e, e_o, atol=6 * tol, rtol=0)
