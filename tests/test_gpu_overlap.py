"""Passes that start while the one before still runs: the same bits as with an
event between any two launches (the profiled evolution), for passes of fewer
blocks than SMs, of one to a few blocks an SM, and of several tiles a block."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,mode,L", [
    ("c64", "plain", 16), ("c64", "plain", 20), ("c64", "plain", 22),
    ("df64", "plain", 13), ("df64", "plain", 17), ("c128", "plain", 9), ("c128", "plain", 13),
    ("c64", "drive", 18), ("c64", "drive", 19), ("c64", "drive", 21),
    ("c64", "block", 13), ("c64", "block", 14), ("c64", "block", 20), ("c64", "block", 22)])
def test_overlapped_passes_same_bits(svlib, precision, mode, L):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 5
    cfg = inputs.ChainConfig(L=L, seed=L)
    if mode == "drive":
        cfg.theta_p, cfg.hx_p = np.linspace(0.2, 0.4, P), np.linspace(0.7, 0.9, P)
    out = []
    for profiled in (False, True):
        with FloquetSimulator(L, precision=precision) as sim:
            sim.init_product_state(cfg.spinors())
            form = dict(mode=capi.SV_MODE_BLOCK, block_n=6) if mode == "block" else {}
            sim.build(**chain_params(cfg, renorm_every=2, **form))
            r = sim.evolve_profiled(P) if profiled else sim.evolve(P)
            out.append((r[0], r[1], sim.host_state()))
    for x, y in zip(*out):
        assert np.array_equal(x, y)
