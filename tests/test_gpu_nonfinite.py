"""States with NaN, infinite or vanishing amplitudes: what is read off them."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 0.0])
def test_batch_chains_without_a_norm(svlib, value):
    """Every form of a short chain reports such a chain the same way."""
    import torch
    from paper_2111_08044_gb300.sim import FloquetBatch
    Ls = (4, 9, 10, 11, 13, 14)
    chains = [inputs.ChainConfig(L=L, seed=L) for L in Ls]
    with FloquetBatch(chains, form=capi.SV_BATCH_RESIDENT) as b:
        for c, L in enumerate(Ls):
            psi = b.state[b.offsets[c]:b.offsets[c] + (8 << L)].view(torch.complex64)
            if value == 0.0:
                psi.zero_()
            else:
                psi[1] = value
        e, n = b.evolve(2)
    assert np.isnan(e).all()
    assert (n == 0).all() if value == 0.0 else np.isnan(n).all()


@pytest.mark.parametrize("L", [4, 8, 12, 14, 16, 18])
def test_norm_beyond_fp32(svlib, L):
    """Amplitudes whose squares overflow: the norm is infinite, the energy density
    (infinite terms of both signs) NaN, and moments are refused."""
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, seed=L)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg))
        sim.state.mul_(1e25)
        e, n = sim.energy()
        assert np.isnan(e) and n == np.inf
        with pytest.raises(capi.SvError, match="SV_ESTATE"):
            sim.energy_moments()
        e, n = sim.evolve(2)
        assert np.isnan(e).all() and (n == np.inf).all()
