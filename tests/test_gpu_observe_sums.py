"""Energy density and norm of complex64 states from 13 sites where FP32 sums would
lose them: squares of very different size, and diagonal energies that FP32 rounds."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sim(L, ew, **kw):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, edge_field_weight=ew, **kw)
    sim = FloquetSimulator(L)
    sim.init_product_state(cfg.spinors())
    sim.build(**chain_params(cfg))
    return sim


@pytest.mark.parametrize("L", [13, 16, 21])
@pytest.mark.parametrize("bits", [(0, 4), (4, 4), (8, 4), (0, 2), (9, 3)])
def test_norm_of_uneven_squares(svlib, L, bits):
    """Squares of 1 where the given bits are clear, of 2^-25 elsewhere: each square is
    exact, and so is a sum of 2^L of them in FP32 pairs and FP64."""
    first, count = bits
    x = np.arange(1 << L)
    big = ((x >> first) & ((1 << count) - 1)) == 0
    psi = np.where(big, 1.0, 2.0 ** -13 * (1 + 1j)).astype(np.complex64)
    with _sim(L, 0.5) as sim:
        sim.set_host_state(psi)
        _, n = sim.energy()
    want = big.sum() + (~big).sum() * 2.0 ** -25
    assert abs(n / want - 1) < 2.0 ** -44


@pytest.mark.parametrize("L,ew", [(13, 0.5), (14, 1.0), (20, 0.5), (24, 1.0)])
def test_energy_density_of_basis_states(svlib, L, ew):
    """A basis state's energy is its diagonal energy, an FP32 pair (2^-47 of its value
    and of its two terms, each at most 2 L) in the tile and FP64 behind it."""
    J, hz = 0.937, 0.413
    rng = np.random.default_rng(L)
    with _sim(L, ew, J=J, hz=hz, hx=0.77) as sim:
        for x in [0, (1 << L) - 1] + [int(v) for v in rng.integers(0, 1 << L, 6)]:
            sim.state.zero_()
            sim.state[x] = 1
            e, n = sim.energy()
            z = 1 - 2 * ((x >> np.arange(L)) & 1)
            cz = np.full(L, hz)
            cz[[0, -1]] *= ew
            assert n == 1
            assert abs(e * L - (J * (z[1:] * z[:-1]).sum() + (cz * z).sum())) < 3 * 2 * L * 2.0 ** -46
