"""GPU parity of the tiled measurements of complex64 states (energy density,
moments, product and pair overlaps, pair states) against the FP64 oracle, from
the shortest chains that take them: 13 sites (one site above the tile), window
passes that overlap the lowest tile, and whole edge fields."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,ew", [(13, 0.5), (14, 1.0), (17, 0.5), (20, 1.0), (21, 0.5)])
def test_measurements_match_oracle(svlib, L, ew):
    """The oracle measures the state the device holds, so only the
    measurement's own rounding is left: FP32 products summed over 2^L
    amplitudes, below 2e-7 of |H0| < 3 L, |H0|^2 and the norm."""
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, seed=20 + L, edge_field_weight=ew)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg))
        sim.evolve(2)
        density, norm = sim.energy()
        E, s, n = sim.energy_moments()
        ov = sim.overlap_product(cfg.spinors())
        psi = sim.host_state().astype(np.complex128)
    _, hobs = orc.chain_inputs(cfg)
    Eo, so, no = orc.energy_moments(psi, hobs)
    tol = 2e-7 * 3 * L
    assert abs(density * L - Eo) < tol and abs(E - Eo) < tol
    assert abs(s * s - so * so) < 2 * 3 * L * tol
    assert abs(norm - no) < 2e-7 and abs(n - no) < 2e-7
    # FP32 pairs: exact products, sums to 2^-47
    assert abs(ov - np.vdot(orc.product_state(cfg.spinors()), psi)) < 1e-13


@pytest.mark.parametrize("L", [14, 16, 20])
def test_pair_states_and_bond_moments_match_oracle(svlib, L):
    from paper_2111_08044_gb300.sim import FloquetSimulator
    cfg = inputs.CircuitConfig(L=L, seed=L)
    pairs = cfg.pair_states()
    with FloquetSimulator(L) as sim:
        sim.init_pairs(pairs)
        psi0 = sim.host_state()
        sim.build(**cfg.build_kwargs())
        sim.evolve(2, record=False)
        E, s, n = sim.energy_moments()
        ov = sim.overlap_pairs(pairs)
        psi = sim.host_state().astype(np.complex128)
    ref = orc.pair_product_state(pairs)
    # rounded once: half a unit in the last place of each part
    assert np.max(np.abs(psi0.real - ref.real)) <= np.max(np.abs(ref)) * 2.0 ** -24
    assert np.max(np.abs(psi0.imag - ref.imag)) <= np.max(np.abs(ref)) * 2.0 ** -24
    Eo, so, no = orc.energy_moments(psi, cfg.h_bonds())
    tol = 2e-7 * 3 * L
    assert abs(E - Eo) < tol and abs(n - no) < 2e-7
    assert abs(s * s - so * so) < 2 * 3 * L * tol
    assert abs(ov - np.vdot(ref, psi)) < 1e-13


@pytest.mark.parametrize("L,hz,ew", [(13, 0.57, 0.5), (16, 0.31, 1.0), (24, 0.57, 0.5), (25, 0.43, 1.0)])
def test_moments_of_a_sum_near_zero(svlib, L, hz, ew):
    """|+>^L without a transverse field: the diagonal energies, of up to L (1 + hz),
    cancel to E = 0, and sigma_E^2 = (L - 1) J^2 + sum_i cz_i^2."""
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, J=0.93, hx=0.0, hz=hz, edge_field_weight=ew, seed=1)
    with FloquetSimulator(L) as sim:
        sim.init_product_state(np.tile([np.sqrt(0.5), 0.0], (L, 2)))
        sim.build(**chain_params(cfg))
        e, s, _ = sim.energy_moments()
    # four roundings of 2^-24 an amplitude on terms d p, |d| <= L (1 + hz), independent
    # over 2^L amplitudes of p = 2^-L: six standard deviations
    tol = 6 * 4 * 2.0 ** -24 * L * (1 + hz) * 2.0 ** (-L / 2)
    assert abs(e) < tol
    var = (L - 1) * 0.93 ** 2 + hz ** 2 * (L - 2 + 2 * ew ** 2)
    assert abs(s / np.sqrt(var) - 1) < 8 * 2.0 ** -24
