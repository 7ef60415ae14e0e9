"""Overlaps of complex64 states from 13 sites with product states, in FP64's precision
and over FP64's range: factors FP32 cannot hold, tiny and large amplitudes."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import inputs

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _basis(sim, x, value=1.0):
    sim.state.zero_()
    sim.state[x] = value


def _sim(L):
    from paper_2111_08044_gb300.sim import FloquetSimulator
    sim = FloquetSimulator(L)
    sim.init_product_state(np.tile([1.0, 0.0, 0.0, 0.0], (L, 1)))
    return sim


@pytest.mark.parametrize("L", [13, 18])
@pytest.mark.parametrize("site", [0, 1, 5, 11, 12])
def test_factor_of_one_site_exactly(svlib, L, site):
    """Every other factor is 1, so the overlap is the site's normalised component."""
    rng = np.random.default_rng(site)
    with _sim(L) as sim:
        for _ in range(4):
            sp = np.tile([1.0, 0.0, 0.0, 0.0], (L, 1))
            sp[site] = rng.normal(size=4)
            f = sp[site] / np.sqrt((sp[site] ** 2).sum())
            for bit in (0, 1):
                _basis(sim, bit << site)
                o = sim.overlap_product(sp)
                # the norm's sum may be rounded in another order: two units
                assert abs(o - np.conj(f[2 * bit] + 1j * f[2 * bit + 1])) < 4 * EPS


@pytest.mark.parametrize("eps", [1e-2, 1e-3, 1e-4, 1e-9, 1e-20])
@pytest.mark.parametrize("up", ["low", "high", "all"])
def test_small_factors(svlib, eps, up):
    """A basis state's overlap is a product of L factors: 2 L roundings."""
    L = 16
    bits = {"low": (1 << 12) - 1, "high": 15 << 12, "all": (1 << 16) - 1}[up]
    sp = np.zeros((L, 4))
    sp[:, 0], sp[:, 2] = 1.0, eps
    n = bin(bits).count("1")
    want = np.longdouble(eps) ** n / np.sqrt(np.longdouble(1 + eps * eps)) ** L
    with _sim(L) as sim:
        # small and large amplitudes, where the overlap is within FP64's range
        for a in (1.0, 2.0 ** -100, 2.0 ** -126, 2.0 ** 100):
            _basis(sim, bits, a)
            o = np.longdouble(sim.overlap_product(sp).real)
            if want * a > 1e-300:
                assert abs(o / (want * a) - 1) < 4 * L * EPS


@pytest.mark.parametrize("L", [13, 15, 18])
def test_sums_match_long_double(svlib, L):
    """Random states whose amplitudes span 40 powers of two: below 2 L + 8 roundings
    of the sum of the terms' sizes (FP64 tables; sums over fewer than 2^12 blocks)."""
    rng = np.random.default_rng(L)
    with _sim(L) as sim:
        for k in range(3):
            psi = (rng.normal(size=1 << L) + 1j * rng.normal(size=1 << L)) * 2.0 ** -rng.integers(0, 41, 1 << L)
            psi = psi.astype(np.complex64)
            psi[rng.random(1 << L) < 0.2 * k] = 0
            sp = rng.normal(size=(L, 4)) * np.where(rng.random((L, 4)) < 0.2 * k, 0, 1)
            sp[:, 0] += 0.1
            sim.set_host_state(psi)
            o = sim.overlap_product(sp)
            phi = np.ones(1, dtype=np.clongdouble)
            for s in sp:
                f = np.array([s[0] + 1j * s[1], s[2] + 1j * s[3]]) / np.sqrt((s ** 2).sum())
                phi = (f[:, None].astype(np.clongdouble) * phi[None, :]).reshape(-1)
            terms = np.conj(phi) * psi
            # random signs: the roundings of 2^L terms add up to far less than their bound
            assert abs(np.clongdouble(o) - terms.sum()) < (2 * L + 8) * EPS * np.abs(terms).sum()


@pytest.mark.parametrize("L", [13, 16])
def test_overlap_of_non_finite_amplitudes(svlib, L):
    with _sim(L) as sim:
        sp = inputs.ChainConfig(L=L, seed=3).spinors()
        _basis(sim, 5, float("nan"))
        assert np.isnan(sim.overlap_product(sp).real)
        sim.state.fill_(3e38)
        sp = np.tile([1.0, 0.0, 1.0, 0.0], (L, 1))
        want = np.float64(np.float32(3e38)) * 2.0 ** (L / 2)
        assert abs(sim.overlap_product(sp).real / want - 1) < 4 * L * EPS


@pytest.mark.parametrize("L,eps", [(14, 1.0), (16, 1e-2), (16, 1e-3), (18, 1e-4), (24, 0.03)])
def test_small_amplitudes_of_pair_states(svlib, L, eps):
    """Each component rounded once to FP32 (2^-24 of it, 2^-150 where that is subnormal)
    from FP64 products, off by L + 4 roundings of the amplitude."""
    from paper_2111_08044_gb300.sim import FloquetSimulator
    rng = np.random.default_rng(L)
    pairs = (rng.normal(size=(L // 2, 4)) + 1j * rng.normal(size=(L // 2, 4))) * np.array([1, eps, eps, eps ** 2])
    pairs[0, 1] = 0
    with FloquetSimulator(L) as sim:
        sim.init_pairs(pairs)
        psi = sim.host_state()
    want = np.ones(1, dtype=np.clongdouble)
    for p in pairs:
        f = p.astype(np.clongdouble) / np.sqrt((np.abs(p.astype(np.clongdouble)) ** 2).sum())
        want = (f[[0, 2, 1, 3]][:, None] * want[None, :]).reshape(-1)  # memory order 2 b_1 + b_0
    bound = (L + 4) * EPS * np.abs(want) + 2.0 ** -150
    for got, x in ((psi.real, want.real), (psi.imag, want.imag)):
        assert np.all(np.abs(got - x) <= 2.0 ** -24 * np.abs(x) * (1 + 1e-6) + bound)
