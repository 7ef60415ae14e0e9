"""Tensor-core chain groups of a batch in one launch a pass: against each chain
alone, over what the CTAs' shares depend on (lengths of few and many tiles, more
groups than one launch takes, lengths of different numbers of passes, periods that
start off site 0)."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu


def _run(chains, P):
    from paper_2111_08044_gb300.sim import FloquetBatch
    with FloquetBatch(chains, form=capi.SV_BATCH_BLOCK_TC) as b:
        assert set(b.forms()) == {capi.SV_BATCH_BLOCK_TC}
        e, n = b.evolve(P)
        return e, n, [b.chain_state(c) for c in range(len(chains))]


@pytest.mark.parametrize("Ls,K", [
    # one tile a chain, and one chain; together 3 to 146 tiles
    ([13], [4]), ([13, 13, 14], [4, 4, 4]), ([17, 13, 18, 15, 16, 14, 18], [4] * 7),
    # below and from three tiles an SM (456 on 152 SMs): 448 and 480 tiles
    ([15, 16, 17] * 16, [4] * 48), ([16, 17] * 20, [2] * 40),
    # more structures than one launch takes
    ([13, 14, 15] * 7, [1] * 3 + [2] * 3 + [3] * 3 + [4] * 3 + [5] * 3 + [6] * 3 + [7] * 3)])
def test_groups_match_single_chains(svlib, Ls, K):
    """The state's bits, and its energies to the order of their FP32 sums."""
    P = 5
    cs = inputs.batch_preset(n_chains=len(Ls), seed=9, Lmin=2, Lmax=2, periods=P)
    chains = [inputs.ChainConfig(L=L, K=k, J=c.J, hx=c.hx, hz=c.hz, theta=c.theta, periods=P,
                                 seed=c.seed) for L, k, c in zip(Ls, K, cs)]
    e, n, psi = _run(chains, P)
    for c in sorted({Ls.index(L) for L in Ls} | {len(Ls) // 2, len(Ls) - 1}):
        e1, n1, psi1 = _run([chains[c]], P)
        assert np.array_equal(psi[c], psi1[0])
        # sums of at most 2^18 terms, |term| <= 3 |psi_x|^2, in FP32 per row (64
        # terms) and compensated over rows: 64 roundings of 2^-24 and a few more
        np.testing.assert_allclose(e[c], e1[0], atol=3 * 70 * 2.0 ** -24, rtol=0)
        np.testing.assert_allclose(n[c], n1[0], atol=70 * 2.0 ** -24, rtol=0)
