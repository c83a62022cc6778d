"""The DO-coefficient sampler judges its attempts in FP32 and takes the FP64
steps once per pair: every coefficient must still be the oracle's, bit for bit,
over enough draws to meet the ones that FP32 cannot judge."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


# 640,000 pairs: about 800,000 attempts, of which two in 2^20 (an annulus of
# area 2 pi 2^-20 in the square of area 4, within 2^-20 of s = 1) are undecided
@pytest.mark.parametrize("nt, N, K", [(40, 4000, 7), (1, 1, 1), (1, 31, 2), (3, 33, 16), (2, 4097, 3)])
def test_sampler_is_the_oracles_bit_for_bit(mdp, nt, N, K):
    sig = [0.4 * 0.9 ** k for k in range(K)]
    Y64 = mdp.mdp_sample_coeffs(nt, N, K, sig, seed=917, mdp_id=5, precision=mdp.MDP_FP64_CHECK).cpu().numpy()
    ref = oracle.sample_coeffs(nt, N, K, sig, seed=917, mdp_id=5)
    assert np.array_equal(Y64.view(np.int64), ref.reshape(Y64.shape).view(np.int64))
    Y32 = mdp.mdp_sample_coeffs(nt, N, K, sig, seed=917, mdp_id=5, precision=mdp.MDP_FP32).cpu().numpy()
    assert np.array_equal(Y32, Y64.astype(np.float32))
