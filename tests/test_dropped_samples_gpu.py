"""Dropped pairs and subnormal links in the sample rollouts, seen in dR and W
and not only in the costs: the zeros of a dropped pair and the values of the
kept ones come from different lanes of a warp, so an entry that the wrong lane
wrote last would be a silent zero (or a stale value) in P and S."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N = 6


def run(prec, M, sampling, x0, sigma, K=96):
    prob = G.chain_problem(M, N=N, K=K, precision=prec, sigma0=0.2, seed=3, sampling=sampling)
    s = G.Solver(prob, 1)
    _, _, rep = s.step(x0, I.chain_target(M, 0.2), np.zeros(2 * N), sigma, 0)
    Kp = 2 * N if sampling == G.SAMPLE_SIGMA else K // 2
    F = M - 1
    dR = s.debug("dR").reshape(N * (2 * F + 2) + 2 * F, Kp)
    W = s.debug("W").reshape(2 * N, Kp)
    out = dR, W, s.debug("C"), s.debug("e"), rep[0].n_masked, np.max(np.abs(s.debug("r")))
    s.close()
    return out


@pytest.mark.parametrize("M", [4, 10, 20, 40])
@pytest.mark.parametrize("sampling", [G.SAMPLE_RANDOM, G.SAMPLE_SIGMA])
@pytest.mark.parametrize("prec", [G.PREC_FP32, G.PREC_BF16])
def test_a_subnormal_link_loses_no_entry(M, sampling, prec):
    x0 = I.chain_rest_state(M)
    x0[0:2] = (1e-20, 0.0)  # the first free mass beside the fixed one at the origin
    sig = np.full(2 * N, 0.2)
    dR, W, C, e, masked, rmax = run(prec, M, sampling, x0, sig)
    dR64, W64, C64, e64, masked64, _ = run(G.PREC_FP64, M, sampling, x0, sig)
    assert masked == 0 and masked64 == 0
    F = M - 1
    u = (np.arange(N)[:, None] * (2 * F + 2) + 2 * F + np.arange(2)).ravel()  # control rows: 0.1 W, never rounded to zero
    assert np.array_equal(W != 0, W64 != 0) and np.array_equal(dR[u] != 0, dR64[u] != 0)
    # the reduced modes' stated bound, against the largest entry
    assert np.max(np.abs(W - W64)) <= 1e-4 * np.max(np.abs(W64))
    assert np.max(np.abs(dR - dR64)) <= 1e-4 * rmax


@pytest.mark.parametrize("M", [4, 10, 20, 40])
@pytest.mark.parametrize("prec", [G.PREC_FP64, G.PREC_FP32, G.PREC_BF16])
@pytest.mark.parametrize("gap", [None, 1e-20])
def test_a_dropped_pair_leaves_the_others_as_they_are(M, prec, gap):
    # sigma points: pair j perturbs control j alone, and a scale of 1e30 (1e200 in
    # FP64) makes that pair's cost overflow
    x0 = I.chain_rest_state(M)
    if gap:
        x0[0:2] = (gap, 0.0)
    sig = np.full(2 * N, 0.2)
    dR, W, C, e, masked, _ = run(prec, M, G.SAMPLE_SIGMA, x0, sig)
    assert masked == 0
    for j in (0, 5):
        big = sig.copy()
        big[j] = 1e200 if prec == G.PREC_FP64 else 1e30
        dRj, Wj, Cj, ej, maskedj, _ = run(prec, M, G.SAMPLE_SIGMA, x0, big)
        keep = np.arange(2 * N) != j
        assert maskedj == 1 and not np.all(np.isfinite(Cj.reshape(-1, 2)[j]))
        assert not np.any(dRj[:, j]) and not np.any(Wj[:, j]) and ej[j] == 0.0
        assert np.array_equal(dRj[:, keep], dR[:, keep]) and np.array_equal(Wj[:, keep], W[:, keep])
        assert np.array_equal(ej[keep], e[keep])
        assert np.array_equal(Cj.reshape(-1, 2)[keep], C.reshape(-1, 2)[keep])
