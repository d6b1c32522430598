"""The FP32 sample rollouts' reciprocal square root: a link whose squared
length is subnormal in FP32 (two masses 1e-20 apart) has a finite force, so no
sample is dropped and the costs match the FP64 mode's; coincident masses have
none, and every sample is dropped, as in the FP64 mode."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def run(prec, M, gap):
    x0 = I.chain_rest_state(M)
    x0[0:2] = (gap, 0.0)  # the first free mass beside the fixed one at the origin
    tgt = I.chain_target(M, 0.2)
    N, K = 6, 96
    prob = G.chain_problem(M, N=N, K=K, precision=prec, sigma0=0.2, seed=3)
    s = G.Solver(prob, 1)
    st, _, rep = s.step(x0, tgt, np.zeros(2 * N), np.full(2 * N, 0.2), 0)
    C = s.debug("C")
    s.close()
    return st, rep[0].n_masked, C


@pytest.mark.parametrize("M", [4, 10, 20, 40])
@pytest.mark.parametrize("prec", [G.PREC_FP32, G.PREC_BF16])
def test_subnormal_link_length(M, prec):
    # FP32 chains of 18 and more masses carry positions relative to the initial
    # ones: the same link there is the reference link vector itself
    st, masked, C = run(prec, M, 1e-20)
    _, masked64, C64 = run(G.PREC_FP64, M, 1e-20)
    assert masked == 0 and masked64 == 0
    assert np.all(np.abs(C - C64) <= 1e-4 * np.abs(C64))  # the stated bound of the reduced modes' sample costs


@pytest.mark.parametrize("M", [4, 20])
def test_coincident_masses_drop_every_sample(M):
    for prec in (G.PREC_FP32, G.PREC_FP64):
        st, masked, C = run(prec, M, 0.0)
        assert st == G.E_NONFINITE and masked == 48 and not np.any(np.isfinite(C))
