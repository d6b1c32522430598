"""A kernel's shared-memory limit belongs to the function, not to a handle: a
handle with a short horizon created after one with a long horizon must not
lower it under the first one's launches."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# nR beyond the 48 KB that need no opting in: chains of one thread per rollout and of a group
@pytest.mark.parametrize("M,N", [(16, 500), (24, 300)])
def test_a_smaller_handle_leaves_a_larger_one_running(M, N):
    def make(n):
        return G.Solver(G.chain_problem(M, N=n, K=64, precision=G.PREC_FP32, sigma0=0.2, method=G.METHOD_MPPI), 1)

    x0, tgt = I.chain_instances(2, 1, M)
    big = make(N)
    first = big.step(x0, tgt, np.zeros(2 * N), np.full(2 * N, 0.2), 0)[1]
    small = make(10)
    small.step(x0, tgt, np.zeros(20), np.full(20, 0.2), 0)
    again = big.step(x0, tgt, np.zeros(2 * N), np.full(2 * N, 0.2), 0)[1]
    assert np.array_equal(first, again)
    small.close()
    big.close()
