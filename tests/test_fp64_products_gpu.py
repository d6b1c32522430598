"""The FP64 mode's tiled products ([P^T | S], A, S2) against numpy's FP64
products of the same operands, at sizes around the 16-wide tiles, within the
rounding bound of a K-term dot product (K u sum |a||b|, either order), and the
stored symmetric halves equal bit for bit."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


def near(got, a, b):
    """got = a b^T with rounding bounded term by term."""
    bound = 2 * a.shape[1] * U64 * (np.abs(a) @ np.abs(b).T)
    assert np.all(np.abs(got - a @ b.T) <= bound)


# n = N: one entry, around one tile, around two, several; K' odd, below and above a k block
@pytest.mark.parametrize("N,K", [(1, 2), (3, 30), (15, 34), (16, 64), (17, 62), (31, 200), (33, 130), (50, 256), (97, 66)])
def test_products_match_their_definition(N, K):
    prob = G.pendulum_problem(N=N, K=K, sigma0=0.5, seed=N)
    s = G.Solver(prob, 2)
    s.step(I.pendulum_x0(N, 2), None, np.full(2 * N, 0.1), np.full(2 * N, 0.5), 0)
    n, nR, kp = N, 3 * N + 2, K // 2
    for b in range(2):
        dR = s.debug("dR", b).reshape(nR, kp)
        W = s.debug("W", b).reshape(n, kp)
        PS = s.debug("PS", b).reshape(n, nR + n)
        P, S, A = PS[:, :nR], PS[:, nR:], s.debug("A", b).reshape(n, n)
        near(P, W, dR)
        near(S, W, W)
        near(A, P, P)
        assert np.array_equal(S, S.T) and np.array_equal(A, A.T)
        if kp >= n:  # LSQ mode
            S2 = s.debug("S2", b).reshape(n, n)
            near(S2, S, S)
            assert np.array_equal(S2, S2.T)
    s.close()
