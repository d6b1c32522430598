"""Which kernel solves the damped system: the tests that compare the cluster
Cholesky with the single-CTA kernel say something only where a cluster was
taken, so the report names the CTAs per instance and this file pins them."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the sizes of test_cluster_solve_gpu.py (but N = 333, whose system does not fit a cluster's shared
# memory) and the longest horizon that fits
SIZES = [(17, 1), (24, 3), (41, 2), (100, 1), (100, 9), (100, 30), (100, 70), (200, 1), (200, 12), (320, 1)]


def ctas(N, batch, prec, nt=None, shapes=None, M=4, **kw):
    s = G.Solver(G.chain_problem(M, N=N, K=4 * N + 64, precision=prec, sigma0=0.2, seed=5, **kw), batch, shapes)
    if nt:
        G.gnmppi_tune_set(s.h, 1, nt)
    r = G.gnmppi_tune_report(s.h)
    s.close()
    return r["solve_ctas"]


@pytest.mark.parametrize("prec", [G.PREC_BF16, G.PREC_FP32, G.PREC_FP64])
def test_a_cluster_where_the_batch_leaves_sms_idle(prec):
    sizes = {(N, b): ctas(N, b, prec) for N, b in SIZES if prec != G.PREC_FP64 or N * b <= 400}
    assert all(2 <= c <= 16 and b * c <= 152 for (_, b), c in sizes.items()), sizes
    assert len(set(sizes.values())) >= 3, sizes
    assert ctas(17, 1, prec, nt=512) == sizes[17, 1]


def test_one_cta_otherwise():
    assert ctas(100, 1, G.PREC_BF16, nt=256) == 1 and ctas(100, 1, G.PREC_BF16, nt=128) == 1
    assert ctas(16, 1, G.PREC_FP64) == 1  # n = 32: two panels
    assert ctas(20, 77, G.PREC_BF16) == 1  # two CTAs each would need 154 SMs
    assert ctas(20, 160, G.PREC_BF16) == 1
    assert ctas(333, 1, G.PREC_BF16) == 1  # 16 CTAs' shared memory does not hold the system
    assert ctas(100, 1, G.PREC_BF16, method=G.METHOD_MPPI) == 1  # no system to solve


def test_the_other_cases_of_the_cluster_tests_take_a_cluster():
    shapes = [(30 + 7 * b, 3 + b, 256 + 64 * b) for b in range(6)]
    assert ctas(30, 6, G.PREC_FP32, shapes=shapes) >= 2
    assert ctas(40, 2, G.PREC_BF16) >= 2
    assert ctas(100, 8, G.PREC_BF16, M=10) >= 2
    s = G.Solver(G.pendulum_problem(K=256, sigma0=0.5, seed=7), 2)
    assert G.gnmppi_tune_report(s.h)["solve_ctas"] >= 2
    s.close()


def test_the_longest_horizon_as_one_cta():
    x0, tgt = I.chain_instances(331, 1, 4)
    out = []
    for nt in (512, 256):
        s = G.Solver(G.chain_problem(4, N=320, K=1344, precision=G.PREC_BF16, sigma0=0.2, seed=5), 1)
        G.gnmppi_tune_set(s.h, 1, nt)
        assert G.gnmppi_tune_report(s.h)["solve_ctas"] == (16 if nt == 512 else 1)
        st, U, _ = s.step(x0, tgt, np.full(640, 0.01), np.full(640, 0.2), 0)
        out.append((st, U, s.debug("delta")))
        s.close()
    assert out[0][0] == out[1][0] == G.OK
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])


def test_systems_without_a_factor_on_a_cluster():
    # K' = n at almost no damping: the retries of test_cluster_solve_gpu.py do
    # happen, so factorisations that fail part-way through are among its cases
    x0, tgt = I.chain_instances(4, 8, 10)
    s = G.Solver(G.chain_problem(10, N=100, K=400, precision=G.PREC_BF16, sigma0=0.2, seed=9, lam=1e-9), 8)
    assert G.gnmppi_tune_report(s.h)["solve_ctas"] >= 2
    _, _, rep = s.step(x0, tgt, np.zeros(1600), np.full(1600, 0.2), 0)
    s.close()
    assert any(r.chol_retries > 0 for r in rep)
