"""The cluster Cholesky (several CTAs per instance) against the single-CTA
kernel: the same operations on every matrix entry in the same order, so one
iteration gives the same bits, whatever the cluster size, the number of
16-wide panels and the last panel's width, and also where factorisations fail
and are retried."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def both(prob, batch, shapes, x0, tgt, U, sig, inject=0):
    out = []
    for nt in (512, 256):  # 512: one cluster (or CTA) per instance; 256: one CTA, two per SM
        s = G.Solver(prob, batch, shapes)
        G.gnmppi_tune_set(s.h, 1, nt)
        if inject:
            G.gnmppi_debug_inject(s.h, inject, 0)
        st, V, rep = s.step(x0, tgt, U, sig, 0)
        d = [s.debug("delta", b) for b in range(batch)]
        out.append((st, V, np.concatenate(d), [(r.status, r.chol_retries, r.jac_mode_used, r.j_star) for r in rep]))
        s.close()
    (s0, U0, d0, r0), (s1, U1, d1, r1) = out
    assert s0 == s1 and r0 == r1
    assert np.array_equal(d0, d1) and np.array_equal(U0, U1)
    return r0


# n = 2 N: two panels and a bit, a full last panel, one row in it, the
# longest horizon of the sweep; batches from one cluster to more than fit
@pytest.mark.parametrize("N,batch", [(17, 1), (24, 3), (41, 2), (100, 1), (100, 9), (100, 30), (100, 70), (200, 1),
                                     (200, 12), (333, 1)])
@pytest.mark.parametrize("prec", [G.PREC_BF16, G.PREC_FP64])
def test_bitwise_as_one_cta(N, batch, prec):
    if prec == G.PREC_FP64 and N * batch > 400:
        pytest.skip("the FP64 products of this size are slow and add nothing to the factorisation")
    M = 4
    x0, tgt = I.chain_instances(11 + N, batch, M)
    K = 4 * N + 64
    prob = G.chain_problem(M, N=N, K=K, precision=prec, sigma0=0.2, seed=5)
    both(prob, batch, None, x0, tgt, np.full(batch * 2 * N, 0.01), np.full(batch * 2 * N, 0.2))


def test_bitwise_uneven_batch_and_pendulum():
    shapes = [(30 + 7 * b, 3 + b, 256 + 64 * b) for b in range(6)]
    x0 = np.concatenate([I.chain_instances(b, 1, M)[0].ravel() for b, (_, M, _) in enumerate(shapes)])
    tgt = np.concatenate([I.chain_instances(b, 1, M)[1].ravel() for b, (_, M, _) in enumerate(shapes)])
    n = sum(2 * s[0] for s in shapes)
    prob = G.chain_problem(3, N=30, K=256, precision=G.PREC_FP32, sigma0=0.2, seed=6)
    both(prob, 6, shapes, x0, tgt, np.zeros(n), np.full(n, 0.2))
    prob = G.pendulum_problem(K=256, sigma0=0.5, seed=7)
    both(prob, 2, None, I.pendulum_x0(3, 2), None, np.zeros(100), np.full(100, 0.5))


@pytest.mark.parametrize("kind", [1, 2])
def test_failed_factorisations_take_the_same_ladder(kind):
    x0, tgt = I.chain_instances(3, 2, 4)
    prob = G.chain_problem(4, N=40, K=256, precision=G.PREC_BF16, sigma0=0.2, seed=8)
    reps = both(prob, 2, None, x0, tgt, np.zeros(160), np.full(160, 0.2), inject=kind)
    assert all(r[0] == (G.E_NOT_PD if kind == 2 else G.OK) for r in reps)


def test_indefinite_systems_are_retried_alike():
    # K' = n: S is nearly singular and the reduced-precision Gram's rounding
    # leaves some systems without a factor at the stated damping
    x0, tgt = I.chain_instances(4, 8, 10)
    prob = G.chain_problem(10, N=100, K=400, precision=G.PREC_BF16, sigma0=0.2, seed=9, lam=1e-9)
    both(prob, 8, None, x0, tgt, np.zeros(1600), np.full(1600, 0.2))
