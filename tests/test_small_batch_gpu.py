"""A few instances run with other launch shapes than many (cluster Cholesky,
one-sub-tile Gram tiles with a deeper ring, one A sub-tile per contraction
tile): an instance alone gives the bits it gives inside a batch that fills the
chip, in the products and in the step."""
import numpy as np
import pytest

from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# n below and above one 128-row sub-tile and one 256-row tile; nR below and
# above one 2048-column Gram chunk; K' short and long for a contraction tile
@pytest.mark.parametrize("M,N,K,batch", [(4, 60, 512, 170), (5, 90, 700, 170), (10, 110, 2048, 170), (4, 140, 640, 160)])
@pytest.mark.parametrize("prec", [G.PREC_FP32, G.PREC_BF16])
def test_alone_as_in_a_full_batch(M, N, K, batch, prec):
    x0, tgt = I.chain_instances(21, batch, M)
    n = 2 * N
    U, sig = np.full(batch * n, 0.02), np.full(batch * n, 0.2)
    kw = dict(N=N, K=K, precision=prec, sigma0=0.2, seed=12)
    full = G.Solver(G.chain_problem(M, **kw), batch)
    _, V, _ = full.step(x0, tgt, U, sig, 0)
    for b in (0, batch - 1):
        one = G.Solver(G.chain_problem(M, first_instance=b, **kw), 1)
        _, v, _ = one.step(x0[b], tgt[b], U[:n], sig[:n], 0)
        for name in ("PS", "A", "S2", "delta"):
            assert np.array_equal(one.debug(name), full.debug(name, b)), name
        assert np.array_equal(v, V[b * n:(b + 1) * n])
        one.close()
    full.close()
