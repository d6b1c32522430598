"""The network's products at the edges of their tiles: output tiles of 32, 64
and 128 columns (batches that make the launch wide enough), ragged row and
column remainders, batches around one tile and one k-block, one and three
controls per scale, and a second call at another batch size on the same handle.
Against the FP64 oracle within the three-pass products' FP32-level accuracy
(2^-17 per operand, a few products deep)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2512_04579_gb300 import gnmppi as G

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300)


def net(dims, seed):
    rng = np.random.default_rng(seed)
    ps = []
    for a, b in zip(dims[:-1], dims[1:]):
        ps += [rng.normal(0, 1.0 / math.sqrt(a), size=a * b), rng.normal(0, 0.1, size=b)]
    return np.concatenate(ps).astype(np.float32).astype(np.float64), rng


# (widths, nu, batches on one handle): one sample; one k-block of batch and one
# past it; one row tile and one past it; enough tiles for 64 and 128 columns
@pytest.mark.parametrize("dims,nu,batches", [
    ([3, 5, 4], 1, (1, 2)),
    ([7, 33, 31, 12], 2, (1, 64, 65)),
    ([36, 64, 129, 32], 3, (127, 128, 129)),
    ([5, 20], 1, (31, 33)),
    ([40, 256, 96, 300], 2, (700, 4000, 12000)),
])
def test_products_at_tile_edges(dims, nu, batches):
    params, rng = net(dims, len(dims) + nu)
    nmu = dims[-1] // (nu + 1) * nu
    xm, xs = np.zeros(dims[0]), np.ones(dims[0])
    m = G.Mlp(dims, nu=nu, weights_bf16=False, max_batch=max(batches))
    m.set_params(params)
    m.set_normalization(xm, xs, 1.0)
    for B in tuple(batches) + (batches[0],):
        X, T = rng.normal(size=(B, dims[0])), rng.normal(size=(B, nmu))
        assert rel(m.forward(X), O.mlp_forward(dims, params, xm, xs, X)) < 3e-5
        loss, g = m.loss_grad(X, T)
        lo, go = O.mlp_loss_grad(dims, params, xm, xs, X, T, nu)
        assert loss == pytest.approx(lo, rel=3e-5)
        off = 0
        for a, b in zip(dims[:-1], dims[1:]):
            for size in (a * b, b):
                assert rel(g[off:off + size], go[off:off + size]) < 3e-4, (B, a, b, size)
                off += size
    m.close()
