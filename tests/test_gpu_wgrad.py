"""GPU test of the tensor-core weight gradients at the edges of their tiles
(8 x 16 x 4 points): one point below and above a tile along every axis, grids
smaller than a tile, several tiles per CTA and more tiles than one
accumulation window (4), with more samples allocated than used."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# BF16 operands (relative rounding 2^-9 each) through three layers; the
# gradients' own sums are FP32.  A missing or doubled row, plane or shift of a
# tile moves a tensor by 1 / n or more (n <= 33), above this bound.
GRAD_TOL = 2e-2


@pytest.mark.parametrize("n,batch,parts", [(4, 1, 0), (5, 3, 2), (7, 1, 0), (9, 2, 1), (15, 1, 3),
                                           (16, 1, 1), (17, 2, 0), (20, 1, 5), (33, 1, 11)])
def test_weight_gradients_at_tile_edges(n, batch, parts):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    p = ocnn.init_params(21)
    p["W3"] *= 10.0
    rng = np.random.default_rng(n)
    for k in ("b1", "b2", "b3"):
        p[k] = 0.05 * rng.standard_normal(p[k].shape)
    xs = rng.standard_normal((batch, 5, n, n, n))
    tgt = rng.standard_normal((batch, 5, n, n, n))
    net = gbfd.CNN(n, batch=batch + 1)
    net.set_params(p)
    net.set_norm(np.zeros(5), np.ones(5), np.ones(5))
    net.set_option(gbfd.GBFD_CNN_OPT_WGRAD_PARTS, parts)
    g, _ = net.gradients(torch.from_numpy(xs.astype(np.float32)).cuda(),
                         torch.from_numpy((xs + tgt).astype(np.float32)).cuda())
    _, ref = ocnn.loss_and_grads(list(xs), list(tgt), p)
    got = net.unflatten(g)
    for k in ref:
        err = np.linalg.norm((got[k] - ref[k]).ravel()) / np.linalg.norm(ref[k].ravel())
        assert err < GRAD_TOL, (k, err)
    net.close()
