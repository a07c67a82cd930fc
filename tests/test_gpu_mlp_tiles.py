"""The network's row and gradient kernels at the edges of their tiles (needs a GB300).

Rows go 128 to a CTA and gradients sum over chunks of 64 rows, two stages in
turn: one row, one below, at and above a tile, and batches that end inside the
first, second and third chunk.  Every row is independent, so a batch gives the
bits of its rows alone; a gradient over n rows is the mean of the rows' own, up
to the rounding of its parts: BF16 deltas (relative 2^-8 each, n of them
averaged) and FP32 sums, held to the oracle's 2e-2 bar of the gradient test.
"""
import numpy as np
import pytest

from helpers import rel_l2
from oracle import mlp_oracle as M
from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def net():
    from paper_2505_10171_gb300 import build, lbm
    build.build()
    c = lbm.Context(dict(W.COMMON, nx=16, ny=16, nz=16, store_velocity=1), "fp32")
    th = M.init_params(31)
    c.lbm_surrogate_load(th)
    rng = np.random.default_rng(32)
    X = rng.normal(size=(4300, M.N_IN)).astype(np.float32)
    T = rng.normal(scale=0.5, size=(4300, M.N_OUT)).astype(np.float32)
    yield c, th.astype(np.float32).astype(np.float64), X, T
    c.close()


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 4096, 4097])
def test_rows_of_a_batch_are_independent(net, n):
    c, th, X, _ = net
    Y = c.lbm_surrogate_predict(X[:n])
    assert rel_l2(Y, M.forward(th, X[:n], bf=True)[0]) < 2e-2
    for r in {0, n // 2, n - 1}:
        assert np.array_equal(c.lbm_surrogate_predict(X[r:r + 1])[0], Y[r])


@pytest.mark.parametrize("n", [1, 7, 63, 64, 65, 128, 129, 191, 193, 4096])
def test_gradient_at_chunk_edges(net, n):
    c, th, X, T = net
    g, loss = c.lbm_surrogate_gradient(X[:n], T[:n])
    lo, go = M.loss_and_grad(th, X[:n], T[:n], bf=True)
    assert abs(loss - lo) <= 5e-3 * lo
    o = 0
    for name, shp in M.SHAPES:
        k = int(np.prod(shp))
        assert rel_l2(g[o:o + k], go[o:o + k]) < 2e-2, name
        o += k
