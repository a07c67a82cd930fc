"""Network rows 32 to a CTA, eight to a warp, and gradients with eight stages of 64
rows in flight (needs a GB300): batches that end at, below and above a group of
eight, a tile, the last stage and the first refilled one, against the oracle in
the bars of its BF16 form (2e-2 relative in the outputs and gradients, whose
deltas are BF16: 2^-8 each; 5e-3 in the loss)."""
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
    th = M.init_params(41)
    c.lbm_surrogate_load(th)
    rng = np.random.default_rng(42)
    X = rng.normal(size=(1100, M.N_IN)).astype(np.float32)
    T = rng.normal(scale=0.5, size=(1100, M.N_OUT)).astype(np.float32)
    yield c, th.astype(np.float32).astype(np.float64), X, T
    c.close()


@pytest.mark.parametrize("n", [2, 8, 9, 32, 33, 40, 511, 512, 513, 576, 577, 1025])
def test_tile_and_stage_edges(net, n):
    c, th, X, T = net
    Y = c.lbm_surrogate_predict(X[:n])
    assert rel_l2(Y, M.forward(th, X[:n], bf=True)[0]) < 2e-2
    assert np.array_equal(c.lbm_surrogate_predict(X[n - 1:n])[0], Y[-1])
    g, loss = c.lbm_surrogate_gradient(X[:n], T[:n])
    lo, go = M.loss_and_grad(th, X[:n], T[:n], bf=True)
    assert abs(loss - lo) <= 5e-3 * lo
    o = 0
    for name, shp in M.SHAPES:
        k = int(np.prod(shp))
        assert rel_l2(g[o:o + k], go[o:o + k]) < 2e-2, name
        o += k
