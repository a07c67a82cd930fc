"""The boundary-bit pass scans only the cube around a particle that its surface can
reach: radii around whole and half numbers, whose reach (radius + move + 1.52)
crosses a node, on spheres that move through the periodic box, against the oracle
(owners exactly, populations to 1e-12 as everywhere in FP64)."""
import numpy as np
import pytest

from helpers import gpu_ctx, oracle_sim
from test_gpu_grad_fp64 import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


@pytest.mark.parametrize("radius", [1.47, 1.5, 2.45, 2.49, 3.4, 3.48, 3.99])
def test_moving_spheres_match_the_oracle(radius):
    w = workload((20, 17, 19), False, [((0.3, 16.8, 18.6), radius, 60.0), ((10.5, 8.0, 9.99), radius, 100.0)])
    for q, v in zip(w["particles"], ((0.11, -0.09, 0.1), (-0.08, 0.12, -0.1))):
        q["v"] = v
    s, c = oracle_sim(w), gpu_ctx(w, "fp64")
    for _ in range(4):
        s.step(3)
        c.lbm_step(3)
        own = s.owner()
        assert (c.owner() == own).all()
        for g, f in zip(c.pops(), s.pops()):
            assert np.abs(g - f)[:, own == 0].max() <= 1e-12
    c.close()
