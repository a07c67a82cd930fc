"""FP64 wall velocity and momentum exchange from one lever per node where all its
links have the same periodic image, per link where they may not: spheres that
spin and move in boxes of which they fill little, most, and all that is accepted
(their surface then reaches half the period, where images change along a link),
against the oracle: populations to 1e-12, records to 1e-9 as everywhere in FP64."""
import numpy as np
import pytest

from helpers import gpu_ctx, oracle_sim
from test_gpu_grad_fp64 import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


@pytest.mark.parametrize("shape,radius", [((24, 20, 22), 3.7), ((12, 13, 14), 4.6), ((12, 13, 14), 4.95),
                                          ((11, 24, 23), 4.45), ((23, 11, 12), 4.4)])
def test_links_match_the_oracle(shape, radius):
    w = workload(shape, False, [((0.37 * shape[0], 0.9 * shape[1], 0.03 * shape[2]), radius, 75.0)])
    w["particles"][0].update(v=(0.02, -0.03, 0.01), w=(4e-3, -3e-3, 5e-3))
    s, c = oracle_sim(w), gpu_ctx(w, "fp64")
    s.step(6)
    c.lbm_step(6)
    own = s.owner()
    assert (c.owner() == own).all()
    for g, f in zip(c.pops(), s.pops()):
        assert np.abs(g - f)[:, own == 0].max() <= 1e-12
    assert np.abs(c.lbm_particle_forces() - s.particles()).max() <= 1e-9
    c.close()
