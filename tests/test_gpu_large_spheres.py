"""Spheres whose momentum exchange has more partial sums than one warp of the DEM
kernel takes (96, 64 nodes each of a cube of 2 R + 5 a side), against the oracle."""
import numpy as np
import pytest

from helpers import gpu_ctx, oracle_sim
from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


@pytest.mark.parametrize("R,blocks", [(6.0, 77), (6.6, 108), (11.0, 308)])
def test_forces_match_the_oracle(R, blocks):
    """2e-12 of 1 or the value where that is larger: some 8000 links with terms of up to
    1.2 (torque, R = 11) at 1.1e-16 each."""
    n = 32
    assert -(-(2 * int(np.ceil(R)) + 5) ** 3 // 64) == blocks
    p = dict(W.COMMON, nx=n, ny=n, nz=n, wall_z0=0, nu_a=1 / 6, nu_b=1 / 12, body_force_a=(1e-5, 0.0, 0.0))
    w = dict(params=p, phi=W.drop_phi(n, n, n, (8.0, 16.0, 16.0), 9.0),
             particles=[dict(x=(19.3, 15.8, 16.4), R=R, rho_p=2.0, theta_deg=70.0, v=(1e-2, -5e-3, 2e-3),
                             w=(1e-3, 2e-3, -1e-3))])
    sim = oracle_sim(w)
    sim.step(4)
    c = gpu_ctx(w, "fp64")
    c.lbm_step(4)
    got, want = c.lbm_particle_forces()[0], sim.particles()[0]
    c.close()
    assert np.abs(want[:12]).max() > 0.0
    assert (np.abs(got[:12] - want[:12]) <= 2e-12 * np.maximum(1.0, np.abs(want[:12]))).all()
