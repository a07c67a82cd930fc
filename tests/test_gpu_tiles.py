"""FP64 parity with the oracle at the edges of the marching tiles (needs a GB300).

The order-parameter and gradient passes cover 32-node columns of 4 to 16 rows in
z-chunks chosen by the grid's size; nodes next to solids take their bounced
offsets and marks from lists in node order.  Sizes one below, at and above the
tile's edges, single rows and planes, walls on both sides of a chunk, spheres
across tile borders and the periodic box.  Bar: the FP64 parity bar of the
whole path, 1e-12 on every population.
"""
import numpy as np
import pytest

from helpers import gpu_ctx, oracle_sim, rel_l2
from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def workload(shape, wall, spheres):
    nx, ny, nz = shape
    p = dict(W.COMMON, nx=nx, ny=ny, nz=nz, wall_z0=int(wall), wall_velocity=(2e-3, -1e-3, 0.0) if wall else (0, 0, 0),
             theta_wall_deg=70.0, nu_a=1 / 6, nu_b=1 / 20, mu_s=0.3, mu_r=0.1, body_force_a=(1e-6, 2e-6, -1e-6))
    R = max(1.5, min(shape) / 3.0)
    phi = W.drop_phi(nx, ny, nz, (0.4 * nx, 0.5 * ny, 0.45 * nz), R)
    rng = np.random.default_rng(nx * ny + nz)
    u = 1e-3 * rng.standard_normal((3, nx * ny * nz))
    parts = [dict(x=x, R=r, rho_p=2.5, theta_deg=t, v=(0.01, -0.02, 0.015), w=(1e-3, 2e-3, -1e-3))
             for x, r, t in spheres]
    return dict(params=p, phi=phi, u=u, particles=parts)


CASES = [
    ((31, 7, 5), False, []), ((33, 9, 3), True, []), ((1, 17, 33), False, []), ((64, 1, 9), True, []),
    ((32, 16, 2), False, []), ((65, 15, 12), True, []), ((5, 33, 67), True, []),
    # spheres at tile borders (x = 32, y = 8 and 16) and across the periodic box
    ((40, 20, 18), True, [((32.2, 8.1, 6.0), 3.6, 50.0), ((10.0, 16.3, 8.5), 3.2, 110.0)]),
    ((34, 18, 17), False, [((0.4, 17.6, 16.7), 4.0, 80.0)]),
]


@pytest.mark.parametrize("shape,wall,spheres", CASES)
def test_fp64_parity_at_tile_edges(shape, wall, spheres):
    w = workload(shape, wall, spheres)
    s = oracle_sim(w)
    s.step(6)
    fa, fb = s.pops()
    fl = s.owner() == 0
    c = gpu_ctx(w, "fp64")
    c.lbm_step(6)
    ga, gb = c.pops()
    assert (c.owner() == s.owner()).all()
    err = max(np.abs(ga[:, fl] - fa[:, fl]).max(), np.abs(gb[:, fl] - fb[:, fl]).max())
    if spheres:
        assert np.abs(c.lbm_particle_forces() - s.particles()).max() <= 1e-9
    c.close()
    assert err <= 1e-12, err


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-4), ("fp16", 2e-3), ("bf16", 2e-3)])
@pytest.mark.parametrize("case", [1, 5, 7, 8])
def test_other_storage_at_tile_edges(case, precision, tol):
    """rho and phi of the other storage types within the path's bars (1e-4, 2e-3) of the oracle."""
    w = workload(*CASES[case])
    s = oracle_sim(w)
    s.step(6)
    f, own = s.fields(), s.owner()
    c = gpu_ctx(w, precision)
    c.lbm_step(6)
    g, gown = c.fields(), c.owner()
    c.close()
    fl = (own == 0) & (gown == 0)
    assert (own != gown).sum() <= 4
    assert rel_l2((g["rho_a"] + g["rho_b"])[fl], (f["rho_a"] + f["rho_b"])[fl]) <= tol
    assert rel_l2(g["phi"][fl], f["phi"][fl]) <= tol
