"""FP64 gradient and curvature, a node per thread in CTAs of one warp: domains whose
node counts leave a part of a warp and of a work item of 64 nodes, alone and
as uneven instances of one context, against the oracle."""
import numpy as np
import pytest

from helpers import oracle_sim
from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def workload(shape, wall, spheres):
    nx, ny, nz = shape
    p = dict(W.COMMON, nx=nx, ny=ny, nz=nz, wall_z0=int(wall), theta_wall_deg=65.0, nu_a=1 / 6, nu_b=1 / 12, mu_s=0.2,
             mu_r=0.1)
    phi = W.drop_phi(nx, ny, nz, (0.45 * nx, 0.5 * ny, 0.4 * nz), max(1.5, min(shape) / 3.0))
    u = 1e-3 * np.random.default_rng(nx + 7 * ny + 31 * nz).standard_normal((3, nx * ny * nz))
    return dict(params=p, phi=phi, u=u, particles=[dict(x=x, R=r, rho_p=2.0, theta_deg=t) for x, r, t in spheres])


DOMAINS = [
    ((3, 1, 7), False, []),                                   # 21 nodes: less than a warp
    ((5, 5, 5), True, []),                                    # 125: a part of the second item
    ((11, 9, 13), False, []),                                 # 1287 = 20 items and 7 nodes
    # two spheres that share boundary nodes, one across the periodic box
    ((19, 17, 15), True, [((6.0, 8.2, 6.5), 3.1, 40.0), ((12.3, 8.0, 6.1), 3.1, 120.0)]),
]


@pytest.mark.parametrize("which", [[0], [1], [2], [3], [3, 0, 2, 1]])
def test_populations_match_the_oracle(which):
    """Absolute 1e-12 of the offsets after five steps (offsets of order 1, rounding of
    some 1e2 operations a node and step at 1.1e-16)."""
    from paper_2505_10171_gb300 import lbm
    ws = [workload(*DOMAINS[k]) for k in which]
    c = lbm.Context([w["params"] for w in ws], "fp64")
    for k, w in enumerate(ws):
        if w["particles"]:
            c.lbm_add_particles(w["particles"], inst=k)
        c.lbm_init_fields(w["phi"], None, w["u"], inst=k)
    c.lbm_step(5)
    for k, w in enumerate(ws):
        s = oracle_sim(w)
        s.step(5)
        own = s.owner()
        assert (c.owner(k) == own).all()
        for g, f in zip(c.pops(k), s.pops()):
            assert np.abs(g - f)[:, own == 0].max() <= 1e-12
    c.close()
