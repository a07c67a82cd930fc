"""Order parameter of narrow and thin domains (a node per thread) against the same
domain repeated along its periodic axes until it fills the marching tiles."""
import numpy as np
import pytest

from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def run(shape, times, wall, spheres, precision):
    from paper_2505_10171_gb300 import lbm
    nx, ny, nz = shape
    p = dict(W.COMMON, nx=nx * times[0], ny=ny * times[1], nz=nz, wall_z0=int(wall), theta_wall_deg=110.0, nu_a=1 / 6,
             nu_b=1 / 12)
    rng = np.random.default_rng(nx + 7 * ny + 31 * nz)
    rep = lambda a: np.tile(a.reshape(nz, ny, nx), (1, times[1], times[0])).ravel()  # noqa: E731
    c = lbm.Context(p, precision)
    if spheres:
        c.lbm_add_particles([dict(x=(x + nx * i, y + ny * j, z), R=R, rho_p=2.0, theta_deg=60.0, kinematic=1)
                             for x, y, z, R in spheres for i in range(times[0]) for j in range(times[1])])
    c.lbm_init_fields(rep(W.drop_phi(nx, ny, nz, (0.4 * nx, 0.5 * ny, 0.4 * nz), max(1.5, 0.3 * min(shape)))), None,
                      np.stack([rep(1e-3 * rng.standard_normal(nx * ny * nz)) for _ in range(3)]))
    c.lbm_step(6)
    out = np.concatenate([np.asarray(a) for a in c.pops()]).reshape(38, nz, ny * times[1], nx * times[0])[:, :, :ny, :nx]
    c.close()
    return out


@pytest.mark.parametrize("shape,times,wall,spheres", [
    ((8, 8, 20), (4, 1), False, []),
    ((16, 4, 33), (2, 2), True, []),
    ((1, 1, 50), (32, 8), False, []),
    ((20, 6, 7), (8, 4), True, []),
    ((16, 16, 20), (2, 1), True, [(8.25, 7.5, 5.25, 3.0)]),
])
@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
def test_narrow_as_repeated(shape, times, wall, spheres, precision):
    """FP32: the same bits.  16-bit storage sums the two forms in different groups: a unit
    of the stored type's last place per step."""
    a, b = run(shape, (1, 1), wall, spheres, precision), run(shape, times, wall, spheres, precision)
    assert np.isfinite(a).all()
    if precision == "fp32":
        assert np.array_equal(a, b)
    else:
        ulp = {"fp16": 2.0 ** -11, "bf16": 2.0 ** -8}[precision]
        assert np.abs(a - b).max() <= 6 * ulp * np.abs(b).max()
