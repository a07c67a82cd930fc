"""The density and order-parameter read against the populations of the same state.

The read sums the 19 offsets of a node by error-free FP32 transformations (FP64
for FP64 storage); the populations are formed one by one in FP64.  Both describe
the same stored values, so they agree to a few FP64 roundings whatever the
cancellation between the offsets: each population carries at most 3 roundings of
values below |f|, their exact sum and the read's five operations add 8 more, of
2^-53 each: |difference| <= 11 2^-53 sum |f| (component) and twice that for phi.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape,spread", [((5, 3, 4), 1e-2), ((33, 7, 9), 0.9), ((64, 8, 3), 1e-6)])
def test_densities_are_the_sums_of_the_populations(precision, shape, spread):
    from paper_2505_10171_gb300 import lbm
    from paper_2505_10171_gb300 import workloads as W
    nx, ny, nz = shape
    N = nx * ny * nz
    rng = np.random.default_rng(nx)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    # offsets of mixed size and sign, so that partial sums cancel
    F = rng.uniform(-1.0, 1.0, (19, N)) * spread * 10.0 ** rng.uniform(-5.0, 0.0, (19, N))
    phi = rng.uniform(-1.0, 1.0, N)
    f = w[:, None] * (1.0 + F)
    pops = np.concatenate([0.5 * (1 + phi) * f, 0.5 * (1 - phi) * f])
    c = lbm.Context(dict(W.COMMON, nx=nx, ny=ny, nz=nz), precision)
    c.lbm_init_fields(pops=pops)
    fa, fb = c.pops()
    got = c.lbm_read_fields(lbm.FIELD_RHO_A | lbm.FIELD_RHO_B | lbm.FIELD_PHI).reshape(3, N)
    mass = c.lbm_diagnostics()
    c.close()
    eps = 2.0 ** -53
    for n in range(N):
        ra, rb = math.fsum(fa[:, n]), math.fsum(fb[:, n])
        size = np.abs(fa[:, n]).sum() + np.abs(fb[:, n]).sum()
        assert abs(got[0, n] - ra) <= 11 * eps * size
        assert abs(got[1, n] - rb) <= 11 * eps * size
        assert abs(got[2, n] - (ra - rb) / (ra + rb)) <= 22 * eps * size / (ra + rb)
    total = math.fsum(got[0]), math.fsum(got[1])
    assert np.allclose(mass[:2], total, rtol=(11 + N) * eps, atol=0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_zero_and_infinite_densities(precision):
    """A node of zero density has no order parameter; an infinite offset leaves no finite one."""
    from paper_2505_10171_gb300 import lbm
    from paper_2505_10171_gb300 import workloads as W
    c = lbm.Context(dict(W.COMMON, nx=4, ny=3, nz=3), precision)
    rho = np.ones(36)
    rho[5], rho[7] = 0.0, np.inf
    c.lbm_init_fields(np.full(36, 0.25), rho=rho)
    ra, rb, phi = c.lbm_read_fields(lbm.FIELD_RHO_A | lbm.FIELD_RHO_B | lbm.FIELD_PHI).reshape(3, 36)
    c.close()
    ok = np.ones(36, bool)
    ok[[5, 7]] = False
    assert np.allclose(ra[ok], 0.625, rtol=1e-7) and np.allclose(phi[ok], 0.25, rtol=1e-7)
    assert ra[5] == 0.0 and rb[5] == 0.0 and np.isnan(phi[5])
    # F = inf, G = phi inf: f^a = inf, f^b = inf - inf
    assert np.isinf(ra[7]) and np.isnan(rb[7]) and np.isnan(phi[7])
