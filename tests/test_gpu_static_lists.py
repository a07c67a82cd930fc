"""The first step's lists of nodes next to walls, when a call runs out of memory
between the two: the next call builds them anew for the solid map of then."""
import numpy as np
import pytest

from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N = 288


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def grid_mask(every):
    m = np.zeros((N, N, N), dtype=np.uint8)
    m[::every, ::every, ::every] = 1
    return m


def test_lists_after_out_of_memory():
    """Single solid nodes, every third: 7 MB of solid nodes, 127 MB of fluid ones next to
    them, with 64 MB free.  Then every second: 24 MB and 150 MB."""
    import torch
    from paper_2505_10171_gb300 import lbm
    params, phi = dict(W.COMMON, nx=N, ny=N, nz=N, body_force_a=(1e-6, 0.0, 0.0)), np.full(N ** 3, 1.0)

    def context(every):
        c = lbm.Context(params, "fp16")
        c.lbm_set_solid_mask(grid_mask(every))
        c.lbm_init_fields(phi, None, None)
        return c

    c = context(3)
    torch.cuda.init()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - (64 << 20), dtype=torch.uint8, device="cuda")
    with pytest.raises(lbm.LbmError) as err:
        c.lbm_step(1)
    assert lbm.STATUS_NAMES[err.value.status] == "LBM_ERR_OOM"
    del hog
    torch.cuda.empty_cache()
    c.lbm_set_solid_mask(grid_mask(2))
    c.lbm_init_fields(phi, None, None)
    c.lbm_step(3)
    got = np.asarray(c.lbm_read_fields(lbm.FIELD_RHO_A))
    c.close()
    c = context(2)
    c.lbm_step(3)
    want = np.asarray(c.lbm_read_fields(lbm.FIELD_RHO_A))
    c.close()
    assert np.isfinite(want).all() and np.array_equal(got, want)
