"""The autotuner's choice where the gradient pass marches: never worse than the planned chunk."""
import numpy as np
import pytest

from paper_2505_10171_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def test_planned_chunk_is_kept_where_it_is_fastest():
    """32 x 8 columns, 4096 planes: chunks of 9 planes are 456 CTAs, three for each of 152
    SMs; 8, 16 and 32 planes take 5, 14 and 40% longer a step."""
    from paper_2505_10171_gb300 import lbm
    c = lbm.Context(dict(W.COMMON, nx=32, ny=8, nz=4096), "fp32")
    c.lbm_init_fields(np.full(32 * 8 * 4096, -1.0), None, None)
    _, zchunks, _ = c.lbm_autotune(1000)
    c.close()
    assert zchunks == [9]
