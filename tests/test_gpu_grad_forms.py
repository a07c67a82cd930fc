"""FP32 gradient pass: a domain in a small context (a node per thread) and beside a
domain that takes the context past the line (marching tiles) has the same bits."""
import numpy as np
import pytest

from paper_2505_10171_gb300 import workloads as W
from test_gpu_grad_fp64 import DOMAINS, workload

pytestmark = pytest.mark.gpu
NODES_MAX = 768 * 1024


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("which", [[0], [1], [2], [3], [3, 0, 2, 1]])
def test_both_forms_same_bits(which, precision):
    from paper_2505_10171_gb300 import lbm
    ws = [workload(*DOMAINS[k]) for k in which]
    nodes = sum(w["phi"].size for w in ws)
    big = dict(W.COMMON, nx=128, ny=128, nz=-(-(NODES_MAX + 1 - nodes) // (128 * 128)))
    out = []
    for extra in ([], [big]):
        c = lbm.Context([w["params"] for w in ws] + extra, precision)
        for k, w in enumerate(ws):
            if w["particles"]:
                c.lbm_add_particles(w["particles"], inst=k)
            c.lbm_init_fields(w["phi"], None, w["u"], inst=k)
        if extra:
            c.lbm_init_fields(np.full(128 * 128 * big["nz"], -1.0), None, None, inst=len(ws))
        c.lbm_step(5)
        out.append([np.concatenate([np.asarray(p).ravel() for p in c.pops(k)]) for k in range(len(ws))])
        c.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)
