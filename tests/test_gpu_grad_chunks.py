"""The marching gradient pass at the edges of its tiles and of requested z-chunks:
domains in a context past the line, against the node-per-thread form of the
same domains alone."""
import numpy as np
import pytest

from paper_2505_10171_gb300 import workloads as W
from test_gpu_grad_fp64 import workload

pytestmark = pytest.mark.gpu

# columns and rows around multiples of the tiles (32 by 8 and 32 by 16), walls,
# spheres across the tiles' edges and the periodic box
DOMAINS = [
    ((31, 7, 9), True, []),
    ((33, 9, 11), False, []),
    ((32, 8, 5), False, []),
    ((64, 16, 12), True, [((20.3, 8.1, 5.2), 3.2, 150.0), ((32.5, 7.9, 4.7), 3.1, 60.0)]),
    ((65, 17, 13), True, [((31.6, 15.8, 6.0), 3.4, 120.0)]),
    ((1, 3, 40), False, []),
]
FILLER = dict(W.COMMON, nx=128, ny=128, nz=49)


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_10171_gb300 import build
    build.build()


def run(precision, zchunk=None):
    from paper_2505_10171_gb300 import lbm
    ws = [workload(*d) for d in DOMAINS]
    c = lbm.Context([w["params"] for w in ws] + ([FILLER] if zchunk is not None else []), precision)
    for k, w in enumerate(ws):
        if w["particles"]:
            c.lbm_add_particles(w["particles"], inst=k)
        c.lbm_init_fields(w["phi"], None, w["u"], inst=k)
    if zchunk is not None:
        c.lbm_init_fields(np.full(128 * 128 * FILLER["nz"], -1.0), None, None, inst=len(ws))
        c.lbm_set_fluid_kernel(lbm.FORM_PLAIN, 0, zchunk)
    c.lbm_step(5)
    out = [np.concatenate([np.asarray(p).ravel() for p in c.pops(k)]) for k in range(len(ws))]
    c.close()
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
def test_every_chunk_same_bits(precision):
    want = run(precision)
    for zchunk in (0, 1, 2, 5, 64):
        for d, a, b in zip(DOMAINS, want, run(precision, zchunk)):
            assert np.isfinite(a).all() and np.array_equal(a, b), (zchunk, d[0])
