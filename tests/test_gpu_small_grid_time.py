"""Steps of small grids last as long as the chain of work of one tile.  Their time against the time of a larger grid on the
same GPU, so that a longer chain shows: a limit stands half way between the chain that it is to keep and the one that
was found too long."""
import time

import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_bulk import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _us(ibm, spec, prep=None, n=60):  # noqa: F811
    c = ibm.Case(spec)
    if prep:
        prep(c)
    c.step(4)
    c.sync()
    best = 1e9
    for _ in range(12):
        t = time.perf_counter()
        c.step(n)
        c.sync()
        best = min(best, (time.perf_counter() - t) / n)
    c.close()
    return 1e6 * best


def _open(nx, ny, **kw):
    return W.case_spec(None, nx, ny, (0.0, nx / 32.0, 0.0, ny / 32.0), 0.3, 100.0, W.FAR, precision=W.PREC_FP32_BULK, **kw)


def test_body_tiles(ibm):  # noqa: F811
    """A body tile's node rebuild beside the other tiles' work: the quadratic form at 1024 x 512, 1.31 times the step
    without a body with every node walked through twice, 1.16 with each class of nodes walked through once."""
    quad = _us(ibm, W.cylinder_m02_re40(1024, 512, precision=W.PREC_FP32_BULK, ib_interp=W.INTERP_QUADRATIC))
    none = _us(ibm, _open(1024, 512))
    print("quadratic %.1f us, no body %.1f us" % (quad, none))
    assert quad <= 1.235 * none, (quad, none)
