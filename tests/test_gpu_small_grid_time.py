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


LARGE = (768, 384)


@pytest.mark.parametrize("name,make,prep,limit", [
    # the smallest steps against a step of one full wave of tiles: 18 us with wide blocks, 29 with 128 threads, of 49
    ("no body", lambda: _open(64, 64), None, 0.48),
    ("cylinder", lambda: W.cylinder_m02_re40(64, 64, precision=W.PREC_FP32_BULK), None, 0.67),
    ("cylinder 256 x 128", lambda: W.cylinder_m02_re40(256, 128, precision=W.PREC_FP32_BULK), None, 0.83),
    ("no body, persistent", lambda: _open(64, 64), lambda c: c.use_persistent(1), 0.66),
    ("no body 512 x 256, persistent", lambda: _open(512, 256), lambda c: c.use_persistent(1), 1.10),
])
def test_small_steps(ibm, name, make, prep, limit):  # noqa: F811
    large = _us(ibm, _open(*LARGE), lambda c: c.stage_launches(2))
    small = _us(ibm, make(), prep, 200)
    print("%s %.1f us, %d x %d %.1f us: %.2f" % ((name, small) + LARGE + (large, small / large)))
    assert small <= limit * large, (small, large)


@pytest.mark.parametrize("nx,ny,limit", [(64, 64, 0.32), (512, 256, 0.66)])
def test_small_dual_steps(ibm, nx, ny, limit):  # noqa: F811
    """Dual time, ten sub-iterations, against 768 x 384 (1600 us): 417 and 829 us with wide blocks, 625 and 1445 with two
    cells per thread in turn."""
    kw = dict(precision=W.PREC_FP32_BULK, subiters=10)
    large = _us(ibm, W.naca0012_a5_m0001(*LARGE, **kw), n=4)
    small = _us(ibm, W.naca0012_a5_m0001(nx, ny, **kw), n=4)
    print("%d x %d %.0f us, %d x %d %.0f us: %.2f" % ((nx, ny, small) + LARGE + (large, small / large)))
    assert small <= limit * large, (small, large)
