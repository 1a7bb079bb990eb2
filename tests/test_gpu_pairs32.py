"""FP32-bulk stages on grids at the edges of the 16 x 16 tiles (interior tiles, tiles with domain halos, tiles cut by
the grid, one tile, no interior tile), against the FP64 oracle.  Bar: a stage's residual has about 200 dependent FP32
roundings of 2^-24, 1.2e-5 of the perturbations' scale if they all added up; three steps are nine stages: 1.1e-4."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_bulk import _compare, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

BAR = 1.1e-4
GRIDS = [(16, 16), (17, 16), (16, 31), (32, 33), (48, 48), (49, 47), (64, 64), (67, 41), (151, 113)]


def _spec(nx, ny, p, **kw):
    h = 12.0 / nx
    return W.case_spec(W.cylinder(64, 2.0) if nx >= 64 else None, nx, ny, (-4.0, 8.0, -0.5 * ny * h, 0.5 * ny * h),
                       kw.pop("mach", 0.3), 200.0, W.FAR, precision=p, **kw)


def _run(ibm, orc, nx, ny, **kw):  # noqa: F811
    rng = np.random.default_rng(nx)
    g, o = ibm.Case(_spec(nx, ny, W.PREC_FP32_BULK, **kw)), orc.Case(_spec(nx, ny, W.PREC_FP64, **kw))
    a = o.state() * (1.0 + 0.01 * rng.uniform(-1.0, 1.0, (4, ny, nx)))
    g.set_state(a)
    o.set_state(a)
    g.step(3)
    o.step(3)
    err = _compare(g, o)
    assert max(err.values()) <= BAR, err


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("scheme", [W.SCHEME_WENO5, W.SCHEME_TVD2])
@pytest.mark.parametrize("mach", [0.3, 1.5])
def test_explicit(ibm, orc, nx, ny, scheme, mach):  # noqa: F811
    _run(ibm, orc, nx, ny, scheme=scheme, mach=mach)


@pytest.mark.parametrize("nx,ny", [(17, 16), (48, 48), (67, 41), (151, 113)])
def test_dual(ibm, orc, nx, ny):  # noqa: F811
    _run(ibm, orc, nx, ny, time_scheme=W.TIME_DUAL, dt_phys=0.5 * 12.0 / nx, subiters=4)
