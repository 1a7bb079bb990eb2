"""FP64 stages at the grid sizes where the tile shape changes (16 x 16, 16 x 8 and 8 x 8 cells, by the work of the
fullest SM) and at ragged edges of each, against the FP64 oracle: state within 1e-10 relative, the repository's FP64
bar, or the dual-time bar of the oracle's own conditioning."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from flowmetrics import fp64_bar
from test_gpu_dual import _err, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

GRIDS = [(160, 240), (151, 235), (257, 131), (129, 97), (64, 64), (67, 41), (8, 8), (9, 11)]


def _spec(nx, ny, **kw):
    h = 12.0 / nx
    return W.case_spec(W.cylinder(64, 2.0) if nx > 16 else None, nx, ny, (-4.0, 8.0, -0.5 * ny * h, 0.5 * ny * h), 0.3,
                       200.0, W.FAR, **kw)


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("scheme", [W.SCHEME_WENO5, W.SCHEME_TVD2])
def test_explicit(ibm, orc, nx, ny, scheme):  # noqa: F811
    spec = _spec(nx, ny, scheme=scheme)
    rng = np.random.default_rng(nx)
    g, o = ibm.Case(spec), orc.Case(spec)
    a = o.state() * (1.0 + 0.01 * rng.uniform(-1.0, 1.0, (4, ny, nx)))
    g.set_state(a)
    o.set_state(a)
    g.step(3)
    o.step(3)
    e = _err(g.state(), o.state(), o.tags())
    assert e <= 1e-10, e


@pytest.mark.parametrize("nx,ny", [(151, 235), (257, 131), (67, 41)])
def test_dual(ibm, orc, nx, ny):  # noqa: F811
    spec = dict(_spec(nx, ny, time_scheme=W.TIME_DUAL, dt_phys=0.5 * 12.0 / nx, subiters=4), mach=0.01)
    g, o = ibm.Case(spec), orc.Case(spec)
    g.step(3)
    o.step(3)
    e, bar = _err(g.state(), o.state(), o.tags()), fp64_bar(orc, spec, 3)
    assert e <= bar, (e, bar)
