"""FP32-bulk tiles convert a cell to primitives with the same rounding wherever they do it: with a field that does not vary
along x and zero-gradient ends, every column of cells stays the same bit for bit, in tiles at the domain's edge (read
with per-thread loads), interior tiles (tensor copy) and ragged ones; likewise along y."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_bulk import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(83, 67), (128, 96), (1003, 251)])
@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("mach,kw", [(0.3, {}), (1.5, {}), (0.01, {}), (0.3, dict(scheme=W.SCHEME_TVD2)),
                                     (0.05, dict(time_scheme=W.TIME_DUAL, dt_phys=0.02, subiters=3))])
@pytest.mark.parametrize("tma", [0, 1])
def test_rows_and_columns(ibm, n, axis, mach, kw, tma):  # noqa: F811
    nx, ny = n
    spec = W.case_spec(None, nx, ny, (0.0, nx / 16.0, 0.0, ny / 16.0), mach, 200.0, (W.BC_OUTFLOW,) * 4,
                       precision=W.PREC_FP32_BULK, **kw)
    g = ibm.Case(spec)
    g.use_tma(tma)
    shape = [4, ny, nx]
    shape[axis] = 1
    line = 1.0 + 0.02 * np.random.default_rng(nx).uniform(-1.0, 1.0, shape)
    g.set_state(g.state() * line)
    g.step(2)
    u = g.state()
    assert np.isfinite(u).all() and np.ptp(u, axis=axis).max() == 0.0
