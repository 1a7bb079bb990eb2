"""Grids longer than a launch dimension holds (65,535 blocks along y): with a field that does not vary along y and
zero-gradient ends, every row of cells repeats the rows of a short grid bit for bit."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_flow3d import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

BC3 = (W.BC_FREESTREAM, W.BC_OUTFLOW) + (W.BC_OUTFLOW,) * 4


def _run3d(ibm, ny, line, precision):  # noqa: F811
    nz, nx = line.shape[1], line.shape[3]
    spec = W.case3d_spec(None, None, (nx, ny, nz), (0.0, 0.0, 0.0), (nx / 16.0, ny / 16.0, nz / 16.0), 0.4, 100.0, BC3,
                         precision=precision)
    g = ibm.Case3D(spec)
    g.set_state(np.broadcast_to(line, (5, nz, ny, nx)) * g.state())
    g.step(2)
    return g.state()


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_BULK])
@pytest.mark.parametrize("ny", [65535, 65536, 131077])
def test_3d_rows(ibm, ny, precision):  # noqa: F811
    line = 1.0 + 0.02 * np.random.default_rng(3).uniform(-1.0, 1.0, (5, 5, 1, 7))
    short, long_ = _run3d(ibm, 33, line, precision), _run3d(ibm, ny, line, precision)
    assert np.ptp(short, axis=2).max() == 0.0
    np.testing.assert_array_equal(long_, np.broadcast_to(short[:, :, :1], long_.shape))


def _run2d(ibm, ny, line, precision):  # noqa: F811
    nx = line.shape[2]
    spec = W.case_spec(None, nx, ny, (0.0, nx / 16.0, 0.0, ny / 16.0), 0.4, 100.0,
                       (W.BC_FREESTREAM,) + (W.BC_OUTFLOW,) * 3, precision=precision)
    g = ibm.Case(spec)
    g.set_state(np.broadcast_to(line, (4, ny, nx)) * g.state())
    g.step(2)
    g.sync()
    return g.state()


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_BULK])
@pytest.mark.parametrize("ny", [524280, 524288, 1048560])
def test_2d_rows(ibm, ny, precision):  # noqa: F811
    line = 1.0 + 0.02 * np.random.default_rng(4).uniform(-1.0, 1.0, (4, 1, 8))
    short, long_ = _run2d(ibm, 64, line, precision), _run2d(ibm, ny, line, precision)
    assert np.ptp(short, axis=1).max() == 0.0
    np.testing.assert_array_equal(long_, np.broadcast_to(short[:, :1], long_.shape))
