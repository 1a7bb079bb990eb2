"""The 3-D sweeps at the sizes where their warps and rows end: cells around a warp's 30 along x, the rows that the y and
z sweeps' blocks take around 14, the smallest blocks; shocks in the field so that the first-order fallback and the
supersonic branches are taken.  Both precisions against the FP64 oracle, the repository's bars (1e-10 and 1e-4)."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_flow3d import _state_error, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SIZES = [(29, 13, 14), (30, 14, 15), (31, 15, 29), (61, 28, 5), (4, 43, 6), (5, 4, 17), (90, 7, 9)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_BULK])
@pytest.mark.parametrize("re", [50.0, 0.0])
def test_field(ibm, orc, n, precision, re):  # noqa: F811
    spec = W.case3d_spec(None, None, n, (0.0, 0.0, 0.0), (1.0, 0.7, 0.9), 1.5, re,
                         (W.BC_FREESTREAM, W.BC_OUTFLOW) + (W.BC_PERIODIC,) * 2 + (W.BC_OUTFLOW,) * 2,
                         uinf=(0.9, 0.3, -0.2), precision=precision)
    g, o = ibm.Case3D(spec), orc.Case3D(spec)
    rng = np.random.default_rng(sum(n))
    a = o.state() * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, (5, n[2], n[1], n[0])))
    a[1:4] *= 1.0 + np.sign(np.sin(7.0 * np.arange(n[0]) / n[0]))  # stepped momentum: subsonic and supersonic slabs
    a[4] += 0.5 * (a[1:4] ** 2).sum(0) / a[0]
    g.set_state(a)
    o.set_state(a)
    g.step(2)
    o.step(2)
    e = _state_error(g.state(), o.state(), o.tags())
    assert e <= (1e-10 if precision == W.PREC_FP64 else 1e-4), e
