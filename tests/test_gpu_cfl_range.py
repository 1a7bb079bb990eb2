"""The CFL bound of FP64 cases in cells whose state leaves the range of ordinary flow: a cell with an infinite energy
drives dt to zero, one near the largest double gives its own finite bound, and one with a NaN bound (a negative
pressure) is left out, as IEEE arithmetic and a maximum that ignores NaN have it.  One step; t is then the dt taken."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_flow3d import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

CELLS = [("energy", np.inf), ("energy", 1e308), ("energy", 3e307), ("energy", -1e300), ("energy", 1e300),
         ("momentum", 1e200), ("momentum", np.inf), ("density", 1e-300)]
ROW = {"density": 0, "momentum": 1, "energy": -1}


def _dt(u, spec, h):
    """CFL / max of the bound over the cells, in numpy's IEEE arithmetic."""
    g, n = spec["gamma"], u.shape[0] - 2
    mu = 1.0 / spec["re"]
    with np.errstate(all="ignore"):
        v = u[1:1 + n] / u[0]
        c = np.sqrt(g * (g - 1.0) * (u[-1] - 0.5 * u[0] * (v * v).sum(0)) / u[0])
        lam = sum((np.abs(v[a]) + c) / h[a] for a in range(n))
        lam = lam + 2.0 * g * mu / (spec["prandtl"] * u[0]) * sum(1.0 / h[a] ** 2 for a in range(n))
        return spec["cfl"] / np.fmax.reduce(lam.ravel())


@pytest.mark.parametrize("what,value", CELLS)
@pytest.mark.parametrize("dim", [2, 3])
def test_dt(ibm, dim, what, value):  # noqa: F811
    if dim == 2:
        spec = W.case_spec(None, 40, 24, (0.0, 5.0, 0.0, 3.0), 0.4, 100.0, W.FAR)
        g = ibm.Case(spec)
    else:
        spec = W.case3d_spec(None, None, (12, 10, 9), (0.0,) * 3, (1.5, 1.25, 1.125), 0.4, 100.0, W.FAR3D)
        g = ibm.Case3D(spec)
    u = g.state()
    u[(ROW[what],) + (4,) * dim] = value
    g.set_state(u)
    g.step(1)
    want = _dt(u, spec, (0.125,) * dim)
    np.testing.assert_allclose(g.time()[0], want, rtol=1e-12)
