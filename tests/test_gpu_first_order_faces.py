"""Faces where WENO5 gives a density or pressure that is not positive take the cells' values instead (Sec. 2's first-order
fallback), and supersonic faces the one-sided splits, in every tile shape: fields with runs of cells (0.2, 0.1, 0.01
times the free stream's density or pressure, then the free stream again) along every axis in both senses, placed so
that of two adjacent lines mostly one falls back.  The faces that do are counted on the CPU, with the distance of every
other face's density and pressure from zero, far above rounding.  Against the FP64 oracle after one step: 1e-10 in FP64;
FP32-bulk 1e-3 of the deviations' scale -- a residual's 200 dependent roundings of 2^-24 on energy fluxes of up to 40
times the state's scale; a face that took the wrong line's or cell's states is off by 1e-2 and more."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_bulk import _compare
from test_gpu_dual import _err
from test_gpu_flow3d import _state_error, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

RUN = np.array([0.2, 0.1, 0.01])


def _weno(f0, f1, f2, f3, f4):
    b = [13.0 / 12.0 * (f0 - 2 * f1 + f2) ** 2 + 0.25 * (f0 - 4 * f1 + 3 * f2) ** 2,
         13.0 / 12.0 * (f1 - 2 * f2 + f3) ** 2 + 0.25 * (f1 - f3) ** 2,
         13.0 / 12.0 * (f2 - 2 * f3 + f4) ** 2 + 0.25 * (3 * f2 - 4 * f3 + f4) ** 2]
    a = [d / (1e-6 + x) ** 2 for d, x in zip((0.1, 0.6, 0.3), b)]
    q = [(2 * f0 - 7 * f1 + 11 * f2) / 6, (-f1 + 5 * f2 + 2 * f3) / 6, (2 * f2 + 5 * f3 - f4) / 6]
    return sum(x * y for x, y in zip(a, q)) / sum(a)


def _states(f, axis):
    """Left and right states of the faces between cells 2, 3 .. n - 4, n - 3 along the axis."""
    f = np.moveaxis(f, axis, -1)
    n = f.shape[-1]
    s = [f[..., k:n - 5 + k] for k in range(6)]
    return np.moveaxis(_weno(*s[:5]), -1, axis), np.moveaxis(_weno(*s[5:0:-1]), -1, axis)


def _falls(rho, p, axis, margin=2e-3):
    """Faces along the axis that fall back; every state is clear of zero by the margin."""
    s = _states(rho, axis) + _states(p / p.max(), axis)
    assert min(np.abs(x).min() for x in s) > margin
    return np.any([x <= 0.0 for x in s], axis=0)


def _field(shape, seed, size=9):
    """Density and pressure factors with a run of cells in every block of the given size along each axis."""
    rng = np.random.default_rng(seed)
    out = [np.ones(shape), np.ones(shape)]
    for block in np.ndindex(*[n // size for n in shape]):
        axis = rng.integers(len(shape))
        at = [int(b * size + rng.integers(0, size - 3)) for b in block]
        run = RUN[::rng.choice([-1, 1])]
        sl = [slice(a, a + 1) for a in at]
        sl[axis] = slice(at[axis], at[axis] + 3)
        f = out[rng.integers(2)]
        f[tuple(sl)] = run[:f[tuple(sl)].size].reshape(f[tuple(sl)].shape)
    return out


def _conserved(spec, rho, pf, vel):
    g = spec["gamma"]
    p = pf / (g * spec["mach"] ** 2)
    m = [rho * v for v in vel]
    return np.stack([rho] + m + [p / (g - 1.0) + 0.5 * rho * sum(v * v for v in vel)]), p


def _mixed(falls):
    """Pairs of adjacent lines (even, odd along the last axis of falls) of which exactly one falls back."""
    n = falls.shape[-1] // 2 * 2
    return int((falls[..., 0:n:2] != falls[..., 1:n:2]).sum())


@pytest.mark.parametrize("nx,ny", [(64, 64), (97, 83), (257, 131), (160, 240), (1009, 249)])
@pytest.mark.parametrize("mach", [0.3, 2.0])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_BULK])
@pytest.mark.parametrize("form", [0, 2, "persistent"])
def test_2d(ibm, orc, nx, ny, mach, precision, form):  # noqa: F811
    if precision == W.PREC_FP64 and (form != 0 or nx > 1000):
        pytest.skip("one form")
    spec = W.case_spec(None, nx, ny, (0.0, nx / 16.0, 0.0, ny / 16.0), mach, 200.0, (W.BC_FREESTREAM,) + (W.BC_OUTFLOW,) * 3,
                       precision=precision)
    rho, pf = _field((ny, nx), nx)
    vel = (np.where(np.arange(nx) // 20 % 2, 1.0, -0.9) + 0.0 * rho, np.where(np.arange(ny) // 20 % 2, 0.8, -0.7)[:, None] + 0.0 * rho)
    a, p = _conserved(spec, rho, pf, vel)
    fx, fy = _falls(rho, p, 1), _falls(rho, p, 0)
    counts = (int(fx.sum()), int(fy.sum()), _mixed(fx.T), _mixed(fy))
    assert min(counts) >= 4, counts
    g, o = ibm.Case(spec), orc.Case(dict(spec, precision=W.PREC_FP64))
    if precision == W.PREC_FP32_BULK:
        g.use_persistent(form == "persistent")
        if form != "persistent":
            g.stage_launches(form)
    g.set_state(a)
    o.set_state(a)
    g.step(1)
    o.step(1)
    if precision == W.PREC_FP64:
        assert _err(g.state(), o.state(), o.tags()) <= 1e-10
    else:
        err = _compare(g, o)
        assert max(err.values()) <= 1e-3, err


@pytest.mark.parametrize("n", [(31, 15, 29), (62, 30, 16), (20, 43, 18)])
@pytest.mark.parametrize("mach", [0.3, 2.0])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_BULK])
def test_3d(ibm, orc, n, mach, precision):  # noqa: F811
    spec = W.case3d_spec(None, None, n, (0.0,) * 3, tuple(k / 16.0 for k in n), mach, 200.0,
                         (W.BC_FREESTREAM,) + (W.BC_OUTFLOW,) * 5, precision=precision)
    shape = n[::-1]
    rho, pf = _field(shape, n[0], 6)
    k = np.indices(shape)
    vel = [np.where(k[2 - a] // 10 % 2, 1.0, -0.9 + 0.1 * a) for a in range(3)]
    a, p = _conserved(spec, rho, pf, vel)
    counts = [int(_falls(rho, p, 2 - d).sum()) for d in range(3)]
    assert min(counts) >= 3, counts
    g, o = ibm.Case3D(spec), orc.Case3D(dict(spec, precision=W.PREC_FP64))
    g.set_state(a)
    o.set_state(a)
    g.step(1)
    o.step(1)
    if precision == W.PREC_FP64:
        assert _state_error(g.state(), o.state(), o.tags()) <= 1e-10
    else:
        x, y = g.state(), o.state()
        for v in range(5):
            dev = np.abs(y[v] - np.median(y[v])).max()
            assert np.abs(x[v] - y[v]).max() <= 1e-3 * dev, v
