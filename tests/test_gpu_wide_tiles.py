"""FP32-bulk stages on both sides of the rule that gives grids of few tiles wide blocks: ragged grids of more tiles than
that (128-thread blocks) against the FP64 oracle with the bar of the tile-edge tests, and the same tiles through wide
blocks (alone) and 128-thread blocks (a group of many requests)."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_bulk import ibm  # noqa: F401  (fixture)
from test_gpu_pairs32 import _run

pytestmark = pytest.mark.gpu

GRIDS = [(1009, 249), (497, 507), (1009, 331), (661, 507)]  # 1,024 tiles each, then 1,344: all four sides ragged


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("scheme,interp,mach", [
    (W.SCHEME_WENO5, W.INTERP_LINEAR, 0.3), (W.SCHEME_WENO5, W.INTERP_LINEAR, 1.5),
    (W.SCHEME_TVD2, W.INTERP_LINEAR, 1.5), (W.SCHEME_WENO5, W.INTERP_QUADRATIC, 0.3)])
def test_many_tiles(ibm, orc, nx, ny, scheme, interp, mach):  # noqa: F811
    _run(ibm, orc, nx, ny, scheme=scheme, ib_interp=interp, mach=mach)


@pytest.mark.parametrize("scheme", [W.SCHEME_WENO5, W.SCHEME_TVD2])
@pytest.mark.parametrize("interp", [W.INTERP_LINEAR, W.INTERP_QUADRATIC])
@pytest.mark.parametrize("count", [2, 24])
def test_alone_and_in_a_group(ibm, scheme, interp, count):  # noqa: F811
    """2 cases of 55 tiles: wide blocks in the group too; 24 of them: 128 threads.  Equal up to FP32 rounding."""
    spec = W.cylinder_m02_re40(171, 75, precision=W.PREC_FP32_BULK, scheme=scheme, ib_interp=interp)
    c = ibm.Case(spec)
    c.step(20)
    want = c.forces()
    s = ibm.Server(max_active=32, steps_per_chunk=10)
    ids = [s.submit(spec, 20) for _ in range(count)]
    s.drain()
    for i in ids:
        r = s.poll(i)
        assert r["status"] == ibm.IBM_OK and r["steps_done"] == 20
        np.testing.assert_allclose(r["forces"], want, rtol=2e-5, atol=2e-5 * np.abs(want).max())
    s.close()


def test_residency_of_the_table_kernels(ibm):  # noqa: F811
    """Eight 128-thread blocks or three wide ones per SM, as their launch bounds and the group tuner count on."""
    import ctypes
    f = ibm.lib().ibm__batch_blocks_per_sm
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    for wide, want in ((0, 8), (1, 3)):
        assert [f(wide, t, q) for t in (0, 1) for q in (0, 1)] == [want] * 4


def test_residency_for_few_tiles(ibm):  # noqa: F811
    """Six 128-thread blocks per SM of the form that groups of a wave or two take."""
    import ctypes
    f = ibm.lib().ibm__batch_blocks_per_sm
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    assert [f(2, t, q) for t in (0, 1) for q in (0, 1)] == [6] * 4


@pytest.mark.parametrize("scheme", [W.SCHEME_WENO5, W.SCHEME_TVD2])
@pytest.mark.parametrize("interp", [W.INTERP_LINEAR, W.INTERP_QUADRATIC])
@pytest.mark.parametrize("count", [1, 3])
def test_groups_of_many_tiles(ibm, scheme, interp, count):  # noqa: F811
    """1,344 tiles (six blocks per SM), three times as many (eight), a case alone: equal up to FP32 rounding."""
    spec = W.cylinder_m02_re40(1009, 331, precision=W.PREC_FP32_BULK, scheme=scheme, ib_interp=interp)
    c = ibm.Case(spec)
    c.step(20)
    want = c.forces()
    s = ibm.Server(max_active=32, steps_per_chunk=10)
    ids = [s.submit(spec, 20) for _ in range(count)]
    s.drain()
    for i in ids:
        r = s.poll(i)
        assert r["status"] == ibm.IBM_OK and r["steps_done"] == 20
        np.testing.assert_allclose(r["forces"], want, rtol=2e-5, atol=2e-5 * np.abs(want).max())
    s.close()
