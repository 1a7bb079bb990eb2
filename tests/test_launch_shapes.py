"""Host-side launch rules: tile shapes of the FP64 stages."""
import ctypes
import random

import pytest


@pytest.fixture(scope="module")
def shape():
    from paper_1912_11908_gb300 import _build, ibm as mod
    _build.build()
    f = mod.lib().ibm__tile_shape_f64
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    return f


TILES = [(16, 16), (16, 8), (8, 8)]


def test_shape_fits_the_grid_dimension(shape):
    """Every grid that 16 x 16 tiles can cover (65,535 of them along y) gets a shape that can."""
    rng = random.Random(5)
    for ny in [8, 524272, 524280, 524281, 524288, 1048559, 1048560] + [rng.randint(8, 1048560) for _ in range(200)]:
        for nx in (8, 9, 16, 33, rng.randint(8, 1023)):
            ty = TILES[shape(nx, ny, 152)][1]
            assert (ny + ty - 1) // ty <= 65535, (nx, ny, ty)


def test_shape_is_the_least_work_of_the_fullest_sm(shape):
    work = [1.0, 0.53, 0.30]
    rng = random.Random(6)
    for nx, ny, sms in [(257, 131, 152), (257, 131, 76)] + [(rng.randint(8, 2000), rng.randint(8, 2000),
                                                             rng.randint(1, 200)) for _ in range(500)]:
        cost = [-(-(-(-nx // tx) * -(-ny // ty)) // sms) * w for (tx, ty), w in zip(TILES, work)]
        assert cost[shape(nx, ny, sms)] == min(cost), (nx, ny, sms)
    assert shape(257, 131, 152) == 1 and shape(768, 384, 152) == 0 and shape(64, 64, 152) == 2


@pytest.fixture(scope="module")
def wide():
    from paper_1912_11908_gb300 import _build, ibm as mod
    _build.build()
    f = mod.lib().ibm__stage_wide
    f.argtypes = [ctypes.c_int] * 4
    f.restype = ctypes.c_int
    return f


def test_wide_blocks_for_few_tiles(wide):
    """One wave of wide blocks (three per SM) without body tiles, two with them, one of 128-thread blocks (eight per
    SM) where IB nodes are rebuilt in them."""
    for sms in (1, 76, 148, 152):
        for nt, nb, rebuild, want in ((1, 0, 1, 1), (3 * sms, 0, 1, 1), (3 * sms + 1, 0, 1, 0), (3 * sms + 1, 1, 0, 1),
                                      (6 * sms, 9, 0, 1), (6 * sms + 1, 9, 0, 0), (8 * sms, 9, 1, 1),
                                      (8 * sms + 1, 9, 1, 0)):
            assert bool(wide(nt, nb, rebuild, sms)) == bool(want), (nt, nb, rebuild, sms)


def test_wide_blocks_in_dual_time(wide):
    """Up to sixteen tiles per SM for a case alone, six for a group."""
    from paper_1912_11908_gb300 import ibm as mod
    f = mod.lib().ibm__dual_wide
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    for sms in (1, 152):
        assert [f(16 * sms, 1, sms), f(16 * sms + 1, 1, sms), f(6 * sms, 2, sms), f(6 * sms + 1, 2, sms)] == [1, 0, 1, 0]


def test_beside_other_cases(wide):
    """Crowded from 24 tiles per SM on, a case's or group's own and those beside it; never alone."""
    from paper_1912_11908_gb300 import ibm as mod
    f = mod.lib().ibm__crowded
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    for sms in (1, 152):
        assert [f(4 * sms, 20 * sms, sms), f(4 * sms, 20 * sms + 1, sms), f(100 * sms, 0, sms)] == [0, 1, 0]
        assert f(1, 1 << 30, sms) == 1


def test_blocks_of_a_group(wide):
    """Six 128-thread blocks per SM for explicit groups of up to 20 tiles per SM, eight for larger ones."""
    from paper_1912_11908_gb300 import ibm as mod
    f = mod.lib().ibm__batch_blocks
    f.argtypes = [ctypes.c_int] * 2
    f.restype = ctypes.c_int
    for sms in (1, 152):
        assert [f(1, sms), f(20 * sms, sms), f(20 * sms + 1, sms), f(2 ** 31 - 1, sms)] == [6, 6, 8, 8]
