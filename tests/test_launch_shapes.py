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
