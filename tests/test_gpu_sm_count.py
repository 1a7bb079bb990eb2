"""The launch rules count the device's own multiprocessors."""
import ctypes

import pytest

from test_gpu_flow3d import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_sm_count(ibm):  # noqa: F811
    torch = pytest.importorskip("torch")
    f = ibm.lib().ibm__sm_count
    f.restype = ctypes.c_int
    assert f() == torch.cuda.get_device_properties(0).multi_processor_count
