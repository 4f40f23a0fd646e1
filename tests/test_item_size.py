"""The work item size of a plan (host function of the library, no GPU)."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def item_size():
    from paper_2503_22695_gb300 import _build
    f = C.CDLL(_build.build())["_ZN4ibfe9item_sizeEili"]
    f.argtypes, f.restype = [C.c_int, C.c_int64, C.c_int], C.c_int
    return f


POINTS = [0, 1, 1024, 14400, 38912, 38913, 64000, 144000, 622592, 622593, 10 ** 8]


@pytest.mark.parametrize("Q", POINTS)
def test_fp64_items_do_not_depend_on_the_device(item_size, Q):
    from paper_2503_22695_gb300 import ibfe
    sizes = {item_size(ibfe.IB_FP64, Q, sms) for sms in (1, 16, 76, 132, 148, 152, 160)}
    assert len(sizes) == 1


@pytest.mark.parametrize("Q", POINTS)
@pytest.mark.parametrize("sms", [1, 76, 152])
def test_items_are_whole_steps_within_the_kernels_limits(item_size, Q, sms):
    from paper_2503_22695_gb300 import ibfe
    for prec, step in ((ibfe.IB_FP32_SPLIT, 128), (ibfe.IB_FP64, 64)):
        n = item_size(prec, Q, sms)
        assert step <= n <= 1024 and n % step == 0
