"""The fixed-point FP64 product takes the shapes its sums and indices are made for (host
code: no GPU needed)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def supported():
    from paper_2605_30379_gb300 import build
    fn = ctypes.CDLL(build.build())._Z19mrc_pairq_supportediii  # bool mrc_pairq_supported(int, int, int)
    fn.restype = ctypes.c_bool
    fn.argtypes = [ctypes.c_int] * 3
    return fn


@pytest.mark.parametrize("r,m,c,ok", [
    (1, 1, 1, True), (56, 56, 56, True), (57, 57, 57, False), (78, 78, 1, True), (80, 80, 5, False),
    (64, 1, 128, True), (255, 1, 257, True), (256, 1, 256, False), (200, 1, 400, False),
    (2, 79, 2, True), (2, 80, 2, False), (1, 128, 1, False), (1, 3000, 1, False)])
def test_shapes(supported, r, m, c, ok):
    assert supported(r, m, c) is ok
