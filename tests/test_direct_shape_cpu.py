"""The shapes that the GPU tests of the direct convolution's single GEMM run through: every layout of the pixels, with and without
split channel ranges, for both strides, and wide tiles (host logic only; 148 SMs)."""
import pytest

from tests.test_gpu_direct_conv import SHAPES
from tests.test_gpu_direct_windows import WINDOW_SHAPES


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    return binding


def test_the_tested_layers_cover_the_variants(B):
    seen = set()
    for stride, C, K, H, W, N in SHAPES + WINDOW_SHAPES:
        shape = B.sdwino_selftest_direct_shape(N, C, H, W, K, stride)
        if shape:
            flat, n_tile, splits = shape
            seen.add((stride, flat, splits > 1))
            seen.add((flat, "wide") if n_tile >= 144 else (flat, "narrow"))
    assert {(s, f, p) for s in (1, 2) for f in (0, 1) for p in (False, True)} <= seen
    assert {(f, w) for f in (0, 1) for w in ("wide", "narrow")} <= seen


def test_which_layers_take_it(B):
    assert B.sdwino_selftest_direct_shape(2, 320, 64, 64, 320, 2) is not None
    assert B.sdwino_selftest_direct_shape(7, 64, 8, 8, 64, 1) is None        # 448 pixels
    assert B.sdwino_selftest_direct_shape(1, 31, 32, 32, 64, 1) is None      # 31 channels
    assert B.sdwino_selftest_direct_shape(9, 320, 16, 16, 320, 2) is None    # 576 pixels of 640
    assert B.sdwino_selftest_direct_shape(640, 64, 1, 1, 20, 2) is None      # padding makes the packed input too large
