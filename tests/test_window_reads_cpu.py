"""The activation transforms of any width load x in aligned 4-byte words of two pixels.  No word may reach outside x: not
where x begins at an odd pixel, not where it ends at one (the walk computes the addresses as the kernels do, with their rules for what may be loaded)."""
import pytest


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    return binding


@pytest.mark.parametrize("odd_start", [False, True])
@pytest.mark.parametrize("tile", [2, 4])
@pytest.mark.parametrize("shape", [
    # N, C, H, W: x of an even and of an odd number of pixels, rows narrower than a window, one pixel
    (1, 1, 1, 1), (1, 1, 1, 2), (1, 3, 5, 1), (2, 2, 3, 3), (1, 1, 9, 9), (1, 9, 4, 5), (3, 1, 7, 11), (1, 5, 33, 129),
    (1, 2, 6, 16), (1, 1, 8, 8), (2, 640, 5, 37),
])
def test_no_read_outside_x(B, shape, tile, odd_start):
    assert B.sdwino_selftest_window_reads(*shape, tile, odd_start) == (0, 0)


def test_arguments(B):
    with pytest.raises(B.SdwinoError):
        B.sdwino_selftest_window_reads(1, 1, 1, 0, 2, False)
    with pytest.raises(B.SdwinoError):
        B.sdwino_selftest_window_reads(1, 1, 1, 1, 1, False)
