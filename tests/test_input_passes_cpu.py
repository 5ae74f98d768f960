"""Which activation transform the passes of an F(4x4) layer take (host logic only)."""
import pytest


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    return binding


@pytest.mark.parametrize("shape", [(1, 512, 1024, 1024, 512), (2, 256, 1024, 1024, 256), (1, 640, 1024, 896, 640), (1, 512, 768, 1536, 512)])
def test_passes_of_large_layers_are_cut_for_the_staged_transform(B, shape):
    # more tiles than one pass of the default workspace holds, and rows of tiles that its size is no multiple of
    ws = B.sdwino_workspace_bytes(*shape, 4)
    passes, staged = B.sdwino_selftest_input_passes(*shape, ws)
    assert passes >= 2 and staged >= passes - 1      # the last pass may be small
    # a third of it: still gigabytes of transformed activations per pass
    passes, staged = B.sdwino_selftest_input_passes(*shape, ws // 3)
    assert passes >= 4 and staged >= passes - 1


def test_one_pass(B):
    ws = B.sdwino_workspace_bytes(1, 512, 512, 512, 512, 4)
    assert B.sdwino_selftest_input_passes(1, 512, 512, 512, 512, ws) == (1, 1)
    assert B.sdwino_selftest_input_passes(1, 320, 64, 64, 320, 1 << 30) == (1, 0)        # small: registers
    assert B.sdwino_selftest_input_passes(1, 512, 516, 516, 512, 4 << 30) == (1, 0)      # rows that are not whole sectors of V
    assert B.sdwino_selftest_input_passes(1, 512, 512, 512, 512, 1000)[0] == 0


@pytest.mark.parametrize("shape, expected", [
    # N, C, H, W, K: rows of 64 tiles or more from half the L2 cache on
    ((1, 512, 256, 256, 512), 1), ((1, 256, 256, 256, 256), 1), ((1, 256, 512, 512, 128), 1), ((1, 128, 512, 512, 128), 1),
    ((1, 128, 256, 256, 128), 0), ((1, 256, 320, 320, 256), 0), ((2, 512, 320, 320, 512), 1),
    # narrower rows: 2.5 times the L2 cache
    ((2, 960, 128, 128, 320), 0), ((4, 1280, 128, 128, 640), 1), ((1, 512, 128, 128, 512), 0),
])
def test_where_the_staged_transform_is_taken(B, shape, expected):
    assert B.sdwino_selftest_input_passes(*shape, B.sdwino_workspace_bytes(*shape, 4)) == (1, expected)
