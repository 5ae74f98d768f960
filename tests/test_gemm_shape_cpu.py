"""The GEMM's launch shape where the HBM stream of V and M bounds it (host logic only): one block of tiles per CTA tile and few
stages in flight, from twice the L2 cache of V and M on."""
import pytest


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    return binding


@pytest.mark.parametrize("shape, expected", [
    # N, C, H, W, K: (CTAs, n_tile, blocks, stages)
    ((1, 256, 1024, 1024, 128), (1, 128, 1, 5)), ((1, 256, 512, 512, 128), (1, 128, 1, 5)),
    ((1, 128, 1024, 1024, 128), (1, 128, 1, 4)), ((1, 128, 512, 512, 128), (1, 128, 1, 4)),
    ((1, 128, 768, 768, 64), (1, 64, 1, 5)), ((1, 192, 768, 768, 128), (1, 128, 1, 4)),
])
def test_streaming_launches(B, shape, expected):
    assert B.sdwino_selftest_gemm_shape(*shape, 4, B.sdwino_workspace_bytes(*shape, 4)) == expected


@pytest.mark.parametrize("shape, blocks", [((1, 256, 256, 256, 128), None), ((1, 512, 512, 512, 128), 2), ((4, 320, 96, 96, 320), None)])
def test_other_launches_keep_their_shape(B, shape, blocks):
    # V and M within twice the L2 cache, many channels, several k tiles: the deep ring
    ctas, n_tile, got, stages = B.sdwino_selftest_gemm_shape(*shape, 4, B.sdwino_workspace_bytes(*shape, 4))
    assert ctas == 1 and (blocks is None or got == blocks)
    assert stages * (got * 16 + n_tile // 8) >= 160        # KB
