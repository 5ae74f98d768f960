"""The direct convolution with less workspace than one pass takes: it runs window by window, and the header's promise holds
that the workspace only changes how many passes are made.  Every output sums the same channels in the same order in every
window, so the bound is equality of all bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_05781_b200 import workloads
from paper_2412_05781_b200.workloads import ConvLayer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    assert torch.cuda.is_available()
    return binding


def _kinds(B, call):
    """The kinds of the kernels a call launches, in order."""
    B.sdwino_profile_enable(1)
    try:
        call()
        torch.cuda.synchronize()
        return [k for k, _ in B.sdwino_profile_records()]
    finally:
        B.sdwino_profile_enable(0)


# (layouts, channel ranges and wide tiles: test_direct_shape_cpu.py checks that the model still picks each for one of them)
WINDOW_SHAPES = [
    # stride, C, K, H, W, N: one image or many, odd sizes, channels that end inside a block, split channel ranges
    (1, 64, 64, 16, 16, 2), (1, 72, 200, 30, 26, 2), (1, 640, 136, 16, 16, 2), (1, 33, 300, 17, 40, 1), (1, 40, 17, 600, 1, 1),
    (1, 64, 16, 1, 1, 512), (1, 32, 9, 1, 600, 1), (1, 32, 1, 23, 24, 1), (1, 1280, 1280, 8, 8, 8),
    (2, 48, 56, 48, 55, 2), (2, 33, 1, 64, 64, 1), (2, 320, 328, 16, 16, 10), (2, 40, 24, 5, 900, 1), (2, 1280, 48, 50, 51, 1),
    (1, 32, 320, 23, 56, 5), (1, 200, 160, 66, 41, 5), (1, 100, 16, 15, 37, 1), (2, 32, 100, 10, 66, 5), (2, 100, 16, 27, 45, 2),
]


@pytest.mark.parametrize("shape", WINDOW_SHAPES)
def test_the_workspace_does_not_change_the_bits(B, shape):
    stride, C, K, H, W, N = shape
    x, w, b = workloads.make_inputs(ConvLayer(C=C, K=K, H=H, W=W, N=N), seed=sum(shape))
    ref = oracle.direct_conv3x3_strided(x.numpy(), w.numpy(), b.numpy(), stride)
    xd, bd, wT = x.cuda(), b.cuda(), B.sdwino_filter_transform(w.cuda(), 1)
    full = B.sdwino_workspace_bytes_direct(N, C, H, W, K, stride)
    least = 128 * 9 * (C + K) * 2
    n, pad = ref.size, 64
    first = None
    launches, parts_in_turn = [], False
    for size in sorted({full, full // 2, full // 3, full // 7, 3 * least, least + 1024, least}, reverse=True):
        if size < least:
            continue
        ws = B.alloc_workspace(size + 4096)
        ws.fill_(255)                              # a workspace of NaNs, canaries behind it and around y
        canary = torch.full((n + 2 * pad,), 1234.0, dtype=torch.float16, device="cuda")
        y = canary[pad:pad + n].view(ref.shape)
        kinds = _kinds(B, lambda: B.sdwino_conv3x3_direct(xd, wT, bd, K, stride, ws[:size], y=y))
        assert B.sdwino_last_device_status() == B.OK
        assert "fused" in kinds and "wino_gemm" not in kinds
        assert bool((ws[size:] == 255).all())
        assert bool((canary[:pad] == 1234.0).all()) and bool((canary[pad + n:] == 1234.0).all())
        if first is None:
            first = y.clone()
            assert np.abs(y.cpu().double().numpy() - ref).max() <= 1e-3 * np.abs(ref).max()
        assert torch.equal(first, y), size
        launches.append(len(kinds))
        # one packed input, but the parts of the channel ranges of some tiles at a time
        parts_in_turn |= kinds.count("input_transform") == 1 and kinds.count("output_transform") > 1
    # the smallest workspace does take several windows, unless the layer's packed input fits it
    positions = N * ((H - 1) // stride + 2) * ((W - 1) // stride + 2)
    if positions * (4 if stride == 2 else 1) * -(-C // 64) * 128 > least:
        assert launches[-1] >= 4
    if shape in ((1, 640, 136, 16, 16, 2), (1, 1280, 1280, 8, 8, 8)):
        assert parts_in_turn


def test_residual_and_activation_window_by_window(B):
    C, K, H, W, N = 96, 40, 24, 32, 2
    x, w, b = workloads.make_inputs(ConvLayer(C=C, K=K, H=H, W=W, N=N), seed=5)
    res = torch.randn(N, K, H, W, generator=torch.Generator().manual_seed(1)).half().cuda()
    wT = B.sdwino_filter_transform(w.cuda(), 1)
    full = B.sdwino_conv3x3_ex(x.cuda(), wT, b.cuda(), res, K, 1, B.ACT_SILU, B.alloc_workspace(B.sdwino_workspace_bytes(N, C, H, W, K, 1)))
    y = res.clone()                                # the residual may be y itself
    B.sdwino_conv3x3_ex(x.cuda(), wT, b.cuda(), y, K, 1, B.ACT_SILU, B.alloc_workspace(B.sdwino_workspace_min_bytes(N, C, H, W, K, 1)), y=y)
    assert B.sdwino_last_device_status() == B.OK
    assert torch.equal(full, y)


@pytest.mark.parametrize("shape", [(1, 64, 64, 8, 8, 7), (1, 31, 64, 32, 32, 1), (2, 320, 320, 16, 16, 9)])
def test_small_layers_take_the_three_steps(B, shape):
    """Below the number of pixels or channels from which the single GEMM pays: several passes give the bits of one."""
    stride, C, K, H, W, N = shape
    x, w, b = workloads.make_inputs(ConvLayer(C=C, K=K, H=H, W=W, N=N), seed=sum(shape))
    wT = B.sdwino_filter_transform(w.cuda(), 1)
    ys, passes = [], []
    for size in (B.sdwino_workspace_bytes_direct(N, C, H, W, K, stride), 128 * 9 * (C + K) * 2 + 1024):
        ws = B.alloc_workspace(size)
        kinds = _kinds(B, lambda: ys.append(B.sdwino_conv3x3_direct(x.cuda(), wT, b.cuda(), K, stride, ws)))
        assert kinds == ["input_transform", "wino_gemm", "output_transform"] * (len(kinds) // 3)
        passes.append(len(kinds) // 3)
    assert passes[0] == 1 and passes[1] > 1
    assert torch.equal(ys[0], ys[1])
