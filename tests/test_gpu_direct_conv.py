"""The direct convolution as one implicit GEMM (tile 1 from 512 output pixels, 640 with stride 2, and 32 channels) where
it can go wrong: both layouts of the pixels on the tensor core's lanes, images smaller than a tile of 128 pixels, rows
wider than a patch, the last row and column of each parity plane, channels and filters that end inside a block, channel
ranges split over CTAs, outputs that are not whole aligned pieces of eight.  Sums are kept in fp32 and rounded once, so
the bound is that of one fp16 rounding, 2^-11 of the value, plus the fp32 sum's 9 C 2^-24 of the largest: 1e-3 * max|ref|."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_05781_b200 import workloads
from paper_2412_05781_b200.workloads import ConvLayer

pytestmark = pytest.mark.gpu

BOUND = 1e-3


@pytest.fixture(scope="module")
def B():
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding
    assert torch.cuda.is_available()
    return binding


SHAPES = [
    # stride, C, K, H, W, N
    (1, 64, 64, 16, 16, 2), (1, 100, 36, 23, 23, 1), (1, 640, 136, 16, 16, 2), (1, 32, 9, 1, 600, 1), (1, 40, 17, 600, 1, 1),
    (1, 64, 16, 1, 1, 512), (1, 33, 300, 17, 40, 1), (1, 130, 24, 2, 1100, 1),
    (2, 48, 56, 48, 55, 2), (2, 40, 16, 51, 53, 1), (2, 100, 70, 64, 64, 1), (2, 33, 9, 3, 700, 1), (2, 40, 24, 2, 2047, 1),
    (2, 320, 328, 16, 16, 10), (2, 64, 20, 1, 1, 640), (2, 32, 40, 33, 80, 1), (2, 1280, 48, 50, 51, 1),
]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_implicit_gemm(B, shape, offset):
    stride, C, K, H, W, N = shape
    layer = ConvLayer(C=C, K=K, H=H, W=W, N=N)
    x, w, b = workloads.make_inputs(layer, seed=sum(shape) + offset)
    ref = oracle.direct_conv3x3_strided(x.numpy(), w.numpy(), b.numpy(), stride)
    # x and y one element into their buffers: 2-byte aligned pointers, canaries around y, a workspace of NaNs
    xb = torch.zeros(x.numel() + 1, dtype=torch.float16, device="cuda")
    xb[offset:offset + x.numel()] = x.flatten().cuda()
    xd = xb[offset:offset + x.numel()].view(x.shape)
    n, pad = ref.size, 64
    canary = torch.full((n + 2 * pad + 1,), 1234.0, dtype=torch.float16, device="cuda")
    y = canary[pad + offset:pad + offset + n].view(ref.shape)
    wT = B.sdwino_filter_transform(w.cuda(), 1)
    ws = B.alloc_workspace(B.sdwino_workspace_bytes_direct(N, C, H, W, K, stride))
    ws.view(torch.uint8).fill_(255)
    B.sdwino_profile_enable(1)
    try:
        B.sdwino_conv3x3_direct(xd, wT, b.cuda(), K, stride, ws, y=y)
        assert B.sdwino_last_device_status() == B.OK
        kinds = [k for k, _ in B.sdwino_profile_records()]
    finally:
        B.sdwino_profile_enable(0)
    # packing, GEMM, parts; the three steps where the padding makes the packed input larger than their workspace (1x1, stride 2)
    packed = N * ((H - 1) // stride + 2) * ((W - 1) // stride + 2) * (4 if stride == 2 else 1) * -(-C // 64) * 128
    routes = [["input_transform", "fused"], ["input_transform", "fused", "output_transform"]]
    assert kinds in ([["input_transform", "wino_gemm", "output_transform"]] if packed > ws.numel() else routes)
    assert np.abs(y.cpu().double().numpy() - ref).max() <= BOUND * np.abs(ref).max()
    assert bool((canary[:pad + offset] == 1234.0).all()) and bool((canary[pad + offset + n:] == 1234.0).all())
    first = y.clone()
    B.sdwino_conv3x3_direct(xd, wT, b.cuda(), K, stride, ws, y=y)
    assert torch.equal(first, y)      # parts are added in a fixed order
    if stride == 1:                   # residual and activation
        res = torch.randn(ref.shape, generator=torch.Generator().manual_seed(1)).half()
        refe = oracle.epilogue(ref, res.numpy(), "silu")
        B.sdwino_conv3x3_ex(xd, wT, b.cuda(), res.cuda(), K, 1, B.ACT_SILU, ws, y=y)
        assert np.abs(y.cpu().double().numpy() - refe).max() <= BOUND * np.abs(refe).max()
        assert bool((canary[:pad + offset] == 1234.0).all()) and bool((canary[pad + offset + n:] == 1234.0).all())
    # the smallest workspace: other windows, the same bits (and the same bound, which the three steps would miss)
    small = B.alloc_workspace(B.sdwino_workspace_min_bytes(N, C, H, W, K, 1))
    B.sdwino_conv3x3_direct(xd, wT, b.cuda(), K, stride, small, y=y)
    assert B.sdwino_last_device_status() == B.OK
    assert torch.equal(first, y)


def test_filters_of_another_layer_are_refused(B):
    layer = ConvLayer(C=64, K=64, H=32, W=32, N=1)
    x, w, b = workloads.make_inputs(layer, seed=1)
    other = B.sdwino_filter_transform(torch.zeros(72, 64, 3, 3, dtype=torch.float16, device="cuda"), 1)
    ws = B.alloc_workspace(B.sdwino_workspace_bytes_direct(1, 64, 32, 32, 64, 1))
    y = torch.full((1, 64, 32, 32), 7.0, dtype=torch.float16, device="cuda")
    B.sdwino_conv3x3_direct(x.cuda(), other, b.cuda(), 64, 1, ws, y=y)
    assert B.sdwino_last_device_status() != B.OK
    assert bool((y == 7.0).all())
