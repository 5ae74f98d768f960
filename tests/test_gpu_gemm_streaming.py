"""GEMM launches that HBM bounds run a shorter operand ring: the bits of the same layer with the full ring (forced shape)."""
import pytest
import torch

from paper_2412_05781_b200 import workloads
from paper_2412_05781_b200.workloads import ConvLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(256, 128, 400, 404, 1), (130, 120, 520, 516, 1), (64, 16, 1024, 1024, 1)])
def test_short_ring_has_the_bits_of_the_full_ring(shape):
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding as B
    C, K, H, W, N = shape
    x, w, b = workloads.make_inputs(ConvLayer(C=C, K=K, H=H, W=W, N=N), seed=sum(shape))
    wT = B.sdwino_filter_transform(w.cuda(), 4)
    nbytes = B.sdwino_workspace_bytes(N, C, H, W, K, 4)
    _, n_tile, blocks, stages = B.sdwino_selftest_gemm_shape(N, C, H, W, K, 4, nbytes)
    assert blocks == 1 and stages <= 5
    ws = B.alloc_workspace(nbytes)
    ys = []
    try:
        for force in (0, n_tile):
            B.sdwino_set_gemm_shape(1 if force else 0, force)
            ws.fill_(255)
            ys.append(B.sdwino_conv3x3(x.cuda(), wT, b.cuda(), K, 4, workspace=ws))
            assert B.sdwino_last_device_status() == B.OK
    finally:
        B.sdwino_set_gemm_shape(0, 0)
    assert torch.equal(ys[0], ys[1]) and bool(torch.isfinite(ys[0]).all())
