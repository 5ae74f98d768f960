"""The staged F(4x4) activation transform at the widths whose blocks hang over the right edge of the image (rows of tiles that
are no multiple of the block's 32 or 48): the bits of the register-only kernel."""
import pytest
import torch

from paper_2412_05781_b200 import workloads
from paper_2412_05781_b200.workloads import ConvLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(10, 16, 24, 320, 1), (9, 16, 37, 448, 2), (16, 16, 9, 576, 1), (12, 16, 20, 704, 1), (9, 16, 40, 832, 1)])
def test_widths_of_partial_blocks(shape):
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding as B
    C, K, H, W, N = shape
    x, w, b = workloads.make_inputs(ConvLayer(C=C, K=K, H=H, W=W, N=N), seed=sum(shape))
    wT = B.sdwino_filter_transform(w.cuda(), 4)
    ys = []
    try:
        for mode in (2, 0):
            B.sdwino_set_input_staging(mode)
            ws = B.alloc_workspace(B.sdwino_workspace_bytes(N, C, H, W, K, 4))
            ws.fill_(255)
            ys.append(B.sdwino_conv3x3(x.cuda(), wT, b.cuda(), K, 4, workspace=ws))
            assert B.sdwino_last_device_status() == B.OK
    finally:
        B.sdwino_set_input_staging(1)
    assert torch.equal(ys[0], ys[1]) and bool(torch.isfinite(ys[0]).all())
