"""ddflb_nn_conv3x3 with 64 channels on either side of the rule between its two kernels:
the same bits as with one TMA box per tap."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W", [(4, 32, 32), (16, 32, 32), (2, 64, 64), (4, 64, 64), (8, 64, 64),
                                   (16, 64, 64), (4, 128, 128)])
@pytest.mark.parametrize("N", [32, 64, 72, 96, 128, 192])
def test_same_bits_on_both_sides(B, H, W, N):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lib, C, P = D.load(), 64, B * H * W
    g = torch.Generator().manual_seed(P + N)
    x = torch.randn(B, H, W, C, generator=g).to(torch.bfloat16).cuda()
    w = (0.1 * torch.randn(N * 9 * C, generator=g)).to(torch.bfloat16).cuda()
    b = torch.randn(N, generator=g).cuda()
    out = []
    try:
        for path in (0, 1):
            lib.ddflb_nn_set_conv_path(path)
            y = torch.full((P, N), 7.0, device="cuda")
            D._check(lib.ddflb_nn_conv3x3(x.data_ptr(), B, H, W, C, C, w.data_ptr(), N,
                                          y.data_ptr(), N, None, 0, b.data_ptr(), 1, 0,
                                          torch.cuda.current_stream().cuda_stream))
            out.append(y)
        torch.cuda.synchronize()
    finally:
        lib.ddflb_nn_set_conv_path(0)
    assert torch.equal(*out)
