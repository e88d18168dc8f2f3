"""The convolutions with few input channels (ddflb_nn_conv3x3_narrow, _dgrad)
against im2col + GEMM and GEMM + col2im on the same BF16 data: the same products
in the same order, so bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


def _setup(B, H, W, C, cs, off, n, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    buf = torch.randn(B, H, W, cs, generator=g).to(torch.bfloat16).cuda()
    wt = (0.1 * torch.randn(n, generator=g)).to(torch.bfloat16).cuda()
    return buf, buf[..., off:], buf[..., off:off + C].contiguous(), wt, g


# row segments (W a multiple of 128) and padded rows: sizes at the edges of the
# 128-position tiles, one-row images, several N tiles, channel-strided input
SHAPES = [(2, 5, 128, 16, 16, 0, 32), (1, 3, 256, 32, 64, 32, 32), (2, 4, 128, 64, 64, 0, 96),
          (1, 1, 384, 32, 32, 0, 64), (3, 7, 9, 16, 24, 8, 16), (2, 16, 16, 32, 32, 0, 40),
          (5, 12, 30, 64, 64, 0, 64), (2, 33, 62, 32, 32, 0, 72), (1, 64, 126, 16, 16, 0, 64),
          (2, 24, 192, 32, 40, 0, 32), (1, 2, 130, 64, 64, 0, 128), (4, 1, 1, 16, 16, 0, 8)]


@pytest.mark.parametrize("B,H,W,C,cs,off,N", SHAPES)
def test_narrow_conv_equals_im2col_gemm(B, H, W, C, cs, off, N):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lib = D.load()
    buf, x, xc, wt, g = _setup(B, H, W, C, cs, off, N * 9 * C, B * H + W + C + N)
    bias = torch.randn(N, generator=g).cuda()
    P, s = B * H * W, torch.cuda.current_stream().cuda_stream
    yf, yb = torch.full((P, N), 7.0, device="cuda"), torch.empty(P, N, dtype=torch.bfloat16,
                                                                 device="cuda")
    D._check(lib.ddflb_nn_conv3x3_narrow(x.data_ptr(), B, H, W, C, cs, wt.data_ptr(), N,
                                         yf.data_ptr(), N, yb.data_ptr(), N, bias.data_ptr(), 1, 0,
                                         s))
    col = torch.empty(P * 9 * C, dtype=torch.bfloat16, device="cuda")
    D._check(lib.ddflb_nn_im2col(xc.data_ptr(), B, H, W, C, C, col.data_ptr(), 0, s))
    rf, rb = torch.empty_like(yf), torch.empty_like(yb)
    D._check(lib.ddflb_nn_gemm(col.data_ptr(), wt.data_ptr(), P, N, 9 * C, 9 * C, 9 * C,
                               rf.data_ptr(), N, rb.data_ptr(), N, bias.data_ptr(), 1, 0, 1, None,
                               s))
    torch.cuda.synchronize()
    assert torch.equal(yf, rf) and torch.equal(yb, rb)


@pytest.mark.parametrize("B,H,W,C,cs,off,N", SHAPES)
def test_dgrad_equals_gemm_col2im(B, H, W, C, cs, off, N):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lib = D.load()
    buf, dy, dyc, wt, _ = _setup(B, H, W, C, cs, off, C * 9 * N, B + H + W + C + N)
    P, s = B * H * W, torch.cuda.current_stream().cuda_stream
    dx = torch.full((P, N), 7.0, device="cuda")
    D._check(lib.ddflb_nn_conv3x3_dgrad(dy.data_ptr(), B, H, W, C, cs, wt.data_ptr(), N,
                                        dx.data_ptr(), N, s))
    wT = torch.empty(9 * N, C, dtype=torch.bfloat16, device="cuda")
    D._check(lib.ddflb_nn_transpose(wt.data_ptr(), C, 9 * N, 9 * N, wT.data_ptr(), s))
    dcol, ref = torch.empty(P, 9 * N, device="cuda"), torch.empty_like(dx)
    D._check(lib.ddflb_nn_gemm(dyc.data_ptr(), wT.data_ptr(), P, 9 * N, C, C, C, dcol.data_ptr(),
                               9 * N, None, 0, None, 0, 0, 1, None, s))
    D._check(lib.ddflb_nn_col2im(dcol.data_ptr(), B, H, W, N, ref.data_ptr(), N, s))
    torch.cuda.synchronize()
    assert torch.equal(dx, ref)


@pytest.mark.parametrize("B,H,W,Ci,Co,splits", [
    (2, 5, 128, 16, 32, 3), (1, 3, 256, 32, 16, 1), (2, 4, 64, 64, 128, 5), (1, 1, 384, 32, 64, 2),
    (3, 7, 9, 16, 8, 2), (2, 16, 16, 96, 40, 4), (5, 12, 30, 64, 64, 7), (2, 33, 62, 32, 72, 3),
    (2, 24, 192, 32, 32, 11), (16, 16, 16, 128, 128, 2), (4, 1, 1, 32, 16, 1),
    (2, 200, 128, 32, 32, 25)])
def test_wgrad(B, H, W, Ci, Co, splits):
    """Against the transposed im2col + split GEMM: bit for bit where the width is
    a multiple of 64 (the same order of pixels), and everywhere within FP32
    rounding of the FP64 sum."""
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lib = D.load()
    g = torch.Generator().manual_seed(B * H * W + Ci + Co)
    csx, csg, P = Ci + 16, Co + 8, B * H * W
    s = torch.cuda.current_stream().cuda_stream
    x = torch.randn(B, H, W, csx, generator=g).to(torch.bfloat16).cuda()
    dy = torch.randn(B, H, W, csg, generator=g).to(torch.bfloat16).cuda()
    part = torch.full((splits * Co * 9 * Ci,), float("nan"), device="cuda")
    dw = torch.empty(Co, 9 * Ci, device="cuda")
    D._check(lib.ddflb_nn_conv3x3_wgrad(x[..., 8:].data_ptr(), B, H, W, Ci, csx, dy.data_ptr(), Co,
                                        csg, dw.data_ptr(), splits, part.data_ptr(), s))
    xc, dyc = x[..., 8:8 + Ci].contiguous(), dy[..., :Co].contiguous()
    if W % 64 == 0:
        col = torch.empty(9 * Ci * P, dtype=torch.bfloat16, device="cuda")
        D._check(lib.ddflb_nn_im2col(xc.data_ptr(), B, H, W, Ci, Ci, col.data_ptr(), 1, s))
        gT, ref = dyc.reshape(P, Co).t().contiguous(), torch.empty_like(dw)
        D._check(lib.ddflb_nn_gemm(gT.data_ptr(), col.data_ptr(), Co, 9 * Ci, P, P, P,
                                   ref.data_ptr(), 9 * Ci, None, 0, None, 0, 0, splits,
                                   part.data_ptr(), s))
        assert torch.equal(dw, ref)
    xp, gd = torch.nn.functional.pad(xc.double(), (0, 0, 1, 1, 1, 1)), dyc.double().reshape(-1, Co)
    ref, mag = [], []
    for t in range(9):
        xs = xp[:, t // 3:t // 3 + H, t % 3:t % 3 + W].reshape(-1, Ci)
        ref.append(gd.t() @ xs)
        mag.append(gd.abs().t() @ xs.abs())
    ref, mag = torch.stack(ref, 1).reshape(Co, -1), torch.stack(mag, 1).reshape(Co, -1)
    # one FP32 rounding (or truncation) per 16 pixels and per slice, of a running
    # sum no larger than the sum of magnitudes
    bound = 2.0 ** -23 * (P / 16 + splits + 16) * mag
    assert bool(((dw.double() - ref).abs() <= bound).all())
