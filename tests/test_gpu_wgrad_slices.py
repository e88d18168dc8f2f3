"""Weight gradient of a 3x3 convolution where the asked-for slices are more than
the units of 64 positions fill: every slice that is summed holds pixels."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,Ci,Co,splits", [
    (1, 16, 16, 32, 32, 4), (1, 32, 32, 32, 32, 13), (1, 32, 32, 16, 64, 16),
    (3, 12, 24, 32, 16, 13), (1, 8, 8, 96, 128, 1), (1, 24, 1, 32, 8, 24),
    (8, 120, 120, 32, 64, 48)])
def test_every_summed_slice_holds_pixels(B, H, W, Ci, Co, splits):
    """A constant output gradient and activation make every weight gradient the
    number of pixels that a tap reaches, exactly, whatever the order of the sum.
    Another convolution first leaves accumulators of its own in tensor memory."""
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lib = D.load()
    s = torch.cuda.current_stream().cuda_stream
    bf = dict(dtype=torch.bfloat16, device="cuda")
    big, w = torch.ones(16, 128, 128, 64, **bf), torch.ones(64 * 9 * 64, **bf)
    out = torch.empty(16, 128, 128, 64, device="cuda")
    x, dy = torch.ones(B, H, W, Ci, **bf), torch.ones(B, H, W, Co, **bf)
    part = torch.empty(splits * Co * 9 * Ci, device="cuda")
    dw = torch.empty(Co, 9, Ci, device="cuda")
    for _ in range(3):
        D._check(lib.ddflb_nn_conv3x3_dgrad(big.data_ptr(), 16, 128, 128, 64, 64, w.data_ptr(), 64,
                                            out.data_ptr(), 64, s))
        D._check(lib.ddflb_nn_conv3x3_wgrad(x.data_ptr(), B, H, W, Ci, Ci, dy.data_ptr(), Co, Co,
                                            dw.data_ptr(), splits, part.data_ptr(), s))
        n = torch.tensor([float(B * (H - (t // 3 != 1)) * (W - (t % 3 != 1))) for t in range(9)],
                         device="cuda")
        assert torch.equal(dw, n[None, :, None].expand_as(dw))
