"""Which layers the convolutions straight from the activation take: one rule, the
library's, for the C entry points and for the network that falls back on im2col."""
import pytest

from paper_1908_06742_gb300 import build as B
from paper_1908_06742_gb300 import ddflb as D

NARROW, DGRAD, WGRAD = 0, 1, 2


@pytest.mark.parametrize("form,B_,H,W,C,N,ok", [
    (NARROW, 16, 128, 128, 16, 32, 1), (NARROW, 1, 8, 1536, 64, 64, 1),
    (NARROW, 1, 1608, 1600, 16, 16, 1), (NARROW, 1, 1640, 1640, 16, 16, 0),
    (NARROW, 1, 2048, 1592, 16, 16, 0), (NARROW, 1, 2048, 2048, 16, 16, 1),
    (NARROW, 4, 64, 64, 48, 32, 0), (NARROW, 1, 8, 1000, 64, 64, 0),
    (DGRAD, 1, 2048, 1592, 16, 16, 0), (DGRAD, 1, 1608, 1592, 16, 16, 1),
    (WGRAD, 1, 1640, 1640, 32, 32, 0), (WGRAD, 1, 1024, 2040, 16, 8, 0),
    (WGRAD, 1, 1600, 1624, 32, 32, 1),
    (WGRAD, 1, 1640, 1664, 32, 32, 1), (WGRAD, 4, 64, 64, 16, 128, 1),
    (WGRAD, 4, 64, 64, 48, 32, 0), (WGRAD, 4, 64, 64, 32, 136, 0),
    (WGRAD, 4, 64, 64, 32, 12, 0), (3, 4, 64, 64, 32, 32, 0), (NARROW, 0, 64, 64, 32, 32, 0)])
def test_takes(form, B_, H, W, C, N, ok):
    B.build()
    assert D.load().ddflb_nn_conv3x3_takes(form, B_, H, W, C, N) == ok


@pytest.mark.gpu
@pytest.mark.parametrize("c,H,W,form,train", [(8, 1024, 2040, WGRAD, True),
                                              (16, 2048, 1592, NARROW, False)])
def test_network_beyond_the_limits(c, H, W, form, train):
    """Images beyond a limit run through im2col + GEMM, as with implicit=False,
    beside layers that are within it: equal outputs and gradients within the
    rounding of BF16 gradients summed in another order."""
    import torch
    from paper_1908_06742_gb300 import surrogate as S
    g = torch.Generator().manual_seed(3)
    x = torch.randn(1, H, W, S.CIN, generator=g).to(torch.bfloat16).cuda()
    t = torch.randn(1, H, W, S.COUT, generator=g).cuda()
    got = []
    for implicit in (True, False):
        net = S.UNet(c=c, batch=1, H=H, W=W)
        net.implicit = implicit
        assert not net.direct["e1a"][form] and any(d[form] for d in net.direct.values())
        got.append([net.forward(x).clone()])
        if train:
            net.backward(t)
            got[-1] += [net.p[n]["gw"].clone() for n in net.p]
        torch.cuda.synchronize()
        del net
    for a, b in zip(*got):
        assert float((a - b).norm()) <= 2.0 ** -8 * float(b.norm())
