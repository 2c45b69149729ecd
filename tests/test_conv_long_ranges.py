"""Backward of the convolution where a CTA's range is 64 tokens and more: the sums of dw and dbias left after every 64 tokens, ranges
that end on a sum's edge, just behind one and inside a stage, and the last, shorter range."""
import pytest
import torch

from oracle import ssd_oracle as orc
from tests.parity_util import TOL, relerr


@pytest.mark.gpu
@pytest.mark.parametrize("L", [190, 193, 256, 385, 400, 513])      # three blocks of channels x 50 sequences: two or three ranges each
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_sums_of_long_ranges(L, dtype):
    from paper_2411_19460_b200 import libssd

    B, C = 50, 1032
    td = torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator().manual_seed(L)
    u, g = (torch.randn(B, L, C, generator=gen).to(td).cuda() for _ in range(2))
    st = torch.randn(B, 3, C, generator=gen).to(td).cuda()
    dtail = torch.randn(B, 3, C, generator=gen).cuda()
    w, bias = (torch.randn(C, 4, generator=gen) * 0.5).cuda(), (torch.randn(C, generator=gen) * 0.1).cuda()
    f64 = lambda t: t.detach().double().cpu().numpy()
    refs = orc.conv_bwd(f64(u), f64(w), f64(bias), f64(st), f64(g), f64(dtail))
    got = libssd.ssd_conv_bwd(u, w, bias, st, g, dtail)
    for k, (a, r) in enumerate(zip(got, refs)):
        assert relerr(a, r) <= TOL[dtype]
        # dstate, dw, dbias are fp32 sums in either mode: 64 terms rounded to 2^-24 each, the reciprocal and exponential of a sigmoid to
        # 2^-22, and what the sum loses by terms of either sign (sqrt of their number)
        if k:
            assert relerr(a, r) <= 2.0 ** -22 * 8 * (B * L) ** 0.25
