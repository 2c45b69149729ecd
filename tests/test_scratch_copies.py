"""Segments side by side on the tensor-core path: each copy of the scratch used two times and more, on both sides of the size
(16 MiB of bf16 states a segment) up to which there is one copy more, against the same call in order on one stream."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs
from tests import parity_util as pu


def config(L, H, G, seg, B=1):
    return CONFIGS[0].scaled(name="copies", dtype="bf16", B=B, L=L, H=H, P=64, N=128, G=G, chunk=256, seg=seg, h0_std=0.1, dh_std=0.1)


@pytest.mark.gpu
@pytest.mark.parametrize("L,H,G,seg,B", [
    (2304, 8, 2, 256, 1),          # nine segments of two blocks
    (3328, 6, 3, 512, 2),          # six and a half
    (1024, 4, 1, 256, 1),          # the fewest that are run side by side
    (14336, 64, 1, 2048, 1),       # 16 MiB
    (14336, 66, 1, 2048, 1),       # just above
    (8192, 80, 8, 1024, 2),
])
def test_same_bits_as_in_order(L, H, G, seg, B):
    cfg = config(L, H, G, seg, B)
    inp = make_inputs(cfg, "cuda", seed=11)
    ref = pu.run_gpu(cfg, inp, flags=libssd.SSD_FLAG_SERIAL)
    for _ in range(3):
        got = pu.run_gpu(cfg, inp)
        for k in ref:
            assert torch.equal(got[k], ref[k]), k


@pytest.mark.gpu          # without the CUDA driver the query answers for the split path, which has none of these copies
@pytest.mark.parametrize("op", ["fwd", "bwd"])
def test_one_copy_more_of_small_segments(op):
    code = dict(fwd=libssd.SSD_OP_FWD_SEG, bwd=libssd.SSD_OP_BWD_SEG)[op]

    def states(cfg):              # copies of the bf16 states: what a call needs beyond the same one in order, in units of them
        mk = lambda flags: libssd.SSDShape(cfg.B, cfg.L, cfg.H, 64, cfg.N, cfg.G, cfg.chunk, cfg.seg, libssd.SSD_DTYPE_BF16, flags, 0, 0, 0)
        return (libssd.workspace_bytes(mk(0), code) - libssd.workspace_bytes(mk(libssd.SSD_FLAG_SERIAL), code)) / (
            cfg.B * cfg.H * cfg.seg // 128 * 64 * 128 * 2)

    small, large = states(config(14336, 64, 1, 2048)), states(config(14336, 66, 1, 2048))
    assert small > 1.5 and large > 1.5
    assert (small - large > 1.5) == (op == "bwd")
