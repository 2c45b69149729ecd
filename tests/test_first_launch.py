"""The first launch of a call: it clears the status word, and the inputs that it reads ahead of its dependency are complete although
the kernel before it in the stream, the library's own or not, has just been launched."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs

pytestmark = pytest.mark.gpu

SHAPES = [("bf16", 2048, 24, 128, 256, 256), ("bf16", 1024, 8, 128, 256, 1024), ("bf16", 1024, 6, 64, 128, 256), ("fp32", 512, 4, 64, 64, 128)]


def setup(dtype, L, H, N, chunk, seg):
    cfg = CONFIGS[0].scaled(name="first", dtype=dtype, B=1, L=L, H=H, P=64, N=N, G=1, chunk=chunk, seg=seg, h0_std=0.1)
    return cfg, make_inputs(cfg, "cuda", seed=17)


@pytest.mark.parametrize("flags", [0, libssd.SSD_FLAG_SERIAL])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%s-%d-%d-%d-%d-%d" % s)
def test_status_word_is_cleared(shape, flags):
    cfg, i = setup(*shape)
    ins = (i["x"], i["dt"], i["A"], i["Bm"], i["Cm"], i["D"])
    s = libssd.make_shape(i["x"], i["Bm"], cfg.chunk, cfg.seg, flags=flags)
    for op in (libssd.SSD_OP_FWD_SEG, libssd.SSD_OP_BWD_SEG):
        ws = libssd.alloc_workspace(s, op, torch.device("cuda"))
        ws[:256] = 255
        if op == libssd.SSD_OP_FWD_SEG:
            _, _, boundary = libssd.ssd_fwd_segmented(*ins, i["h0"], chunk=cfg.chunk, seg=cfg.seg, flags=flags, ws=ws)
        else:
            libssd.ssd_bwd_segmented(*ins, boundary, i["dy"], None, chunk=cfg.chunk, seg=cfg.seg, flags=flags, ws=ws)
        torch.cuda.synchronize()
        assert libssd.poll_status(ws) == libssd.SSD_OK


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%s-%d-%d-%d-%d-%d" % s)
def test_inputs_written_just_before_the_call(shape):
    """y of a call is x (then dy) of the next ones, with nothing but the stream between them; the same with a wait after each."""
    cfg, i = setup(*shape)
    args = (i["dt"], i["A"], i["Bm"], i["Cm"], i["D"])

    def run(wait):
        x = i["x"].clone()
        out = []
        for _ in range(6):
            y, _, boundary = libssd.ssd_fwd_segmented(x, *args, i["h0"], chunk=cfg.chunk, seg=cfg.seg)
            wait()
            g = libssd.ssd_bwd_segmented(x, *args, boundary, y, None, chunk=cfg.chunk, seg=cfg.seg)
            wait()
            x = (y + g["dx"]) * 0.01
            wait()
            out += [y, g["dB"], g["ddt"]]
        torch.cuda.synchronize()
        return out

    ref = run(torch.cuda.synchronize)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(run(lambda: None), ref))
