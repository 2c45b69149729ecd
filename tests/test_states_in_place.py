"""States and state gradients in place: h_final given as h0, dh0 as dh_final or as the boundary state.  Where a segment's readers would
make its states beside the CTAs that store the new one (csrc/ssd_api.cu), the call has to take the state pass, whose threads read and
store an element of their own."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs

pytestmark = pytest.mark.gpu

NAMES = ("x", "dt", "A", "Bm", "Cm", "D")


def case(dtype, B, H, N, chunk, nc, seg):
    cfg = CONFIGS[0].scaled(name="in_place", dtype=dtype, B=B, L=nc * chunk, H=H, P=64, N=N, G=1, chunk=chunk, seg=seg * chunk,
                            h0_std=0.5, dh_std=0.5)
    inp = make_inputs(cfg, "cuda", seed=21)
    return cfg, inp, [inp[k] for k in NAMES]


CASES = [
    # one segment of 1, 4 and 8 chunks, heads enough for more CTAs than are resident at once
    ("fp32", 1, 640, 64, 64, 1, 1), ("fp32", 1, 160, 64, 64, 4, 4), ("fp32", 1, 36, 64, 64, 8, 8), ("fp32", 2, 36, 128, 128, 4, 4),
    ("bf16", 1, 640, 64, 64, 1, 1), ("bf16", 1, 160, 64, 64, 4, 4), ("bf16", 1, 36, 64, 64, 8, 8), ("bf16", 2, 36, 128, 128, 4, 4),
    ("fp32", 1, 64, 64, 64, 9, 9),          # nine chunks: state passes in any case
    ("fp32", 1, 64, 64, 64, 8, 4),          # two segments
    ("bf16", 1, 160, 128, 256, 3, 3),       # tensor cores
    ("bf16", 1, 80, 128, 256, 8, 1),        # tensor cores, segments side by side
]


@pytest.mark.parametrize("flags", [0, libssd.SSD_FLAG_SERIAL])
@pytest.mark.parametrize("shape", CASES, ids=lambda s: "%s-%d-%d-%d-%d-%d-%d" % s)
def test_states_in_place_give_the_bits_of_separate_buffers(shape, flags):
    cfg, inp, ins = case(*shape)
    kw = dict(chunk=cfg.chunk, seg=cfg.seg, flags=flags)
    y0, hf0 = libssd.ssd_fwd(*ins, inp["h0"], **kw)
    y1, hf1, bd1 = libssd.ssd_fwd_segmented(*ins, inp["h0"], **kw)
    g0 = libssd.ssd_bwd_segmented(*ins, bd1, inp["dy"], inp["dh_final"], **kw)
    assert torch.equal(y0, y1) and torch.equal(hf0, hf1)
    one_row = cfg.B == 1 or cfg.seg >= cfg.L
    for _ in range(20):
        h = inp["h0"].clone()
        y, hf = libssd.ssd_fwd(*ins, h, h_final=h, **kw)
        assert torch.equal(y, y0) and torch.equal(h, hf0)
        h = inp["h0"].clone()
        y, hf, bd = libssd.ssd_fwd_segmented(*ins, h, h_final=h, **kw)
        assert torch.equal(y, y0) and torch.equal(h, hf0) and torch.equal(bd, bd1)
        if one_row:
            bd = torch.zeros_like(bd1)
            bd.view(-1)[:h.numel()] = inp["h0"].view(-1)
            y, hf, _ = libssd.ssd_fwd_segmented(*ins, bd.view(-1)[:h.numel()].view_as(h), boundary=bd, **kw)
            assert torch.equal(y, y0) and torch.equal(hf, hf0) and torch.equal(bd, bd1)
        for source in ("dh_final", "boundary"):
            if source == "boundary" and not one_row:
                continue
            bd, dh = bd1.clone(), inp["dh_final"].clone()
            out = {k: torch.empty_like(v) for k, v in g0.items()}
            out["dh0"] = dh if source == "dh_final" else bd.view(-1)[:dh.numel()].view_as(dh)
            libssd.ssd_bwd_segmented(*ins, bd, inp["dy"], dh, out=out, **kw)
            for k, v in g0.items():
                assert torch.equal(out[k], v), (source, k)


def launches(kind, call):
    libssd.profile(True)
    call()
    torch.cuda.synchronize()
    n = libssd.profile_read()[kind][1]
    libssd.profile(False)
    return n


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("nc,seg", [(1, 1), (4, 4), (8, 8), (8, 4)])
def test_in_place_states_take_the_state_pass(dtype, nc, seg):
    """Which way a call goes, by its launches: that in-place calls happen to come out right on one run shows nothing."""
    cfg, inp, ins = case(dtype, 1, 4, 64, 64, nc, seg)
    kw = dict(chunk=cfg.chunk, seg=cfg.seg)
    alone = nc == seg
    _, hf, bd = libssd.ssd_fwd_segmented(*ins, inp["h0"], **kw)
    nh = hf.numel()

    def fwd(h0, h_final, boundary=None):
        if boundary is None:
            return launches("state_pass_fwd", lambda: libssd.ssd_fwd(*ins, h0, h_final=h_final, **kw))
        return launches("state_pass_fwd", lambda: libssd.ssd_fwd_segmented(*ins, h0, h_final=h_final, boundary=boundary, **kw))

    def bwd(dh0, dh_final, boundary):
        g = libssd.ssd_bwd_segmented(*ins, bd, inp["dy"], inp["dh_final"], **kw)
        return launches("state_pass_bwd", lambda: libssd.ssd_bwd_segmented(*ins, boundary, inp["dy"], dh_final, out=dict(g, dh0=dh0), **kw))

    h, spare = inp["h0"].clone(), torch.empty_like(hf)
    wide = torch.zeros(2 * nh, device="cuda")
    half = wide[nh // 2:nh // 2 + nh].view_as(hf)
    assert fwd(h, spare) == 0 and fwd(None, h) == 0 and fwd(h, spare, bd.clone()) == 0
    assert fwd(h, h) == (1 if alone else 0)
    assert fwd(wide[:nh].view_as(hf), half) == (1 if alone else 0)          # any byte in common
    b2 = bd.clone()
    assert fwd(b2.view(-1)[:nh].view_as(hf), spare, b2) == nc // seg
    assert bwd(spare, h, bd) == 0 and bwd(spare, None, bd) == 0
    assert bwd(h, h, bd) == (1 if alone else 0)
    assert bwd(b2.view(-1)[:nh].view_as(hf), h, b2) == nc // seg
