"""Split path, short segments: states made by their readers from the chunk sums against state passes, which the same call in order on
one stream runs: the same bits.  Both sides of the rule (eight chunks a segment, 1024 tiles), short last segments, one segment."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,L,H,N,G,chunk,seg", [
    ("fp32", 1, 64, 1, 64, 1, 64, 64),          # one chunk
    ("fp32", 1, 1024, 4, 64, 1, 64, 512),       # eight chunks
    ("fp32", 1, 1152, 4, 64, 1, 64, 576),       # nine: state passes
    ("fp32", 2, 1792, 3, 128, 1, 256, 512),     # a short last segment
    ("fp32", 1, 1280, 6, 128, 2, 128, 1280),    # one segment, ten chunks: state passes
    ("bf16", 1, 768, 5, 64, 1, 128, 384),
    ("bf16", 2, 1344, 4, 128, 2, 64, 320),
    ("bf16", 1, 2048, 64, 64, 1, 128, 512),     # 768 tiles
    ("bf16", 1, 2048, 88, 64, 1, 128, 512),     # 1056: state passes
])
@pytest.mark.parametrize("ends", [True, False])
def test_same_bits_as_with_state_passes(dtype, B, L, H, N, G, chunk, seg, ends):
    cfg = CONFIGS[0].scaled(name="readers", dtype=dtype, B=B, L=L, H=H, P=64, N=N, G=G, chunk=chunk, seg=seg, h0_std=0.1, dh_std=0.1)
    inp = make_inputs(cfg, "cuda", seed=13)
    if not ends:
        inp["h0"] = inp["dh_final"] = None
    got, ref = pu.run_gpu(cfg, inp), pu.run_gpu(cfg, inp, flags=libssd.SSD_FLAG_SERIAL)
    for k in ref:
        assert torch.equal(got[k], ref[k]), k
