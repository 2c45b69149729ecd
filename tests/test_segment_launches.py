"""The edges of what a launch covers, against the fp64 oracle: blocks of 128 steps on the tensor-core path (chunks of 256, N = 128,
an even number of heads per group: one chunk, two heads, five and more segments so that every scratch copy is used twice, a
short last segment, stiff and mild decays, head ranges of dB/dC, one and two heads per CTA of the forward chain), and CUDA-core
launches that carry the sums of the neighbouring segment (one segment, two, a short last one, one 64-step tile per chunk and
four, both state sizes, odd numbers of heads, both dtypes).  In order on one stream the same bits come out."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

STIFF = dict(a_max=64.0, dt_lo=1e-4, dt_hi=1.0)


@pytest.mark.parametrize("dtype,L,H,G,N,chunk,seg,extra", [
    ("bf16", 128, 1, 1, 128, 128, 128, {}),
    ("bf16", 640, 3, 1, 64, 128, 256, {}),
    ("bf16", 1152, 5, 1, 128, 128, 128, {}),
    ("bf16", 1792, 6, 2, 128, 256, 256, STIFF),
    ("bf16", 768, 9, 1, 64, 128, 128, dict(B=2)),
    ("bf16", 1024, 20, 1, 128, 256, 512, {}),
    ("bf16", 256, 2, 1, 128, 256, 256, {}),
    ("bf16", 1792, 12, 2, 128, 256, 256, STIFF),
    ("bf16", 2304, 6, 3, 128, 256, 512, dict(B=2)),
    ("bf16", 1280, 76, 2, 128, 256, 256, {}),          # two heads per CTA of the forward chain
    ("bf16", 1280, 76, 1, 128, 256, 256, STIFF),
    ("bf16", 768, 76, 1, 128, 256, 768, dict(B=2)),
    ("bf16", 1152, 76, 2, 128, 128, 256, {}),
    ("bf16", 640, 76, 1, 64, 128, 128, STIFF),
    ("bf16", 384, 76, 1, 128, 128, 384, dict(B=2)),
    ("fp32", 64, 1, 1, 64, 64, 64, {}),
    ("fp32", 320, 3, 1, 64, 64, 128, {}),
    ("fp32", 1280, 5, 1, 128, 256, 512, STIFF),
    ("fp32", 512, 2, 2, 128, 128, 256, dict(B=2)),
    ("bf16", 192, 3, 1, 128, 64, 64, {}),
    ("fp32", 4096, 16, 4, 64, 256, 1024, {}),          # long sequences: fewer head ranges of dB/dC
    ("fp32", 8192, 5, 1, 64, 128, 2048, STIFF),
    ("fp32", 8320, 32, 1, 128, 64, 4160, {}),          # segments too large to run side by side in the forward
])
def test_launch_edges(dtype, L, H, G, N, chunk, seg, extra):
    cfg = CONFIGS[0].scaled(**dict(dict(name="edge", dtype=dtype, B=1, L=L, H=H, P=64, N=N, G=G, chunk=chunk, seg=seg, h0_std=0.1,
                                        dh_std=0.1), **extra))
    pu.full_parity(cfg, flags=0)
    inp = make_inputs(cfg, "cuda")
    a, b = pu.run_gpu(cfg, inp), pu.run_gpu(cfg, inp, flags=libssd.SSD_FLAG_SERIAL)
    for k in a:
        assert torch.equal(a[k], b[k]), k
