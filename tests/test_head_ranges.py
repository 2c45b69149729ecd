"""Split path: ranges of one, two, four and eight heads of the dB / dC sums, even and uneven ones, against the oracle."""
import pytest

from paper_2411_19460_b200.inputs import CONFIGS
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,L,H,G,N,chunk,seg", [
    ("fp32", 256, 3, 1, 64, 64, 128),           # one head each
    ("fp32", 1024, 7, 1, 64, 256, 512),         # two, the last one
    ("fp32", 1024, 12, 1, 64, 256, 512),        # four
    ("fp32", 1024, 24, 1, 64, 256, 256),        # eight
    ("fp32", 1024, 26, 1, 128, 256, 1024),      # seven, seven, seven, five
    ("bf16", 2048, 34, 2, 64, 128, 512),        # two groups of 17: six, six, five
])
def test_parity(dtype, L, H, G, N, chunk, seg):
    cfg = CONFIGS[0].scaled(name="ranges", dtype=dtype, B=1, L=L, H=H, P=64, N=N, G=G, chunk=chunk, seg=seg, h0_std=0.1, dh_std=0.1)
    pu.full_parity(cfg)
