"""What is held and computed in fp32 between a bf16 call's inputs and its fp32 outputs, against the fp64 oracle."""
import pytest

from paper_2411_19460_b200.inputs import CONFIGS, make_inputs, to_f64_numpy
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def config(L, H, N, G, chunk, seg, **extra):
    return CONFIGS[0].scaled(**dict(dict(name="precision", dtype="bf16", B=1, L=L, H=H, P=64, N=N, G=G, chunk=chunk, seg=seg, h0_std=0.1,
                                         dh_std=0.1), **extra))


@pytest.mark.parametrize("L,H,N,G,chunk,seg", [
    (1024, 8, 64, 1, 128, 256),
    (1024, 4, 64, 2, 256, 512),
    (640, 6, 128, 1, 128, 256),
    (1024, 6, 128, 2, 256, 256),       # three heads per group
    (768, 3, 128, 1, 256, 256),
    (512, 8, 128, 1, 64, 128),
])
def test_fp32_outputs_of_shapes_with_fp32_intermediates(L, H, N, G, chunk, seg):
    """bf16 inputs are exact to the oracle, so where weights, masked tiles and states stay in fp32 the fp32 outputs meet the
    fp32 tolerance; with any of them rounded to bf16 they are off by the order of 2^-9."""
    cfg = config(L, H, N, G, chunk, seg)
    inp = make_inputs(cfg, "cuda")
    ref = pu.run_oracle(to_f64_numpy(inp), cfg.seg)
    got = pu.run_gpu(cfg, inp)
    errs = {k: pu.relerr(got[k], ref[k]) for k in ("h_final", "boundary", "ddt", "dA", "dD", "dh0")}
    assert max(errs.values()) <= pu.TOL["fp32"], errs
