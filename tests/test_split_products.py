"""Tile products whose fp32 operands go to the tensor cores as three bf16 parts (csrc/ssd_split.cuh)."""
import math

import pytest
import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import CONFIGS, make_inputs, to_f64_numpy
from tests import parity_util as pu


def parts(x):
    """The three parts as the kernels make them: upper half of the bits, the rest to nearest, the rest of that."""
    p0 = (x.view(torch.int32) & -65536).view(torch.float32)
    r = x - p0
    p1 = r.bfloat16().float()
    s = r - p1
    return p0, p1, (s.view(torch.int32) & -65536).view(torch.float32)


@pytest.mark.parametrize("exponent", [-100, -60, 0, 60, 127])
def test_parts_are_exact_and_what_is_left_out_is_small(exponent):
    g = torch.Generator().manual_seed(exponent + 1000)
    x = (1 + torch.rand(1 << 16, generator=g)) * 2.0 ** exponent
    x[:3] = torch.tensor([2.0 ** exponent, (2 - 2.0 ** -23) * 2.0 ** exponent, (1 + 2.0 ** -23) * 2.0 ** exponent])
    x[::2] *= -1
    p = parts(x)
    assert torch.equal(sum(v.double() for v in p), x.double())
    for v in p:
        assert torch.equal(v.bfloat16().float(), v)
    assert ((p[1] / x).abs() < 2.0 ** -7).all() and ((p[2] / x).abs() <= 2.0 ** -16).all()
    # left out of x y: p1 q2 + p2 q1 + p2 q2, of either sign
    left = (p[2].double() / x.double()).mean().abs()
    assert left < 2.0 ** -16 / math.sqrt(len(x)) * 4


def config(dtype, L, H, N, G, chunk, seg, **extra):
    return CONFIGS[0].scaled(**dict(dict(name="split", dtype=dtype, B=1, L=L, H=H, P=64, N=N, G=G, chunk=chunk, seg=seg, h0_std=0.1,
                                         dh_std=0.1), **extra))


SHAPES = [("fp32", 64, 1, 64, 1, 64, 64), ("fp32", 512, 3, 128, 1, 256, 256), ("fp32", 384, 2, 64, 2, 128, 256),
          ("bf16", 64, 2, 64, 1, 64, 64), ("bf16", 768, 3, 128, 1, 256, 512), ("bf16", 384, 2, 128, 1, 128, 128)]


@pytest.mark.gpu
@pytest.mark.parametrize("decay", [0.0, 7.5, 8.5, 80.0])       # of 64 steps: masks by factors up to 8, beyond element by element
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%s-%d-%d-%d-%d-%d-%d" % s)
def test_products_against_the_oracle_on_both_sides_of_the_mask_rule(shape, decay):
    """fp32 outputs to 2^-24 of the largest argument of an exponential (a chunk's cumulative sum, twice: of t and of s) plus that of the
    sums, whose roundings are counted as one per 16 steps of a contraction of up to Q + N and one per chunk; eight units for what
    follows (head and row sums, suffix sums).  dA and dD add 64 L terms of either sign, about sqrt(64 L) times larger in all than
    their sum."""
    cfg = config(*shape)
    inp = make_inputs(cfg, "cuda", seed=int(decay) + 3)
    inp["A"][:] = -decay / 64 / 0.05
    inp["dt"][:] = 0.05
    if decay == 0.0:
        inp["A"][:] = -1e-6
    ref, got = pu.run_oracle(to_f64_numpy(inp), cfg.seg), pu.run_gpu(cfg, inp)
    unit = 2.0 ** -24 * (2 * decay * cfg.chunk / 64 + (cfg.chunk + cfg.N) / 16 + cfg.L / cfg.chunk + 8)
    for k, r in ref.items():
        e = pu.relerr(got[k], r)
        limit = 2.0 ** -8 if shape[0] == "bf16" and k in ("y", "dx", "dB", "dC") else unit * (math.sqrt(64 * cfg.L) if k in ("dA", "dD") else 1)
        assert e <= limit, (k, e, limit)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES[:3], ids=lambda s: "%s-%d-%d-%d-%d-%d-%d" % s)
@pytest.mark.parametrize("up", [40, -40, 100])
def test_powers_of_two_go_through_exactly(shape, up):
    """Every output is linear in x and h0 (y, states) or in dy and dh_final: scaled by a power of two they give the same bits,
    scaled, as long as no part leaves the range of bf16 (its smallest normal is that of fp32)."""
    cfg = config(*shape)
    inp = make_inputs(cfg, "cuda", seed=5)
    base = pu.run_gpu(cfg, inp)
    s = 2.0 ** up
    big = dict(inp, x=inp["x"] * s, h0=inp["h0"] * s)
    got = pu.run_gpu(cfg, big)
    for k in ("y", "h_final", "boundary", "dB", "dC", "ddt", "dA", "dD"):
        assert torch.equal(got[k], base[k] * s), k
    for k in ("dx", "dh0"):
        assert torch.equal(got[k], base[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_values_that_are_not_finite_stay_so_and_do_not_go_back_in_time(value):
    cfg = config("fp32", 512, 2, 64, 1, 128, 256)
    inp = make_inputs(cfg, "cuda", seed=6)
    base = pu.run_gpu(cfg, inp, want=("fwd",))
    inp["x"][0, 200, 1, 7] = value
    got = pu.run_gpu(cfg, inp, want=("fwd",))
    assert not torch.isfinite(got["y"][0, 200:, 1, 7]).any() and not torch.isfinite(got["h_final"][0, 1, 7]).any()
    assert torch.equal(got["y"][0, :128], base["y"][0, :128]) and torch.equal(got["y"][:, :, 0], base["y"][:, :, 0])
