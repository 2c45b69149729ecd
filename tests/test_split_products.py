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


@pytest.mark.parametrize("exponent", [-110, -111, -120, -126, -135, -148])
def test_parts_of_the_smallest_values(exponent):
    """Exact from 2^-110 up, where the last bit of an fp32 value is bf16's smallest number; below, what lies under that is missing."""
    g = torch.Generator().manual_seed(exponent + 1000)
    x = ((1 + torch.rand(1 << 14, generator=g).double()) * 2.0 ** exponent).float()
    x[::2] *= -1
    off = (sum(v.double() for v in parts(x)) - x.double()).abs().max().item()
    assert off < 2.0 ** -133 and (off == 0) == (exponent >= -110)


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


INFINITE = [("fp32", 64, 128), ("fp32", 128, 256), ("bf16", 64, 128), ("bf16", 128, 64)]


def same(a, b):
    return torch.equal(a.float().view(torch.int32), b.float().view(torch.int32))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,N,chunk", INFINITE)
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_infinities_come_out_as_infinities(dtype, N, chunk, sign):
    """An infinite operand times the parts of either sign of the other is NaN; the recurrence has an infinity there, whose sign the
    inputs say.  Whatever the infinity does not reach keeps its bits, in the same tile too."""
    cfg = config(dtype, 512, 2, N, 1, chunk, 256)
    inp = make_inputs(cfg, "cuda", seed=6)
    base = pu.run_gpu(cfg, inp)
    inf = sign * float("inf")
    t, h, p, n = 200, 1, 7, 9
    c0, c1 = t // chunk * chunk, (t // chunk + 1) * chunk               # its chunk
    B, C = inp["Bm"][0, :, 0].double(), inp["Cm"][0, :, 0].double()
    others = [i for i in range(64) if i != p]

    def run(name, at):
        i = dict(inp, **{name: inp[name].clone()})
        i[name][at] = inf
        got = pu.run_gpu(cfg, i)
        for k, v in pu.run_gpu(cfg, i, flags=libssd.SSD_FLAG_SERIAL).items():
            assert same(v, got[k]), (name, k)
        return got

    def expect(got, signs, what):
        assert torch.equal(got.double(), (torch.sign(signs) * inf).expand_as(got).double()), what

    got = run("x", (0, t, h, p))
    expect(got["y"][0, t + 1:c1, h, p], C[t + 1:c1] @ B[t], "x -> y")
    expect(got["h_final"][0, h, p], B[t], "x -> h_final")
    expect(got["boundary"][0, 1, h, p], B[t], "x -> boundary")
    assert same(got["y"][0, :, h, others], base["y"][0, :, h, others]) and same(got["y"][:, :, 0], base["y"][:, :, 0])
    assert same(got["y"][0, :t // 64 * 64], base["y"][0, :t // 64 * 64]) and same(got["h_final"][0, h, others], base["h_final"][0, h, others])
    dy = inp["dy"][0, :, h].double()
    rows = slice(t + 1, c1)
    if c1 > t + 1:                     # W_ts = (dy_t . x_s) e dt: one infinite column, added up over the heads into dC = W B
        expect(got["dC"][0, rows, 0], torch.sign(dy[rows, p])[:, None] * torch.sign(B[t])[None], "x -> dC")

    got = run("h0", (0, h, p, n))
    expect(got["y"][0, :, h, p], C[:, n], "h0 -> y")
    expect(got["dC"][0, :, 0, n], dy[:, p], "h0 -> dC")
    assert got["h_final"][0, h, p, n] == inf and same(got["y"][0, :, h, others], base["y"][0, :, h, others])
    keep = [i for i in range(N) if i != n]
    assert same(got["h_final"][0, h, p, keep], base["h_final"][0, h, p, keep]) and same(got["dC"][0, :, 0, keep], base["dC"][0, :, 0, keep])

    got = run("dy", (0, t, h, p))
    expect(got["dx"][0, c0:t, h, p], B[c0:t] @ C[t], "dy -> dx")
    expect(got["dh0"][0, h, p], C[t], "dy -> dh0")
    assert same(got["dx"][0, :, h, others], base["dx"][0, :, h, others]) and same(got["dh0"][0, h, others], base["dh0"][0, h, others])
    assert same(got["dx"][0, (t // 64 + 1) * 64:], base["dx"][0, (t // 64 + 1) * 64:])

    got = run("Bm", (0, t, 0, n))
    x = inp["x"][0, t].double()                                          # [H, P]
    expect(got["h_final"][0, :, :, n], x, "B -> h_final")
    expect(got["y"][0, t + 1:c1], torch.sign(C[t + 1:c1, n])[:, None, None] * torch.sign(x)[None], "B -> y")
    assert same(got["h_final"][0, :, :, keep], base["h_final"][0, :, :, keep])


@pytest.mark.gpu
def test_infinities_where_every_tile_of_y_makes_its_own_products():
    """24 heads in 8 groups, segments of 1024 steps: the built-in scratch has no room for C B^T."""
    cfg = config("fp32", 2048, 24, 64, 8, 64, 1024)
    inp = make_inputs(cfg, "cuda", seed=8)
    inp["x"][0, 300, 3, 5] = float("inf")
    inp["Cm"][0, 700, 2, 11] = float("-inf")
    kw = dict(chunk=cfg.chunk, seg=cfg.seg)
    ins = [inp[k] for k in ("x", "dt", "A", "Bm", "Cm", "D", "h0")]
    y, hf = libssd.ssd_fwd(*ins, **kw)
    ys, hs = libssd.ssd_fwd_static_ws(*ins, y=torch.empty_like(y), h_final=torch.empty_like(hf), **kw)
    assert torch.isinf(y).any() and same(y, ys) and same(hf, hs)


@pytest.mark.gpu
@pytest.mark.parametrize("up", [-112, -118])
def test_values_below_the_exact_range_miss_only_bf16s_smallest_number(up):
    """x and h0 scaled to where their last bits lie below 2^-133: y is off by no more than what all its operands of that size miss."""
    cfg = config("fp32", 512, 3, 128, 1, 128, 256)
    inp = make_inputs(cfg, "cuda", seed=5)
    base, s = pu.run_gpu(cfg, inp, want=("fwd",)), 2.0 ** up
    got = pu.run_gpu(cfg, dict(inp, x=inp["x"] * s, h0=inp["h0"] * s), want=("fwd",))
    B, C, dt = (inp[k].double() for k in ("Bm", "Cm", "dt"))
    B, C, dt, Q = B[0, :, 0].abs(), C[0, :, 0].abs(), dt[0], cfg.chunk
    # every operand of that size misses less than 2^-133: x in the masked products of a chunk, the weighted x in the sums of all chunks
    # before, the state in C H
    cb = (inp["Cm"][0, :, 0].double() @ inp["Bm"][0, :, 0].double().T).abs()
    rows = max((cb[c:c + Q, c:c + Q] @ dt[c:c + Q]).max().item() for c in range(0, cfg.L, Q))
    states = (C @ (1 + B.sum(0))).max().item()
    bound = 2.0 ** -133 * (rows + states) + 2.0 ** -23 * base["y"].abs().max().item() * s
    off = (got["y"].double() - base["y"].double() * s).abs().max().item()
    assert off <= bound, (off, bound)
