"""What is held and computed in fp32 between a bf16 call's inputs and its fp32 outputs, against the fp64 oracle."""
import pytest
import torch

from paper_2411_19460_b200 import libssd
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


def rounded_algebra(i, T=128):
    """ddt, dB and dC with the roundings that the tensor-core path cannot do without, in fp64 otherwise: bf16 states (where they meet
    dy, x and the other state), bf16 decayed rows where they meet a state or make a state sum, bf16 dB and dC.  Everything between
    two steps of one block is exact.  B = G = 1."""
    def bf(v):
        return v.float().bfloat16().double()

    i = {k: v.double() for k, v in i.items()}
    x, dy = i["x"][0].transpose(0, 1), i["dy"][0].transpose(0, 1)                   # [H, L, P]
    dt, A, Bm, Cm = i["dt"][0].T, i["A"], i["Bm"][0, :, 0], i["Cm"][0, :, 0]
    H, L = dt.shape
    cs = torch.cumsum((dt * A[:, None]).view(H, L // T, T), -1)
    states, h = [], i["h0"][0]
    for c in range(L // T):
        s = slice(c * T, (c + 1) * T)
        states.append(h)
        w = torch.exp(cs[:, c, -1:] - cs[:, c]) * dt[:, s]
        h = torch.exp(cs[:, c, -1])[:, None, None] * h + torch.einsum("hsp,sn->hpn", bf(x[:, s] * w[..., None]), Bm[s])
    ddt, dB, dC, g = torch.empty_like(dt), torch.empty_like(Bm), torch.empty_like(Cm), i["dh_final"][0]
    causal = torch.tril(torch.ones(T, T, dtype=torch.bool, device=x.device))
    for c in reversed(range(L // T)):
        s, k = slice(c * T, (c + 1) * T), cs[:, c]
        mask = torch.exp((k[:, :, None] - k[:, None, :]).masked_fill(~causal, -1e9))
        wd = torch.einsum("htp,hsp->hts", dy[:, s], x[:, s]) * mask
        z = wd * (Cm[s] @ Bm[s].T)
        rho2 = torch.einsum("htp,hpn,tn->ht", dy[:, s] * torch.exp(k)[..., None], bf(states[c]), Cm[s])
        inter = torch.exp(k[:, -1:] - k) * torch.einsum("hsp,hpn,sn->hs", x[:, s], bf(g), Bm[s])
        gh = torch.exp(k[:, -1]) * (g * bf(states[c])).sum((1, 2))
        right = (z * dt[:, None, s]).sum(2) - z.sum(1) * dt[:, s] + rho2
        psi2 = dt[:, s] * inter
        da = right.flip(-1).cumsum(-1).flip(-1) + psi2.cumsum(-1) - psi2 + gh[:, None]
        ddt[:, s] = z.sum(1) + inter + A[:, None] * da
        dyd, xd = bf(dy[:, s] * torch.exp(k)[..., None]), bf(x[:, s] * (torch.exp(k[:, -1:] - k) * dt[:, s])[..., None])
        wsum = (wd * dt[:, None, s]).sum(0)
        dC[s] = wsum @ Bm[s] + torch.einsum("htp,hpn->tn", dyd, bf(states[c]))
        dB[s] = wsum.T @ Cm[s] + torch.einsum("hsp,hpn->sn", xd, bf(g))
        g = torch.exp(k[:, -1])[:, None, None] * g + torch.einsum("htp,tn->hpn", dyd, Cm[s])
    return dict(ddt=ddt.T[None], dB=bf(dB)[None, :, None], dC=bf(dC)[None, :, None])


@pytest.mark.parametrize("extra", [{}, dict(a_max=64.0, dt_lo=1e-4, dt_hi=1.0)], ids=["mild", "stiff"])
def test_gradients_of_the_tensor_core_path_have_only_the_states_roundings(extra):
    """Masked tiles rounded to bf16 stay out of ddt, dB and dC: their errors, of ddt head by head, are those of the algebra above (a
    rounding differs from the kernels' where an fp32 sum falls on the other side: 10 % for that and for fp32 itself)."""
    cfg = config(2048, 16, 128, 1, 256, 512, **extra)
    errs = {k: [0.0, 0.0] for k in ("ddt", "dB", "dC")}
    for seed in (1, 2):
        inp = make_inputs(cfg, "cuda", seed=seed)
        ref, got, algebra = pu.run_oracle(to_f64_numpy(inp), cfg.seg), pu.run_gpu(cfg, inp), rounded_algebra(inp)
        for k, e in errs.items():
            r = torch.from_numpy(ref[k]).cuda()
            for j, v in enumerate((got[k].double(), algebra[k])):
                e[j] += ((v - r).norm(dim=1) / r.norm(dim=1)).pow(2).mean().item()
    assert all(gpu <= 1.1 ** 2 * alg for gpu, alg in errs.values()), errs
    print(errs)


@pytest.mark.parametrize("flags", [0, libssd.SSD_FLAG_FORCE_SIMT])
def test_ddt_where_the_step_size_is_zero(flags):
    """A step of size zero leaves the state alone, and its ddt is the direct term, which no product with dt shows."""
    cfg = config(1024, 4, 128, 1, 256, 512)
    inp = make_inputs(cfg, "cuda")
    inp["dt"][:, 5::7] = 0.0
    inp["dt"][:, 6::7] = 1e-25
    ref = pu.run_oracle(to_f64_numpy(inp), cfg.seg)
    got = pu.run_gpu(cfg, inp, flags=flags)
    for k in ("y", "ddt", "dA", "dx"):
        assert pu.relerr(got[k], ref[k]) <= pu.TOL["bf16"], k
    for first in (5, 6):
        assert pu.relerr(got["ddt"][:, first::7], ref["ddt"][:, first::7]) <= pu.TOL["bf16"], first
