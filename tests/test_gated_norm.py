"""Gated RMS normalisation behind the SSD layer: the oracle is pinned by a brute-force loop and by finite differences; the
CUDA kernels are compared with it (whole-row and grouped normalisation, both dtypes, several group widths)."""
import numpy as np
import pytest
import torch

from oracle import ssd_oracle as orc


def test_oracle_gated_norm_equals_brute_force_loop():
    rng = np.random.default_rng(0)
    y, z = rng.standard_normal((3, 12)), rng.standard_normal((3, 12))
    gamma = rng.standard_normal(12)
    for group in (12, 4):
        out, _, _ = orc.gated_norm_fwd(y, z, gamma, group, eps=1e-3)
        for r in range(3):
            for g0 in range(0, 12, group):
                v = [y[r, c] * z[r, c] / (1 + np.exp(-z[r, c])) for c in range(g0, g0 + group)]
                ms = sum(a * a for a in v) / group
                for j, c in enumerate(range(g0, g0 + group)):
                    assert abs(out[r, c] - v[j] / np.sqrt(ms + 1e-3) * gamma[c]) < 1e-12


def test_oracle_gated_norm_backward_matches_finite_differences():
    rng = np.random.default_rng(1)
    y, z = rng.standard_normal((2, 8)), rng.standard_normal((2, 8))
    gamma, g = rng.standard_normal(8), rng.standard_normal((2, 8))
    for group in (8, 4):
        dy, dz, dg = orc.gated_norm_bwd(y, z, gamma, g, group, eps=1e-3)
        loss = lambda a, b, c: float(np.sum(orc.gated_norm_fwd(a, b, c, group, eps=1e-3)[0] * g))
        eps = 1e-6
        for arr, grad, pos in ((y, dy, 0), (z, dz, 1), (gamma, dg, 2)):
            for idx in np.ndindex(arr.shape):
                hi, lo = arr.copy(), arr.copy()
                hi[idx] += eps
                lo[idx] -= eps
                args_hi = [y, z, gamma]
                args_lo = [y, z, gamma]
                args_hi[pos], args_lo[pos] = hi, lo
                fd = (loss(*args_hi) - loss(*args_lo)) / (2 * eps)
                assert abs(fd - grad[idx]) < 1e-6 * max(1.0, abs(fd)), (group, pos, idx)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,rows,D,group", [("fp32", 37, 512, 512), ("bf16", 37, 512, 128), ("bf16", 300, 5120, 5120),
                                                 ("bf16", 100, 5120, 640), ("fp32", 20, 8192, 8192)])
def test_gated_norm_matches_oracle(dtype, rows, D, group):
    from paper_2411_19460_b200 import libssd
    from tests.parity_util import TOL, relerr

    tol = TOL[dtype]
    td = torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator().manual_seed(5)
    y = torch.randn(rows, D, generator=gen).to(td).cuda()
    z = torch.randn(rows, D, generator=gen).to(td).cuda()
    g = torch.randn(rows, D, generator=gen).to(td).cuda()
    gamma = (1.0 + 0.1 * torch.randn(D, generator=gen)).cuda()
    f64 = lambda t: t.detach().double().cpu().numpy()
    out_ref, _, _ = orc.gated_norm_fwd(f64(y), f64(z), f64(gamma), group)
    dy_ref, dz_ref, dg_ref = orc.gated_norm_bwd(f64(y), f64(z), f64(gamma), f64(g), group)
    out = libssd.ssd_gated_norm_fwd(y, z, gamma, group=group)
    dy, dz, dg = libssd.ssd_gated_norm_bwd(y, z, gamma, g, group=group)
    # in two row ranges with accumulation: the same values
    dg2 = torch.zeros_like(dg)
    half = rows // 2
    libssd.ssd_gated_norm_bwd(y[:half], z[:half], gamma, g[:half], group=group, dgamma=dg2, accumulate=True)
    libssd.ssd_gated_norm_bwd(y[half:], z[half:], gamma, g[half:], group=group, dgamma=dg2, accumulate=True)
    torch.cuda.synchronize()
    errs = dict(out=relerr(out, out_ref), dy=relerr(dy, dy_ref), dz=relerr(dz, dz_ref), dgamma=relerr(dg, dg_ref),
                dgamma_split=relerr(dg2, dg_ref))
    assert all(v <= tol for v in errs.values()), errs


@pytest.mark.gpu
def test_gated_norm_rejects_bad_arguments():
    from paper_2411_19460_b200 import libssd

    y = torch.zeros(4, 24, device="cuda")
    gamma = torch.ones(24, device="cuda")
    with pytest.raises(libssd.SSDError):
        libssd.ssd_gated_norm_fwd(y, y, gamma, group=10)              # D % group
    with pytest.raises(libssd.SSDError):
        libssd.ssd_gated_norm_fwd(y, y, gamma, group=6)               # group % 4


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("rows,D,group", [(1, 5120, 5120), (5, 1536, 512), (1205, 2048, 2048), (2500, 64, 64), (37, 24, 12), (9, 8192, 8192)])
def test_gated_norm_row_splits_and_rings(rows, D, group, dtype):
    """One row, few rows per CTA, an uneven last CTA, more rows than the ring holds, rows that no ring takes."""
    from paper_2411_19460_b200 import libssd
    from tests.parity_util import TOL, relerr

    td = torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator().manual_seed(rows)
    y, z, g = (torch.randn(rows, D, generator=gen).to(td).cuda() for _ in range(3))
    gamma = (1.0 + 0.1 * torch.randn(D, generator=gen)).cuda()
    f64 = lambda t: t.detach().double().cpu().numpy()
    out_ref, _, _ = orc.gated_norm_fwd(f64(y), f64(z), f64(gamma), group)
    refs = orc.gated_norm_bwd(f64(y), f64(z), f64(gamma), f64(g), group)
    assert relerr(libssd.ssd_gated_norm_fwd(y, z, gamma, group=group), out_ref) <= TOL[dtype]
    for a, r in zip(libssd.ssd_gated_norm_bwd(y, z, gamma, g, group=group), refs):
        assert relerr(a, r) <= TOL[dtype]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("scale,eps", [(1e15, 1e-5), (1e-15, 0.0)])
@pytest.mark.parametrize("D,group", [(1024, 1024), (8192, 8192)])
def test_gated_norm_of_rows_far_from_one(D, group, scale, eps, dtype):
    """A normalisation does not depend on its input's scale: whatever fp32 holds the squares of has the same accuracy."""
    from paper_2411_19460_b200 import libssd
    from tests.parity_util import TOL, relerr

    td = torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator().manual_seed(3)
    y, z, g = (torch.randn(12, D, generator=gen).to(td).cuda() for _ in range(3))
    y = y * scale
    gamma = (1.0 + 0.1 * torch.randn(D, generator=gen)).cuda()
    f64 = lambda t: t.detach().double().cpu().numpy()
    out_ref, _, _ = orc.gated_norm_fwd(f64(y), f64(z), f64(gamma), group, eps=eps)
    refs = orc.gated_norm_bwd(f64(y), f64(z), f64(gamma), f64(g), group, eps=eps)
    assert relerr(libssd.ssd_gated_norm_fwd(y, z, gamma, group=group, eps=eps), out_ref) <= TOL[dtype]
    for a, r in zip(libssd.ssd_gated_norm_bwd(y, z, gamma, g, group=group, eps=eps), refs):
        assert relerr(a, r) <= TOL[dtype]


@pytest.mark.gpu
@pytest.mark.parametrize("rows,D,group", [(65536, 256, 256), (8192, 1024, 128), (4099, 2048, 2048)])
def test_gated_norm_dgamma_of_long_calls_is_summed_in_short_pieces(rows, D, group):
    """However many rows a CTA takes, fp32 sums of dgamma end after 16 of them.  Relative error of 16 terms of either sign in order:
    sqrt(16 / 2) 2^-25; of a term itself (reciprocal root, sigmoid, products): about 2^-23.  One sum over 222 rows: 3e-7."""
    from paper_2411_19460_b200 import libssd

    gen = torch.Generator(device="cuda").manual_seed(rows)
    y, z, g = (torch.randn(rows, D, generator=gen, device="cuda") for _ in range(3))
    gamma = 1.0 + 0.1 * torch.randn(D, generator=gen, device="cuda")
    v = (y.double() * z.double() * torch.sigmoid(z.double())).view(rows, -1, group)
    ref = ((v * torch.rsqrt((v * v).mean(-1, keepdim=True) + 1e-5)).view(rows, D) * g.double()).sum(0)
    _, _, dg = libssd.ssd_gated_norm_bwd(y, z, gamma, g, group=group)
    assert ((dg.double() - ref).norm() / ref.norm()).item() <= 2e-7
