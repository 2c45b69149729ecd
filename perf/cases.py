"""What is timed of this library: whole passes through the public entry points of
`paper_2411_19460_b200.libssd` and `paper_2411_19460_b200.stack`, as a user's program calls them.

A case is a dict of plain values; its "kind" says which calls a pass makes:
  layer    ssd_fwd_segmented + ssd_bwd_segmented of one layer: a training step under sequence checkpoints
  prefill  ssd_fwd with nothing but inputs in hand (the wrapper allocates outputs and scratch)
  decode   one ssd_decode_step on a carried state
  stack    LayerStack.forward + LayerStack.backward: both checkpoint axes
  conv     ssd_conv_fwd over all segments, then ssd_conv_bwd right to left
  norm     ssd_gated_norm_fwd and ssd_gated_norm_bwd, a segment of rows at a time
Head counts are those of the Mamba-2 sizes this repository's workloads and tests use (24, 32, 64 and 80 heads of
64 channels) and the 4 and 8 heads of its small ones; lengths run from one chunk to a quarter of a million tokens.
"""
import math

import torch

from paper_2411_19460_b200 import libssd
from paper_2411_19460_b200.inputs import SSDConfig, make_inputs, make_stack_params
from paper_2411_19460_b200.stack import LayerStack

P = 64


def _layer(name, dtype, B, L, H, N, G, chunk, seg, stiff=False, dh=False):
    return dict(name=name, kind="layer", dtype=dtype, B=B, L=L, H=H, N=N, G=G, chunk=chunk, seg=seg, stiff=stiff, dh=dh)


def listed():
    return [
        # one token of one sequence through the largest layer: latency of a generation loop
        dict(name="decode_one", kind="decode", dtype="bf16", B=1, H=80, N=128, G=1),
        # one token for each of many sequences: a serving batch, the state read and written once
        dict(name="decode_batch", kind="decode", dtype="bf16", B=48, H=64, N=128, G=1),
        # a prompt batch whose length is an odd number of chunks and whose last scratch segment is short
        dict(name="prefill_ragged", kind="prefill", dtype="bf16", B=3, L=9472, H=64, N=128, G=1, chunk=256, seg=4096),
        # the fp32 reference workload: a few microseconds of work, many launches
        _layer("layer_fp32_small", "fp32", 1, 1024, 4, 64, 1, 64, 256),
        # an fp32 training step of the smallest model's layer: gradients to 1e-4 and better
        _layer("layer_fp32_130m", "fp32", 2, 4096, 24, 128, 1, 256, 1024),
        # the smallest model's layer in bf16, short segments
        _layer("layer_bf16_130m", "bf16", 1, 16384, 24, 128, 1, 256, 2048),
        # half the state size and half the chunk, a batch of sequences
        _layer("layer_bf16_n64", "bf16", 2, 8192, 32, 64, 1, 128, 2048),
        # the largest model's layer over a long video
        _layer("layer_bf16_2p7b", "bf16", 1, 131072, 80, 128, 1, 256, 4096),
        # grouped B and C, stiff decays, a quarter of a million tokens: the largest
        _layer("layer_bf16_stiff_g8", "bf16", 1, 262144, 80, 128, 8, 256, 8192, stiff=True),
        # stacked layers with only every second layer's input kept
        dict(name="stack_l2", kind="stack", dtype="bf16", B=1, L=16384, H=80, N=128, G=1, chunk=256, seg=4096, layers=6,
             interval=2),
        # the convolution in front of the layer, 5376 channels, segment by segment
        dict(name="conv_segments", kind="conv", dtype="bf16", B=1, L=32768, C=5376, seg=4096),
        # the gated normalisation behind it, 5120 channels
        dict(name="norm_segments", kind="norm", dtype="bf16", B=1, L=32768, D=5120, group=5120, seg=4096),
    ]


def _spread(rng, lo, hi):
    """An integer between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _groups(rng, H):
    return rng.choice([g for g in (1, 1, 2, 4, 8) if H % g == 0])


def draw(rng):
    kind = rng.choice(["decode", "prefill", "layer_fp32", "layer_bf16", "layer_bf16", "layer_bf16", "layer_bf16_option", "stack",
                       "conv", "norm"])
    H = rng.choice([24, 32, 64, 80])
    if kind == "decode":
        return dict(kind="decode", dtype=rng.choice(["bf16", "bf16", "fp32"]), B=_spread(rng, 1, 64), H=H, N=rng.choice([64, 128, 128]),
                    G=_groups(rng, H))
    if kind == "prefill":
        nc, B = _spread(rng, 1, 128), _spread(rng, 1, 4)
        return dict(kind="prefill", dtype="bf16", B=B, L=256 * nc, H=H, N=128, G=_groups(rng, H), chunk=256,
                    seg=256 * min(nc, _spread(rng, 8, 64)))
    if kind == "layer_fp32":
        H, chunk = rng.choice([4, 8, 24]), rng.choice([64, 128, 256])
        L = chunk * _spread(rng, max(1, 512 // chunk), 8192 // chunk)
        return _drawn_layer(rng, "fp32", _spread(rng, 1, 2), L, H, rng.choice([64, 128]), chunk)
    if kind == "layer_bf16":       # the chunk and state size of every model of the repository's workloads
        L = 256 * _spread(rng, 4, 512)
        B = _spread(rng, 1, 4) if L <= 16384 else 1
        return _drawn_layer(rng, "bf16", B, L, H, 128, 256)
    if kind == "layer_bf16_option":
        chunk = rng.choice([64, 128, 256])
        L = chunk * _spread(rng, 1024 // chunk, 16384 // chunk)
        return _drawn_layer(rng, "bf16", 1, L, rng.choice([4, 8, 24, 32]), 64 if chunk == 256 else rng.choice([64, 128]), chunk)
    if kind == "stack":
        seg, layers = 256 * _spread(rng, 4, 16), rng.randint(2, 6)
        return dict(kind="stack", dtype="bf16", B=1, L=seg * rng.randint(2, 4), H=H, N=128, G=_groups(rng, H), chunk=256, seg=seg,
                    layers=layers, interval=rng.randint(1, 2))
    L = 64 * _spread(rng, 16, 512) + rng.choice([0, 0, 1, 37])
    seg = min(L, 256 * _spread(rng, 4, 32))
    if L % seg in (1, 2):          # the convolution's state is three tokens: no shorter last segment
        L += 3
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    if kind == "conv":
        return dict(kind="conv", dtype=dtype, B=1, L=L, C=H * P + 2 * _groups(rng, H) * 128, seg=seg)
    D = H * P
    return dict(kind="norm", dtype=dtype, B=1, L=L, D=D, group=D // _groups(rng, H), seg=seg)


def _drawn_layer(rng, dtype, B, L, H, N, chunk):
    nc = L // chunk
    c = _layer("", dtype, B, L, H, N, _groups(rng, H), chunk, chunk * min(nc, _spread(rng, min(nc, max(4, 1024 // chunk)), 32)),
               stiff=rng.random() < 0.3, dh=rng.random() < 0.3)
    del c["name"]
    return c


def _config(c):
    stiff = dict(a_max=64.0, dt_lo=1e-4, dt_hi=1.0) if c.get("stiff") else {}
    return SSDConfig("case", c["dtype"], c["B"], c.get("L", 1), c["H"], P, c["N"], c["G"], c.get("chunk", 256), c.get("seg", 0),
                     h0_std=0.1, dh_std=0.1 if c.get("dh") else 0.0, layers=c.get("layers", 1), **stiff)


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def prepare(case, seed):
    c, dev = case, torch.device("cuda")
    s = dict(case=c)
    if c["kind"] in ("layer", "prefill", "decode", "stack"):
        cfg = _config(c)
        s.update(make_inputs(cfg, dev, seed=seed))
    if c["kind"] == "layer":
        # a training program keeps its outputs, checkpoints and scratch from step to step
        shape = libssd.make_shape(s["x"], s["Bm"], c["chunk"], c["seg"])
        B, H, N = c["B"], c["H"], c["N"]
        nseg = -(-c["L"] // c["seg"])
        f32 = dict(dtype=torch.float32, device=dev)
        s.update(y=torch.empty_like(s["x"]), h_final=torch.empty(B, H, P, N, **f32), boundary=torch.empty(B, nseg, H, P, N, **f32),
                 ws_f=libssd.alloc_workspace(shape, libssd.SSD_OP_FWD_SEG, dev),
                 ws_b=libssd.alloc_workspace(shape, libssd.SSD_OP_BWD_SEG, dev),
                 out=dict(dx=torch.empty_like(s["x"]), ddt=torch.empty_like(s["dt"]), dA=torch.empty(H, **f32),
                          dB=torch.empty_like(s["Bm"]), dC=torch.empty_like(s["Cm"]), dD=torch.empty(H, **f32),
                          dh0=torch.empty(B, H, P, N, **f32)))
    elif c["kind"] == "stack":
        sp = make_stack_params(cfg, dev)
        st = LayerStack(s["x"], s["dt"], s["Bm"], s["Cm"], sp["A"], sp["D"], sp["W"], chunk=c["chunk"], seg=c["seg"],
                        layer_interval=c["interval"])
        for j in range(c["layers"]):
            st.set_h0(j, sp["h0"][j])
        s.update(stack=st, out=dict(dx0=torch.empty_like(s["x"]), dA=torch.zeros(c["layers"], c["H"], device=dev),
                                    dD=torch.zeros(c["layers"], c["H"], device=dev)))
    elif c["kind"] in ("conv", "norm"):
        g = torch.Generator(device=dev).manual_seed(seed)
        randn = lambda *shape: torch.randn(*shape, generator=g, device=dev, dtype=torch.float32)
        B, L, td = c["B"], c["L"], _dtype(c)
        cuts = [(a, min(a + c["seg"], L)) for a in range(0, L, c["seg"])]
        s["cuts"] = cuts
        if c["kind"] == "conv":
            C = c["C"]
            u = randn(B, L, C).to(td)
            s.update(u=u, dout=randn(B, L, C).to(td), w=randn(C, 4) * 0.5, bias=randn(C) * 0.1, y=torch.empty_like(u),
                     du=torch.empty_like(u), states=torch.zeros(len(cuts) + 1, B, 3, C, dtype=td, device=dev),
                     dstates=torch.zeros(2, B, 3, C, device=dev), dw=torch.zeros(C, 4, device=dev), dbias=torch.zeros(C, device=dev),
                     ws=torch.empty(int(libssd.lib().ssd_conv_workspace_bytes(B, c["seg"], C)), dtype=torch.uint8, device=dev))
        else:
            D = c["D"]
            y = randn(B * L, D).to(td)
            s.update(y=y, z=randn(B * L, D).to(td), dout=randn(B * L, D).to(td), gamma=1.0 + 0.1 * randn(D), o=torch.empty_like(y),
                     dy=torch.empty_like(y), dz=torch.empty_like(y), dgamma=torch.zeros(D, device=dev),
                     ws=torch.empty(int(libssd.lib().ssd_gated_norm_workspace_bytes(c["seg"], D)), dtype=torch.uint8, device=dev))
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "layer":
        ins = (s["x"], s["dt"], s["A"], s["Bm"], s["Cm"], s["D"])
        y, hf, bd = libssd.ssd_fwd_segmented(*ins, s["h0"], chunk=c["chunk"], seg=c["seg"], y=s["y"], h_final=s["h_final"],
                                             boundary=s["boundary"], ws=s["ws_f"])
        grads = libssd.ssd_bwd_segmented(*ins, bd, s["dy"], s["dh_final"], chunk=c["chunk"], seg=c["seg"], out=s["out"], ws=s["ws_b"])
        return dict(y=y, h_final=hf, boundary=bd, **grads)
    if c["kind"] == "prefill":
        return libssd.ssd_fwd(s["x"], s["dt"], s["A"], s["Bm"], s["Cm"], s["D"], chunk=c["chunk"], seg=c["seg"])
    if c["kind"] == "decode":
        y = libssd.ssd_decode_step(s["x"], s["dt"], s["A"], s["Bm"], s["Cm"], s["D"], s["h0"])
        return y, s["h0"]
    if c["kind"] == "stack":
        s["out"]["dA"].zero_()
        s["out"]["dD"].zero_()
        top = s["stack"].forward()
        out = s["stack"].backward(s["dy"], out=s["out"])
        return dict(top=top, states=s["stack"].bnd[:, -1], dx0=out["dx0"], dA=out["dA"], dD=out["dD"], dh0=out["dh0"])
    cuts, last = s["cuts"], len(s["cuts"]) - 1
    if c["kind"] == "conv":
        st, ds = s["states"], s["dstates"]
        for k, (a, b) in enumerate(cuts):
            libssd.ssd_conv_fwd(s["u"][:, a:b], s["w"], s["bias"], st[k], out=s["y"][:, a:b], state_out=st[k + 1])
        for k in range(last, -1, -1):
            a, b = cuts[k]
            cur = (last - k) & 1
            libssd.ssd_conv_bwd(s["u"][:, a:b], s["w"], s["bias"], st[k], s["dout"][:, a:b], None if k == last else ds[cur],
                                du=s["du"][:, a:b], dstate=ds[1 - cur], dw=s["dw"], dbias=s["dbias"], accumulate=k != last, ws=s["ws"])
        return dict(y=s["y"], state=st[last + 1], du=s["du"], dw=s["dw"], dbias=s["dbias"], dstate=ds[(last + 1) & 1])
    for a, b in cuts:
        libssd.ssd_gated_norm_fwd(s["y"][a:b], s["z"][a:b], s["gamma"], group=c["group"], out=s["o"][a:b])
    for k in range(last, -1, -1):
        a, b = cuts[k]
        libssd.ssd_gated_norm_bwd(s["y"][a:b], s["z"][a:b], s["gamma"], s["dout"][a:b], group=c["group"], dy=s["dy"][a:b],
                                  dz=s["dz"][a:b], dgamma=s["dgamma"], accumulate=k != last, ws=s["ws"])
    return dict(o=s["o"], dy=s["dy"], dz=s["dz"], dgamma=s["dgamma"])


def work(case):
    """Bytes: each call's inputs once and its outputs once.  Flops: the products of the chunked scan, the causal half
    of the intra-chunk ones only."""
    c = case
    e = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] == "decode":
        state = c["B"] * c["H"] * P * c["N"]
        return dict(bytes=8 * state + c["B"] * (2 * e * c["H"] * P + 2 * e * c["G"] * c["N"] + 4 * c["H"]), flops=5 * state)
    if c["kind"] == "conv":
        n = c["B"] * c["L"] * c["C"]
        return dict(bytes=5 * e * n, flops=40 * n)
    if c["kind"] == "norm":
        n = c["B"] * c["L"] * c["D"]
        return dict(bytes=8 * e * n, flops=30 * n)
    tok, HP, GN, H, Q = c["B"] * c["L"], c["H"] * P, c["G"] * c["N"], c["H"], c["chunk"]
    HPN, half = HP * c["N"], (Q + 1) / 2
    states = 4 * HPN * c["B"]
    fwd = dict(bytes=tok * (e * (2 * HP + 2 * GN) + 4 * H) + 2 * states, flops=tok * (4 * HPN + 2 * half * (GN + HP)))
    if c["kind"] == "prefill":
        return fwd
    nseg = -(-c["L"] // c["seg"])
    bwd = dict(bytes=tok * (e * (3 * HP + 4 * GN) + 8 * H) + (2 * nseg + 2) * states, flops=tok * (10 * HPN + 2 * half * (3 * GN + 3 * HP)))
    n = 1
    if c["kind"] == "stack":       # the hand-over between layers: x, y in and x out; its transpose on the way back
        n = c["layers"]
        fwd = dict(bytes=fwd["bytes"] + tok * 3 * e * HP, flops=fwd["flops"] + tok * 2 * P * HP)
        bwd = dict(bytes=bwd["bytes"] + tok * 2 * e * HP, flops=bwd["flops"] + tok * 2 * P * HP)
    return {k: n * (fwd[k] + bwd[k]) for k in fwd}


def tolerance(case):
    # bf16: outputs rounded to 8 bits, bf16 products summed in fp32 in another order.  fp32: sums of thousands of
    # terms in another order; dA is a sum with cancellation over the whole sequence.
    return dict(rel=1e-2) if case["dtype"] == "bf16" else dict(rel=2e-5, max=1e-3)
