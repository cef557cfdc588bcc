"""The element-wise pre- and post-operations of the layer (Sec. 3.3) on the GPU against the numpy
oracle: the Swish feature map on q, k, v inside gsa_fwd / gsa_bwd / gsa_decode_step, and the
output path Swish -> RMSNorm over the heads of a token, forward and backward."""
import numpy as np
import pytest
import torch

import gsa_workloads as W
import oracle
from oracle import layer
import paper_2409_07146_b200 as gsa
from util import BF16_IO, TOL, bf16_half_ulp, rand_inputs, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu


def activated(x, io):
    a = layer.swish(x).astype(np.float32)
    return W.round_to_bf16(a) if io == "bf16" else a


@pytest.mark.parametrize("io,impl,d,m", [("f32", "auto", 64, 32), ("bf16", "tc", 128, 64), ("bf16", "tc", 512, 64)])
def test_feature_map_fwd_bwd(io, impl, d, m):
    B, T, H = 2, 260, 2
    x = rand_inputs(17 + d, B, T, H, d, d, m, io, init=True)
    for n in ("q", "k", "v"):                      # pre-activations of a wider range than N(0,1) q
        x[n] = (x[n] * (4.0 if n == "q" else 1.5)).astype(np.float32)
        if io == "bf16":
            x[n] = W.round_to_bf16(x[n])
    p = gsa.Params(B, T, H, d, d, m, io=io, impl=impl, feature_map="swish", scale=d ** -0.5)
    q, k, v, dO = (to_dev(x[n], io) for n in ("q", "k", "v", "dO"))
    gate, K0, V0 = to_dev(x["gate"]), to_dev(x["K0"]), to_dev(x["V0"])
    ok = torch.empty(B, T, H, m, device="cuda")
    o = gsa.gsa_fwd(p, q, k, v, gate, K0, V0, ok_save=ok)
    dq, dk, dv, dg = gsa.gsa_bwd(p, q, k, v, gate, dO, K0, V0, ok_saved=ok)
    torch.cuda.synchronize()
    qa, ka, va = (activated(x[n], io) for n in ("q", "k", "v"))
    rf = oracle.fwd(qa, ka, va, x["gate"], K0=x["K0"], V0=x["V0"], scale=d ** -0.5)
    rb = oracle.bwd(qa, ka, va, x["gate"], x["dO"], K0=x["K0"], V0=x["V0"], scale=d ** -0.5)
    ref = dict(o=rf["o"], ok=rf["ok"], dgate=rb["dgate"])
    for n in ("q", "k", "v"):
        ref["d" + n] = rb["d" + n] * layer.swish_grad(x[n])
    got = dict(o=to_np(o), ok=to_np(ok), dq=to_np(dq), dk=to_np(dk), dv=to_np(dv), dgate=to_np(dg))
    errs = {n: rel_err(got[n], ref[n], io == "bf16" and n in BF16_IO) for n in got}
    if io == "bf16":
        # dq, dk, dv are rounded to bfloat16 twice here: by the scan that writes the gradient w.r.t. the
        # activated tensor, and again after the multiplication by Swish' (in place, bfloat16 storage): two
        # half-ulps of the output format are taken off instead of one
        for n in ("dq", "dk", "dv"):
            diff = np.maximum(np.abs(got[n] - ref[n]) - 2.0 * bf16_half_ulp(ref[n]), 0.0)
            errs[n] = float(diff.max() / np.sqrt(np.mean(ref[n] ** 2)))
    print("feature map", io, d, {n: float("%.2g" % e) for n, e in errs.items()})
    assert all(e <= TOL[io] for e in errs.values()), errs


def test_feature_map_in_the_decode_step():
    S, H, d, m = 3, 4, 128, 64
    w = W.CONFIGS["decode"].scaled(B=S, H=H, d_k=d, d_v=d, m=m)
    st = W.make_decode_states(w)
    Ks, Vs = to_dev(st["K"]), to_dev(st["V"])
    Kr, Vr = st["K"].astype(np.float64), st["V"].astype(np.float64)
    p = gsa.Params(S, 1, H, d, d, m, io="bf16", feature_map="swish")
    for step in range(3):
        x = W.make_decode_step_inputs(w, step)
        o = gsa.gsa_decode_step(p, to_dev(x["q"], "bf16"), to_dev(x["k"], "bf16"), to_dev(x["v"], "bf16"),
                                to_dev(x["gate"]), Ks, Vs)
        ro = oracle.decode_step(layer.swish(x["q"]), layer.swish(x["k"]), layer.swish(x["v"]), x["gate"], Kr, Vr)
    assert rel_err(to_np(o), ro, True) <= TOL["bf16"] and rel_err(to_np(Ks), Kr) <= 1e-5 and rel_err(to_np(Vs), Vr) <= 1e-5


@pytest.mark.parametrize("io,H,dv,T", [("f32", 2, 64, 37), ("bf16", 4, 512, 100), ("bf16", 5, 512, 33), ("bf16", 32, 128, 20)])
@pytest.mark.parametrize("with_weight", [False, True])
def test_output_norm_fwd_bwd(io, H, dv, T, with_weight):
    B = 2
    r = np.random.default_rng(H + dv)
    o = (1.5 * r.standard_normal((B, T, H, dv))).astype(np.float32)
    dy = r.standard_normal((B, T, H, dv)).astype(np.float32)
    if io == "bf16":
        o, dy = W.round_to_bf16(o), W.round_to_bf16(dy)
    wgt = (1.0 + 0.3 * r.standard_normal(H * dv)).astype(np.float32) if with_weight else None
    eps = 1e-5
    p = gsa.Params(B, T, H, 128, dv, 64, io=io)
    od, dyd = to_dev(o, io), to_dev(dy, io)
    wd = to_dev(wgt) if with_weight else None
    y = gsa.gsa_out_norm_fwd(p, od, wd, eps)
    d_o, dw = gsa.gsa_out_norm_bwd(p, od, dyd, wd, eps)
    torch.cuda.synchronize()
    ry = layer.out_norm_fwd(o, wgt, eps)
    rdo, rdw = layer.out_norm_bwd(o, dy, wgt, eps)
    tol = TOL[io]
    assert rel_err(to_np(y), ry, io == "bf16") <= tol
    assert rel_err(to_np(d_o), rdo, io == "bf16") <= tol
    assert rel_err(to_np(dw), rdw) <= (1e-4 if io == "f32" else 2e-3)      # fp32 sums of bf16-exact inputs
    # deterministic
    d2, dw2 = gsa.gsa_out_norm_bwd(p, od, dyd, wd, eps)
    torch.cuda.synchronize()
    assert torch.equal(d_o, d2) and torch.equal(dw, dw2)


@pytest.mark.parametrize("io,H,dv,T", [("bf16", 1, 64, 1), ("f32", 3, 64, 7), ("bf16", 8, 512, 9), ("f32", 4, 512, 5), ("bf16", 7, 64, 17)])
def test_output_norm_edges(io, H, dv, T):
    # tokens that do not fill the four of a forward CTA or the pair of a backward one, rows from 8 vectors to the widest, a CTA of a partial last warp
    test_output_norm_fwd_bwd(io, H, dv, T, True)


@pytest.mark.parametrize("io,T,dk,dv", [("bf16", 1, 64, 512), ("f32", 33, 128, 64), ("bf16", 67, 256, 64)])
def test_feature_map_of_unequal_widths(io, T, dk, dv):
    # q, k and v share a launch: a short tensor beside a long one, sizes that do not fill the last block
    B, H, m = 1, 1, 64
    d = rand_inputs(5 + T, B, T, H, dk, dv, m, io)
    q, k, v, dO = (to_dev(d[n], io) for n in ("q", "k", "v", "dO"))
    p = gsa.Params(B, T, H, dk, dv, m, io=io, feature_map="swish")
    pn = gsa.Params(B, T, H, dk, dv, m, io=io)
    g = to_dev(d["gate"])
    sq, sk, sv = (torch.nn.functional.silu(x.float()).to(x.dtype) for x in (q, k, v))
    # the same kernels on features made by torch.  fp32: the two Swish differ by 2^-22 of the value, the gradients w.r.t. q
    # and k are differences of terms that many times larger (dq ~ p (dp - <p, dp>)), at the worst of all elements by rms a
    # hundredfold: 2.4e-5.  bf16: features and gradients are rounded to 8 bits on either side.
    tol = 1e-4 if io == "f32" else 2e-2
    assert rel_err(to_np(gsa.gsa_fwd(p, q, k, v, g)), to_np(gsa.gsa_fwd(pn, sq, sk, sv, g)), io == "bf16") <= tol
    got = gsa.gsa_bwd(p, q, k, v, g, dO)
    want = gsa.gsa_bwd(pn, sq, sk, sv, g, dO)
    for x, a, b in zip((q, k, v), got[:3], want[:3]):
        s = torch.sigmoid(x.double())
        assert rel_err(to_np(a), to_np((b.double() * s * (1 + x.double() * (1 - s))).float()), io == "bf16") <= tol


@pytest.mark.parametrize("io", ["f32", "bf16"])
def test_output_norm_weight_gradient_of_tiny_activations(io):
    # the weight gradient leaves in fp32 whatever the io type, also where 1 + exp(-o) is above 2^126 and its approximate
    # reciprocal is 0: Swish(o) = -5e-37 here, 1 / sqrt(eps) times that comes out.  (1 / (1 + exp(-o)) is a denormal of 22
    # bits there, exp's argument has a rounding of 2^-18: 4e-6)
    o = torch.tensor([-87.5, -88.0, -88.5, -88.0] * 16, device="cuda").view(1, 1, 1, 64)
    dy = torch.linspace(1, 2, 64, device="cuda").view(1, 1, 1, 64)
    p = gsa.Params(1, 1, 1, 64, 64, 64, io=io)
    dw = gsa.gsa_out_norm_bwd(p, o.to(p.io_dtype), dy.to(p.io_dtype), None, 1e-6)[1]
    x, g = o.double().flatten(), dy.to(p.io_dtype).double().flatten()
    want = g * x * torch.sigmoid(x) * 1e3
    assert float(((dw.double() - want) / want).abs().max()) <= 2e-5


@pytest.mark.parametrize("io,H,dv,T", [("bf16", 8, 512, 1301), ("bf16", 1, 64, 5003), ("f32", 1, 64, 5003)])
def test_output_norm_bwd_of_more_tokens_than_ctas(io, H, dv, T):
    # at most 148 * (2 .. 8) CTAs: each takes several pairs of tokens here, the last pair has one
    r = np.random.default_rng(T)
    o, dy = r.standard_normal((1, T, H, dv)).astype(np.float32), r.standard_normal((1, T, H, dv)).astype(np.float32)
    if io == "bf16":
        o, dy = W.round_to_bf16(o), W.round_to_bf16(dy)
    wgt = (1.0 + 0.3 * r.standard_normal(H * dv)).astype(np.float32)
    p = gsa.Params(1, T, H, 64, dv, 64, io=io)
    d_o, dw = gsa.gsa_out_norm_bwd(p, to_dev(o, io), to_dev(dy, io), to_dev(wgt), 1e-5)
    again = gsa.gsa_out_norm_bwd(p, to_dev(o, io), to_dev(dy, io), to_dev(wgt), 1e-5)
    without = gsa.gsa_out_norm_bwd(p, to_dev(o, io), to_dev(dy, io), to_dev(wgt), 1e-5, want_dweight=False)[0]
    rdo, rdw = layer.out_norm_bwd(o, dy, wgt, 1e-5)
    assert rel_err(to_np(d_o), rdo, io == "bf16") <= TOL[io]
    # terms of N(0, 1) size with 2^-21 from the exponential and the divisions, the worst of 4096 sums of them
    assert rel_err(to_np(dw), rdw) <= 5e-6
    assert torch.equal(d_o, again[0]) and torch.equal(dw, again[1]) and torch.equal(d_o, without)


@pytest.mark.parametrize("io,H,dv,T", [("bf16", 8, 512, 37889), ("f32", 4, 512, 37889)])
def test_output_norm_weight_gradient_does_not_drift(io, H, dv, T):
    # All tokens alike, so that every addition to a CTA's sum (128 tokens of it) rounds the same way.  Against T times the
    # gradient of one token: a run of 16 equal fp32 terms, (2 + .. + 16) / 16 half-ulps at the most; three roundings of sums.
    # (128 in one run: 1.9e-6.)
    g = torch.Generator(device="cuda").manual_seed(3)
    row = torch.randn(2, 1, 1, H, dv, generator=g, device="cuda").to(torch.bfloat16 if io == "bf16" else torch.float32)
    one = gsa.Params(1, 1, H, 64, dv, 64, io=io)
    d_one, dw_one = gsa.gsa_out_norm_bwd(one, row[0], row[1])
    p = gsa.Params(1, T, H, 64, dv, 64, io=io)
    o, dy = (x.expand(1, T, H, dv).contiguous() for x in row)
    d_o, dw = gsa.gsa_out_norm_bwd(p, o, dy)
    want = dw_one.double() * T
    assert float(((dw.double() - want) / want).abs().max()) <= (135 / 16 + 3) * 2.0 ** -24
    assert bool((d_o == d_one).all())


def test_exponential_of_the_sigmoid():
    # Swish over the range of fp32's exponential, by itself: with a large eps the output path divides by sqrt(eps).
    # exp(-x): 2^-21 + |x| 2^-23; the addition, two divisions or products, the square root's reciprocal (2 ulp): 8 half-ulps.
    o = torch.linspace(-70, 80, 32 * 1024 * 64, device="cuda").view(1, 1024, 32, 64)
    p = gsa.Params(1, 1024, 32, 64, 64, 64, io="f32")
    y = gsa.gsa_out_norm_fwd(p, o, None, 1e12)
    x = o.double()
    want = x * torch.sigmoid(x) * 1e-6
    bound = 2.0 ** -21 + x.abs() * 2.0 ** -23 + 8 * 2.0 ** -24
    # (mean(Swish^2) <= 6400 beside 1e12: another 3.2e-9)
    assert bool(((y.double() - want).abs() <= (bound + 3.2e-9) * want.abs()).all())
    far = torch.full((1, 1, 1, 64), -200.0, device="cuda")
    assert bool((gsa.gsa_out_norm_fwd(gsa.Params(1, 1, 1, 64, 64, 64, io="f32"), far, None, 1.0) == 0).all())       # (-3e-85)
