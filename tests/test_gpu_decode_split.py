"""The decode step of few pairs, dealt out over clusters: every number of slots and rows a warp, heads whose value channels are
fewer than a warp's lanes in a CTA, unequal widths, both sides of the lines between the kernels; against the step in 64 bits.
"""
import numpy as np
import pytest
import torch


import paper_2409_07146_b200 as gsa
from util import TOL, rel_err, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io", ["bf16", "f32"])
@pytest.mark.parametrize("m", [32, 64, 128])
@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (512, 64), (64, 512), (256, 128), (512, 512)])
@pytest.mark.parametrize("B", [1, 10, 50])
def test_split_steps(io, m, dk, dv, B):
    H = 2
    dt = torch.bfloat16 if io == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(m + dk + B)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda") * scale
    q, k, v = normal(B, H, dk, scale=dk ** -0.5).to(dt), normal(B, H, dk).to(dt), normal(B, H, dv).to(dt)
    gate = torch.sigmoid(normal(B, H, m))
    K, V = normal(B, H, m, dk), normal(B, H, m, dv)
    refs = [to_np(t) for t in (q, k, v, gate, K, V)]
    p = gsa.Params(B, 1, H, dk, dv, m, io=io)
    o = gsa.gsa_decode_step(p, q, k, v, gate, K, V)
    torch.cuda.synchronize()
    for n, t in (("o", o), ("K", K), ("V", V)):
        assert torch.isfinite(t.float()).all(), n
    qn, kn, vn, a, Kr, Vr = (t.astype(np.float64) for t in refs)
    Kr = a[..., None] * Kr + (1 - a)[..., None] * kn[:, :, None]
    Vr = a[..., None] * Vr + (1 - a)[..., None] * vn[:, :, None]
    z = np.einsum("bhmd,bhd->bhm", Kr, qn)
    w = np.exp(z - z.max(-1, keepdims=True))
    w /= w.sum(-1, keepdims=True)
    ref = np.einsum("bhm,bhmd->bhd", w, Vr)
    assert rel_err(to_np(K), Kr) <= TOL["f32"] and rel_err(to_np(V), Vr) <= TOL["f32"]
    assert rel_err(to_np(o), ref, io == "bf16") <= TOL[io]
