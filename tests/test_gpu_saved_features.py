"""With a feature map the block that a forward leaves for its backward holds the activated q and k, and v of a sequence cut into
segments: the gradients are those of a backward that forms them again, to the bit, and a short block is refused."""
import pytest
import torch

import paper_2409_07146_b200 as gsa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,m,T", [("bf16", 64, 130), ("bf16", 32, 17), ("bf16", 128, 65), ("f32", 32, 200), ("bf16", 64, 1300)])
def test_block_with_a_feature_map(io, m, T):
    B, H, dk, dv = 2, 2, 128, 64
    p = gsa.Params(B, T, H, dk, dv, m, io=io, gate_is_log=True, feature_map="swish")
    g = torch.Generator(device="cuda").manual_seed(T + m)
    dt = torch.bfloat16 if io == "bf16" else torch.float32

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")
    q, k, v, dO = (normal(B, T, H, d).to(dt) for d in (dk, dk, dv, dv))
    gate = torch.nn.functional.logsigmoid(normal(B, T, H, m)) / 8
    logits = [torch.empty(B, T, H, m, device="cuda") for _ in range(2)]
    block = gsa.gate_block(p, "cuda")
    ws = torch.empty(gsa.gsa_workspace_bytes(p, 0), dtype=torch.uint8, device="cuda")
    o = [gsa.gsa_fwd(p, q, k, v, gate, ok_save=logits[0]), gsa.gsa_fwd(p, q, k, v, gate, ok_save=logits[1], ws=ws, gate_save=block)]
    ws.fill_(0x7f)                                  # (nothing of the forward's workspace is left)
    grads = [gsa.gsa_bwd(p, q, k, v, gate, dO, ok_saved=logits[0]),
             gsa.gsa_bwd(p, q, k, v, gate, dO, ok_saved=logits[1], gate_saved=block)]
    assert torch.equal(o[0], o[1]) and torch.equal(logits[0], logits[1])
    for a, b in zip(*[x.values() if isinstance(x, dict) else x for x in grads]):
        assert (a is None and b is None) or torch.equal(a, b)
    short = block[:-256].contiguous()
    with pytest.raises(RuntimeError):
        gsa.gsa_fwd(p, q, k, v, gate, ok_save=logits[1], gate_save=short)
    with pytest.raises(RuntimeError):
        gsa.gsa_bwd(p, q, k, v, gate, dO, ok_saved=logits[1], gate_saved=short)


# (one segment: what the block holds beside q and k depends on the gate alone, and the logits on q and k)
@pytest.mark.parametrize("io,m,T", [("bf16", 64, 130), ("bf16", 32, 17), ("bf16", 128, 65), ("f32", 32, 60)])
def test_a_block_serves_other_tensors_where_nothing_in_it_depends_on_them(io, m, T):
    B, H, dk, dv = 2, 2, 128, 64
    p = gsa.Params(B, T, H, dk, dv, m, io=io, gate_is_log=True, feature_map="swish")
    g = torch.Generator(device="cuda").manual_seed(T + m)
    dt = torch.bfloat16 if io == "bf16" else torch.float32

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")
    q, k, v, dO, q2, k2, v2 = (normal(B, T, H, d).to(dt) for d in (dk, dk, dv, dv, dk, dk, dv))
    gate = torch.nn.functional.logsigmoid(normal(B, T, H, m)) / 8
    logits = torch.empty(B, T, H, m, device="cuda")
    block = gsa.gate_block(p, "cuda")
    gsa.gsa_fwd(p, q, k, v, gate, ok_save=logits, gate_save=block)
    for args, ok in (((q, k, v2), logits), ((q2, k2, v2), None)):
        want = gsa.gsa_bwd(p, *args, gate, dO, ok_saved=ok)
        got = gsa.gsa_bwd(p, *args, gate, dO, ok_saved=ok, gate_saved=block)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
