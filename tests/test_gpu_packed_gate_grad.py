"""Packed sequences, gate gradient: the 16-row blocks that hold the first token of a sequence.  Offsets on, before and behind
the edges of a block, several in one, empty sequences, offsets that repeat T."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_07146_b200 as gsa
from util import TOL, rand_inputs, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("T,cuts", [(97, [1, 15, 16, 17, 96]), (300, [31, 32, 33, 40, 47, 48, 256]), (160, [64, 64, 65, 160, 160]),
                                    (1041, [1, 500, 1024, 1040])])
def test_gate_gradient_at_the_edges_of_blocks(T, cuts, io):
    B, H, dk, dv, m = 1, 2, 64, 128, 64
    d = rand_inputs(77 + T, B, T, H, dk, dv, m, io)
    cu = [0] + cuts + [T]
    p = gsa.Params(B, T, H, dk, dv, m, io=io, cu_seqlens=torch.tensor(cu, dtype=torch.int32, device="cuda"))
    q, k, v, dO = (to_dev(d[n], io) for n in ("q", "k", "v", "dO"))
    dgate = gsa.gsa_bwd(p, q, k, v, to_dev(d["gate"]), dO)[3]
    torch.cuda.synchronize()
    ref = np.zeros_like(d["gate"], dtype=np.float64)
    for a, b in zip(cu, cu[1:]):
        if a < b:
            part = {n: d[n][:, a:b] for n in ("q", "k", "v", "gate", "dO")}
            ref[:, a:b] = oracle.bwd(part["q"], part["k"], part["v"], part["gate"], part["dO"])["dgate"]
    # on the fp32 kernels a start drops the running log gate by 100: n of them in a chunk of 64 tokens make |G| reach 100 n, whose
    # fp32 rounding, 100 n 2^-24, is a relative error of every decay factor, four of which multiply the terms of a gradient
    n = max(sum(c <= x < c + 64 for x in cuts) for c in range(0, T, 64))
    assert rel_err(to_np(dgate), ref) <= TOL[io] + (4 * 100 * n * 2.0 ** -24 if io == "f32" else 0.0)


def test_more_blocks_than_the_bits_of_the_scan():
    # 65537 blocks of 16 rows: the scan over the block totals searches the offsets instead.  Against each sequence by
    # itself, which needs neither.
    T = 65536 * 16 + 5
    cu = [0, 17, 600000, 600007, T - 30, T]
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v, dO = (torch.randn(1, T, 1, 64, generator=g, device="cuda") for _ in range(4))
    q *= 0.125
    gate = torch.sigmoid(torch.randn(1, T, 1, 32, generator=g, device="cuda")) ** 0.125
    p = gsa.Params(1, T, 1, 64, 64, 32, io="f32", cu_seqlens=torch.tensor(cu, dtype=torch.int32, device="cuda"))
    dgate = gsa.gsa_bwd(p, q, k, v, gate, dO)[3]
    want = torch.empty_like(dgate)
    for a, b in zip(cu, cu[1:]):
        part = [t[:, a:b].contiguous() for t in (q, k, v, gate, dO)]
        want[:, a:b] = gsa.gsa_bwd(gsa.Params(1, b - a, 1, 64, 64, 32, io="f32"), *part)[3]
    # (two starts in a chunk of 64 tokens: the bound of the test above)
    assert float((dgate - want).abs().max() / want.square().mean().sqrt()) <= TOL["f32"] + 4 * 200 * 2.0 ** -24
