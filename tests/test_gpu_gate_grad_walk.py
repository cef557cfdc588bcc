"""The gate gradient in one pass from the last tile to the first, which calls with enough (batch, head) pairs take: all, half or
a quarter of a pair's slots to a CTA (100, 50, 28 pairs); tiles of 64, 128 and 256 rows, whole and ragged; every kind of gate;
final memories; packed sequences whose offsets fall on groups of eight rows, inside them and on tiles."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_07146_b200 as gsa
from test_gpu_parity import check_bwd, run_bwd
from util import TOL, rand_inputs, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H", [(50, 2), (25, 2), (14, 2)])
@pytest.mark.parametrize("T,log", [(1, False), (64, True), (150, False), (257, True)])
def test_whole_and_ragged_tiles(B, H, T, log):
    d = rand_inputs(300 + B + T, B, T, H, 64, 64, 64, "bf16", init=True, final_grads=True)
    gb, rb = run_bwd(d, B, T, H, 64, 64, 64, "bf16", log=log)
    check_bwd(gb, rb, TOL["bf16"], tc=True)


@pytest.mark.parametrize("io,dk,dv", [("bf16", 512, 256), ("f32", 64, 128)])
def test_several_slices(io, dk, dv):
    B, H, T = 14, 2, 130
    d = rand_inputs(55, B, T, H, dk, dv, 64, io, final_grads=True)
    gb, rb = run_bwd(d, B, T, H, dk, dv, 64, io, log=True)
    check_bwd(gb, rb, TOL[io], tc=io == "bf16")


@pytest.mark.parametrize("B,H", [(100, 1), (25, 2), (7, 4)])
def test_packed_sequences_and_logits(B, H):
    T, m, d_ = 300, 64, 64
    cuts = [1, 8, 9, 63, 64, 128, 128, 200, 256, 299]
    cu = [0] + cuts + [T]
    d = rand_inputs(9 + B, B, T, H, d_, d_, m, "bf16")
    x = np.random.default_rng(B).standard_normal(d["gate"].shape).astype(np.float32)
    p = gsa.Params(B, T, H, d_, d_, m, io="bf16", gate_is_logits=True, tau=8.0,
                   cu_seqlens=torch.tensor(cu, dtype=torch.int32, device="cuda"))
    q, k, v, dO = (to_dev(d[n], "bf16") for n in ("q", "k", "v", "dO"))
    dgate = to_np(gsa.gsa_bwd(p, q, k, v, to_dev(x), dO)[3])
    ref = np.zeros(x.shape)
    a = (1 / (1 + np.exp(-x.astype(np.float64)))) ** 0.125
    for lo, hi in zip(cu, cu[1:]):
        if lo < hi:
            part = {n: d[n][:, lo:hi] for n in ("q", "k", "v", "dO")}
            g = oracle.bwd(part["q"], part["k"], part["v"], a[:, lo:hi], part["dO"])["dgate"]
            ref[:, lo:hi] = g * a[:, lo:hi] / (8 * (1 + np.exp(x[:, lo:hi].astype(np.float64))))
    assert rel_err(dgate, ref) <= TOL["bf16"]
