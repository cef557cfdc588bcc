"""1 - a, which the gate kernel leaves out where only the general scans read it: pairs with strong and moderate chunks side by
side, every way a call comes to its first scan, every kind of gate."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_07146_b200 as gsa
import test_gpu_fused as fused
from test_gpu_parity import check_bwd, check_fwd, run_bwd, run_fwd
from util import TOL, rand_inputs, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu


def inputs(T, H, seed, final=True):
    d = rand_inputs(seed, 1, T, H, 128, 64, 64, "bf16", init=True, final_grads=final)
    a = d["gate"]
    a[:, 130:200, 0, 7] = 0.3                    # a strong chunk (the second), a run that two chunks share ...
    a[:, 380:400, 0, 9] = 1e-6                   # ... and one of 20 tokens across a boundary
    if T > 500:
        a[:, 460:500, H - 1, :] = 0.05
    return d


@pytest.mark.parametrize("T,H", [(139, 1), (384, 2), (523, 3), (2700, 1)])       # (2700: several segments)
@pytest.mark.parametrize("log,saved", [(False, False), (False, True), (True, False)])
def test_strong_and_moderate_chunks_in_a_pair(T, H, log, saved):
    d = inputs(T, H, T)
    got, g = run_fwd(d, 1, T, H, 128, 64, 64, "bf16", impl="tc", log=log)
    check_fwd(d, got, g, "bf16", log=log, tc=True, storage=False)
    gb, rb = run_bwd(d, 1, T, H, 128, 64, 64, "bf16", impl="tc", log=log, saved=saved)
    if not log:
        # d(log a) / a amplifies its fp32 noise where a is small (1e-6 here): that gate's gradient is held by the log form
        small = d["gate"] < 0.01
        gb["dgate"], rb["dgate"] = np.where(small, 0, gb["dgate"]), np.where(small, 0, rb["dgate"])
    check_bwd(gb, rb, TOL["bf16"], tc=True, storage=False)


@pytest.mark.parametrize("T", [384, 2700])
def test_the_forwards_block_serves_the_backward(T):
    d = inputs(T, 2, 5, final=False)
    p = gsa.Params(1, T, 2, 128, 64, 64, io="bf16")
    q, k, v, dO = (to_dev(d[n], "bf16") for n in ("q", "k", "v", "dO"))
    gate, K0, V0 = (to_dev(d[n]) for n in ("gate", "K0", "V0"))
    ok, block = torch.empty(1, T, 2, 64, device="cuda"), gsa.gate_block(p, "cuda")
    block.fill_(0x7f)                            # (what is left out is nowhere taken for something)
    gsa.gsa_fwd(p, q, k, v, gate, K0, V0, ok_save=ok, gate_save=block)
    x = gsa.gsa_bwd(p, q, k, v, gate, dO, K0, V0, ok_saved=ok, gate_saved=block)
    y = gsa.gsa_bwd(p, q, k, v, gate, dO, K0, V0, ok_saved=ok)
    torch.cuda.synchronize()
    for a, b in zip(x, y):
        assert rel_err(to_np(a), to_np(b)) <= 1e-6


@pytest.mark.parametrize("T,H", [(139, 1), (523, 3), (2700, 1)])
@pytest.mark.parametrize("bf16_gate", [False, True])
def test_logits(T, H, bf16_gate):
    # (forwards alone: where a backward follows, the gate kernel writes all of 1 - a for this kind)
    d = inputs(T, H, T + 1)
    a = d["gate"].astype(np.float64)
    x = (np.log(a) - np.log1p(-a)).astype(np.float32)            # a = sigmoid(x)
    xd = to_dev(x).to(torch.bfloat16) if bf16_gate else to_dev(x)
    a = 1.0 / (1.0 + np.exp(-to_np(xd)))
    ref = oracle.fwd(d["q"], d["k"], d["v"], a, K0=d["K0"], V0=d["V0"])
    p = gsa.Params(1, T, H, 128, 64, 64, io="bf16", impl="tc", gate_is_logits=True, tau=1.0, gate_bf16=bf16_gate)
    q, k, v = (to_dev(d[n], "bf16") for n in ("q", "k", "v"))
    KT, VT, ok = torch.empty(1, H, 64, 128, device="cuda"), torch.empty(1, H, 64, 64, device="cuda"), torch.empty(1, T, H, 64, device="cuda")
    ws = torch.full((gsa.gsa_workspace_bytes(p, 0),), 0x7f, dtype=torch.uint8, device="cuda")       # (3.4e38)
    o = gsa.gsa_fwd(p, q, k, v, xd, to_dev(d["K0"]), to_dev(d["V0"]), ok_save=ok, KT=KT, VT=VT, ws=ws)
    for n, t in (("o", o), ("ok", ok), ("KT", KT), ("VT", VT)):
        assert rel_err(to_np(t), ref[n], n == "o") <= TOL["bf16"], n


@pytest.mark.parametrize("T", [384, 523, 2048])
@pytest.mark.parametrize("saved", [False, True])
def test_the_fused_kernels_flagged_pairs(T, saved):
    B, H, w, m = 1, 3, 128, 64
    d = rand_inputs(T, B, T, H, w, w, m, "bf16", init=True)
    a = d["gate"]
    a[:, 130:200, 0, 7] = 0.3                    # the first and the last pair, each with chunks of both kinds
    a[:, 300:340, H - 1, :] = 0.05
    fused.check(fused.run(d, B, T, H, w, w, m, fuse=True, saved=saved), fused.reference(d))


@pytest.mark.parametrize("T,H", [(139, 1), (523, 3)])
@pytest.mark.parametrize("log", [False, True])
def test_shard_states(T, H, log):
    d = inputs(T, H, T + 2)
    p = gsa.Params(1, T, H, 128, 64, 64, io="bf16", impl="tc", gate_is_log=log)
    g = np.log(d["gate"].astype(np.float64)).astype(np.float32) if log else d["gate"]
    ws = torch.full((gsa.gsa_workspace_bytes(p, 4),), 0x7f, dtype=torch.uint8, device="cuda")
    KT, VT, decay = gsa.gsa_shard_states(p, to_dev(d["k"], "bf16"), to_dev(d["v"], "bf16"), to_dev(g), ws=ws)
    ref = oracle.fwd(d["q"], d["k"], d["v"], g, gate_is_log=log)
    assert rel_err(to_np(KT), ref["KT"]) <= TOL["bf16"] and rel_err(to_np(VT), ref["VT"]) <= TOL["bf16"]
    want = (g.astype(np.float64) if log else np.log(d["gate"].astype(np.float64))).sum(1)
    # log a to 2^-21 each (the hardware's logarithm), the sum of a chunk to 2^-24 of it
    assert np.abs(to_np(decay) - want).max() <= T * 2.0 ** -21 + 2.0 ** -23 * np.abs(want).max()
