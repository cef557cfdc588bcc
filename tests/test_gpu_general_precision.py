"""How exact the scans of flagged (batch, head) pairs are beyond the tolerance of the other tests, root mean square against the fp64
oracle: the fp32 outputs (logits, gate gradient, final memories), slots that keep nearly all over thousands of tokens beside one
that forgets, and gradients near the ends of what fp32 holds."""
import numpy as np
import pytest
import torch

import paper_2409_07146_b200 as gsa
from test_gpu_parity import run_bwd, run_fwd
from util import rand_inputs, to_dev, to_np

import oracle

pytestmark = pytest.mark.gpu


def rms_err(x, ref):
    return float(np.sqrt(np.mean((x - ref) ** 2)) / np.sqrt(np.mean(ref ** 2)))


def sigmoid(x):
    return 1 / (1 + np.exp(-x))


# Bounds: a third above what the kernels gave that formed these chunks row by row in fp32 (logits 1.2e-6, gate gradient 8.2e-6 and
# 1.4e-5; the size of the latter is that of the running sum over the tokens, fp32 G of a few hundred gives 1.5e-5 a factor)
@pytest.mark.parametrize("mu,bound", [(0.0, 1.1e-5), (-2.0, 1.9e-5)])
def test_fp32_outputs_of_flagged_pairs(mu, bound):
    B, T, H, d, m = 1, 2048, 2, 128, 64
    x = rand_inputs(3, B, T, H, d, d, m, "bf16", init=True)
    x["gate"] = sigmoid(np.random.default_rng(4).standard_normal((B, T, H, m)) + mu).astype(np.float32)
    got, gate = run_fwd(x, B, T, H, d, d, m, "bf16", impl="tc", log=True)
    ref = oracle.fwd(x["q"], x["k"], x["v"], gate, gate_is_log=True, K0=x["K0"], V0=x["V0"])
    assert rms_err(got["ok"], ref["ok"]) <= 1.6e-6
    gb, rb = run_bwd(x, B, T, H, d, d, m, "bf16", impl="tc", log=True)
    assert rms_err(gb["dgate"], rb["dgate"]) <= bound


def test_slots_that_keep_over_many_tokens():
    # one segment (50 pairs), 1024 steps of 16 tokens: each rounds the decay and the state, 2^-24 at most each, as a random walk
    # sqrt(2 * 1024 / 3) 2^-24 = 1.6e-6 of what the memory held all along
    B, T, H, d, m = 1, 16384, 50, 64, 64
    x = rand_inputs(8, B, T, H, d, d, m, "bf16", init=True)
    r = np.random.default_rng(9)
    a = np.exp(-1e-5 * r.random((B, T, H, m)))
    a[..., 0] = sigmoid(r.standard_normal((B, T, H)) - 1)
    x["gate"] = a.astype(np.float32)
    few = 4                                                # of the pairs, which are alike, for the oracle
    got, gate = run_fwd(x, B, T, H, d, d, m, "bf16", impl="tc", log=True)
    ref = oracle.fwd(*(t[:, :, :few] for t in (x["q"], x["k"], x["v"], gate)), gate_is_log=True, K0=x["K0"][:, :few], V0=x["V0"][:, :few])
    errs = {n: rms_err(got[n][:, :few, 1:], ref[n][:, :, 1:]) for n in ("KT", "VT")}
    assert max(errs.values()) <= 1.6e-6, errs


# e^-20 to e^-50 a step of 16 tokens in some slot, no more
@pytest.mark.parametrize("size", [1e-20, 1e-17, 1.0, 1e17])
def test_gradients_of_any_size(size):
    B, T, H, d, m = 1, 400, 2, 128, 64
    x = rand_inputs(17, B, T, H, d, d, m, "bf16")
    x["dO"] = (x["dO"] * np.float32(2.0 ** np.round(np.log2(size)))).astype(np.float32)
    x["gate"] = np.exp(-np.minimum(np.random.default_rng(5).gamma(3.0, 1.1, (B, T, H, m)), 3.4)).astype(np.float32)
    got, ref = run_bwd(x, B, T, H, d, d, m, "bf16", impl="tc", log=True)
    for n in ("dq", "dk", "dv"):                           # (the rounding to bfloat16 is 1.66e-3)
        assert rms_err(got[n], ref[n]) <= 1.7e-3, n


# calls of packed sequences, whose scans have twice the state warps: half a slice, one slice and two; a segment with two offsets in a chunk
@pytest.mark.parametrize("dk,dv", [(64, 128), (128, 64), (256, 256)])
def test_packed_calls(dk, dv):
    B, T, H, m = 1, 1400, 2, 64
    cu = [0, 300, 310, 1025, T]
    x = rand_inputs(21 + dk, B, T, H, dk, dv, m, "bf16")
    x["gate"] = np.log(sigmoid(np.random.default_rng(dk).standard_normal((B, T, H, m)))).astype(np.float32)
    p = gsa.Params(B, T, H, dk, dv, m, io="bf16", gate_is_log=True, cu_seqlens=torch.tensor(cu, dtype=torch.int32, device="cuda"))
    q, k, v, dO = (to_dev(x[n], "bf16") for n in ("q", "k", "v", "dO"))
    gate = to_dev(x["gate"])
    logits, KT, VT = torch.empty(B, T, H, m, device="cuda"), torch.empty(B, H, m, dk, device="cuda"), torch.empty(B, H, m, dv, device="cuda")
    o = gsa.gsa_fwd(p, q, k, v, gate, ok_save=logits, KT=KT, VT=VT)
    dq, dk_, dv_, dgate = gsa.gsa_bwd(p, q, k, v, gate, dO, ok_saved=logits)
    args = (x["q"], x["k"], x["v"], x["gate"])
    ref = dict(oracle.fwd_packed(*args, cu, gate_is_log=True), **oracle.bwd_packed(*args, x["dO"], cu, gate_is_log=True))
    # (two offsets in a chunk of eleven: its G goes beyond -200, and an fp32 rounding of that is 200 * 2^-25 = 6e-6 to 1.2e-5 of a decay;
    # a root of eleven less of the whole, beside the 1.2e-6 of the other chunks; the gate gradient of the scans
    # in fp32 was 6.0e-6)
    for n, t, bound in (("ok", logits, 3e-6), ("KT", KT, 4e-6), ("VT", VT, 4e-6), ("dgate", dgate, 8e-6),     # (memories: pairs in the state runs' products)
                        ("o", o, 1.7e-3), ("dq", dq, 1.7e-3), ("dk", dk_, 1.7e-3), ("dv", dv_, 1.7e-3)):
        assert rms_err(to_np(t), ref[n]) <= bound, (n, rms_err(to_np(t), ref[n]))
