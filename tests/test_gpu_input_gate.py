"""1 - a, which the gate kernel leaves out where only the general scans read it: pairs with strong and moderate chunks side by
side, every way a call comes to its first scan, every kind of gate."""
import numpy as np
import pytest

import paper_2409_07146_b200 as gsa
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
    import torch
    ok, block = torch.empty(1, T, 2, 64, device="cuda"), gsa.gate_block(p, "cuda")
    block.fill_(0x7f)                            # (what is left out is nowhere taken for something)
    gsa.gsa_fwd(p, q, k, v, gate, K0, V0, ok_save=ok, gate_save=block)
    x = gsa.gsa_bwd(p, q, k, v, gate, dO, K0, V0, ok_saved=ok, gate_saved=block)
    y = gsa.gsa_bwd(p, q, k, v, gate, dO, K0, V0, ok_saved=ok)
    torch.cuda.synchronize()
    for a, b in zip(x, y):
        assert rel_err(to_np(a), to_np(b)) <= 1e-6
