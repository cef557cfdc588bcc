"""The walking gate gradient of calls that are cut into segments, some of them flagged for strong decay and their neighbours not:
a tile of 256 (128) rows may span two segments, of which one has a row factor pending and the other has not."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_07146_b200 as gsa
from util import TOL, rand_inputs, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu

CHUNK = 128


def strong_in_one_chunk_a_head(d, T):
    """Head h forgets e^-76 in slot h within chunk h of its tokens (the heads past the last chunk nowhere)."""
    for h in range(min(d["gate"].shape[2], T // CHUNK)):
        t = h * CHUNK + 40
        d["gate"][:, t:t + 40, h, h % d["gate"].shape[3]] = 0.15


def dgate_of(d, kind, T, cu=None):
    """(dgate of the library, of the oracle) for the gates d["gate"] = a, handed over as `kind`."""
    B, _, H, dk = d["q"].shape
    dv, m = d["v"].shape[-1], d["gate"].shape[-1]
    a, tau = d["gate"].astype(np.float64), 8.0
    if kind == "a":
        gate = d["gate"]
    elif kind == "log":
        gate = np.log(a).astype(np.float32)
    else:                                  # a = sigmoid(x)^(1/tau)
        sig = np.minimum(a ** tau, 1 - 1e-7)
        gate = (np.log(sig) - np.log1p(-sig)).astype(np.float32)
    p = gsa.Params(B, T, H, dk, dv, m, io="bf16", gate_is_log=kind == "log", gate_is_logits=kind == "logits", tau=tau,
                   cu_seqlens=None if cu is None else torch.tensor(cu, dtype=torch.int32, device="cuda"))
    q, k, v, dO = (to_dev(d[n], "bf16") for n in ("q", "k", "v", "dO"))
    x = to_dev(gate)
    K0, V0, dKT, dVT = (to_dev(d.get(n)) for n in ("K0", "V0", "dKT", "dVT"))
    got = to_np(gsa.gsa_bwd(p, q, k, v, x, dO, K0, V0, dKT=dKT, dVT=dVT)[3])
    kw = dict(gate_is_log=kind == "log", gate_is_logits=kind == "logits", tau=tau,
              **{n: d.get(n) for n in ("K0", "V0", "dKT", "dVT")})
    args = (d["q"], d["k"], d["v"], gate, d["dO"])
    ref = oracle.bwd(*args, **kw) if cu is None else oracle.bwd_packed(*args, cu, **kw)
    return got, ref["dgate"]


# 16 slots a CTA (28 .. 37 pairs, tiles of 256 rows), 32 (45 .. 74, tiles of 128; at 3200 tokens logits take the three kernels), 128 slots
@pytest.mark.parametrize("B,H,T,dk,dv,m", [(1, 32, 1500, 128, 128, 64), (1, 32, 2304, 128, 128, 64), (2, 16, 1500, 128, 256, 64),
                                           (1, 47, 1500, 64, 128, 64), (1, 48, 3200, 64, 64, 64),
                                           (1, 16, 1500, 128, 128, 128)])
@pytest.mark.parametrize("kind", ["a", "log", "logits"])
def test_flagged_segments_beside_others(B, H, T, dk, dv, m, kind):
    d = rand_inputs(T + H + m, B, T, H, dk, dv, m, "bf16", init=True, final_grads=True)
    strong_in_one_chunk_a_head(d, T)
    got, ref = dgate_of(d, kind, T)
    assert np.isfinite(got).all()
    # (by head: a wrong one is not hidden behind the others' rms)
    errs = [rel_err(got[:, :, h], ref[:, :, h]) for h in range(H)]
    assert max(errs) <= TOL["bf16"], errs


@pytest.mark.parametrize("kind", ["a", "logits"])
def test_offsets_that_flag_a_segment(kind):
    B, H, T, dk, m = 1, 32, 1500, 128, 64
    cu = [0, 400, 430, 780, 1200, 1210, 1499, T]         # two of one chunk in the second segment, and in the last
    d = rand_inputs(5, B, T, H, dk, dk, m, "bf16")
    got, ref = dgate_of(d, kind, T, cu)
    assert np.isfinite(got).all() and rel_err(got, ref) <= TOL["bf16"]
