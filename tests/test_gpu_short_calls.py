"""A call of one chunk: the gate kernel's CTA writes its pair's strong-decay flag itself, whatever the workspace holds, so that
moderate pairs take the pipelined scans and strong ones the general scans.  Two chunks share a flag that is cleared first."""
import numpy as np
import pytest
import torch

import paper_2409_07146_b200 as gsa
from paper_2409_07146_b200.binding import GSA_WS_FWD
from test_gpu_parity import check_fwd
from util import rand_inputs, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 100, 128, 129])
@pytest.mark.parametrize("m", [32, 64, 128])
@pytest.mark.parametrize("log", [False, True])
def test_flags_do_not_depend_on_the_workspace(T, m, log):
    B, H, dk, dv = 2, 2, 128, 128
    d = rand_inputs(900 + T, B, T, H, dk, dv, m, "bf16", init=True)
    d["gate"][0, T // 2, 1, :5] = 1e-30            # (e^-69 in one pair of four)
    gate = np.log(d["gate"].astype(np.float64)).astype(np.float32) if log else d["gate"]
    p = gsa.Params(B, T, H, dk, dv, m, io="bf16", gate_is_log=log)
    io = [to_dev(d[n], "bf16") for n in "qkv"]
    got = []
    for fill in (0, 255):
        ws = torch.full((gsa.gsa_workspace_bytes(p, GSA_WS_FWD),), fill, dtype=torch.uint8, device="cuda")
        KT, VT = torch.empty(B, H, m, dk, device="cuda"), torch.empty(B, H, m, dv, device="cuda")
        ok = torch.empty(B, T, H, m, device="cuda")
        o = gsa.gsa_fwd(p, *io, to_dev(gate), to_dev(d["K0"]), to_dev(d["V0"]), ok_save=ok, KT=KT, VT=VT, ws=ws)
        torch.cuda.synchronize()
        got.append(dict(o=to_np(o), ok=to_np(ok), KT=to_np(KT), VT=to_np(VT)))
    check_fwd(d, got[0], gate, "bf16", log=log, tc=True)
    for n in got[0]:
        assert np.array_equal(got[0][n], got[1][n]), n
