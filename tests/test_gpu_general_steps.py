"""The scans of flagged (batch, head) pairs, which walk 16 tokens at a time: steps that end within a tile, gates that lose
everything between two tokens (the decay over a step is far below e^-60 then), half a slice of channels and several slices,
both directions; and state runs that leave out the chunks of which nothing is left."""
import numpy as np
import pytest

from test_gpu_parity import check_bwd, check_fwd, run_bwd, run_fwd
from util import TOL, rand_inputs

pytestmark = pytest.mark.gpu


def check(d, B, T, H, dk, dv, m):
    got, g = run_fwd(d, B, T, H, dk, dv, m, "bf16", impl="tc", log=True)
    check_fwd(d, got, g, "bf16", log=True, tc=True)
    gb, rb = run_bwd(d, B, T, H, dk, dv, m, "bf16", impl="tc", log=True)
    check_bwd(gb, rb, TOL["bf16"], tc=True)


@pytest.mark.parametrize("T", [2, 15, 16, 17, 31, 145])
@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 256)])
def test_gates_that_lose_everything(T, dk, dv):
    B, H, m = 2, 2, 64
    d = rand_inputs(700 + T, B, T, H, dk, dv, m, "bf16", init=True, final_grads=True)
    r = np.random.default_rng(T)
    a = 0.9 ** r.uniform(0.0, 2.0, d["gate"].shape)
    a[r.random(d["gate"].shape) < 0.1] = 1e-30            # e^-69
    a[:, T // 2] = 1e-30                                  # every slot at once
    a[:, :, :, 7] = 1.0
    a[:, -1, :, 3] = 1e-30                                # (every pair is flagged)
    d["gate"] = a.astype(np.float32)
    check(d, B, T, H, dk, dv, m)


@pytest.mark.parametrize("T", [897, 1300])
@pytest.mark.parametrize("slow", [0.2, 0.9, 1.0])         # one slot keeps e^-206, e^-13 or all of a chunk
def test_state_runs_of_forgetful_segments(T, slow):
    B, H, dk, dv, m = 1, 2, 128, 128, 64
    d = rand_inputs(800 + T, B, T, H, dk, dv, m, "bf16", init=True, final_grads=True)
    r = np.random.default_rng(T)
    a = 0.2 ** r.uniform(0.5, 1.5, d["gate"].shape)
    a[..., 11] = slow
    d["gate"] = a.astype(np.float32)
    check(d, B, T, H, dk, dv, m)
