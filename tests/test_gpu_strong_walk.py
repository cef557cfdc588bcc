"""Chunks of strong decay on the tensor-core kernels.  One slot that forgets hard sends the pair to the scans that walk 16 tokens at
a time; the others remember a step or two, a few of them, or all of the chunk; ragged chunks and steps; both directions."""
import numpy as np
import pytest

from test_gpu_parity import check_bwd, check_fwd, run_bwd, run_fwd
from util import TOL, rand_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 33, 128, 161, 300])
@pytest.mark.parametrize("keep", [0.2, 0.55, 0.999])     # below 2^-40 after 18 steps, 47 steps, 27713
def test_strong_decay_walk(T, keep):
    B, H, dk, dv, m = 1, 2, 128, 64, 64
    d = rand_inputs(900 + T, B, T, H, dk, dv, m, "bf16", init=True, final_grads=True)
    r = np.random.default_rng(T)
    a = keep ** r.uniform(0.5, 1.5, d["gate"].shape)
    a[..., 5] = 0.2                                       # e^-206 over a chunk of 128 tokens
    a[..., 40] = 0.3
    d["gate"] = a.astype(np.float32)
    got, g = run_fwd(d, B, T, H, dk, dv, m, "bf16", impl="tc", log=True)
    check_fwd(d, got, g, "bf16", log=True, tc=True)
    gb, rb = run_bwd(d, B, T, H, dk, dv, m, "bf16", impl="tc", log=True)
    check_bwd(gb, rb, TOL["bf16"], tc=True)
