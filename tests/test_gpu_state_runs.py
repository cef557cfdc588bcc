"""State runs of segment-parallel scheduling on the CUDA-core kernels (K and V side in one launch, which also leaves the
segments' log-decay): ragged last segments, every slot count, chunks that decay too hard for one reference point."""
import numpy as np
import pytest

from test_gpu_parity import check_bwd, check_fwd, run_bwd, run_fwd
from util import TOL, rand_inputs, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [32, 64, 128])
@pytest.mark.parametrize("T,dk,dv,gate", [(193, 64, 128, "tau8"), (200, 128, 64, "strong"), (449, 256, 64, "tau8")])
def test_state_runs_on_cuda_cores(T, dk, dv, m, gate):
    d = rand_inputs(600 + T + m, 2, T, 2, dk, dv, m, "f32", init=True, final_grads=True, gate=gate)
    got, g = run_fwd(d, 2, T, 2, dk, dv, m, "f32", log=True)
    check_fwd(d, got, g, "f32", log=True)
    gb, rb = run_bwd(d, 2, T, 2, dk, dv, m, "f32", log=True)
    if gate == "strong":
        # |G| reaches 200 in a chunk: its fp32 rounding makes every decay factor 200 2^-24 wrong whatever the state runs do,
        # and up to four of them multiply the terms of a gradient, the largest of which are largest / rms times the rms
        # (4e-4 on the gate gradient, 2e-4 on dq)
        assert all(np.isfinite(t).all() for t in gb.values())
        for n, t in gb.items():
            largest = np.abs(rb[n]).max() / np.sqrt(np.mean(rb[n] ** 2))
            assert rel_err(t, rb[n]) <= TOL["f32"] + 4 * 200 * 2.0 ** -24 * largest, n
        return
    check_bwd(gb, rb, TOL["f32"])
