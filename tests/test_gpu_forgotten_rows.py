"""State runs of segments that forget leave out the chunks of which nothing is left at their ends.  An infinity or a NaN is left
however hard the gates forget, in one segment as in several, and so are numbers that no decay to the end makes nothing of."""
import numpy as np
import pytest

from test_gpu_parity import run_bwd, run_fwd
from util import TOL, rand_inputs, rel_err

import oracle

pytestmark = pytest.mark.gpu


def forgetful(seed, T, H, dk, dv):
    d = rand_inputs(seed, 1, T, H, dk, dv, 64, "bf16", init=True, final_grads=True)
    d["gate"] = (0.2 ** np.random.default_rng(seed).uniform(0.5, 1.5, d["gate"].shape)).astype(np.float32)
    return d


# 3 heads: state runs of one memory a CTA; 8 of 4700 tokens: of both
@pytest.mark.parametrize("H,T,dk,dv", [(3, 1300, 128, 256), (8, 4700, 64, 128)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_what_never_fades_reaches_the_final_memories(H, T, dk, dv, bad):
    d = forgetful(T, T, H, dk, dv)
    d["k"][0, 70, 1, 9] = bad
    d["v"][0, 3, 2, 40] = bad
    with np.errstate(invalid="ignore"):
        got, gate = run_fwd(d, 1, T, H, dk, dv, 64, "bf16", impl="tc", log=True)
        ref = oracle.fwd(d["q"], d["k"], d["v"], gate, gate_is_log=True, K0=d["K0"], V0=d["V0"])
    for n, h, c in (("KT", 1, 9), ("VT", 2, 40)):
        want = ~np.isfinite(ref[n])
        assert want[0, h, :, c].all()
        if n == "KT":                                     # (from the logits on everything of head 1 is lost, its V as well)
            assert np.array_equal(~np.isfinite(got[n]), want), n
        assert (~np.isfinite(got[n][0, h, :, c])).all(), n
        assert np.isfinite(got[n][0, 0]).all()


@pytest.mark.parametrize("H,T", [(3, 1300), (8, 4700)])
def test_a_gate_that_is_no_number(H, T):
    d = forgetful(T + 1, T, H, 128, 128)
    d["gate"][0, 50, 1, 33] = np.nan
    got, _ = run_fwd(d, 1, T, H, 128, 128, 64, "bf16", impl="tc")
    assert (~np.isfinite(got["KT"][0, 1, 33])).all() and np.isfinite(got["KT"][0, 0]).all()


def test_what_never_fades_reaches_the_gradients_of_the_initial_memories():
    H, T, d_ = 3, 1300, 128
    d = forgetful(77, T, H, d_, d_)
    d["dO"][0, T - 60, 1, 5] = np.nan
    with np.errstate(invalid="ignore"):
        got, ref = run_bwd(d, 1, T, H, d_, d_, 64, "bf16", impl="tc", log=True)
    assert (~np.isfinite(ref["dV0"][0, 1, :, 5])).all() and (~np.isfinite(got["dV0"][0, 1, :, 5])).all()
    assert np.isfinite(got["dV0"][0, 0]).all()


@pytest.mark.parametrize("large", [1e5, 1e6, 1e30])       # below the bound and beyond
def test_large_rows_that_the_gates_forget(large):
    H, T, d_ = 3, 1300, 128
    d = forgetful(5, T, H, d_, d_)
    d["v"][0, 20, 1] = large                              # (the chunk is walked, and nothing is left of it)
    got, gate = run_fwd(d, 1, T, H, d_, d_, 64, "bf16", impl="tc", log=True)
    ref = oracle.fwd(d["q"], d["k"], d["v"], gate, gate_is_log=True, K0=d["K0"], V0=d["V0"])
    assert rel_err(got["VT"], ref["VT"]) <= TOL["bf16"] and rel_err(got["KT"], ref["KT"]) <= TOL["bf16"]
    assert rel_err(got["o"][:, 600:], ref["o"][:, 600:], True) <= TOL["bf16"]


@pytest.mark.parametrize("size", [4.0, 1e6])              # weights dz beyond 2, and beyond the bound
def test_gradients_that_the_gates_forget(size):
    H, T, d_ = 3, 1300, 128
    d = forgetful(6, T, H, d_, d_)
    d["dO"] = (d["dO"] * np.float32(2.0 ** np.round(np.log2(size)))).astype(np.float32)
    d["dO"][:, 900:] *= 4
    d["dKT"], d["dVT"] = d["dKT"] * np.float32(size), d["dVT"] * np.float32(size)
    got, ref = run_bwd(d, 1, T, H, d_, d_, 64, "bf16", impl="tc", log=True)
    for n in ("dK0", "dV0"):
        assert rel_err(got[n], ref[n]) <= TOL["bf16"], n
