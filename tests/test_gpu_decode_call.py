"""The decode step's two ways into the library -- the native check-and-call and the Python one -- accept and refuse the same
calls: memories and outputs alike, errors as the Python path words them."""
import copy

import pytest
import torch

import paper_2409_07146_b200 as gsa
from paper_2409_07146_b200 import binding

pytestmark = pytest.mark.gpu


def call(io="bf16", m=64, **kw):
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *s, dt=torch.float32: torch.randn(*s, generator=g, device="cuda").to(dt)
    p = gsa.Params(2, 1, 3, 64, 128, m, io=io, gate_is_logits=True, **kw)
    dt = p.io_dtype
    gate = r(*p.gate_shape(decode=True), dt=p.gate_torch_dtype)
    return p, [r(2, 3, 64, dt=dt), r(2, 3, 64, dt=dt), r(2, 3, 128, dt=dt), gate, r(2, 3, m, 64), r(2, 3, m, 128), torch.empty(2, 3, 128, dtype=dt, device="cuda")]


@pytest.mark.parametrize("kw", [dict(), dict(io="f32", m=32), dict(gate_bf16=True, m=128), dict(gate_broadcast=True)])
def test_both_ways_do_the_same(kw):
    p, x = call(**kw)
    y = [t.clone() for t in x]
    assert binding._decode_step(p._made_at(), *x) == 0            # the plain call is a native one
    by_python = gsa.gsa_decode_step(p, *y[:6])                    # (no o given: the Python way)
    q = copy.copy(p)                                              # (a copy makes a struct of its own)
    z = [t.clone() for t in call(**kw)[1]]
    assert gsa.gsa_decode_step(q, *z[:6], o=z[6]) is z[6]
    torch.cuda.synchronize()
    for a, b, c in zip(x[4:], y[4:6] + [by_python], z[4:]):
        assert torch.equal(a, b) and torch.equal(a, c)


@pytest.mark.parametrize("at,bad,error", [(0, lambda t: t.float(), TypeError), (2, lambda t: t[..., :64], ValueError),
                                          (4, lambda t: t.transpose(2, 3), ValueError), (5, lambda t: t.cpu(), TypeError),
                                          (3, lambda t: t[:1], ValueError), (6, lambda t: t.tolist(), TypeError)])
def test_what_is_refused(at, bad, error):
    p, x = call()
    keep = [t.clone() for t in x]
    y = list(x)
    y[at] = bad(y[at])
    with pytest.raises(error):
        gsa.gsa_decode_step(p, *y[:6], o=y[6])
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(x[:6], keep))
    with pytest.raises(gsa.GsaError):
        gsa.gsa_decode_step(gsa.Params(2, 1, 3, 96, 128, 64), *[t.new_empty(2, 3, 96) for t in x[:2]], *x[2:4], x[4].new_empty(2, 3, 64, 96),
                            x[5], o=x[6])


@pytest.mark.parametrize("B", [30, 31, 37, 38])
def test_steps_of_a_little_more_than_half_of_what_the_gpu_holds(B):
    # 360 .. 456 pairs of d = 64: 31 and 37 on either edge of the steps that leave an SM three CTAs.  Two steps, one placed
    # while the other runs, against the same pairs in calls of 24.
    H, d, m = 12, 64, 64
    g = torch.Generator(device="cuda").manual_seed(B)
    r = lambda *s, dt=torch.float32: torch.randn(*s, generator=g, device="cuda").to(dt)
    x = [r(B, H, d, dt=torch.bfloat16) for _ in range(3)] + [r(B, H, m), r(B, H, m, d), r(B, H, m, d)]
    y = [t.clone() for t in x]
    p = gsa.Params(B, 1, H, d, d, m, gate_is_logits=True)
    o = torch.empty(2, B, H, d, dtype=torch.bfloat16, device="cuda")
    for i in range(2):
        gsa.gsa_decode_step(p, *x, o=o[i])
    for b in range(0, B, 2):
        n = min(2, B - b)
        part = gsa.Params(n, 1, H, d, d, m, gate_is_logits=True)
        for i in range(2):
            assert torch.equal(gsa.gsa_decode_step(part, *[t[b:b + n] for t in y]), o[i, b:b + n])
    assert torch.equal(x[4], y[4]) and torch.equal(x[5], y[5])
