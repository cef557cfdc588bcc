"""The five independent scans of an fp32 backward run side by side on the library's streams: a step captured into a graph by a
process whose first calls it holds, on a stream of its own, replays what plain calls give, bit for bit."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
import paper_2409_07146_b200 as gsa
T, m = {T}, {m}
g = torch.Generator(device="cuda").manual_seed(1)
r = lambda *s: torch.randn(*s, generator=g, device="cuda")
p = gsa.Params(2, T, 2, 128, 64, m, io="f32", gate_is_logits=True)
q, k, v, gate, dO = r(2, T, 2, 128) * 0.09, r(2, T, 2, 128), r(2, T, 2, 64), r(2, T, 2, m), r(2, T, 2, 64)
w = [torch.empty(gsa.gsa_workspace_bytes(p, i), dtype=torch.uint8, device="cuda") for i in (0, 1)]
ok, o = torch.empty(2, T, 2, m, device="cuda"), torch.empty_like(v)
out = [torch.empty_like(t) for t in (q, k, v, gate)]
def step():
    gsa.gsa_fwd(p, q, k, v, gate, o=o, ok_save=ok, ws=w[0])
    gsa.gsa_bwd(p, q, k, v, gate, dO, ok_saved=ok, dq=out[0], dk=out[1], dv=out[2], dgate=out[3], ws=w[1])
side = torch.cuda.Stream()
graph = torch.cuda.CUDAGraph()
torch.cuda.synchronize()
with torch.cuda.graph(graph, stream=side):
    step()
step()
torch.cuda.synchronize()
plain = [t.clone() for t in [o, ok] + out]
for _ in range(3):
    for t in [o, ok] + out:
        t.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip([o, ok] + out, plain))
del graph
gsa.gsa_release_streams()
step()
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip([o, ok] + out, plain))
print("same")
"""


@pytest.mark.parametrize("T,m", [(65, 32), (700, 64)])
def test_captured_and_plain_steps_agree(T, m):
    done = subprocess.run([sys.executable, "-c", PROGRAM.format(T=T, m=m)], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0 and "same" in done.stdout, done.stderr[-2000:]


BESIDE = """
import torch
import paper_2409_07146_b200 as gsa
g = torch.Generator(device="cuda").manual_seed(2)
r = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.{dtype})
p = gsa.Params(2, 130, 2, 128, 64, 64, io="{io}", gate_is_logits=True)
q, k, v, dO = r(2, 130, 2, 128) * 0.09, r(2, 130, 2, 128), r(2, 130, 2, 64), r(2, 130, 2, 64)
gate = r(2, 130, 2, 64).float()
ws = [torch.empty(gsa.gsa_workspace_bytes(p, 1), dtype=torch.uint8, device="cuda") for _ in range(2)]
out = [[torch.empty_like(t) for t in (q, k, v, gate)] for _ in range(2)]
def step(i):
    gsa.gsa_bwd(p, q, k, v, gate, dO, dq=out[i][0], dk=out[i][1], dv=out[i][2], dgate=out[i][3], ws=ws[i])
step(0)
torch.cuda.synchronize()
want = [t.clone() for t in out[0]]
graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
with torch.cuda.graph(graph, capture_error_mode="relaxed"):
    step(0)
    with torch.cuda.stream(other):
        step(1)
    step(0)
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip(out[1], want))
for t in out[0]:
    t.fill_(7.0)
graph.replay()
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip(out[0], want))
step(1)
torch.cuda.synchronize()
print("same")
"""


@pytest.mark.parametrize("io,dtype", [("f32", "float32"), ("bf16", "bfloat16")])
def test_a_plain_call_between_two_captured_ones(io, dtype):
    # the captured calls hold the thread's lanes until the capture ends: a call on another stream does without
    done = subprocess.run([sys.executable, "-c", BESIDE.format(io=io, dtype=dtype)], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0 and "same" in done.stdout, done.stderr[-2000:]
