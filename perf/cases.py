"""The work that users of the GSA library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  Three kinds of use:

  train    a training step of the layer: gsa_fwd with the logits and the gate kernel's products kept, then
           gsa_bwd on them.  With `out_norm` the layer's element-wise output path (Swish -> RMSNorm) and its
           backward stand between the two, with `feature` the Swish feature map is applied by the library.
  forward  a prefill: gsa_fwd over whole prompts; with `carry` from given memories, the final memories
           (what decoding goes on from) are returned either way.
  decode   one token through `layers` GSA layers for B sequences, the memories updated in place.

Sizes: B sequences of T tokens, H heads of width d_k = d_v = d, m slots.  nseq > 0: B rows of T tokens hold
nseq sequences of random lengths back to back.  The gate tensor holds a, log a or the logits x of
a = sigmoid(x)^(1/tau), x ~ N(mu, 1).
"""
import random

import torch

import paper_2409_07146_b200 as gsa

DEFAULTS = dict(B=1, T=1, H=4, d=128, m=64, io="bf16", gate="a", gate_bf16=False, mu=0.0, tau=8.0, k_sigma=0.0,
                feature=False, out_norm=False, nseq=0, carry=False, layers=1)


def _case(**kw):
    return dict(DEFAULTS, **kw)


def listed():
    return [
        # the smallest call: a short fp32 sequence, two heads (a unit test, a numerics check, a toy model): latency
        _case(name="forward_tiny_f32", kind="forward", B=1, T=256, H=2, d=64, m=32, io="f32"),
        # a training step in fp32 (debugging a bf16 run, gradient checks): the CUDA-core kernels
        _case(name="train_f32", kind="train", B=2, T=1024, H=4, d=256, io="f32", gate="log"),
        # pre-training, the 1.3B model's layer: 4 heads of width 512 over 2K windows (the benchmark's workload)
        _case(name="train_1p3b", kind="train", B=8, T=2048, H=4, d=512),
        # finetuning a pretrained 7B transformer: 32 heads of width 128, outlier channels in the keys
        _case(name="train_7b_geometry", kind="train", B=4, T=4096, H=32, d=128, k_sigma=0.5),
        # the 2.7B model's whole layer, as a model calls it: projections' outputs in, bf16 gate logits, Swish feature
        # map, Swish -> RMSNorm output; a window length that no tile divides
        _case(name="train_2p7b_layer_ragged", kind="train", B=4, T=1999, H=5, d=512, gate="logits", gate_bf16=True,
              feature=True, out_norm=True),
        # finetuning on packed variable-length sequences: 13 of them in one row of 8K tokens
        _case(name="train_packed", kind="train", B=1, T=8192, H=4, d=512, gate="logits", nseq=13),
        # the largest slot count of the ablation on the number of slots, on the 1.3B model's layer
        _case(name="train_128_slots", kind="train", B=8, T=2048, H=4, d=512, m=128),
        # serving: the prefill of one prompt of odd length with the 1.3B model's layer, memories handed to decoding
        _case(name="forward_prompt", kind="forward", B=1, T=1431, H=4, d=512, gate="logits"),
        # long context with carried memories, gates that keep nearly everything ...
        _case(name="forward_long_keep", kind="forward", B=1, T=32768, H=16, d=128, mu=2.0, tau=16.0, carry=True),
        # ... and gates that forget within a few tokens
        _case(name="forward_long_forget", kind="forward", B=1, T=32768, H=16, d=128, mu=-2.0, tau=1.0, carry=True),
        # serving: one token for a batch of 256 sequences (a pure stream of the memories)
        _case(name="decode_batch", kind="decode", B=256, H=32, d=128),
        # serving: one token of one sequence through the 24 layers of the 1.3B model: latency and launches
        _case(name="decode_one_sequence", kind="decode", B=1, H=4, d=512, layers=24),
    ]


# H heads of width d that layers are built with: the 1.3B and 2.7B models, the 7B geometry, and generic ones
GEOMETRIES = ((4, 512), (5, 512), (32, 128), (16, 128), (8, 256), (12, 64))
MAX_ELEMENTS = 4 * 4096 * 32 * 128      # B T H d of the largest listed training step
MAX_MEMORY = 256 * 32 * 64 * 128        # B H m d (and layers) of the largest listed decode step


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform over its logarithm; mostly odd."""
    x = int(round(lo * (hi / lo) ** rng.random()))
    if rng.random() < 0.25:
        x = (x + 32) // 64 * 64         # a quarter of the lengths are round
    return max(lo, min(hi, x))


def draw(rng):
    use = rng.choice(("train", "train", "train", "packed", "slots", "f32", "forward", "forward", "long", "decode", "decode"))
    gate, gate_bf16 = rng.choice((("a", False), ("log", False), ("logits", False), ("logits", True)))
    H, d = rng.choice(GEOMETRIES)
    if use == "f32":
        H, d = rng.choice(((2, 64), (4, 128), (4, 256)))
        T = _log_int(rng, 64, 1024)
        return _case(kind=rng.choice(("forward", "train")), B=rng.randint(1, 2), T=T, H=H, d=d,
                     m=rng.choice((32, 64)), io="f32", gate=gate, carry=rng.random() < 0.5)
    if use == "packed":
        H, d = rng.choice(((4, 512), (16, 128)))
        return _case(kind="train", B=1, T=_log_int(rng, 1024, 8192), H=H, d=d, gate=gate, gate_bf16=gate_bf16,
                     nseq=rng.randint(2, 16))
    if use == "slots":
        B = rng.randint(1, 8)
        T = _log_int(rng, 128, 2048)
        return _case(kind="train", B=B, T=T, H=4, d=512, m=rng.choice((32, 128)), gate=gate, gate_bf16=gate_bf16)
    if use == "train":
        B = rng.randint(1, 8)
        T = _log_int(rng, 128, max(128, min(8192, MAX_ELEMENTS // (B * H * d))))
        layer = H * d <= 4096 and rng.random() < 0.4
        return _case(kind="train", B=B, T=T, H=H, d=d, gate=gate, gate_bf16=gate_bf16, feature=layer, out_norm=layer)
    if use == "forward":
        B = rng.choice((1, 1, 2, 4))
        return _case(kind="forward", B=B, T=_log_int(rng, 64, 8192), H=H, d=d, gate=gate, gate_bf16=gate_bf16,
                     carry=rng.random() < 0.5)
    if use == "long":
        mu, tau = rng.choice(((2.0, 16.0), (0.0, 8.0), (-2.0, 1.0)))
        T = _log_int(rng, 8192, 32768)
        return _case(kind="forward", B=1, T=T, H=16, d=128, mu=mu, tau=tau, gate=gate, carry=True)
    layers = rng.choice((1, 8, 24))
    most = max(1, min(256, MAX_MEMORY // (layers * H * 64 * d)))
    return _case(kind="decode", B=_log_int(rng, 1, most), H=H, d=d, gate=gate, gate_bf16=gate_bf16, layers=layers)


# ------------------------------------------------------------------ what a program has in hand before the call
def _params(c, cu=None):
    return gsa.Params(c["B"], c["T"], c["H"], c["d"], c["d"], c["m"], io=c["io"], gate_is_log=c["gate"] == "log",
                      gate_is_logits=c["gate"] == "logits", tau=c["tau"], gate_bf16=c["gate_bf16"],
                      feature_map="swish" if c["feature"] else "none", cu_seqlens=cu)


def _offsets(c, seed):
    """nseq + 1 ascending offsets of sequences of random lengths that fill T tokens."""
    rng = random.Random(seed)
    cuts = sorted(rng.sample(range(1, c["T"]), c["nseq"] - 1))
    return torch.tensor([0] + cuts + [c["T"]], dtype=torch.int32, device="cuda")


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)
    io = torch.bfloat16 if c["io"] == "bf16" else torch.float32
    B, T, H, d, m = (c[n] for n in ("B", "T", "H", "d", "m"))
    decode = c["kind"] == "decode"

    def normal(*shape, scale=1.0, dtype=io):
        return (torch.randn(*shape, generator=g, device="cuda") * scale).to(dtype)

    def gate_tensor(*shape):
        x = torch.randn(*shape, generator=g, device="cuda") + c["mu"]
        if c["gate"] == "logits":
            gate = x
        else:
            gate = torch.nn.functional.logsigmoid(x) / c["tau"]
            gate = gate.exp() if c["gate"] == "a" else gate
        return gate.to(torch.bfloat16 if c["gate_bf16"] else torch.float32).contiguous()

    def token_inputs(*lead):
        # (with the feature map the tensors are the projections' outputs and scaling q is theirs too)
        x = {"q": normal(*lead, H, d, scale=d ** -0.5), "k": normal(*lead, H, d), "v": normal(*lead, H, d),
             "gate": gate_tensor(*lead, H, m)}
        if c["k_sigma"]:
            scale = torch.exp(c["k_sigma"] * torch.randn(H, d, generator=g, device="cuda"))
            x["k"] = (x["k"].float() * scale).to(io)
        return x

    s = {"case": c}
    if decode:
        s["p"] = _params(dict(c, T=1))
        s["layers"] = [dict(token_inputs(B), K=normal(B, H, m, d, scale=0.1, dtype=torch.float32),
                            V=normal(B, H, m, d, scale=0.1, dtype=torch.float32),
                            o=torch.empty(B, H, d, dtype=io, device="cuda")) for _ in range(c["layers"])]
        return s
    p = s["p"] = _params(c, _offsets(c, seed) if c["nseq"] else None)
    s["x"] = token_inputs(B, T)
    s["ws_fwd"] = torch.empty(gsa.gsa_workspace_bytes(p, 0), dtype=torch.uint8, device="cuda")
    if c["carry"]:
        s["K0"] = normal(B, H, m, d, scale=0.1, dtype=torch.float32)
        s["V0"] = normal(B, H, m, d, scale=0.1, dtype=torch.float32)
    if c["kind"] == "train":
        s["dy"] = normal(B, T, H, d)
        s["ws_bwd"] = torch.empty(gsa.gsa_workspace_bytes(p, 1), dtype=torch.uint8, device="cuda")
        s["saved"] = gsa.gate_block(p, "cuda")
        s["logits"] = torch.empty(B, T, H, m, device="cuda")
        s["norm_weight"] = 1.0 + normal(H * d, scale=0.1, dtype=torch.float32)
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    s = state
    c, p = s["case"], s["p"]
    if c["kind"] == "decode":
        for x in s["layers"]:
            gsa.gsa_decode_step(p, x["q"], x["k"], x["v"], x["gate"], x["K"], x["V"], o=x["o"])
        first, last = s["layers"][0], s["layers"][-1]
        return [first["o"], first["K"], first["V"], last["o"], last["K"], last["V"]]
    q, k, v, gate = (s["x"][n] for n in ("q", "k", "v", "gate"))
    K0, V0 = s.get("K0"), s.get("V0")
    if c["kind"] == "forward":
        KT = torch.empty(c["B"], c["H"], c["m"], c["d"], device="cuda")
        VT = torch.empty_like(KT)
        o = gsa.gsa_fwd(p, q, k, v, gate, K0, V0, KT=KT, VT=VT, ws=s["ws_fwd"])
        return {"o": o, "KT": KT, "VT": VT}
    o = gsa.gsa_fwd(p, q, k, v, gate, K0, V0, ok_save=s["logits"], ws=s["ws_fwd"], gate_save=s["saved"])
    out = {}
    d_o = s["dy"]
    if c["out_norm"]:
        out["y"] = gsa.gsa_out_norm_fwd(p, o, s["norm_weight"])
        d_o, out["dweight"] = gsa.gsa_out_norm_bwd(p, o, s["dy"], s["norm_weight"])
    out["o"] = o
    out["dq"], out["dk"], out["dv"], out["dgate"] = gsa.gsa_bwd(
        p, q, k, v, gate, d_o, K0, V0, ok_saved=s["logits"], ws=s["ws_bwd"], gate_saved=s["saved"])
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c = case
    e = 2 if c["io"] == "bf16" else 4
    eg = 2 if c["gate_bf16"] else 4
    H, d, m = c["H"], c["d"], c["m"]
    memories = 8 * c["B"] * H * m * d                     # K~ and V~, fp32
    if c["kind"] == "decode":
        rows = c["B"] * H
        return {"bytes": c["layers"] * (2 * memories + rows * (4 * d * e + m * eg)),
                "flops": c["layers"] * rows * 8.0 * m * d}
    rows = c["B"] * c["T"] * H
    forward = rows * (4 * d * e + m * eg)                 # q, k, v, gate -> o
    flops = rows * 8.0 * m * d                            # two memories updated and read
    if c["kind"] == "forward":
        return {"bytes": forward + memories * (2 if c["carry"] else 1), "flops": flops}
    # q, k, v, gate, the output's gradient -> three gradients and the gate's; the output path reads o and dy again
    backward = rows * (7 * d * e + m * (eg + 4))
    if c["out_norm"]:
        backward += rows * d * e * 3                      # y out; o and dy in again for the norm's gradient
    return {"bytes": forward + backward, "flops": 3.0 * flops}


def tolerance(case):
    # About four times what the outputs differ by from the fp64 recurrence (2-norms, and the worst element over the rms
    # or its own value): fp32 io 6e-7 and 1.1e-5; bf16 io 1.7e-3 and 3.9e-3, the rounding of the outputs' own format; a
    # whole layer hands bf16 tensors (o and its gradient, gradients before the feature map's) on to the next step and
    # shows 4e-3 and 3.5e-2.
    if case["io"] == "f32":
        return {"rel": 3e-6, "max": 5e-5}
    if case["feature"] or case["out_norm"]:
        return {"rel": 1.6e-2, "max": 0.14}
    return {"rel": 6.6e-3, "max": 1.6e-2}


# ------------------------------------------------------------------ the same in 64 bits
def _swish_slope(x):
    g = torch.sigmoid(x)
    return g * (1.0 + x * (1.0 - g))


def _decay(c, gate):
    """a (the share of its memory that a slot keeps) and d a / d gate."""
    x = gate.double()
    if c["gate"] == "a":
        return x, torch.ones_like(x)
    if c["gate"] == "log":
        return x.exp(), x.exp()
    a = torch.exp(torch.nn.functional.logsigmoid(x) / c["tau"])
    return a, a * torch.sigmoid(-x) / c["tau"]


def _step(K, V, a, q, k, v):
    """One token of the recurrence; the memories K, V [N, m, d] are updated in place.  Returns o and the slot weights."""
    w = (1.0 - a).unsqueeze(2)
    K.mul_(a.unsqueeze(2)).baddbmm_(w, k.unsqueeze(1))
    V.mul_(a.unsqueeze(2)).baddbmm_(w, v.unsqueeze(1))
    p = torch.softmax(torch.bmm(K, q.unsqueeze(2)).squeeze(2), 1)
    return torch.bmm(p.unsqueeze(1), V).squeeze(1), p


def _exact_decode(s):
    c, out = s["case"], []
    for x in (s["layers"][0], s["layers"][-1]):
        n = c["B"] * c["H"]
        q, k, v = (x[t].double().view(n, c["d"]) for t in ("q", "k", "v"))
        K, V = (x[t].double().view(n, c["m"], c["d"]).clone() for t in ("K", "V"))
        o, _ = _step(K, V, _decay(c, x["gate"])[0].view(n, c["m"]), q, k, v)
        out += [o.view(x["o"].shape), K.view(x["K"].shape), V.view(x["V"].shape)]
    return out


@torch.no_grad()
def exact(case, seed):
    s = prepare(case, seed)
    c = s["case"]
    if c["kind"] == "decode":
        return _exact_decode(s)
    B, T, H, d, m = (c[n] for n in ("B", "T", "H", "d", "m"))
    N = B * H

    def by_time(x):                                       # [B, T, H, n] -> [T, B H, n]
        return x.double().permute(1, 0, 2, 3).reshape(T, N, -1)

    def by_batch(x):
        return x.view(T, B, H, -1).permute(1, 0, 2, 3).contiguous()

    raw = {n: by_time(s["x"][n]) for n in ("q", "k", "v")}
    q, k, v = (torch.nn.functional.silu(raw[n]) if c["feature"] else raw[n] for n in ("q", "k", "v"))
    a, slope = _decay(c, by_time(s["x"]["gate"]))
    starts = set(_offsets(c, seed).tolist()[1:-1]) if c["nseq"] else set()
    K = s["K0"].double().view(N, m, d).clone() if c["carry"] else torch.zeros(N, m, d, dtype=torch.float64, device="cuda")
    V = s["V0"].double().view(N, m, d).clone() if c["carry"] else torch.zeros_like(K)
    o, p = torch.empty_like(v), torch.empty_like(a)
    kept = {}                                             # the memories before every 64th token, for the way back

    def forward(t):
        if t in starts:
            K.zero_(), V.zero_()
        o[t], p[t] = _step(K, V, a[t], q[t], k[t], v[t])

    for t in range(T):
        if c["kind"] == "train" and t % 64 == 0:
            kept[t] = K.clone(), V.clone()
        forward(t)
    if c["kind"] == "forward":
        return {"o": by_batch(o), "KT": K.view(B, H, m, d).clone(), "VT": V.view(B, H, m, d).clone()}
    out = {}
    d_o = by_time(s["dy"])
    ob = by_batch(o)
    if c["out_norm"]:
        with torch.enable_grad():
            x, w = ob.clone().requires_grad_(), s["norm_weight"].double().requires_grad_()
            y = torch.nn.functional.rms_norm(torch.nn.functional.silu(x).view(B, T, H * d), (H * d,), w, 1e-6)
            gx, out["dweight"] = torch.autograd.grad(y, (x, w), s["dy"].double().view(B, T, H * d))
        out["y"] = y.detach().view(B, T, H, d)
        d_o = by_time(gx)
    out["o"] = ob
    dq, dk, dv, da = torch.empty_like(q), torch.empty_like(k), torch.empty_like(v), torch.empty_like(a)
    gK, gV = torch.zeros_like(K), torch.zeros_like(V)     # gradients w.r.t. the memories after token t
    for t0 in reversed(range(0, T, 64)):
        K.copy_(kept[t0][0]), V.copy_(kept[t0][1])
        before, after = [], []
        for t in range(t0, min(t0 + 64, T)):
            if t in starts:
                K.zero_(), V.zero_()
            before.append((K.clone(), V.clone()))
            forward(t)
            after.append((K.clone(), V.clone()))
        for t in reversed(range(t0, min(t0 + 64, T))):
            (K0, V0), (K1, V1) = before[t - t0], after[t - t0]
            dp = torch.bmm(V1, d_o[t].unsqueeze(2)).squeeze(2)
            dz = p[t] * (dp - (p[t] * dp).sum(1, keepdim=True))
            dq[t] = torch.bmm(dz.unsqueeze(1), K1).squeeze(1)
            gK.baddbmm_(dz.unsqueeze(2), q[t].unsqueeze(1))
            gV.baddbmm_(p[t].unsqueeze(2), d_o[t].unsqueeze(1))
            w = (1.0 - a[t]).unsqueeze(1)
            dk[t], dv[t] = torch.bmm(w, gK).squeeze(1), torch.bmm(w, gV).squeeze(1)
            da[t] = ((gK * K0).sum(2) + (gV * V0).sum(2) - torch.bmm(gK, k[t].unsqueeze(2)).squeeze(2)
                     - torch.bmm(gV, v[t].unsqueeze(2)).squeeze(2))
            keep = torch.zeros_like(a[t]) if t in starts else a[t]
            gK.mul_(keep.unsqueeze(2)), gV.mul_(keep.unsqueeze(2))
    for n, g in (("q", dq), ("k", dk), ("v", dv)):
        out["d" + n] = by_batch(g * _swish_slope(raw[n]) if c["feature"] else g)
    out["dgate"] = by_batch(da * slope)
    return out
