"""The work that programs have this library do, as cases to measure.

A case is one call of the MoE layer (or of its steps one by one) on a shape of
the families this library is built for:

  decode     the Mixtral-shaped bf16 layer on decode batches of 1..256 tokens
             (d = 4096, 8 SwiGLU experts, d_ff = 14336, Top-2, codec rank
             128..512, 4 to 8 experts allowed on the device)
  mixtral    the same layer on prefill batches, whole or in ragged chunks
  switch     Switch-Transformer-base layers (d = 768, d_ff = 3072, GELU,
             Top-1, 8..64 experts with a share of them allowed): the paper's
             own evaluation (batch 4 x 256 tokens, 64 experts, 40% cap) and
             the batch 8 x 512 preset
  fine       fine-grained bf16 layers (d = 2048, 64 SwiGLU experts of width
             1408, Top-6 over 8 groups, 2 shared experts, Zipf popularity),
             from decode steps to full prefill batches
  fp32       layers kept in fp32 (PyTorch's default type): the tiny preset and
             Switch-sized ones

op "layer" is ec2moe_layer_forward, "pipelined" the end/cloud two-stream call,
"steps" the same layer as a program composes it from the single entry points
(gate, encode, decode, route + gather, experts, shared experts, combine), whose
intermediate results are all returned.

Inputs: X ~ N(0, 1), weights ~ N(0, 1 / fan_in), biases zero or Zipf, bf16
tensors rounded once to their storage type.
"""

from __future__ import annotations

import math

import torch

from paper_2508_06024_gb300 import ec2moe as C

MIXTRAL = dict(d=4096, E=8, d_ff=14336, k=2, act="swiglu", dtype="bf16", n_shared=0, zipf=0.0)
SWITCH = dict(d=768, d_ff=3072, k=1, act="gelu", dtype="bf16", n_shared=0, zipf=0.0)
FINE = dict(d=2048, E=64, d_ff=1408, k=6, act="swiglu", dtype="bf16", n_shared=2, zipf=1.2)


def _case(family, op, T, groups, allowed, r, renorm=0, top_groups=0, micro=0, **over):
    return dict(family, op=op, T=T, groups=groups, allowed=allowed, r=r, renorm=renorm, top_groups=top_groups,
                micro=micro, **over)


def listed():
    named = [
        # One token of a Mixtral-shaped decoder: latency, two experts' weights.
        ("decode_1", _case(MIXTRAL, "layer", 1, 1, 8, 256)),
        # A serving batch's decode step: every expert's weights, few rows each.
        ("decode_64", _case(MIXTRAL, "layer", 64, 1, 8, 512)),
        # A ragged chunk of a chunked prefill.
        ("mixtral_chunk_777", _case(MIXTRAL, "layer", 777, 2, 6, 512)),
        # The largest prefill batch: the benchmark's default workload.
        ("mixtral_8192", _case(MIXTRAL, "layer", 8192, 2, 6, 512)),
        # The paper's end/cloud pipeline over micro-batches.
        ("mixtral_pipelined_4096", _case(MIXTRAL, "pipelined", 4096, 2, 6, 512, micro=4)),
        # The paper's evaluation batch (4 x 256 tokens), 64 experts, 40% of them allowed.
        ("switch_1024_e64", _case(SWITCH, "layer", 1024, 1, 25, 128, E=64)),
        # The Switch preset (8 x 512 tokens).
        ("switch_4096", _case(SWITCH, "layer", 4096, 1, 12, 128, E=16)),
        # A decode step of a fine-grained model: many experts, few rows each.
        ("fine_decode_32", _case(FINE, "layer", 32, 8, 32, 256)),
        # Its full prefill batch.
        ("fine_16384", _case(FINE, "layer", 16384, 8, 32, 256)),
        # The fine-grained layer composed from the single entry points.
        ("fine_steps_2001", _case(FINE, "steps", 2001, 8, 32, 256)),
        # The tiny fp32 preset.
        ("fp32_tiny_256", _case(SWITCH, "layer", 256, 2, 4, 64, d=512, E=8, d_ff=1024, k=2, dtype="fp32")),
        # The paper's batch with the weights left in fp32.
        ("fp32_switch_1024", _case(SWITCH, "layer", 1024, 1, 12, 128, E=16, dtype="fp32")),
    ]
    return [dict(_merge(c), name=n) for n, c in named]


def _merge(c):
    return {key: c[key] for key in sorted(c)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "mixtral", "switch", "switch", "fine", "fine", "fp32", "fp32"])
    renorm = rng.choice([0, 0, 1])
    if kind == "decode":
        g = rng.choice([1, 2])
        c = _case(MIXTRAL, "layer", _log_int(rng, 1, 256), g, rng.choice([4, 6, 8]), rng.choice([128, 256, 512]),
                  renorm=renorm)
    elif kind == "mixtral":
        op = rng.choice(["layer", "layer", "layer", "pipelined", "steps"])
        c = _case(MIXTRAL, op, _log_int(rng, 257, 4096 if op == "steps" else 8192), 2, rng.choice([4, 6, 8]),
                  rng.choice([256, 512]), renorm=renorm, micro=rng.choice([2, 3, 4]) if op == "pipelined" else 0)
    elif kind == "switch":
        E = rng.choice([8, 16, 32, 64])
        op = rng.choice(["layer", "layer", "layer", "steps"])
        c = _case(SWITCH, op, _log_int(rng, 8, 8192), 1, max(2, int(E * rng.choice([0.4, 0.75, 1.0]))),
                  rng.choice([0, 128, 256]), E=E, renorm=renorm)
        c["k"] = rng.choice([1, 1, 2])
    elif kind == "fine":
        op = rng.choice(["layer", "layer", "layer", "pipelined", "steps"])
        c = _case(FINE, op, _log_int(rng, 1, 4096 if op == "steps" else 16384), 8, rng.choice([32, 64]), 256,
                  renorm=renorm, top_groups=rng.choice([0, 0, 4]),
                  micro=rng.choice([2, 4]) if op == "pipelined" else 0)
        c["zipf"] = rng.choice([0.0, 1.2])
    else:
        E = rng.choice([8, 16])
        op = rng.choice(["layer", "layer", "layer", "steps"])
        c = _case(SWITCH, op, _log_int(rng, 8, 2048), rng.choice([1, 2]), max(2, int(E * rng.choice([0.5, 0.75]))),
                  rng.choice([0, 64, 128]), E=E, renorm=renorm, dtype="fp32")
        c["d"], c["d_ff"] = rng.choice([(512, 1024), (512, 2048), (768, 3072)])
        c["k"] = rng.choice([1, 2])
        c["act"] = rng.choice(["gelu", "swiglu"])
    return _merge(c)


# ----------------------------------------------------------------- inputs
def _inputs(case, seed):
    """Tensors of one layer call on the GPU, from the seed alone."""
    T, d, E, f, K = case["T"], case["d"], case["E"], case["d_ff"], case["groups"]
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    h = torch.Generator()
    h.manual_seed(seed)

    def normal(*shape, fan_in=1, dtype=dt):
        return (torch.randn(*shape, generator=g, device="cuda") * (1.0 / math.sqrt(fan_in))).to(dtype)

    glu = case["act"] == "swiglu"
    t = {"X": normal(T, d), "W_local": normal(E, d, fan_in=d, dtype=torch.float32)}
    # Zipf popularity: the expert of rank j is biased by -s ln(j + 1).
    rank = torch.empty(E)
    rank[torch.randperm(E, generator=h)] = torch.arange(E, dtype=torch.float32)
    t["b_local"] = (-case["zipf"] * torch.log(rank + 1.0)).cuda()
    t["W_global"] = normal(K, d, fan_in=d, dtype=torch.float32) if K > 1 else None
    t["b_global"] = torch.zeros(K, device="cuda") if K > 1 else None
    # The experts allowed on this device, as many in each group.
    mask = torch.zeros(E, dtype=torch.uint8)
    for j in range(K):
        n = case["allowed"] * (j + 1) // K - case["allowed"] * j // K
        mask[j * (E // K) + torch.randperm(E // K, generator=h)[:n]] = 1
    t["mask"] = mask
    t["W1"] = normal(E, f, d, fan_in=d)
    t["W3"] = normal(E, f, d, fan_in=d) if glu else None
    t["W2"] = normal(E, d, f, fan_in=f)
    s = case["n_shared"]
    t["W1s"] = normal(s, f, d, fan_in=d) if s else None
    t["W3s"] = normal(s, f, d, fan_in=d) if s and glu else None
    t["W2s"] = normal(s, d, f, fan_in=f) if s else None
    t["V_enc"] = normal(case["r"], d, fan_in=d) if case["r"] else None
    t["V_dec"] = normal(d, case["r"], fan_in=case["r"]) if case["r"] else None
    return t


def prepare(case, seed):
    t = _inputs(case, seed)
    T, d, E, k, r = case["T"], case["d"], case["E"], case["k"], case["r"]
    dt = t["X"].dtype
    s = case["n_shared"]
    desc = C.make_desc(T=T, d=d, E=E, d_ff=case["d_ff"], k=k, n_groups=case["groups"],
                       act=C.SWIGLU if case["act"] == "swiglu" else C.GELU, dtype=C.F32 if dt == torch.float32 else C.BF16,
                       r=r, n_shared=s, d_ff_shared=case["d_ff"] if s else 0, renorm_topk=case["renorm"],
                       top_groups=case["top_groups"])

    def empty(*shape, dtype=dt):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    st = dict(op=case["op"], micro=case["micro"], desc=desc, t=t, mask=C.host_mask(t["mask"]),
              Y=empty(T, d), topk_idx=empty(T, k, dtype=torch.int32), topk_w=empty(T, k, dtype=torch.float32),
              counts=empty(E, dtype=torch.int32), Z=empty(T, r) if r else None)
    if st["op"] == "steps":
        st["ws_route"] = empty(max(16, C.ec2moe_route_workspace_size(desc)), dtype=torch.uint8)
        st["ws"] = empty(C.ec2moe_experts_workspace_size(desc), dtype=torch.uint8)
        st.update(offsets=empty(E + 1, dtype=torch.int32), perm=empty(T * k, dtype=torch.int32),
                  inv_perm=empty(T * k, dtype=torch.int32), X_hat=empty(T, d) if r else None, X_perm=empty(T * k, d),
                  slot=empty(T * k, d), shared=empty(s * T, d) if s else None)
    else:
        st["weights"] = C.make_weights(**{key: t[key] for key in ("W_local", "b_local", "W_global", "b_global", "W1", "W3",
                                                                  "W2", "W1s", "W3s", "W2s", "V_enc", "V_dec")})
        need = C.ec2moe_workspace_size(desc)
        if st["op"] == "pipelined":
            need = C.ec2moe_pipelined_workspace_size(desc, case["micro"])
            st["cloud"] = torch.cuda.Stream()
        st["ws"] = empty(max(16, need), dtype=torch.uint8)
    return st


# ----------------------------------------------------------------- one pass
def run(state):
    st, desc, t = state, state["desc"], state["t"]
    out = {key: st[key] for key in ("Y", "topk_idx", "topk_w", "counts", "Z") if st[key] is not None}
    ws = st["ws"]
    if st["op"] == "layer":
        C.ec2moe_layer_forward(desc, st["weights"], t["X"], st["mask"], st["Y"], st["topk_idx"], st["topk_w"],
                               st["counts"], st["Z"], ws, ws.numel())
        return out
    if st["op"] == "pipelined":
        C.ec2moe_layer_forward_pipelined(desc, st["weights"], t["X"], st["mask"], st["Y"], st["topk_idx"], st["topk_w"],
                                         st["counts"], st["Z"], ws, ws.numel(), st["micro"], None, st["cloud"])
        return out
    C.ec2moe_gate(desc, t["X"], t["W_local"], t["b_local"], t["W_global"], t["b_global"], st["mask"], st["topk_idx"],
                  st["topk_w"])
    x = t["X"]
    if st["Z"] is not None:
        C.ec2moe_lr_encode(desc, x, t["V_enc"], st["Z"])
        C.ec2moe_lr_decode(desc, st["Z"], t["V_dec"], st["X_hat"])
        x = st["X_hat"]
        out["X_hat"] = x
    C.ec2moe_route(desc, st["topk_idx"], st["counts"], st["offsets"], st["perm"], st["inv_perm"], x, x.shape[1],
                   st["X_perm"], st["ws_route"], st["ws_route"].numel())
    C.ec2moe_experts(desc, st["X_perm"], st["offsets"], t["W1"], t["W3"], t["W2"], st["topk_w"], st["perm"], st["slot"],
                     ws, ws.numel())
    if st["shared"] is not None:
        C.ec2moe_shared_experts(desc, x, t["W1s"], t["W3s"], t["W2s"], st["shared"], ws, ws.numel())
        out["shared"] = st["shared"]
    C.ec2moe_combine(desc, st["slot"], st["shared"], st["Y"])
    out.update({key: st[key] for key in ("offsets", "perm", "inv_perm", "X_perm", "slot")})
    return out


# ----------------------------------------------------------------- floors and tolerances
def work(case):
    T, d, E, f, k, r, s = (case[key] for key in ("T", "d", "E", "d_ff", "k", "r", "n_shared"))
    es = 4 if case["dtype"] == "fp32" else 2
    mats = 3 if case["act"] == "swiglu" else 2
    n = T * k
    a = case["allowed"]
    # experts expected to receive a row (popularity near uniform over the allowed ones)
    touched = a * (1.0 - (1.0 - k / a) ** T)
    flops = 2.0 * T * d * (E + (case["groups"] if case["groups"] > 1 else 0)) + 4.0 * T * d * r
    flops += 2.0 * mats * d * f * (n + s * T)
    byts = 2.0 * T * d * es + n * 8 + 4 * E + 4.0 * (E + case["groups"]) * d + T * r * es + 2.0 * d * r * es
    byts += (touched + s) * mats * d * f * es
    if case["op"] == "steps":
        # every step reads its inputs and writes its results: X_hat, X_perm, slot, shared
        byts += es * d * T * ((2 if r else 0) + 2 * k + (2 if s else 0) + k + s) + es * T * r + n * 16
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["dtype"] == "fp32":
        return {"rel": 5e-6, "max": 1e-4}
    # bf16 results of bf16 intermediates: another order of the fp32 sums moves
    # single roundings of Z, X_hat and the hidden rows by one unit (2^-8)
    return {"rel": 1e-2, "max": 1e-1}


# ----------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    t = _inputs(case, seed)
    T, d, E, k, K, s = (case[key] for key in ("T", "d", "E", "k", "groups", "n_shared"))
    D = torch.float64
    X = t["X"].to(D)
    neg = float("-inf")
    allowed = t["mask"].cuda().bool()
    local = (X @ t["W_local"].to(D).T + t["b_local"].to(D)).masked_fill(~allowed, neg).view(T, K, E // K)
    live = allowed.view(K, E // K).any(1)
    if K > 1:
        m = (X @ t["W_global"].to(D).T + t["b_global"].to(D)).masked_fill(~live, neg)
        if 0 < case["top_groups"] < int(live.sum()):
            keep = torch.zeros_like(m, dtype=torch.bool).scatter_(1, m.topk(case["top_groups"], 1).indices, True)
            m = m.masked_fill(~keep, neg)
        p_group = torch.softmax(m, 1)
    else:
        p_group = torch.ones(T, 1, dtype=D, device="cuda")
    p_local = torch.softmax(local, 2).nan_to_num(0.0)
    g = (p_group[:, :, None] * p_local).reshape(T, E)
    w, idx = torch.topk(g, k, dim=1)
    if case["renorm"]:
        w = w / w.sum(1, keepdim=True)
    out = {"topk_idx": None, "topk_w": w, "counts": None}
    x = X
    if case["r"]:
        z = X @ t["V_enc"].to(D).T
        x = z @ t["V_dec"].to(D).T
        out["Z"] = z

    def ffn(rows, w1, w3, w2):
        u = rows @ w1.to(D).T
        if w3 is not None:
            u = torch.nn.functional.silu(u) * (rows @ w3.to(D).T)
        else:
            u = torch.nn.functional.gelu(u)
        return u @ w2.to(D).T

    slot = torch.zeros(T * k, d, dtype=D, device="cuda")
    flat = idx.reshape(-1)
    for e in range(E):
        entries = (flat == e).nonzero().flatten()
        if entries.numel():
            y = ffn(x[entries // k], t["W1"][e], None if t["W3"] is None else t["W3"][e], t["W2"][e])
            slot[entries] = y * w.reshape(-1, 1)[entries]
    Y = slot.view(T, k, d).sum(1)
    shared = torch.empty(s * T, d, dtype=D, device="cuda")
    for j in range(s):
        shared[j * T:(j + 1) * T] = ffn(x, t["W1s"][j], None if t["W3s"] is None else t["W3s"][j], t["W2s"][j])
        Y = Y + shared[j * T:(j + 1) * T]
    out["Y"] = Y
    if case["op"] == "steps":
        out.update(offsets=None, perm=None, inv_perm=None, slot=slot)
        out["X_perm"] = x[torch.argsort(flat, stable=True) // k]
        if case["r"]:
            out["X_hat"] = x
        if s:
            out["shared"] = shared
    return out
