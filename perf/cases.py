"""What this library is used for, as measurable cases: the verify step of
speculative decoding and its parts, called as a serving loop calls them.

Every case goes through `paper_2606_31160_gb300.sd`. Two manners of use:

  * whole steps (verify, draft) run as a serving loop runs them: captured once
    per slot in a CUDA graph over the slot's buffers, replayed for every step.
    Each pass begins with the copy that brings the step's new rows and the
    committed lengths into the slot (in a model, the projections write them),
    so a pass is the same work on the same values however often it runs;
  * single calls (attention, acceptance, the attention budget) run eagerly on
    preallocated outputs and workspaces.

Sizes are those of the repository's workloads, tests and benchmark: 32 query /
8 KV heads x 128 (target), 16 / 4 x 128 (draft), 4 / 1 x 64 (tiny), prefixes of
up to 16384 keys, K up to 16, a vocabulary of 151936. `draw` spreads over the
same ranges, with odd batch sizes, group sizes, prefixes and vocabularies.
"""

import math

import numpy as np
import torch

from paper_2606_31160_gb300 import sd

DEV = "cuda"
SECTIONS = {128: (16, 24, 24), 64: (8, 12, 12)}
BASE = 1e6
TEMPERATURE = 0.6


def listed():
    return [
        # the smallest whole step: one head_dim-64 layer of 4 query heads over 256 keys,
        # fp32 logits over 4096 tokens; five short launches, all latency
        dict(name="tiny_step", kind="step", layers=1, B=1, Hq=4, Hkv=1, D=64, L=256, K=4, block=False,
             accept="greedy_f32", V=4096),
        # the draft's propose loop: 7 dependent single-row decode steps of one layer with
        # flat positions, then the rollback to what the target accepted
        dict(name="draft_propose", kind="draft", steps=7, Hq=16, Hkv=4, D=128, L=4096, committed=3),
        # the headline: one scene's verify pass of an 8B-class target (36 layers, 4096 keys,
        # K = 7), greedy acceptance over bf16 logits, rollback of every layer
        dict(name="target_step", kind="step", layers=36, B=1, Hq=32, Hkv=8, D=128, L=4096, K=7, block=False,
             accept="greedy_bf16", V=151936),
        # block-diffusion drafts: blocks of 16 tokens under the block mask, 68 packed rows a KV head
        dict(name="block_step", kind="step", layers=36, B=1, Hq=32, Hkv=8, D=128, L=4096, K=16, block=True,
             accept="greedy_bf16", V=151936),
        # sampled decoding of 8 scenes with ragged prefixes: rejection sampling over fp32 logits
        dict(name="stochastic_step", kind="step", layers=12, B=8, Hq=32, Hkv=8, D=128, L=4096, K=7, block=False,
             accept="sample", V=151936),
        # one scene with a long prefix (all cameras and history), short drafts
        dict(name="long_step", kind="step", layers=8, B=1, Hq=32, Hkv=8, D=128, L=16384, K=4, block=False,
             accept="greedy_bf16", V=151936),
        # batched serving: the attention alone over 32 ragged scenes, K = 8
        dict(name="attention_b32", kind="attention", B=32, Hq=32, Hkv=8, D=128, L=8192, K=8, block=False),
        # causal verification of 16-token drafts over 8 ragged scenes
        dict(name="attention_k16", kind="attention", B=8, Hq=32, Hkv=8, D=128, L=8192, K=16, block=False),
        # head_dim 64, seven query heads a KV head, an odd batch and capacity
        dict(name="attention_d64", kind="attention", B=5, Hq=28, Hkv=4, D=64, L=4099, K=5, block=False),
        # greedy acceptance of a batch
        dict(name="accept_greedy", kind="greedy", B=32, K=7, V=151936, dtype="bf16"),
        # rejection sampling of a batch
        dict(name="accept_sample", kind="sample", B=8, K=7, V=151936),
        # the attention-budget diagnostic of one target layer
        dict(name="attention_budget", kind="budget", B=1, Hq=32, Hkv=8, D=128, L=4096, K=7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_BYTES = 1.9e9  # of one drawn pass: below the largest listed cases


def draw(rng):
    kind = rng.choice(["step", "step", "draft", "attention", "attention", "greedy", "sample", "budget"])
    Hq, Hkv, D = rng.choice([(32, 8, 128), (32, 8, 128), (16, 4, 128), (28, 4, 128), (8, 8, 128), (4, 1, 64), (16, 4, 64)])
    V = rng.choice([4096, 32000, 50257, 128256, 151936, 151936])
    while True:
        if kind == "step":
            c = dict(kind="step", layers=rng.randint(1, 36), B=_log_int(rng, 1, 8), Hq=Hq, Hkv=Hkv, D=D,
                     L=_log_int(rng, 200, 16384), K=rng.randint(1, 16), block=rng.random() < 0.25,
                     accept=rng.choice(["greedy_bf16", "greedy_bf16", "greedy_f32", "sample"]), V=V)
        elif kind == "draft":
            c = dict(kind="draft", steps=rng.randint(1, 16), Hq=rng.choice([16, 32]), Hkv=rng.choice([4, 8]), D=128,
                     L=_log_int(rng, 200, 16384), committed=0)
            c["committed"] = rng.randint(0, c["steps"])
        elif kind == "attention":
            c = dict(kind="attention", B=_log_int(rng, 1, 32), Hq=Hq, Hkv=Hkv, D=D, L=_log_int(rng, 200, 16384),
                     K=rng.randint(0, 16), block=rng.random() < 0.2)
        elif kind == "greedy":
            c = dict(kind="greedy", B=_log_int(rng, 1, 32), K=rng.randint(0, 16), V=V, dtype=rng.choice(["bf16", "f32"]))
        elif kind == "sample":
            c = dict(kind="sample", B=_log_int(rng, 1, 16), K=rng.randint(1, 16), V=V)
        else:
            c = dict(kind="budget", B=_log_int(rng, 1, 8), Hq=Hq, Hkv=Hkv, D=D, L=_log_int(rng, 200, 16384),
                     K=rng.randint(0, 16))
        if c.get("Hq", 0) // c.get("Hkv", 1) * (c.get("K", 0) + 1) <= 128 and work(c)["bytes"] <= MAX_BYTES:
            return c


# ------------------------------------------------------------------ inputs

def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + 7919 * stream + 12345) & 0x7FFFFFFF)
    return g


def _prefixes(case):
    """Keys cached per scene: L for a single scene, U[0.75 L, L] for a batch (a
    property of the workload: every seed's batch is equally ragged)."""
    B, L = case.get("B", 1), case["L"]
    if B == 1:
        return np.array([L], dtype=np.int64)
    return np.random.RandomState(1000 + 31 * B + L).randint(-(-3 * L // 4), L + 1, size=B).astype(np.int64)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)


def _positions(prefix, R):
    """(t, h, w) of the new rows: text after 7/8 vision patches on 28 x 32 grids."""
    pos = np.empty((len(prefix), R, 3), dtype=np.int32)
    for b, n in enumerate(prefix):
        n_vis = 7 * int(n) // 8
        start = max((n_vis - 1) // 896, min(27, (n_vis - 1) // 32), min(31, n_vis - 1)) + 1 if n_vis else 0
        pos[b] = (np.arange(R) + start + int(n) - n_vis)[:, None]
    return torch.from_numpy(pos).to(DEV)


def _views(buf, shapes):
    """Views of consecutive parts of a byte buffer: [(dtype, shape), ...]."""
    out, at = [], 0
    for dtype, shape in shapes:
        n = math.prod(shape) * torch.empty(0, dtype=dtype).element_size()
        out.append(buf[at:at + n].view(dtype).view(shape))
        at += -(-n // 16) * 16
    return out


def _bytes_for(shapes):
    return sum(-(-math.prod(s) * torch.empty(0, dtype=d).element_size() // 16) * 16 for d, s in shapes)


def _greedy_inputs(case, g, seed, dtype):
    """Logits N(0, 2) with a planted maximum 8 sigma up; drafts that match a random
    number of leading rows."""
    B, K, V = case["B"], case["K"], case["V"]
    z = torch.randn((B, K + 1, V), generator=g, device=DEV, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32) * 2.0
    target = torch.randint(0, V, (B, K + 1, 1), generator=g, device=DEV)
    z.scatter_(2, target, 16.0)
    ell = torch.randint(0, K + 1, (B, 1), generator=g, device=DEV)
    j = torch.arange(K, device=DEV)[None]
    t = target[:, :K, 0]
    draft = torch.where(j < ell, t, (t + 1) % V).to(torch.int32).contiguous()
    return z, draft


def _sample_inputs(case, g):
    """Target logits N(0, 3), draft logits = target + N(0, 0.5), drafts drawn from the
    draft distribution (Gumbel-max), uniforms of 24 bits."""
    B, K, V = case["B"], case["K"], case["V"]
    z_t = torch.randn((B, K + 1, V), generator=g, device=DEV) * 3.0
    z_d = z_t[:, :K] + torch.randn((B, K, V), generator=g, device=DEV) * 0.5
    e = torch.empty_like(z_d).exponential_(generator=g).clamp_min_(1e-30)
    draft = (z_d / TEMPERATURE - e.log()).argmax(-1).to(torch.int32)
    u = torch.randint(0, 1 << 24, (B, K + 1), generator=g, device=DEV).float() * 2.0 ** -24
    return z_t, z_d.contiguous(), draft, u


def _empty_i32(*shape):
    return torch.empty(shape, dtype=torch.int32, device=DEV)


def _accept_state(case, g, seed):
    accept = case["accept"] if case["kind"] == "step" else case["kind"]
    B, K, V = case["B"], case["K"], case["V"]
    s = dict(n_emit=_empty_i32(B), tokens=_empty_i32(B, K + 1))
    if accept == "sample":
        s["z_t"], s["z_d"], s["draft"], s["u"] = _sample_inputs(case, g)
        s["accept_ws"] = sd.workspace(sd.sample_workspace_bytes(B, K, V))
    else:
        dtype = case.get("dtype") or ("bf16" if accept == "greedy_bf16" else "f32")
        s["logits"], s["draft"] = _greedy_inputs(case, g, seed, dtype)
        s["argmax"] = _empty_i32(B, K + 1)
        s["accept_ws"] = sd.workspace(sd.greedy_workspace_bytes(B, K, V))
    return s


def _accept(s):
    if "z_t" in s:
        sd.accept_sample(s["z_t"], s["z_d"], s["draft"], s["u"], TEMPERATURE, ws=s["accept_ws"], n_emit=s["n_emit"],
                         tokens=s["tokens"])
        return {"n_emit": s["n_emit"], "tokens": s["tokens"]}
    sd.accept_greedy(s["logits"], s["draft"], ws=s["accept_ws"], n_emit=s["n_emit"], tokens=s["tokens"], argmax=s["argmax"])
    return {"n_emit": s["n_emit"], "tokens": s["tokens"], "argmax": s["argmax"]}


def _step_rows(case):
    """Buffers that a step rewrites: rotated query and key rows of every layer, and the lengths."""
    n, B, R = case["layers"], case["B"], case["K"] + 1
    return [(torch.bfloat16, (n, B, R, case["Hq"], case["D"])), (torch.bfloat16, (n, B, R, case["Hkv"], case["D"])),
            (torch.int32, (n, B))]


def _draft_rows(case):
    n = case["steps"]
    return [(torch.bfloat16, (n, 1, 1, case["Hq"], case["D"])), (torch.bfloat16, (n, 1, 1, case["Hkv"], case["D"])),
            (torch.int32, (1,))]


def _step_inputs(case, seed):
    """Everything a step reads, before any call: raw rows, caches, positions, logits."""
    g = _gen(seed)
    n, B, R, Hkv, D = case["layers"], case["B"], case["K"] + 1, case["Hkv"], case["D"]
    prefix = _prefixes(case)
    cap = case["L"] + 17
    shapes = _step_rows(case)
    raw = torch.zeros(_bytes_for(shapes), dtype=torch.uint8, device=DEV)
    q, k, lens = _views(raw, shapes)
    q.copy_(_normal(g, *q.shape))
    k.copy_(_normal(g, *k.shape))
    lens.copy_(torch.from_numpy(prefix.astype(np.int32))[None].expand(n, B))
    s = dict(raw=raw, v_new=_normal(g, n, B, R, Hkv, D), pos=_positions(prefix, R), k_cache=_normal(g, n, B, Hkv, cap, D),
             v_cache=_normal(g, n, B, Hkv, cap, D))
    s.update(_accept_state(case, g, seed))
    return s


def _draft_inputs(case, seed):
    g = _gen(seed)
    n, Hkv, D, L = case["steps"], case["Hkv"], case["D"], case["L"]
    shapes = _draft_rows(case)
    raw = torch.zeros(_bytes_for(shapes), dtype=torch.uint8, device=DEV)
    q, k, lens = _views(raw, shapes)
    q.copy_(_normal(g, *q.shape))
    k.copy_(_normal(g, *k.shape))
    lens.fill_(L)
    pos = (L + torch.arange(n, dtype=torch.int32, device=DEV))[:, None, None, None].expand(n, 1, 1, 3).contiguous()
    return dict(raw=raw, v_new=_normal(g, n, 1, 1, Hkv, D), pos=pos, k_cache=_normal(g, 1, Hkv, L + 17, D),
                v_cache=_normal(g, 1, Hkv, L + 17, D),
                committed=torch.full((1,), case["committed"], dtype=torch.int32, device=DEV))


def _attention_inputs(case, seed):
    g = _gen(seed)
    B, R, Hkv, D, cap = case["B"], case["K"] + 1, case["Hkv"], case["D"], case["L"] + 17
    prefix = _prefixes(case)
    return dict(q=_normal(g, B, R, case["Hq"], D), k_cache=_normal(g, B, Hkv, cap, D), v_cache=_normal(g, B, Hkv, cap, D),
                lens=torch.from_numpy((prefix + R).astype(np.int32)).to(DEV),
                n_visual=torch.from_numpy((7 * prefix // 8).astype(np.int32)).to(DEV))


# ---------------------------------------------------------------- the passes

def _step_body(s):
    s["work"].copy_(s["raw"])
    for i, cache in enumerate(s["caches"]):
        sd.verify_layer(s["q"][i], s["k"][i], s["v_new"][i], s["pos"], s["sections"], cache, 0, BASE, out=s["out"][i],
                        early=i > 0, block=s["block"])
    res = _accept(s)
    sd.kv_rollback(s["lens"], s["n_emit"], s["R"])
    return {"out": s["out"], "q": s["q"], "k": s["k"], "lens": s["lens"], "k_cache": s["k_cache"], "v_cache": s["v_cache"], **res}


def _draft_body(s):
    s["work"].copy_(s["raw"])
    for i in range(s["steps"]):
        sd.verify_layer(s["q"][i], s["k"][i], s["v_new"][i], s["pos"][i], s["sections"], s["cache"], 0, BASE, out=s["out"][i])
    sd.kv_rollback(s["lens"], s["committed"], s["steps"])
    return {"out": s["out"], "q": s["q"], "k": s["k"], "lens": s["lens"], "k_cache": s["k_cache"], "v_cache": s["v_cache"]}


def _capture(s, body):
    """One eager pass (kernel attributes, workspaces), then the slot's graph."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        body(s)
    torch.cuda.current_stream().wait_stream(side)
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["graph"]):
        s["result"] = body(s)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        s = _step_inputs(case, seed)
        s["work"] = s["raw"].clone()
        s["q"], s["k"], s["lens"] = _views(s["work"], _step_rows(case))
        s["out"] = torch.zeros_like(s["q"])
        s["caches"] = [sd.KVCache(s["k_cache"][i], s["v_cache"][i], s["lens"][i]) for i in range(case["layers"])]
        s.update(sections=SECTIONS[case["D"]], block=case["block"], R=case["K"] + 1)
        return _capture(s, _step_body)
    if kind == "draft":
        s = _draft_inputs(case, seed)
        s["work"] = s["raw"].clone()
        s["q"], s["k"], s["lens"] = _views(s["work"], _draft_rows(case))
        s["out"] = torch.zeros_like(s["q"])
        s["cache"] = sd.KVCache(s["k_cache"], s["v_cache"], s["lens"])
        s.update(sections=SECTIONS[case["D"]], steps=case["steps"])
        return _capture(s, _draft_body)
    if kind in ("attention", "budget"):
        s = _attention_inputs(case, seed)
        B, R, Hq, D = s["q"].shape
        s["cache"] = sd.KVCache(s["k_cache"], s["v_cache"], s["lens"])
        if kind == "attention":
            s["out"] = torch.zeros_like(s["q"])
            s["ws"] = sd.workspace(sd.attention_workspace_bytes(B, R, Hq, case["Hkv"], D, s["cache"].shape[2]))
            s["block"] = case["block"]
        else:
            s["mass"] = torch.zeros((B, R, Hq, 3), dtype=torch.float32, device=DEV)
            s["entropy"] = torch.zeros((B, R, Hq), dtype=torch.float32, device=DEV)
        s["kind"] = kind
        return s
    s = _accept_state(case, _gen(seed), seed)
    s["kind"] = kind
    return s


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["result"]
    if state["kind"] == "attention":
        return sd.verify_attention(state["q"], state["cache"], out=state["out"], ws=state["ws"], block=state["block"])
    if state["kind"] == "budget":
        sd.attention_budget(state["q"], state["cache"], state["n_visual"], mass=state["mass"], entropy=state["entropy"])
        return {"mass": state["mass"], "entropy": state["entropy"]}
    return _accept(state)


# ------------------------------------------------------------- work, tolerance

def _accept_bytes(case):
    accept = case["accept"] if case["kind"] == "step" else case["kind"]
    B, K, V = case["B"], case["K"], case["V"]
    if accept == "sample":  # every target and draft logit once
        return B * (2 * K + 1) * V * 4
    elem = 2 if accept == "greedy_bf16" or case.get("dtype") == "bf16" else 4
    return B * (K + 1) * V * elem


def work(case):
    kind = case["kind"]
    if kind in ("greedy", "sample"):
        b = _accept_bytes(case)
        return {"bytes": b, "flops": b / 2}
    Hq, Hkv, D = case["Hq"], case["Hkv"], case["D"]
    if kind == "draft":
        n, L = case["steps"], case["L"]
        keys = n * L + n * (n - 1) // 2
        # raw and rotated q and k rows, v, the two appended rows, out
        rows = n * (3 * Hq + 5 * Hkv) * D * 2
        return {"bytes": keys * Hkv * D * 4 + rows, "flops": 4 * (keys + n) * Hq * D}
    prefix, B, R = _prefixes(case), case["B"], case["K"] + 1
    keys = int(prefix.sum())
    flops = 4 * R * keys * Hq * D
    if kind == "step":
        rows = B * R * (3 * Hq + 5 * Hkv) * D * 2
        return {"bytes": case["layers"] * (keys * Hkv * D * 4 + rows) + _accept_bytes(case), "flops": case["layers"] * flops}
    if kind == "attention":
        return {"bytes": (keys + B * R) * Hkv * D * 4 + 2 * B * R * Hq * D * 2, "flops": flops}
    # the budget reads keys only
    return {"bytes": (keys + B * R) * Hkv * D * 2 + B * R * Hq * (D * 2 + 16), "flops": flops / 2}


def tolerance(case):
    kind = case["kind"]
    if kind == "greedy":
        return "exact"  # token ids
    if kind == "sample":
        # token ids; fp32 sums in another order move a draw at a cumulative step
        return {"rel": 0.0, "max": 0.0, "differ": 0.01}
    if kind == "budget":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}  # fp32 sums of bf16 products
    # bf16 outputs from bf16 weights and fp32 sums (error against 64 bits 2e-3 to 3e-3)
    return {"rel": 1e-2, "max": 6e-2, "differ": 0.01}


# ---------------------------------------------------------------- in 64 bits

def _rotate(x, pos, D):
    """x [..., D] (adjacent pairs) by theta_d * pos[axis(d)]; pos [..., 3], broadcast over heads."""
    s_t, s_h, s_w = SECTIONS[D]
    axis = torch.tensor([0] * s_t + [1] * s_h + [2] * s_w, device=DEV)
    theta = BASE ** (-2.0 * torch.arange(D // 2, device=DEV, dtype=torch.float64) / D)
    phi = pos.double()[..., axis] * theta
    c, s = phi.cos(), phi.sin()
    a, b = x.double()[..., 0::2], x.double()[..., 1::2]
    return torch.stack([a * c - b * s, a * s + b * c], -1).flatten(-2)


def _attend(q, k, v, n, block, n_visual=None):
    """q [R, Hq, D], k / v [Hkv, cap, D], n valid keys (the last R of them new)."""
    R, Hq, D = q.shape
    Hkv = k.shape[0]
    G = Hq // Hkv
    qq = q.double().reshape(R, Hkv, G, D).permute(1, 0, 2, 3).reshape(Hkv, R * G, D)
    y = qq @ k[:, :n].double().transpose(1, 2) / math.sqrt(D)
    row = torch.arange(R, device=DEV).repeat_interleave(G)
    key = torch.arange(n, device=DEV)
    if not block:
        y.masked_fill_((key[None] > n - R + row[:, None])[None], -math.inf)
    if n_visual is None:
        o = torch.softmax(y, -1) @ v[:, :n].double()
        return o.reshape(Hkv, R, G, D).permute(1, 0, 2, 3).reshape(R, Hq, D)
    p = torch.softmax(y, -1)
    L = n - R
    mass = torch.stack([p[..., :n_visual].sum(-1), p[..., n_visual:L].sum(-1), p[..., L:].sum(-1)], -1)
    rest = torch.log_softmax(y[..., n_visual:], -1)
    h = -(rest.exp() * rest.masked_fill(rest == -math.inf, 0.0)).sum(-1)
    count = (L - n_visual + row + 1).double()
    ent = torch.where(count > 1, h / count.clamp_min(2).log(), torch.zeros_like(h))
    back = lambda t: t.reshape(Hkv, R, G, -1).permute(1, 0, 2, 3).reshape(R, Hq, -1)  # noqa: E731
    return back(mass), back(ent)[..., 0]


def _accept_exact(s):
    out = {}
    draft = s["draft"].long()
    if "z_t" in s:
        p = torch.softmax(s["z_t"].double() / TEMPERATURE, -1)
        q = torch.softmax(s["z_d"].double() / TEMPERATURE, -1)
        B, K = draft.shape
        ok = s["u"][:, :K].double() * q.gather(2, draft[..., None])[..., 0] <= p[:, :K].gather(2, draft[..., None])[..., 0]
        ell = ok.long().cumprod(1).sum(1)
        last = torch.empty(B, dtype=torch.long, device=DEV)
        for b in range(B):
            n = int(ell[b])
            w = (p[b, n] - q[b, n]).clamp_min(0) if n < K else p[b, K]
            c = w.cumsum(0)
            last[b] = (c <= s["u"][b, K].double() * c[-1]).sum().clamp_max(w.numel() - 1)
    else:
        star = s["logits"].float().argmax(-1)
        B, K = draft.shape
        ell = (draft == star[:, :K]).long().cumprod(1).sum(1)
        last = star.gather(1, ell[:, None])[:, 0]
        out["argmax"] = star.to(torch.int32)
    j = torch.arange(K + 1, device=DEV)[None]
    pad = torch.cat([draft, draft.new_zeros(B, 1)], 1)
    tokens = torch.where(j < ell[:, None], pad, torch.where(j == ell[:, None], last[:, None], torch.full_like(pad, -1)))
    out.update(n_emit=(ell + 1).to(torch.int32), tokens=tokens.to(torch.int32))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        s = _step_inputs(case, seed)
        q, k, lens = _views(s["raw"], _step_rows(case))
        R, D, prefix = case["K"] + 1, case["D"], _prefixes(case)
        qr, kr = _rotate(q, s["pos"][None, :, :, None], D), _rotate(k, s["pos"][None, :, :, None], D)
        # the attention reads the rotated rows as they are stored
        qb, kb = qr.to(torch.bfloat16), kr.to(torch.bfloat16)
        kc, vc = s["k_cache"].double(), s["v_cache"].double()
        out = torch.empty_like(qr)
        for i in range(case["layers"]):
            for b in range(case["B"]):
                n = int(prefix[b])
                kc[i, b, :, n:n + R] = kr[i, b].transpose(0, 1)
                vc[i, b, :, n:n + R] = s["v_new"][i, b].double().transpose(0, 1)
                kk = s["k_cache"][i, b, :, :n + R].double()
                kk[:, n:] = kb[i, b].double().transpose(0, 1)
                out[i, b] = _attend(qb[i, b], kk, vc[i, b], n + R, case["block"])
        res = _accept_exact(s)
        return {"out": out, "q": qr, "k": kr, "lens": lens + res["n_emit"][None], "k_cache": kc, "v_cache": vc, **res}
    if kind == "draft":
        s = _draft_inputs(case, seed)
        q, k, lens = _views(s["raw"], _draft_rows(case))
        D, n = case["D"], case["L"]
        pos = s["pos"][:, :, :, None]
        qr, kr = _rotate(q, pos, D), _rotate(k, pos, D)
        kc, vc, kk = s["k_cache"].double(), s["v_cache"].double(), s["k_cache"].double()
        out = torch.empty_like(qr)
        for i in range(case["steps"]):
            kc[0, :, n + i] = kr[i, 0, 0]
            kk[0, :, n + i] = kr[i, 0, 0].to(torch.bfloat16).double()
            vc[0, :, n + i] = s["v_new"][i, 0, 0].double()
            out[i, 0] = _attend(qr[i, 0].to(torch.bfloat16), kk[0], vc[0], n + i + 1, False)
        return {"out": out, "q": qr, "k": kr, "lens": lens + case["committed"], "k_cache": kc, "v_cache": vc}
    if kind in ("attention", "budget"):
        s = _attention_inputs(case, seed)
        R, prefix = case["K"] + 1, _prefixes(case)
        got = [_attend(s["q"][b], s["k_cache"][b], s["v_cache"][b], int(prefix[b]) + R, case.get("block", False),
                       7 * int(prefix[b]) // 8 if kind == "budget" else None) for b in range(case["B"])]
        if kind == "attention":
            return torch.stack(got)
        return {"mass": torch.stack([m for m, _ in got]), "entropy": torch.stack([e for _, e in got])}
    return _accept_exact(_accept_state(case, _gen(seed), seed))
