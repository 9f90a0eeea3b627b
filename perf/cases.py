"""The work that a program built on this framework has it do, as cases to time.

A block-diffusion language model calls the MoE layer once per layer and
denoising forward, for the tokens that forward processes: one active block of
32 tokens where earlier keys and values are cached, whole sequences where they
are not, batches of sequences in serving.  The cases span that range: the
tiny fp32 layer, one block, short and ragged batches, the layers of both
model shapes, the largest token count of the token sweep, layers of the
benchmark's stack in a row, and the steps that are called by themselves (the routing
without workspace, the refinement state of a denoising loop).

A case's "call" is the public entry point:
  step     api.MoELayer.step: counts from the refinement state, then the layer
  forward  api.MoELayer.forward: the layer at counts that the caller holds
  stack    api.MoEStack.forward: one denoising forward through all layers
  route    reflex_route_noalloc: scores, TopK and weights, no workspace
  loop     api.allocate and api.update_state: a denoising loop's own work
With "graph" the call is captured once and replayed, as a serving loop does.
Everything is synthetic and seeded; weights and hidden states have the
benchmark's distributions (hidden N(0, 1), weights N(0, 0.02), or
1 / sqrt(fan_in) in fp32).
"""
import math

import numpy as np
import torch

from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import api

# layer shapes: the two model shapes of the benchmark and its tiny fp32 layer
MOE = dict(dtype="bf16", d=2048, E=64, inter=1024, shared=0)
MINI = dict(dtype="bf16", d=2048, E=256, inter=512, shared=512)
TINY = dict(dtype="f32", d=256, E=8, inter=128, shared=0)
# count bounds and allocation offsets that go with them
K12 = dict(k_min=2, k_base=8, k_max=12, delta_role=4, delta_cur=2)
K4 = dict(k_min=1, k_base=2, k_max=4, delta_role=1, delta_cur=1)
THETA, V_REF, TAU, Q, W_CF = 0.9, 0.01, 0.05, 0.25, 0.30


def seqs(n_seq, prompt, gen, block=32, ragged=0):
    """Sequences of a batch; sequence s has (37 s) mod (ragged + 1) more prompt tokens."""
    return dict(n_seq=n_seq, prompt=prompt, gen=gen, block=block, ragged=ragged)


def listed():
    return [
        # the smallest call: 96 tokens of the fp32 layer, all launch latency
        dict(name="tiny_f32_96", call="step", **TINY, **K4, **seqs(1, 32, 64)),
        # fp32 storage at a working size (checking a model in full precision)
        dict(name="f32_1024", call="step", dtype="f32", d=1024, E=16, inter=512, shared=0, **K4,
             **seqs(4, 128, 128)),
        # one active block with cached keys and values, captured by a serving loop
        dict(name="moe_block32_graph", call="step", graph=True, **MOE, **K12, **seqs(1, 0, 32)),
        # the shortest batch of the token sweep, at the most uneven counts
        dict(name="mini_256_skew", call="forward", tokens=256, skew=1.0, **MINI, **K12),
        # one sequence of 512 + 512 tokens, no cache
        dict(name="moe_1024", call="step", **MOE, **K12, **seqs(1, 512, 512)),
        # a few sequences of unequal, odd lengths
        dict(name="moe_ragged_3k", call="step", **MOE, **K12, **seqs(7, 211, 233, ragged=40)),
        # the serving batch of the second model shape, with its shared expert
        dict(name="mini_8192", call="step", **MINI, **K12, **seqs(8, 256, 768)),
        # counts from the router's own mass (Top-p), bounds [1, 12]
        dict(name="mini_topp_2048", call="step", rule="top_p", threshold=0.25, **MINI,
             **dict(K12, k_min=1), **seqs(2, 256, 768)),
        # the largest token count of the sweep, fixed top-8
        dict(name="mini_65536", call="forward", tokens=65536, skew=0.0, **MINI, **K12),
        # routing alone, in a plugin that has no workspace
        dict(name="route_4096", call="route", tokens=4096, skew=0.5, **MOE, **K12),
        # allocation and state update of a denoising loop, ragged batch
        dict(name="loop_32seq", call="loop", **K12, **seqs(32, 500, 500, ragged=60)),
        # four of the benchmark's 16 layers at its 32 x 1024 tokens, counts once per forward
        dict(name="moe_stack4_32768", call="stack", layers=4, **MOE, **K12, **seqs(32, 512, 512)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_seqs(rng, most):
    """A batch of sequences of at most `most` tokens, odd lengths among them."""
    block = rng.choice([16, 32, 32, 32, 48])
    total = _log(rng, 32, most)
    if total < 96 or rng.random() < 0.15:  # active blocks alone
        return seqs(max(1, total // block), 0, block, block)
    n = min(_log(rng, 1, 32), max(1, total // 64))
    each = total // n
    gen = max(block, int(each * rng.uniform(0.3, 0.8)))
    prompt = max(1, each - gen)
    return seqs(n, prompt, gen, block, rng.choice([0, 0, min(prompt, 40)]) if n > 1 else 0)


def draw(rng):
    what = rng.choice(["moe", "moe", "mini", "mini", "mini_fwd", "other", "other", "f32", "rule",
                       "route", "loop", "stack"])
    if what == "moe":
        c = dict(call="step", **MOE, **K12, **_draw_seqs(rng, 32000))
        if rng.random() < 0.25:
            c["graph"] = True
        return c
    if what == "mini":
        return dict(call="step", **MINI, **K12, **_draw_seqs(rng, 32000))
    if what == "mini_fwd":
        return dict(call="forward", tokens=_log(rng, 1, 60000), skew=round(rng.random(), 2), **MINI,
                    **K12)
    if what == "other":  # other widths and expert counts that the layer takes
        shape = dict(dtype="bf16", d=rng.choice([1024, 2048, 4096]),
                     E=rng.choice([16, 32, 60, 96, 128, 160]),
                     inter=rng.choice([512, 768, 1024]), shared=rng.choice([0, 0, 512]))
        return dict(call="forward", tokens=_log(rng, 8, 16000), skew=round(rng.random(), 2), **shape,
                    **K12)
    if what == "f32":
        shape = dict(dtype="f32", d=rng.choice([256, 512, 1024]), E=rng.choice([8, 16, 32]),
                     inter=rng.choice([128, 256, 512]), shared=0)
        return dict(call="step", **shape, **K4, **_draw_seqs(rng, 2048))
    if what == "rule":
        top_p = rng.random() < 0.5
        return dict(call="step", rule="top_p" if top_p else "expert_threshold",
                    threshold=rng.choice([0.15, 0.25, 0.325] if top_p else [0.019, 0.027]),
                    **rng.choice([MOE, MINI]), **dict(K12, k_min=1), **_draw_seqs(rng, 8000))
    if what == "route":
        shape = rng.choice([MOE, MINI])
        most = B.REFLEX_NOALLOC_MAX_SCORES // shape["E"]
        return dict(call="route", tokens=_log(rng, 1, most), skew=round(rng.random(), 2), **shape,
                    **K12)
    if what == "loop":
        return dict(call="loop", **K12, **_draw_seqs(rng, 64000))
    return dict(call="stack", layers=rng.randint(2, 4), **MOE, **K12, **_draw_seqs(rng, 16000))


# ---- inputs -----------------------------------------------------------------
def _lengths(c):
    prompts = [c["prompt"] + (37 * s) % (c["ragged"] + 1) for s in range(c["n_seq"])]
    return prompts, c["gen"]


def _tokens(c):
    if "tokens" in c:
        return c["tokens"]
    prompts, gen = _lengths(c)
    return sum(prompts) + gen * len(prompts)


def _state(c, seed):
    """Refinement state of one forward: blocks before the active one resolved,
    the active one partly, later ones masked; confidences Beta(2, 2) on masked
    and Beta(5, 1) on resolved positions, a few positions with a short history."""
    g = np.random.default_rng([seed, 1])
    prompts, gen = _lengths(c)
    n_blocks = -(-gen // c["block"])
    bid, off, active, masked = [], [0], [], []
    for p in prompts:
        a = int(g.integers(1, n_blocks + 1))
        b = np.concatenate([np.zeros(p, np.int32), 1 + np.arange(gen, dtype=np.int32) // c["block"]])
        frac = g.uniform(0.1, 1.0)
        m = (b > a) | ((b == a) & (g.random(b.size) < frac))
        bid.append(b)
        masked.append(m)
        active.append(a)
        off.append(off[-1] + b.size)
    bid, masked = np.concatenate(bid), np.concatenate(masked)
    n = bid.size
    conf1 = np.where(masked, g.beta(2.0, 2.0, n), g.beta(5.0, 1.0, n)).astype(np.float32)
    conf2 = np.clip(conf1 - g.uniform(-0.2, 0.2, n), 0, 1).astype(np.float32)
    hist = g.choice(np.array([0, 1, 2], np.uint8), n, p=[0.03, 0.07, 0.9])
    return dict(block_id=bid, seq_offsets=np.array(off, np.int32),
                active_block=np.array(active, np.int32), masked=masked.astype(np.uint8),
                conf1=conf1, conf2=conf2, hist_len=hist)


def _given_counts(c, seed):
    """Counts that the caller holds: 0.7 skew of the tokens at k_min, 0.3 skew at k_max, the
    others at k_base."""
    u = np.random.default_rng([seed, 2]).random(c["tokens"])
    s, most = c["skew"], min(c["k_max"], c["E"])
    k = np.where(u < 0.7 * s, c["k_min"], np.where(u < s, c["k_max"], c["k_base"]))
    return np.minimum(k, most).astype(np.int32)


def _normal(g, shape, std, dtype):
    t = torch.empty(shape, dtype=dtype, device="cuda")
    return t.normal_(0.0, std, generator=g)


def _weights(c, g):
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    d, e, i, s = c["d"], c["E"], c["inter"], c["shared"]
    std = (lambda fan: 0.02) if c["dtype"] == "bf16" else (lambda fan: 1 / math.sqrt(fan))
    w = dict(w_router=_normal(g, (e, d), std(d), dt), w_gate_up=_normal(g, (e, 2 * i, d), std(d), dt),
             w_down=_normal(g, (e, d, i), std(i), dt))
    if s:
        w["shared_gate_up"] = _normal(g, (2 * s, d), std(d), dt)
        w["shared_down"] = _normal(g, (d, s), std(s), dt)
    return w


def _inputs(c, seed):
    """Host state or counts, and hidden states and weights on the GPU."""
    inp = {}
    if "tokens" in c:
        inp["k"] = _given_counts(c, seed)
    else:
        inp["state"] = _state(c, seed)
    if c["call"] != "loop":
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
        inp["hidden"] = _normal(g, (_tokens(c), c["d"]), 1.0, dt)
        inp["layers"] = [_weights(c, g) for _ in range(c.get("layers", 1))]
    return inp


def _params(c):
    p = dict(k_min=c["k_min"], k_base=c["k_base"], k_max=c["k_max"], delta_role=c["delta_role"],
             delta_cur=c["delta_cur"], q=Q, theta=THETA, w_cf=W_CF, v_ref=V_REF, tau=TAU)
    if "rule" in c:
        p["count_rule"] = dict(top_p=B.REFLEX_RULE_TOP_P,
                               expert_threshold=B.REFLEX_RULE_EXPERT_THRESHOLD)[c["rule"]]
        p["rule_threshold"] = c["threshold"]
    return B.make_params(**p)


def prepare(case, seed):
    c, inp = case, _inputs(case, seed)
    T = _tokens(c)
    i32 = dict(dtype=torch.int32, device="cuda")
    s = dict(case=c, params=_params(c), status=torch.zeros(1, **i32), k=torch.zeros(T, **i32),
             k_sum=torch.zeros(1, dtype=torch.int64, device="cuda"))
    if "state" in inp:
        s["state"] = api.state_to_device(inp["state"])
    else:
        s["k"] = torch.from_numpy(inp["k"]).cuda()
    if c["call"] == "loop":
        g = np.random.default_rng([seed, 3])
        # confidences of this forward: some active positions reach the threshold
        s["conf"] = torch.from_numpy(g.beta(4.0, 1.2, T).astype(np.float32)).cuda()
        s["blocks"] = torch.full((c["n_seq"],), -(-c["gen"] // c["block"]), **i32)
        s["committed"] = torch.zeros(c["n_seq"], **i32)
        s["work"] = {n: t.clone() for n, t in s["state"].items()}
        return s
    s["hidden"] = inp["hidden"]
    if c["call"] == "route":
        s["w_router"] = inp["layers"][0]["w_router"]
        s["ids"] = torch.empty((T, c["k_max"]), **i32)
        s["alpha"] = torch.empty((T, c["k_max"]), dtype=torch.float32, device="cuda")
        return s
    s["out"] = torch.empty_like(s["hidden"])
    shape = dict(dtype=c["dtype"], d=c["d"], E=c["E"], inter=c["inter"], shared_inter=c["shared"],
                 k_max=c["k_max"], max_tokens=T)
    if c["call"] == "stack":
        s["stack"] = api.MoEStack(inp["layers"], **shape)
    else:
        s["layer"] = api.MoELayer(inp["layers"][0], **shape)
    if c.get("graph"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _call(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _call(s)
    return s


# ---- one pass ---------------------------------------------------------------
def _call(s):
    c = s["case"]
    if c["call"] == "step":
        s["layer"].step(s["state"], s["params"], s["hidden"], out=s["out"], k_out=s["k"],
                        k_sum=s["k_sum"], status=s["status"])
    elif c["call"] == "forward":
        s["layer"].forward(s["hidden"], s["k"], s["out"])
    else:
        s["stack"].forward(s["state"], s["params"], s["hidden"], s["out"], s["k"], s["k_sum"],
                           s["status"])


def run(state):
    s = state
    c = s["case"]
    if c["call"] == "route":
        B.reflex_route_noalloc(B.REFLEX_DTYPE_BF16, s["hidden"], s["w_router"], s["k"],
                               s["hidden"].shape[0], c["d"], c["E"], c["k_max"],
                               B.REFLEX_FLAG_RENORM_TOPK, s["ids"], s["alpha"], s["status"])
        return dict(ids=s["ids"], alpha=s["alpha"])
    if c["call"] == "loop":
        w = s["work"]
        for n in ("masked", "conf1", "conf2", "hist_len", "active_block"):
            w[n].copy_(s["state"][n])  # this forward's state
        api.allocate(w, s["params"], k_out=s["k"], k_sum=s["k_sum"], status=s["status"])
        api.update_state(w, s["conf"], s["blocks"], THETA, committed=s["committed"])
        return dict(k=s["k"], k_sum=s["k_sum"], committed=s["committed"], masked=w["masked"],
                    conf1=w["conf1"], conf2=w["conf2"], hist=w["hist_len"], active=w["active_block"])
    if "graph" in s:
        s["graph"].replay()
    else:
        _call(s)
    if c["call"] == "forward":
        return dict(out=s["out"])
    return dict(out=s["out"], k=s["k"], k_sum=s["k_sum"])


# ---- what a pass cannot do without ------------------------------------------
def work(case):
    c = case
    T = _tokens(c)
    if c["call"] == "loop":
        # per token: two confidences, history, mask, block in; count out; the
        # state update reads the new confidence and writes the same arrays
        return dict(bytes=T * (14 + 4 + 4 + 10), flops=0)
    es = 2 if c["dtype"] == "bf16" else 4
    d, e, i, sh = c["d"], c["E"], c["inter"], c["shared"]
    if "tokens" in c:
        pairs = int(_given_counts(c, 0).sum())
    elif "rule" in c:  # about what the rules give on these inputs
        lo = c["rule"] == "top_p" and e == 64
        hi = c["rule"] == "top_p" or e == 64
        pairs = int(T * (3.0 if lo else 11.9 if hi else 2.0))
    else:
        st, p = _state(c, 0), c
        pairs = int(_allocate64(st, p).sum())
    route = dict(bytes=T * d * es + e * d * es + T * c["k_max"] * 8, flops=2 * T * e * d)
    if c["call"] == "route":
        return route
    touched = e * (1 - (1 - 1 / e) ** pairs)  # experts that at least one pair needs
    layer = dict(bytes=touched * 3 * d * i * es + 3 * d * sh * es + e * d * es + 2 * T * d * es,
                 flops=route["flops"] + 6 * pairs * d * i + 6 * T * d * sh)
    n = c.get("layers", 1)
    return dict(bytes=n * layer["bytes"], flops=n * layer["flops"])


def tolerance(case):
    c = case
    if c["call"] == "loop":
        return "exact"
    if c["call"] == "route":  # fp32 softmax of scores in a fixed order
        return dict(rel=4e-6, max=4e-5, differ=0.0)
    if c["dtype"] == "f32":  # sums in another order: 1.0e-6, largest 7.7e-6
        return dict(rel=4e-6, max=4e-5, differ=0.0)
    if c["call"] == "stack":
        # bf16 hidden states between the layers, and experts that change with
        # them: 1.8e-3 after two layers in another order, 1.9e-2 after eight
        return dict(rel=2e-2, max=0.9, differ=0.0)
    # SIMT instead of tensor-core sums: 7.1e-4, largest 1.9e-2 (two bf16 ulps)
    return dict(rel=3e-3, max=8e-2, differ=0.0)


# ---- the same in 64 bits ----------------------------------------------------
def _allocate64(st, c):
    """Counts of Eq. 5 and Eq. 9 in 64 bits."""
    k = np.zeros(st["block_id"].size, np.int64)
    sig = lambda x: 1.0 / (1.0 + np.exp(-x))  # noqa: E731
    off = st["seq_offsets"]
    for s, a in enumerate(st["active_block"]):
        r = slice(off[s], off[s + 1])
        b, dist = st["block_id"][r], np.abs(st["block_id"][r] - a)
        ks = c["k_base"] + np.where(dist <= 1, 1, np.where(dist == 2, 0, -1)) * c["delta_role"]
        h = st["hist_len"][r]
        j = np.nonzero((b == a) & (st["masked"][r] == 1) & (h >= 1))[0]
        c1, c2 = st["conf1"][r][j].astype(np.float64), st["conf2"][r][j].astype(np.float64)
        v = np.clip(np.where(h[j] >= 2, c1 - c2, 0.0), -W_CF / 2, W_CF / 2)
        ahead = np.clip(c1 + v, 0, 1)
        front = sig((ahead - THETA + W_CF) / TAU) * sig((THETA - ahead) / TAU)
        score = front * np.where(h[j] >= 2, sig((V_REF - v) / TAU), 1.0)
        order = j[np.argsort(-score, kind="stable")]
        n = int(math.floor(Q * j.size))
        ks[order[:n]] += c["delta_cur"]
        ks[order[j.size - n:]] -= c["delta_cur"]
        k[r] = np.clip(ks, c["k_min"], c["k_max"])
    return k


def _route64(c, h, w_router, k):
    """Top-k_t experts of every token [T, k_max] (score order) and their weights."""
    z = h @ w_router.double().T
    if "rule" in c:
        p = torch.softmax(z, 1)
        if c["rule"] == "top_p":
            mass = torch.sort(p, 1, descending=True).values.cumsum(1)
            k = (mass < c["threshold"]).sum(1) + 1
        else:
            k = (p > c["threshold"]).sum(1)
        k = k.clamp(c["k_min"], min(c["k_max"], c["E"]))
    top = torch.topk(z, min(c["k_max"], c["E"]), dim=1)
    used = torch.arange(top.values.shape[1], device=h.device)[None] < k[:, None]
    alpha = torch.softmax(top.values.masked_fill(~used, -math.inf), 1)
    return top.indices.masked_fill(~used, -1), alpha


def _swiglu64(x, gate_up, down):
    n = gate_up.shape[0] // 2
    g = x @ gate_up[:n].double().T
    g = g * torch.sigmoid(g)
    return (g * (x @ gate_up[n:].double().T)) @ down.double().T


def _layer64(c, w, h, k):
    ids, alpha = _route64(c, h, w["w_router"], k)
    out = torch.zeros_like(h)
    for e in range(c["E"]):
        t, j = torch.nonzero(ids == e, as_tuple=True)
        if t.numel():
            y = _swiglu64(h[t], w["w_gate_up"][e], w["w_down"][e])
            out.index_add_(0, t, alpha[t, j, None] * y)
    if c["shared"]:
        out += _swiglu64(h, w["shared_gate_up"], w["shared_down"])
    return out


def exact(case, seed):
    c = case
    # 64-bit products run at about 1 TFLOP/s here; counts and state are integers and copies
    if c["call"] == "loop" or work(c)["flops"] > 1e13:
        return None
    inp = _inputs(c, seed)
    k = torch.from_numpy(np.asarray(inp["k"] if "k" in inp else _allocate64(inp["state"], c))).cuda()
    h = inp["hidden"].double()
    if c["call"] == "route":
        _, alpha = _route64(c, h, inp["layers"][0]["w_router"], k)
        full = torch.zeros((h.shape[0], c["k_max"]), dtype=torch.float64, device="cuda")
        full[:, :alpha.shape[1]] = alpha
        return dict(ids=None, alpha=full)
    for w in inp["layers"]:
        out = _layer64(c, w, h, k)
        h = h + out
    out = h if c["call"] == "stack" else out
    return dict(out=out) if c["call"] == "forward" else dict(out=out, k=None, k_sum=None)
