"""The work that programs built on this library have it do, as cases that can be timed.

A case is one of six kinds of use:

  generate   a decoding loop on the library's own drafter: the state saved after the prompt is restored, then `rounds`
             rounds of draft -> verify -> update with the target's logits of every round on the device
  host       the same loop through the host-buffer call (pinned buffers, results back on the host)
  prompt     the prompts of every drafting input are fed (image embeddings, pooled image embeddings, text), then one
             decoder step gives the first logits
  engine     one round on drafter logits that the caller's own engine computed (a handle without a drafter)
  ensemble   one ensemble step on the caller's logits, with every distribution returned
  plain      the ensemble step without a handle (nothing allocated)

A drafter's weights are random, but its LM head favours a known successor of every token, so that its distributions are
peaked as a trained model's are; the target's logits of every round follow the successors, accept a planned number of
drafts and emit a planned token.  Where the caller brings the logits they are flat, and every result is exact.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2601_20357_b200 import binding as TB
from paper_2601_20357_b200 import workloads as W

STATIC, GRID, SOFTMAX, ADABOOST = "static", "grid", "softmax", "adaboost"
_POLICY = {STATIC: TB.POLICY_STATIC, GRID: TB.POLICY_GRID_MT, SOFTMAX: TB.POLICY_SOFTMAX_INV_ERR, ADABOOST: TB.POLICY_ADABOOST}

_SMALL = dict(layers=4, width=768, heads=12, kv_heads=12, ffn=3072, vocab=32000, dtype="bf16")
_WIDE = dict(layers=12, width=896, heads=14, kv_heads=2, ffn=4864, vocab=152064, dtype="bf16")
_TINY = dict(layers=2, width=128, heads=4, kv_heads=4, ffn=512, vocab=1024, dtype="fp32")


def listed():
    return [
        # one chat request: image + text, text alone and caption + text as the three inputs (a small drafter, sampled)
        dict(name="chat_one_request", kind="generate", **_SMALL, inputs=3, requests=1, gamma=5, window=8, policy=SOFTMAX,
             distance="kl", greedy=False, tree=1, context_low=128, context_high=704, rounds=6),
        # the same drafter serving two requests at once on short contexts, greedy as the paper's reported runs are
        dict(name="chat_two_requests", kind="generate", **_SMALL, inputs=3, requests=2, gamma=3, window=4, policy=SOFTMAX,
             distance="tvd", greedy=True, tree=1, context_low=61, context_high=531, rounds=6),
        # a drafter of a large vocabulary with grouped queries, four inputs (two of them with a 1024-token image)
        dict(name="large_vocabulary", kind="generate", **_WIDE, inputs=4, requests=1, gamma=5, window=8, policy=SOFTMAX,
             distance="kl", greedy=False, tree=1, context_low=128, context_high=1152, rounds=3),
        # a long document under all three inputs
        dict(name="long_context", kind="generate", **_SMALL, inputs=3, requests=1, gamma=7, window=16, policy=SOFTMAX,
             distance="kl", greedy=True, tree=1, context_low=8192, context_high=8192, rounds=3),
        # serving: 32 requests of 3 inputs with contexts of all lengths
        dict(name="serving_32_requests", kind="generate", **_SMALL, inputs=3, requests=32, gamma=5, window=8, policy=SOFTMAX,
             distance="kl", greedy=False, tree=1, context_low=256, context_high=4096, rounds=3),
        # a token tree of width 3 for a handful of requests, hard-label weights
        dict(name="token_tree", kind="generate", **_SMALL, inputs=3, requests=6, gamma=5, window=8, policy=ADABOOST,
             distance="kl", greedy=True, tree=3, context_low=200, context_high=1999, rounds=3),
        # the fp32 drafter, two inputs, grid policy: launches and latency
        dict(name="fp32_drafter", kind="generate", **_TINY, inputs=2, requests=1, gamma=3, window=4, policy=GRID,
             distance="kl", greedy=False, tree=1, context_low=16, context_high=64, rounds=6),
        # rounds with host buffers: a target model whose logits arrive in pinned memory
        dict(name="host_buffers", kind="host", **_SMALL, inputs=3, requests=8, gamma=5, window=8, policy=SOFTMAX,
             distance="kl", greedy=False, tree=1, context_low=300, context_high=1500, rounds=3),
        # time to the first logits of a chat request: 576 image tokens + text, text, pooled image + text
        dict(name="prompt_chat", kind="prompt", **_SMALL, inputs=3, requests=1, image_grid=24, text=128),
        # the same for the large-vocabulary drafter: 1024 image tokens and longer text
        dict(name="prompt_large_vocabulary", kind="prompt", **_WIDE, inputs=4, requests=1, image_grid=32, text=131),
        # an engine that runs its own drafter and hands over logits: 16 requests, flat distributions
        dict(name="engine_logits", kind="engine", vocab=32000, inputs=3, requests=16, gamma=5, window=8, policy=SOFTMAX,
             distance="kl", greedy=False),
        # one ensemble step of one request: the smallest call
        dict(name="ensemble_step", kind="ensemble", vocab=32000, inputs=3, requests=1, greedy=False),
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["generate"] * 5 + ["host", "prompt", "prompt", "engine", "engine", "ensemble", "plain"])
    if kind in ("engine", "ensemble", "plain"):
        c = dict(kind=kind, vocab=_log_int(rng, 97, 152064), inputs=rng.choice([1, 2, 3, 3, 4, 5]), greedy=rng.random() < 0.3)
        most = max(1, min(64, 3_000_000 // (c["vocab"] * c["inputs"])))
        c["requests"] = _log_int(rng, 1, most)
        if kind == "engine":
            c.update(gamma=rng.choice([3, 5, 7]), window=rng.choice([0, 4, 8, 16]), distance=rng.choice(["kl", "tvd"]),
                     policy=rng.choice([SOFTMAX, SOFTMAX, STATIC] + ([GRID] if c["inputs"] == 2 else [])))
        return c
    fp32 = kind == "generate" and rng.random() < 0.15
    if fp32:
        hd, heads = rng.choice([32, 64]), rng.choice([2, 4])
        c = dict(kind=kind, layers=rng.randint(1, 3), width=hd * heads, heads=heads, kv_heads=heads, ffn=rng.choice([256, 512, 520]),
                 vocab=_log_int(rng, 500, 8000), dtype="fp32")
    else:
        hd = rng.choice([64, 64, 64, 128, 32])
        heads = rng.randint(max(4, 256 // hd), 1024 // hd)
        kv = rng.choice([k for k in range(1, heads + 1) if heads % k == 0 and heads // k <= 8])
        width = hd * heads
        c = dict(kind=kind, layers=rng.randint(2, 8), width=width, heads=heads, kv_heads=kv,
                 ffn=16 * rng.randint(width // 8, width // 4), vocab=_log_int(rng, 4001, 80000), dtype="bf16")
    c["inputs"] = rng.choice([2, 3, 3, 3, 4])
    if kind == "prompt":
        c.update(requests=rng.choice([1, 1, 2]), image_grid=2 * rng.randint(4, 14), text=_log_int(rng, 5, 500))
        return c
    c["requests"] = _log_int(rng, 1, 2 if fp32 else 24)
    tree = rng.choice([1, 1, 1, 2, 3]) if kind == "generate" and not fp32 else 1
    greedy = tree > 1 or rng.random() < 0.4
    high = _log_int(rng, 24, 300 if fp32 else 6000)
    # no more cache to read than the largest listed case has
    most = 96 * 2176 * 4 * 768 // (c["requests"] * c["inputs"] * c["layers"] * c["kv_heads"] * hd)
    high = max(20, min(high, most))
    c.update(gamma=rng.choice([3, 5, 7]), window=rng.choice([4, 8, 16]), policy=ADABOOST if tree > 1 else SOFTMAX,
             distance=rng.choice(["kl", "kl", "tvd"]), greedy=greedy, tree=tree, context_low=max(4, high // rng.choice([1, 4, 16])),
             context_high=high, rounds=rng.choice([2, 3]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniforms(g, shape, low=0.0, high=1.0):
    """Uniforms of [low, high) on the library's lattice (k + 1/2) 2^-23."""
    k = torch.randint(int(low * (1 << 23)), int(high * (1 << 23)), shape, generator=g, device="cuda")
    return ((k.double() + 0.5) * 2.0 ** -23).float()


def _lengths(c):
    """Cached positions of every row, spread over the case's range in no order."""
    rows, lo, hi = c["inputs"] * c["requests"], c["context_low"], c["context_high"]
    lens = [lo + (hi - lo) * r // max(1, rows - 1) for r in range(rows)]
    random.Random(rows).shuffle(lens)
    return lens


def _drafter(c):
    return W.DrafterCfg(c["layers"], c["width"], c["heads"], c["kv_heads"], c["ffn"], c["vocab"], c["dtype"])


def _weights(c, g):
    """Random weights (std 0.02); the LM head's row of a token's successors holds that token's embedding."""
    d, F, V = c["width"], c["ffn"], c["vocab"]
    kvd = d // c["heads"] * c["kv_heads"]
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    rnd = lambda *s: (0.02 * torch.randn(s, generator=g, device="cuda")).to(dt)
    w = {"embed": torch.randn((V, d), generator=g, device="cuda").to(dt), "final_norm": torch.ones(d, device="cuda", dtype=dt)}
    sharp = c.get("greedy", True)
    top = math.log(V) + (3.0 if sharp else 14.0)
    top += 0.5 * (top / (0.8 * math.sqrt(d))) ** 2
    scale = top / (0.8 * d)
    ranks = [1.0] if c.get("tree", 1) == 1 else [1.15, 1.0, 0.85, 0.7][:c["tree"]]
    head = torch.zeros((V, d), device="cuda")
    succ = []
    for a in ranks:
        s = torch.randperm(V, generator=g, device="cuda")
        head[s] += (a * scale) * w["embed"].float()
        succ.append(s.cpu().numpy())
    w["lm_head"] = head.to(dt)
    shapes = dict(wq=(d, d), wk=(kvd, d), wv=(kvd, d), wo=(d, d), w_gate=(F, d), w_up=(F, d), w_down=(d, F))
    for nm, s in shapes.items():
        w[nm] = [rnd(*s) for _ in range(c["layers"])]
    for nm in ("norm1", "norm2"):
        w[nm] = [torch.ones(d, device="cuda", dtype=dt) for _ in range(c["layers"])]
    return w, succ


def _caches(c, g):
    hd = c["width"] // c["heads"]
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    one = lambda n: (0.5 * torch.randn((c["layers"], c["kv_heads"], n, hd), generator=g, device="cuda")).to(dt)
    for n in _lengths(c):
        yield one(n), one(n)


def _boosted(c, g, rows, favourite):
    """Target logits [rows][V]: noise and one favourite a row; greedy decoding meets softer rows."""
    V = c["vocab"]
    lg = torch.randn((rows, V), generator=g, device="cuda")
    lg.scatter_(1, favourite.view(-1, 1), math.log(V) + (2.0 if c["greedy"] else 3.0))
    return lg


def _plan(c, succ, g, seed):
    """Rounds of target logits and uniforms, and the tokens pending before the first: every round accepts a planned
    number of drafts (a sibling after them, in a tree) and emits a planned token."""
    B, G, D, V, m = c["requests"], c["gamma"], c["tree"], c["vocab"], c["inputs"]
    rng = random.Random(seed)
    first = last = [rng.randrange(V) for _ in range(B)]
    rounds = []
    for _ in range(c["rounds"]):
        favourite, keep, after = [], [], []
        for b in range(B):
            chain, t = [], last[b]
            kids = []
            for _ in range(G):
                kids.append([int(s[t]) for s in succ])
                t = kids[-1][0]
                chain.append(t)
            a, z = rng.choice([G, G, *range(G)]), rng.randrange(V)
            sibling = rng.randrange(1, D) if D > 1 and a < G and rng.random() < 0.5 else 0
            while z in chain or any(z in k for k in kids):
                z = rng.randrange(V)
            rows = chain[:a] + [kids[a][sibling] if sibling else z] * (G + 1 - a)
            rows += [z] * (G * (D - 1))
            favourite += rows
            keep.append(a)
            after.append(z)
        rows = G + 1 + G * (D - 1)
        target = _boosted(c, g, B * rows, torch.tensor(favourite, device="cuda"))
        if not c["greedy"]:
            # the row of a rejected draft and the bonus row leave no doubt about what they emit
            at = torch.tensor([b * rows + a for b, a in enumerate(keep)], device="cuda")
            z = torch.tensor(after, device="cuda")
            target[at, z] += 12.0
        rounds.append(dict(target=target.view(B, rows, V), u_draft=_uniforms(g, (B, G, D) if D > 1 else (B, G)),
                           u_accept=_uniforms(g, (B, G, D) if D > 1 else (B, G), 0.01, 0.8), u_resid=_uniforms(g, (B,))))
        last = after
    return first, rounds


def _handle(c, weights=None, capacity=0):
    return TB.Tabed(n_inputs=c["inputs"], n_requests=c["requests"], gamma=c.get("gamma", 1), window_h=c.get("window", 0),
                    policy=_POLICY[c.get("policy", STATIC)], vocab=c["vocab"],
                    distance=TB.DIST_TVD if c.get("distance") == "tvd" else TB.DIST_KL,
                    sample_mode=TB.MODE_GREEDY if c.get("greedy") else TB.MODE_SAMPLE, tau=1.0,
                    drafter=_drafter(c) if weights is not None else None, weights=weights, kv_capacity=capacity,
                    tree_width=c.get("tree", 1))


def _view(h, what):
    """One of the handle's own buffers; the handle lives as long as the tensor does."""
    t = h.debug_view(what)
    t.owner = h
    return t


def _set_pending(h, first):
    tok = torch.zeros((len(first), 2), dtype=torch.int32, device="cuda")
    tok[:, 0] = torch.tensor(first, dtype=torch.int32)
    h.set_pending(tok, torch.ones(len(first), dtype=torch.int32, device="cuda"))


def _prompt_inputs(c, g):
    """Segments of every row: [("embeds" | "pool" | "tokens", tensor)]; image, text, pooled image and noisy image in turn."""
    n, d = c["image_grid"], c["width"]
    rows = []
    for _ in range(c["requests"]):
        image = torch.randn((n * n, d), generator=g, device="cuda")
        for k in range(c["inputs"]):
            text = torch.randint(0, c["vocab"], (c["text"],), generator=g, device="cuda", dtype=torch.int32)
            if k == 0:
                rows.append([("embeds", image), ("tokens", text)])
            elif k == 1:
                rows.append([("tokens", text)])
            elif k == 2:
                rows.append([("pool", image), ("tokens", text)])
            else:
                noisy = image + 0.5 * torch.randn(image.shape, generator=g, device="cuda")
                rows.append([("embeds", noisy), ("tokens", text)])
    return rows


def _flat(c, g, steps):
    """Flat drafter logits [steps][B][m][V] and, with steps > 1, a target near their mean."""
    B, m, V = c["requests"], c["inputs"], c["vocab"]
    base = torch.randn((steps, B, 1, V), generator=g, device="cuda")
    drafts = base + 0.4 * torch.randn((steps, B, m, V), generator=g, device="cuda")
    return drafts


def _target_for(c, g, drafts):
    mean = drafts.mean(2).transpose(0, 1)                                     # [B][G][V]
    mean = torch.cat([mean, mean[:, -1:]], 1)
    return (mean + 0.5 * torch.randn(mean.shape, generator=g, device="cuda")).contiguous()


def _inputs(c, seed):
    """Everything random of a case, from the seed alone."""
    g = _gen(seed)
    s = {}
    B, m = c["requests"], c["inputs"]
    if c["kind"] in ("generate", "host"):
        s["weights"], succ = _weights(c, g)
        s["first"], s["rounds"] = _plan(c, succ, g, seed)
        s["generator"] = g                                                    # the caches follow, row by row
    elif c["kind"] == "prompt":
        s["weights"], _ = _weights(c, g)
        s["prompts"] = _prompt_inputs(c, g)
        s["first"] = torch.randint(0, c["vocab"], (B,), generator=g, device="cuda", dtype=torch.int32)
    elif c["kind"] == "engine":
        s["drafts"] = _flat(c, g, c["gamma"])
        s["target"] = _target_for(c, g, s["drafts"])
        s["u_draft"], s["u_accept"], s["u_resid"] = _uniforms(g, (B, c["gamma"])), _uniforms(g, (B, c["gamma"])), _uniforms(g, (B,))
    else:
        s["logits"] = _flat(c, g, 1)[0]
        s["w"] = torch.softmax(torch.randn((B, m), generator=g, device="cuda"), 1)
        s["u"] = _uniforms(g, (B,))
    return s


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    s["case"] = c
    B, m, V = c["requests"], c["inputs"], c["vocab"]
    new = lambda *shape, dtype=torch.float32: torch.empty(shape, dtype=dtype, device="cuda")
    i32 = torch.int32
    if c["kind"] in ("generate", "host"):
        G, D, n = c["gamma"], c["tree"], c["rounds"]
        h = s["handle"] = _handle(c, s["weights"], c["context_high"] + n * (G + 1) + 2)
        for row, (k, v) in enumerate(_caches(c, s.pop("generator"))):
            h.load_prefix_kv(row, k, v)
        _set_pending(h, s["first"])
        s["saved"] = h.state_export()
        out = dict(tokens=new(n, B, G * D, dtype=i32), accepted=new(n, B, dtype=i32), next=new(n, B, dtype=i32), weights=new(n, B, m))
        if c["kind"] == "host":
            pin = lambda t: t.cpu().pin_memory()
            s["rounds"] = [{k: pin(t) for k, t in r.items()} for r in s["rounds"]]
            out = {k: pin(t) for k, t in out.items()}
        else:
            # what the last round drafted from
            out["logits"], out["mix"] = _view(h, TB.VIEW_LOGITS), _view(h, TB.VIEW_Q)
        s["out"] = out
    elif c["kind"] == "prompt":
        longest = max(sum(t.shape[0] for _, t in segs) for segs in s["prompts"])
        h = s["handle"] = _handle(c, s["weights"], longest + 8)
        s["saved"] = h.state_export()
        s["pooled"] = new(c["image_grid"] ** 2 // 4, c["width"])
        s["out"] = dict(logits=new(B, m, V))
    elif c["kind"] == "engine":
        h = s["handle"] = _handle(c)
        s["saved"] = h.state_export()
        s["out"] = dict(tokens=new(B, c["gamma"], dtype=i32), accepted=new(B, dtype=i32), next=new(B, dtype=i32),
                        weights=new(B, m), best=new(B, dtype=i32), mix=new(B, c["gamma"], V), each=_view(h, TB.VIEW_QK))
    else:
        if c["kind"] == "ensemble":
            s["handle"] = _handle(c)
        s["out"] = dict(token=new(B, dtype=i32), mix=new(B, V), each=new(B, m, V))
    return s


def run(state):
    s, c, out = state, state["case"], state["out"]
    if c["kind"] == "generate":
        h = s["handle"]
        h.state_import(s["saved"])
        for i, r in enumerate(s["rounds"]):
            h.draft_round(r["u_draft"], out["tokens"][i])
            h.verify(r["target"], r["u_accept"], r["u_resid"], out["accepted"][i], out["next"][i])
            h.update_weights(out["weights"][i])
    elif c["kind"] == "host":
        h = s["handle"]
        h.state_import(s["saved"])
        for i, r in enumerate(s["rounds"]):
            h.round_host(r["u_draft"], r["u_accept"], r["u_resid"], r["target"], out["tokens"][i], out["accepted"][i], out["next"][i],
                         out["weights"][i])
    elif c["kind"] == "prompt":
        h, n = s["handle"], c["image_grid"]
        h.state_import(s["saved"])
        for row, segments in enumerate(s["prompts"]):
            for what, data in segments:
                if what == "tokens":
                    h.prefill_tokens(row, data)
                elif what == "pool":
                    h.pool_embeds(data, n, n, s["pooled"])
                    h.prefill_embeds(row, s["pooled"])
                else:
                    h.prefill_embeds(row, data)
        h.decode_step(s["first"], out["logits"])
    elif c["kind"] == "engine":
        h = s["handle"]
        h.state_import(s["saved"])
        h.draft_round_logits(s["drafts"], s["u_draft"], out["tokens"], out["mix"])
        h.verify(s["target"], s["u_accept"], s["u_resid"], out["accepted"], out["next"])
        h.update_weights(out["weights"], out["best"])
    elif c["kind"] == "ensemble":
        s["handle"].ensemble_step(s["logits"], s["w"], s["u"], out["token"], out["mix"], out["each"])
    else:
        TB.ensemble_step_static(s["logits"], s["w"], s["u"], out["token"], out["mix"], out["each"],
                                sample_mode=TB.MODE_GREEDY if c["greedy"] else TB.MODE_SAMPLE)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    c = case
    B, m, V = c["requests"], c["inputs"], c["vocab"]
    R = B * m
    if c["kind"] in ("ensemble", "plain"):
        return {"bytes": 4.0 * V * (2 * R + B), "flops": 8.0 * R * V}
    if c["kind"] == "engine":
        G = c["gamma"]
        # logits read, distributions and their mix written, target logits and drafter distributions compared
        return {"bytes": 4.0 * V * B * (G * (2 * m + 1) + G + 1), "flops": 20.0 * V * B * G * (m + 1)}
    d, F, L, e = c["width"], c["ffn"], c["layers"], 4 if c["dtype"] == "fp32" else 2
    kvd = d // c["heads"] * c["kv_heads"]
    layer, head = 2 * d * d + 2 * d * kvd + 3 * d * F, V * d
    if c["kind"] == "prompt":
        n2, lens = c["image_grid"] ** 2, []
        for k in range(m):
            lens.append(c["text"] + (n2, 0, n2 // 4, n2)[min(k, 3)])
        lens = [n + 1 for n in lens] * B
        flops = sum(2.0 * L * layer * n + 2.0 * L * d * n * n for n in lens) + 2.0 * head * R
        embeds = sum(n - 1 - c["text"] for n in lens)
        size = e * (L * layer + head) + 4.0 * d * embeds + e * 2.0 * L * kvd * sum(lens) + 4.0 * R * V
        return {"bytes": size, "flops": flops}
    G, n, D = c["gamma"], c["rounds"], c["tree"]
    tokens = sum(_lengths(c))
    step = e * (L * layer + head) + e * 2.0 * L * kvd * tokens + 4.0 * V * (2 * R + B) + 4.0 * R * V
    size = n * (G * step + 4.0 * V * B * (G + 1 + G * (D - 1)))
    flops = n * G * (2.0 * R * (L * layer + head) + 4.0 * L * d * tokens)
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["kind"] in ("engine", "ensemble", "plain"):
        return "exact"                       # every result is a function of the logits' bits
    if case["dtype"] == "fp32":
        return {"rel": 2e-6, "max": 2e-5}     # logits 1e-7 off the same in 64 bits, weights a little more
    return {"rel": 1e-2, "max": 0.1}         # bf16 operands and caches: logits 2e-3 to 3e-3 off


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

class _Plain:
    """The drafter in 64 bits: rows with caches of their own."""

    def __init__(self, c, w, capacity):
        f = lambda t: t.double()
        self.c, self.w = c, {k: [f(t) for t in v] if isinstance(v, list) else f(v) for k, v in w.items()}
        self.R, self.H, self.K, self.hd = c["inputs"] * c["requests"], c["heads"], c["kv_heads"], c["width"] // c["heads"]
        z = lambda: [torch.zeros((self.R, self.K, capacity, self.hd), dtype=torch.float64, device="cuda") for _ in range(c["layers"])]
        self.k, self.v, self.len = z(), z(), torch.zeros(self.R, dtype=torch.long, device="cuda")
        inv = 10000.0 ** (-2.0 * torch.arange(self.hd // 2, dtype=torch.float64, device="cuda") / self.hd)
        ang = torch.arange(capacity, dtype=torch.float64, device="cuda")[:, None] * inv
        self.cos, self.sin = ang.cos(), ang.sin()

    def norm(self, x, gain):
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gain

    def turn(self, x, pos):                                                   # [n][heads][hd] at pos [n]
        a, b = x.chunk(2, -1)
        cs, sn = self.cos[pos][:, None], self.sin[pos][:, None]
        return torch.cat([a * cs - b * sn, b * cs + a * sn], -1)

    def layers(self, x, rows, pos):
        """Feeds x [n][d], position pos of row rows each (positions of one row in order), through every layer."""
        w, n, grp = self.w, x.shape[0], self.H // self.K
        one = len(set(rows.tolist())) == 1 and n > 1
        for l in range(self.c["layers"]):
            h = self.norm(x, w["norm1"][l])
            q = self.turn((h @ w["wq"][l].T).view(n, self.H, self.hd), pos)
            k = self.turn((h @ w["wk"][l].T).view(n, self.K, self.hd), pos)
            self.k[l][rows, :, pos] = k
            self.v[l][rows, :, pos] = (h @ w["wv"][l].T).view(n, self.K, self.hd)
            q = q.view(n, self.K, grp, self.hd)
            top = int(pos.max()) + 1
            if one:
                kk, vv = self.k[l][rows[0], :, :top], self.v[l][rows[0], :, :top]
                s = torch.einsum("nkgd,ktd->nkgt", q, kk)
            else:
                kk, vv = self.k[l][rows, :, :top], self.v[l][rows, :, :top]
                s = torch.einsum("nkgd,nktd->nkgt", q, kk)
            s = s / math.sqrt(self.hd)
            s = s.masked_fill((torch.arange(top, device="cuda")[None] > pos[:, None])[:, None, None], -math.inf).softmax(-1)
            o = torch.einsum("nkgt,ktd->nkgd" if one else "nkgt,nktd->nkgd", s, vv).reshape(n, -1)
            x = x + o @ w["wo"][l].T
            h = self.norm(x, w["norm2"][l])
            x = x + (torch.nn.functional.silu(h @ w["w_gate"][l].T) * (h @ w["w_up"][l].T)) @ w["w_down"][l].T
        return x

    def step(self, rows, tokens, pos):
        return self.layers(self.w["embed"][tokens], rows, pos)

    def logits(self, x):
        return self.norm(x, self.w["final_norm"]) @ self.w["lm_head"].T


def _pick(q, u, greedy):
    if greedy:
        return q.argmax(-1)
    cdf = q.cumsum(-1)
    return (cdf > (u.double() * cdf[..., -1]).unsqueeze(-1)).double().argmax(-1)


def _decide(c, qk, q, cand, r, p, history, w):
    """Verification and weight update of one round: (accepted, accepted of the primary chain, emitted, pending) a request."""
    B, G, D, V = c["requests"], c["gamma"], c.get("tree", 1), c["vocab"]
    accepted, primary, emitted, pending = [], [], [], []
    for b in range(B):
        a, sib = 0, -1
        while a < G:
            y = int(cand[b, a, 0])
            ok = int(p[b, a].argmax()) == y if c["greedy"] else float(p[b, a, y]) > float(r["u_accept"].reshape(B, G, D)[b, a, 0]) * float(q[b, a, y])
            if not ok:
                break
            a += 1
        if a < G and D > 1:                                                   # greedy trees
            best = int(p[b, a].argmax())
            sib = next((i for i in range(1, D) if int(cand[b, a, i]) == best), -1)
        row = p[b, G + 1 + a * (D - 1) + sib - 1] if sib > 0 else p[b, a]
        if a < G and sib < 0 and not c["greedy"]:
            row = (row - q[b, a]).clamp(min=0)
        z = int(_pick(row, r["u_resid"][b], c["greedy"]))
        accepted.append(a + (sib > 0))
        primary.append(a)
        emitted.append(z)
        pending.append([int(cand[b, a, sib]), z] if sib > 0 else [int(cand[b, G - 1, 0]), z] if a == G else [z])
        grid = c["policy"] == GRID
        for i in range(min(a, G - 1) + 1):
            pi, label = p[b, i], int(cand[b, i, 0]) if i < a else int(cand[b, a, sib]) if sib > 0 else z
            if grid:
                t = torch.arange(11, dtype=torch.float64, device="cuda")[:, None] / 10
                qs = (1 - t) * qk[b, i, 0] + t * qk[b, i, 1]
            else:
                qs = qk[b, i]
            if c["policy"] == ADABOOST:
                dev = (qs.argmax(-1) != label).double()
            elif c["distance"] == "tvd":
                dev = 0.5 * (pi - qs).abs().sum(-1)
            else:
                dev = (pi * (pi.clamp(min=1e-300).log() - qs.clamp(min=1.1754943508222875e-38).log())).sum(-1)
            history[b].append(dev)
        seen = torch.stack(history[b][-c["window"]:] if c["window"] else history[b])
        e, m = seen.sum(0), c["inputs"]
        if c["policy"] == SOFTMAX:
            w[b] = torch.softmax(1.0 / e.clamp(min=1e-8), 0)
        elif grid:
            j = int(e.argmin()) / 10
            w[b] = torch.tensor([1 - j, j], dtype=torch.float64)
        elif c["policy"] == ADABOOST:
            eps = (e + 1) / (len(seen) + 2)
            alpha = ((1 / eps - 1).log() + math.log(V - 1)).clamp(min=0)
            w[b] = alpha / alpha.sum() if float(alpha.sum()) > 0 else torch.full((m,), 1.0 / m, dtype=torch.float64)
    return accepted, primary, emitted, pending


def exact(case, seed):
    c = case
    s = _inputs(c, seed)
    B, m, V = c["requests"], c["inputs"], c["vocab"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if c["kind"] in ("ensemble", "plain"):
        each = s["logits"].double().softmax(-1)
        return dict(token=None, mix=(each * s["w"].double()[..., None]).sum(1), each=each)
    history = [[] for _ in range(B)]
    w = torch.full((B, m), 1.0 / m, **f64)
    if c["kind"] == "engine":
        each = s["drafts"].double().softmax(-1).transpose(0, 1).contiguous()  # [B][G][m][V]
        mix = (each * w[:, None, :, None]).sum(2)
        cand = _pick(mix, s["u_draft"], c["greedy"])[..., None]
        r = dict(u_accept=s["u_accept"], u_resid=s["u_resid"])
        _decide(c, each, mix, cand, r, s["target"].double().softmax(-1), history, w)
        return dict(tokens=None, accepted=None, next=None, weights=w, best=None, mix=mix, each=each)
    if c["kind"] == "prompt":
        lens = [sum((t.shape[0] // 4 if what == "pool" else t.shape[0]) for what, t in segs) for segs in s["prompts"]]
        net = _Plain(c, s["weights"], max(lens) + 1)
        n = c["image_grid"]
        for row, segs in enumerate(s["prompts"]):
            xs = []
            for what, t in segs:
                if what == "tokens":
                    xs.append(net.w["embed"][t.long()])
                elif what == "pool":
                    xs.append(t.double().view(n // 2, 2, n // 2, 2, -1).mean((1, 3)).reshape(n * n // 4, -1))
                else:
                    xs.append(t.double())
            net.layers(torch.cat(xs), torch.full((lens[row],), row, device="cuda"), torch.arange(lens[row], device="cuda"))
        rows = torch.arange(B * m, device="cuda")
        x = net.step(rows, s["first"].long().repeat_interleave(m), torch.tensor(lens, device="cuda"))
        return dict(logits=net.logits(x).view(B, m, V))
    G, D, n = c["gamma"], c["tree"], c["rounds"]
    net = _Plain(c, s["weights"], c["context_high"] + n * (G + 1) + 2)
    lens = _lengths(c)
    for row, (k, v) in enumerate(_caches(c, s["generator"])):
        for l in range(c["layers"]):
            net.k[l][row, :, :lens[row]], net.v[l][row, :, :lens[row]] = k[l].double(), v[l].double()
    lens = torch.tensor(lens, device="cuda")
    pending = [[t] for t in s["first"]]
    rows, weights = torch.arange(B * m, device="cuda"), []
    for r in s["rounds"]:
        double = [b for b in range(B) if len(pending[b]) == 2]
        pos = lens.clone()
        if double:
            sel = torch.tensor([b * m + k for b in double for k in range(m)], device="cuda")
            net.step(sel, torch.tensor([pending[b][0] for b in double], device="cuda").repeat_interleave(m), pos[sel])
            pos[sel] += 1
        tok = torch.tensor([p[-1] for p in pending], device="cuda")
        lgs, mixes, eachs, cands = [], [], [], []
        for i in range(G):
            lg = net.logits(net.step(rows, tok.repeat_interleave(m), pos)).view(B, m, V)
            each = lg.softmax(-1)
            mix = (each * w[..., None]).sum(1)
            cand = mix.topk(D).indices if D > 1 else _pick(mix, r["u_draft"][:, i], c["greedy"])[:, None]
            tok, pos = cand[:, 0], pos + 1
            lgs.append(lg), mixes.append(mix), eachs.append(each), cands.append(cand)
        mix = torch.stack(mixes, 1)
        before = pending
        _, primary, _, pending = _decide(c, torch.stack(eachs, 1), mix, torch.stack(cands, 1), r, r["target"].double().softmax(-1), history, w)
        weights.append(w.clone())
        lens = lens + torch.tensor([len(before[b]) + min(primary[b], G - 1) for b in range(B)], device="cuda").repeat_interleave(m)
    out = dict(tokens=None, accepted=None, next=None, weights=torch.stack(weights))
    if c["kind"] == "generate":
        out["logits"], out["mix"] = torch.stack(lgs), mix
    return out
