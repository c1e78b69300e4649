"""The calls that a user of this library makes, as cases that can be timed and compared.

A request is: prompt pass, choice of the domain's skip mask, rounds of draft and verification passes (greedy or
sampled); anchors are built once beforehand.  Each listed case is one of these calls through the binding, at the widths
of the shapes this repository names.  Models are cut to a few layers where the call does the same thing layer after
layer; `request-7b-512` runs one model at its full depth.

A case holds plain values; `kind` says which call it is:

  select    Session.select_skipset on a given query (domains x 10 anchors)
  draft     Session.draft of one token with 45 % of the sublayers skipped, logits returned
  verify    Session.verify of k given drafts at a given context, logits and hidden states returned
  prompt    Session.prefill of `rows` tokens, pooled hidden state and first token returned
  round     one round of sampled decoding on given logits: both models' filtered distributions, keep-or-resample
  pick      one sampled draft token from given logits: filtered distribution, draw
  anchors   knnssd_build_anchors on `domains` x `per` vectors
  request   prompt pass, mask choice, first draft step and first verification pass of one request
"""
from __future__ import annotations

import math

import numpy as np
import torch

import synthetic_inputs as si
from paper_2505_16162_b200 import binding as kb

ANCHORS_PER_DOMAIN = 10


def listed():
    return [
        # choosing the domain of a request among 5 x 10 anchors: the smallest call, once per request
        {"name": "select-5x10-13b", "kind": "select", "shape": "llama13b", "domains": 5},
        # the small fp32 configuration, whole: a verification pass that is nothing but latency
        {"name": "verify-tiny-fp32-k4", "kind": "verify", "shape": "tiny", "layers": 4, "context": 96, "k": 4},
        # one draft step, the call made most often: 13B widths in mid-generation after a 1024-token prompt
        {"name": "draft-13b-ctx1280", "kind": "draft", "shape": "llama13b", "layers": 8, "context": 1280},
        # one verification pass at the usual draft length, same context
        {"name": "verify-13b-k4-ctx1280", "kind": "verify", "shape": "llama13b", "layers": 8, "context": 1280, "k": 4},
        # a longer draft on the narrower model: nine rows
        {"name": "verify-7b-k8-ctx640", "kind": "verify", "shape": "llama7b", "layers": 8, "context": 640, "k": 8},
        # grouped query heads, a long context and a vocabulary of 152064
        {"name": "verify-qwen14b-k4-ctx2304", "kind": "verify", "shape": "qwen14b", "layers": 8, "context": 2304, "k": 4},
        # a short question of ragged length: time to the first token
        {"name": "prompt-7b-77", "kind": "prompt", "shape": "llama7b", "layers": 8, "rows": 77},
        # the prompt of the benchmark's workload
        {"name": "prompt-13b-1024", "kind": "prompt", "shape": "llama13b", "layers": 8, "rows": 1024},
        # sampled decoding at temperature 0.2 and top-p 0.85: what follows a verification pass of k = 4
        {"name": "round-k4-v32000", "kind": "round", "vocab": 32000, "k": 4, "temperature": 0.2, "top_p": 0.85},
        # and what follows each draft step, on the largest vocabulary
        {"name": "pick-v152064", "kind": "pick", "vocab": 152064, "temperature": 0.2, "top_p": 0.85},
        # anchors from 1000 sampled vectors of each of 5 domains
        {"name": "anchors-5x1000-d5120", "kind": "anchors", "domains": 5, "per": 1000, "d": 5120},
        # the first round of a whole request at full depth
        {"name": "request-7b-512", "kind": "request", "shape": "llama7b", "layers": 32, "rows": 512, "k": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select", "draft", "verify", "verify", "prompt", "prompt", "round", "pick", "anchors", "request"])
    shape = rng.choice(["llama7b", "llama13b", "qwen14b"])
    layers = rng.randint(2, 8)
    if kind == "select":
        return {"kind": kind, "shape": shape, "domains": rng.randint(2, 40)}
    if kind == "draft":
        return {"kind": kind, "shape": shape, "layers": layers, "context": _log_int(rng, 40, 2600)}
    if kind == "verify":
        if rng.random() < 0.15:
            return {"kind": kind, "shape": "tiny", "layers": 4, "context": rng.randint(20, 400), "k": rng.randint(0, 8)}
        return {"kind": kind, "shape": shape, "layers": layers, "context": _log_int(rng, 40, 2600), "k": rng.randint(0, 15)}
    if kind == "prompt":
        return {"kind": kind, "shape": shape, "layers": layers, "rows": _log_int(rng, 8, 2100)}
    if kind == "round":
        return {"kind": kind, "vocab": _log_int(rng, 1000, 152064), "k": rng.randint(1, 8), "temperature": rng.choice([0.2, 0.5, 0.7, 1.0]),
                "top_p": rng.choice([0.8, 0.85, 0.9, 0.95])}
    if kind == "pick":
        return {"kind": kind, "vocab": _log_int(rng, 1000, 152064), "temperature": rng.choice([0.2, 0.5, 0.7, 1.0]),
                "top_p": rng.choice([0.8, 0.85, 0.9, 0.95])}
    if kind == "anchors":
        return {"kind": kind, "domains": rng.randint(2, 10), "per": _log_int(rng, 60, 1000), "d": 64 * rng.randint(16, 80) + rng.choice([0, 0, 0, 4, 1])}
    return {"kind": kind, "shape": "llama7b", "layers": rng.randint(4, 24), "rows": _log_int(rng, 20, 512), "k": rng.randint(1, 8)}


# ---- inputs -------------------------------------------------------------------------------------------------------
def _shape(case):
    return si.SHAPES[case["shape"]].with_layers(case.get("layers", 1))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _mask(shape, seed):
    return si.skip_mask(seed + 102, 2 * shape.n_layers, int(round(0.45 * 2 * shape.n_layers)))


def _tokens(case, shape, seed):
    """(context or prompt, pending token and drafts)"""
    n = case.get("context", case.get("rows", 0))
    return (si.uniform_tokens(seed, 0, n, shape.vocab).numpy(),
            si.uniform_tokens(seed, 1, case.get("k", 0) + 1, shape.vocab).numpy())


def _anchor_set(shape, domains, seed):
    g = _gen(seed + 5)
    c = torch.randn(domains, shape.d_model, generator=g, device="cuda")
    a = c.repeat_interleave(ANCHORS_PER_DOMAIN, 0)
    a = a + 0.5 * torch.randn(a.shape, generator=g, device="cuda")
    q = c[seed % domains] + 0.5 * torch.randn(shape.d_model, generator=g, device="cuda")
    return (a / a.norm(dim=1, keepdim=True)).contiguous(), q.contiguous()


def _model(case, seed):
    shape = _shape(case)
    return shape, si.make_model_weights(shape, seed, device="cuda", gain_spread=0.1)


def _logits(case, seed):
    """Logits of the spread a random-init model gives; the draft model's follow the full model's."""
    g = _gen(seed)
    rows = case.get("k", 0) + 1
    p = 1.4 * torch.randn(rows, case["vocab"], generator=g, device="cuda")
    q = p + 0.3 * torch.randn(p.shape, generator=g, device="cuda")
    return p.contiguous(), q[:rows - 1].contiguous()


def _vectors(case, seed):
    g = _gen(seed)
    n, d = case["domains"], case["d"]
    c = torch.randn(n, d, generator=g, device="cuda").repeat_interleave(case["per"], 0)
    x = (c + 0.5 * torch.randn(c.shape, generator=g, device="cuda")).contiguous()
    return x, x[:n].contiguous()


def _session(case, shape, w, seed, max_seq, anchors=None):
    kw = {}
    if anchors is not None:
        n = anchors.shape[0] // ANCHORS_PER_DOMAIN
        kw = {"anchors": anchors, "skip_masks": np.stack([_mask(shape, seed + i) for i in range(n)]), "anchors_per_domain": ANCHORS_PER_DOMAIN}
    return kb.Session.from_shape(shape, w, max_seq, max_draft=15, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "round":
        p, q = _logits(case, seed)
        u = si.uniforms(seed, 3, case["k"] + 1)
        return {"case": case, "p": p, "q": q, "drafts": q.argmax(dim=1).cpu().numpy(), "u": u}
    if kind == "pick":
        return {"case": case, "p": _logits(case, seed)[0], "u": float(si.uniforms(seed, 3, 1)[0])}
    if kind == "anchors":
        x, start = _vectors(case, seed)
        return {"case": case, "x": x, "start": start}
    shape, w = _model(case, seed)
    st = {"case": case}
    if kind == "select":
        anchors, st["query"] = _anchor_set(shape, case["domains"], seed)
        st["session"] = _session(case, shape, w, seed, 64, anchors)
        return st
    prompt, rows = _tokens(case, shape, seed)
    st["prompt"], st["pending"], st["drafts"] = prompt, int(rows[0]), rows[1:]
    anchors = _anchor_set(shape, 5, seed)[0] if kind == "request" else None
    s = st["session"] = _session(case, shape, w, seed, len(prompt) + 64, anchors)
    if kind in ("draft", "verify"):
        s.prefill(prompt)
        s.set_skipmask(_mask(shape, seed))
        s.set_pending(st["pending"])
    return st


# ---- one pass ------------------------------------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "select":
        return list(st["session"].select_skipset(st["query"]))
    if kind == "round":
        p = kb.knnssd_filtered_probs(st["p"], case["temperature"], case["top_p"])
        q = kb.knnssd_filtered_probs(st["q"], case["temperature"], case["top_p"])
        kept, token = kb.knnssd_spec_accept(p, q, st["drafts"], st["u"][:-1], st["u"][-1])
        return {"p": p, "q": q, "kept": kept, "token": token}
    if kind == "pick":
        p = kb.knnssd_filtered_probs(st["p"], case["temperature"], case["top_p"])
        return {"p": p, "token": kb.knnssd_sample_token(p[0], st["u"])}
    if kind == "anchors":
        r = kb.knnssd_build_anchors(st["x"], st["start"], 50, ANCHORS_PER_DOMAIN)
        return {k: r[k] for k in ("labels", "centroids", "anchors", "rounds")}
    s = st["session"]
    if kind == "draft":
        tokens, logits = s.draft(1, want_logits=True)
        return {"tokens": tokens, "logits": logits}
    if kind == "verify":
        s.set_length(len(st["prompt"]))          # a pass commits its rows: the next one starts from the same context
        s.set_pending(st["pending"])
        return s.verify(st["drafts"], want_logits=True, want_hidden=True)
    first, pooled = s.prefill(st["prompt"], want_pooled=True)
    if kind == "prompt":
        return {"first": first, "pooled": pooled}
    # a greedy token is the arg-max of logits that a full-depth model gives to ~1e-2 only: the pending token and the
    # drafts are given, and the logits are returned in the place of the tokens
    s.select_skipset()
    s.set_pending(st["pending"])
    draft_logits = s.draft(1, want_logits=True)[1]
    logits = s.verify(st["drafts"], want_logits=True)["logits"]
    return {"pooled": pooled, "draft_logits": draft_logits, "logits": logits}


# ---- what a pass cannot do without ---------------------------------------------------------------------------------
def _pass_work(shape, rows, context, mask=None, head_rows=None):
    b = 2 if shape.dtype == "bf16" else 4
    d, hd = shape.d_model, shape.head_dim
    keep = lambda j: mask is None or not mask[j]  # noqa: E731
    n_attn = sum(1 for l in range(shape.n_layers) if keep(2 * l))
    n_mlp = sum(1 for l in range(shape.n_layers) if keep(2 * l + 1))
    weights = n_attn * 2 * d * hd * (shape.n_heads + shape.n_kv_heads) + n_mlp * 3 * d * shape.d_ff
    head_rows = rows if head_rows is None else head_rows
    kv = n_attn * 2 * shape.n_kv_heads * hd
    seen = sum(context + r + 1 for r in range(rows))            # (row, position) pairs attention looks at
    return {"bytes": b * (weights + shape.vocab * d + kv * (context + rows) + rows * d) + 4 * head_rows * shape.vocab,
            "flops": 2 * rows * weights + 2 * head_rows * shape.vocab * d + 4 * n_attn * shape.n_heads * hd * seen}


def work(case):
    kind = case["kind"]
    if kind == "select":
        n = case["domains"] * ANCHORS_PER_DOMAIN * _shape(case).d_model
        return {"bytes": 4 * n, "flops": 2 * n}
    if kind == "round":
        n = (2 * case["k"] + 1) * case["vocab"]
        return {"bytes": 8 * n, "flops": 4 * n}
    if kind == "pick":
        return {"bytes": 8 * case["vocab"], "flops": 4 * case["vocab"]}
    if kind == "anchors":                                        # at least one assignment and one mean of every point
        n = case["domains"] * case["per"] * case["d"]
        return {"bytes": 4 * n, "flops": 3 * n * case["domains"]}
    shape = _shape(case)
    if kind == "draft":
        return _pass_work(shape, 1, case["context"], _mask(shape, 0))
    if kind == "verify":
        return _pass_work(shape, case["k"] + 1, case["context"])
    w = _pass_work(shape, case["rows"], 0, head_rows=1)
    if kind == "request":
        for more in (_pass_work(shape, 1, case["rows"], _mask(shape, 0)), _pass_work(shape, case["k"] + 1, case["rows"])):
            w = {k: w[k] + more[k] for k in w}
    return w


def tolerance(case):
    kind = case["kind"]
    if kind in ("select", "round", "pick"):
        return {"rel": 5e-6}                                     # 32-bit sums
    if kind == "anchors":
        return {"rel": 1e-9}                                     # centroids are summed in 64 bits
    if case["shape"] == "tiny":
        return {"rel": 1e-5}
    # bf16 K and V: an entry that rounds the other way is off by 4e-3 of itself, and more of them do with every
    # layer: 1e-3 against 64 bits at 8 layers, 2.6e-3 at 32
    return {"rel": 1e-2} if kind == "request" else {"rel": 4e-3}


# ---- the same in 64 bits -------------------------------------------------------------------------------------------
def _map64(x, w):
    out = torch.empty(x.shape[0], w.shape[0], dtype=torch.float64, device=x.device)
    for r in range(0, w.shape[0], 16384):
        out[:, r:r + 16384] = x @ w[r:r + 16384].double().T
    return out


def _norm64(x, gain, eps):
    return x * torch.rsqrt((x * x).mean(dim=1, keepdim=True) + eps) * gain.double()


def _rope64(x, pos, theta):
    half = x.shape[-1] // 2
    ang = pos[:, None].double() * theta ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


def _pass64(shape, w, cache, tokens, pos0, mask=None):
    """Hidden states after the final norm of the rows `tokens` at positions pos0 ..; cache[l] = (K, V) is extended."""
    tok = torch.as_tensor(np.asarray(tokens), dtype=torch.int64, device="cuda")
    T, hd, group = tok.numel(), shape.head_dim, shape.n_heads // shape.n_kv_heads
    pos = torch.arange(pos0, pos0 + T, device="cuda")
    stored = lambda t: t.to(torch.bfloat16).double() if shape.dtype == "bf16" else t  # noqa: E731
    x = w["tok_embed"][tok].double()
    for l in range(shape.n_layers):
        if mask is None or not mask[2 * l]:
            h = _norm64(x, w["attn_norm"][l], shape.rms_eps)
            q = _rope64(_map64(h, w["wq"][l]).view(T, -1, hd), pos, shape.rope_theta)
            k = stored(_rope64(_map64(h, w["wk"][l]).view(T, -1, hd), pos, shape.rope_theta))
            v = stored(_map64(h, w["wv"][l]).view(T, -1, hd))
            if l in cache:
                k, v = torch.cat([cache[l][0][:pos0], k]), torch.cat([cache[l][1][:pos0], v])
            if mask is None:
                cache[l] = (k, v)
            hide = torch.arange(pos0 + T, device="cuda")[None] > pos[:, None]
            o = torch.empty(T, shape.n_heads, hd, dtype=torch.float64, device="cuda")
            for i in range(shape.n_heads):
                sc = (q[:, i] @ k[:, i // group].T / math.sqrt(hd)).masked_fill(hide, -math.inf)
                o[:, i] = sc.softmax(dim=1) @ v[:, i // group]
            x = x + _map64(o.view(T, -1), w["wo"][l])
        if mask is None or not mask[2 * l + 1]:
            h = _norm64(x, w["mlp_norm"][l], shape.rms_eps)
            gate = _map64(h, w["w_gate"][l])
            x = x + _map64(gate * torch.sigmoid(gate) * _map64(h, w["w_up"][l]), w["w_down"][l])
    return _norm64(x, w["final_norm"], shape.rms_eps)


def _filtered64(logits, temperature, top_p):
    p = (logits.double() / temperature).softmax(dim=1)
    order = torch.sort(p, dim=1, descending=True, stable=True)
    keep = order.values.cumsum(dim=1) - order.values < top_p
    p = p * torch.zeros_like(p).scatter(1, order.indices, keep.double())
    return p / p.sum(dim=1, keepdim=True)


def _clusters64(x, start):
    x, mu, labels, rounds = x.double(), start.double(), None, 0
    while rounds < 50:
        dist = torch.stack([(x - m).square().sum(dim=1) for m in mu], dim=1)
        new = dist.argmin(dim=1)
        rounds += 1
        if labels is not None and torch.equal(new, labels):
            break
        labels = new
        for c in range(len(mu)):
            if (labels == c).any():
                mu[c] = x[labels == c].mean(dim=0)
    return mu


def exact(case, seed):
    kind = case["kind"]
    if kind == "round":
        p, q = _logits(case, seed)
        return {"p": _filtered64(p, case["temperature"], case["top_p"]), "q": _filtered64(q, case["temperature"], case["top_p"]), "kept": None, "token": None}
    if kind == "pick":
        return {"p": _filtered64(_logits(case, seed)[0], case["temperature"], case["top_p"]), "token": None}
    if kind == "anchors":
        return {"labels": None, "centroids": _clusters64(*_vectors(case, seed)), "anchors": None, "rounds": None}
    if kind == "select":
        anchors, query = (t.double() for t in _anchor_set(_shape(case), case["domains"], seed))
        return [None, None, float((anchors @ query / anchors.norm(dim=1) / query.norm()).max())]
    shape, w = _model(case, seed)
    prompt, rows = _tokens(case, shape, seed)
    cache, n = {}, len(prompt)
    hidden = _pass64(shape, w, cache, prompt, 0)
    if kind == "prompt":
        return {"first": None, "pooled": hidden.mean(dim=0)}
    mask = _mask(shape, seed)
    if kind == "draft":
        return {"tokens": None, "logits": _map64(_pass64(shape, w, cache, rows[:1], n, mask), w["lm_head"])}
    if kind == "request":
        pooled = hidden.mean(dim=0)
        anchors = _anchor_set(shape, 5, seed)[0].double()
        best = int((anchors @ pooled / anchors.norm(dim=1)).argmax())
        drafted = _map64(_pass64(shape, w, cache, rows[:1], n, _mask(shape, seed + best // ANCHORS_PER_DOMAIN)), w["lm_head"])
        return {"pooled": pooled, "draft_logits": drafted, "logits": _map64(_pass64(shape, w, cache, rows, n), w["lm_head"])}
    hidden = _pass64(shape, w, cache, rows, n)
    return {"n_accepted": None, "next_token": None, "logits": _map64(hidden, w["lm_head"]), "hidden": hidden}
