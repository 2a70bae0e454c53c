"""Performance cases of the ConfLayers hot path: what a program that decodes with this library has it do.

Every case goes through the public binding (`paper_2604_14612_b200.Context` and the context-free scoring call).  The
kinds of work are

  cycle     one draft / verify / accept cycle driven by the caller, which looks at the logits (a server that samples or
            streams tokens itself)
  draft     the draft half of a cycle alone: K single-row steps through the kept layers
  verify    the verify half alone: one (K + 1)-row pass of the whole model
  generate  the library's own loop (K = 0: plain decoding), then the logits of the position after the last token
  prompt    a new prompt into an empty cache, then the logits of the position after its first token
  search    a new prompt with hidden-state taps, then the confidences of all layers on the tapped positions: the step
            with which the layer search begins on an input
  scores    confidences of hidden rows that the caller holds
  rounds    the search rounds of one input: score all layers on each round's hidden states, select a skip set
  static    confidences of hidden rows through the call that allocates nothing

Sizes are those of this repository's workloads (4-layer fp32 model, 12-layer bf16 model, layers of width 4096 and 5120,
32 layers for the headline model and 8 elsewhere, all-layer scoring over 32 x 64 rows), with ragged prompts and context
lengths, grouped-query attention, fp16 storage and the 128256-token vocabulary as its tests have them.

Weights are random with one property of a trained model put in: the head's row of token v + 1 leans towards the embedding
of token v, so that the next token is predicted with a probability of some tens of per cent and drafts are mostly accepted.
With unstructured weights the two largest logits lie closer together than the rounding of a 16-bit cache and no two
correct implementations would emit the same tokens.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2604_14612_b200 as cl

DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
STD = 0.02
EPS = 1e-5
THETA = 10000.0
LOGIT_STD = 1.28      # spread of the head's logits (N(0, 0.02) rows of 4096 elements on a normalised row)
NEXT_LOGIT = 12.0     # logit that the head gives the embedded token's successor


def _model(layers, d, heads, ffn, vocab, dtype="bf16", kv_heads=None):
    return dict(layers=layers, d=d, heads=heads, kv_heads=kv_heads or heads, ffn=ffn, vocab=vocab, dtype=dtype)


def _tiny():
    return _model(4, 256, 4, 688, 1024, "fp32")


def _small(layers=12, dtype="bf16"):
    return _model(layers, 768, 12, 2048, 32000, dtype)


def _wide(layers=8, dtype="bf16", kv_heads=32, vocab=32000):
    return _model(layers, 4096, 32, 11008, vocab, dtype, kv_heads)


def _wider(layers=8, dtype="bf16"):
    return _model(layers, 5120, 40, 13824, 32000, dtype)


def listed():
    return [
        # the smallest calls: a 4-layer fp32 model, all launches and latency
        dict(name="cycle_fp32_tiny", kind="cycle", ctx=24, K=4, skip=1, **_tiny()),
        # a 12-layer bf16 model whose layers take a few microseconds each
        dict(name="cycle_bf16_12layers", kind="cycle", ctx=200, K=4, skip=3, **_small()),
        # the two halves of the headline cycle: 32 layers of width 4096, 18 of them kept while drafting
        dict(name="draft_k4_32layers", kind="draft", ctx=640, K=4, skip=14, **_wide(32)),
        dict(name="verify_k4_32layers", kind="verify", ctx=640, K=4, **_wide(32)),
        # the widest verify pass, a ragged context, grouped-query attention, fp16 storage
        dict(name="verify_k8_grouped_fp16", kind="verify", ctx=1003, K=8, **_wide(8, "fp16", 8)),
        # the library's own loop on the wider model
        dict(name="generate_k6_wider", kind="generate", ctx=1024, K=6, skip=3, tokens=32, **_wider()),
        # prompts: short and ragged (a zero-shot question), a few-shot prompt, a long one
        dict(name="prompt_61_grouped_fp16", kind="prompt", n=61, **_wide(8, "fp16", 8)),
        dict(name="prompt_512", kind="prompt", n=512, **_wide()),
        dict(name="prompt_1024_wider", kind="prompt", n=1024, **_wider()),
        # the start of the layer search on a new input
        dict(name="search_333", kind="search", n=333, P=32, **_wide()),
        # all-layer scoring, 8 rounds over 32 layers x 64 positions
        dict(name="rounds_8x32x64", kind="rounds", iters=8, P=64, skip=14, **_wide(32)),
        # one layer's context window of 100 positions, scored without allocating
        dict(name="static_100", kind="static", rows=1, P=100, **_wide(1)),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["cycle", "draft", "verify", "generate", "prompt", "prompt", "search", "scores", "rounds", "static"])
    dtype = rng.choice(["bf16", "bf16", "fp16"])
    size = rng.choice(["small", "wide", "wide", "wider"])
    if size == "small":
        m = _small(rng.randint(3, 12), dtype)
    elif size == "wide":
        m = _wide(rng.randint(2, 8), dtype, rng.choice([32, 32, 8]), rng.choice([32000, 32000, 128256]))
    else:
        m = _wider(rng.randint(2, 8), dtype)
    if kind in ("cycle", "draft", "verify", "generate"):
        if kind == "cycle" and rng.random() < 0.3:
            m = _tiny()
        top = 100 if m["layers"] == 4 and m["d"] == 256 else 1100
        c = dict(kind=kind, ctx=_log_int(rng, 12, top), K=rng.randint(1, 8), **m)
        if kind != "verify":
            c["skip"] = rng.randint(0, max(0, m["layers"] // 2))
        if kind == "generate":
            c["K"] = rng.choice([0, c["K"], c["K"]])
            c["tokens"] = rng.randint(4, 18)
        return c
    if kind == "prompt":
        return dict(kind=kind, n=_log_int(rng, 3, 1024), **m)
    if kind == "search":
        P = rng.randint(4, 64)
        return dict(kind=kind, n=_log_int(rng, P + 1, 1024), P=P, **m)
    m["layers"] = rng.randint(3, 32)
    if rng.random() < 0.3:
        m["vocab"] = 5003
    if kind == "rounds":
        m["layers"] = max(8, m["layers"])
        return dict(kind=kind, iters=rng.randint(1, 8), P=_log_int(rng, 4, 50), skip=rng.randint(1, m["layers"] - 4), **m)
    if kind == "static":
        m["dtype"] = "bf16"
        return dict(kind=kind, rows=1, P=_log_int(rng, 1, 400), **m)
    return dict(kind=kind, rows=rng.randint(1, m["layers"]), P=_log_int(rng, 1, 100), **m)


# ---- inputs ------------------------------------------------------------------------------------------------------


def _normal(gen, shape, std, dtype):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype).mul_(std)


def _stream_rms(c):
    """RMS of what the random layers add to the residual stream, roughly (sizes the embedding)."""
    z = np.linspace(-6, 6, 1201)
    w = np.exp(-z * z / 2)
    g = STD * math.sqrt(c["d"]) * z
    silu = g / (1 + np.exp(-g))
    ffn = STD * math.sqrt(c["ffn"]) * STD * math.sqrt(c["d"]) * math.sqrt(float((w * silu * silu).sum() / w.sum()))
    att = 0.4 * (STD * math.sqrt(c["d"])) ** 2
    return math.sqrt(c["layers"] * (ffn * ffn + att * att))


def _head(c, gen):
    """(unit-variance token vectors [V, d], head [V, d], final gain): the head's row of token v + 1 is token v's vector."""
    e = torch.randn((c["vocab"], c["d"]), generator=gen, device="cuda", dtype=torch.float32)
    head = (torch.roll(e, 1, 0) * (LOGIT_STD / math.sqrt(c["d"]))).to(DTYPES[c["dtype"]])
    gain = 1.0 + 0.1 * torch.randn((c["d"],), generator=gen, device="cuda", dtype=torch.float32)
    return e, head, gain


def _weights(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 1)
    dt, d, F, L = DTYPES[c["dtype"]], c["d"], c["ffn"], c["layers"]
    kvd = c["kv_heads"] * (d // c["heads"])
    e, head, gain = _head(c, gen)
    rho = min(0.8, NEXT_LOGIT / (LOGIT_STD * math.sqrt(d)))
    w = dict(embed=(e * (rho / math.sqrt(1 - rho * rho) * _stream_rms(c))).to(dt), lm_head=head, final_norm=gain)
    del e
    dims = dict(wq=(d, d), wk=(kvd, d), wv=(kvd, d), wo=(d, d), wg=(F, d), wu=(F, d), wd=(d, F))
    for n, shape in dims.items():
        w[n] = [_normal(gen, shape, STD, dt) for _ in range(L)]
    for n in ("norm1", "norm2"):
        w[n] = [1.0 + 0.1 * torch.randn((d,), generator=gen, device="cuda", dtype=torch.float32) for _ in range(L)]
    return w


def _tokens(c, seed, n):
    return np.random.RandomState(seed % (1 << 31)).randint(0, c["vocab"], n).astype(np.int32)


def _skip_mask(c):
    """`skip` layers spread evenly, first and last layer left out."""
    L, S = c["layers"], min(c.get("skip", 0), max(0, c["layers"] - 2))
    m = np.zeros(L, np.uint8)
    for i in range(S):
        m[1 + (i * (L - 2)) // max(1, S)] = 3
    return m


def _drafts(c, seed, t0):
    """Candidates of a verify pass: the first half follows the model, the others do not."""
    t = (t0 + 1 + np.arange(c["K"])) % c["vocab"]
    bad = _tokens(c, seed + 5, c["K"])
    t[(c["K"] + 1) // 2:] = bad[(c["K"] + 1) // 2:]
    return t.astype(np.int32)


def _hidden(c, seed, n, P, e):
    """n x P hidden rows of the storage type: layer l's rows lean towards a token's vector, later layers more so."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 3)
    rs = np.random.RandomState((seed + 17) % (1 << 31))
    want = 9.5 + 5.0 * np.arange(n) / max(1, n) + rs.uniform(-1, 1, n)      # the leading logit of the row, by layer
    rho = torch.tensor(np.minimum(0.9, want / (LOGIT_STD * math.sqrt(c["d"]))), device="cuda", dtype=torch.float32)
    tok = torch.randint(0, c["vocab"], (n, P), generator=gen, device="cuda")
    x = e[tok] * rho[:, None, None]
    x += torch.randn((n, P, c["d"]), generator=gen, device="cuda") * torch.sqrt(1 - rho * rho)[:, None, None]
    return (3.0 * x).to(DTYPES[c["dtype"]]).contiguous()


def _select_cfg(c):
    # w_max given: counting the layers that share the first one's value has no meaning on these inputs
    return cl.SelectCfg.make(1, c["layers"] - 2, n_skip=c["skip"], w_max=4.0)


def prepare(case, seed):
    c, s = case, dict(case=case)
    kind = c["kind"]
    if kind in ("scores", "rounds", "static"):
        gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 1)
        e, head, gain = _head(c, gen)
        if kind == "rounds":
            s["hidden"] = [_hidden(c, seed * 31 + i, c["layers"], c["P"], e) for i in range(c["iters"])]
            s["scores"] = np.random.RandomState(seed % (1 << 31)).uniform(0, 4, c["iters"]).astype(np.float32)
            s["cfg"] = _select_cfg(c)
        else:
            s["hidden"] = _hidden(c, seed * 31, c["rows"], c["P"], e)
        if kind == "static":
            s["head"], s["gain"] = head, gain
        else:
            s["ctx"] = cl.Context(c["layers"], c["d"], c["heads"], c["ffn"], c["vocab"], 8, c["dtype"], EPS, THETA)
            s["ctx"].cl_load(dict(lm_head=head, final_norm=gain), head_only=True)
        return s
    n = c["n"] if kind in ("prompt", "search") else c["ctx"]
    room = n + c.get("tokens", 0) + 16
    s["ctx"] = cl.Context(c["layers"], c["d"], c["heads"], c["ffn"], c["vocab"], room, c["dtype"], EPS, THETA,
                          tap_positions=c.get("P", 0), n_kv_heads=c["kv_heads"])
    s["ctx"].cl_load(_weights(c, seed))
    s["tokens"] = _tokens(c, seed + 3, n)
    if kind not in ("prompt", "search"):
        s["t0"] = s["ctx"].cl_prefill(s["tokens"])
        s["ctx"].cl_set_skip_set(_skip_mask(c))
        if kind == "verify":
            s["drafts"] = _drafts(c, seed, s["t0"])
    return s


# ---- the work ----------------------------------------------------------------------------------------------------


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "static":
        return cl.cl_layer_confidences_static(state["head"], state["gain"], state["hidden"], EPS)
    ctx = state["ctx"]
    if kind == "scores":
        r = ctx.cl_layer_confidences(state["hidden"])
        return dict(conf=r["conf"], p_max=r["p_max"], argmax=r["argmax"])
    if kind == "rounds":
        r = ctx.cl_score_loop(state["cfg"], state["hidden"], state["scores"])
        return dict(c_layers=r["c_layers"], masks=r["masks"])
    if kind == "prompt":
        first = ctx.cl_prefill(state["tokens"])
        v = ctx.cl_verify(1, want_logits=True)
        return dict(first=first, target=v["targets"], logits=v["logits"])
    if kind == "search":
        first = ctx.cl_prefill(state["tokens"], tap_hidden=True)
        r = ctx.cl_layer_confidences()
        return dict(first=first, conf=r["conf"], p_max=r["p_max"])
    ctx.cl_rollback(c["ctx"], state["t0"])
    if kind == "generate":
        toks, _ = ctx.cl_generate(c["K"], c["tokens"])
        ctx.cl_rollback(c["ctx"] + c["tokens"], int(toks[-1]))     # the last cycle may have committed more than was asked for
        v = ctx.cl_verify(1, want_logits=True)
        return dict(tokens=toks, target=v["targets"], logits=v["logits"])
    out = {}
    if kind in ("cycle", "draft"):
        d = ctx.cl_draft(c["K"], want_logits=True)
        out.update(draft_tokens=d["tokens"], draft_logits=d["logits"])
    else:
        ctx.cl_force_tokens(state["drafts"])
    if kind in ("cycle", "verify"):
        v = ctx.cl_verify(c["K"] + 1, want_logits=True)
        out.update(targets=v["targets"], logits=v["logits"])
    if kind == "cycle":
        n, emitted = ctx.cl_accept()
        out.update(accepted=n, emitted=emitted)
    return out


def work(case):
    c = case
    kind, es = c["kind"], 4 if c["dtype"] == "fp32" else 2
    d, F, V, L = c["d"], c["ffn"], c["vocab"], c["layers"]
    kvd = c["kv_heads"] * (d // c["heads"])
    per_layer = 2 * d * d + 2 * kvd * d + 3 * d * F
    head = V * d
    if kind in ("scores", "rounds", "static"):
        rows = (L if kind == "rounds" else c["rows"]) * c["P"]
        it = c.get("iters", 1)
        # (the head is read once for all rounds' worth of rows: nothing forces it to be read again)
        return dict(bytes=head * es + it * rows * (d * es + 12), flops=2.0 * it * rows * head)
    kv_pos = 2 * kvd * es                       # cached bytes of one position of one layer

    def passes(n_pass, layers, rows, ctx):
        att = 4.0 * rows * (ctx + rows / 2) * d
        return (n_pass * (layers * (per_layer * es + (ctx + rows) * kv_pos) + head * es + rows * V * 4),
                n_pass * (2.0 * rows * (layers * per_layer + head) + layers * att))

    kept = L - int((_skip_mask(c) == 3).sum())
    b = f = 0.0
    if kind in ("prompt", "search"):
        n = c["n"]
        b = L * (per_layer * es + n * kv_pos) + head * es
        f = 2.0 * n * L * per_layer + 2.0 * head + L * 2.0 * n * n * d
        if kind == "prompt":
            b2, f2 = passes(1, L, 1, n)
        else:
            rows = L * c["P"]
            b2, f2 = head * es + rows * (d * es + 8), 2.0 * rows * head
        return dict(bytes=b + b2, flops=f + f2)
    if kind == "generate":
        K, n = c["K"], c["tokens"]
        cycles = n if K == 0 else -(-n // (K + 1))      # as few as can emit n tokens
        b, f = passes(cycles, L, K + 1, c["ctx"])
        b1, f1 = passes(cycles * K, kept, 1, c["ctx"])
        b2, f2 = passes(1, L, 1, c["ctx"] + n)
        return dict(bytes=b + b1 + b2, flops=f + f1 + f2)
    if kind in ("cycle", "draft"):
        b, f = passes(c["K"], kept, 1, c["ctx"])
    if kind in ("cycle", "verify"):
        b1, f1 = passes(1, L, c["K"] + 1, c["ctx"])
        b, f = b + b1, f + f1
    return dict(bytes=b, flops=f)


def tolerance(case):
    """Relative errors measured against exact(): bf16 models 5e-4 .. 1.3e-3 in the logits, 3e-4 .. 8e-4 in a row's confidence,
    6e-5 in a mean over 64 rows; fp16 8e-5 .. 2.3e-4 (the cache's and the normalised rows' storage type decides); fp32 models and
    the static call, whose activations stay fp32, 2e-7 .. 1.2e-6.  Four times that and more, rounded."""
    kind, half = case["kind"], case["dtype"] == "fp16"
    if case["dtype"] == "fp32" or kind == "static":
        return dict(rel=1e-5)
    if kind == "rounds":
        return dict(rel=1e-4 if half else 5e-4, differ=0.01)      # two layers at the edge of the selection may trade places
    if kind in ("scores", "search"):
        return dict(rel=5e-4 if half else 3e-3)
    return dict(rel=1e-3 if half else 5e-3)


# ---- the same in 64 bits -------------------------------------------------------------------------------------------


class _Exact:
    """Llama-style decoder in fp64; keys, values and taps are rounded to the storage type, which is part of the model."""

    def __init__(self, c, seed):
        self.c, self.w = c, _weights(c, seed)
        self.hd = c["d"] // c["heads"]
        self.k = [torch.empty((0, c["kv_heads"], self.hd), device="cuda", dtype=torch.float64) for _ in range(c["layers"])]
        self.v = [t.clone() for t in self.k]

    def stored(self, x):
        return x.to(DTYPES[self.c["dtype"]]).double()

    @staticmethod
    def norm(x, g):
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * g.double()

    def rope(self, x, pos):
        half = self.hd // 2
        inv = THETA ** (-2.0 * torch.arange(half, device="cuda", dtype=torch.float64) / self.hd)
        a = pos.double()[:, None] * inv
        cos, sin = a.cos()[:, None, :], a.sin()[:, None, :]
        p, q = x[..., :half], x[..., half:]
        return torch.cat([p * cos - q * sin, q * cos + p * sin], -1)

    def rows(self, tokens, pos0, mask=None, taps=None):
        """The normalised last rows [T, d] after a pass over `tokens` at pos0 ..; cached rows past pos0 are dropped."""
        c, w, hd = self.c, self.w, self.hd
        t = torch.as_tensor(np.asarray(tokens), device="cuda", dtype=torch.long)
        T = t.shape[0]
        pos = torch.arange(pos0, pos0 + T, device="cuda")
        x = w["embed"][t].double()
        for l in range(c["layers"]):
            if mask is not None and mask[l] == 3:
                continue
            xn = self.norm(x, w["norm1"][l])
            q = self.rope((xn @ w["wq"][l].double().T).view(T, c["heads"], hd), pos)
            k = self.stored(self.rope((xn @ w["wk"][l].double().T).view(T, c["kv_heads"], hd), pos))
            v = self.stored((xn @ w["wv"][l].double().T).view(T, c["kv_heads"], hd))
            self.k[l], self.v[l] = torch.cat([self.k[l][:pos0], k]), torch.cat([self.v[l][:pos0], v])
            g = c["heads"] // c["kv_heads"]
            K, V = (a.repeat_interleave(g, 1).transpose(0, 1) for a in (self.k[l], self.v[l]))
            s = q.transpose(0, 1) @ K.transpose(1, 2) / math.sqrt(hd)
            s = s.masked_fill(torch.arange(K.shape[1], device="cuda")[None, :] > pos[:, None], -math.inf)
            x = x + (torch.softmax(s, -1) @ V).transpose(0, 1).reshape(T, -1) @ w["wo"][l].double().T
            xn = self.norm(x, w["norm2"][l])
            h = torch.nn.functional.silu(xn @ w["wg"][l].double().T) * (xn @ w["wu"][l].double().T)
            x = x + h @ w["wd"][l].double().T
            if taps is not None:
                taps.append(self.stored(x))
        return self.norm(x, w["final_norm"])

    def logits(self, tokens, pos0, mask=None, last=False):
        r = self.rows(tokens, pos0, mask)
        return (r[-1:] if last else r) @ self.w["lm_head"].double().T


def _exact_scores(hidden, head, gain):
    """(conf, p_max, argmax) of rows [n, d]: softmax of the clamped early-exit logits, 1 - H / log V."""
    conf, pm, am = [], [], []
    W = head.double()
    for i in range(0, hidden.shape[0], 1024):
        lg = (_Exact.norm(hidden[i:i + 1024].double(), gain) @ W.T).clamp(-1e4, 1e4)
        lp = torch.log_softmax(lg, -1)
        conf.append(1 + (lp.exp() * lp).sum(-1) / math.log(head.shape[0]))
        pm.append(lp.max(-1).values.exp())
        am.append(lg.argmax(-1))
    return torch.cat(conf), torch.cat(pm), torch.cat(am)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("scores", "rounds", "static"):
        gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 1)
        e, head, gain = _head(c, gen)
        if kind == "rounds":
            cls = []
            for i in range(c["iters"]):
                h = _hidden(c, seed * 31 + i, c["layers"], c["P"], e)
                conf, _, _ = _exact_scores(h.view(-1, c["d"]), head, gain)
                cls.append(conf.view(c["layers"], c["P"]).mean(1))
            return dict(c_layers=torch.stack(cls), masks=None)
        h = _hidden(c, seed * 31, c["rows"], c["P"], e)
        r = _exact_scores(h.view(-1, c["d"]), head, gain)
        shape = (c["rows"], c["P"])
        return dict(conf=r[0].view(shape), p_max=r[1].view(shape), argmax=r[2].view(shape))
    m = _Exact(c, seed)
    n = c["n"] if kind in ("prompt", "search") else c["ctx"]
    prompt = _tokens(c, seed + 3, n)
    if kind == "search":
        taps = []
        r = m.rows(prompt, 0, taps=taps)
        first = int((r[-1] @ m.w["lm_head"].double().T).argmax())
        P = c["P"]
        slots = torch.as_tensor([p for _, p in sorted((p % P, p) for p in range(n - P, n))], device="cuda")
        h = torch.stack([t[slots] for t in taps]).view(-1, c["d"])
        conf, pm, _ = _exact_scores(h, m.w["lm_head"], m.w["final_norm"])
        return dict(first=first, conf=conf.view(-1, P), p_max=pm.view(-1, P))
    t0 = int(m.logits(prompt, 0, last=True).argmax())
    if kind == "prompt":
        lg = m.logits([t0], n)
        return dict(first=t0, target=lg.argmax(-1).cpu().numpy(), logits=lg)
    if kind == "generate":      # greedy decoding with the full model: what speculation has to reproduce
        toks = [t0]
        for i in range(c["tokens"]):
            toks.append(int(m.logits([toks[-1]], n + i).argmax()))
        lg = m.logits([toks[-1]], n + c["tokens"])
        return dict(tokens=np.array(toks[1:]), target=lg.argmax(-1).cpu().numpy(), logits=lg)
    out = {}
    if kind in ("cycle", "draft"):
        t, rows, mask = [t0], [], _skip_mask(c)
        for i in range(c["K"]):
            rows.append(m.logits([t[-1]], n + i, mask))
            t.append(int(rows[-1].argmax()))
        drafts = np.array(t[1:])
        out.update(draft_tokens=drafts, draft_logits=torch.cat(rows))
    else:
        drafts = _drafts(c, seed, t0)
    if kind in ("cycle", "verify"):
        lg = m.logits(np.concatenate([[t0], drafts]), n)
        targets = lg.argmax(-1).cpu().numpy()
        out.update(targets=targets, logits=lg)
    if kind == "cycle":
        acc = 0
        while acc < c["K"] and drafts[acc] == targets[acc]:
            acc += 1
        out.update(accepted=acc, emitted=np.concatenate([drafts[:acc], targets[acc:acc + 1]]))
    return out
