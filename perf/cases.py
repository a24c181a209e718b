"""The work that users of this framework have it do, as cases that can be timed and compared.

Every case goes through the package's public entry points (SpdContext and the batched calls) on seeded inputs: weights
N(0, 0.02), RMSNorm gains 1 + N(0, 0.1), n-gram tables counted over a Zipf stream, prefixes of Zipf-distributed
tokens.  Model shapes, draft counts, prefix and generation lengths are those of the named workloads (tiny, 7b, 13b;
prefixes of 15, 64 and 2048 tokens, drafts of 10 tokens) and of the tests and the batch benchmark.  The weights and the
tables of a shape are kept between preparations, as a serving program keeps them; a prefix, a context and its cache
are made anew for each.

Kinds of case:
  request   spd_prefill on a new prefix, then one spd_step per token: a client that shows the drafts as they grow
  generate  spd_prefill, then the remaining tokens with one spd_generate
  prefill   spd_prefill alone: the time to the first drafts
  decode    spd_generate on a context that already holds its prefix; the context goes on from where it is and takes
            its prefix again once its positions have run out
  sample    spd_prefill, then a nucleus-sampled continuation that ends in fresh drafts (spd_sample)
  batch     several requests of different prefix lengths over the same weights, stepped together (spd_batch_generate);
            they go on from where they are, as `decode`
Outputs are the logits of the last pass (of every request of a batch), which hang on every earlier choice, and the
sampled ids (the order of two drafts of nearly the same probability is no property of a correct program).  With random
weights the logits are flat, and a temperature of 0.06 makes the drafts' weights, and with them the next input, hang on
the last bits of the logits: two correct programs drift apart within a few timesteps.  So the temperature is 1, and
cases of several timesteps use the float32 cache (a bf16 one rounds a value in a hundred the other way).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_18400_b200 as P
import spd_inputs as si

DEVICE = "cuda:0"
ALPHA, DELTA = 0.54, 0.01                     # the workloads' values
TAU = 1.0                                     # the workloads' 0.06 suits a trained model: see below
LAMBDA = (0.01, 0.04, 0.15, 0.18, 0.12)       # orders 2..6
TOP_P, TEMPERATURE = 0.9, 0.2                  # of the nucleus sampler
ROPE_THETA, RMS_EPS = 10000.0, 1e-5


def listed():
    return [
        # the smallest model and prefix: latency of single launches and of the host path
        {"name": "tiny_request", "kind": "request", "shape": "tiny", "k": 3, "prefix": 16, "tokens": 9, "kv": "bf16"},
        # the headline workload: a 15-token prefix, 3 drafts of 10 tokens, read step by step
        {"name": "request_7b", "kind": "request", "shape": "7b", "k": 3, "prefix": 15, "tokens": 10, "kv": "f32"},
        # the widest draft set of the k sweep, in one call, float32 cache
        {"name": "generate_7b_k8", "kind": "generate", "shape": "7b", "k": 8, "prefix": 15, "tokens": 10, "kv": "f32"},
        # decoding behind a long document
        {"name": "decode_7b_2048", "kind": "decode", "shape": "7b", "k": 3, "prefix": 2048, "tokens": 10, "kv": "bf16"},
        # time to the first drafts: a short question, a paragraph, a page, a long document
        {"name": "prefill_7b_27", "kind": "prefill", "shape": "7b", "k": 3, "prefix": 27, "kv": "bf16"},
        {"name": "prefill_7b_100", "kind": "prefill", "shape": "7b", "k": 3, "prefix": 100, "kv": "bf16"},
        {"name": "prefill_7b_400", "kind": "prefill", "shape": "7b", "k": 3, "prefix": 400, "kv": "bf16"},
        {"name": "prefill_7b_2048", "kind": "prefill", "shape": "7b", "k": 3, "prefix": 2048, "kv": "bf16"},
        # a few requests with three drafts each and many plain ones, served together
        {"name": "batch_7b_8", "kind": "batch", "shape": "7b", "k": 3, "prefix": 15, "requests": 8, "tokens": 4, "kv": "f32"},
        {"name": "batch_7b_64", "kind": "batch", "shape": "7b", "k": 1, "prefix": 15, "requests": 64, "tokens": 4, "kv": "f32"},
        # drafts that start from a nucleus-sampled continuation
        {"name": "sample_7b", "kind": "sample", "shape": "7b", "k": 3, "prefix": 15, "tokens": 10, "kv": "f32"},
        # the larger model, five drafts behind a 64-token prefix
        {"name": "generate_13b_k5", "kind": "generate", "shape": "13b", "k": 5, "prefix": 64, "tokens": 4, "kv": "f32"},
    ]


def _spread(rng, lo, hi):
    """A whole number of lo..hi, spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["request", "generate", "decode", "prefill", "prefill", "batch", "sample"])
    shape = rng.choice(["tiny", "7b", "7b", "7b", "13b"]) if kind in ("request", "generate") else "7b"
    c = {"kind": kind, "shape": shape, "k": rng.choice([2, 3, 3, 4, 5, 6, 8]), "kv": "bf16" if kind in ("prefill", "decode") else "f32"}
    if kind == "prefill":
        c["prefix"] = _spread(rng, 8, 1900)
        if c["prefix"] <= 600:
            c["kv"] = rng.choice(["bf16", "bf16", "f32"])
        return c
    c["prefix"] = _spread(rng, 100, 1900) if kind == "decode" else _spread(rng, 8, 90)
    c["tokens"] = rng.randint(2, 5) if shape == "13b" else rng.randint(4, 10)
    if kind == "batch":
        c["k"], c["prefix"], c["tokens"] = rng.choice([1, 1, 2, 3]), rng.randint(8, 20), rng.randint(3, 4)
        c["requests"] = _spread(rng, 2, 64 if c["k"] == 1 else 12)  # every further draft is a further choice that can be a near-tie
    return c


# ---------------------------------------------------------------- inputs
_kept = {}


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _normal(g, rows, cols, std=0.02):
    return torch.randn(rows, cols, generator=g, device=DEVICE, dtype=torch.float32).mul_(std).to(torch.bfloat16)


def _gain(g, n):
    return torch.randn(n, generator=g, device=DEVICE, dtype=torch.float32).mul_(0.1).add_(1.0).to(torch.bfloat16)


def _layer(shape, l):
    """The tensors of layer l, bf16, [out][in]."""
    g, d, f = _generator(1000 + l), shape.d_model, shape.d_ffn
    out = {n: _normal(g, d, d) for n in ("wq", "wk", "wv", "wo")}
    out["wgate"], out["wup"], out["wdown"] = _normal(g, f, d), _normal(g, f, d), _normal(g, d, f)
    out["attn_norm"], out["ffn_norm"] = _gain(g, d), _gain(g, d)
    return out


def _ends(shape):
    g = _generator(999)
    return {"tok_emb": _normal(g, shape.vocab, shape.d_model), "lm_head": _normal(g, shape.vocab, shape.d_model, 0.02),
            "final_norm": _gain(g, shape.d_model)}


def _orders(case):
    return (2, 3, 4) if case["shape"] == "tiny" else (2, 3, 4, 5, 6)


def _lambdas(case):
    return [LAMBDA[n - 2] if n in _orders(case) else 0.0 for n in range(2, 10)]


def _model(case):
    """The shape's weights and n-gram tables as the library takes them; the last shape's are kept."""
    name = case["shape"]
    if _kept.get("name") != name:
        _kept.clear()
        torch.cuda.empty_cache()
        shape = si.SHAPES[name]
        weights = _ends(shape)
        layers = [_layer(shape, l) for l in range(shape.n_layers)]
        for key in list(layers[0]):
            weights[key] = [layer.pop(key) for layer in layers]
        packed = P.pack_weights(weights, DEVICE, consume=True)
        del weights, layers
        long = name != "tiny"
        counted = si.make_ngram_tables(shape.vocab, 1.1, 1_000_000 if long else 200_000, _orders(case), 100_000 if long else 20_000,
                                       seed=1, device=DEVICE)
        _kept.update(name=name, shape=shape, packed=packed, counted=counted, tables=P.build_ngram_tables(counted, DEVICE))
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    return _kept


def _prefixes(case, seed):
    """The prefix of each request (a batch: lengths up to four apart)."""
    vocab = si.SHAPES[case["shape"]].vocab
    rng = np.random.default_rng([int(seed), 77])
    cdf = si.zipf_cdf(vocab, 1.1)
    return [np.minimum(np.searchsorted(cdf, rng.random(case["prefix"] + r % 5)), vocab - 1).astype(np.int32)
            for r in range(case.get("requests", 1))]


def _uniforms(case, seed):
    return np.random.default_rng([int(seed), 78]).random(case["tokens"]).astype(np.float32)


def _positions(case):
    """Positions that the context's cache holds: room for the prefix and, where a context goes on, for many calls."""
    if case["kind"] in ("decode", "batch"):
        return case["prefix"] + 256
    return max(192, case["prefix"] + case.get("tokens", 1) + 64)


def prepare(case, seed):
    kept = _model(case)
    ctxs = [P.SpdContext(kept["shape"], kept["packed"], kept["tables"], case["k"], _orders(case), _lambdas(case), ALPHA, TAU, DELTA,
                         _positions(case), case["kv"]) for _ in range(case.get("requests", 1))]
    state = {"case": case, "ctxs": ctxs, "prefixes": _prefixes(case, seed), "left": 0}
    if case["kind"] == "sample":
        state["uniforms"] = _uniforms(case, seed)
    if case["kind"] in ("decode", "batch"):
        _begin(state)
    return state


def _begin(state):
    for ctx, prefix in zip(state["ctxs"], state["prefixes"]):
        ctx.spd_prefill(prefix)
    state["len"], state["left"] = 1, 240 // state["case"]["tokens"]


def run(state):
    case, ctx, prefix = state["case"], state["ctxs"][0], state["prefixes"][0]
    kind, n = case["kind"], case.get("tokens", 1)
    if kind in ("decode", "batch"):
        if state["left"] == 0:
            _begin(state)
        state["left"] -= 1
        state["len"] += n - 1
        if kind == "decode":
            ctx.spd_generate(n - 1, state["len"])
        else:
            P.spd_batch_generate(state["ctxs"], n - 1)
        return {"logits": [c.spd_debug_read("LOGITS") for c in state["ctxs"]]}
    ctx.spd_prefill(prefix)
    if kind == "prefill":
        return {"logits": ctx.spd_debug_read("LOGITS")}
    if kind == "request":
        for _ in range(n - 1):
            ctx.spd_step()
        return {"logits": ctx.spd_debug_read("LOGITS")}
    if kind == "generate":
        ctx.spd_generate(n - 1, n)
        return {"logits": ctx.spd_debug_read("LOGITS")}
    new, _, _ = ctx.spd_sample(state["uniforms"], TOP_P, TEMPERATURE)
    return {"logits": ctx.spd_debug_read("LOGITS"), "ids": new}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    shape = si.SHAPES[case["shape"]]
    d, f, v, layers = shape.d_model, shape.d_ffn, shape.vocab, shape.n_layers
    body, head = layers * (4 * d * d + 3 * d * f), v * d
    kv_row = layers * 2 * d * (2 if case["kv"] == "bf16" else 4)
    rows, n = case.get("requests", 1), case.get("tokens", 1)
    k, probes = case["k"], (case["k"] + case["k"] ** 2) * len(_orders(case)) * 32
    total = flops = 0
    if case["kind"] not in ("decode", "batch"):
        m = case["prefix"]
        total += 2 * (body + head) + m * (2 * d + kv_row)
        flops += 2 * (m * body + head) + 2 * layers * d * m * (m + 1)
    if case["kind"] != "prefill":
        steps = n if case["kind"] == "sample" else n - 1
        t = case["prefix"] + n / 2
        total += steps * (2 * (body + head) + rows * (t * kv_row + k * 2 * d + probes))
        flops += steps * rows * (2 * (body + head) + 4 * layers * d * t)
    return {"bytes": total + rows * 4 * v, "flops": flops}


def tolerance(case):
    """Four times and more what the library showed against 64 bits over several seeds.  float32 cache: sums in another
    order, which superposed timesteps enlarge through the drafts' weights.  bf16 cache: a value in a hundred rounds the
    other way, and the difference travels through the layers and positions that follow."""
    if case["kind"] in ("decode",):
        return {"rel": 3e-2, "max": 0.15}
    if case["kv"] == "bf16" and case["shape"] != "tiny":
        return {"rel": 1.4e-2, "max": 6e-2}
    if case["kind"] in ("prefill", "sample") or case["k"] == 1:
        return {"rel": 1e-4, "max": 5e-4}
    return {"rel": 1e-2, "max": 5e-2}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _rms(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + RMS_EPS) * gain.double()


def _rotate(x, pos, heads):
    """x [rows][d], adjacent pairs of each head turned by pos * theta^(-2i / head size)."""
    rows, d = x.shape
    hd = d // heads
    i = torch.arange(hd // 2, device=x.device, dtype=torch.float64)
    ang = pos.double()[:, None] * torch.pow(torch.tensor(ROPE_THETA, dtype=torch.float64, device=x.device), -2.0 * i / hd)
    cos, sin = torch.cos(ang)[:, None, :], torch.sin(ang)[:, None, :]
    y = x.view(rows, heads, hd // 2, 2)
    return torch.stack([y[..., 0] * cos - y[..., 1] * sin, y[..., 0] * sin + y[..., 1] * cos], -1).reshape(rows, d)


class _Exact:
    """The decoder and the method of one case in float64; cache values are rounded as the cache's type says."""

    def __init__(self, case, seed):
        self.case, self.shape = case, si.SHAPES[case["shape"]]
        self.prefixes = _prefixes(case, seed)
        self.rounds = case["kv"] == "bf16"
        self.ends = _ends(self.shape)
        self.cache = [[[None, None] for _ in self.prefixes] for _ in range(self.shape.n_layers)]
        self.counts = None

    def forward(self, xs):
        """xs: per request the new rows [t][d]; their keys and values join the cache.  Returns the rows' outputs."""
        heads, lens = self.shape.n_heads, [x.shape[0] for x in xs]
        hd = self.shape.d_model // heads
        seen = [0 if c[0] is None else c[0].shape[0] for c in self.cache[0]]
        pos = torch.cat([torch.arange(s, s + n, device=DEVICE) for s, n in zip(seen, lens)])
        h = torch.cat(xs)
        for l in range(self.shape.n_layers):
            w = _layer(self.shape, l)
            a = _rms(h, w["attn_norm"])
            q, k = (_rotate(a @ w[n].double().T, pos, heads) for n in ("wq", "wk"))
            v = a @ w["wv"].double().T
            if self.rounds:
                k, v = (t.to(torch.float32).to(torch.bfloat16).double() for t in (k, v))
            else:
                k, v = (t.to(torch.float32).double() for t in (k, v))
            o = torch.empty_like(h)
            at = 0
            for r, n in enumerate(lens):
                c = self.cache[l][r]
                for j, t in ((0, k), (1, v)):
                    new = t[at:at + n]
                    c[j] = new if c[j] is None else torch.cat([c[j], new])
                kk, vv = (t.view(-1, heads, hd).transpose(0, 1) for t in c)
                s = torch.matmul(q[at:at + n].view(n, heads, hd).transpose(0, 1), kk.transpose(1, 2)) / math.sqrt(hd)
                ahead = torch.arange(kk.shape[1], device=DEVICE)[None, :] > pos[at:at + n][:, None]
                s.masked_fill_(ahead[None], -math.inf)
                o[at:at + n] = torch.matmul(torch.softmax(s, -1), vv).transpose(0, 1).reshape(n, -1)
                at += n
            h = h + o @ w["wo"].double().T
            a = _rms(h, w["ffn_norm"])
            g = a @ w["wgate"].double().T
            h = h + (g * torch.sigmoid(g) * (a @ w["wup"].double().T)) @ w["wdown"].double().T
        return list(torch.split(h, lens))

    def logits(self, rows):
        return _rms(rows, self.ends["final_norm"]) @ self.ends["lm_head"].double().T

    def embed(self, ids):
        return self.ends["tok_emb"][torch.as_tensor(np.asarray(ids), device=DEVICE, dtype=torch.long)].double()

    def keep(self, z):
        """The k most probable tokens and their log-probabilities under the temperature."""
        top = torch.sort(z, descending=True, stable=True).indices[: self.case["k"]]
        lp = torch.log_softmax(z / TAU, -1)[top]
        return top.tolist(), lp.tolist()

    def first(self):
        rows = self.forward([self.embed(p) for p in self.prefixes])
        z = self.logits(torch.stack([r[-1] for r in rows]))
        self.drafts, self.logp = [], []
        for r, p in enumerate(self.prefixes):
            ids, lp = self.keep(z[r])
            self.drafts.append([p.tolist() + [t] for t in ids])
            self.logp.append(lp)
        return z

    def probability(self, history, token):
        """Interpolated n-gram probability of a token behind a draft."""
        if self.counts is None:
            self.counts = []
            for t in _model(self.case)["counted"]:
                grams, totals = {}, {}
                for row, c in zip(t["keys"].tolist(), t["counts"].tolist()):
                    grams[tuple(row)] = c
                    ctx = tuple(row[:-1])
                    totals[ctx] = totals.get(ctx, 0) + c
                self.counts.append((int(t["n"]), grams, totals))
        p = 0.0
        for n, grams, totals in self.counts:
            if len(history) >= n - 1:
                ctx = tuple(history[-(n - 1):])
                if ctx in totals:
                    p += LAMBDA[n - 2] * grams.get(ctx + (token,), 0) / totals[ctx]
        return p

    def weights(self, r):
        w = np.exp(np.asarray(self.logp[r]) - max(self.logp[r]))
        return w / w.sum()

    def step(self):
        xs = []
        for r in range(len(self.prefixes)):
            gamma = torch.as_tensor(self.weights(r), device=DEVICE, dtype=torch.float64)
            xs.append((gamma[:, None] * self.embed([d[-1] for d in self.drafts[r]])).sum(0, keepdim=True))
        z = self.logits(torch.cat(self.forward(xs)))
        for r in range(len(self.prefixes)):
            ids, lp = self.keep(z[r])
            options = []
            for i, draft in enumerate(self.drafts[r]):
                png = [self.probability(draft, t) for t in ids]
                for j, t in enumerate(ids):
                    score = self.logp[r][i] + (1 - ALPHA) * lp[j]
                    if not any(png):
                        options.append((score + math.log(DELTA), draft + [t]))
                    elif png[j] > 0:
                        options.append((score + ALPHA * math.log(png[j]), draft + [t]))
            options.sort(key=lambda o: -o[0])
            best = options[: self.case["k"]]
            if len(best) < self.case["k"]:
                raise ArithmeticError("fewer options than drafts")
            self.logp[r], self.drafts[r] = [o[0] for o in best], [o[1] for o in best]
        return z

    def nucleus(self, z, u):
        p = torch.softmax(z / TEMPERATURE, -1)
        order = torch.sort(p, descending=True, stable=True).indices
        cum = torch.cumsum(p[order], 0)
        size = int((cum < TOP_P).sum()) + 1
        at = int((cum[:size] <= float(u) * cum[size - 1]).sum())
        return int(order[min(at, size - 1)])


def exact(case, seed):
    """None for several timesteps of several drafts: there the distance from 64 bits is the first pass's rounding times
    whatever the drafts' weights made of it (1e-5 of it to 5e-3 over six seeds of one case), and says nothing about the
    precision of a sum.  The same kernels are measured by the sampled continuation, the single-draft batch and the
    prefixes."""
    if case["kind"] not in ("prefill", "sample") and case["k"] > 1:
        return None
    e = _Exact(case, seed)
    z = e.first()
    kind, n = case["kind"], case.get("tokens", 1)
    if kind == "prefill":
        return {"logits": z[0]}
    if kind == "sample":
        new = []
        for u in _uniforms(case, seed):
            new.append(e.nucleus(z[0], u))
            z = e.logits(e.forward([e.embed(new[-1:])])[0])
        return {"logits": z[0], "ids": np.asarray(new, np.int32)}
    try:
        for _ in range(n - 1):
            z = e.step()
    except ArithmeticError:
        return None
    return {"logits": list(z) if kind in ("decode", "batch") else z[0]}
