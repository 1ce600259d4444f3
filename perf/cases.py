"""The work that is measured: calls a user of the library makes, over the sizes they come in.

Kinds of case (key "kind"):
  score   dopr.score on a batch of (query, document) pairs against stored prefixes of m keys
          (m = 0: the uncompressed pass over [document ; query ; score token])
  ingest  dopr.build_prefixes for a set of documents, then one query scored against them:
          the built keys and values stay in the store, the scores are what shows them
  select  dopr.select_prefix_inputs: key token selection over whole documents
  pack    dopr.pack_order_noalloc: the packer's ordering step alone

Model widths are the Qwen3 shapes the repository is configured for, at their full depth for the
0.6B model and cut to a few layers otherwise (every layer does the same work).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_03311_gb300 import dopr, synth

MODEL_NAMES = ("qwen3-0.6b", "qwen3-4b", "qwen3-8b")
MIXED_M = (32, 64, 128, 256)  # prefix lengths of a mixed store, drawn per document
MAX_TOKENS = 74000            # packed tokens of the largest call
EXACT_FLOPS = 8e12            # a 64-bit pass above this takes too long


def _score(name, model, layers, queries, cands, q_lo, q_hi, m, docs, **more):
    return dict(name=name, kind="score", model=model, layers=layers, queries=queries, cands=cands, q_lo=q_lo,
                q_hi=q_hi, m=m, docs=docs, zipf=more.get("zipf", 0.0), doc_tokens=more.get("doc_tokens", 0),
                head=more.get("head", 0), io=more.get("io", "device"))


def listed():
    return [
        # one (query, document) pair: the per-pair latency the paper reports
        _score("8b one pair", "qwen3-8b", 4, 1, 1, 24, 24, 64, 100, io="host"),
        # the top of a first-stage ranking, rescored for one short query
        _score("8b ten candidates", "qwen3-8b", 4, 1, 10, 17, 17, 128, 100, io="host"),
        # one query's whole candidate list: the batch whose latency the bench quotes
        _score("8b hundred candidates", "qwen3-8b", 4, 1, 100, 37, 37, 64, 100),
        # a server's batch: 20 queries' lists over one collection with mixed prefix lengths (the largest call)
        _score("8b zipf batch", "qwen3-8b", 4, 20, 100, 8, 64, -1, 1000, zipf=1.1),
        # the two-layer model, short queries: launch-bound
        _score("0.6b two layers", "qwen3-0.6b", 2, 32, 8, 24, 24, 64, 64),
        # a whole model at full depth on one query's list, through host arrays
        _score("0.6b whole model", "qwen3-0.6b", 28, 1, 100, 40, 40, 64, 200, io="host"),
        # long reasoning-style queries, ragged, with the trained MLP scoring head instead of the yes/no rows
        _score("4b long queries", "qwen3-4b", 4, 2, 25, 32, 256, 128, 60, head=1024),
        # the uncompressed baseline: the document's own tokens in front of every query, no prefix
        _score("8b uncompressed", "qwen3-8b", 2, 1, 16, 37, 37, 0, 16, doc_tokens=512),
        # a batch of documents enters the store and is searched
        dict(name="8b ingest", kind="ingest", model="qwen3-8b", layers=2, docs=64, m_lo=64, m_hi=64, q_lo=37),
        # selection over ordinary documents, salience = the column mean
        dict(name="0.6b selection", kind="select", model="qwen3-0.6b", layers=4, docs=32, n_lo=512, n_hi=512, top_k=64,
             top_p=1 << 20),
        # selection over documents up to the longest the library takes, salience = the mean of the top 32
        dict(name="4b selection, long", kind="select", model="qwen3-4b", layers=2, docs=4, n_lo=777, n_hi=2048,
             top_k=256, top_p=32),
        # the ordering step of 200 queries' lists on its own
        dict(name="pack 20000 pairs", kind="pack", queries=200, cands=100, q_lo=8, q_hi=64, docs=1000, zipf=1.1),
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], even over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("score", "score", "score", "score", "uncompressed", "ingest", "select", "pack"))
    model = rng.choice(MODEL_NAMES)
    layers = rng.randint(2, 4)
    if kind in ("score", "uncompressed"):
        q_lo = _spread(rng, 1, 128)
        q_hi = min(256, q_lo + rng.randint(0, q_lo))
        doc_tokens = _spread(rng, 100, 600) if kind == "uncompressed" else 0
        per_pair = doc_tokens + (q_lo + q_hi) / 2 + 1
        cands = max(1, min(_spread(rng, 1, 100), int(20000 / per_pair) if doc_tokens else 100))
        queries = max(1, min(_spread(rng, 1, 20), int((20000 if doc_tokens else MAX_TOKENS) / (per_pair * cands))))
        m = 0 if doc_tokens else rng.choice((-1, _spread(rng, 1, 256), _spread(rng, 1, 256)))
        return {k: v for k, v in _score("", model, layers, queries, cands, q_lo, q_hi, m,
                                        max(cands, _spread(rng, 10, 400)), zipf=rng.choice((0.0, 1.1)),
                                        doc_tokens=doc_tokens, head=rng.choice((0, 0, 0, _spread(rng, 64, 1024))),
                                        io=rng.choice(("device", "host"))).items() if k != "name"}
    if kind == "ingest":
        m_lo = _spread(rng, 8, 200)
        return dict(kind="ingest", model=model, layers=layers, docs=_spread(rng, 1, 100), m_lo=m_lo,
                    m_hi=min(256, m_lo + rng.randint(0, m_lo)), q_lo=_spread(rng, 4, 64))
    if kind == "select":
        n_lo = _spread(rng, 100, 1500)
        n_hi = min(2048, n_lo + rng.randint(0, n_lo))
        return dict(kind="select", model=model, layers=layers, docs=max(1, min(_spread(rng, 1, 32), 16000 // n_hi)),
                    n_lo=n_lo, n_hi=n_hi, top_k=_spread(rng, 16, 256), top_p=rng.choice((1 << 20, _spread(rng, 4, 256))))
    return dict(kind="pack", queries=_spread(rng, 1, 300), cands=_spread(rng, 10, 100), q_lo=_spread(rng, 1, 32),
                q_hi=rng.randint(32, 64), docs=_spread(rng, 100, 1000), zipf=rng.choice((0.0, 1.1)))


# ---------------------------------------------------------------- inputs


def _shape(case):
    return synth.MODELS[case["model"]].with_layers(case["layers"])


def _between(lo, hi, n):
    """n lengths from lo to hi, evenly spaced: their sum does not depend on the seed."""
    return np.round(np.linspace(lo, hi, n) if n > 1 else np.array([(lo + hi) / 2])).astype(np.int64)


def _doc_lengths(case):
    """Prefix length of each document of a score case's store."""
    if case["m"] >= 0:
        return np.full(case["docs"], case["m"], np.int64)
    return np.asarray(MIXED_M, np.int64)[np.random.default_rng(5).integers(0, len(MIXED_M), case["docs"])]


def _candidates(case, seed):
    """Distinct documents of each query [queries, cands], uniform or Zipf-weighted."""
    rng = np.random.default_rng([seed, 1])
    weight = -case["zipf"] * np.log(np.arange(1, case["docs"] + 1))
    keys = weight + rng.gumbel(size=(case["queries"], case["docs"]))
    return rng.permutation(case["docs"])[np.argsort(-keys, axis=1)[:, :case["cands"]]].astype(np.int64)


def _pairs(case, seed, vocab, doc_tokens=None):
    """(q_offsets, q_tokens, doc_ids): every query's tokens once per candidate."""
    rng = np.random.default_rng([seed, 2])
    cand = _candidates(case, seed)
    lens = rng.permutation(_between(case["q_lo"], case["q_hi"], case["queries"]))
    parts, sizes = [], []
    for q, n in enumerate(lens):
        tok = rng.integers(0, vocab, n).astype(np.int32)
        for d in cand[q]:
            parts.append(tok if doc_tokens is None else np.concatenate([doc_tokens[d], tok]))
            sizes.append(len(parts[-1]))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    return off, np.concatenate(parts), cand.reshape(-1)


def _normal(gen, shape, std):
    return (torch.randn(shape, generator=gen, device="cuda") * std).to(torch.bfloat16)


def _weights(shape, seed):
    """Random-init bf16 decoder weights: matrices N(0, 0.02), norm gains 1 + N(0, 0.1)."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 7)
    H, F, D = shape.hidden, shape.ffn, shape.head_dim
    q, kv = shape.n_q_heads * D, shape.n_kv_heads * D

    def mat(*s):
        return _normal(g, s, 0.02)

    def gain(n):
        return (1 + 0.1 * torch.randn(n, generator=g, device="cuda")).to(torch.bfloat16)

    w = {"embed": mat(shape.vocab, H), "final_norm": gain(H), "score_head": mat(2, H)}
    each = {"attn_norm": lambda: gain(H), "wq": lambda: mat(q, H), "wk": lambda: mat(kv, H), "wv": lambda: mat(kv, H),
            "q_norm": lambda: gain(D), "k_norm": lambda: gain(D), "wo": lambda: mat(H, q), "mlp_norm": lambda: gain(H),
            "w_gate": lambda: mat(F, H), "w_up": lambda: mat(F, H), "w_down": lambda: mat(H, F)}
    w.update({k: [f() for _ in range(shape.n_layers)] for k, f in each.items()})
    return w


def _head(case, shape, seed):
    """An MLP scoring head of the case's width (GELU), or None for the yes/no rows."""
    n = case.get("head", 0)
    if not n:
        return None
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 11)
    return {"w1": _normal(g, (n, shape.hidden), 0.02), "b1": _normal(g, (n,), 0.1), "w2": _normal(g, (n,), n ** -0.5),
            "b2": 0.1, "act": 1}


def _prefixes(case, shape, seed):
    """Stored keys and values, N(0, 1): per layer bf16 [sum of m, kv heads, 128] twice, and the documents' first rows."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 13)
    m = _doc_lengths(case)
    first = np.concatenate([[0], np.cumsum(m)])
    size = (int(first[-1]), shape.n_kv_heads, shape.head_dim)
    return [(_normal(g, size, 1.0), _normal(g, size, 1.0)) for _ in range(shape.n_layers)], first


def _doc_texts(case, seed, vocab, lens):
    rng = np.random.default_rng([seed, 3])
    return [rng.integers(0, vocab, int(n)).astype(np.int32) for n in lens]


def _score_inputs(case, seed):
    shape = _shape(case)
    texts = _doc_texts(case, seed, shape.vocab, [case["doc_tokens"]] * case["docs"]) if case["doc_tokens"] else None
    return shape, _pairs(case, seed, shape.vocab, texts)


def _ingest_inputs(case, seed):
    """Documents' representations N(0, 1), and one query scored against all of them."""
    shape = _shape(case)
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    rng = np.random.default_rng([seed, 4])
    lens = rng.permutation(_between(case["m_lo"], case["m_hi"], case["docs"]))
    x_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    x = _normal(g, (int(x_off[-1]), shape.hidden), 1.0)
    tok = rng.integers(0, shape.vocab, case["q_lo"]).astype(np.int32)
    q_off = (np.arange(case["docs"] + 1) * case["q_lo"]).astype(np.int32)
    ids = np.arange(case["docs"], dtype=np.int64)
    return shape, x_off, x, (q_off, np.tile(tok, case["docs"]), ids)


def _select_inputs(case, seed):
    shape = _shape(case)
    lens = np.random.default_rng([seed, 5]).permutation(_between(case["n_lo"], case["n_hi"], case["docs"]))
    texts = _doc_texts(case, seed, shape.vocab, lens)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    return shape, off, np.concatenate(texts)


# ---------------------------------------------------------------- the measured passes


def _model(shape, seed, max_position):
    cfg = dopr.make_config(shape, max_position=max_position)
    return cfg, dopr.Model(cfg, _weights(shape, seed))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "score":
        shape, pairs = _score_inputs(case, seed)
        cfg, model = _model(shape, seed, 1024)
        dopr.set_mlp_head(model, _head(case, shape, seed))
        m = _doc_lengths(case)
        store = dopr.Store(cfg, case["docs"] - 1, dopr.prefix_bytes(cfg, int(m.sum())))
        layers, first = _prefixes(case, shape, seed)
        for d in range(case["docs"]):
            for l, (k, v) in enumerate(layers):
                store.put_layer(d, l, k[first[d]:first[d + 1]], v[first[d]:first[d + 1]])
        if case["io"] == "device":
            pairs = tuple(torch.from_numpy(a).cuda() for a in pairs)
        return dict(kind=kind, model=model, store=store, pairs=pairs)
    if kind == "ingest":
        shape, x_off, x, pairs = _ingest_inputs(case, seed)
        cfg, model = _model(shape, seed, 1024)
        store = dopr.Store(cfg, case["docs"] - 1, dopr.prefix_bytes(cfg, int(x_off[-1])))
        return dict(kind=kind, model=model, store=store, x_off=x_off, x=x, pairs=pairs)
    if kind == "select":
        shape, off, tok = _select_inputs(case, seed)
        _, model = _model(shape, seed, 2048)
        return dict(kind=kind, model=model, off=off, tok=tok, top_k=case["top_k"], top_p=case["top_p"])
    # pack: a store whose documents have one stored key each (the ordering reads slots and lengths only)
    shape = synth.MODELS["qwen3-0.6b"].with_layers(1)
    cfg = dopr.make_config(shape, max_position=1024)
    store = dopr.Store(cfg, case["docs"] - 1, dopr.prefix_bytes(cfg, case["docs"]))
    one = torch.zeros(1, shape.n_kv_heads, shape.head_dim, dtype=torch.bfloat16, device="cuda")
    for d in range(case["docs"]):
        store.put_layer(d, 0, one, one)
    q_off, _, ids = _pairs(case, seed, shape.vocab)
    n = len(ids)
    return dict(kind=kind, store=store, q_off=torch.from_numpy(q_off).cuda(), ids=torch.from_numpy(ids).cuda(),
                perm=torch.empty(n, dtype=torch.int32, device="cuda"),
                tok_off=torch.empty(n + 1, dtype=torch.int32, device="cuda"))


def run(s):
    if s["kind"] == "score":
        return {"scores": dopr.score(s["model"], s["store"], *s["pairs"])}
    if s["kind"] == "ingest":
        dopr.build_prefixes(s["model"], s["store"], s["pairs"][2], s["x_off"], s["x"])
        return {"scores": dopr.score(s["model"], s["store"], *s["pairs"])}
    if s["kind"] == "select":
        pos, x, u = dopr.select_prefix_inputs(s["model"], s["off"], s["tok"], s["top_k"], s["top_p"])
        return {"positions": pos, "states": x, "salience": u}
    dopr.pack_order_noalloc(s["store"], s["q_off"], s["ids"], s["perm"], s["tok_off"])
    return {"perm": s["perm"], "tok_off": s["tok_off"]}


# ---------------------------------------------------------------- what a pass cannot do without


def _layer_sizes(shape):
    """Weights of a layer: (QKV projection's, the others')."""
    q, kv = shape.n_q_heads * shape.head_dim, shape.n_kv_heads * shape.head_dim
    return shape.hidden * (q + 2 * kv), shape.hidden * q + 3 * shape.hidden * shape.ffn


def _decoder_work(shape, lens, keys_before, out_rows):
    """Bytes and flops of a decoder pass over sequences of `lens` tokens, each behind `keys_before` stored keys.
    out_rows: rows of the last layer anything after its keys and values is needed for, per sequence (0: none)."""
    lens, before = np.asarray(lens, float), np.asarray(keys_before, float)
    T, L = lens.sum(), shape.n_layers
    q, kv = shape.n_q_heads * shape.head_dim, shape.n_kv_heads * shape.head_dim
    w_qkv, w_rest = _layer_sizes(shape)
    attn = 4 * q * (lens * before + lens * (lens + 1) / 2).sum()
    flops = (L - 1) * (2 * T * (w_qkv + w_rest) + attn)
    out = np.minimum(lens, out_rows)
    flops += 2 * T * shape.hidden * 2 * kv + 2 * out.sum() * (shape.hidden * q + w_rest)
    flops += 4 * q * (out * before + lens * out - out * (out - 1) / 2).sum()
    weights = 2 * (L * (w_qkv + w_rest) - (0 if out_rows else w_rest + shape.hidden * q))
    return weights + T * (4 + 2 * shape.hidden), flops


def work(case):
    kind = case["kind"]
    if kind == "pack":
        n = case["queries"] * case["cands"]
        return {"bytes": 20.0 * n, "flops": 0}
    shape = _shape(case)
    stored = 4.0 * shape.n_layers * shape.n_kv_heads * shape.head_dim  # bytes of a stored position
    if kind == "score":
        cand = _candidates(case, 0).reshape(-1)
        m = _doc_lengths(case)
        lens = np.repeat(_between(case["q_lo"], case["q_hi"], case["queries"]), case["cands"]) + 1 + case["doc_tokens"]
        b, f = _decoder_work(shape, lens, m[cand], 1)
        b += m[np.unique(cand)].sum() * stored + 4 * len(cand)
        f += 2 * len(cand) * shape.hidden * max(2, case["head"])
        return {"bytes": float(b), "flops": float(f)}
    if kind == "ingest":
        m = _between(case["m_lo"], case["m_hi"], case["docs"])
        b, f = _decoder_work(shape, m, 0 * m, 0)
        b2, f2 = _decoder_work(shape, 0 * m + case["q_lo"] + 1, m, 1)
        return {"bytes": float(b + b2 + 2 * m.sum() * stored), "flops": float(f + f2)}
    n = _between(case["n_lo"], case["n_hi"], case["docs"])
    b, f = _decoder_work(shape, n, 0 * n, 1 << 30)
    probs = (n * (n + 1.0) / 2).sum()
    return {"bytes": float(b + case["docs"] * case["top_k"] * (2 * shape.hidden + 4) + 4 * n.sum()),
            "flops": float(f + shape.n_q_heads * probs * 4)}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    # 16-bit operands of the tensor-core products (10 stored bits) through all layers: a pass is 0.8e-3 to 1.6e-3 of the
    # scores' size off the 64-bit result (2.2e-3 in the full-depth model), so two correct passes differ by as much.
    # Four times that, and room for a call of a few scores, one of them near 0.
    if case["kind"] == "select":
        return {"rel": 1e-2, "max": 0.2, "differ": 0.01}  # the states come back in bf16 (2e-3 each), a tie may swap rows
    deep = case["layers"] > 8
    return {"rel": 1.5e-2 if deep else 1e-2, "max": 0.1 if deep else 0.05}


# ---------------------------------------------------------------- the same in 64 bits, plain torch


def _rms(x, gain, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain.double()


def _rope(x, pos, theta):
    """x [n, heads, 128]: pairs (i, i + 64) rotated by pos * theta^(-2i/128)."""
    half = x.shape[-1] // 2
    ang = pos.double()[:, None] * theta ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    c, s = ang.cos()[:, None, :], ang.sin()[:, None, :]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _decode(shape, w, x, lens, before, probs_of_last=False):
    """The decoder over rows x, sequences of `lens` rows end to end; sequence i's stored keys and values in layer l:
    before(i, l) = (k, v) [m, kv heads, 128] in 64 bits or None.  Returns the last residual rows, every layer's keys and
    values of these rows, and (asked) the head-averaged attention weights of the last layer per sequence."""
    D, Hq, Hkv, eps = shape.head_dim, shape.n_q_heads, shape.n_kv_heads, shape.rms_eps
    first = np.concatenate([[0], np.cumsum(lens)])
    made, probs = [], []
    m0 = [0 if before(i, 0) is None else before(i, 0)[0].shape[0] for i in range(len(lens))]
    pos = torch.cat([torch.arange(m, m + int(n), device=x.device) for m, n in zip(m0, lens)])
    for l in range(shape.n_layers):
        h = _rms(x, w["attn_norm"][l], eps)
        q, k, v = ((h @ w[n][l].double().T).view(len(x), -1, D) for n in ("wq", "wk", "wv"))
        q = _rope(_rms(q, w["q_norm"][l], eps), pos, shape.rope_theta)
        k = _rope(_rms(k, w["k_norm"][l], eps), pos, shape.rope_theta)
        made.append((k, v))
        o = torch.empty_like(q)
        for i, n in enumerate(int(n) for n in lens):
            rows = slice(int(first[i]), int(first[i]) + n)
            old = before(i, l)
            ki, vi = (k[rows], v[rows]) if old is None else (torch.cat([old[0], k[rows]]), torch.cat([old[1], v[rows]]))
            ki, vi = (t.repeat_interleave(Hq // Hkv, 1) for t in (ki, vi))
            s = torch.einsum("qhd,khd->hqk", q[rows], ki) / math.sqrt(D)
            s = s.masked_fill(torch.ones(s.shape[1:], dtype=torch.bool, device=x.device).triu(m0[i] + 1), -math.inf)
            p = s.softmax(-1)
            if probs_of_last and l == shape.n_layers - 1:
                probs.append(p.mean(0))
            o[rows] = torch.einsum("hqk,khd->qhd", p, vi)
        x = x + o.view(len(x), -1) @ w["wo"][l].double().T
        h = _rms(x, w["mlp_norm"][l], eps)
        up = torch.nn.functional.silu(h @ w["w_gate"][l].double().T) * (h @ w["w_up"][l].double().T)
        x = x + up @ w["w_down"][l].double().T
    return x, made, probs


def _exact_scores(shape, w, head, pairs, before):
    q_off, q_tok, ids = pairs
    lens = np.diff(q_off) + 1
    ends = np.cumsum(lens) - 1
    tok = np.insert(q_tok, q_off[1:], shape.score_token_id)
    x = w["embed"][torch.from_numpy(tok.astype(np.int64)).cuda()].double()
    x, _, _ = _decode(shape, w, x, lens, lambda i, l: before(int(ids[i]), l))
    h = _rms(x[torch.from_numpy(ends).cuda()], w["final_norm"], shape.rms_eps)
    if head is None:
        return h @ (w["score_head"][0].double() - w["score_head"][1].double())
    z = torch.nn.functional.gelu(h @ head["w1"].double().T + head["b1"].double())
    return z @ head["w2"].double() + head["b2"]


def exact(case, seed):
    if case["kind"] == "pack" or work(case)["flops"] > EXACT_FLOPS:
        return None
    if case["kind"] == "score":
        shape, pairs = _score_inputs(case, seed)
        layers, first = _prefixes(case, shape, seed)

        def stored(d, l):
            return tuple(t[first[d]:first[d + 1]].double() for t in layers[l])

        scores = _exact_scores(shape, _weights(shape, seed), _head(case, shape, seed), pairs, stored)
        return {"scores": scores if case["io"] == "device" else scores.cpu()}
    if case["kind"] == "ingest":
        shape, x_off, x, pairs = _ingest_inputs(case, seed)
        w = _weights(shape, seed)
        _, made, _ = _decode(shape, w, x.double(), np.diff(x_off), lambda i, l: None)
        scores = _exact_scores(shape, w, None, pairs,
                               lambda d, l: tuple(t[x_off[d]:x_off[d + 1]] for t in made[l]))
        return {"scores": scores.cpu()}
    shape, off, tok = _select_inputs(case, seed)
    w = _weights(shape, seed)
    lens = np.diff(off)
    x, _, probs = _decode(shape, w, w["embed"][torch.from_numpy(tok.astype(np.int64)).cuda()].double(), lens,
                          lambda i, l: None, probs_of_last=True)
    salience = []
    for p in probs:
        n = p.shape[0]
        count = torch.arange(n, 0, -1, device=p.device).clamp(max=case["top_p"])
        run_sum = p.sort(0, descending=True).values.cumsum(0)  # entries above the diagonal are 0 and come last
        salience.append(run_sum.gather(0, count[None] - 1)[0] / count)
    # which rows come back turns on gaps far below the rounding of 16-bit operands, unless all of them do
    states = None
    if lens.max() <= case["top_k"]:
        states = torch.zeros(len(lens), case["top_k"], shape.hidden, dtype=torch.float64)
        h = _rms(x, w["final_norm"], shape.rms_eps)
        for i, n in enumerate(lens):
            states[i, :n] = h[off[i]:off[i + 1]].cpu()
    return {"positions": None, "states": states, "salience": torch.cat(salience).cpu()}
