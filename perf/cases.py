"""Performance cases of the Ouroboros decoding path on one GPU.

What a user of this framework has it do: prefill a prompt, draft with the small model, verify a packed candidate block
with the large one, decode greedily with or without drafts, and (for callers without a workspace) run the LM head
alone.  Shapes are those of this repository's configurations (``synth.config``), whole where three states fit one card
and cut to fewer layers where they do not, or small generic ones.

Models are synthetic but peaked like trained ones: the embedding dominates the residual stream and the LM head is
aligned with it through a permutation of the vocabulary made of cycles, so that the greedy text is a fixed chain with a
wide top-2 margin (tokens do not hang on rounding).  A draft model follows the same chain except on an eighth of the
vocabulary, which gives partly and fully accepted drafts; the text comes back to earlier phrases, which feeds the pool.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2402_13720_b200 import binding, build, synth

CYCLE = 48            # tokens until the greedy text comes back to where it was
DRAFT_MISS = 0.12     # share of the vocabulary where the draft model predicts something else

# layers, d_model, heads, kv heads, head dim, FFN, vocabulary
SHAPES = {
    "7b": (32, 4096, 32, 32, 128, 11008, 32000),
    "1b": (22, 2048, 32, 4, 64, 5632, 32000),
    "34b": (60, 7168, 56, 8, 128, 20480, 64000),
    "6b": (32, 4096, 32, 4, 128, 11008, 64000),
    "70b": (80, 8192, 64, 8, 128, 28672, 32000),
    "small": (2, 512, 4, 2, 128, 512, 1024),
    "tiny": (2, 128, 4, 4, 32, 344, 512),
}


def listed():
    return [
        # The smallest whole use: the fp32 pair of configuration C1 (early-exit draft), prompt 32, 64 new tokens.
        dict(name="generate_tiny_f32", kind="generate", shape="tiny", layers=2, draft="early_exit", draft_layers=1, dtype="f32",
             prompt=32, new=64, gamma=4, beta=4, K=4),
        # The smallest bf16 call: one verification step of a two-layer model, where only latency and launches count.
        dict(name="step_small", kind="step", shape="small", layers=2, dtype="bf16", cache=67, gamma=3, beta=4, K=3, phrases=3,
             hits=2, logits=False),
        # Configuration C2 (the repository's benchmark): one layer + LM head on a long cache, 37 rows, one library call.
        dict(name="step_7b_layer", kind="step", shape="7b", layers=1, dtype="bf16", cache=4096, gamma=4, beta=9, K=4, phrases=4,
             hits=2, logits=False),
        # The verification step of configuration C3's whole target in mid-generation: draft accepted, a suffix moved.
        dict(name="step_7b", kind="step", shape="7b", layers=32, dtype="bf16", cache=411, gamma=4, beta=9, K=4, phrases=4,
             hits=4, logits=True),
        # Plain greedy decoding of the 7B-shaped target (no draft): one token per forward, after a one-chunk prompt.
        dict(name="vanilla_7b", kind="vanilla", shape="7b", layers=32, dtype="bf16", prompt=129, new=24),
        # Prompt processing of the same model: a ragged prompt, three full chunks and a rest; phrases seed the pool.
        dict(name="prefill_7b", kind="prefill", shape="7b", layers=32, dtype="bf16", prompt=467, gamma=4, beta=9, K=4),
        # Drafting: four single-row forwards of the 1.1B-shaped draft model (grouped queries, head dim 64).
        dict(name="draft_1b", kind="draft", shape="1b", layers=22, dtype="bf16", cache=389, gamma=4, beta=9, K=4, window=0),
        # Drafting with phrase generation (lookahead window), at the paper's settings for long drafts.
        dict(name="draft_1b_window", kind="draft", shape="1b", layers=22, dtype="bf16", cache=521, gamma=6, beta=6, K=3, window=18),
        # Whole generation with configuration C3's pair: prefill, drafting, verification, acceptance, harvest, host loop.
        dict(name="generate_7b", kind="generate", shape="7b", layers=32, draft="1b", draft_layers=22, dtype="bf16",
             prompt=256, new=96, gamma=4, beta=9, K=4),
        # Configuration C4's block (K = 8, 69 rows, GQA 7:1, vocabulary 64000) on a slice of its 60 layers.
        dict(name="step_34b_slice", kind="step", shape="34b", layers=8, dtype="bf16", cache=777, gamma=4, beta=9, K=8, phrases=8,
             hits=4, logits=True),
        # Configuration C5's widths on a slice of its 80 layers over a long context, two phrases found.
        dict(name="step_70b_slice_long", kind="step", shape="70b", layers=6, dtype="bf16", cache=12345, gamma=6, beta=7, K=4,
             phrases=2, hits=5, logits=True),
        # LM head for callers that cannot allocate: logits and greedy tokens of one block.
        dict(name="lm_head_static", kind="lm_head", rows=37, d=4096, vocab=32000, logits=True),
    ]


def _between(rng, lo, hi):
    """Whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "prefill", "vanilla", "draft", "draft", "generate", "generate_tiny", "lm_head"])
    if kind == "lm_head":
        return dict(kind=kind, rows=_between(rng, 1, 128), d=64 * _between(rng, 8, 128), vocab=8 * _between(rng, 128, 8000),
                    logits=rng.random() < 0.5)
    gamma, beta, K = rng.randint(2, 12), rng.randint(3, 9), rng.randint(1, 8)
    while 1 + gamma + K * (beta - 1) > 100:
        K -= 1
    if kind == "generate_tiny":
        return dict(kind="generate", shape="tiny", layers=rng.randint(2, 4), draft="early_exit", draft_layers=1, dtype="f32",
                    prompt=_between(rng, 9, 120), new=_between(rng, 16, 96), gamma=gamma, beta=beta, K=K)
    if kind == "step":
        shape = rng.choice(["small", "1b", "7b", "6b", "34b", "70b"])
        most = {"small": 4, "1b": 22, "7b": 12, "6b": 12, "34b": 6, "70b": 4}[shape]
        hits = rng.randint(0, gamma)
        # (a fully accepted draft corrects the pool's phrases: only with candidates in hand is every pass the same)
        return dict(kind=kind, shape=shape, layers=rng.randint(1, most), dtype="bf16", cache=_between(rng, 33, 12000), gamma=gamma,
                    beta=beta, K=K, phrases=rng.randint(0, K), hits=hits, logits=hits == gamma or rng.random() < 0.5)
    if kind == "draft":
        shape = rng.choice(["small", "1b", "1b", "6b", "7b"])
        window = rng.choice([0, rng.randint(beta - 1, 20)])
        return dict(kind=kind, shape=shape, layers={"small": 2, "1b": 22}.get(shape, 8), dtype="bf16", cache=_between(rng, 33, 4000),
                    gamma=gamma, beta=beta, K=K, window=window)
    shape = rng.choice(["small", "1b", "7b", "6b"])
    layers = {"small": 2, "1b": 22}.get(shape, rng.randint(2, 12))
    if kind == "prefill":
        return dict(kind=kind, shape=shape, layers=layers, dtype="bf16", prompt=_between(rng, 17, 1500), gamma=gamma, beta=beta, K=K)
    if kind == "vanilla":
        return dict(kind=kind, shape=shape, layers=layers, dtype="bf16", prompt=_between(rng, 2, 1200), new=_between(rng, 8, 48))
    return dict(kind=kind, shape=shape, layers=layers, draft="small" if shape == "small" else "1b", draft_layers=2 if shape == "small" else 12,
                dtype="bf16", prompt=_between(rng, 17, 700), new=_between(rng, 24, 96), gamma=gamma, beta=beta, K=K)


# ------------------------------------------------------------------------------------------ inputs

def _desc(shape, layers, dtype, max_seq):
    _, d, h, kv, hd, f, v = SHAPES[shape]
    return synth.ModelDesc(layers, d, h, kv, hd, f, v, max_seq, dtype)


def _params(case):
    return synth.DecodeParams(case.get("gamma", 1), case.get("beta", 2), case.get("K", 0), 128, 32, window=case.get("window", 0))


def _rows(case):
    """Rows of a step's block."""
    return 1 + case["gamma"] + min(case["phrases"], case["K"]) * (case["beta"] - 1)


def _positions(case):
    """Cache slots a case needs."""
    block = 1 + case.get("gamma", 0) + max(case.get("K", 0) * (case.get("beta", 1) - 1), case.get("window", 0))
    text = case["cache"] if "cache" in case else case["prompt"] + case.get("new", 0)
    return text + 2 * block + 16


def _chain(rs, vocab):
    """Successor of every token in the greedy text: a permutation made of cycles of CYCLE tokens."""
    order = rs.permutation(vocab)
    nxt = np.empty(vocab, dtype=np.int64)
    for a in range(0, vocab, CYCLE):
        part = order[a: a + CYCLE]
        nxt[part] = np.roll(part, -1)
    return nxt


def _weights(m, seed, nxt):
    w = synth.model_weights(m, seed, device="cuda")
    w["embed"].mul_(50.0)                                            # unit variance: it dominates the residual stream,
    for lw in w["layers"]:                                           # to which every branch adds its share of one layer's
        for name in ("wo", "w_down"):
            lw[name].mul_((2 * m.n_layers) ** -0.5)
    before = np.empty_like(nxt)
    before[nxt] = np.arange(len(nxt))
    w["lm_head"].add_(w["embed"][torch.as_tensor(before, device="cuda")], alpha=0.02)
    return w


def _follow(nxt, token, n):
    out = []
    for _ in range(n):
        token = int(nxt[token])
        out.append(token)
    return out


def _prompt(rs, nxt, n):
    """Stretches of 8 to 32 tokens of the model's own text, started from a few places again and again."""
    starts = rs.randint(0, len(nxt), 6)
    out = []
    while len(out) < n:
        out += _follow(nxt, int(starts[rs.randint(6)]), int(rs.randint(8, 33)))
    return np.asarray(out[:n], dtype=np.int32)


def _fill_cache(mem, length, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for cache in (mem.k_cache, mem.v_cache):
        cache[:, :length].normal_(generator=gen)


def prepare(case, seed):
    build.build()
    rs = np.random.RandomState(seed % (1 << 31))
    if case["kind"] == "lm_head":
        return dict(case=case, x=synth.tensor(seed, 1, (case["rows"], case["d"]), 1.0, torch.bfloat16, "cuda"),
                    w=synth.tensor(seed, 2, (case["vocab"], case["d"]), 0.02, torch.bfloat16, "cuda"))
    kind, P, room = case["kind"], _params(case), _positions(case)
    if kind == "draft":     # the drafts are what is used here: the target is one layer of the same widths
        draft = _desc(case["shape"], case["layers"], case["dtype"], room)
        target = dataclasses.replace(draft, n_layers=1)
    else:
        target = _desc(case["shape"], case["layers"], case["dtype"], room)
        draft = None
        if kind == "generate":
            draft = target.early_exit(case["draft_layers"]) if case["draft"] == "early_exit" else \
                dataclasses.replace(_desc(case["draft"], case["draft_layers"], case["dtype"], room), vocab=target.vocab)
    nxt = _chain(rs, target.vocab)
    w = _weights(target, seed, nxt)
    wd = None
    if kind == "draft" or case.get("draft") == "early_exit":
        wd = w if draft.n_layers <= target.n_layers else _weights(draft, seed + 1, nxt)
    elif draft is not None:
        miss = nxt.copy()
        at = rs.permutation(target.vocab)[: int(DRAFT_MISS * target.vocab)]
        miss[at] = nxt[np.roll(at, 1)]
        wd = _weights(draft, seed + 1, miss)
    eng = binding.Engine(target, w, P, draft, wd, device="cuda:0")
    state = dict(case=case, eng=eng, next=nxt)
    if kind in ("prefill", "vanilla", "generate"):
        state["prompt"] = _prompt(rs, nxt, case["prompt"])
        return state
    L = case["cache"]
    state["pending"] = int(rs.randint(target.vocab))
    _fill_cache(eng.tm, L, seed)
    if kind == "draft":
        _fill_cache(eng.dm, L, seed + 1)
        return state
    # a step: a draft whose first `hits` tokens the target agrees with, and phrases that start with its last token, the
    # first of them right and each of the others wrong from some place on
    tokens = _follow(nxt, state["pending"], P.gamma)
    for i in range(case["hits"], P.gamma):
        tokens[i] = int(rs.randint(target.vocab))
    eng.draft_tokens.copy_(torch.as_tensor(tokens, dtype=torch.int32))
    if case["phrases"] > 0:
        grams = np.array([[tokens[-1]] + _follow(nxt, tokens[-1], P.S) for _ in range(case["phrases"])], dtype=np.int32)
        for j in range(1, case["phrases"]):
            at = int(rs.randint(1, P.beta))
            grams[j, at:] = rs.randint(0, target.vocab, P.beta - at)
        eng.phrase_update(np.roll(grams, int(rs.randint(case["phrases"])), axis=0))
    eng.phrase_lookup(tokens[-1])         # candidates in hand, for the calls that pack them without another lookup
    return state


# -------------------------------------------------------------------------------------------- runs

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lm_head":
        argmax, logits = binding.lm_head_static(state["x"], state["w"], want_logits=case["logits"])
        return {"argmax": argmax, "logits": logits}
    eng = state["eng"]
    T, D = eng.tm, eng.dm
    if kind == "generate":
        out, _ = eng.generate(state["prompt"], case["new"])
        n = case["prompt"] + case["new"] - 1
        return {"tokens": out, "k": T.k_cache[:, :n], "v": T.v_cache[:, :n]}
    if kind == "vanilla":
        out, _ = eng.generate_vanilla(state["prompt"], case["new"])
        n = case["prompt"] + case["new"] - 1
        return {"tokens": out, "k": T.k_cache[:, :n], "v": T.v_cache[:, :n]}
    if kind == "prefill":
        eng.reset()
        eng.prefill(state["prompt"])
        n = case["prompt"] - 1
        return {"k": T.k_cache[:, :n], "v": T.v_cache[:, :n]}
    eng.set_state(case["cache"], state["pending"])
    if kind == "draft":
        tokens = eng.draft()
        n = case["cache"] + case["gamma"]
        return {"tokens": tokens, "k": D.k_cache[:, :n], "v": D.v_cache[:, :n]}
    logits = None
    if case["logits"]:
        eng.assemble_candidates(lookup_here=False)
        _, logits = eng.verify_forward(want_logits=True)
        n, chosen, accurate, accepted = eng.accept_and_compact()
        logits = logits[: _rows(case)]
    else:
        n, chosen, accurate, accepted = eng.verify_step()
    end = case["cache"] + n
    return {"accepted": np.array(accepted[:n]), "logits": logits, "k": T.k_cache[:, :end], "v": T.v_cache[:, :end]}


# ------------------------------------------------------------------------- the same in 64 bits

def _norm64(x, gain, eps):
    return gain.double() * x / (x.square().mean(-1, keepdim=True) + eps).sqrt()


def _rope64(x, pos, theta):
    half = x.shape[-1] // 2
    inv = theta ** (-torch.arange(half, dtype=torch.float64, device=x.device) / half)
    angle = pos.double()[:, None, None] * inv
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * angle.cos() - b * angle.sin(), b * angle.cos() + a * angle.sin()], -1)


def _matmul64(x, w):
    """x w^T, the bf16 or fp32 weights widened a slab at a time."""
    return torch.cat([x @ part.double().T for part in w.split(8192)], -1)


def _attend64(q, k, v, hidden):
    """q [rows, heads, h]; k, v [keys, kv heads, h]; hidden [rows, rows] for the last keys (the block's own)."""
    group = q.shape[1] // k.shape[1]
    out = torch.empty_like(q)
    for j in range(k.shape[1]):
        s = torch.einsum("rah,kh->ark", q[:, j * group: (j + 1) * group], k[:, j]) / math.sqrt(q.shape[-1])
        s[..., s.shape[-1] - len(hidden):].masked_fill_(hidden, -math.inf)
        out[:, j * group: (j + 1) * group] = torch.einsum("ark,kh->rah", s.softmax(-1), v[:, j])
    return out


def _forward64(m, w, tokens, pos, hidden, before, logits=True):
    """Keys and values of a block in every layer ([layers, rows, kv heads, h] each), and its logits.  `before`: the cached
    keys and values in front of it, or None."""
    device = w["embed"].device
    pos = torch.as_tensor(np.asarray(pos), device=device)
    x = w["embed"][torch.as_tensor(np.asarray(tokens), dtype=torch.int64, device=device)].double()
    rows = len(pos)
    ks, vs = [], []
    for layer in range(m.n_layers):
        lw = w["layers"][layer]
        n1 = _norm64(x, lw["attn_norm"], m.rms_eps)
        q = _rope64(_matmul64(n1, lw["wq"]).view(rows, m.n_heads, m.head_dim), pos, m.rope_theta)
        k = _rope64(_matmul64(n1, lw["wk"]).view(rows, m.n_kv_heads, m.head_dim), pos, m.rope_theta)
        v = _matmul64(n1, lw["wv"]).view(rows, m.n_kv_heads, m.head_dim)
        ks.append(k)
        vs.append(v)
        if before is not None:
            k, v = torch.cat([before[0][layer].double(), k]), torch.cat([before[1][layer].double(), v])
        x = x + _matmul64(_attend64(q, k, v, hidden).reshape(rows, -1), lw["wo"])
        n2 = _norm64(x, lw["ffn_norm"], m.rms_eps)
        gate = _matmul64(n2, lw["w_gate"])
        x = x + _matmul64(gate * gate.sigmoid() * _matmul64(n2, lw["w_up"]), lw["w_down"])
    return torch.stack(ks), torch.stack(vs), _matmul64(_norm64(x, w["final_norm"], m.rms_eps), w["lm_head"]) if logits else None


def _causal(n):
    return torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1)


def exact(case, seed):
    """Token choices have wide margins, so keys and values are those of one causal forward over the greedy text."""
    state = prepare(case, seed)
    torch.cuda.synchronize()
    if case["kind"] == "lm_head":
        return {"argmax": None, "logits": _matmul64(state["x"].double(), state["w"]) if case["logits"] else None}
    kind, eng, nxt = case["kind"], state["eng"], state["next"]
    if kind in ("prefill", "vanilla", "generate"):
        text = [int(t) for t in state["prompt"]]
        if kind != "prefill":
            text += _follow(nxt, text[-1], case["new"])
        text = text[:-1]
        k, v, _ = _forward64(eng.target_desc, eng.tm.w, text, range(len(text)), _causal(len(text)), None, logits=False)
        return {"k": k, "v": v} if kind == "prefill" else {"tokens": None, "k": k, "v": v}
    L, P = case["cache"], eng.params
    mem, m = (eng.dm, eng.draft_desc) if kind == "draft" else (eng.tm, eng.target_desc)
    before = mem.k_cache[:, :L], mem.v_cache[:, :L]
    if kind == "draft":
        text = [state["pending"]] + _follow(nxt, state["pending"], P.gamma - 1)
        logits = None
    else:
        # accepted: the draft's right tokens and, behind a whole draft, the right phrase's, then one of the target's own
        matched = case["hits"]
        if matched == P.gamma and case["phrases"] > 0:
            matched += P.S
        text = [state["pending"]] + _follow(nxt, state["pending"], matched)
        logits = None
        if case["logits"]:
            draft = [int(t) for t in eng.draft_tokens[: P.gamma]]
            suffixes = eng.suffix[: int(eng.count) * P.S].view(-1, P.S).tolist()
            trunk = 1 + P.gamma
            tokens = [state["pending"]] + draft + sum(suffixes, [])
            pos = list(range(L, L + trunk)) + list(range(L + trunk, L + trunk + P.S)) * len(suffixes)
            hidden = _causal(len(tokens))
            group = torch.as_tensor([0] * trunk + [1 + j for j in range(len(suffixes)) for _ in range(P.S)], device="cuda")
            hidden |= (group[None, :] != group[:, None]) & (group[None, :] != 0)
            logits = _forward64(m, mem.w, tokens, pos, hidden, before)[2]
    k, v, _ = _forward64(m, mem.w, text, range(L, L + len(text)), _causal(len(text)), before, logits=False)
    k, v = (torch.cat([old.double(), new], 1) for old, new in zip(before, (k, v)))
    return {"tokens": None, "k": k, "v": v} if kind == "draft" else {"accepted": None, "logits": logits, "k": k, "v": v}


# -------------------------------------------------------------------------------- least work, tolerance

def _forward(m, rows, cached, size, logits=False):
    """(bytes, flops) of one forward of `rows` rows on a cache of `cached` tokens: every weight once, the visible keys and
    values once, the new ones written, the embedding rows, the logits where they are asked for."""
    layer = m.layer_weight_elems()
    kv = 2 * m.d_kv
    b = size * (m.n_layers * (layer + 2 * m.d_model + kv * (cached + rows)) + m.vocab * m.d_model + m.d_model + rows * m.d_model)
    f = 2.0 * rows * (m.n_layers * layer + m.vocab * m.d_model) + 4.0 * m.n_layers * m.d_q * rows * (cached + rows)
    return b + (4 * rows * m.vocab if logits else 0), f


def work(case):
    kind = case["kind"]
    if kind == "lm_head":
        r, d, v = case["rows"], case["d"], case["vocab"]
        return {"bytes": 2 * (r * d + v * d) + 4 * r + (4 * r * v if case["logits"] else 0), "flops": 2.0 * r * d * v}
    m = _desc(case["shape"], case["layers"], case["dtype"], _positions(case))
    size = 4 if case["dtype"] == "f32" else 2
    if kind == "step":
        b, f = _forward(m, _rows(case), case["cache"], size, case["logits"])
        return {"bytes": b, "flops": f}
    if kind == "draft":
        parts = [_forward(m, 1 + case["window"], case["cache"] + i, size) for i in range(case["gamma"])]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n = case["prompt"] - 1
    head = m.vocab * m.d_model
    parts = []
    if n > 0:               # the prompt's keys and values need no LM head
        b, f = _forward(m, n, 0, size)
        parts.append((b - size * head, f - 2.0 * n * head))
    if kind == "vanilla":
        parts += [_forward(m, 1, n + i, size) for i in range(case["new"])]
    if kind == "generate":  # at best every draft and a whole phrase is accepted in every step
        e = m.early_exit(case["draft_layers"]) if case["draft"] == "early_exit" else \
            dataclasses.replace(_desc(case["draft"], case["draft_layers"], case["dtype"], m.max_seq), vocab=m.vocab)
        for i in range(0, case["new"], case["gamma"] + case["beta"]):
            parts.append(_forward(m, 1 + case["gamma"], n + i, size))
            parts += [_forward(e, 1, n + i, size)] * case["gamma"]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    if case["kind"] == "lm_head":          # products of bf16 values summed in 32 bits, in whatever order
        return {"rel": 2e-6, "differ": 0.0}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "differ": 0.0}
    # Sums in another order move single roundings of the bf16 activations, and every layer carries that on.  Against the
    # same path with its sums in another order: logits 0.002 (one layer), 0.006 to 0.008 (6 to 32 layers), keys and values
    # up to 0.006; against the path in float64 without those roundings: 0.003 and 0.005 to 0.007.  Tokens: top-2 margins
    # are 7 to 35 where logits differ by less than 0.5.
    return {"rel": 1e-2 if case["layers"] <= 2 else 2e-2, "differ": 0.0}
