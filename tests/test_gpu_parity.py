"""GPU parity: the CUDA library, called through its C ABI, against the CPU oracle on the same seeded inputs.

Floating point: fp32 logits within 1e-3 max-abs; bf16 logits within 3e-2 of the row's largest |logit|.
Integers (block layout, acceptance, compaction indices, pool contents, tokens) are bit exact.
"""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import ouroboros as ob
from oracle import transformer as tf
from paper_2402_13720_b200 import binding, build, synth

pytestmark = pytest.mark.gpu

FP32_TOL = 1e-3
BF16_REL = 3e-2

TINY = synth.ModelDesc(2, 64, 4, 2, 32, 96, 100, 192, "f32")
MIDB = synth.ModelDesc(3, 256, 8, 2, 64, 512, 1000, 320, "bf16")     # GQA 4:1, head_dim 64, bf16
C1T, C1D, C1P, C1R = synth.config("C1")


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def make(desc, params, seed=0, draft=None):
    """Engine on cuda:0 and the oracle's weights; the generator gives identical values on both devices."""
    w = synth.model_weights(desc, seed, device="cuda:0")
    eng = binding.Engine(desc, w, params, draft, w if draft is not None else None)
    return eng, tf.Weights(desc, synth.model_weights(desc, seed))


def test_generated_inputs_are_device_independent():
    a = synth.model_weights(MIDB, 7, device="cuda:0")
    b = synth.model_weights(MIDB, 7)
    assert torch.equal(a["lm_head"].cpu(), b["lm_head"]) and torch.equal(a["layers"][2]["w_down"].cpu(), b["layers"][2]["w_down"])
    assert torch.equal(a["layers"][0]["attn_norm"].cpu(), b["layers"][0]["attn_norm"])


def oracle_pool(P):
    return ob.PhrasePool(P.pool_sets, P.pool_ways, P.beta)


def pool_rows(pool):
    ex = pool.export()
    return [list(p) for _, p in ex], [s for s, _ in ex]


def gpu_pool_rows(eng):
    ng, st = eng.pool_export()
    return ng.tolist(), st.tolist()


# ------------------------------------------------------------------------------------ pool

@pytest.mark.parametrize("sets,ways,beta", [(4, 3, 3), (1, 2, 2), (8, 40, 5)])
def test_pool_matches_oracle(sets, ways, beta):
    P = synth.DecodeParams(2, beta, 3, sets, ways)
    eng, _ = make(TINY, P)
    ref = oracle_pool(P)
    rng = np.random.default_rng(sets * 100 + ways)
    for rnd in range(12):
        grams = rng.integers(0, 7, (int(rng.integers(1, 40)), beta))
        eng.phrase_update(grams)
        for g in grams:
            ref.insert(g)
        assert gpu_pool_rows(eng) == pool_rows(ref)
        for key in range(8):
            got = eng.phrase_lookup(key).tolist()
            assert got == ref.lookup(key, P.K)
            assert all(len(s) == beta - 1 for s in got)
    # export -> reset -> import reproduces the same retrieval order
    ng, _ = eng.pool_export()
    eng.reset(keep_pool=False)
    assert eng.pool_export()[0].shape[0] == 0 and eng.phrase_lookup(3).shape[0] == 0
    eng.pool_import(ng)
    for key in range(8):
        assert eng.phrase_lookup(key).tolist() == ref.lookup(key, P.K)
    eng.close()


@pytest.mark.parametrize("sets,ways,beta,tokens", [(1, 40, 3, 9), (64, 4, 2, 90), (256, 8, 16, 12), (32, 33, 6, 40)])
def test_pool_takes_long_lists_in_order(sets, ways, beta, tokens):
    """A list of phrases is shared by the warps of a block, a set's phrases staying in one warp: lists of 1 to 700 sliding windows
    with few tokens (the same set and phrase again and again, sets that overflow), one set and more sets than warps.  Entries,
    stamps and the counter for what follows as in the oracle, which inserts one after the other."""
    P = synth.DecodeParams(2, beta, 3, sets, ways)
    eng, _ = make(TINY, P)
    ref = oracle_pool(P)
    rng = np.random.default_rng(tokens)
    for n in (1, 31, 32, 33, 700, 5):
        text = rng.integers(0, tokens, n + beta - 1)
        grams = np.stack([text[i: i + beta] for i in range(n)])
        eng.phrase_update(grams)
        for g in grams:
            ref.insert(g)
        assert gpu_pool_rows(eng) == pool_rows(ref), n
    eng.close()


# ------------------------------------------------------------------------- candidate packing

@pytest.mark.parametrize("gamma,beta,K,n_fill", [(4, 4, 4, 60), (3, 9, 4, 80), (2, 3, 0, 10), (5, 6, 3, 0), (1, 2, 16, 50)])
def test_assemble_matches_oracle(gamma, beta, K, n_fill):
    P = synth.DecodeParams(gamma, beta, K, 4, 8, seed_prompt=False)
    eng, _ = make(TINY, P)
    ref = oracle_pool(P)
    rng = np.random.default_rng(gamma * 10 + beta)
    if n_fill:
        grams = rng.integers(0, 5, (n_fill, beta))
        eng.phrase_update(grams)
        for g in grams:
            ref.insert(g)
    prompt = rng.integers(0, TINY.vocab, 21).astype(np.int32)
    eng.prefill(prompt)
    L = len(prompt) - 1
    for trial in range(4):
        d = rng.integers(0, 5, gamma).tolist()
        eng.assemble_candidates(draft=d)
        tok, pos, grp, mask = eng.block_get()
        cands = ref.lookup(d[-1], K)
        t2, p2, g2, vis = ob.build_block(L, prompt[-1], d, cands)
        assert tok.tolist() == t2 and pos.tolist() == p2 and grp.tolist() == g2
        B = len(t2)
        bits = np.array([[(int(mask[r, c // 64]) >> (c % 64)) & 1 for c in range(B)] for r in range(B)], dtype=bool)
        assert np.array_equal(bits, vis[:, L:])
        assert all(c[0] is not None for c in cands) and B == 1 + gamma + len(cands) * (beta - 1)
        # the same block through an explicit lookup
        got = eng.phrase_lookup(d[-1])
        eng.assemble_candidates(draft=d, lookup_here=False)
        assert eng.block_get()[0].tolist() == t2 and got.tolist() == cands
    eng.close()


# ------------------------------------------------------------------------------ forward logits

def _verify_case(eng, W, desc, P, seed, L_prompt, tol_fn, full_block=False):
    rng = np.random.default_rng(seed)
    prompt = synth.prompt(seed, desc.vocab, L_prompt, 0.4, 4, 8)
    eng.reset()
    eng.prefill(prompt)
    ref_pool = oracle_pool(P)
    ref_pool.apply(ob.prompt_ops(prompt, P.beta, P))
    d = rng.integers(0, desc.vocab, P.gamma).tolist()
    d[-1] = int(prompt[5])                     # a key that the seeded pool knows
    if full_block:                             # K phrases with that key, so that the block has all its rows
        grams = rng.integers(0, desc.vocab, (P.K, P.beta)).astype(np.int32)
        grams[:, 0] = d[-1]
        eng.phrase_update(grams)
        for g in grams:
            ref_pool.insert(g)
    eng.assemble_candidates(draft=d)
    tok, pos, grp, mask = eng.block_get()
    cands = ref_pool.lookup(d[-1], P.K)
    t2, p2, g2, vis = ob.build_block(len(prompt) - 1, prompt[-1], d, cands)
    assert tok.tolist() == t2 and len(cands) >= 1 and (not full_block or len(t2) == P.block_max)
    am, logits = eng.verify_forward(want_logits=True)
    cache = tf.KVCache(desc)
    ob.prefill(W, cache, list(prompt[:-1]))
    L = cache.length
    want = tf.forward(W, cache, t2, p2, vis)
    got = logits[: len(t2)].cpu().numpy().astype(np.float64)
    tol_fn(got, want)
    # greedy choice agrees wherever the oracle's top-2 margin exceeds the numeric error
    err = np.abs(got - want).max(axis=1)
    srt = np.sort(want, axis=1)
    safe = (srt[:, -1] - srt[:, -2]) > 2 * err + 1e-12
    assert safe.sum() >= 1
    assert np.array_equal(am[: len(t2)].cpu().numpy()[safe], tf.argmax_rows(want)[safe])
    # K/V appended by the forward equal the oracle's (cache slots L .. L+B-1 of every layer)
    k_gpu = eng.tm.k_cache[:, : L + len(t2)].float().cpu().numpy()
    v_gpu = eng.tm.v_cache[:, : L + len(t2)].float().cpu().numpy()
    kv_tol = 1e-4 if desc.dtype == "f32" else 2e-2 * max(np.abs(cache.k).max(), np.abs(cache.v).max())
    assert np.abs(k_gpu - cache.k[:, : L + len(t2)]).max() < kv_tol
    assert np.abs(v_gpu - cache.v[:, : L + len(t2)]).max() < kv_tol


def _fp32_tol(got, want):
    assert np.abs(got - want).max() < FP32_TOL


def _bf16_tol(got, want):
    rel = np.abs(got - want).max(axis=1) / np.abs(want).max(axis=1)
    assert rel.max() < BF16_REL, rel.max()


@pytest.mark.parametrize("seed,L_prompt", [(0, 32), (1, 33), (2, 130), (3, 9)])
def test_verify_logits_fp32_c1(seed, L_prompt):
    eng, W = make(C1T, C1P, seed)
    _verify_case(eng, W, C1T, C1P, seed, L_prompt, _fp32_tol)
    eng.close()


@pytest.mark.parametrize("seed,L_prompt", [(0, 40), (1, 257)])
def test_verify_logits_bf16(seed, L_prompt):
    P = synth.DecodeParams(4, 9, 4, 16, 8)
    eng, W = make(MIDB, P, seed)
    _verify_case(eng, W, MIDB, P, seed, L_prompt, _bf16_tol)
    eng.close()


def test_packed_block_equals_separate_causal_forwards_on_gpu():
    """Eq. 8 on the GPU itself, bit for bit: a suffix row's logits equal those of the same token decoded
    as plain causal text (which is what makes the method lossless on this library)."""
    P = synth.DecodeParams(3, 4, 2, 4, 8, seed_prompt=False)
    eng, _ = make(MIDB, P, 5)
    rng = np.random.default_rng(5)
    prompt = rng.integers(0, MIDB.vocab, 70).astype(np.int32)
    d = rng.integers(0, MIDB.vocab, 3).tolist()
    cands = rng.integers(0, MIDB.vocab, (2, 3))
    eng.phrase_update(np.concatenate([np.full((2, 1), d[-1]), cands], axis=1))
    eng.prefill(prompt)
    eng.assemble_candidates(draft=d)
    tok = eng.block_get()[0]
    assert len(tok) == 10
    _, logits = eng.verify_forward(want_logits=True)
    packed = logits[:10].clone()
    order = [tok[4:7].tolist(), tok[7:10].tolist()]
    for j, suffix in enumerate(order):
        eng.reset()
        eng.prefill(prompt)
        lin = [int(prompt[-1])] + d + suffix
        rows = []
        for t in lin:                                  # one token per forward, like plain decoding
            eng.assemble_causal(binding.OURO_TARGET, [t])
            _, lg = eng.verify_forward(want_logits=True)
            rows.append(lg[0].clone())
            eng.advance(binding.OURO_TARGET, 1)
        rows = torch.stack(rows)
        assert torch.equal(rows[:4], packed[:4])
        assert torch.equal(rows[4:], packed[4 + 3 * j: 7 + 3 * j])
    eng.close()


# ------------------------------------------------------------- acceptance, compaction, harvest

def _hand_trace(name):
    from test_oracle_ouroboros import load_trace
    return load_trace(name)


@pytest.mark.parametrize("name", ["trace_partial_accept.txt", "trace_full_accept.txt", "trace_tie.txt"])
def test_hand_traces_on_gpu(name):
    t = _hand_trace(name)
    gamma, beta = t["gamma"], t["beta"]
    P = synth.DecodeParams(gamma, beta, max(1, len(t["candidates"])), 8, 4, harvest_accepted=False, seed_prompt=False)
    eng, _ = make(TINY, P)
    for c in t["candidates"]:
        eng.phrase_update([[t["draft"][-1]] + c])
    prompt = np.array([1, 2, 3, 4, 5, 6, 7, t["pending"]], dtype=np.int32)
    eng.prefill(prompt)
    # candidates come back newest first; the traces list them in block order
    eng.count.fill_(len(t["candidates"]))
    if t["candidates"]:
        eng.suffix[: len(t["candidates"]) * (beta - 1)] = torch.tensor(np.array(t["candidates"]).ravel(), dtype=torch.int32, device="cuda")
    eng.assemble_candidates(draft=t["draft"], lookup_here=False)
    eng.verify_forward()
    o = torch.tensor(t["outputs"], dtype=torch.int32, device="cuda")
    n, chosen, A, acc = eng.accept_and_compact(o)
    assert (A, chosen, acc.tolist()) == (t["A"], t["chosen"], t["accepted"]) and n == len(t["accepted"])
    assert eng.get_state()[0] == 7 + t["new_length_minus_L"] and eng.get_state()[2] == t["accepted"][-1]
    if "pool_after" in t:
        assert gpu_pool_rows(eng)[0] == t["pool_after"]
    if "ops_matched_only" in t:
        assert gpu_pool_rows(eng)[0] == [op[1] for op in t["ops_matched_only"]]
    eng.close()


@pytest.mark.parametrize("gamma,beta,K,flags", [
    (4, 4, 4, {}), (3, 3, 2, {}), (2, 9, 4, {}), (5, 2, 3, {}), (4, 4, 0, {}),
    (4, 4, 4, dict(harvest_accepted=False, seed_prompt=False)),
    (6, 3, 3, dict(harvest_candidates=False)), (4, 5, 4, dict(harvest_matched=False, harvest_accepted=False))])
def test_accept_compact_harvest_fuzz(gamma, beta, K, flags):
    """Random verification outcomes injected as the argmax vector: every integer result, the moved KV rows
    and the pool contents must equal the oracle's, step after step."""
    P = synth.DecodeParams(gamma, beta, K, 4, 6, **flags)
    S = beta - 1
    eng, _ = make(TINY, P)
    rng = np.random.default_rng(gamma * 100 + beta * 10 + K)
    V = 4                                                     # tiny alphabet: matches happen all the time
    prompt = rng.integers(0, V, 12).astype(np.int32)
    eng.prefill(prompt)
    pool = oracle_pool(P)
    pool.apply(ob.prompt_ops(prompt, beta, P))
    seq = prompt.tolist()
    moved = full = 0
    for step in range(40):
        L = len(seq) - 1
        assert eng.get_state()[0] == L and eng.get_state()[2] == seq[-1]
        d = rng.integers(0, V, gamma).tolist()
        cands = pool.lookup(d[-1], K)
        eng.assemble_candidates(draft=d)
        tokens, pos, group, vis = ob.build_block(L, seq[-1], d, cands)
        assert eng.block_get()[0].tolist() == tokens
        B = len(tokens)
        eng.verify_forward()
        torch.cuda.synchronize()
        k_before = eng.tm.k_cache.clone(); v_before = eng.tm.v_cache.clone()
        # outputs that agree with the row's successor most of the time
        o = rng.integers(0, V, B)
        for b in range(B):
            if rng.random() < 0.8:
                if b < gamma:
                    o[b] = tokens[b + 1]
                elif b == gamma and cands:
                    o[b] = cands[int(rng.integers(0, len(cands)))][0]
                elif b > gamma and (b - gamma) % S != 0:          # not the last row of its suffix
                    o[b] = tokens[b + 1]
        o_dev = torch.tensor(o, dtype=torch.int32, device="cuda")
        n, chosen, A, acc = eng.accept_and_compact(o_dev)
        A2, j2, m2, acc2 = ob.accept(tokens, o.tolist(), gamma, S, len(cands))
        assert (n, chosen, A, acc.tolist()) == (len(acc2), j2, A2, acc2)
        # compaction: expected cache = before + the oracle's moves
        cache = tf.KVCache(dataclasses.replace(TINY, n_layers=1, max_seq=TINY.max_seq))
        cache.length = L
        moves = ob.compact(cache, L, gamma, S, A2, j2, m2)
        k_exp, v_exp = k_before.clone(), v_before.clone()
        for s, dst in moves:
            k_exp[:, dst] = k_before[:, s]; v_exp[:, dst] = v_before[:, s]
        Ln = cache.length
        assert torch.equal(eng.tm.k_cache[:, :Ln], k_exp[:, :Ln]) and torch.equal(eng.tm.v_cache[:, :Ln], v_exp[:, :Ln])
        moved += len(moves); full += A2 == gamma
        seq += acc2
        pool.apply(ob.harvest_ops(tokens, o.tolist(), gamma, S, len(cands), A2, seq, len(acc2), P))
        assert gpu_pool_rows(eng) == pool_rows(pool)
        if len(seq) + P.block_max + 1 >= TINY.max_seq:
            break
    assert full > 3 and (moved > 0 or K < 2 or S == 0)
    eng.close()


# -------------------------------------------------------------------------- end to end (C1)

@pytest.fixture(scope="module")
def c1():
    w = synth.model_weights(C1T, 0, device="cuda:0")
    eng = binding.Engine(C1T, w, C1P, C1D, w)
    W = tf.Weights(C1T, synth.model_weights(C1T, 0))
    yield eng, W, tf.Weights(C1D, synth.model_weights(C1T, 0))
    eng.close()


C1_SEEDS = [0, 1, 2, 4]
_c1_seen = {}


@pytest.mark.parametrize("seed", C1_SEEDS)
def test_generate_c1_matches_oracle_and_vanilla(c1, seed):
    eng, W, Wd = c1
    prompt = synth.prompt(seed, C1T.vocab, C1R["n"], C1R["copy_frac"], *C1R["span"])
    gen = C1R["gen"]
    out, stats = eng.generate(prompt, gen)
    pool_gpu = gpu_pool_rows(eng)
    van, vstats = eng.generate_vanilla(prompt, gen)
    assert np.array_equal(out, van)                                   # lossless on the GPU, bit for bit
    assert vstats["target_calls"] == gen and stats["target_calls"] <= gen
    trace = []
    ref, rstats = ob.generate(W, ob.ModelDrafter(Wd), prompt, gen, C1P, trace=trace)
    assert out.tolist() == ref                                        # and equal to the oracle's text
    assert stats["target_calls"] == rstats["target_calls"]
    assert stats["full_accepts"] == sum(a == C1P.gamma for a in rstats["A"])
    assert stats["suffix_tokens"] == sum(rstats["m"])
    assert stats["candidates"] == sum(rstats["n_cand"])
    assert pool_gpu[0] == [list(p) for _, p in trace[-1]["pool"]]    # same pool, same order
    assert pool_gpu[1] == [s for s, _ in trace[-1]["pool"]]
    _c1_seen[seed] = (sum(rstats["A"]), stats["suffix_tokens"], stats["target_calls"])
    if len(_c1_seen) == len(C1_SEEDS):
        # The early-exit draft (one of the target's two layers) agrees with the target only now and then: seed 0 runs
        # with block efficiency 1 (no draft token is ever accepted).  Over the seeds draft tokens must have been
        # accepted, or this comparison would not exercise acceptance at all.  Phrase suffixes are never accepted
        # with these natural drafts; the replayed-draft test below asserts suffix_tokens > 0.
        assert sum(v[0] for v in _c1_seen.values()) > 20, _c1_seen
        assert any(v[2] < gen for v in _c1_seen.values()), _c1_seen


def test_teacher_forced_steps_c1(c1):
    """Step the GPU through its own API; at every step the oracle evaluates the same block on the same
    history: logits within tolerance, integer results and pool bit exact."""
    eng, W, Wd = c1
    P = C1P
    prompt = synth.prompt(4, C1T.vocab, 32, 0.5, 8, 8)
    eng.reset(); eng.prefill(prompt)
    cache = tf.KVCache(C1T); ob.prefill(W, cache, list(prompt[:-1]))
    pool = oracle_pool(P); pool.apply(ob.prompt_ops(prompt, P.beta, P))
    seq = prompt.tolist()
    for step in range(12):
        L = cache.length
        d = eng.draft().cpu().numpy()[: P.gamma].tolist()
        eng.assemble_candidates()
        tok = eng.block_get()[0].tolist()
        cands = pool.lookup(d[-1], P.K)
        tokens, pos, group, vis = ob.build_block(L, seq[-1], d, cands)
        assert tok == tokens
        am, logits = eng.verify_forward(want_logits=True)
        want = tf.forward(W, cache, tokens, pos, vis)
        assert np.abs(logits[: len(tokens)].cpu().numpy() - want).max() < FP32_TOL
        o = am[: len(tokens)].cpu().numpy().tolist()
        n, chosen, A, acc = eng.accept_and_compact()
        A2, j2, m2, acc2 = ob.accept(tokens, o, P.gamma, P.S, len(cands))
        assert (n, chosen, A, acc.tolist()) == (len(acc2), j2, A2, acc2)
        ob.compact(cache, L, P.gamma, P.S, A2, j2, m2)
        seq += acc2
        pool.apply(ob.harvest_ops(tokens, o, P.gamma, P.S, len(cands), A2, seq, len(acc2), P))
        assert gpu_pool_rows(eng) == pool_rows(pool)
        Ln = cache.length
        assert np.abs(eng.tm.k_cache[:, :Ln].cpu().numpy() - cache.k[:, :Ln]).max() < 1e-4
        assert np.abs(eng.tm.v_cache[:, :Ln].cpu().numpy() - cache.v[:, :Ln]).max() < 1e-4


def test_external_drafter_replay_is_lossless(c1):
    eng, W, _ = c1
    prompt = synth.prompt(9, C1T.vocab, 32, 0.5, 8, 8)
    van, _ = eng.generate_vanilla(prompt, 64)
    truth = np.concatenate([prompt, van, np.zeros(16, dtype=np.int32)])
    eng.set_drafter(lambda seq, g, step: synth.corrupt_drafts(3, truth, len(seq), g, C1T.vocab, 0.05, 0.05, step))
    try:
        out, stats = eng.generate(prompt, 64)
        pool_gpu = gpu_pool_rows(eng)
    finally:
        eng.set_drafter(None)
    assert np.array_equal(out, van)
    drafter = ob.FixedDrafter(lambda seq, g, step: synth.corrupt_drafts(3, truth, len(seq), g, C1T.vocab, 0.05, 0.05, step))
    trace = []
    ref, rstats = ob.generate(W, drafter, prompt, 64, C1P, trace=trace)
    assert out.tolist() == ref and stats["target_calls"] == rstats["target_calls"]
    assert stats["suffix_tokens"] == sum(rstats["m"]) > 0
    assert pool_gpu[0] == [list(p) for _, p in trace[-1]["pool"]]


def test_history_reuse_and_eos(c1):
    eng, W, Wd = c1
    p1 = synth.prompt(10, C1T.vocab, 24, 0.5, 8, 8)
    p2 = synth.prompt(11, C1T.vocab, 24, 0.5, 8, 8)
    eng.generate(p1, 24)
    n1 = eng.pool_export()[0].shape[0]
    out2, _ = eng.generate(p2, 24, keep_pool=True)                    # Section 3.4: the pool survives the query
    assert eng.pool_export()[0].shape[0] > 0 and n1 > 0
    assert np.array_equal(out2, eng.generate_vanilla(p2, 24)[0])
    pool = oracle_pool(C1P)
    for p in (p1, p2):
        ref, _ = ob.generate(W, ob.ModelDrafter(Wd), p, 24, C1P, pool=pool)
    eng.generate(p1, 24); eng.generate(p2, 24, keep_pool=True)
    assert gpu_pool_rows(eng)[0] == pool_rows(pool)[0]
    # stop token
    van, _ = eng.generate_vanilla(p1, 24)
    eos = int(van[7])
    Pe = dataclasses.replace(C1P, eos_token=eos)
    w = synth.model_weights(C1T, 0, device="cuda:0")
    e2 = binding.Engine(C1T, w, Pe, C1D, w)
    cut = van[: van.tolist().index(eos) + 1]
    assert np.array_equal(e2.generate(p1, 24)[0], cut) and np.array_equal(e2.generate_vanilla(p1, 24)[0], cut)
    e2.close()


# ------------------------------------------------------------------ lossless in bf16, edge cases

def test_bf16_ouroboros_is_bit_identical_to_vanilla():
    P = synth.DecodeParams(4, 9, 4, 32, 8)
    eng, _ = make(MIDB, P, 3)
    prompt = synth.prompt(3, MIDB.vocab, 96, 0.3, 8, 32)
    van, _ = eng.generate_vanilla(prompt, 160)
    truth = np.concatenate([prompt, van, np.zeros(32, dtype=np.int32)])
    for p_sub in (0.0, 0.15):
        eng.set_drafter(lambda seq, g, step: synth.corrupt_drafts(1, truth, len(seq), g, MIDB.vocab, p_sub, 0.05, step))
        out, stats = eng.generate(prompt, 160)
        assert np.array_equal(out, van)
        assert stats["target_calls"] < 160 and stats["suffix_tokens"] > 0
    eng.set_drafter(None)
    eng.close()


def test_edge_cases():
    P = synth.DecodeParams(4, 4, 4, 8, 4)
    eng, W = make(TINY, P)
    # a one-token prompt: nothing to prefill, the pool stays empty at first
    out, _ = eng.generate_vanilla(np.array([5], dtype=np.int32), 6)
    assert out.tolist() == ob.vanilla_greedy(W, [5], 6)
    # capacity: the cache cannot take prompt + block
    with pytest.raises(binding.OuroError) as e:
        eng.reset(); eng.prefill(np.zeros(TINY.max_seq - 3, dtype=np.int32))
    assert e.value.status == binding.OURO_ECAPACITY
    # call order: verify without a block, accept without a verification
    eng.reset(); eng.prefill(np.array([1, 2, 3], dtype=np.int32))
    with pytest.raises(binding.OuroError) as e:
        eng.verify_forward()
    assert e.value.status == binding.OURO_ESTATE
    with pytest.raises(binding.OuroError) as e:
        eng.accept_and_compact()
    assert e.value.status == binding.OURO_ESTATE
    # no draft model and no drafter
    with pytest.raises(binding.OuroError):
        eng.draft()
    # token out of range
    with pytest.raises(binding.OuroError) as e:
        eng.reset(); eng.prefill(np.array([1, TINY.vocab], dtype=np.int32))
    assert e.value.status == binding.OURO_EINVAL
    # widest block the library takes: 1 + 7 + 8*15 = 128 rows
    Pw = synth.DecodeParams(7, 16, 8, 2, 16, seed_prompt=False)
    e2, W2 = make(TINY, Pw, 1)
    grams = np.random.default_rng(0).integers(0, TINY.vocab, (8, 16)); grams[:, 0] = 9
    e2.phrase_update(grams)
    prompt = synth.prompt(0, TINY.vocab, 20, 0.0, 4, 4)
    e2.prefill(prompt)
    d = [1, 2, 3, 4, 5, 6, 9]
    e2.assemble_candidates(draft=d)
    tok, pos, grp, mask = e2.block_get()
    assert len(tok) == 128
    _, logits = e2.verify_forward(want_logits=True)
    cache = tf.KVCache(TINY); ob.prefill(W2, cache, list(prompt[:-1]))
    cands = [tok[8 + 15 * j: 8 + 15 * (j + 1)].tolist() for j in range(8)]
    t2, p2, g2, vis = ob.build_block(19, prompt[-1], d, cands)
    assert np.abs(logits.cpu().numpy() - tf.forward(W2, cache, t2, p2, vis)).max() < FP32_TOL
    eng.close(); e2.close()


# ----------------------------------------------- full-size verify step (the benchmark's configuration)

@pytest.mark.parametrize("L", [1024, 4096])
def test_verify_step_full_size_c2(L):
    """One 7B-shaped layer + LM head, 37-row candidate block on a random KV cache of L tokens, exactly as
    bench.py runs it: logits of every row against the oracle, acceptance and pool bit exact."""
    T, _, P, _ = synth.config("C2")
    w = synth.model_weights(T, 0, device="cuda:0")
    eng = binding.Engine(T, w, P)
    k, v = synth.kv_fill(T, 1, L, device="cuda:0")
    eng.tm.k_cache.copy_(k); eng.tm.v_cache.copy_(v)
    W = tf.Weights(T, {n: (t.cpu() if n != "layers" else [{a: b.cpu() for a, b in lw.items()} for lw in t]) for n, t in w.items()})
    cache = tf.KVCache(T, k.double().cpu().numpy(), v.double().cpu().numpy(), L)
    rng = np.random.default_rng(L)
    d = rng.integers(0, T.vocab, P.gamma).tolist()
    grams = np.concatenate([np.full((P.K, 1), d[-1]), rng.integers(0, T.vocab, (P.K, P.S))], axis=1)
    eng.phrase_update(grams)
    pool = oracle_pool(P)
    for g in grams:
        pool.insert(g)
    eng.set_state(L, 17)
    eng.assemble_candidates(draft=d)
    tok = eng.block_get()[0].tolist()
    tokens, pos, group, vis = ob.build_block(L, 17, d, pool.lookup(d[-1], P.K))
    assert tok == tokens and len(tok) == 37
    am, logits = eng.verify_forward(want_logits=True)
    want = tf.forward(W, cache, tokens, pos, vis)
    got = logits[:37].cpu().numpy().astype(np.float64)
    _bf16_tol(got, want)
    o = am[:37].cpu().numpy().tolist()
    n, chosen, A, acc = eng.accept_and_compact()
    A2, j2, m2, acc2 = ob.accept(tokens, o, P.gamma, P.S, P.K)
    assert (n, chosen, A, acc.tolist()) == (len(acc2), j2, A2, acc2)
    seq = [0] * L + [17] + acc2
    pool.apply(ob.harvest_ops(tokens, o, P.gamma, P.S, P.K, A2, seq, len(acc2), P))
    assert gpu_pool_rows(eng) == pool_rows(pool)
    eng.close()


# ------------------------------------------------------------ 7B-shaped pair: lossless at scale

def test_c3_shapes_ouroboros_is_bit_identical_to_vanilla():
    """Target 7B-shaped (32 layers), draft 1.1B-shaped (GQA 8:1, head_dim 64), bf16, replayed drafts and a
    replayed phrase source: the generated text must equal plain greedy decoding on the same kernels bit for
    bit, with phrase suffixes actually accepted along the way."""
    T, D, P, R = synth.config("C3")
    wt = synth.model_weights(T, 0, device="cuda:0")
    wd = synth.model_weights(D, 100, device="cuda:0")
    eng = binding.Engine(T, wt, P, D, wd)
    prompt = synth.prompt(0, T.vocab, 96, R["copy_frac"], *R["span"])
    gen = 72
    van, _ = eng.generate_vanilla(prompt, gen)
    truth = np.concatenate([prompt, van, np.zeros(64, dtype=np.int32)])

    def drafter(seq, g, step):
        d = synth.corrupt_drafts(5, truth, len(seq), g, T.vocab, 0.12, 0.03, step)
        grams = np.empty((P.K, P.beta), dtype=np.int32)
        for j in range(P.K):
            grams[j, 0] = d[-1]
            grams[j, 1:] = synth.corrupt_drafts(11 + j, truth, len(seq) + g, P.S, T.vocab, 0.08 * (j + 1), 0.0, step)
        eng.phrase_update(grams[::-1])
        return d

    eng.set_drafter(drafter)
    out, st = eng.generate(prompt, gen)
    eng.set_drafter(None)
    assert np.array_equal(out, van)
    assert st["suffix_tokens"] > 0 and st["target_calls"] < gen // 2
    nat, st2 = eng.generate(prompt, 24)                      # the draft model's own (chance-level) drafts
    assert np.array_equal(nat, van[:24]) and st2["draft_calls"] == 4 * st2["target_calls"]
    eng.close()


# ------------------------------------------------------------------- phrase-level drafting (Section 3.1)

def test_phrase_level_drafting_c1_matches_oracle():
    """The draft model drafts phrase by phrase: same text, same target calls and the oracle's number of draft
    forwards; against token-level drafting on the GPU only the number of draft forwards may differ."""
    import dataclasses
    P = dataclasses.replace(C1P, draft_phrases=True)
    w = synth.model_weights(C1T, 0, device="cuda:0")
    eng = binding.Engine(C1T, w, P, C1D, w)
    tok = binding.Engine(C1T, w, C1P, C1D, w)
    W = tf.Weights(C1T, synth.model_weights(C1T, 0))
    Wd = tf.Weights(C1D, synth.model_weights(C1T, 0))
    fewer = 0
    for seed in (0, 1, 4):
        prompt = synth.prompt(seed, C1T.vocab, C1R["n"], C1R["copy_frac"], *C1R["span"])
        gen = C1R["gen"]
        out, stats = eng.generate(prompt, gen)
        pool_gpu = gpu_pool_rows(eng)
        pool = oracle_pool(P)
        drafter = ob.PhraseDrafter(Wd, P, pool)
        trace = []
        ref, rstats = ob.generate(W, drafter, prompt, gen, P, pool=pool, trace=trace)
        assert out.tolist() == ref
        assert stats["target_calls"] == rstats["target_calls"] and stats["draft_calls"] == drafter.calls
        assert stats["suffix_tokens"] == sum(rstats["m"]) and stats["candidates"] == sum(rstats["n_cand"])
        assert pool_gpu[0] == [list(p) for _, p in trace[-1]["pool"]]
        out2, stats2 = tok.generate(prompt, gen)
        assert np.array_equal(out, out2) and stats2["target_calls"] == stats["target_calls"]
        assert stats2["draft_calls"] == P.gamma * stats2["target_calls"] >= stats["draft_calls"]
        fewer += stats2["draft_calls"] - stats["draft_calls"]
    assert fewer > 0                                   # some round did accept a phrase on the draft side
    eng.close()
    tok.close()


def test_phrase_level_drafting_bf16_self_draft():
    """bf16 on the tensor-core path, the target's own weights as the draft model: drafts are always accepted, the
    pool fills with the text's own phrases, and drafting by phrases must leave text and target calls untouched."""
    import dataclasses
    P0 = synth.DecodeParams(4, 9, 4, 32, 8)
    P1 = dataclasses.replace(P0, draft_phrases=True)
    w = synth.model_weights(MIDB, 3, device="cuda:0")
    prompt = synth.prompt(3, MIDB.vocab, 96, 0.3, 8, 32)
    res = []
    for P in (P0, P1):
        eng = binding.Engine(MIDB, w, P, MIDB, w)
        van, _ = eng.generate_vanilla(prompt, 120)
        out, st = eng.generate(prompt, 120)
        assert np.array_equal(out, van)
        res.append(st)
        eng.close()
    assert res[0]["target_calls"] == res[1]["target_calls"] and res[0]["full_accepts"] == res[0]["target_calls"]
    assert res[1]["draft_calls"] < res[0]["draft_calls"] == 4 * res[0]["target_calls"]     # c of Eq. 6 above 1


@pytest.mark.parametrize("kind", ["phrases", "window"])
@pytest.mark.parametrize("desc", [TINY, MIDB], ids=["f32", "bf16"])
def test_drafting_leaves_an_assembled_target_block_alone(desc, kind):
    """A candidate block's row and candidate counts stay on the device until the forward and the acceptance read them.
    Drafting in between (its blocks have counts of their own) must not change them: block, logits and acceptance are those
    of the same calls without it."""
    P = synth.DecodeParams(3, 4, 3, 16, 8, harvest_matched=False, harvest_candidates=False, harvest_accepted=False,
                           draft_phrases=kind == "phrases", window=6 if kind == "window" else 0)
    eng, _ = make(desc, P, 2, draft=desc)
    prompt = synth.prompt(2, desc.vocab, 40, 0.5, 4, 8)
    L, d = len(prompt) - 1, torch.tensor([1, 2, int(prompt[5])], dtype=torch.int32, device="cuda:0")
    eng.prefill(prompt)
    res = []
    for between in (False, True):
        eng.set_state(L, int(prompt[-1]))
        eng._ck(eng.L.ouro_assemble_candidates(eng.ctx, d.data_ptr(), None, None))
        if between:
            eng.draft()
        am, lg = eng.verify_forward(want_logits=True)
        logits = lg.clone()
        tok = eng.block_get()[0].tolist()
        assert len(tok) > 1 + P.gamma                             # some phrase was found, and not all rows of K candidates
        res.append((tok, logits[: len(tok)], eng.accept_and_compact()[3].tolist()))
    assert res[0][0] == res[1][0] and torch.equal(res[0][1], res[1][1]) and res[0][2] == res[1][2]
    eng.close()


def test_phrase_level_drafting_edge_cases():
    """Long catch-up (the uncached text does not fit one block beside the candidates), K = 0 (every round is a plain
    single-token forward) and beta = 1 (phrases have no suffix): the drafts stay those of token-level drafting."""
    import dataclasses
    w = synth.model_weights(TINY, 2, device="cuda:0")
    prompt = synth.prompt(2, TINY.vocab, 125, 0.5, 4, 8)             # 125 + K*S rows > OURO_MAX_ROWS on the first round
    for gamma, beta, K in ((3, 4, 4), (3, 4, 0), (2, 1, 3)):
        P0 = synth.DecodeParams(gamma, beta, K, 8, 4)
        P1 = dataclasses.replace(P0, draft_phrases=True)
        outs = []
        for P in (P0, P1):
            eng = binding.Engine(TINY, w, P, TINY, w)
            van, _ = eng.generate_vanilla(prompt, 20)
            out, st = eng.generate(prompt, 20)
            assert np.array_equal(out, van)
            outs.append(st)
            eng.close()
        assert outs[0]["target_calls"] == outs[1]["target_calls"]
        assert outs[1]["draft_calls"] <= outs[0]["draft_calls"]
        if K == 0 or beta == 1:
            assert outs[1]["draft_calls"] == outs[0]["draft_calls"]


# --------------------------------------- tcgen05 attention: GQA, several rounds of query rows, span boundaries

GQAB = synth.ModelDesc(2, 512, 8, 2, 128, 1024, 1000, 1200, "bf16")   # 4 query heads per kv head, head_dim 128


def _gqa_case(P, seed, L_prompt):
    eng, W = make(GQAB, P, seed)
    rng = np.random.default_rng(seed)
    prompt = synth.prompt(seed, GQAB.vocab, L_prompt, 0.4, 4, 8)
    eng.reset()
    eng.prefill(prompt)
    d = rng.integers(0, GQAB.vocab, P.gamma).tolist()
    grams = rng.integers(0, GQAB.vocab, (P.K, P.beta)).astype(np.int32)
    grams[:, 0] = d[-1]
    eng.phrase_update(grams)
    pool = oracle_pool(P)
    for g in grams:
        pool.insert(g)
    eng.assemble_candidates(draft=d)
    tok = eng.block_get()[0]
    cands = pool.lookup(d[-1], P.K)
    t2, p2, g2, vis = ob.build_block(len(prompt) - 1, prompt[-1], d, cands)
    assert tok.tolist() == t2 and len(t2) == P.block_max
    am, logits = eng.verify_forward(want_logits=True)
    cache = tf.KVCache(GQAB)
    ob.prefill(W, cache, list(prompt[:-1]))
    want = tf.forward(W, cache, t2, p2, vis)
    got = logits[: len(t2)].cpu().numpy().astype(np.float64)
    _bf16_tol(got, want)
    err = np.abs(got - want).max(axis=1)
    srt = np.sort(want, axis=1)
    safe = (srt[:, -1] - srt[:, -2]) > 2 * err + 1e-12
    assert np.array_equal(am[: len(t2)].cpu().numpy()[safe], tf.argmax_rows(want)[safe])
    eng.close()


@pytest.mark.parametrize("seed,L_prompt", [(0, 40), (1, 509), (2, 1000), (3, 129)])
def test_verify_logits_bf16_gqa_head_dim_128(seed, L_prompt):
    """69 block rows x 4 query heads per kv head = 276 query rows (three rounds of 128) with 8 candidates, at
    cache lengths that put the block inside a chunk, across a span boundary (512) and at the end of a span."""
    _gqa_case(synth.DecodeParams(4, 9, 8, 16, 16, seed_prompt=False), seed, L_prompt)


@pytest.mark.parametrize("gamma,beta,K,L_prompt", [(7, 16, 8, 300), (3, 8, 16, 505)])
def test_verify_logits_bf16_widest_blocks(gamma, beta, K, L_prompt):
    """The widest block (128 rows: four rounds of query rows) and the most groups (16 candidates + trunk)."""
    _gqa_case(synth.DecodeParams(gamma, beta, K, 2, 32, seed_prompt=False), 5, L_prompt)


# ------------------------------------------------------------------ full-width shapes against the oracle

def _oracle_weights(desc, w):
    return tf.Weights(desc, {n: (t.cpu() if n != "layers" else [{a: b.cpu() for a, b in lw.items()} for lw in t]) for n, t in w.items()})


@pytest.mark.parametrize("name,K", [("C4", 8), ("C5", 4)])
def test_verify_logits_full_width_one_layer(name, K):
    """One decoder layer + LM head at the widths of the 34B- and 70B-shaped targets (d 7168 / 8192, 56 / 64 query
    heads on 8 kv heads, FFN 20480 / 28672, vocabulary 64000 / 32000): the candidate block (69 / 37 rows) on a
    prefilled cache, logits, greedy tokens and appended K/V against the oracle."""
    T, _, P, _ = synth.config(name)
    desc = dataclasses.replace(T, n_layers=1, max_seq=448)
    assert P.K == K and P.block_max == 1 + 4 + K * 8
    w = synth.model_weights(desc, 0, device="cuda:0")
    eng = binding.Engine(desc, w, P)
    W = _oracle_weights(desc, w)
    _verify_case(eng, W, desc, P, 2, 150, _bf16_tol, full_block=True)
    eng.close()


def test_teacher_forced_bf16_four_layer_7b_stack():
    """Four 7B-shaped layers (d 4096, FFN 11008, vocabulary 32000), bf16, ten decoding steps with replayed drafts and
    phrases: at every step the oracle evaluates the same block on the same history - logits within the bf16 bound,
    greedy tokens equal wherever the oracle's margin allows, acceptance / compaction / pool bit exact."""
    T, _, P, R = synth.config("C3")
    desc = dataclasses.replace(T, n_layers=4, max_seq=320)
    w = synth.model_weights(desc, 0, device="cuda:0")
    eng = binding.Engine(desc, w, P)
    W = _oracle_weights(desc, w)
    prompt = synth.prompt(1, desc.vocab, 48, R["copy_frac"], 4, 8)
    van, _ = eng.generate_vanilla(prompt, 96)
    truth = np.concatenate([prompt, van, np.zeros(64, dtype=np.int32)])
    eng.reset(); eng.prefill(prompt)
    cache = tf.KVCache(desc); ob.prefill(W, cache, list(prompt[:-1]))
    pool = oracle_pool(P); pool.apply(ob.prompt_ops(prompt, P.beta, P))
    seq = prompt.tolist()
    worst, suffix_tokens, full = 0.0, 0, 0
    for step in range(10):
        L = cache.length
        d = synth.corrupt_drafts(5, truth, len(seq), P.gamma, desc.vocab, 0.10, 0.03, step).tolist()
        grams = np.empty((P.K, P.beta), dtype=np.int32)
        for j in range(P.K):                                   # phrases that continue the draft, more or less corrupted
            grams[j, 0] = d[-1]
            grams[j, 1:] = synth.corrupt_drafts(11 + j, truth, len(seq) + P.gamma, P.S, desc.vocab, 0.08 * (j + 1), 0.0, step)
        eng.phrase_update(grams[::-1])
        for g in grams[::-1]:
            pool.insert(g)
        eng.assemble_candidates(draft=d)
        tok = eng.block_get()[0].tolist()
        cands = pool.lookup(d[-1], P.K)
        tokens, pos, group, vis = ob.build_block(L, seq[-1], d, cands)
        assert tok == tokens
        am, logits = eng.verify_forward(want_logits=True)
        want = tf.forward(W, cache, tokens, pos, vis)
        got = logits[: len(tokens)].cpu().numpy().astype(np.float64)
        rel = np.abs(got - want).max(axis=1) / np.abs(want).max(axis=1)
        worst = max(worst, rel.max())
        assert rel.max() < BF16_REL, (step, rel.max())
        err = np.abs(got - want).max(axis=1)
        srt = np.sort(want, axis=1)
        safe = (srt[:, -1] - srt[:, -2]) > 2 * err + 1e-12
        o = am[: len(tokens)].cpu().numpy()
        assert np.array_equal(o[safe], tf.argmax_rows(want)[safe])
        n, chosen, A, acc = eng.accept_and_compact()
        A2, j2, m2, acc2 = ob.accept(tokens, o.tolist(), P.gamma, P.S, len(cands))
        assert (n, chosen, A, acc.tolist()) == (len(acc2), j2, A2, acc2)
        ob.compact(cache, L, P.gamma, P.S, A2, j2, m2)
        seq += acc2
        pool.apply(ob.harvest_ops(tokens, o.tolist(), P.gamma, P.S, len(cands), A2, seq, len(acc2), P))
        assert gpu_pool_rows(eng) == pool_rows(pool)
        Ln = cache.length
        kv_tol = 2e-2 * max(np.abs(cache.k[:, :Ln]).max(), np.abs(cache.v[:, :Ln]).max())
        assert np.abs(eng.tm.k_cache[:, :Ln].float().cpu().numpy() - cache.k[:, :Ln]).max() < kv_tol
        assert np.abs(eng.tm.v_cache[:, :Ln].float().cpu().numpy() - cache.v[:, :Ln]).max() < kv_tol
        suffix_tokens += m2 if j2 >= 0 else 0
        full += A2 == P.gamma
        assert seq[len(prompt):] == van[: len(seq) - len(prompt)].tolist()      # the accepted text is the greedy text
    assert full >= 3 and suffix_tokens > 0, (full, suffix_tokens)
    eng.close()


@pytest.mark.parametrize("rows", [1, 37])
def test_exact_logit_ties_take_the_smallest_id(rows):
    """Identical rows of the LM head give bit-identical logits when they are accumulated the same way: inside one
    128-entry tile of the head GEMM, or in different tiles that one CTA handles over the whole K range (a tile whose
    K range is split across CTAs adds its partial sums in another order, so it rounds differently).  The greedy
    choice among such equals must be the smallest id - for a single row (plain decoding) and for a candidate block."""
    desc = synth.ModelDesc(1, 256, 4, 4, 64, 512, 32000, 192, "bf16")       # 250 head tiles: whole and split ones
    w = synth.model_weights(desc, 4, device="cuda:0")
    P = synth.DecodeParams(4, 9, 4, 16, 8, seed_prompt=False)
    eng = binding.Engine(desc, w, P)
    tokens = (np.arange(rows) * 7 + 3).astype(np.int32)
    eng.assemble_causal(binding.OURO_TARGET, tokens)
    _, lg = eng.verify_forward(want_logits=True)
    base = lg[:rows].clone()
    # a head row that wins for every token: a large multiple of the mean normalised activation direction is not
    # available from outside, so take the current winner's row of token 0 and scale it up
    win_id = int(base[0].argmax())
    boosted = (w["lm_head"][win_id].float() * 4.0).to(torch.bfloat16)
    # 250 tiles on 148 CTAs: tiles 0..147 are handled whole, 148..249 are split along K
    for ids in ((700, 731, 5000), (18900, 130, 131), (19050, 19000)):
        saved = {i: w["lm_head"][i].clone() for i in ids}
        for i in ids:
            w["lm_head"][i] = boosted
        am, lg = eng.verify_forward(want_logits=True)
        torch.cuda.synchronize()
        vals = {float(lg[0, i]) for i in ids}
        assert len(vals) == 1 and int(lg[0].argmax()) in ids, (vals, int(lg[0].argmax()))
        assert int(am[0]) == min(ids)
        for r in range(rows):                              # every row: the choice is the smallest index among the maxima
            mx = lg[r].max()
            assert int(am[r]) == int(torch.nonzero(lg[r] == mx)[0])
        am2, _ = eng.verify_forward()                      # and the same without materialised logits
        assert torch.equal(am2[:rows], am[:rows])
        for i in ids:
            w["lm_head"][i] = saved[i]
    eng.close()


# ------------------------------------------------------------------ a bounded device-side wait that runs out

def test_bounded_wait_gives_up_and_the_context_recovers():
    """The wait of a split-K tile for its other contributors is bounded.  With the bound set to zero polls it runs out
    at once (nothing is made to fault: the kernels return normally with the status word raised): the call that reads
    results back reports OURO_ETIMEOUT, plain decoding reports it too, and after a reset the same context computes
    oracle-equal logits again."""
    P = synth.DecodeParams(4, 9, 4, 16, 8)
    eng, W = make(MIDB, P, 2)                      # d 256: every q,k,v tile is split four ways
    _verify_case(eng, W, MIDB, P, 2, 40, _bf16_tol)
    eng.accept_and_compact()
    prompt = synth.prompt(2, MIDB.vocab, 40, 0.4, 4, 8)
    eng.set_wait_limit(0)
    eng.reset(); eng.prefill(prompt[:2])           # one causal row: raises the status word on the device
    eng.assemble_candidates(draft=[1, 2, 3, int(prompt[5])])
    eng.verify_forward()
    with pytest.raises(binding.OuroError) as e:
        eng.accept_and_compact()
    assert e.value.status == binding.OURO_ETIMEOUT
    with pytest.raises(binding.OuroError) as e:
        eng.generate_vanilla(prompt, 4)
    assert e.value.status == binding.OURO_ETIMEOUT
    eng.set_wait_limit(-1)
    _verify_case(eng, W, MIDB, P, 2, 40, _bf16_tol)     # reset + prefill + verify: as before the give-up
    eng.accept_and_compact()
    van, _ = eng.generate_vanilla(prompt, 12)
    eng.set_drafter(lambda seq, g, step: [int(van[min(len(seq) - len(prompt) + i, 11)]) for i in range(g)])
    out, _ = eng.generate(prompt, 12)
    eng.set_drafter(None)
    assert len(van) == 12 and np.array_equal(out, van)
    eng.close()


@pytest.mark.parametrize("fuse", ["0", "1"])
@pytest.mark.parametrize("ffn", [512, 7168])
def test_give_up_that_nobody_read_ends_with_the_state(monkeypatch, ffn, fuse):
    """Only acceptance and the whole loops read the status word.  A wait that runs out in a forward or while drafting leaves
    sums nobody fetched in the partial-tile slots; set_state clears the status, so the slots must be empty again with it: the
    step that follows gives the bits it gave before and no time-out.  One launch per GEMM (no hand-over counter in the way)
    and chained launches; one row (on the single rows' kernel, which waits for packets, and, with the long FFN, on the kernel of all blocks),
    a few and a candidate block.  Each time a wait must really have run out."""
    monkeypatch.setenv("OURO_FUSE", fuse)
    P = synth.DecodeParams(4, 9, 4, 16, 8, harvest_matched=False, harvest_candidates=False, harvest_accepted=False)
    desc = dataclasses.replace(MIDB, d_ffn=ffn)
    eng, _ = make(desc, P, 2, draft=desc)          # d 256: every q,k,v tile is split four ways
    prompt = synth.prompt(2, MIDB.vocab, 40, 0.4, 4, 8)
    eng.reset(); eng.prefill(prompt)
    L, d = len(prompt) - 1, [1, 2, 3, int(prompt[5])]

    def step():
        eng.set_state(L, int(prompt[-1]))
        eng.assemble_candidates(draft=d)
        am, lg = eng.verify_forward(want_logits=True)
        n = len(eng.block_get()[0])
        return am[:n].clone(), lg[:n].clone(), eng.accept_and_compact()[3].tolist()

    def one_row():
        eng.assemble_causal(binding.OURO_TARGET, [5])
        eng.verify_forward()

    def few_rows():
        eng.assemble_causal(binding.OURO_TARGET, [5, 6, 7, 8, 9])
        eng.verify_forward()

    def candidates():
        eng.assemble_candidates(draft=d)
        eng.verify_forward()

    want = step()
    for give_up in (one_row, few_rows, candidates, eng.draft):
        eng.set_state(L, int(prompt[-1]))
        eng.set_wait_limit(0)
        before = eng.debug_counts()
        give_up()
        after = eng.debug_counts()
        eng.set_wait_limit(-1)
        assert before["status"] == 0 and after["status"] != 0, give_up
        if give_up is one_row:
            assert (after["rows_launches"] > before["rows_launches"]) == (ffn == 512)
        got = step()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and got[2] == want[2], give_up
    for give_up in (one_row, few_rows):
        eng.set_wait_limit(0)
        give_up()
        assert eng.debug_counts()["status"] != 0
        eng.set_wait_limit(-1)
        eng.reset()
        eng.prefill(prompt)
        got = step()
        assert torch.equal(got[1], want[1]), give_up
    eng.close()


def _partial_tile_slots(eng):
    """The words of the workspace that carry partial sums between CTAs, all 0xffffffff in a fresh context: the run of that
    length that ends in front of the hand-over counters."""
    n = 160 * 2 * 128 * 256
    ws = eng.workspace.view(torch.int32)
    other = torch.cat([(ws != -1).nonzero().flatten(), torch.tensor([ws.numel()], device=ws.device)])
    ends = other[1:][other.diff() > n].tolist()
    assert len(ends) == 1
    return ws[ends[0] - n: ends[0]]


@pytest.mark.parametrize("heads,kv,hd,ffn", [(8, 2, 64, 704), (4, 2, 128, 704), (4, 2, 128, 7168)])
def test_every_launch_leaves_the_partial_tile_slots_empty(heads, kv, hd, ffn):
    """A scratch word counts as arrived when it is anything but EMPTY, so whoever fetches a sum empties the word again.
    After forwards of every kernel size (up to 32, 48, 128 and 256 rows, whose slots are laid out differently), with the row count
    on the device or on the host, and after whole loops, no word may be left full.  (Single rows use slots with the long FFN only.)"""
    desc = synth.ModelDesc(2, 256, heads, kv, hd, ffn, 1000, 700, "bf16")
    P = synth.DecodeParams(4, 9, 4, 16, 8)
    eng, _ = make(desc, P, 3, draft=desc)
    slots = _partial_tile_slots(eng)
    prompt = synth.prompt(3, desc.vocab, 420, 0.4, 4, 8)

    def empty():
        torch.cuda.synchronize()
        return bool((slots == -1).all())

    for n in (1, 2, 15, 48, 49, 100, 128):
        eng.reset()
        eng.assemble_causal(binding.OURO_TARGET, prompt[:n])
        eng.verify_forward()
        assert empty(), n
        if n == 1:
            assert (eng.debug_counts()["rows_launches"] > 0) == (ffn == 704)
    for n in (130, 200, 257, 420):
        eng.reset()
        eng.prefill(prompt[:n])
        assert empty(), n
    eng.draft()
    assert empty()
    eng.assemble_candidates(draft=[1, 2, 3, int(prompt[5])])
    eng.verify_forward()
    eng.accept_and_compact()
    assert empty()
    eng.generate(prompt[:140], 24)
    assert empty()
    eng.close()


def test_partial_sums_that_are_nan_arrive():
    """The word that stands for "not there yet" is a NaN.  Sums that are NaN must arrive all the same: a token whose embedding is
    NaN gives NaN logits and no time-out, and leaves no word full."""
    P = synth.DecodeParams(4, 9, 4, 16, 8)
    w = synth.model_weights(MIDB, 2, device="cuda:0")
    w["embed"][7] = float("nan")
    eng = binding.Engine(MIDB, w, P)
    slots = _partial_tile_slots(eng)
    eng.prefill(np.arange(20, 40))
    eng.assemble_candidates(draft=[1, 2, 3, 7])
    _, logits = eng.verify_forward(want_logits=True)
    eng.accept_and_compact()                                      # (would raise on a time-out)
    assert bool(logits[4].isnan().all()) and bool((slots == -1).all())
    eng.close()


@pytest.mark.parametrize("start", [(1 << 31) - 300, (1 << 32) - 300])
def test_hand_over_counters_pass_the_ends_of_their_range(monkeypatch, start):
    """The counters by which the GEMMs of a chain hand over are never reset and are compared by their distance; the marks of single
    rows' packets begin anew, on cleared packets, before they run out.  Started 300 below 2^31 and 2^32 (a forward of
    a block counts 8 to 100 per chain position, one of a single row 20 marks), every one of them goes across; the text equals that of a
    context that starts at zero, and the resets and the set_state in between leave the counters alone."""
    P = synth.DecodeParams(4, 9, 4, 32, 8)
    prompt = synth.prompt(5, MIDB.vocab, 64, 0.3, 8, 32)
    eng0, _ = make(MIDB, P, 5)
    want, _ = eng0.generate_vanilla(prompt, 48)
    eng0.close()
    monkeypatch.setenv("OURO_COUNT_START", str(start))
    eng, _ = make(MIDB, P, 5)
    van, _ = eng.generate_vanilla(prompt, 20)
    assert np.array_equal(van, want[:20])
    truth = np.concatenate([prompt, want, np.zeros(32, dtype=np.int32)])
    eng.set_drafter(lambda seq, g, step: synth.corrupt_drafts(1, truth, len(seq), g, MIDB.vocab, 0.1, 0.05, step))
    out, stats = eng.generate(prompt, 48)
    eng.set_drafter(None)
    assert np.array_equal(out, want) and stats["target_calls"] < 48
    eng.set_state(70, 3)
    assert np.array_equal(eng.generate_vanilla(prompt, 48)[0], want)
    counts = eng.debug_counts()
    gone = [(v - start) % (1 << 32) for i, v in enumerate(counts["counters"]) if i != 3]     # (nobody waits for the last of four GEMMs)
    assert all(300 < g < 1 << 30 for g in gone), gone
    assert counts["rows_launches"] > 100
    if start > 1 << 31:                                            # all launches but the 59 until the marks ran out
        assert counts["mark"] == 1 + 5 * (counts["rows_launches"] - 59), counts
    else:
        assert counts["mark"] == start + 5 * counts["rows_launches"], counts
    eng.close()


@pytest.mark.parametrize("ffn", [9408, 9472, 9536, 1600])
def test_cut_tiles_at_the_edges_of_their_number(ffn):
    """Gate / up tiles of 64 features, eight k-blocks each, on 148 CTAs: 147 of them (a CTA's share of the k-blocks is a whole tile,
    so nothing is cut), 148 (all whole), 149 (one cut into eight pieces), 25 (every CTA has a piece of two k-blocks).  One, 40 and 100 rows,
    whose tokens are finished one or four at a time: logits against the oracle, and a row's bits do not show its block."""
    desc = synth.ModelDesc(1, 512, 4, 2, 128, ffn, 1000, 192, "bf16")
    P = synth.DecodeParams(4, 5, 3, 16, 8)
    eng, W = make(desc, P, 7)
    _verify_case(eng, W, desc, P, 7, 40, _bf16_tol)
    tokens = np.random.default_rng(ffn).integers(0, desc.vocab, 100).astype(np.int32)
    rows = []
    for n in (40, 100):
        eng.set_state(30, 1)
        eng.assemble_causal(binding.OURO_TARGET, tokens[:n])
        rows.append(eng.verify_forward(want_logits=True)[1][:40].clone())
    assert torch.equal(rows[0], rows[1])
    eng.set_state(30, 1)
    for i in range(4):
        eng.assemble_causal(binding.OURO_TARGET, tokens[i: i + 1])
        assert torch.equal(eng.verify_forward(want_logits=True)[1][0], rows[0][i])
        eng.advance(binding.OURO_TARGET, 1)
    eng.close()


# ------------------------------------------------- phrase generation during the draft forward (Section 3.1)

def test_lookahead_window_matches_oracle_c1():
    """Every draft forward carries a lookahead window whose outputs refill it and feed the pool on the device: same text,
    target calls, accepted suffix tokens and pool as the oracle's LookaheadDrafter; candidates come up and get accepted
    without any phrase injected from outside."""
    P = dataclasses.replace(C1P, window=6)
    w = synth.model_weights(C1T, 0, device="cuda:0")
    W = tf.Weights(C1T, synth.model_weights(C1T, 0))
    for draft_desc in (C1D, C1T):                       # the early-exit draft, then the target as its own draft model
        eng = binding.Engine(C1T, w, P, draft_desc, w)
        Wd = tf.Weights(draft_desc, synth.model_weights(C1T, 0))
        got_suffix = got_cand = 0
        for seed in (1, 4):
            prompt = synth.prompt(seed, C1T.vocab, C1R["n"], C1R["copy_frac"], *C1R["span"])
            gen = C1R["gen"]
            out, stats = eng.generate(prompt, gen)
            pool_gpu = gpu_pool_rows(eng)
            van, _ = eng.generate_vanilla(prompt, gen)
            assert np.array_equal(out, van)
            pool = oracle_pool(P)
            drafter = ob.LookaheadDrafter(Wd, P, pool, P.window)
            trace = []
            ref, rstats = ob.generate(W, drafter, prompt, gen, P, pool=pool, trace=trace)
            assert out.tolist() == ref
            assert stats["target_calls"] == rstats["target_calls"] and stats["draft_calls"] == drafter.calls
            assert stats["suffix_tokens"] == sum(rstats["m"]) and stats["candidates"] == sum(rstats["n_cand"])
            assert pool_gpu[0] == [list(p) for _, p in trace[-1]["pool"]]
            got_suffix += stats["suffix_tokens"]
            got_cand += stats["candidates"]
        assert got_cand > 0
        if draft_desc is C1T:
            assert got_suffix > 0                       # the window's phrases are the target's own continuation
        eng.close()


def test_lookahead_window_bf16_self_draft():
    """The same on the tensor-core path (bf16, GQA, head dim 64): lossless, and the window's phrases extend accepted
    drafts although nothing but the prompt and the draft model's own forwards feeds the pool."""
    P0 = synth.DecodeParams(4, 9, 4, 32, 8)
    P1 = dataclasses.replace(P0, window=10)
    w = synth.model_weights(MIDB, 3, device="cuda:0")
    prompt = synth.prompt(3, MIDB.vocab, 96, 0.3, 8, 32)
    res = []
    for P in (P0, P1):
        eng = binding.Engine(MIDB, w, P, MIDB, w)
        van, _ = eng.generate_vanilla(prompt, 120)
        out, st = eng.generate(prompt, 120)
        assert np.array_equal(out, van)
        res.append(st)
        eng.close()
    assert res[1]["candidates"] > 0 and res[1]["suffix_tokens"] > 0
    assert res[1]["target_calls"] <= res[0]["target_calls"]
    with pytest.raises(binding.OuroError):              # a window together with phrase-level drafting is refused
        binding.Engine(MIDB, w, dataclasses.replace(P1, draft_phrases=True), MIDB, w)


# ------------------------------------------------------------ wide blocks of known text

@pytest.mark.parametrize("heads,kv,hd", [(4, 2, 128), (8, 2, 64)])
def test_prefill_in_wide_blocks_is_bit_identical_to_short_blocks(heads, kv, hd):
    """Prompts beyond 128 tokens are prefilled up to 512 rows at a time, without the LM head and the last layer's second
    half.  A token's keys and values must not show it: they equal, bit for bit, those left by blocks of 1 to 100 rows.
    Lengths around the block edges, one that ends a span of 512 keys, and one with a one-row rest."""
    desc = synth.ModelDesc(3, 512, heads, kv, hd, 704, 1024, 900, "bf16")
    P = synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False)
    eng, _ = make(desc, P, 6)
    rng = np.random.default_rng(6)
    text = rng.integers(0, desc.vocab, 780).astype(np.int32)
    eng.reset()
    at = 0
    for n in (1, 100, 47, 100, 3, 96, 100, 100, 100, 100, 32):
        eng.assemble_causal(binding.OURO_TARGET, text[at: at + n])
        eng.verify_forward()
        eng.advance(binding.OURO_TARGET, n)
        at += n
    torch.cuda.synchronize()
    want = [c[:, :at].clone() for c in (eng.tm.k_cache, eng.tm.v_cache)]
    assert bool(torch.isfinite(want[0].float()).all()) and float(want[1].float().abs().max()) > 0
    for n in (129, 130, 256, 257, 258, 385, 513, 514, 600, 770):
        eng.reset()
        eng.tm.k_cache.zero_(); eng.tm.v_cache.zero_()
        eng.prefill(text[:n])                                      # caches n - 1 positions
        for got, ref in zip((eng.tm.k_cache, eng.tm.v_cache), want):
            assert torch.equal(got[:, : n - 1], ref[:, : n - 1]), n
            assert not bool(got[:, n - 1:].any()), n               # and nothing behind them
    eng.close()


@pytest.mark.parametrize("d,heads,kv,hd,ffn", [(4928, 2, 2, 64, 9536), (256, 91, 91, 64, 640), (512, 75, 25, 128, 4800)])
def test_long_text_blocks_with_two_tiles_per_pair(d, heads, kv, hd, ffn):
    """Prompts beyond 256 rows, widths for which a pair of SMs takes two weight tiles at a time: an odd number of tiles (the last
    one is contracted twice), matrices whose last tile is half empty, rows up to and around the edges of a pair's 256 tokens and of its
    two halves.  Keys and values equal, bit for bit, those left by blocks of up to 100 rows."""
    desc = synth.ModelDesc(2, d, heads, kv, hd, ffn, 520, 560, "bf16")
    P = synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False)
    eng = binding.Engine(desc, synth.model_weights(desc, 6, device="cuda:0"), P)
    text = np.random.default_rng(6).integers(0, desc.vocab, 530).astype(np.int32)
    eng.reset()
    at = 0
    while at < 520:
        n = min(100, 520 - at)
        eng.assemble_causal(binding.OURO_TARGET, text[at: at + n])
        eng.verify_forward()
        eng.advance(binding.OURO_TARGET, n)
        at += n
    torch.cuda.synchronize()
    want = [c[:, :at].clone() for c in (eng.tm.k_cache, eng.tm.v_cache)]
    assert bool(torch.isfinite(want[0].float()).all()) and float(want[1].float().abs().max()) > 0
    for n in (258, 300, 385, 386, 513, 520):
        eng.reset()
        eng.tm.k_cache.zero_(); eng.tm.v_cache.zero_()
        eng.prefill(text[:n])
        for got, ref in zip((eng.tm.k_cache, eng.tm.v_cache), want):
            assert torch.equal(got[:, : n - 1], ref[:, : n - 1]), n
            assert not bool(got[:, n - 1:].any()), n
    eng.close()


def _round_bf16(x):
    u = np.asarray(x, dtype=np.float32).view(np.uint32)
    return ((u + 0x7fff + ((u >> 16) & 1)) & 0xffff0000).astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("rows", [16, 200, 300, 512])
def test_norm_factor_of_an_embedding_row_to_the_last_bit(rows):
    """The first norm divides by the root of a sum of squares over 128-column tiles, added up two by two in 32 bits: the columns of a
    group of four, then the 32 groups in halves, then the tiles in order.  Embeddings for which this sum and one along the columns of a
    group give neighbouring factors; values in front of the norm (single weights on columns that are one, so no sum can round) that
    land on different sides of a bf16 rounding with the two.  Gathered by the chained launch (16 and 200 rows) and by the kernel of
    long blocks."""
    d, kv, n_tok, per_tok = 512, 4, 16, 16
    rng = np.random.default_rng(1)
    x = _round_bf16(rng.standard_normal((20000, d)).astype(np.float32))
    x[:, :3] = 1
    sq = (x * x).reshape(-1, d // 128, 32, 4)

    def factor(groups):
        i = np.arange(32)
        for o in (16, 8, 4, 2, 1):
            groups = groups + groups[..., i ^ o]
        total = np.zeros(len(groups), dtype=np.float32)
        for tile in range(groups.shape[1]):
            total = total + groups[:, tile, 0]
        return np.float32(1) / np.sqrt((total.astype(np.float64) / d + np.float64(np.float32(1e-5))).astype(np.float32))

    by_twos = factor((sq[..., 0] + sq[..., 1]) + (sq[..., 2] + sq[..., 3]))
    in_a_row = factor(((sq[..., 0] + sq[..., 1]) + sq[..., 2]) + sq[..., 3])
    pick = np.flatnonzero(by_twos != in_a_row)[:n_tok]
    assert len(pick) == n_tok
    values = []
    for t in pick:
        found = 0
        while found < per_tok:
            middle = np.float32(1 + (2 * int(rng.integers(0, 128)) + 1) / 256)         # between two bf16 values
            near = (middle / by_twos[t]).view(np.int32) + np.arange(-6, 7, dtype=np.int32)
            near = near.view(np.float32)
            split = _round_bf16(near * by_twos[t]) != _round_bf16(near * in_a_row[t])
            if split.any():
                values.append(near[split][0])
                found += 1
    values = np.array(values, dtype=np.float32)                                       # one per feature of the values: 16 per token
    desc = synth.ModelDesc(1, d, kv, kv, 64, 64, 64, 600, "bf16")
    w = synth.model_weights(desc, 1, device="cuda:0")
    w["embed"].zero_()
    w["embed"][:n_tok] = torch.as_tensor(x[pick], device="cuda:0").bfloat16()
    lw = w["layers"][0]
    lw["attn_norm"].fill_(1)
    lw["wv"].zero_()
    rest = values.copy()
    for column in range(3):                                                           # 24 bits in three bf16 weights
        part = _round_bf16(rest)
        lw["wv"][:, column] = torch.as_tensor(part, device="cuda:0").bfloat16()
        rest = rest - part
    assert not rest.any()
    eng = binding.Engine(desc, w, synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False))
    text = np.resize(np.arange(n_tok, dtype=np.int32), rows + 1)
    eng.prefill(text)
    got = eng.tm.v_cache[0, :rows].reshape(rows, -1).float().cpu().numpy()
    assert np.array_equal(got, _round_bf16(values[None, :] * by_twos[pick][text[:rows], None]))
    eng.close()


@pytest.mark.parametrize("heads,kv,hd,ffn", [(2, 1, 128, 704), (32, 32, 128, 704), (6, 3, 128, 4800), (256, 1, 128, 64), (8, 2, 64, 704)])
def test_long_text_block_behind_a_short_cache(heads, kv, hd, ffn):
    """A draft model that has cached 1 to 300 tokens catches up on a text that ends beyond 512: one block of more than 256 rows, whose
    attention runs in two parts, the first of which sees one span of keys (nothing to fold) up to a cache of 256.  Keys and values equal,
    bit for bit, those left by blocks of up to 100 rows, and no read comes ahead of the block's own keys: what stands in the cache
    before is large and finite."""
    desc = synth.ModelDesc(3, 256, heads, kv, hd, ffn, 520, 830, "bf16")
    P = synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False)
    w = synth.model_weights(desc, 6, device="cuda:0")
    eng = binding.Engine(dataclasses.replace(desc, n_layers=1), w, P, desc, w)
    text = np.random.default_rng(6).integers(0, desc.vocab, 780).astype(np.int32)

    def cache(begin, end, most=100):
        while begin < end:
            n = min(most, end - begin)
            eng.assemble_causal(binding.OURO_DRAFT, text[begin: begin + n])
            eng.verify_forward(binding.OURO_DRAFT)
            eng.advance(binding.OURO_DRAFT, n)
            begin += n

    eng.reset()
    cache(0, 767)
    torch.cuda.synchronize()
    want = [c[:, :767].clone() for c in (eng.dm.k_cache, eng.dm.v_cache)]
    assert bool(torch.isfinite(want[0].float()).all()) and float(want[1].float().abs().max()) > 0
    for L in (1, 100, 200, 255, 256, 257, 300):
        for n in (513, 600, 767):
            if n - L <= 257:
                continue
            for turn in range(20 if heads < 256 else 2):
                eng.reset()
                cache(0, L)
                eng.dm.k_cache[:, L:].fill_(30 + turn); eng.dm.v_cache[:, L:].fill_(-30 - turn)
                eng.prefill(text[:n])
                eng.draft()
                for got, ref in zip((eng.dm.k_cache, eng.dm.v_cache), want):
                    assert torch.equal(got[:, :n], ref[:, :n]), (L, n, turn)
    eng.close()


@pytest.mark.parametrize("heads,kv,hd", [(4, 2, 64), (2, 1, 128)])
def test_long_text_blocks_in_a_cache_beyond_the_span_kernels(heads, kv, hd):
    """A cache of more than 16384 positions is attended to by the generic kernel, which leaves no pieces (and has no room for them):
    blocks of 257 to 512 rows of a prompt too.  Keys and values equal, bit for bit, those left by blocks of up to 100 rows."""
    desc = synth.ModelDesc(2, 256, heads, kv, hd, 704, 520, 16500, "bf16")
    P = synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False)
    eng, _ = make(desc, P, 6)
    text = np.random.default_rng(6).integers(0, desc.vocab, 900).astype(np.int32)
    eng.reset()
    for at in range(0, 900, 100):
        eng.assemble_causal(binding.OURO_TARGET, text[at: at + 100])
        eng.verify_forward()
        eng.advance(binding.OURO_TARGET, 100)
    torch.cuda.synchronize()
    want = [c[:, :900].clone() for c in (eng.tm.k_cache, eng.tm.v_cache)]
    assert bool(torch.isfinite(want[0].float()).all()) and float(want[1].float().abs().max()) > 0
    for n in (258, 513, 600, 900):
        eng.reset()
        eng.tm.k_cache.zero_(); eng.tm.v_cache.zero_()
        eng.prefill(text[:n])
        for got, ref in zip((eng.tm.k_cache, eng.tm.v_cache), want):
            assert torch.equal(got[:, : n - 1], ref[:, : n - 1]), n
            assert not bool(got[:, n - 1:].any()), n
    eng.close()


@pytest.mark.parametrize("heads,kv,hd", [(4, 2, 64), (2, 1, 128)])
def test_candidates_fewer_than_the_launch_is_sized_for_in_a_cache_beyond_the_span_kernels(heads, kv, hd):
    """The forward of a candidate block is launched for the largest block; a fresh context's first block finds one phrase of eight, and
    nobody has described the other rows.  The generic attention kernel, which serves caches of more than 16384 positions, leaves them
    out.  The rows that are there equal, bit for bit, the same tokens decoded one by one."""
    desc = synth.ModelDesc(2, 256, heads, kv, hd, 704, 520, 16500, "bf16")
    P = synth.DecodeParams(4, 9, 8, 4, 8)
    eng, _ = make(desc, P, 6)
    rng = np.random.default_rng(6)
    d = [3, 1, 4, 15]
    eng.set_state(0, 9)
    eng.phrase_update(np.concatenate([[15], rng.integers(0, desc.vocab, 8)]))
    eng.assemble_candidates(draft=d)
    packed = eng.verify_forward(want_logits=True)[1][:13].clone()
    assert bool(torch.isfinite(packed).all())
    tok = eng.block_get()[0]
    assert len(tok) == 13
    eng.set_state(0, 9)
    for r in range(13):
        eng.assemble_causal(binding.OURO_TARGET, [int(tok[r])])
        assert torch.equal(eng.verify_forward(want_logits=True)[1][0], packed[r]), r
        eng.advance(binding.OURO_TARGET, 1)
    eng.close()


def test_draft_catches_up_on_a_long_prompt():
    """The draft model's first block is the whole prompt, the last 128 rows of it or fewer with outputs: its drafts equal
    those of the same model as the target (self-draft), which accepts every one of them."""
    desc = synth.ModelDesc(2, 512, 8, 2, 64, 704, 1024, 700, "bf16")
    P = synth.DecodeParams(4, 5, 2, 16, 8)
    w = synth.model_weights(desc, 8, device="cuda:0")
    eng = binding.Engine(desc, w, P, desc, w)
    for n in (130, 200, 257, 385, 400):
        prompt = synth.prompt(n, desc.vocab, n, 0.4, 4, 8)
        van, _ = eng.generate_vanilla(prompt, 24)
        out, st = eng.generate(prompt, 24)
        assert np.array_equal(out, van) and st["full_accepts"] == st["target_calls"]
    eng.close()


# ------------------------------------------------------------ the one-launch forward of small generic models

@pytest.mark.parametrize("dtype,d,heads,kv,hd,ffn,vocab", [
    ("f32", 128, 4, 4, 32, 344, 512), ("f32", 72, 3, 1, 32, 104, 1000), ("f32", 512, 4, 2, 128, 2048, 264),
    ("bf16", 96, 2, 1, 96, 136, 520), ("bf16", 200, 4, 2, 64, 72, 1032),
    ("f32", 136, 4, 4, 32, 1208, 4739), ("bf16", 328, 2, 1, 96, 2040, 5001)])
def test_one_launch_forward_matches_oracle_and_single_kernels(dtype, d, heads, kv, hd, ffn, vocab):
    """Widths that are no multiple of a warp's stride, one kv head, head dims 32 to 128, the widest model the one-launch
    forward takes, vocabularies whose columns are taken four at a time with a rest; blocks of 1 to 100 rows (units of two and
    eight rows).  Against the oracle, against the same block through the single kernels (which
    run while one kernel class is being timed), and a row's logits do not depend on the block."""
    desc = synth.ModelDesc(2, d, heads, kv, hd, ffn, vocab, 192, dtype)
    P = synth.DecodeParams(4, 5, 3, 16, 8)
    eng, W = make(desc, P, 9)
    _verify_case(eng, W, desc, P, 9, 40, _fp32_tol if dtype == "f32" else _bf16_tol)
    rng = np.random.default_rng(9)
    for n in (1, 3, 4, 5, 37, 100):
        tokens = rng.integers(0, vocab, n).astype(np.int32)
        outs = []
        for timed in (False, True):
            eng.profile_enable("norm" if timed else "off")
            eng.set_state(30, 1)                      # on the keys the prefill above left
            eng.assemble_causal(binding.OURO_TARGET, tokens)
            am, lg = eng.verify_forward(want_logits=True)
            outs.append((am[:n].clone(), lg[:n].clone()))
        eng.profile_enable("off")
        scale = outs[1][1].abs().amax()
        # fp32: sums of at most 2048 products in another order; bf16: one rounding of an activation may fall the other way
        assert float((outs[0][1] - outs[1][1]).abs().amax() / scale) < (1e-5 if dtype == "f32" else BF16_REL)
        eng.set_state(30, 1)
        for i in range(min(n, 5)):                    # token by token
            eng.assemble_causal(binding.OURO_TARGET, tokens[i: i + 1])
            _, lg = eng.verify_forward(want_logits=True)
            assert torch.equal(lg[0], outs[0][1][i])
            eng.advance(binding.OURO_TARGET, 1)
    eng.close()


@pytest.mark.parametrize("heads,kv,hd", [(4, 2, 32), (3, 1, 128)])
def test_one_launch_forward_rotates_as_spelled_out(heads, kv, hd):
    """A rotated pair (a, b) of a key is (a c - b s, b c + a s) with the second product of each rounded first and the first one fused into
    the sum.  With the key weights equal to the value weights the value cache holds the pair in front of the rotation: keys to the
    last bit, one row per unit, two and eight."""
    desc = synth.ModelDesc(2, 72, heads, kv, hd, 104, 1000, 400, "f32")
    w = synth.model_weights(desc, 3, device="cuda:0")
    for lw in w["layers"]:
        lw["wk"].copy_(lw["wv"])
    eng = binding.Engine(desc, w, synth.DecodeParams(3, 4, 2, 16, 8, seed_prompt=False))
    text = np.random.default_rng(3).integers(0, desc.vocab, 139).astype(np.int32)
    at = 0
    for n in (1, 10, 128):
        eng.assemble_causal(binding.OURO_TARGET, text[at: at + n])
        eng.verify_forward()
        eng.advance(binding.OURO_TARGET, n)
        at += n
    half = hd // 2
    v = eng.tm.v_cache[:, :at].cpu().numpy()
    angle = np.arange(at)[:, None] * np.power(desc.rope_theta, -np.arange(half) / half)
    c, s = (f(angle).astype(np.float32)[None, :, None, :] for f in (np.cos, np.sin))
    a, b = v[..., :half], v[..., half:]
    want = np.concatenate([(a.astype(np.float64) * c - (b * s)).astype(np.float32), (b.astype(np.float64) * c + (a * s)).astype(np.float32)], -1)
    assert np.array_equal(eng.tm.k_cache[:, :at].cpu().numpy(), want)
    eng.close()


def test_one_launch_forward_with_scores_that_overflow():
    """Keys so large that a whole group's scores are -infinity in fp32 have the weight zero, whichever of the four warps of a row
    walks the group and whether it comes first, alone or last there.  wk = wq makes the cached key of the row itself its
    rotated query; the oracle's float64 scores stay finite and give those keys exactly nothing."""
    desc = synth.ModelDesc(1, 64, 2, 2, 32, 96, 100, 256, "f32")
    w = synth.model_weights(desc, 6, device="cuda:0")
    w["layers"][0]["wq"].mul_(40.0)
    w["layers"][0]["wk"].copy_(w["layers"][0]["wq"])
    eng = binding.Engine(desc, w, synth.DecodeParams(2, 3, 1, 4, 4))
    W = tf.Weights(desc, {k: ([{n: t.cpu() for n, t in lw.items()} for lw in v] if k == "layers" else v.cpu()) for k, v in w.items()})
    L = 210                                                       # seven groups: warps 0 to 2 walk two, warp 3 one
    k, v = synth.kv_fill(desc, 3, L, device="cuda:0")
    for groups in ((1,), (2, 6), (3,), (4,), (1, 2, 3, 5), (0, 4, 5)):
        eng.tm.k_cache.copy_(k); eng.tm.v_cache.copy_(v)
        eng.set_state(L, 5)
        eng.assemble_causal(binding.OURO_TARGET, [5])
        eng.verify_forward()
        q = eng.tm.k_cache[0, L].clone()
        assert float(q.abs().sum(1).min()) > 4.0
        for g in groups:
            eng.tm.k_cache[0, 32 * g: 32 * g + 32] = -1e38 * q.sign()
        cache = tf.KVCache(desc, eng.tm.k_cache.double().cpu().numpy(), eng.tm.v_cache.double().cpu().numpy(), L)
        eng.assemble_causal(binding.OURO_TARGET, [5])
        _, logits = eng.verify_forward(want_logits=True)
        want = tf.forward(W, cache, [5], [L], np.ones((1, L + 1), dtype=bool))
        _fp32_tol(logits[:1].cpu().numpy().astype(np.float64), want)
    eng.close()


def test_one_launch_forward_gives_up_and_the_context_recovers():
    """The barriers of the one-launch forward are bounded.  With no polls allowed they give up at once (every CTA leaves, the
    status word is raised): acceptance and plain decoding report it, and a reset, or set_state without anybody having read
    the status, makes the context compute what it did before."""
    P = synth.DecodeParams(3, 4, 4, 8, 4)
    eng, W = make(TINY, P, 2, draft=TINY)
    _verify_case(eng, W, TINY, P, 2, 40, _fp32_tol)
    eng.accept_and_compact()
    prompt = synth.prompt(2, TINY.vocab, 40, 0.4, 4, 8)
    want, _ = eng.generate_vanilla(prompt, 12)

    def logits():
        eng.set_state(30, 7)                                    # on the keys of the prompt
        eng.assemble_causal(binding.OURO_TARGET, [4, 9, 2])
        return eng.verify_forward(want_logits=True)[1][:3].clone()

    ref = logits()
    for call in (eng.verify_forward, eng.draft):
        eng.set_state(30, 7)
        eng.set_wait_limit(0)
        eng.assemble_causal(binding.OURO_TARGET, [4, 9, 2])
        call()
        eng.set_wait_limit(-1)
        assert torch.equal(logits(), ref)
    eng.set_wait_limit(0)
    with pytest.raises(binding.OuroError) as e:
        eng.generate_vanilla(prompt, 4)
    assert e.value.status == binding.OURO_ETIMEOUT
    eng.reset(); eng.prefill(prompt)
    eng.assemble_candidates(draft=[1, 2, int(prompt[5])])
    eng.verify_forward()
    with pytest.raises(binding.OuroError) as e:
        eng.accept_and_compact()
    assert e.value.status == binding.OURO_ETIMEOUT
    eng.set_wait_limit(-1)
    _verify_case(eng, W, TINY, P, 2, 40, _fp32_tol)
    eng.accept_and_compact()
    assert np.array_equal(eng.generate_vanilla(prompt, 12)[0], want)
    eng.close()


@pytest.mark.parametrize("layers", [1, 2])
def test_one_launch_forward_replays_from_a_graph(layers):
    """A captured forward (block assembled inside the graph) gives at every replay what the same calls give uncaptured, with
    other forwards of the context in between: nothing of the barriers is counted on the host."""
    desc = dataclasses.replace(TINY, n_layers=layers)
    P = synth.DecodeParams(3, 4, 4, 8, 4)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        eng, _ = make(desc, P, 4)
        eng.prefill(synth.prompt(4, desc.vocab, 50, 0.4, 4, 8))
        tokens = torch.zeros(9, dtype=torch.int32, device="cuda:0")

        def block():
            eng._ck(eng.L.ouro_assemble_causal(eng.ctx, binding.OURO_TARGET, tokens.data_ptr(), 9))
            return eng.verify_forward(want_logits=True)

        block()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            block()
        rng = np.random.default_rng(4)
        for _ in range(6):
            tokens.copy_(torch.as_tensor(rng.integers(0, desc.vocab, 9).astype(np.int32)))
            am, lg = block()
            want = am[:9].clone(), lg[:9].clone()
            eng.argmax.zero_(); eng.logits.zero_()
            for _ in range(3):
                graph.replay()
            assert torch.equal(eng.argmax[:9], want[0]) and torch.equal(eng.logits[:9], want[1])
            eng.assemble_causal(binding.OURO_TARGET, [1, 2])
            eng.verify_forward()
        side.synchronize()
        del graph
        eng.close()


# ------------------------------------------------------------ spans of the attention

@pytest.mark.parametrize("heads,kv,hd", [(2, 1, 128), (4, 2, 64)])
@pytest.mark.parametrize("L", [120, 127, 1018, 1023, 1024, 5114, 13306])
def test_attention_spans_match_oracle(heads, kv, hd, L):
    """Blocks that straddle the end of a chunk (128), of the short spans (1024), of the first batch of the fold (16 spans:
    5120 keys) and of a lane's first span (32 spans: 13312): logits against the oracle, and a suffix row's logits equal
    those of the same token decoded alone, bit for bit."""
    desc = synth.ModelDesc(1, 256, heads, kv, hd, 256, 520, 13400, "bf16")
    P = synth.DecodeParams(3, 6, 2, 4, 8, seed_prompt=False)
    eng, W = make(desc, P, 10)
    k, v = synth.kv_fill(desc, 3, L, device="cuda:0")
    eng.tm.k_cache.copy_(k); eng.tm.v_cache.copy_(v)
    cache = tf.KVCache(desc, k.double().cpu().numpy(), v.double().cpu().numpy(), L)
    rng = np.random.default_rng(L)
    d = rng.integers(0, desc.vocab, 3).tolist()
    eng.phrase_update(np.concatenate([np.full((2, 1), d[-1]), rng.integers(0, desc.vocab, (2, 5))], axis=1))
    eng.set_state(L, 17)
    eng.assemble_candidates(draft=d)
    tok = eng.block_get()[0].tolist()
    assert len(tok) == 14
    _, logits = eng.verify_forward(want_logits=True)
    got = logits[:14].clone()
    tokens, pos, _, vis = ob.build_block(L, 17, d, [tok[4:9], tok[9:14]])
    assert tok == tokens
    _bf16_tol(got.cpu().numpy().astype(np.float64), tf.forward(W, cache, tokens, pos, vis))
    for rows in ([0, 1, 2, 3, 4, 5, 6, 7, 8], [0, 1, 2, 3, 9, 10, 11, 12, 13]):
        eng.set_state(L, 17)
        for r in rows:
            eng.assemble_causal(binding.OURO_TARGET, [tok[r]])
            _, lg = eng.verify_forward(want_logits=True)
            assert torch.equal(lg[0], got[r]), r
            eng.advance(binding.OURO_TARGET, 1)
    eng.close()


@pytest.mark.parametrize("kv,K,L", [(1, 16, 300), (16, 4, 411), (37, 4, 127), (74, 3, 500), (30, 4, 505), (100, 2, 411)])
def test_groups_shared_by_several_ctas_are_bit_identical_to_plain_decoding(kv, K, L):
    """Head dim 128: trunk and candidates of one span are shared by as many CTAs as SMs are left (here all groups alone, five
    groups on four CTAs, four on two, two spans with block keys, one CTA).  A suffix row's logits equal, bit for bit, those of the
    same token decoded as plain text."""
    desc = synth.ModelDesc(1, 256, kv, kv, 128, 320, 512, L + 80, "bf16")
    P = synth.DecodeParams(3, 4, K, 4, 32, seed_prompt=False)
    eng, _ = make(desc, P, 5)
    k, v = synth.kv_fill(desc, 3, L, device="cuda:0")
    eng.tm.k_cache.copy_(k); eng.tm.v_cache.copy_(v)
    rng = np.random.default_rng(L)
    d = rng.integers(0, desc.vocab, 3).tolist()
    eng.set_state(L, 9)
    eng.phrase_update(np.concatenate([np.full((K, 1), d[-1]), rng.integers(0, desc.vocab, (K, 3))], axis=1).astype(np.int32))
    eng.assemble_candidates(draft=d)
    tok = eng.block_get()[0]
    assert len(tok) == 4 + 3 * K
    packed = eng.verify_forward(want_logits=True)[1][: len(tok)].clone()
    for j in (0, K // 2, K - 1):
        eng.set_state(L, 9)
        own = list(range(4)) + list(range(4 + 3 * j, 7 + 3 * j))
        for r in own:
            eng.assemble_causal(binding.OURO_TARGET, [int(tok[r])])
            assert torch.equal(eng.verify_forward(want_logits=True)[1][0], packed[r]), (j, r)
            eng.advance(binding.OURO_TARGET, 1)
    eng.close()


# ------------------------------------------------------------------ a handful of rows

@pytest.mark.parametrize("d,heads,kv,hd,ffn,vocab", [
    (512, 4, 2, 128, 512, 1000),          # one unit per CTA, every GEMM in pieces of one k-block; half a unit of the vocabulary
    (320, 5, 5, 64, 9536, 520),           # heads that leave half a tile of every matrix empty, one tile cut beside whole ones
    (320, 5, 5, 64, 1280, 520),           # the same on a single row's kernel
    (2048, 32, 4, 64, 5632, 64000),       # pieces taken in turn, more of them than warps share (q,k,v) and fewer; three passes of the head
    (2048, 32, 32, 64, 512, 4104),        # three units per CTA that no tile holds together
    (1024, 8, 8, 128, 24576, 1000),       # activations of 48 KB, three passes of seven units, twenty pieces: too long for a single row's kernel
    (1536, 12, 3, 128, 12288, 1000),      # activations of 24 KB, two passes of six units
    (1024, 8, 2, 128, 11264, 1000),       # ten units per CTA, one tile cut beside whole ones; nineteen pieces
    (1024, 8, 2, 128, 4096, 1000),        # four units per CTA, two warps each
    (256, 2, 1, 128, 1536, 1000),         # as many pieces as are parked at a time
    (7168, 8, 8, 128, 512, 1000),         # four units per CTA, two warps each, k-blocks by the hundred
    (4096, 32, 32, 128, 11008, 1000),     # a layer beyond the single row's kernels
    (1792, 14, 2, 128, 4864, 1000),       # seven query heads per kv head: two rows fill the attention's tile but for two
    (1024, 16, 2, 128, 2816, 1000),       # eight: two rows fill it
])
def test_few_rows_are_bit_identical_to_wider_blocks(d, heads, kv, hd, ffn, vocab):
    """A single row of a model of small layers runs on GEMM kernels of its own, and up to 16 query rows of a kv head without
    candidates on attention of their own (head dim 128), both where they are faster.  A token's logits,
    choice, keys and values must not show which: blocks of 1, 2, 5, 8, 9 and 16 rows against one block of 40, behind 490 keys, so
    that the rows pass the end of a span."""
    desc = synth.ModelDesc(1 if d > 2048 else 2, d, heads, kv, hd, ffn, vocab, 640, "bf16")
    w = synth.model_weights(desc, 5, device="cuda:0")
    eng = binding.Engine(desc, w, synth.DecodeParams(4, 5, 3, 16, 8))
    k, v = synth.kv_fill(desc, 1, 490, device="cuda:0")
    eng.tm.k_cache.copy_(k)
    eng.tm.v_cache.copy_(v)
    tokens = np.random.default_rng(d).integers(0, vocab, 40).astype(np.int32)

    def run(n):
        eng.set_state(490, 1)
        argmax, logits = [], []
        for at in range(0, 40, n):
            part = tokens[at: at + n]
            eng.assemble_causal(binding.OURO_TARGET, part)
            am, lg = eng.verify_forward(want_logits=True)
            argmax.append(am[: len(part)].clone())
            logits.append(lg[: len(part)].clone())
            eng.advance(binding.OURO_TARGET, len(part))
        return torch.cat(argmax), torch.cat(logits), eng.tm.k_cache[:, :530].clone(), eng.tm.v_cache[:, :530].clone()

    want = run(40)
    assert bool(want[1].isfinite().all()) and float(want[1].std()) > 0
    for n in (1, 2, 5, 8, 9, 16):
        for got, ref in zip(run(n), want):
            assert torch.equal(got, ref), n
    eng.close()


@pytest.mark.parametrize("fuse", ["0", "1"])
def test_single_rows_with_every_gemm_a_launch_of_its_own(monkeypatch, fuse):
    """The kernels of a single row hand activations over inside a launch and through memory between launches: plain decoding gives
    the same logits whether GEMMs are chained or not, and those of the wider kernels."""
    monkeypatch.setenv("OURO_FUSE", fuse)
    eng, _ = make(MIDB, synth.DecodeParams(4, 9, 4, 16, 8), 2)
    tokens = np.arange(20, 44, dtype=np.int32)
    eng.set_state(30, 1)
    eng.assemble_causal(binding.OURO_TARGET, tokens)
    want = eng.verify_forward(want_logits=True)[1][:24].clone()
    eng.set_state(30, 1)
    for i in range(24):
        eng.assemble_causal(binding.OURO_TARGET, tokens[i: i + 1])
        assert torch.equal(eng.verify_forward(want_logits=True)[1][0], want[i]), i
        eng.advance(binding.OURO_TARGET, 1)
    eng.close()


@pytest.mark.parametrize("fuse", ["0", "1"])
def test_single_rows_with_a_late_warp(monkeypatch, fuse):
    """One warp of a single row's kernel works out the norm's factor and has nothing to hand back for the GEMMs without one.  It
    may be late by more than such a GEMM and the hand-over behind it (here 30 us a GEMM; they take 1 to 5): no time-out, and the same
    logits.  All GEMMs of this model are a few k-blocks long, so that nothing else holds the others back."""
    desc = synth.ModelDesc(3, 128, 1, 1, 128, 128, 512, 64, "bf16")
    w = synth.model_weights(desc, 4, device="cuda:0")
    prompt = np.arange(3, 20, dtype=np.int32)
    want = None
    for late in ("0", "30000"):
        monkeypatch.setenv("OURO_LATE_NS", late)
        monkeypatch.setenv("OURO_FUSE", fuse)
        eng = binding.Engine(desc, w, synth.DecodeParams(4, 5, 3, 16, 8))
        got = eng.generate_vanilla(prompt, 24)[0].tolist()             # (would raise on a time-out)
        eng.assemble_causal(binding.OURO_TARGET, [5])
        got = got, eng.verify_forward(want_logits=True)[1][0].clone()
        eng.close()
        if want is None:
            want = got
    assert got[0] == want[0] and torch.equal(got[1], want[1])


@pytest.mark.parametrize("layers,d,heads,kv,hd,ffn,vocab,owned", [
    (1, 512, 4, 2, 128, 512, 1000, True),
    (1, 256, 2, 1, 128, 2048, 1000, True),         # 32 k-blocks walked by one warp a unit, in a layer of 3 MB
    (1, 512, 4, 1, 128, 3072, 1000, True),         # 48
    (1, 384, 3, 1, 128, 3072, 1000, False),        # ... in a smaller layer
    (1, 512, 4, 1, 128, 28672, 1000, False),       # 448
    (1, 256, 15, 5, 64, 1600, 1000, True),         # head dim 64: 25
    (1, 384, 48, 6, 64, 1024, 1000, False),        # ... an output projection of 48
    (1, 1024, 8, 2, 128, 11264, 1000, True),       # 72 MB
    (1, 1536, 12, 3, 128, 16896, 1000, False),     # 88 k-blocks of the down projection, 48 of gate and up, in 152 MB
    (1, 2048, 32, 4, 64, 5632, 32000, True),
    (1, 2560, 20, 5, 128, 10240, 1000, False),     # beyond 160 MB
    (2, 256, 2, 1, 128, 256, 262144, False),       # twelve passes of the head behind two layers
    (3, 256, 2, 1, 128, 256, 262144, True),        # ... and three
    (1, 512, 4, 4, 96, 512, 1000, False),          # another head dim
])
def test_single_rows_take_the_kernel_that_is_faster(layers, d, heads, kv, hd, ffn, vocab, owned):
    """Shapes on either side of the lines behind which a single row's own GEMM kernel was measured slower than the
    kernel of wider blocks (narrow layers with a long K: up to twice as slow)."""
    desc = synth.ModelDesc(layers, d, heads, kv, hd, ffn, vocab, 64, "bf16")
    eng = binding.Engine(desc, synth.model_weights(desc, 3, device="cuda:0"), synth.DecodeParams(4, 5, 3, 16, 8))
    for n in (1, 2):
        eng.set_state(20, 1)
        eng.assemble_causal(binding.OURO_TARGET, np.arange(n, dtype=np.int32))
        eng.verify_forward()
        counts = eng.debug_counts()
        assert counts["status"] == 0 and counts["rows_launches"] == (layers + 1 if owned else 0), n     # (layers + 1 launches a row)
    eng.close()


@pytest.mark.parametrize("d,heads,kv,ffn,rows,keys,few", [
    (4096, 32, 32, 11008, 16, 128, True), (4096, 32, 32, 11008, 8, 512, True), (4096, 32, 32, 11008, 9, 129, False),
    (4096, 32, 32, 11008, 1, 513, False), (4096, 32, 8, 11008, 2, 512, True), (4096, 32, 8, 11008, 2, 513, False), (4096, 32, 8, 11008, 3, 129, False),
    (4096, 64, 8, 4096, 2, 128, True), (4096, 64, 8, 4096, 2, 200, False), (512, 4, 2, 512, 8, 512, True), (512, 4, 2, 512, 9, 60, False),
    (512, 4, 2, 512, 2, 513, False), (512, 4, 2, 512, 1, 8192, True), (512, 4, 4, 512, 1, 4096, True), (512, 4, 4, 512, 1, 4097, False),
    (1024, 32, 32, 2816, 1, 512, True), (1024, 32, 32, 2816, 1, 513, False),
])
def test_few_rows_take_the_attention_that_is_faster(d, heads, kv, ffn, rows, keys, few):
    """Blocks on either side of the lines behind which attention with a span's chunks side by side was measured slower: one chunk or
    more, one span or more, query rows, kv heads, kv heads times spans in front of the single rows' GEMMs.  `keys`: those the last row
    sees."""
    desc = synth.ModelDesc(1, d, heads, kv, 128, ffn, 1000, 8448, "bf16")
    eng = binding.Engine(desc, synth.model_weights(desc, 3, device="cuda:0"), synth.DecodeParams(4, 5, 3, 16, 8))
    eng.set_state(keys - rows, 1)
    eng.assemble_causal(binding.OURO_TARGET, np.arange(rows, dtype=np.int32))
    eng.verify_forward()
    counts = eng.debug_counts()
    assert counts["status"] == 0 and counts["few_launches"] == few
    eng.close()
