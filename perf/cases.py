"""Performance cases: what a program that decodes with this library has it do, from one attention
call to a first pass over a long prompt, through the public Python binding.

Model shapes are the repository's configurations at full depth.  Weights are random with the
statistics of a trained decoder in the one respect that matters for comparing two runs: its
predictions are clear-cut.  (With N(0, 0.02) weights everywhere the best of 151936 logits leads by less
than bf16 rounding, so token ids of two correct implementations part within a few steps.)  Matrices are
scaled by their fan-in, the two that write to the residual stream also by the depth, and every LM-head
row leans towards the embedding of the one token it follows.  The acceptance lengths of the decode
steps come from the benchmark's seeded schedule, since no random model drafts what it later verifies.
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2511_08923_b200 import Tidar, pack_weights
from paper_2511_08923_b200.binding import plan_ks
from tidar_synth import CONFIGS, acceptance_schedule

DEVICE = "cuda:0"
EMBED_STD = 0.5          # about the scale of what the layers add to the residual stream
FAVOURITE = 16.0         # the favoured next token's logit, in standard deviations of the others
ROW_BUDGET = 288         # token slots of a step at which the 8b shape turns tensor-bound


def listed():
    return [
        # One layer's attention alone, as a host with its own layers calls it: the smallest call.
        dict(name="attention_1k", kind="attention", hq=32, hkv=8, hd=128, batch=1, k=16, n_lo=1024, n_hi=1024),
        # The same for a ragged batch of four with six query heads per KV head.
        dict(name="attention_ragged", kind="attention", hq=12, hkv=2, hd=128, batch=4, k=8, n_lo=500, n_hi=9001),
        # And over a long context.
        dict(name="attention_32k", kind="attention", hq=32, hkv=8, hd=128, batch=1, k=16, n_lo=32768, n_hi=32768),
        # A short request on the smallest model: all latency and launches.
        dict(name="tiny_generate", kind="generate", model="tiny", k=4, prompt=64, steps=8),
        # One request on a small model, the benchmark's second workload: prompt, then 16 steps (about 128 tokens).
        dict(name="1.5b_generate", kind="generate", model="1.5b", k=16, prompt=512, steps=16),
        # Plain autoregressive decoding with sampling for a small batch (the model's other mode), Q/K/V biases as in that family.
        dict(name="1.5b_ar_batch8", kind="decode", model="1.5b", variant=True, ar=True, temperature=0.7, batch=8, k=1, n_lo=131, n_hi=905, steps=16),
        # One request on the larger model, the benchmark's default workload.
        dict(name="8b_generate", kind="generate", model="8b", k=16, prompt=1024, steps=16),
        # The same with short blocks and an odd prompt: every weight streamed for 20 rows.
        dict(name="8b_generate_k4", kind="generate", model="8b", k=4, prompt=333, steps=32),
        # Continuous batching: eight ragged requests, block lengths planned anew for every step, Q/K norm as in that family.
        dict(name="8b_serve_mixed", kind="decode", model="8b", variant=True, mixed=True, batch=8, k=16, n_lo=203, n_hi=3001, steps=4),
        # A full batch in lock step: the steps that are bound by arithmetic.
        dict(name="8b_serve_batch16", kind="decode", model="8b", batch=16, k=8, n_lo=301, n_hi=2000, steps=2),
        # The first pass over a long prompt, all of it at once.
        dict(name="8b_prefill_4k", kind="prefill", model="8b", k=16, prompt=4096, one_pass=True),
        # Likelihood of a given text.
        dict(name="1.5b_score", kind="score", model="1.5b", prompt=1777, one_pass=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attention", "attention", "generate", "generate", "decode", "decode", "prefill", "score"])
    if kind == "attention":
        hq, hkv, hd = rng.choice([(32, 8, 128), (12, 2, 128), (4, 2, 64)])
        n_hi = _log_int(rng, 64, 32768)
        k = rng.randint(2, 16)
        batch = rng.randint(1, max(1, min(8, 32768 // n_hi, 1088 // (k * (k + 1)))))
        return dict(kind=kind, hq=hq, hkv=hkv, hd=hd, batch=batch, k=k, n_lo=max(1, int(n_hi * rng.uniform(0.2, 1.0))), n_hi=n_hi)
    model = rng.choice(["tiny", "1.5b", "1.5b", "8b", "8b"])
    out = dict(kind=kind, model=model, variant=rng.random() < 0.5)
    if kind == "generate":
        out.update(k=rng.randint(2, 16), prompt=_log_int(rng, 32, 1024), steps=rng.randint(6, 16))
        option = rng.choice(["greedy", "greedy", "sample", "mix"])
        if option == "sample":
            out.update(temperature=0.7)
        elif option == "mix":
            out.update(beta=0.75)
    elif kind == "decode":
        batch = rng.randint(2, 16)
        n_hi = _log_int(rng, 100, 2000)
        out.update(batch=batch, n_lo=max(1, int(n_hi * rng.uniform(0.2, 1.0))), n_hi=n_hi)
        mode = rng.choice(["ar", "mixed", "equal"])
        if mode == "ar":
            out.update(ar=True, k=1, steps=rng.randint(4, 16))
        elif mode == "mixed":
            out.update(mixed=True, k=16, steps=4)
        else:
            out.update(k=rng.randint(2, 8), steps=2)
    elif kind == "prefill":
        out.update(k=rng.randint(2, 16), prompt=_log_int(rng, 100, 4096), one_pass=rng.random() < 0.7)
    else:
        out.update(prompt=_log_int(rng, 100, 2048), one_pass=rng.random() < 0.7)
    return out


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shape(case):
    sh = CONFIGS[case["model"]]
    if case.get("variant"):
        sh = replace(sh, qk_norm=True) if case["model"] == "8b" else replace(sh, qkv_bias=True)
    return sh


def _lengths(case):
    """Cached lengths of the batch, spread over [n_lo, n_hi] out of order."""
    b = case["batch"]
    return [case["n_hi"] - (case["n_hi"] - case["n_lo"]) * (i * 5 % b) // max(1, b - 1) if b > 1 else case["n_hi"] for i in range(b)]


def _weights(sh, gen):
    """(weight dict of the library's layout, favoured next token of every token)."""
    def mat(rows, cols, std):
        return torch.randn(rows, cols, device=DEVICE, dtype=torch.bfloat16, generator=gen).mul_(std)

    def vec(n, std, offset=0.0):
        return (torch.randn(n, device=DEVICE, generator=gen) * std + offset).to(torch.bfloat16)

    d, hd, qo, kvo = sh.d_model, sh.head_dim, sh.n_q_heads * sh.head_dim, sh.n_kv_heads * sh.head_dim
    out_scale = 1.0 / math.sqrt(2 * sh.n_layers)

    def layers():
        for _ in range(sh.n_layers):
            L = dict(attn_norm=vec(d, 0.1, 1.0), ffn_norm=vec(d, 0.1, 1.0),
                     wq=mat(qo, d, d ** -0.5), wk=mat(kvo, d, d ** -0.5), wv=mat(kvo, d, d ** -0.5), wo=mat(d, qo, qo ** -0.5 * out_scale),
                     w_gate=mat(sh.d_ffn, d, d ** -0.5), w_up=mat(sh.d_ffn, d, d ** -0.5), w_down=mat(d, sh.d_ffn, sh.d_ffn ** -0.5 * out_scale))
            if sh.qkv_bias:
                L.update(bq=vec(qo, 0.1), bk=vec(kvo, 0.1), bv=vec(kvo, 0.1))
            if sh.qk_norm:
                L.update(q_norm=vec(hd, 0.1, 1.0), k_norm=vec(hd, 0.1, 1.0))
            yield L

    embed = mat(sh.vocab, d, EMBED_STD)
    if sh.tie_lm_head:
        head, follows = embed, torch.arange(sh.vocab, device=DEVICE)
    else:
        follows = torch.randperm(sh.vocab, device=DEVICE, generator=gen)
        lean = min(1.0, FAVOURITE / math.sqrt(d / 2))
        head = mat(sh.vocab, d, math.sqrt(1 - lean * lean) * d ** -0.5)
        for lo in range(0, sh.vocab, 16384):
            head[lo:lo + 16384].add_(embed[follows[lo:lo + 16384]], alpha=lean * d ** -0.5 / EMBED_STD)
    packed = pack_weights(dict(embed=embed, lm_head=head, final_norm=vec(d, 0.1, 1.0), layers=layers()), DEVICE)
    return packed, torch.argsort(follows).cpu().numpy().astype(np.int32)


def _text(rng, n, favoured):
    """Token ids of which about half are what the model itself would continue with."""
    ids = rng.integers(0, len(favoured) - 1, n).astype(np.int32)          # the last id is the mask token
    for i in np.nonzero(rng.random(n) < 0.5)[0]:
        nxt = favoured[ids[i - 1]] if i else len(favoured) - 1
        if nxt < len(favoured) - 1:
            ids[i] = nxt
    return ids


def _prepare_attention(case, gen):
    hq, hkv, hd, b, k = case["hq"], case["hkv"], case["hd"], case["batch"], case["k"]
    sh = replace(CONFIGS["tiny"], head_dim=hd, n_q_heads=hq, n_kv_heads=hkv, n_layers=1, vocab=64, d_ffn=64, d_model=64)
    lens = _lengths(case)
    pages = (max(lens) + k + 63) // 64

    def rnd(*shape):
        return torch.randn(*shape, device=DEVICE, dtype=torch.bfloat16, generator=gen)
    return dict(
        case=case, lib=Tidar(sh, _weights(sh, gen)[0], k_max=k, max_batch=b, max_seq_len=128),
        args=(rnd(b * k * (k + 1), hq, hd), rnd(b * pages, hkv, 64, hd), rnd(b * pages, hkv, 64, hd),
              torch.randperm(b * pages, device=DEVICE, generator=gen).to(torch.int32).view(b, pages),
              torch.tensor(lens, dtype=torch.int32, device=DEVICE), rnd(b * k * k, hkv, hd), rnd(b * k * k, hkv, hd),
              torch.empty(b * k * (k + 1), hq * hd, dtype=torch.bfloat16, device=DEVICE), b, k))


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    if case["kind"] == "attention":
        return _prepare_attention(case, gen)
    rng = np.random.default_rng(seed)
    sh = _shape(case)
    packed, favoured = _weights(sh, gen)
    k, batch = case.get("k", 1), case.get("batch", 1)
    if case["kind"] == "decode":
        lens = _lengths(case)
        room = max(lens) + 1024
    else:
        lens = [case["prompt"]]
        room = lens[0] + (case.get("steps", 0) + 2) * k
    lib = Tidar(sh, packed, k_max=k, max_batch=batch, max_seq_len=max(room, 2 * k + 1), beta=case.get("beta", 1.0), temperature=case.get("temperature", 0.0),
                sample_seed=seed, prefill_rows=lens[0] + k if case.get("one_pass") else 1024 if case["kind"] == "decode" else 0)
    prompts = [_text(rng, n, favoured) for n in lens]
    base = -lib.arena.data_ptr() % 256                  # the KV pages are the first thing in the arena: [layer][K, V][page][kv head][64][head_dim]
    pages = batch * ((max(room, 2 * k + 1) + 63) // 64)
    n_kv = sh.n_layers * 2 * pages * sh.n_kv_heads * 64 * sh.head_dim
    kv = lib.arena[base:base + 2 * n_kv].view(torch.bfloat16).view(sh.n_layers, 2, pages, sh.n_kv_heads, 64, sh.head_dim)
    seqs = list(range(batch))
    state = dict(case=case, lib=lib, prompts=prompts, kv=kv, seqs=seqs, room=room, turn=0,
                 accept=acceptance_schedule(seed, 64 * batch, max(k, 2)).numpy().reshape(64, batch),
                 want=rng.integers(1, k + 1, (64, batch)))
    if case["kind"] == "decode":
        _fill(state)
    return state


def _fill(state):
    """(Re)starts a standing batch from its prompts."""
    for q, p in zip(state["seqs"], state["prompts"]):
        state["lib"].prefill(q, p, state["case"]["k"])


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _step(state, turn):
    """One decode step of the listed sequences; row i: sequence i's new tokens, then -1."""
    case, lib, seqs = state["case"], state["lib"], state["seqs"]
    if case.get("ar"):
        return np.asarray(lib.ar_step(seqs), dtype=np.int32)[:, None]
    accept = state["accept"][turn % 64]
    if case.get("mixed"):
        ks = plan_ks(len(seqs), case["k"], ROW_BUDGET, state["want"][turn % 64])
        tokens, _ = lib.step_ks(seqs, ks, np.minimum(accept, ks))
    else:
        tokens, _ = lib.step(seqs, np.minimum(accept, case["k"]))
    out = np.full((len(seqs), case["k"]), -1, dtype=np.int32)
    for i, t in enumerate(tokens):
        out[i, :len(t)] = t
    return out


def run(state):
    case, lib = state["case"], state["lib"]
    if case["kind"] == "attention":
        lib.attention(*state["args"])
        return state["args"][7]
    if case["kind"] == "score":
        return lib.score(0, state["prompts"][0])
    if case["kind"] == "prefill":
        return dict(first=lib.prefill(0, state["prompts"][0], case["k"]), kv=state["kv"])
    if case["kind"] == "generate":
        first = lib.prefill(0, state["prompts"][0], case["k"])
        return dict(first=first, tokens=np.stack([_step(state, i) for i in range(case["steps"])]), kv=state["kv"])
    if max(lib.seq_len(q) for q in state["seqs"]) + (case["steps"] + 1) * 2 * case["k"] > state["room"]:
        _fill(state)                                    # the requests are done: the next ones take their places
    turn, state["turn"] = state["turn"], state["turn"] + case["steps"]
    return dict(tokens=np.stack([_step(state, turn + i) for i in range(case["steps"])]), kv=state["kv"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _attention_work(hq, hkv, hd, n, k):
    """(bytes of K and V read, flops) of one sequence's step with n cached positions and block length k."""
    keys = sum(n + j + 1 for j in range(k)) + sum(k * (n + b + 1 + k) for b in range(k))
    return 4 * n * hkv * hd, 4 * hq * hd * keys


def _causal_work(sh, n, rows, head_rows):
    """One pass of n prompt rows (rows in all) with logits for head_rows of them."""
    per_layer = sh.d_model * (2 * sh.n_q_heads + 2 * sh.n_kv_heads) * sh.head_dim + 3 * sh.d_model * sh.d_ffn
    flops = 2 * rows * sh.n_layers * per_layer + 2 * head_rows * sh.vocab * sh.d_model
    flops += sh.n_layers * (2 * sh.n_q_heads * sh.head_dim * n * (n + 1) + 4 * sh.n_q_heads * sh.head_dim * (rows - n) * rows)
    return 2 * (sh.n_layers * per_layer + sh.vocab * sh.d_model) + sh.n_layers * 4 * n * sh.n_kv_heads * sh.head_dim, flops


def _step_work(sh, lens, ks, ar):
    per_layer = sh.d_model * (2 * sh.n_q_heads + 2 * sh.n_kv_heads) * sh.head_dim + 3 * sh.d_model * sh.d_ffn
    params = sh.n_layers * per_layer + sh.vocab * sh.d_model
    total, flops = 2 * params, 0
    for n, k in zip(lens, ks):
        if ar:
            kv, fl, rows = 4 * n * sh.n_kv_heads * sh.head_dim, 4 * sh.n_q_heads * sh.head_dim * (n + 1), 1
        else:
            (kv, fl), rows = _attention_work(sh.n_q_heads, sh.n_kv_heads, sh.head_dim, n, k), k * (k + 1)
        total += sh.n_layers * kv
        flops += sh.n_layers * fl + 2 * rows * params
    return total, flops


def work(case):
    if case["kind"] == "attention":
        hq, hkv, hd, b, k = case["hq"], case["hkv"], case["hd"], case["batch"], case["k"]
        kv, flops = (sum(x) for x in zip(*(_attention_work(hq, hkv, hd, n, k) for n in _lengths(case))))
        rows = b * k * (k + 1)
        return {"bytes": kv + 4 * rows * hq * hd + 4 * b * k * (k + 1) * hkv * hd, "flops": flops}
    sh = _shape(case)
    if case["kind"] == "score":
        n = case["prompt"]
        b, f = _causal_work(sh, n - 1, n - 1, n - 1)
        return {"bytes": b, "flops": f}
    b = f = 0
    if case["kind"] in ("prefill", "generate"):
        n, k = case["prompt"], case["k"]
        b, f = _causal_work(sh, n, n + k, k + 1)
        lens = [n]
    else:
        lens = _lengths(case)
    for _ in range(case.get("steps", 0)):
        ks = plan_ks(len(lens), case["k"], ROW_BUDGET) if case.get("mixed") else [case["k"]] * len(lens)
        sb, sf = _step_work(sh, lens, ks, case.get("ar", False))
        b, f = b + sb, f + sf
        lens = [n + (k + 1) // 2 for n, k in zip(lens, ks)]
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Four times what the tensor-core path and the plain fp32-accumulating kernels (impl=1) differ by:
    attention outputs by 2.5e-3 (rms) and 0.013 (largest, P rounded to bf16); K/V pages up to 3.6e-3 and 0.045 (bf16 activations
    between the kernels); log-probabilities 3e-4 and 1.1e-3.  Token ids were the same in every case."""
    if case["kind"] == "attention":
        return {"rel": 0.01, "max": 0.055}
    if case["kind"] == "score":
        return {"rel": 0.0012, "max": 0.0045}
    return {"rel": 0.014, "max": 0.18, "differ": 0.0}
