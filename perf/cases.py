"""What this library is used for, as measurable cases: score a KV cache, select and compact it, and rescore while decoding.

Every case goes through the public entry points of `paper_2510_07651_b200.api` on inputs that the caller already holds on
the GPU.  Scoring and eviction are separate cases except for fp32 caches: which of two tokens with all but equal scores is
kept, and with it the order of the compacted rows, would otherwise hang on the last bits of a score, so eviction cases
start from given scores (their results are whole numbers and copies, hence exact).
"""
from __future__ import annotations

import math

import torch

from paper_2510_07651_b200 import api

D = 128                                     # head_dim of every model shape the library takes


def listed():
    """The cases that stand for the path; see the comments for what each is in real use."""
    return [
        # The smallest whole eviction: one fp32 attention head with 1024 cached tokens, score, select and compact in one
        # call.  Debugging and validation against other implementations run at this size; latency and launches count.
        dict(name="evict_fp32_head_1k", kind="evict_prefill", dtype="f32", B=1, Hq=1, Hkv=1, W=16, N=1024, budget=256,
             pool="none", pool_kernel=1),
        # A short prompt on a few heads (one tensor-parallel share of a layer): the latency of one scoring call.
        dict(name="score_small_1k", kind="score", dtype="bf16", B=1, Hq=8, Hkv=2, W=16, N=1024, ragged=False, variants="VK"),
        # A layer without grouped queries (every query head has its own KV head): 32 window rows per KV head, odd length.
        dict(name="score_mha_8k", kind="score", dtype="bf16", B=1, Hq=32, Hkv=32, W=32, N=8191, ragged=False, variants="VK"),
        # The Llama-3-8B-shaped layer with 32k cached tokens that the benchmark reports.
        dict(name="score_llama_32k", kind="score", dtype="bf16", B=1, Hq=32, Hkv=8, W=32, N=32768, ragged=False, variants="VK"),
        # The Qwen2.5-7B-shaped layer with 128k cached tokens, two score variants at once, 448 window rows per KV head.
        dict(name="score_qwen_128k", kind="score", dtype="bf16", B=1, Hq=28, Hkv=4, W=64, N=131072, ragged=False, variants="K,VK"),
        # Batched serving: eight prompts of different lengths in one call.  The largest cache.
        dict(name="score_ragged_b8", kind="score", dtype="bf16", B=8, Hq=32, Hkv=8, W=32, N=65536, ragged=True, variants="VK"),
        # Scores from the attention kernel's own outputs (O and log-sum-exp of the window rows): no recompute.
        dict(name="given_llama_32k", kind="given", dtype="bf16", B=1, Hq=32, Hkv=8, W=32, N=32768, variants="VK"),
        # Every query position of a 4k prompt as a window row (the accumulation that H2O uses).
        dict(name="history_4k", kind="history", dtype="bf16", B=1, Hq=32, Hkv=8, W=4096, N=4096, variants="VK"),
        # Pool, select and compact one 32k layer: what follows score_llama_32k.
        dict(name="evict_llama_32k", kind="evict", dtype="bf16", B=1, Hkv=8, N=32768, ragged=False, budget=2048, n_sink=0,
             n_recent=32, pool="max", pool_kernel=7),
        # The same layer with head-adaptive budgets (ranked across heads, safeguard 0.2).
        dict(name="adaptive_llama_32k", kind="adaptive", dtype="bf16", B=1, Hkv=8, N=32768, budget=2048, n_sink=0,
             n_recent=32, pool="max", pool_kernel=7),
        # Serving step: 32 sequences with 4096 kept tokens each, append, rescore, evict one token per head.
        dict(name="decode_b32", kind="decode", B=32, Hq=32, Hkv=8, budget=4096, n_sink=4, n_recent=256, acc_window=0),
        # Interactive decoding: a few sequences, Qwen shapes, scores accumulated over the last 16 steps.
        dict(name="decode_b2_window", kind="decode", B=2, Hq=28, Hkv=4, budget=2048, n_sink=4, n_recent=128, acc_window=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# (query heads, KV heads): no groups, the two model shapes of the benchmark, their tensor-parallel shares, eight queries per KV head
_HEADS = ((32, 32), (32, 8), (28, 4), (8, 2), (7, 1), (64, 8), (16, 8))


def draw(rng):
    """One more case of the ranges above, sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(("evict_prefill", "score", "score", "score", "given", "history", "evict", "evict", "adaptive", "decode", "decode"))
    hq, hkv = rng.choice(_HEADS)
    window = rng.choice((8, 16, 32, 64, rng.randint(4, 64)))
    if kind == "evict_prefill":
        hq, hkv = rng.choice(((1, 1), (4, 2), (8, 2), (32, 8)))
        n = _log_int(rng, 512, 4096)
        return dict(kind=kind, dtype="f32", B=1, Hq=hq, Hkv=hkv, W=min(window, 32), N=n, budget=min(n, min(window, 32) + n // 4),
                    pool=rng.choice(("none", "max")), pool_kernel=7)
    if kind in ("score", "given"):
        batch = rng.choice((1, 1, 1, 2, 4, 8))
        n = _log_int(rng, 512, min(131072, (1 << 22) // (batch * hkv)))       # at most 4 M cached rows: the ragged batch's size
        c = dict(kind=kind, dtype="bf16", B=batch, Hq=hq, Hkv=hkv, W=window, N=n, variants=rng.choice(("VK", "VK", "K,VK", "V,K,VK")))
        return dict(c, ragged=batch > 1 and rng.random() < 0.5) if kind == "score" else c
    if kind == "history":
        hq, hkv = rng.choice(((32, 8), (28, 4), (8, 2), (7, 1)))
        n = _log_int(rng, 256, 4096)
        return dict(kind=kind, dtype="bf16", B=1, Hq=hq, Hkv=hkv, W=n, N=n, variants="VK")
    if kind in ("evict", "adaptive"):
        batch = rng.choice((1, 1, 2, 8))
        n = _log_int(rng, 1024, min(131072, (1 << 22) // (batch * hkv)))
        n_recent = rng.choice((16, 32, 64))
        budget = n_recent + max(1, int(n * rng.uniform(0.03, 0.25)))
        c = dict(kind=kind, dtype="bf16", B=batch, Hkv=hkv, N=n, budget=budget, n_sink=rng.choice((0, 4)), n_recent=n_recent,
                 pool=rng.choice(("none", "avg", "max", "max")), pool_kernel=rng.choice((5, 7)))
        return dict(c, ragged=batch > 1 and rng.random() < 0.5) if kind == "evict" else c
    budget = _log_int(rng, 300, 8192)
    batch = max(1, min(_log_int(rng, 1, 64), (1 << 20) // (budget * hkv)))
    return dict(kind="decode", B=batch, Hq=hq, Hkv=hkv, budget=budget, n_sink=4, n_recent=rng.choice((32, 64, 128)),
                acc_window=rng.choice((0, 0, 16)))


def _variants(case):
    return tuple(case["variants"].split(","))


def _generator(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 64 + tag)
    return g


def _lengths(case, seed):
    """Lengths of a ragged batch, uniform between an eighth of the longest and the longest; the longest is there."""
    if not case.get("ragged"):
        return [case["N"]] * case["B"]
    g = torch.Generator().manual_seed(seed * 64 + 9)
    lens = torch.randint(max(case["N"] // 8, 64), case["N"] + 1, (case["B"],), generator=g).tolist()
    lens[seed % case["B"]] = case["N"]
    return lens


def _cache(case, seed, lens, q=None):
    """K, V [B,Hkv,N,d]: unit normal, one token in a hundred a heavy hitter (its key shifted by 3 along the mean window
    query of its KV head), value norms lognormal(0, 0.5), zero beyond each sequence.  One batch item at a time in fp32."""
    dt = torch.float32 if case.get("dtype") == "f32" else torch.bfloat16
    B, H, N = case["B"], case["Hkv"], case["N"]
    k = torch.empty((B, H, N, D), dtype=dt, device="cuda")
    v = torch.empty_like(k)
    gk, gv = _generator(seed, 2), _generator(seed, 3)
    for b in range(B):
        kb = torch.randn((H, N, D), generator=gk, device="cuda")
        if q is not None:
            mean = q[b].float().reshape(H, -1, D).mean(1)
            mean = mean / mean.norm(dim=-1, keepdim=True).clamp_min(1e-20)
            heavy = (torch.rand((H, N, 1), generator=gk, device="cuda") < 0.01).float()
            kb += 3.0 * heavy * mean[:, None, :]
        vb = torch.randn((H, N, D), generator=gv, device="cuda")
        vb *= torch.exp(0.5 * torch.randn((H, N, 1), generator=gv, device="cuda"))
        kb[:, lens[b]:] = 0
        vb[:, lens[b]:] = 0
        k[b] = kb
        v[b] = vb
    return k, v


def _window_queries(case, seed):
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    return torch.randn((case["B"], case["Hq"], case["W"], D), generator=_generator(seed, 1), device="cuda").to(dt)


def _window_attention(q, k, v):
    """What a model's attention kernel returns for the window rows: O in bf16 and the natural-log log-sum-exp."""
    B, Hq, W, _ = q.shape
    H, N = k.shape[1], k.shape[2]
    o = torch.empty_like(q)
    lse = torch.empty((B, Hq, W), dtype=torch.float32, device="cuda")
    hidden = torch.arange(N, device="cuda")[None, :] > (N - W + torch.arange(W, device="cuda"))[:, None]
    G = Hq // H
    for b in range(B):
        for h in range(H):
            z = (q[b, h * G:(h + 1) * G].float() @ k[b, h].float().T) / math.sqrt(D)
            z.masked_fill_(hidden, float("-inf"))
            lse[b, h * G:(h + 1) * G] = torch.logsumexp(z, dim=-1)
            o[b, h * G:(h + 1) * G] = (torch.softmax(z, dim=-1) @ v[b, h].float()).to(q.dtype)
    return o, lse


def prepare(case, seed):
    """What the caller holds before the call: queries, caches and lengths on the GPU; for decoding also the
    accumulated scores, the slots' bookkeeping, the next tokens and the workspace."""
    kind = case["kind"]
    if kind == "decode":
        return _prepare_decode(case, seed)
    lens = _lengths(case, seed)
    lens_dev = torch.tensor(lens, dtype=torch.int32, device="cuda") if case.get("ragged") else None
    if kind in ("evict", "adaptive"):
        k, v = _cache(case, seed, lens)
        shape = (case["B"], case["Hkv"], case["N"])
        scores = torch.exp(1.5 * torch.randn(shape, generator=_generator(seed, 4), device="cuda")) * 1e-6   # heavy tail, as scores have
        st = dict(case=case, k=k, v=v, scores=scores, lens=lens_dev, budget=case["budget"], budgets=None, stride=case["budget"])
        if kind == "adaptive":
            st["stride"] = min(4 * case["budget"], case["N"])          # the most that one head may keep
        if lens_dev is not None:                                       # every sequence keeps the same share of its length
            share = [max(case["n_sink"] + case["n_recent"] + 1, case["budget"] * n // case["N"]) for n in lens]
            share = [min(s, n) for s, n in zip(share, lens)]
            st.update(budget=0, budgets=torch.tensor(share, dtype=torch.int32, device="cuda"), stride=max(share))
        return st
    q = _window_queries(case, seed)
    k, v = _cache(case, seed, lens, q)
    st = dict(case=case, q=q, k=k, v=v, lens=lens_dev)
    if kind == "given":
        st["o"], st["lse"] = _window_attention(q, k, v)
    return st


_STEPS = 16                                  # distinct tokens a decode state cycles through


def _prepare_decode(case, seed):
    B, H, n0, w = case["B"], case["Hkv"], case["budget"], case["acc_window"]
    cap = n0 + 1
    g = _generator(seed, 5)
    k, v = _cache(dict(case, N=cap), seed, [n0] * B)
    tok = lambda heads: torch.randn((_STEPS, B, heads, 1, D), generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
    pos = torch.full((B, H, cap), -1, dtype=torch.int32, device="cuda")
    pos[:, :, :n0] = torch.arange(n0, dtype=torch.int32, device="cuda")
    acc = torch.zeros((B, H, cap), device="cuda")
    acc[:, :, :n0] = 2e-5 * torch.exp(torch.randn((B, H, n0), generator=g, device="cuda"))     # seeded by the prefill scores
    state = torch.zeros((B, H, 4), dtype=torch.int32, device="cuda")
    state[..., :3] = n0
    hist = torch.zeros((B, H, w, cap), device="cuda") if w else None
    st = dict(case=case, k=k, v=v, q_t=tok(case["Hq"]), k_t=tok(H), v_t=tok(H), pos=pos, acc=acc, state=state, hist=hist, t=0)
    p = api.decode_params(st["q_t"][0], k, budget=n0, n_sink=case["n_sink"], n_recent=case["n_recent"], acc_window=w, s_hist=hist)
    st["ws"] = torch.empty(api.obc_decode_workspace(p), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    """One pass as a user's program makes it."""
    c = st["case"]
    kind = c["kind"]
    if kind in ("score", "history"):
        return api.obc_score(st["q"], st["k"], st["v"], seq_lens=st["lens"], variants=_variants(c))
    if kind == "given":
        return api.obc_score_given(st["q"], st["k"], st["v"], st["o"], st["lse"], variants=_variants(c))
    if kind == "evict_prefill":
        return api.evict_prefill(st["q"], st["k"], st["v"], budget=c["budget"], pool=c["pool"], pool_kernel=c["pool_kernel"])
    if kind == "evict":
        idx = api.obc_select(st["scores"], budget=st["budget"], budgets=st["budgets"], idx_stride=st["stride"], seq_lens=st["lens"],
                             n_sink=c["n_sink"], n_recent=c["n_recent"], pool=c["pool"], pool_kernel=c["pool_kernel"])
        k_out, v_out = api.obc_compact(st["k"], st["v"], idx)
        return idx, k_out, v_out
    if kind == "adaptive":
        idx, counts = api.obc_select_adaptive(st["scores"], budget=c["budget"], safeguard=0.2, idx_stride=st["stride"],
                                              n_sink=c["n_sink"], n_recent=c["n_recent"], pool=c["pool"],
                                              pool_kernel=c["pool_kernel"])
        k_out, v_out = api.obc_compact(st["k"], st["v"], idx)
        return idx, counts, k_out, v_out
    t = st["t"]
    st["t"] = t + 1
    i = t % _STEPS
    api.obc_decode_step(st["q_t"][i], st["k_t"][i], st["v_t"][i], st["k"], st["v"], st["acc"], st["pos"], st["state"],
                        c["budget"] + t, budget=c["budget"], n_sink=c["n_sink"], n_recent=c["n_recent"], workspace=st["ws"],
                        acc_window=c["acc_window"], s_hist=st["hist"])
    out = (st["k"], st["v"], st["acc"], st["pos"], st["state"])
    return out if st["hist"] is None else out + (st["hist"],)


def work(case):
    """K, V, the queries and the scores once; the gathered rows read and written once.  Three contractions over the
    visible (window row, token) pairs (logits, outputs, value-output products), two where the outputs are given."""
    kind = case["kind"]
    es = 4 if case.get("dtype") == "f32" else 2
    if kind == "decode":
        rows, G, w = case["B"] * case["Hkv"] * (case["budget"] + 1), case["Hq"] // case["Hkv"], case["acc_window"]
        # K and V rows, the accumulator read (or the ring's rows of the window) and written, the positions
        return {"bytes": rows * (2 * D * 2 + 4 + (4 * w + 4 if w else 4) + 4), "flops": 3 * 2 * D * G * rows}
    tokens = case["B"] * case["N"] * (9 / 16 if case.get("ragged") else 1.0)       # mean length of a ragged batch
    rows = tokens * case["Hkv"]
    kept = case.get("budget", 0) * case["B"] * case["Hkv"] * (9 / 16 if case.get("ragged") else 1.0)
    if kind in ("evict", "adaptive"):
        return {"bytes": rows * 4 + kept * 4 + kept * 4 * D * es, "flops": 0}
    planes = len(_variants(case)) if "variants" in case else 1
    W, N = case["W"], case["N"]
    pairs = rows * (case["Hq"] // case["Hkv"]) * W * (1 - (W - 1) / (2 * N))
    q = case["B"] * case["Hq"] * W * D * es
    total = rows * (2 * D * es + 4 * planes) + q * (2 if kind == "given" else 1)
    if kind == "evict_prefill":
        total += rows * 4 + kept * 4 + kept * 4 * D * es
    return {"bytes": total, "flops": (2 if kind == "given" else 3) * 2 * D * pairs}


def tolerance(case):
    """Selection and compaction are exact.  Scores: about four times what separates them from a double-precision evaluation of
    the same inputs.  Where everything is summed in 32 bits (fp32 caches, fewer than 64 window rows per KV head, outputs
    given by the caller, decoding) that was up to 1.6e-6 (norm) and 5e-6 (largest); with bf16 attention weights and outputs
    (64 rows and more) 7e-5 and 2.2e-4, and 1.2e-4 and 1.1e-3 where early rows of a whole-sequence window see few tokens."""
    kind = case["kind"]
    if kind in ("evict", "adaptive"):
        return "exact"
    if kind == "evict_prefill":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    if kind == "decode":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}       # `differ`: the slot freed where two accumulators all but tie
    if kind == "history":
        return {"rel": 5e-4, "max": 5e-3}
    if kind == "given" or case["Hq"] // case["Hkv"] * case["W"] < 64:
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 3e-4, "max": 1e-3}
