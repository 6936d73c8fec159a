"""The measured work: what a program that uses the library has it do, through the public entry points.

Three kinds of call:

* ``pass``    one compression pass over prompts (``CompressionPass.run``: score, thresholds and signatures, selection,
              gather), for one layer at a time or for a stack of layers; plain, with the observation window and pooling,
              or with the row log-sum-exp that a prefill attention kernel returned;
* ``decode``  one generated token per sequence: its attention row is added to the running scores;
* ``evict``   the cache has outgrown its budget: thresholds, signatures, selection and gather from the running scores,
              by token or by page, the running scores following the cache.

Sizes are those of the package's workloads (``inputs.paper_workloads``), of the benchmark's options and of the paged
setting of the decode tests (672 tokens = 32 initial + 512 middle + 128 recent, pages of 32); ``draw`` spreads over the
ranges between them.
"""
import math

import numpy as np
import torch

from paper_2503_00022_b200 import binding as kv
from paper_2503_00022_b200 import inputs

DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
ITEM = {"bf16": 2, "fp16": 2, "fp32": 4}
PAGE_INITIAL, PAGE_RECENT = 1, 4            # pages of 32: 32 initial and 128 recent tokens


def _case(name, kind, layers, q_heads, kv_heads, dim, lens, dtype, budget, cache="", window=0, pool=0, lse=False,
          page=0):
    """budget: share of a sequence's tokens (or pages) that is kept; cache: type of the K/V cache when it is not the
    scoring K itself; lens: lengths of the packed sequences."""
    return {"name": name, "kind": kind, "layers": layers, "q_heads": q_heads, "kv_heads": kv_heads, "dim": dim,
            "lens": ",".join(str(int(x)) for x in lens), "dtype": dtype, "cache": cache, "budget": budget,
            "window": window, "pool": pool, "lse": lse, "page": page}


def listed():
    ragged = inputs.paper_workloads()["cfg5_ragged_batch16"].seqlens
    return [
        # a short prompt in float32, one layer: the smallest call, launches and latency
        _case("layer_512_fp32", "pass", 1, 8, 8, 64, [512], "fp32", 0.25),
        # one grouped-query layer of a short prompt of odd length, compressed as soon as its prefill is done
        _case("layer_1k_gqa", "pass", 1, 32, 8, 128, [1001], "bf16", 0.25),
        # one layer of an ordinary prompt
        _case("layer_4k", "pass", 1, 32, 32, 128, [4096], "bf16", 0.25),
        # the whole stack of an ordinary model over a long prompt, the cache in another type than the scoring operands
        _case("prompt_8k", "pass", 32, 32, 32, 128, [8192], "bf16", 0.25, cache="fp16"),
        # the longest prompts, grouped-query heads, a quarter of the layers at a time: the largest call
        _case("prompt_32k_gqa", "pass", 8, 32, 8, 128, [32768], "bf16", 0.20),
        # batched serving: 16 prompts of 1024 to 4096 tokens in one packed call
        _case("batch_ragged", "pass", 8, 32, 32, 128, ragged, "bf16", 0.25),
        # importance from an observation window of the last 64 queries, pooled over 7 neighbours, window kept
        _case("window_8k", "pass", 32, 32, 32, 128, [8192], "bf16", 0.25, cache="fp16", window=64, pool=7),
        # attention was computed by inference: its log-sum-exp is at hand; float16, heads of 96, two odd lengths
        _case("lse_fp16", "pass", 8, 32, 32, 96, [5003, 3117], "fp16", 0.25, lse=True),
        # a generated token over a long cache
        _case("decode_8k", "decode", 32, 32, 32, 128, [8192], "bf16", 0.25),
        # a generated token for each sequence of a batch whose caches are at the paged setting's budget
        _case("decode_batch", "decode", 32, 32, 8, 128, [672 + i for i in range(16)], "bf16", 0.25),
        # the same batch 64 tokens later: eviction of whole pages of 32 down to 21 pages
        _case("evict_pages", "evict", 32, 32, 8, 128, [736] * 16, "bf16", 21 / 23, page=32),
        # eviction by token of a long cache
        _case("evict_32k", "evict", 32, 32, 8, 128, [32768], "bf16", 0.20),
    ]


MOST_FLOPS = 3.6e13                         # no drawn case costs more than the largest listed one; narrower heads
                                            # count as 128 wide, since the exponentials are the same
MOST_BYTES = 1.2e10


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["pass", "pass", "pass", "decode", "evict"])
        layers = _log_int(rng, 1, 32)
        q_heads, kv_heads = rng.choice([(8, 8), (32, 32), (32, 8), (32, 4), (40, 40)])
        dim = rng.choice([64, 96, 128, 128, 128])
        dtype = rng.choice(["bf16", "bf16", "bf16", "fp16"])
        window, pool, lse, page, cache = 0, 0, False, 0, ""
        budget = round(rng.uniform(0.1, 0.5), 3)
        n_seqs = rng.choice([1, 1, _log_int(rng, 2, 16)])
        longest = _log_int(rng, 200, 32768)
        if kind == "pass":
            mode = rng.choice(["plain", "plain", "plain", "window", "lse", "fp32"])
            if mode == "window":
                window, pool = rng.choice([16, 32, 64, 128]), rng.choice([0, 5, 7])
            elif mode == "lse":
                lse = True
            elif mode == "fp32":
                layers, q_heads, kv_heads, dtype, longest = min(layers, 4), 8, 8, "fp32", _log_int(rng, 64, 1024)
            if mode == "plain" and dtype == "bf16" and rng.random() < 0.3:
                cache = "fp16"
        elif kind == "evict" and rng.random() < 0.5:
            page = rng.choice([8, 32])
            budget = round(rng.uniform(0.25, 0.95), 3)
        lens = [longest] + [max(1, int(longest * rng.uniform(0.25, 1.0))) for _ in range(n_seqs - 1)]
        c = _case("", kind, layers, q_heads, kv_heads, dim, lens, dtype, budget, cache, window, pool, lse, page)
        del c["name"]
        w = work(c)
        row = sum(lens) * layers * dim * ITEM[dtype]
        held = row * (q_heads + 4 * kv_heads)                      # a state has to fit the card three times over
        if 2e5 <= w["bytes"] and w["bytes"] + held <= MOST_BYTES and w["flops"] * 128 / dim <= MOST_FLOPS:
            return c


def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _budgets(case):
    """(important, representative) places of every sequence, in tokens or pages: half and half."""
    unit = max(case["page"], 1)
    total = [max(2, int(case["budget"] * ((L + unit - 1) // unit) + 1e-9)) for L in _lens(case)]
    rep = [b // 2 for b in total]
    return np.asarray([[b - r for b, r in zip(total, rep)]], dtype=np.int32), np.asarray([rep], dtype=np.int32)


def _kept_rows(case):
    """Token rows of the reduced cache, per layer."""
    unit = max(case["page"], 1)
    imp, rep = _budgets(case)
    return sum(min(int(b), (L + unit - 1) // unit) for b, L in zip((imp + rep)[0], _lens(case))) * unit


def _heavy(g, L, dev):
    """Gain of every token's key: 4 for the first four tokens, 2 for a random twentieth of the others."""
    gain = torch.where(torch.rand(L, generator=g, device=dev) < 0.05, 2.0, 1.0)
    gain[:inputs.SINK_TOKENS] = inputs.SINK_GAIN
    return gain


def _keys_and_values(case, g, dev, what):
    """Normal tensors [layers, tokens, heads, dim], one for each of (heads, is_key, type) in `what`; keys carry the
    attention sinks and the heavy hitters.  A type "" stands for a copy of the previous tensor's values."""
    T, dim = sum(_lens(case)), case["dim"]
    out = [torch.empty((case["layers"], T, h, dim), dtype=DTYPES[t], device=dev) for h, _, t in what]
    for layer in range(case["layers"]):
        gain = torch.cat([_heavy(g, L, dev) for L in _lens(case)])[:, None, None]
        for x, (h, is_key, _) in zip(out, what):
            v = torch.randn((T, h, dim), generator=g, device=dev)
            x[layer].copy_(v * gain if is_key else v)
    return out


def _column_sums(case, g, dev):
    """Running scores shaped like the column sums of causal attention: older tokens have been seen by more queries, sinks
    and heavy hitters stand out, every head scatters by itself."""
    lens = _lens(case)
    s = torch.empty((case["layers"], case["q_heads"], sum(lens)), dtype=torch.float32, device=dev)
    for layer in range(case["layers"]):
        a = 0
        for L in lens:
            t = torch.arange(L, device=dev, dtype=torch.float32)
            mean = torch.log((L + 0.5) / (t + 0.5)) * _heavy(g, L, dev) ** 2
            x = torch.randn((case["q_heads"], L), generator=g, device=dev)
            s[layer, :, a:a + L] = mean * torch.exp(0.3 * x)
            a += L
    return s


def _prefill_lse(case, q, k):
    """The row log-sum-exp as the prefill attention returned it."""
    lse = torch.empty((case["layers"], case["q_heads"], q.shape[1]), dtype=torch.float32, device=q.device)
    rep = case["q_heads"] // case["kv_heads"]
    for layer in range(case["layers"]):
        a = 0
        for L in _lens(case):
            qs = q[layer, a:a + L].transpose(0, 1)[None].contiguous()
            ks = k[layer, a:a + L].transpose(0, 1)[None].repeat_interleave(rep, dim=1)
            r = torch.ops.aten._scaled_dot_product_flash_attention(qs, ks, ks, 0.0, True, False,
                                                                   scale=1.0 / math.sqrt(case["dim"]))
            lse[layer, :, a:a + L] = r[1][0, :, :L]
            a += L
    return lse


def prepare(case, seed):
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    hq, hk, dt = case["q_heads"], case["kv_heads"], case["dtype"]
    prob = kv.Problem(case["layers"], hq, hk, case["dim"], _lens(case), device=dev, query_window=case["window"])
    st = {"case": case, "prob": prob}
    if case["kind"] == "decode":
        st["k"], = _keys_and_values(case, g, dev, [(hk, True, dt)])
        st["q"] = torch.randn((case["layers"], prob.n_seqs, hq, case["dim"]), generator=g, device=dev).to(DTYPES[dt])
        # the running scores start at zero, so that what comes back is what the steps added
        st["scores"] = torch.zeros((case["layers"], hq, prob.total_tokens), dtype=torch.float32, device=dev)
        st["status"] = torch.zeros(4, dtype=torch.int32, device=dev)
        return st
    imp, rep = _budgets(case)
    cache = case["cache"] or dt
    if case["kind"] == "evict":
        st["kc"], st["vc"] = _keys_and_values(case, g, dev, [(hk, True, cache), (hk, False, cache)])
        st["scores"] = _column_sums(case, g, dev)
        paged = {"page_size": case["page"], "keep_initial": PAGE_INITIAL, "keep_recent": PAGE_RECENT} if case["page"] else {}
        st["cp"] = kv.CompressionPass(prob, imp, rep, cache_dtype=DTYPES[cache], **paged)
        st["new_scores"] = torch.empty((case["layers"], hq, _kept_rows(case)), dtype=torch.float32, device=dev)
        return st
    what = [(hq, False, dt), (hk, True, dt), (hk, False, cache)] + ([(hk, True, cache)] if case["cache"] else [])
    st["q"], st["k"], st["vc"], *more = _keys_and_values(case, g, dev, what)
    st["kc"] = more[0] if more else st["k"]
    st["lse"] = _prefill_lse(case, st["q"], st["k"]) if case["lse"] else None
    st["cp"] = kv.CompressionPass(prob, imp, rep, cache_dtype=DTYPES[cache], pool_kernel=case["pool"],
                                  keep_recent=case["window"])
    return st


def run(st):
    kind = st["case"]["kind"]
    if kind == "decode":
        kv.kvcrush_score_decode(st["prob"], st["q"], st["k"], st["scores"], status=st["status"])
        return {"scores": st["scores"], "status": st["status"]}
    cp = st["cp"]
    if kind == "evict":
        cp.signature(st["scores"])
        cp.select(st["scores"])
        cp.compact(st["kc"], st["vc"])
        kv.kvcrush_compact_scores(st["prob"], st["scores"], cp.page_size, cp.cu_kept, cp.idx, cp.total_kept,
                                  st["new_scores"], status=cp.status)
        return {"theta": cp.theta, "sigs": cp.sigs, "importance": cp.importance, "idx": cp.idx, "kind": cp.kind,
                "n_kept": cp.n_kept, "k": cp.k_out, "v": cp.v_out, "scores": st["new_scores"], "status": cp.status}
    cp.run(st["q"], st["k"], st["kc"], st["vc"], lse_in=st["lse"])
    # The kept list and the rows gathered by it are a step function of the scores: a last-bit difference in one score
    # can move one signature bit, and with it the membership of every later bucket.  They are compared bit for bit by
    # the evict cases, which start from given scores; here everything up to the signatures comes back.
    out = {"scores": cp.scores, "theta": cp.theta, "importance": cp.importance, "sigs": cp.sigs, "n_kept": cp.n_kept,
           "status": cp.status}
    if cp.pooled is not None:
        out["pooled"] = cp.pooled
    if st["lse"] is None and not st["case"]["window"]:
        out["lse"] = cp.lse                 # with a window only the voting rows are written
    return out


def work(case):
    lens, layers, hq, hk, dim = _lens(case), case["layers"], case["q_heads"], case["kv_heads"], case["dim"]
    T, words, eb = sum(lens), (case["q_heads"] + 31) // 32, ITEM[case["dtype"]]
    kept = _kept_rows(case)
    per_head = layers * T * 4                                     # one float per token
    if case["kind"] == "decode":
        return {"bytes": layers * hk * T * dim * eb + layers * len(lens) * hq * dim * eb + 2 * hq * per_head,
                "flops": 2.0 * layers * hq * T * dim}
    # signatures, importance, kept list and kinds; both tensors of the kept rows read and written
    chosen = per_head * words + layers * T * 8 + layers * kept * 5
    gathered = 2 * 2 * layers * kept * hk * dim * (ITEM[case["cache"]] if case["cache"] else eb)
    if case["kind"] == "evict":
        return {"bytes": hq * per_head + chosen + gathered + 2 * layers * hq * kept * 4, "flops": layers * hq * T * 2.0}

    def entries(L):
        first = max(0, L - case["window"]) if case["window"] else 0
        return L * (L + 1) // 2 - first * (first + 1) // 2
    voting = sum(min(L, case["window"]) if case["window"] else L for L in lens)
    if not case["cache"]:
        gathered -= layers * kept * hk * dim * eb                 # the scoring K, read anyway, is the cache
    read = layers * dim * eb * (voting * hq + T * hk)
    # scores, pooled scores and the row log-sum-exp (given or written)
    floats = hq * layers * 4 * (T + (T if case["pool"] else 0) + voting)
    # each logit once
    return {"bytes": read + floats + chosen + gathered, "flops": 2.0 * dim * hq * layers * sum(entries(L) for L in lens)}


def tolerance(case):
    # About four times what one layer of each case differs by from the same path in 64 bits (relative, largest):
    # float32 scores 5e-8, 3e-7 (an exponential of 2 ulp and another order of the sums: 1e-6); bf16 and fp16 scores
    # 3e-6, 3e-5, with few voting queries 1.3e-5, 7e-5; decode 5e-7, 2e-6.  No signature word differed; one score in
    # 1e5 of its threshold makes it a few in 10000.
    if case["kind"] == "evict":
        return "exact"
    if case["kind"] == "decode":
        return {"rel": 2e-6, "max": 2e-5}
    if case["dtype"] == "fp32":
        return {"rel": 4e-6, "max": 4e-5, "differ": 0.002}
    return {"rel": 5e-5, "max": 3e-4, "differ": 0.002}
