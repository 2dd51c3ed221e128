"""What a user of the library has it do, as cases that can be prepared, run and compared.

Five operations, each through the public binding, over the range of sizes that the repository's
configurations, tests and benchmark use (head layouts 32/8, 28/4 and 64/8, one sequence to a batch,
one layer to all layers of a model folded into the batch, 500 to 131072 slots):

  decode   attention of new tokens over merged caches           (kvs_decode_attn)
  stream   a chunk of fresh tokens joins the cache, which is merged back to its budget
                                                                (kvs_append_and_merge)
  merge    the merge pass after a prefill, then the decode of new tokens over its result
                                                                (kvs_merge_layer, kvs_merge_layer_per_head)
  stats    the statistics and the decision of one round         (kvs_window_stats, kvs_window_stats_exact)
  compact  merge and compaction with the caller's decision      (kvs_compact)

Keys drift along the tokens (AR(1)) and have a few outlier channels; values are independent from token
to token around a mean per channel, as the values of a trained model are; queries are N(0, 1).

What is compared.  A merge pass chooses the R smallest scores: two correct sums that differ in their
last bit may swap two pairs at the cutoff, which moves every slot between the two and changes every
later round.  At about 1e-7 of relative difference in a score that happens once in some ten million
candidate pairs, so small passes return the merged cache itself, and larger ones what is read from it
next: the attention output and the log-sum-exp of new tokens, which such a swap hardly changes.  The
statistics and the compaction, which have no such choice before their results, return everything.
"""
import math

import numpy as np
import torch

from paper_2603_00907_b200 import binding as kvs

HEAD_DIM = 128
SINK = 32                      # slots at the start that are never merged
WHOLE_PAIRS = 60_000           # candidate pairs of a pass up to which the cache itself is returned


# ---------------------------------------------------------------------------------------------- cases
def _decode(batch, n_lo, n_hi, n_new, q_heads=32, kv_heads=8, len_seed=7):
    return {"op": "decode", "batch": batch, "n_lo": n_lo, "n_hi": n_hi, "len_seed": len_seed, "n_new": n_new,
            "q_heads": q_heads, "kv_heads": kv_heads}


def _stream(batch, budget, chunk, window=64, q_heads=32, kv_heads=8, n_new=1):
    return {"op": "stream", "batch": batch, "budget": budget, "chunk": chunk, "window": window, "q_heads": q_heads,
            "kv_heads": kv_heads, "n_new": n_new}


def _merge(batch, n_lo, n_hi, window, budget=0, share=0.0, q_heads=32, kv_heads=8, n_new=1, ar=0.9, score_mode=0,
           per_head=False, len_seed=7):
    return {"op": "merge", "batch": batch, "n_lo": n_lo, "n_hi": n_hi, "len_seed": len_seed, "window": window,
            "budget": budget, "share": share, "q_heads": q_heads, "kv_heads": kv_heads, "n_new": n_new, "ar": ar,
            "score_mode": score_mode, "per_head": per_head}


def _stats(batch, n, window, budget, weight_mode=0, q_heads=32, kv_heads=8, first_round=0):
    return {"op": "stats", "batch": batch, "n": n, "window": window, "budget": budget, "weight_mode": weight_mode,
            "q_heads": q_heads, "kv_heads": kv_heads, "first_round": first_round}


def _compact(batch, n, share, window, kv_heads=8, first_round=0, token_major=False):
    return {"op": "compact", "batch": batch, "n": n, "share": share, "window": window, "q_heads": 4 * kv_heads,
            "kv_heads": kv_heads, "first_round": first_round, "token_major": token_major}


def listed():
    return [
        # one decoder layer's attention for the next token of one sequence over a merged cache of the
        # paper's budget: the call that a generation makes most often, and the smallest
        dict(_decode(1, 2048, 2048, 1), name="decode_1tok_b1"),
        # the same for a serving batch whose caches were merged to an eighth of 4 K to 64 K tokens
        dict(_decode(32, 512, 8192, 1), name="decode_1tok_b32"),
        # the paper's operating point: budget 2048, chunks of 512, one layer of one sequence
        dict(_stream(1, 2048, 512), name="stream_1layer"),
        # the same step with all 32 layers in one call, and the next token's attention
        dict(_stream(32, 2048, 512), name="stream_32layers"),
        # a short prompt: one layer, 4096 tokens to 1024
        dict(_merge(1, 4096, 4096, 32, budget=1024), name="merge_8b_4k"),
        # one layer of a 32 K prompt with a budget of its own for every KV head
        dict(_merge(1, 32768, 32768, 64, share=0.125, per_head=True), name="merge_per_head_32k"),
        # Qwen2.5-7B layout (groups of 7: 224 window rows), four sequences of 16 K, one layer
        dict(_merge(4, 16384, 16384, 32, budget=1024, q_heads=28, kv_heads=4), name="merge_qwen_b4_16k"),
        # a ragged serving batch of 4 K to 64 K tokens, budgets of 12.5 %, 32 new tokens each
        dict(_merge(8, 4096, 65536, 32, share=0.125, n_new=32, len_seed=3000), name="merge_ragged_b8"),
        # Llama-3-70B layout, one layer of 128 K tokens, 1024 window rows per KV head
        dict(_merge(1, 131072, 131072, 128, budget=4096, q_heads=64, n_new=32, ar=0.92), name="merge_70b_128k"),
        # the benchmark's workload: all 32 layers of a 32 K prompt in one call
        dict(_merge(32, 32768, 32768, 64, budget=2048, n_new=16), name="merge_8b_32layers_32k"),
        # the diagnostic export of one round, with the weights of the gradient-free form
        dict(_stats(1, 32768, 64, 2048), name="stats_8b_32k"),
        # a decision made elsewhere applied to one layer of 128 K tokens
        dict(_compact(1, 131072, 0.5, 128), name="compact_128k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["decode", "decode", "stream", "stream", "merge", "merge", "merge", "stats", "compact"])
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (28, 4), (64, 8)])
    group = q_heads // kv_heads
    len_seed = rng.randrange(1 << 20)
    if op == "decode":
        batch = _log_int(rng, 1, 64)
        hi = _log_int(rng, 512, min(65536, (1 << 18) // batch))
        lo = hi if rng.random() < 0.3 else max(256, hi // rng.choice([2, 4, 16]))
        n_new = 1 if rng.random() < 0.6 else _log_int(rng, 2, 32)
        return _decode(batch, lo, hi, n_new, q_heads, kv_heads, len_seed)
    window = rng.choice([16, 32, 48, 64] + ([128] if group > 4 else []))
    if op == "stream":
        return _stream(_log_int(rng, 1, 32), _log_int(rng, 512, 4096), _log_int(rng, 64, 1024), window, q_heads, kv_heads,
                       rng.choice([1, 1, 4]))
    if op == "merge":
        hi = _log_int(rng, 2048, 131072)
        batch = _log_int(rng, 1, max(1, min(16, (1 << 18) // hi)))
        lo = hi if rng.random() < 0.5 else max(1500, hi // rng.choice([2, 4]))
        share = round(math.exp(rng.uniform(math.log(1 / 32), math.log(1 / 2))), 4)
        return _merge(batch, lo, hi, window, share=share, q_heads=q_heads, kv_heads=kv_heads,
                      n_new=rng.choice([1, 4, 32]), ar=round(rng.uniform(0.8, 0.95), 3), score_mode=rng.choice([0, 0, 1]),
                      per_head=rng.random() < 0.2, len_seed=len_seed)
    if op == "stats":
        n = _log_int(rng, 1024, 131072)
        return _stats(_log_int(rng, 1, max(1, min(8, (1 << 18) // n))), n, window, n // 3, rng.choice([0, 0, 1, 2]),
                      q_heads, kv_heads, rng.choice([0, 1]))
    n = _log_int(rng, 1024, 131072)
    return _compact(_log_int(rng, 1, max(1, min(16, (1 << 18) // n))), n, round(rng.uniform(0.02, 0.9), 3), window,
                    kv_heads, rng.choice([0, 1]), rng.random() < 0.3)


# ---------------------------------------------------------------------------------------------- sizes
def _lengths(case):
    rng = np.random.default_rng(case["len_seed"])
    return [int(v) for v in rng.integers(case["n_lo"], case["n_hi"] + 1, size=case["batch"])]


def _floor_budget(case):
    return SINK + case["window"] + 8


def _merge_lengths(case):
    """(length, budget) of every sequence, or of every (sequence, KV head)."""
    lens = _lengths(case)
    if case["per_head"]:
        rng = np.random.default_rng(case["len_seed"] + 1)
        lens = [n for n in lens for _ in range(case["kv_heads"])]
        budgets = [int(n * case["share"] * f) for n, f in zip(lens, np.exp(rng.uniform(-0.7, 0.7, len(lens))))]
    else:
        budgets = [case["budget"] or int(n * case["share"]) for n in lens]
    return lens, [min(n, max(b, _floor_budget(case))) for n, b in zip(lens, budgets)]


def _rounds(n, budget, window):
    """(slots, candidate pairs) of every round of one sequence."""
    r = 0
    while n > budget:
        pairs = max(0, (n - SINK - (r & 1) - window) // 2)
        yield n, pairs
        n -= min(n - budget, max(1, pairs // 2))
        r += 1


def _pass_of(case):
    """Over all (sequence, KV head) units of a merging case: slots before, slots after, slots summed over
    the rounds, candidate pairs summed over the rounds."""
    if case["op"] == "stream":
        n = case["budget"] + case["chunk"]
        lens, budgets = [n] * case["batch"], [case["budget"]] * case["batch"]
    else:
        lens, budgets = _merge_lengths(case)
    heads = 1 if case.get("per_head") else case["kv_heads"]
    plan = [list(_rounds(n, b, case["window"])) for n, b in zip(lens, budgets)]
    return (heads * sum(lens), heads * sum(budgets), heads * sum(n for p in plan for n, _ in p),
            heads * sum(k for p in plan for _, k in p))


def _whole(case):
    return _pass_of(case)[3] <= WHOLE_PAIRS


# ---------------------------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _keys(g, batch, heads, n, ar):
    """AR(1) along the tokens with unit variance, plus constant offsets on eight channels of every head."""
    out = torch.empty(batch, heads, n, HEAD_DIM, dtype=torch.bfloat16, device="cuda")
    for b in range(batch):
        x = _normal(g, heads, n, HEAD_DIM)
        x[:, 1:] *= math.sqrt(1 - ar * ar)
        step, weight = 1, ar
        while step < n and weight > 1e-5:          # x_t + a x_(t-1) + a^2 x_(t-2) + ... by doubling
            y = x.clone()
            y[:, step:].add_(x[:, :-step], alpha=weight)
            x, step, weight = y, 2 * step, weight * weight
        channel = torch.rand(heads, HEAD_DIM, generator=g, device="cuda").argsort(-1)[:, :8]
        offset = torch.zeros(heads, HEAD_DIM, device="cuda").scatter_(1, channel, 2.0 * _normal(g, heads, 8))
        out[b] = x + offset[:, None, :]
    return out


def _values(g, batch, heads, n, count=None):
    """Value sums of `count` tokens (1 if None) around a mean per channel."""
    out = torch.empty(batch, heads, n, HEAD_DIM, dtype=torch.bfloat16, device="cuda")
    for b in range(batch):
        x, mean = _normal(g, heads, n, HEAD_DIM), _normal(g, heads, 1, HEAD_DIM)
        if count is not None:
            c = count[b].unsqueeze(-1).float()
            x, mean = x * c.sqrt(), mean * c
        out[b] = x + mean
    return out


def _merged_cache(g, batch, heads, n):
    """A cache as a merge pass leaves it: most slots stand for several tokens, first and last for one."""
    count = torch.empty(batch, heads, n, device="cuda").exponential_(0.08, generator=g).to(torch.int32) + 1
    count[:, :, :SINK] = 1
    count[:, :, -SINK:] = 1
    return _keys(g, batch, heads, n, 0.9), _values(g, batch, heads, n, count), count


def _queries(g, case, rows):
    return _normal(g, case["batch"], case["q_heads"], rows, HEAD_DIM).to(torch.bfloat16)


def _workspace(params, n_max, n_new=0, per_head=False):
    size = kvs.kvs_workspace_size_per_head if per_head else kvs.kvs_workspace_size
    return torch.empty(size(params, n_max, n_new), dtype=torch.uint8, device="cuda")


class State:
    """A plain holder of what the caller's program keeps."""

    def __init__(self, **kw):
        self.__dict__.update(kw)


def _decode_buffers(case):
    shape = (case["batch"], case["q_heads"], case["n_new"])
    return dict(out=torch.empty(*shape, HEAD_DIM, dtype=torch.bfloat16, device="cuda"),
                lse=torch.empty(*shape, dtype=torch.float32, device="cuda"))


def prepare(case, seed):
    g = _generator(seed)
    op, batch, heads, hq = case["op"], case["batch"], case["kv_heads"], case["q_heads"]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if op == "decode":
        lens = _lengths(case)
        K, V, count = _merged_cache(g, batch, heads, max(lens))
        params = kvs.make_params(K, V, hq, 32)
        return State(case=case, K=K, V=V, count=count, q_new=_queries(g, case, case["n_new"]), lens=lens, params=params,
                     ws=_workspace(params, max(lens), case["n_new"]), status=status, **_decode_buffers(case))
    if op == "stream":
        n, chunk = case["budget"] + case["chunk"], case["chunk"]
        K, V, count = _merged_cache(g, batch, heads, n)
        params = kvs.make_params(K, V, hq, case["window"])
        return State(case=case, K=K, V=V, count=count, chunk_k=_keys(g, batch, heads, chunk, 0.9),
                     chunk_v=_values(g, batch, heads, chunk), q_win=_queries(g, case, case["window"]),
                     q_new=_queries(g, case, case["n_new"]), cur=[case["budget"]] * batch, params=params,
                     ws=_workspace(params, n, case["n_new"]), status=status, **_decode_buffers(case))
    if op == "merge":
        lens, budgets = _merge_lengths(case)
        n_max = max(lens)
        K0, V0 = _keys(g, batch, heads, n_max, case["ar"]), _values(g, batch, heads, n_max)
        params = kvs.make_params(K0, V0, hq, case["window"], score_mode=case["score_mode"])
        return State(case=case, K0=K0, V0=V0, K=torch.empty_like(K0), V=torch.empty_like(V0),
                     count=torch.empty(batch, heads, n_max, dtype=torch.int32, device="cuda"),
                     q_win=_queries(g, case, case["window"]), q_new=_queries(g, case, case["n_new"]), lens=lens,
                     budgets=budgets, params=params, ws=_workspace(params, n_max, case["n_new"], case["per_head"]),
                     status=status, **_decode_buffers(case))
    if op == "stats":
        n = case["n"]
        K, V, count = _merged_cache(g, batch, heads, n)
        params = kvs.make_params(K, V, hq, case["window"], first_round=case["first_round"])
        e_win = _queries(g, case, case["window"]) if case["weight_mode"] else None
        slot = {k: torch.zeros(batch, heads, n, device="cuda") for k in ("A", "N1")}
        pair = {k: torch.zeros(batch, heads, n // 2, device="cuda") for k in ("N12", "cosv", "score", "w")}
        return State(case=case, K=K, V=V, count=count, q_win=_queries(g, case, case["window"]), e_win=e_win, slot=slot,
                     pair=pair, mask=torch.zeros(batch, heads, n // 2, dtype=torch.uint8, device="cuda"), params=params,
                     ws=_workspace(params, n), status=status)
    n, off = case["n"], SINK + case["first_round"]
    pairs = (n - off - case["window"]) // 2
    chosen = max(1, int(case["share"] * pairs))
    K0, V0, count0 = _merged_cache(g, batch, heads, n)
    K, V = torch.empty_like(K0), torch.empty_like(V0)
    if case["token_major"]:                        # [B, N, H, D] in memory, as attention kernels often keep it
        K, V = (torch.empty(batch, n, heads, HEAD_DIM, dtype=torch.bfloat16, device="cuda").transpose(1, 2) for _ in "KV")
    mask = torch.zeros(batch, heads, n // 2, dtype=torch.uint8, device="cuda")
    order = torch.rand(batch, heads, pairs, generator=g, device="cuda").argsort(-1)
    mask.scatter_(2, order[:, :, :chosen], 1)
    return State(case=case, K0=K0, V0=V0, count0=count0, K=K, V=V, count=torch.empty_like(count0), mask=mask,
                 w=torch.rand(batch, heads, n // 2, generator=g, device="cuda"), n=n, chosen=chosen,
                 new_index=torch.zeros(batch, heads, n, dtype=torch.int32, device="cuda"),
                 params=kvs.make_params(K, V, hq, case["window"], first_round=case["first_round"]),
                 ws=_workspace(kvs.make_params(K, V, hq, case["window"]), n), status=status)


# ---------------------------------------------------------------------------------------------- one pass
def _cache(s, new_len):
    return {"K": s.K[:, :, :new_len], "V": s.V[:, :, :new_len], "count": s.count[:, :, :new_len]}


def run(s):
    case, op = s.case, s.case["op"]
    if op == "decode":
        kvs.kvs_decode_attn(s.params, s.q_new, s.K, s.V, s.count, s.lens, s.out, s.ws, lse=s.lse, status_dev=s.status)
        return {"out": s.out, "lse": s.lse, "status": s.status}
    if op == "stream":
        # every pass is the next step of the stream: the cache holds what the pass before left
        new_len = kvs.kvs_append_and_merge(s.params, s.K, s.V, s.count, s.chunk_k, s.chunk_v, s.q_win, s.cur, s.cur, s.ws,
                                           status_dev=s.status)
        kvs.kvs_decode_attn(s.params, s.q_new, s.K, s.V, s.count, new_len, s.out, s.ws, lse=s.lse, status_dev=s.status)
        got = {"out": s.out, "lse": s.lse, "status": s.status}
        return dict(got, **_cache(s, case["budget"])) if _whole(case) else got
    if op == "merge":
        # the prefill writes the cache (here a copy of its result), the pass compresses it, decoding reads it
        s.K.copy_(s.K0)
        s.V.copy_(s.V0)
        s.count.fill_(1)
        merge = kvs.kvs_merge_layer_per_head if case["per_head"] else kvs.kvs_merge_layer
        decode = kvs.kvs_decode_attn_per_head if case["per_head"] else kvs.kvs_decode_attn
        new_len = merge(s.params, s.K, s.V, s.count, s.q_win, s.lens, s.budgets, s.ws, status_dev=s.status)
        decode(s.params, s.q_new, s.K, s.V, s.count, new_len, s.out, s.ws, lse=s.lse, status_dev=s.status)
        got = {"out": s.out, "lse": s.lse, "status": s.status, "new_len": np.asarray(new_len)}
        if _whole(case) and len(set(new_len)) == 1:
            got.update(_cache(s, new_len[0]))
        return got
    if op == "stats":
        args = (s.K, s.V, s.count, s.q_win)
        tail = ([case["n"]] * case["batch"], [case["budget"]] * case["batch"], s.ws)
        common = dict(A=s.slot["A"], cosv=s.pair["cosv"], score=s.pair["score"], mask=s.mask, status_dev=s.status)
        if case["weight_mode"] == 0:
            kvs.kvs_window_stats(s.params, *args, *tail, N1=s.slot["N1"], N12=s.pair["N12"], w=s.pair["w"], **common)
        else:
            # (the weight is left to its own arithmetic here: a ratio of signed sums has no bound near its guard)
            kvs.kvs_window_stats_exact(s.params, *args, s.e_win, case["weight_mode"], *tail, g_self=s.slot["N1"],
                                       g_pair=s.pair["N12"], **common)
        return {"slot": s.slot, "pair": s.pair, "mask": s.mask, "status": s.status}
    s.K.copy_(s.K0)
    s.V.copy_(s.V0)
    s.count.copy_(s.count0)
    new_len = kvs.kvs_compact(s.params, s.K, s.V, s.count, s.mask, s.w, [s.n] * case["batch"], [s.chosen] * case["batch"],
                              s.ws, new_index=s.new_index, status_dev=s.status)
    return dict(_cache(s, new_len[0]), new_index=s.new_index, status=s.status)


# ---------------------------------------------------------------------------------------------- what it needs
def work(case):
    """Caches read once and written once, and the contractions over every round: the logits, the attention
    output and the products of values and outputs, 2 * 128 operations each per (query, slot)."""
    op, slot, row = case["op"], 4 * HEAD_DIM + 4, 2 * HEAD_DIM
    group = case["q_heads"] // case["kv_heads"]
    if op == "decode":
        slots = case["kv_heads"] * sum(_lengths(case))
        tokens = case["batch"] * case["q_heads"] * case["n_new"]
        return {"bytes": slots * slot + tokens * (2 * row + 4), "flops": 4.0 * HEAD_DIM * slots * group * case["n_new"]}
    if op == "stats":
        slots = case["batch"] * case["kv_heads"] * case["n"]
        queries = case["batch"] * case["q_heads"] * case["window"]
        return {"bytes": slots * slot + queries * row * (2 if case["weight_mode"] else 1) + slots * 8 + slots * 8.5,
                "flops": 6.0 * HEAD_DIM * slots * group * case["window"]}
    if op == "compact":
        slots = case["batch"] * case["kv_heads"] * case["n"]
        pairs = (case["n"] - SINK - case["first_round"] - case["window"]) // 2
        left = case["batch"] * case["kv_heads"] * (case["n"] - max(1, int(case["share"] * pairs)))
        return {"bytes": (slots + left) * slot + slots * 4 + slots * 2.5, "flops": 0}
    before, after, walked, _ = _pass_of(case)
    tokens = case["batch"] * case["q_heads"] * case["n_new"]
    queries = case["batch"] * case["q_heads"] * case["window"]
    return {"bytes": (before + 2 * after) * slot + queries * row + tokens * (2 * row + 4),
            "flops": 6.0 * HEAD_DIM * walked * group * case["window"] + 4.0 * HEAD_DIM * after * group * case["n_new"]}


def tolerance(case):
    op = case["op"]
    if op == "compact":
        return "exact"                             # bf16 rounding of one fp32 expression; integers
    # four times what another order of the same sums showed (other key ranges, other groups of queries)
    if op == "stats":
        # (with values around a mean, the distance of a value from the output is a difference of larger terms)
        return {"rel": 1.4e-4, "max": 6e-4, "differ": 1e-4} if case["weight_mode"] == 0 else \
            {"rel": 1.3e-3, "max": 0.04, "differ": 1e-4}
    if op == "decode":
        return {"rel": 2.4e-3, "max": 0.03}
    if op == "stream":
        return {"rel": 5e-4, "max": 0.03, "differ": 1e-4}
    # two pairs may swap at the cutoff of a round here and there
    return {"rel": 9e-3, "max": 0.08, "differ": 1e-4}
