"""The performance cases of this library: what a prefill engine asks of it, through the public entry points.

A case is a dict of plain values.  ``path`` names the entry point and the rest the shape and the options:

    prefill        stem_prefill            one attention layer over a packed batch (lists and O come back)
    chunk          stem_prefill_cached     one chunk of a long sequence against its prefix, pooled-K cache updated
    dense          stem_sparse_prefill     the same kernel on every causal block (warm-up layers run dense)
    lists          stem_score_select       the scoring stage alone: an engine with attention kernels of its own
    metric         stem_score, stem_select the metric handed out, then lists from it (a caller that edits the metric)
    token_select   stem_token_select       lists of single tokens from an indexer's scores
    token_attend   stem_token_attention    attention over such lists

Sizes are those of ``workloads.CONFIGS``, of the benchmark's further legs and of the tests.  Q, K and V follow the
recipe of ``workloads.make_qkv`` (heavy keys, an attention sink, log-normal value norms), drawn on the GPU.
"""
from __future__ import annotations

import math

import torch

import paper_2603_06274_b200 as stem

D = 128


def _block_case(name, path, seqlens, hq, hkv, block=128, permille=50, mu="7/10", local=4, share=False, mode=0, chunk=0):
    """``seqlens``: "a,b,..."; ``chunk``: query tokens of the chunk at the end of each (single) sequence, 0 = all."""
    return dict(name=name, path=path, seqlens=seqlens, hq=hq, hkv=hkv, block=block, permille=permille, mu=mu, local=local,
                share=share, mode=mode, chunk=chunk)


def _token_case(name, path, n, hq, hkv, k_start, stem_tokens=0, local=1):
    return dict(name=name, path=path, n=n, hq=hq, hkv=hkv, k_start=k_start, stem_tokens=stem_tokens, local=local)


def listed():
    return [
        # short prompts batched together: two ragged requests on a small layer; launches and latency
        _block_case("prefill_short_ragged", "prefill", "1500,700", 4, 2, permille=300),
        # the smallest configuration: 4K tokens, two heads, blocks of 64
        _block_case("prefill_4k_2h_b64", "prefill", "4096", 2, 2, block=64, permille=250),
        # an ordinary long prompt: one 32K-token layer of 32 / 8 heads
        _block_case("prefill_32k", "prefill", "32768", 32, 8, permille=100),
        # the headline: one 128K-token layer of 32 / 8 heads at a 5 % budget
        _block_case("prefill_128k", "prefill", "131072", 32, 8, permille=50, local=2),
        # two long prompts packed together, 28 / 4 heads
        _block_case("prefill_varlen_64k_40k", "prefill", "65536,40960", 28, 4, permille=50),
        # the largest layer, 64 / 8 heads at 128K, with one list per kv head (block-level top-k shared by a group)
        _block_case("prefill_128k_64h_shared", "prefill", "131072", 64, 8, permille=50, share=True),
        # chunked prefill: the third 32K chunk of a long sequence whose last block is partial
        _block_case("chunk_32k_at_96k", "chunk", "98201", 32, 8, permille=50, local=2, chunk=32665),
        # a dense layer at 16K (layers that are kept dense, and the comparator)
        _block_case("dense_16k", "dense", "16384", 32, 8),
        # the scoring stage alone in the anti-diagonal mode, a ragged 32K prompt
        _block_case("lists_antidiag_32k", "lists", "32700", 32, 8, permille=100, mode=1),
        # metric out and lists from it, two ragged prompts
        _block_case("metric_select_32k", "metric", "20000,12345", 32, 8, permille=100),
        # token-level selector: top 2048 of 8K tokens for each of 8 list heads
        _token_case("token_select_8k", "token_select", 8192, 32, 8, 2048),
        # attention over those lists
        _token_case("token_attend_8k", "token_attend", 8192, 32, 8, 2048),
    ]


# Head layouts of the configurations and of the smoke run.
HEADS = ((2, 2), (4, 2), (28, 4), (32, 8), (64, 8))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: 256 to 131072 tokens in one to four ragged sequences, the listed head layouts,
    both block sizes, the budgets of the configurations and their sweeps; token-level rows of 256 to 12000 tokens."""
    path = rng.choice(("prefill",) * 5 + ("chunk", "chunk", "dense", "lists", "metric", "token_select", "token_attend"))
    if path.startswith("token"):
        n = _log_int(rng, 256, 12000)
        hkv = rng.choice([h for h in (1, 2, 4, 8) if n * n * h <= 8192 * 8192 * 8])
        g = rng.choice((1, 2, 4, 7, 8))
        k_start = rng.choice([k for k in (128, 256, 512, 1024, 2048) if k <= n])
        stem_tokens, local = rng.choice(((0, 1), (4, 8)))
        return {k: v for k, v in _token_case("", path, n, g * hkv, hkv, k_start, stem_tokens, local).items() if k != "name"}
    hq, hkv = rng.choice(HEADS)
    block = rng.choice((128, 128, 64))
    permille = rng.choice((100, 200, 250) if path == "lists" else (30, 50, 100, 200, 250))
    mu = rng.choice(("7/10", "7/10", "1/1", "1/2"))
    if path == "dense":
        cap = 16384 * math.sqrt(32 / hq)
    else:  # no more selected blocks than the largest layer has
        cap = 131072 * min(1.0, math.sqrt(50 / permille * 64 / hq))
    if path == "metric":
        cap = min(cap, 65536)
    # lists alone say nothing about the inputs where every kept block is a forced one: longer sequences there
    total = _log_int(rng, 40000 * block // permille if path == "lists" else 256, int(cap))
    batch = 1 if path == "chunk" else rng.choice((1, 2) if path == "lists" else (1, 1, 2, 3, 4))
    cuts = sorted(rng.sample(range(64, total - 63), batch - 1)) if batch > 1 else []
    lens = [b - a for a, b in zip([0] + cuts, cuts + [total])]
    chunk = 0
    if path == "chunk":
        # the last chunk of the prefix seen so far: it starts on a block and holds up to 32K tokens
        chunk = total - total * rng.randrange(0, 8) // 8 // block * block
        if chunk > 32768:
            chunk = 32768 + total % block
    share = path in ("prefill", "lists") and rng.random() < 0.25
    mode = 1 if path == "lists" and not share and rng.random() < 0.5 else 0
    case = _block_case("", path, ",".join(map(str, lens)), hq, hkv, block, permille, mu, rng.choice((2, 4)), share, mode, chunk)
    return {k: v for k, v in case.items() if k != "name"}


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------

def _normal(gen, shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _make_qkv(gen, seqlens, hq, hkv):
    """Q, K, V bf16 [T, H, 128] by the recipe of ``workloads.make_qkv``: normal rows, 2 % of the keys (and the first of
    every sequence) four times as long, a sink direction on the first four keys, log-normal value norms."""
    T = sum(seqlens)
    u = _normal(gen, (hkv, D))
    u = u / u.norm(dim=1, keepdim=True)
    q = torch.empty((T, hq, D), device="cuda", dtype=torch.bfloat16)
    k = torch.empty((T, hkv, D), device="cuda", dtype=torch.bfloat16)
    v = torch.empty((T, hkv, D), device="cuda", dtype=torch.bfloat16)
    uq = 8.0 * u.repeat_interleave(hq // hkv, dim=0)
    for a in range(0, T, 16384):
        b = min(T, a + 16384)
        q[a:b] = _normal(gen, (b - a, hq, D)).add_(uq)
        kc = _normal(gen, (b - a, hkv, D))
        heavy = torch.rand((b - a, hkv, 1), generator=gen, device="cuda") < 0.02
        k[a:b] = torch.where(heavy, kc * 4.0, kc)
        vc = _normal(gen, (b - a, hkv, D))
        gain = torch.exp(0.5 * _normal(gen, (b - a, hkv, 1)))
        v[a:b] = vc * (gain / vc.norm(dim=2, keepdim=True))
    start = 0
    for n in seqlens:
        m = min(4, n)
        first = _normal(gen, (m, hkv, D))
        first[0] *= 4.0
        k[start:start + m] = first + 8.0 * u
        start += n
    return q, k, v


def _indexer_scores(gen, n, heads):
    """fp32 [heads, n, n]: an indexer's ranking scores, a weighted sum of rectified dot products over four small heads."""
    s = torch.zeros((heads, n, n), device="cuda", dtype=torch.float32)
    for h in range(heads):
        keys = _normal(gen, (n, 32))
        for _ in range(4):
            queries = _normal(gen, (n, 32))
            weight = 0.5 + torch.rand((n, 1), generator=gen, device="cuda")
            s[h] += torch.relu_(queries @ keys.T).mul_(weight)
    return s


def _plan(case):
    seqlens = [int(x) for x in case["seqlens"].split(",")]
    mu = tuple(int(x) for x in case["mu"].split("/"))
    kw = dict(seqlens=seqlens, num_q_heads=case["hq"], num_kv_heads=case["hkv"], block=case["block"],
              budget_permille=case["permille"], mu=mu, local_blocks=case["local"], share_group=case["share"],
              score_mode=case["mode"])
    if case["path"] == "chunk":
        # the cache is allocated for the whole sequence, here a third longer than the prefix seen so far
        total = seqlens[0] + seqlens[0] // 3
        kw.update(q_starts=[seqlens[0] - case["chunk"]], total_lens=[total],
                  kcache_blocks_per_seq=(total + case["block"] - 1) // case["block"])
    return stem.StemPlan(**kw)


def _empty_lists(info):
    return (torch.full((info.list_heads, info.total_q_blocks, info.k_max), -1, dtype=torch.int32, device="cuda"),
            torch.zeros((info.list_heads, info.total_q_blocks), dtype=torch.int32, device="cuda"))


def _prepare_token(case, gen):
    n, hq, hkv = case["n"], case["hq"], case["hkv"]
    k_tok = stem.stem_token_budget(n, case["k_start"], (7, 10), case["stem_tokens"], case["local"])
    k_max = int(k_tok.max())
    state = {"case": case, "k_tok": k_tok.cuda(), "scores": _indexer_scores(gen, n, hkv),
             "idx": torch.full((hkv, n, k_max), -1, dtype=torch.int32, device="cuda"),
             "cnt": torch.zeros((hkv, n), dtype=torch.int32, device="cuda")}
    if case["path"] == "token_attend":
        # the lists come from the selector, as they do in the layer before this call
        stem.stem_token_select(state.pop("scores"), state["k_tok"], state["idx"], state["cnt"], case["stem_tokens"], case["local"])
        state["q"], state["k"], state["v"] = _make_qkv(gen, [n], hq, hkv)
        state["out"] = torch.empty((n, hq, D), dtype=torch.bfloat16, device="cuda")
        state["lse"] = torch.empty((hq, n), dtype=torch.float32, device="cuda")
    return state


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["path"].startswith("token"):
        return _prepare_token(case, gen)
    seqlens = [int(x) for x in case["seqlens"].split(",")]
    q, k, v = _make_qkv(gen, seqlens, case["hq"], case["hkv"])
    plan = _plan(case)
    info = plan.info
    plan.workspace()
    state = {"case": case, "plan": plan, "q": q, "k": k, "v": v}
    if case["path"] == "chunk":
        state["q"] = q[seqlens[0] - case["chunk"]:].contiguous()
        state["kcache"] = torch.zeros(int(info.kcache_bytes), dtype=torch.uint8, device="cuda")
        # the prefix is in the cache already: its key blocks were pooled when its chunks ran
        before = seqlens[0] - case["chunk"]
        if before:
            kw = dict(seqlens=[before], num_q_heads=case["hq"], num_kv_heads=case["hkv"], block=case["block"],
                      budget_permille=case["permille"], total_lens=[seqlens[0] + seqlens[0] // 3],
                      kcache_blocks_per_seq=(seqlens[0] + seqlens[0] // 3 + case["block"] - 1) // case["block"])
            prefix = stem.StemPlan(**kw)
            stem.stem_pool_kv(prefix, k[:before], v[:before], state["kcache"])
            torch.cuda.synchronize()
            prefix.close()
    if case["path"] in ("prefill", "chunk", "dense"):
        state["out"] = torch.empty((info.total_tokens, case["hq"], D), dtype=torch.bfloat16, device="cuda")
    if case["path"] in ("chunk", "dense"):  # partial results of these are merged with others', so their LSE is wanted
        state["lse"] = torch.empty((case["hq"], info.total_tokens), dtype=torch.float32, device="cuda")
    if case["path"] != "dense":
        state["idx"], state["cnt"] = _empty_lists(info)
    if case["path"] == "metric":
        state["M"] = torch.zeros((info.list_heads, info.metric_elems), dtype=torch.float32, device="cuda")
    return state


def run(state):
    path = state["case"]["path"]
    if path == "token_select":
        stem.stem_token_select(state["scores"], state["k_tok"], state["idx"], state["cnt"], state["case"]["stem_tokens"],
                               state["case"]["local"])
        return {"idx": state["idx"], "cnt": state["cnt"]}
    if path == "token_attend":
        stem.stem_token_attention(state["q"], state["k"], state["v"], state["idx"], state["cnt"], state["out"], state["lse"])
        return {"out": state["out"], "lse": state["lse"]}
    plan, q, k, v = state["plan"], state["q"], state["k"], state["v"]
    if path == "prefill":
        stem.stem_prefill(plan, q, k, v, state["out"], state["idx"], state["cnt"])
        return {"out": state["out"], "idx": state["idx"], "cnt": state["cnt"]}
    if path == "chunk":
        stem.stem_prefill_cached(plan, q, k, v, state["out"], state["kcache"], True, state["idx"], state["cnt"], state["lse"])
        return {"out": state["out"], "lse": state["lse"], "idx": state["idx"], "cnt": state["cnt"]}
    if path == "dense":
        stem.stem_sparse_prefill(plan, q, k, v, None, None, state["out"], state["lse"])
        return {"out": state["out"], "lse": state["lse"]}
    if path == "lists":
        stem.stem_score_select(plan, q, k, v, state["idx"], state["cnt"])
        return {"idx": state["idx"], "cnt": state["cnt"]}
    stem.stem_score(plan, q, k, v, state["M"])
    stem.stem_select(plan, state["M"], state["idx"], state["cnt"])
    return {"M": state["M"], "idx": state["idx"], "cnt": state["cnt"]}


def work(case):
    hq, hkv = case["hq"], case["hkv"]
    if case["path"].startswith("token"):
        n = case["n"]
        k_tok = stem.stem_token_budget(n, case["k_start"], (7, 10), case["stem_tokens"], case["local"]).to(torch.int64)
        kept = int(k_tok.sum()) * hkv
        if case["path"] == "token_select":  # causal scores read, padded lists written
            return {"bytes": 4 * hkv * (n * (n + 1) // 2 + n * int(k_tok.max()) + n), "flops": 0}
        return {"bytes": 2 * D * n * (2 * hq + 2 * hkv) + 4 * kept + 4 * hq * n, "flops": 4 * D * kept * (hq // hkv)}
    plan = _plan(case)
    info = plan.info
    plan.close()
    t_q, t_kv, block = info.total_tokens, info.total_kv_tokens, case["block"]
    q_bytes, kv_bytes = 2 * D * t_q * hq, 2 * D * t_kv * hkv * 2
    list_bytes = 4 * info.list_heads * info.total_q_blocks * (info.k_max + 1)
    # metric: one multiply-add per dimension and causal block pair; B of them in the anti-diagonal mode
    metric_flops = 2 * D * info.causal_blocks * info.list_heads // hq * (block if case["mode"] else 1)
    if case["path"] == "dense":
        return {"bytes": 2 * q_bytes + kv_bytes + 4 * hq * t_q, "flops": 4 * D * info.causal_pairs}
    if case["path"] == "lists":
        return {"bytes": q_bytes + kv_bytes + list_bytes, "flops": metric_flops}
    if case["path"] == "metric":
        return {"bytes": q_bytes + kv_bytes + list_bytes + 4 * info.causal_blocks, "flops": metric_flops}
    lse_bytes = 4 * hq * t_q if case["path"] == "chunk" else 0
    return {"bytes": 2 * q_bytes + kv_bytes + list_bytes + lse_bytes, "flops": 4 * D * info.selected_pairs + metric_flops}


def tolerance(case):
    """Lists are decided by comparing sums: another order of summation swaps near-ties (``differ``; the fused path
    against sums in 64 bits: fewer than 2 lists in 10^4 at 128K tokens).  O is bf16 and its probabilities are rounded
    to bf16 before they meet V (``rel``; against 64 bits: 2e-3)."""
    if case["path"] == "token_select":
        return "exact"
    if case["path"] == "lists":
        # the anti-diagonal sums have 8192 or 16384 terms in one fp32 accumulator
        return {"rel": 0.0, "differ": 5e-3 if case["mode"] else 1e-3}
    if case["path"] == "metric":
        return {"rel": 1e-5, "differ": 1e-3}
    if case["path"] in ("dense", "token_attend"):
        return {"rel": 1e-2}
    return {"rel": 1e-2, "differ": 1e-3}
