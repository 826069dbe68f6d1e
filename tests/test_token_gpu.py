"""GPU parity of the token-level path (Main Results: Token Position-Decay on a selector that keeps the top 2048
tokens per query, k_start = 2048, mu = 0.7): the budget k(t) of Eq. 3 at token positions, exact top-k(t) selection
from caller-supplied indexer scores, and gather-style attention over the token lists.  The CPU checker is
Algorithm 1's own code with a block size of one token."""
import numpy as np
import pytest
import torch

from oracle import stem_oracle as so
from paper_2603_06274_b200 import binding, workloads as wl
from tests._util import check_attention, from_dev_bf16, to_dev

pytestmark = pytest.mark.gpu


def _scores(seed, heads, n, ties):
    r = np.random.Generator(np.random.PCG64([seed, 31]))
    m = r.standard_normal((heads, n, n), dtype=np.float32)
    if ties:
        m = np.round(m * 3.0) / 3.0
        m[0, n - 1, 5:40] = np.nan
        m[heads - 1, n // 2, 0:n // 4:3] = np.inf
        m[0, n // 3, 10:20] = -np.inf
        m[m == 0.0] = -0.0
    return m


def _case(n, hq, hkv, k_start, stem, local, seed, ties, sample=None):
    w = wl.small(f"token_{n}", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=True, seed=seed)
    data = wl.make_qkv(w)
    g = hq // hkv
    p = so.StemParams(block=1, k_start_blocks=k_start, mu_num=7, mu_den=10, stem_blocks=stem, local_blocks=local)
    k_ref = so.schedule(n, k_start, p)[1]
    k_tok = binding.stem_token_budget(n, k_start, (7, 10), stem, local)
    assert np.array_equal(k_tok.numpy(), k_ref)
    k_max = int(k_ref.max())
    sc = _scores(seed, hkv, n, ties)
    idx_ref, cnt_ref = so.select(sc.reshape(hkv, -1), np.array([n], np.int32), k_ref, stem, local)
    idx = torch.full((hkv, n, k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((hkv, n), -7, dtype=torch.int32, device="cuda")
    binding.stem_token_select(torch.from_numpy(sc).cuda(), k_tok.cuda(), idx, cnt, stem, local)
    torch.cuda.synchronize()
    assert np.array_equal(cnt.cpu().numpy(), cnt_ref)
    assert np.array_equal(idx.cpu().numpy(), idx_ref)
    # gather attention on those lists; the checker runs Algorithm 1 step d with one token per block
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_token_attention(q, k, v, idx, cnt, out, lse)
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    ei, ec = so.expand_group_lists(idx_ref, cnt_ref, g)
    rows = None
    if sample is not None:
        r = np.random.default_rng(seed)
        toks = np.unique(np.concatenate([[0, 1, k_start - 1, k_start, n // 2, n - 1], r.integers(0, n, sample)]))
        rows = np.array([(h, t) for h in range(hq) for t in toks], dtype=np.int32)
    O_ref, lse_ref = so.attention(data["q"], data["k"], data["v"], data["cu_seqlens"], 1, ei, ec, rows=rows)
    mask = ~np.isnan(O_ref)
    check_attention(from_dev_bf16(out), O_ref, mask, label=f"token-level n={n} k_start={k_start}")
    lm = ~np.isnan(lse_ref)
    assert np.abs(lse.cpu().numpy()[lm] - lse_ref[lm]).max() < 1e-3
    assert torch.isfinite(out.float()).all()


def test_token_level_selection_and_gather_attention_small():
    _case(n=700, hq=4, hkv=2, k_start=200, stem=4, local=8, seed=7, ties=True)
    _case(n=333, hq=3, hkv=3, k_start=64, stem=0, local=1, seed=8, ties=False)
    _case(n=520, hq=8, hkv=1, k_start=300, stem=2, local=3, seed=10, ties=False)   # 8 query heads on one kv head


def test_token_level_top_2048_selector():
    # the paper's setting for that integration: k_start = 2048, mu = 0.7; 4096 tokens, GQA 4
    _case(n=4096, hq=8, hkv=2, k_start=2048, stem=0, local=1, seed=9, ties=True, sample=40)


def test_token_level_rows_of_9000_tokens():
    # lists longer than one 2048-token budget window, rows that span several passes of every thread over the keys
    _case(n=9000, hq=2, hkv=1, k_start=2048, stem=2, local=4, seed=11, ties=True, sample=12)


def test_gather_attention_on_hand_made_lists_with_strided_tensors():
    # 16 query heads on one kv head (the widest group), lists of any length from 0 to 140 tokens (a list need not come
    # from the selector; empty lists give a zero row and lse = -inf), Q / K / V as slices of wider tensors
    n, hq, hkv = 300, 16, 1
    w = wl.small("token_lists", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=False, seed=21)
    data = wl.make_qkv(w)
    r = np.random.default_rng(21)
    k_max = 140
    idx_ref = np.full((hkv, n, k_max), -1, np.int32)
    cnt_ref = np.zeros((hkv, n), np.int32)
    for t in range(n):
        m = 0 if r.random() < 0.1 else int(r.integers(1, min(t + 1, k_max) + 1))
        idx_ref[0, t, :m] = np.sort(r.choice(t + 1, size=m, replace=False))
        cnt_ref[0, t] = m
    q_wide = torch.zeros((n, hq + 4, 128), dtype=torch.bfloat16, device="cuda")
    k_wide = torch.zeros((n, 3, 128), dtype=torch.bfloat16, device="cuda")
    v_wide = torch.zeros((n, 3, 128), dtype=torch.bfloat16, device="cuda")
    q, k, v = q_wide[:, 2:2 + hq], k_wide[:, 1:2], v_wide[:, 1:2]
    q.copy_(to_dev(data["q"])); k.copy_(to_dev(data["k"])); v.copy_(to_dev(data["v"]))
    out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_token_attention(q, k, v, torch.from_numpy(idx_ref).cuda(), torch.from_numpy(cnt_ref).cuda(), out, lse)
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    ei, ec = so.expand_group_lists(idx_ref, cnt_ref, hq // hkv)
    O_ref, lse_ref = so.attention(data["q"], data["k"], data["v"], data["cu_seqlens"], 1, ei, ec)
    check_attention(from_dev_bf16(out), O_ref, label="hand-made token lists, 16 heads per kv head")
    empty = cnt_ref[0] == 0
    assert empty.any()
    assert (from_dev_bf16(out)[empty] == 0).all()
    got_lse = lse.cpu().numpy()
    assert np.isneginf(got_lse[:, empty]).all() and np.isneginf(lse_ref[:, empty]).all()
    assert np.abs(got_lse[:, ~empty] - lse_ref[:, ~empty]).max() < 1e-3


@pytest.mark.parametrize("seed", [31, 32, 33, 34, 35, 36])
def test_gather_attention_on_random_shapes_and_list_lengths(seed):
    # item boundaries in every phase of the pipeline: lists of 0 .. 3 tiles in random order, any group size; the
    # result must also be the same bits on a second run
    r = np.random.default_rng(seed)
    hkv = int(r.integers(1, 4))
    g = int(r.choice([1, 2, 3, 4, 5, 8, 12, 16]))
    hq = hkv * g
    n = int(r.integers(130, 420))
    w = wl.small(f"token_fuzz_{seed}", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=bool(seed & 1), seed=seed)
    data = wl.make_qkv(w)
    k_max = int(r.integers(1, n + 1))
    idx_ref = np.full((hkv, n, k_max), -1, np.int32)
    cnt_ref = np.zeros((hkv, n), np.int32)
    for h in range(hkv):
        for t in range(n):
            top = min(t + 1, k_max)
            m = int(r.choice([0, 1, min(top, 127), min(top, 128), min(top, 129), top, int(r.integers(0, top + 1))]))
            idx_ref[h, t, :m] = np.sort(r.choice(t + 1, size=m, replace=False))
            cnt_ref[h, t] = m
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    idx, cnt = torch.from_numpy(idx_ref).cuda(), torch.from_numpy(cnt_ref).cuda()
    outs = []
    for _ in range(2):
        out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
        binding.stem_token_attention(q, k, v, idx, cnt, out, lse)
        st, detail = binding.stem_token_check_status()
        assert st == 0, detail
        outs.append((out, lse))
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16))
    assert torch.equal(outs[0][1].view(torch.int32), outs[1][1].view(torch.int32))
    ei, ec = so.expand_group_lists(idx_ref, cnt_ref, g)
    O_ref, lse_ref = so.attention(data["q"], data["k"], data["v"], data["cu_seqlens"], 1, ei, ec)
    check_attention(from_dev_bf16(outs[0][0]), O_ref, label=f"random token lists, n={n}, {hq}/{hkv} heads, k_max={k_max}")
    got = outs[0][1].cpu().numpy()
    empty = np.repeat(cnt_ref == 0, g, axis=0)
    assert np.isneginf(got[empty]).all()
    assert np.abs(got[~empty] - lse_ref[~empty]).max() < 1e-3


def test_token_level_argument_errors():
    with pytest.raises(binding.StemError):
        binding.stem_token_budget(100, 10, (11, 10))
    q = torch.zeros((64, 34, 128), dtype=torch.bfloat16, device="cuda")
    kv = torch.zeros((64, 2, 128), dtype=torch.bfloat16, device="cuda")
    idx = torch.zeros((2, 64, 4), dtype=torch.int32, device="cuda")
    cnt = torch.zeros((2, 64), dtype=torch.int32, device="cuda")
    with pytest.raises(binding.StemError) as e:
        binding.stem_token_attention(q, kv, kv, idx, cnt, torch.empty_like(q))     # 17 query heads per kv head
    assert e.value.status == binding.STEM_ERR_UNSUPPORTED


def _lists(r, n, hkv, k_max, order="ascending", repeat=False):
    """Lists of 0 .. min(t + 1, k_max) tokens; with ``repeat`` some lists name a token twice."""
    idx = np.full((hkv, n, k_max), -1, np.int32)
    cnt = np.zeros((hkv, n), np.int32)
    for h in range(hkv):
        for t in range(n):
            top = min(t + 1, k_max)
            m = int(r.choice([0, 1, top, int(r.integers(0, top + 1))], p=[0.05, 0.05, 0.3, 0.6]))
            pick = r.choice(t + 1, size=m, replace=False)
            if repeat and m > 1 and r.random() < 0.3:
                pick[0] = pick[1]
            idx[h, t, :m] = np.sort(pick) if order == "ascending" else pick
            cnt[h, t] = m
    return idx, cnt


def _plain_attention(q, k, v, idx, cnt, rows):
    """fp64 attention of the listed rows (h, t): softmax over the list's entries, a repeated entry counted as often as it appears."""
    hq, hkv = q.shape[1], k.shape[1]
    out, lse = {}, {}
    for h, t in rows:
        kvh = h // (hq // hkv)
        ids = np.clip(idx[kvh, t, :cnt[kvh, t]], 0, t)
        s = k[ids, kvh].astype(np.float64) @ q[t, h].astype(np.float64) / np.sqrt(128.0)
        p = np.exp(s - s.max())
        out[h, t] = (p / p.sum()) @ v[ids, kvh].astype(np.float64)
        lse[h, t] = s.max() + np.log(p.sum())
    return out, lse


# The masked form (every causal key block, the keys outside a list masked out) is taken where it is estimated to be the
# faster one, the gather form for lists that are short against the prefix.  Masks live in the token's own rows of O up to
# 2048 g keys, beyond in rows of earlier tokens.
@pytest.mark.parametrize("n,hq,hkv,k_max,order,repeat,what", [
    (2048, 4, 4, 512, "ascending", False, "masked, masks that just fit the tokens' own rows"),
    (2049, 4, 4, 512, "ascending", False, "masked, two launches: masks in rows of earlier tokens"),
    (4300, 2, 2, 1501, "any", True, "masked, four launches, two windows of flags, entries read one at a time"),
    (897, 28, 4, 300, "ascending", True, "masked, 18-token tiles, lists that name a token twice"),
    (129, 64, 4, 128, "any", True, "masked, 8-token tiles, one token past a key block"),
    (1000, 64, 8, 400, "ascending", True, "masked, an odd number of 16-token tiles in pairs"),
    (2050, 28, 4, 512, "any", False, "masked, 18-token tiles in pairs that span two key blocks"),
    (3000, 2, 2, 20, "ascending", False, "gather: lists short against the prefix"),
    (300, 5, 1, 27, "any", True, "gather, lists in any order and with repeats"),
])
def test_token_attention_forms(n, hq, hkv, k_max, order, repeat, what):
    assert what.startswith(binding.stem_token_attention_form(n, hq, hkv, k_max))
    r = np.random.default_rng(n + k_max)
    w = wl.small("token_forms", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=True, seed=n)
    data = wl.make_qkv(w)
    idx, cnt = _lists(r, n, hkv, k_max, order, repeat)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_token_attention(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), out, lse)
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    g = hq // hkv
    rows = [(h, t) for h in range(hq) for t in sorted({0, 1, 127, 128, n // 2, n - 1, *r.integers(0, n, 150).tolist()}) if t < n and cnt[h // g, t] > 0]
    O_ref, lse_ref = _plain_attention(from_dev_bf16(q), from_dev_bf16(k), from_dev_bf16(v), idx, cnt, rows)
    got, got_lse = from_dev_bf16(out), lse.cpu().numpy()
    ref = np.stack([O_ref[x] for x in rows])
    check_attention(np.stack([got[t, h] for h, t in rows]), ref, np.ones(ref.shape, bool), label=what)
    assert max(abs(got_lse[h, t] - lse_ref[h, t]) for h, t in rows) < 1e-3
    empty = np.repeat(cnt == 0, g, axis=0)
    assert (got.transpose(1, 0, 2)[empty] == 0).all() and np.isneginf(got_lse[empty]).all()
    assert np.isfinite(got).all()


@pytest.mark.parametrize("shape,form", [((1500, 4, 2, 100), "masked"), ((400, 4, 2, 100), None), ((200, 4, 2, 100), "gather")])
def test_token_attention_ignores_rows_no_list_names(shape, form):
    # a value row that is not finite reaches only the queries whose lists name it, and so does a key row, in either form
    n, hq, hkv, k_max = shape
    assert form in (None, binding.stem_token_attention_form(n, hq, hkv, k_max))
    w = wl.small("token_nan", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=False, seed=5)
    data = wl.make_qkv(w)
    r = np.random.default_rng(5)
    idx, cnt = _lists(r, n, hkv, k_max)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    outs = []
    for bad in (False, True):
        if bad:
            v[37] = float("inf")
            k[38] = float("nan")
        out = torch.empty((n, hq, 128), dtype=torch.bfloat16, device="cuda")
        binding.stem_token_attention(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), out)
        st, detail = binding.stem_token_check_status()
        assert st == 0, detail
        outs.append(from_dev_bf16(out))
    named = np.array([[np.isin([37, 38], idx[h, t, :cnt[h, t]]).any() for t in range(n)] for h in range(hkv)])
    clean = np.repeat(~named, hq // hkv, axis=0).T
    assert clean.any() and not clean.all()
    check_attention(outs[1][clean], outs[0][clean], np.ones(outs[0][clean].shape, bool), label="rows whose lists name no bad row")
    assert not np.isfinite(outs[1][~clean]).all(axis=1).any()


@pytest.mark.parametrize("n,heads,k_start,stem,local,ties", [
    (33, 2, 7, 0, 1, True),          # less than a warp's row
    (1024, 1, 300, 3, 5, True),      # one warp to a row, its last row full
    (1025, 2, 1000, 0, 1, False),    # the first row of two warps; N not a multiple of four: scalar loads
    (2052, 1, 64, 1, 2, True),       # rows of two and of four warps
    (4097, 1, 2048, 0, 1, False),    # the first row of eight warps
    (8200, 1, 500, 4, 8, True),      # rows of ten warps
    (15000, 1, 2048, 0, 1, False),   # up to sixteen
    (16388, 1, 700, 0, 1, True),     # longer than the registers hold: the other kernel for all rows
    (1030, 2, 200, 0, 1, "low"),     # scores alike in their upper 16 bits, or in all but the last four
    (4100, 1, 900, 2, 3, "low"),
    (300, 2, 33, 0, 1, "low"),
])
def test_token_selection_row_lengths(n, heads, k_start, stem, local, ties):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    sc = torch.randn((heads, n, n), generator=g, device="cuda")
    if ties == "low":
        last = torch.randint(0, 40000 if n % 4 else 16, (heads, n, n), generator=g, device="cuda", dtype=torch.int32)
        sc = (torch.where(sc < 0.0, -1.5, 1.5).view(torch.int32) + last).view(torch.float32)
    elif ties:
        sc = torch.round(sc * 2.0) / 2.0 * torch.where(torch.rand((heads, n, n), generator=g, device="cuda") < 0.5, 1.0, -1.0)
        sc[0, n - 1, 3:9] = float("nan")
        sc[0, n // 2, ::5] = float("inf")
        sc[0, n // 3, 1::4] = float("-inf")
    k_tok = binding.stem_token_budget(n, k_start, (7, 10), stem, local)
    k_max = int(k_tok.max())
    idx = torch.full((heads, n, k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((heads, n), -7, dtype=torch.int32, device="cuda")
    binding.stem_token_select(sc, k_tok.cuda(), idx, cnt, stem, local)
    torch.cuda.synchronize()
    rows = sorted({0, 1, stem + local - 1, k_start - 1, k_start, n // 3, n // 2, n - 1, 1023, 1024, 2047, 2048, 4095, 4096, 8191, 8192}
                  | {1024 * k + d for k in range(1, 17) for d in (-1, 0)}
                  | set(np.random.default_rng(n).integers(0, n, 40).tolist()))
    for h in range(heads):
        for t in [t for t in rows if 0 <= t < n]:
            s = sc[h, t, :t + 1].cpu().numpy().astype(np.float64)
            s[np.isnan(s)] = -np.inf
            forced = (np.arange(t + 1) < stem) | (np.arange(t + 1) > t - local)
            free = np.flatnonzero(~forced)
            want = max(int(k_tok[t]) - int(forced.sum()), 0)
            best = free[np.lexsort((free, -s[free]))][:want]
            ref = np.sort(np.concatenate([np.flatnonzero(forced), best]))
            got = idx[h, t].cpu().numpy()
            assert int(cnt[h, t]) == len(ref)
            assert np.array_equal(got[:len(ref)], ref), (h, t)
            assert (got[len(ref):] == -1).all()


def _random_lists(r, n, hkv, k_max):
    """Full lists (min(t + 1, k_max) tokens) in random order."""
    idx = np.full((hkv, n, k_max), -1, np.int32)
    for h in range(hkv):
        for t in range(n):
            m = min(t + 1, k_max)
            idx[h, t, :m] = r.permutation(t + 1)[:m]
    return idx, np.broadcast_to(np.minimum(np.arange(n) + 1, k_max).astype(np.int32), (hkv, n)).copy()


# The masked form leaves the rows that a mask cannot express to the gather kernel: lists that name a token twice, and every
# row behind a value that is not finite.  Long lists, where one thread to a row would outlast the bounded waits.
@pytest.mark.parametrize("what", ["a token named twice by every 97th list", "by every list", "an infinite value row"])
def test_rows_that_a_mask_cannot_express_at_long_lists(what):
    n, hq, hkv, k_max = 8300, 4, 2, 8192
    assert binding.stem_token_attention_form(n, hq, hkv, k_max) == "masked"
    r = np.random.default_rng(83)
    g = torch.Generator(device="cuda")
    g.manual_seed(83)
    q, k, v = (torch.randn((n, h, 128), generator=g, device="cuda").to(torch.bfloat16) for h in (hq, hkv, hkv))
    idx, cnt = _random_lists(r, n, hkv, k_max)
    step = 97 if "97" in what else 1
    bad = 5
    if "infinite" in what:
        v[bad, 0] = float("inf")                       # of kv head 0 alone
        for t in range(8193, n, 2):                    # lists without this token, in its place one that they did not name
            if (idx[0, t] == bad).any():
                idx[0, t][idx[0, t] == bad] = np.setdiff1d(np.arange(t + 1), idx[0, t])[0]
    else:
        idx[:, 1::step, 0] = idx[:, 1::step, 1]
    outs = []
    for _ in range(2):
        out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
        binding.stem_token_attention(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), out, lse)
        st, detail = binding.stem_token_check_status()
        assert st == 0, detail
        outs.append((out, lse))
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16))
    got, got_lse = from_dev_bf16(outs[0][0]), outs[0][1].cpu().numpy()
    toks = sorted({0, 1, 2, 96, 97, 98, 127, 128, 4095, 4096, 8191, 8192, n - 2, n - 1, *r.integers(0, n, 60).tolist(), *range(8193, n, 7)})
    rows = [(h, t) for h in range(hq) for t in toks]
    named = {(h, t): "infinite" in what and h < 2 and bool((idx[0, t, :cnt[0, t]] == bad).any()) for h, t in rows}
    clean = [x for x in rows if not named[x]]
    O_ref, lse_ref = _plain_attention(from_dev_bf16(q), from_dev_bf16(k), from_dev_bf16(v), idx, cnt, clean)
    ref = np.stack([O_ref[x] for x in clean])
    check_attention(np.stack([got[t, h] for h, t in clean]), ref, np.ones(ref.shape, bool), label=what)
    assert max(abs(got_lse[h, t] - lse_ref[h, t]) for h, t in clean) < 1e-3
    if "infinite" in what:
        assert any(t > bad and h < 2 for h, t in clean) and any(named.values())
        assert all(not np.isfinite(got[t, h]).any() for h, t in rows if named[h, t])
    else:
        assert np.isfinite(got).all()


def test_marked_rows_over_several_launches_and_streams():
    # masks in rows of earlier tokens (two launches) with repeats; calls without marked rows on another stream meanwhile
    n, hq, hkv, k_max = 2049, 4, 4, 512
    assert binding.stem_token_attention_form(n, hq, hkv, k_max) == "masked"
    r = np.random.default_rng(12)
    g = torch.Generator(device="cuda")
    g.manual_seed(12)
    q, k, v = (torch.randn((n, h, 128), generator=g, device="cuda").to(torch.bfloat16) for h in (hq, hkv, hkv))
    lists = {rep: _lists(r, n, hkv, k_max, "any", rep) for rep in (False, True)}
    dev = {rep: tuple(torch.from_numpy(x).cuda() for x in lists[rep]) for rep in lists}
    outs = {rep: [torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(6)] for rep in lists}
    streams = {rep: torch.cuda.Stream() for rep in lists}
    torch.cuda.synchronize()
    for i in range(6):
        for rep in lists:
            with torch.cuda.stream(streams[rep]):
                binding.stem_token_attention(q, k, v, *dev[rep], outs[rep][i])
    torch.cuda.synchronize()
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    for rep, (idx, cnt) in lists.items():
        rows = [(h, t) for h in range(hq) for t in sorted({0, 1, 127, 128, n - 1, *r.integers(0, n, 100).tolist()}) if cnt[h, t] > 0]
        O_ref, _ = _plain_attention(from_dev_bf16(q), from_dev_bf16(k), from_dev_bf16(v), idx, cnt, rows)
        ref = np.stack([O_ref[x] for x in rows])
        got = from_dev_bf16(outs[rep][0])
        check_attention(np.stack([got[t, h] for h, t in rows]), ref, np.ones(ref.shape, bool), label=f"repeats {rep}")
        for o in outs[rep][1:]:
            assert torch.equal(o.view(torch.int16), outs[rep][0].view(torch.int16))


# O in the place of Q: served by the gather form at every size (the masked one keeps its masks in O).  Also the gather form
# on lists of many tiles: its ring wraps, the row reference is raised more than once, all its completion barriers turn over.
@pytest.mark.parametrize("n,hq,hkv,k_max,order,repeat", [
    (600, 4, 2, 300, "ascending", False),
    (2500, 8, 1, 2048, "ascending", False),     # up to 16 tiles
    (4300, 16, 1, 1501, "any", True),
    (3001, 3, 3, 2900, "any", False),           # up to 23 tiles, one head to a group
    (1200, 28, 4, 900, "ascending", True),
])
def test_output_in_the_place_of_the_queries(n, hq, hkv, k_max, order, repeat):
    assert binding.stem_token_attention_form(n, hq, hkv, k_max) == "masked"     # with an O of its own
    r = np.random.default_rng(n)
    w = wl.small("token_inplace", seqlens=(n,), hq=hq, hkv=hkv, block=64, permille=100, sink=True, seed=n)
    data = wl.make_qkv(w)
    idx, cnt = _lists(r, n, hkv, k_max, order, repeat)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    q_np = from_dev_bf16(q)
    lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_token_attention(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), q, lse)
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    g = hq // hkv
    rows = [(h, t) for h in range(hq) for t in sorted({0, 1, 127, 128, n // 2, n - 1, *r.integers(0, n, 150).tolist()}) if cnt[h // g, t] > 0]
    O_ref, lse_ref = _plain_attention(q_np, from_dev_bf16(k), from_dev_bf16(v), idx, cnt, rows)
    got, got_lse = from_dev_bf16(q), lse.cpu().numpy()
    ref = np.stack([O_ref[x] for x in rows])
    check_attention(np.stack([got[t, h] for h, t in rows]), ref, np.ones(ref.shape, bool), label="O in the place of Q")
    assert max(abs(got_lse[h, t] - lse_ref[h, t]) for h, t in rows) < 1e-3
    empty = np.repeat(cnt == 0, g, axis=0)
    assert (got.transpose(1, 0, 2)[empty] == 0).all() and np.isneginf(got_lse[empty]).all()


@pytest.mark.parametrize("n,hq,hkv", [(1500, 4, 2), (1400, 7, 1)])
def test_row_maxima_that_grow_from_block_to_block_in_the_masked_form(n, hq, hkv):
    # The scores of key block j are about step[j] powers of two: a row's reference stays (growth of less than 8), moves once or
    # moves with every block; some lists name nothing in the blocks that outgrow it.
    k_max = 150
    assert binding.stem_token_attention_form(n, hq, hkv, k_max) == "masked"
    r = np.random.default_rng(n + hq)
    step = np.array([0, 7, 14, 22, 21, 48, 71, 95, 95, 60, 90, 120])[:(n + 127) // 128]
    u = r.standard_normal(128)
    u /= np.linalg.norm(u)
    scale = np.sqrt(128) / np.log2(np.e) / 8  # q = 8 u, so that k = scale * step * u scores `step` powers of two
    dev = lambda t: torch.from_numpy(t).to(device="cuda", dtype=torch.bfloat16)
    k = dev(np.repeat(step, 128)[:n, None, None] * scale * u + 0.3 * r.standard_normal((n, hkv, 128)))
    q = dev(8 * u + 0.3 * r.standard_normal((n, hq, 128)))
    v = dev(r.standard_normal((n, hkv, 128)))
    idx = np.full((hkv, n, k_max), -1, np.int32)
    cnt = np.zeros((hkv, n), np.int32)
    for h in range(hkv):
        for t in range(n):
            tokens = np.arange(t + 1)
            if t % 3 == 1:
                tokens = tokens[tokens // 128 != t // 128] if t >= 128 else tokens
            pick = np.sort(r.choice(tokens, min(len(tokens), k_max), replace=False))
            idx[h, t, :len(pick)] = pick
            cnt[h, t] = len(pick)
    out = torch.full((n, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((hq, n), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_token_attention(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), out, lse)
    st, detail = binding.stem_token_check_status()
    assert st == 0, detail
    g = hq // hkv
    named = torch.zeros((hkv, n, n + 1), dtype=torch.bool, device="cuda")
    named.scatter_(2, torch.from_numpy(np.where(idx < 0, n, idx)).cuda().long(), True)
    s = torch.einsum("thd,shd->hts", q.double(), k.double().repeat_interleave(g, 1)) / np.sqrt(128)
    s = s.masked_fill(~named[:, :, :n].repeat_interleave(g, 0), float("-inf"))
    ref = torch.einsum("hts,shd->thd", torch.softmax(s, 2), v.double().repeat_interleave(g, 1))
    check_attention(from_dev_bf16(out), ref.cpu().numpy(), label=f"growing maxima, token lists, {hq}/{hkv} heads")
    assert (lse - torch.logsumexp(s, 2)).abs().max() < 1e-3
