"""GPU parity of the anti-diagonal scoring mode (Overall Algorithm, "anti-diagonal scoring"; Alg. 1 step 1
comment, stride = B): the metric from the tensor-core contraction of Q with K against the CPU checker's
plain anti-diagonal means, then selection and attention through the fused path."""
import numpy as np
import pytest
import torch

from oracle import stem_oracle as so
from paper_2603_06274_b200 import binding, workloads as wl
from paper_2603_06274_b200.binding import StemPlan
from tests._util import check_attention, compare_selection, from_dev_bf16, oracle_params, sample_rows, to_dev

pytestmark = pytest.mark.gpu

# The contraction adds B * d = 16384 exact bf16 products into one fp32 tensor-memory accumulator over 1024 MMAs, and
# the tensor core's accumulation truncates: a running sum of a few hundred picks up about 1e-2 before the division
# by B, i.e. about 1e-4 on metric values of order 1 (measured 1.4e-4).  The checker sums in fp64.  Lists may then
# differ from the checker's only at near-ties of 1e-3 relative, like on the block-mean path.
METRIC_ABS, METRIC_REL = 3e-4, 1e-4

CASES = {
    # full blocks only, two column tiles
    "full_b128": wl.small("ad_full_b128", seqlens=(130 * 128,), hq=2, hkv=1, block=128, permille=100, sink=True),
    # ragged last block (its metric row comes from the plain-FMA kernel), GQA 3, varlen batch with a tiny sequence
    "ragged_varlen": wl.small("ad_ragged", seqlens=(1000, 50, 1664), hq=6, hkv=2, block=128, permille=300),
    # block 64
    "b64": wl.small("ad_b64", seqlens=(2500,), hq=2, hkv=2, block=64, permille=250),
}


@pytest.mark.parametrize("name", list(CASES))
def test_antidiagonal_metric_and_fused_path_match_checker(name):
    w = CASES[name]
    data = wl.make_qkv(w)
    p = oracle_params(w)
    M_ref, _ = so.score_antidiag(data["q"], data["k"], data["v"], data["cu_seqlens"], p)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    plan = StemPlan.from_workload(w, score_mode=1)
    info = plan.info
    M = torch.full((w.num_q_heads, info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_score(plan, q, k, v, M)
    assert binding.stem_check_status(plan)[0] == 0
    M_g = M.cpu().numpy()
    defined = ~np.isnan(M_ref)
    assert np.array_equal(np.isnan(M_g), ~defined), "exactly the causal blocks j <= r are written"
    err = np.abs(M_g[defined] - M_ref[defined])
    assert np.all(err <= METRIC_ABS + METRIC_REL * np.abs(M_ref[defined])), f"metric max err {err.max()}"
    # fused path
    nblk = so.n_blocks(w.seqlens, w.block)
    k_eff = so.schedule_batch(w.seqlens, p)
    idx_ref, cnt_ref = so.select(M_ref, nblk, k_eff, w.stem_blocks, w.local_blocks)
    idx = torch.full((w.num_q_heads, info.total_q_blocks, info.k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((w.num_q_heads, info.total_q_blocks), -7, dtype=torch.int32, device="cuda")
    out = torch.full((w.total_tokens, w.num_q_heads, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    binding.stem_prefill(plan, q, k, v, out, idx, cnt)
    assert binding.stem_check_status(plan)[0] == 0
    idx_g, cnt_g = idx.cpu().numpy(), cnt.cpu().numpy()
    ties = compare_selection(idx_g, cnt_g, idx_ref, cnt_ref, M_ref, nblk, w)
    assert len(ties) <= max(2, idx_g.shape[0] * idx_g.shape[1] // 100)
    O_ref, _ = so.attention(data["q"], data["k"], data["v"], data["cu_seqlens"], w.block, idx_g, cnt_g)
    check_attention(from_dev_bf16(out), O_ref, label=w.name)
    # the lists differ from the block-mean mode's (another scoring rule), so the mode switch is live
    plan0 = StemPlan.from_workload(w)
    idx0, cnt0 = torch.empty_like(idx), torch.empty_like(cnt)
    binding.stem_score_select(plan0, q, k, v, idx0, cnt0)
    torch.cuda.synchronize()
    assert torch.equal(cnt0, cnt)
    if name != "ragged_varlen":     # (its sequences are so short that every causal block is kept in either mode)
        assert not torch.equal(idx0, idx)
    plan.close(); plan0.close()


def test_antidiagonal_mode_limits():
    w = CASES["b64"]
    for kw in (dict(share_group=True), dict(kcache_blocks_per_seq=64)):
        with pytest.raises(binding.StemError) as e:
            StemPlan.from_workload(w, score_mode=1, **kw)
        assert e.value.status == binding.STEM_ERR_UNSUPPORTED


def test_32k_layer_in_antidiagonal_mode():
    w = wl.CONFIGS["cfg2"]
    data = wl.make_qkv(w)
    p = oracle_params(w)
    # the checker's anti-diagonal metric of two query heads (heads 0 and 9) in full: 33 k block pairs x 128 dots each
    sub = {"q": np.ascontiguousarray(data["q"][:, [0, 9]]), "k": np.ascontiguousarray(data["k"][:, [0, 2]]),
           "v": np.ascontiguousarray(data["v"][:, [0, 2]])}
    M_ref, _ = so.score_antidiag(sub["q"], sub["k"], sub["v"], data["cu_seqlens"], p)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    plan = StemPlan.from_workload(w, score_mode=1)
    info = plan.info
    M = torch.full((w.num_q_heads, info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_score(plan, q, k, v, M)
    assert binding.stem_check_status(plan)[0] == 0
    M_g = M[[0, 9]].cpu().numpy()
    defined = ~np.isnan(M_ref)
    assert np.array_equal(np.isnan(M_g), ~defined)
    err = np.abs(M_g[defined] - M_ref[defined])
    print(f"anti-diagonal metric at 32K: max abs err {err.max():.2e}")
    assert np.all(err <= METRIC_ABS + METRIC_REL * np.abs(M_ref[defined]))
    # fused path: lists of those heads against the checker, attention on sampled lists
    nblk = so.n_blocks(w.seqlens, w.block)
    k_eff = so.schedule_batch(w.seqlens, p)
    idx_ref, cnt_ref = so.select(M_ref, nblk, k_eff, w.stem_blocks, w.local_blocks)
    idx = torch.empty((w.num_q_heads, info.total_q_blocks, info.k_max), dtype=torch.int32, device="cuda")
    cnt = torch.empty((w.num_q_heads, info.total_q_blocks), dtype=torch.int32, device="cuda")
    out = torch.full((w.total_tokens, w.num_q_heads, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    binding.stem_prefill(plan, q, k, v, out, idx, cnt)
    assert binding.stem_check_status(plan)[0] == 0
    idx_g, cnt_g = idx.cpu().numpy(), cnt.cpu().numpy()
    ties = compare_selection(idx_g[[0, 9]], cnt_g[[0, 9]], idx_ref, cnt_ref, M_ref, nblk, w)
    print(f"{len(ties)} of {2 * info.total_q_blocks} lists differ from the checker at near-ties")
    assert len(ties) <= 4
    rows = sample_rows(w.num_q_heads, nblk, [24, 25], n_random=60, seed=11)
    O_ref, _ = so.attention(data["q"], data["k"], data["v"], data["cu_seqlens"], w.block, idx_g, cnt_g, rows=rows, want_lse=False)
    mask = ~np.isnan(O_ref)
    check_attention(from_dev_bf16(out), O_ref, mask, label=f"{w.name} anti-diagonal mode ({len(rows)} lists)")
    assert torch.isfinite(out.float()).all()
    plan.close()


@pytest.mark.parametrize("block,seqlens,hq,hkv", [
    (128, (128 * 33 + 1,), 1, 1),           # one token in the last block, 34 columns: a second column group
    (128, (128 * 31 + 127, 60), 10, 2),     # all but one token; a sequence without any full block; five heads per group
    (64, (64 * 64 + 33,), 16, 1),           # 65 columns, four rounds of heads
])
def test_antidiagonal_metric_row_of_a_partial_last_block(block, seqlens, hq, hkv):
    w = wl.small("ad_partial", seqlens=seqlens, hq=hq, hkv=hkv, block=block, permille=200, seed=77)
    data = wl.make_qkv(w)
    M_ref, _ = so.score_antidiag(data["q"], data["k"], data["v"], data["cu_seqlens"], oracle_params(w))
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    plan = StemPlan.from_workload(w, score_mode=1)
    M = torch.full((hq, plan.info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_score(plan, q, k, v, M)
    assert binding.stem_check_status(plan)[0] == 0
    M_g = M.cpu().numpy()
    defined = ~np.isnan(M_ref)
    assert np.array_equal(np.isnan(M_g), ~defined)
    assert np.all(np.abs(M_g[defined] - M_ref[defined]) <= METRIC_ABS + METRIC_REL * np.abs(M_ref[defined]))
    plan.close()


def test_a_query_without_a_partner_in_the_last_block_leaves_its_own_entry_alone():
    # 40 of 64 tokens: token t of the last block meets key 63 - t of block j; of the block itself only the keys 24 .. 39 exist
    w = wl.small("ad_inf", seqlens=(64 * 5 + 40,), hq=2, hkv=1, block=64, permille=200, seed=3)
    data = wl.make_qkv(w)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    plan = StemPlan.from_workload(w, score_mode=1)
    nb = 6
    rows = []
    for bad in (False, True):
        if bad:
            q[5 * 64 + 5, 0] = float("inf")
        M = torch.full((2, plan.info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
        binding.stem_score(plan, q, k, v, M)
        assert binding.stem_check_status(plan)[0] == 0
        rows.append(M.cpu().numpy()[:, -nb:])
    assert not np.isfinite(rows[1][0, :nb - 1]).any()
    assert rows[1][0, nb - 1] == rows[0][0, nb - 1] and np.isfinite(rows[0][0, nb - 1])
    assert np.array_equal(rows[1][1], rows[0][1])
    plan.close()


@pytest.mark.parametrize("block,seqlens,hq,hkv", [
    (64, (64 * 385, 64 * 130 + 7, 64 * 128), 4, 2),   # a sequence summed at once, one in three parts, one in eight; two heads a tile
    (64, (64 * 384 + 1, 64 * 3), 3, 1),               # just above the limit with the last block, and tiny; an odd group
    (128, (128 * 129, 128 * 128 + 100), 6, 1),        # one block above 128; two heads a tile
])
def test_metric_of_sequences_summed_in_parts(block, seqlens, hq, hkv):
    w = wl.small("ad_parts", seqlens=seqlens, hq=hq, hkv=hkv, block=block, permille=100, seed=sum(seqlens))
    data = wl.make_qkv(w)
    M_ref, _ = so.score_antidiag(data["q"], data["k"], data["v"], data["cu_seqlens"], oracle_params(w))
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])

    def metric(plan, q, k, v):
        M = torch.full((hq, plan.info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
        binding.stem_score(plan, q, k, v, M)
        assert binding.stem_check_status(plan)[0] == 0
        plan.close()
        return M.cpu().numpy()

    M_g = metric(StemPlan.from_workload(w, score_mode=1), q, k, v)
    defined = ~np.isnan(M_ref)
    assert np.array_equal(np.isnan(M_g), ~defined)
    assert np.all(np.abs(M_g[defined] - M_ref[defined]) <= METRIC_ABS + METRIC_REL * np.abs(M_ref[defined]))
    # each sequence alone has the same values: the parts follow from its own length
    tok = off = 0
    for n in seqlens:
        nb = (n + block - 1) // block
        one = wl.small("ad_one", seqlens=(n,), hq=hq, hkv=hkv, block=block, permille=100)
        alone = metric(StemPlan.from_workload(one, score_mode=1), q[tok:tok + n], k[tok:tok + n], v[tok:tok + n])
        assert np.array_equal(alone, M_g[:, off:off + nb * nb], equal_nan=True)
        tok += n
        off += nb * nb


@pytest.mark.parametrize("block,seqlens,hq,hkv", [
    (128, (131072, 1500), 32, 8),              # a sequence that is summed at once beside one of 12 blocks in eight parts
    (64, (131072, 64 * 100), 64, 8),
    (64, (64 * 300, 64 * 1000 + 1, 70), 4, 2),  # three parts, at once, eight parts
])
def test_a_batch_needs_no_more_memory_than_its_sequences_alone(block, seqlens, hq, hkv):
    def bytes_of(lens):
        plan = StemPlan.from_workload(wl.small("ad_ws", seqlens=lens, hq=hq, hkv=hkv, block=block, permille=50), score_mode=1)
        info = plan.info
        plan.close()
        return info.workspace_bytes, info.total_q_blocks * info.k_max * hq * 4

    # (there is room for lists as long as the longest in every row)
    total, lists = bytes_of(seqlens)
    alone = [bytes_of((n,)) for n in seqlens]
    assert total - lists <= sum(n - l for n, l in alone)


@pytest.mark.parametrize("tokens,sums", [
    (128 * 390, 0),                                                # more than 384 blocks: no sums over parts
    (128 * 200 + 1, 3 * (128 * 128 + 96 * 128 + 96 * 96)),         # 200 full blocks: 72 rows and columns beyond the first 128
    (1500, 8 * 32 * 32),                                           # 11 full blocks
    (100, 0),                                                      # no full block
])
def test_the_workspace_has_no_pooled_vectors(tokens, sums):
    # status words, MV, bit planes of the metric, the sums over parts of full rows and columns (rounded up to 32), lists
    hq, hkv, nb = 6, 2, (tokens + 127) // 128
    plan = StemPlan.from_workload(wl.small("ad_ws", seqlens=(tokens,), hq=hq, hkv=hkv, block=128, permille=50), score_mode=1)
    sizes = (32, hkv * nb * 4, hq * nb * ((nb + 31) // 32 * 32) * 4, hq * sums * 4, hq * nb * plan.info.k_max * 4, hq * nb * 4)
    assert plan.info.workspace_bytes == sum((n + 255) // 256 * 256 for n in sizes)
    plan.close()


@pytest.mark.parametrize("seqlens", [(64 * 700 + 5,), (64 * 200,), (64 * 400, 64 * 90 + 60)])
def test_heads_in_pairs_and_alone_have_the_same_metric(seqlens):
    # 32 heads fill the SMs with two to a CTA, the four of one kv head do not
    hq, hkv, n = 32, 8, sum(seqlens)
    gen = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn((n, h, 128), generator=gen, device="cuda").to(torch.bfloat16) for h in (hq, hkv, hkv))

    def metric(heads, kv_heads, q, k, v):
        plan = StemPlan(seqlens, heads, kv_heads, block=64, budget_permille=50, score_mode=1)
        M = torch.full((heads, plan.info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
        idx = torch.full((heads, plan.info.total_q_blocks, plan.info.k_max), -7, dtype=torch.int32, device="cuda")
        cnt = torch.full((heads, plan.info.total_q_blocks), -7, dtype=torch.int32, device="cuda")
        binding.stem_score(plan, q, k, v, M)
        binding.stem_score_select(plan, q, k, v, idx, cnt)
        assert binding.stem_check_status(plan)[0] == 0
        plan.close()
        return M, idx, cnt

    M, idx, cnt = metric(hq, hkv, q, k, v)
    for kvh in (0, 5):
        rows = slice(4 * kvh, 4 * kvh + 4)
        one = metric(4, 1, q[:, rows].contiguous(), k[:, kvh:kvh + 1].contiguous(), v[:, kvh:kvh + 1].contiguous())
        assert torch.equal(one[0].nan_to_num(7e30), M[rows].nan_to_num(7e30))
        assert torch.equal(one[1], idx[rows]) and torch.equal(one[2], cnt[rows])


def _lists_of(plan, q, k, v):
    info = plan.info
    idx = torch.full((plan.num_q_heads, info.total_q_blocks, info.k_max), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((plan.num_q_heads, info.total_q_blocks), -7, dtype=torch.int32, device="cuda")
    binding.stem_score_select(plan, q, k, v, idx, cnt)
    assert binding.stem_check_status(plan)[0] == 0
    return idx.cpu().numpy(), cnt.cpu().numpy()


@pytest.mark.parametrize("block,seqlens,hq,hkv", [
    (64, (64 * 385, 64 * 130 + 7, 64 * 128), 4, 2),   # bit planes of the contraction itself and of the sums in three and eight parts
    (64, (64 * 400 + 9, 64 * 200), 3, 1),             # the same with an odd group
    (128, (128 * 390, 128 * 20 + 100), 2, 1),
    (128, (128 * 386 + 1,), 3, 3),
])
def test_fused_lists_are_those_of_the_metric(block, seqlens, hq, hkv):
    w = wl.small("ad_planes", seqlens=seqlens, hq=hq, hkv=hkv, block=block, permille=100, seed=sum(seqlens))
    data = wl.make_qkv(w)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    plan = StemPlan.from_workload(w, score_mode=1)
    info = plan.info
    idx, cnt = _lists_of(plan, q, k, v)
    M = torch.full((hq, info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
    binding.stem_score(plan, q, k, v, M)
    idx_m = torch.full((hq, info.total_q_blocks, info.k_max), -7, dtype=torch.int32, device="cuda")
    cnt_m = torch.full((hq, info.total_q_blocks), -7, dtype=torch.int32, device="cuda")
    binding.stem_select(plan, M, idx_m, cnt_m)
    assert binding.stem_check_status(plan)[0] == 0
    assert np.array_equal(idx, idx_m.cpu().numpy()) and np.array_equal(cnt, cnt_m.cpu().numpy())
    plan.close()


@pytest.mark.parametrize("block,n,q_start,hq,hkv", [
    (128, 128 * 200 + 50, 128 * 70, 4, 2),    # three parts; the chunk's tiles start inside the sequence's
    (64, 64 * 100, 64 * 33, 4, 2),            # eight parts
    (64, 64 * 390 + 5, 64 * 130, 2, 1),       # at once
    (128, 128 * 3 + 60, 128 * 3, 3, 1),       # the chunk is the partial block alone
])
def test_lists_of_a_chunk_are_those_of_the_whole_sequence(block, n, q_start, hq, hkv):
    w = wl.small("ad_chunk", seqlens=(n,), hq=hq, hkv=hkv, block=block, permille=100, seed=n)
    data = wl.make_qkv(w)
    q, k, v = to_dev(data["q"]), to_dev(data["k"]), to_dev(data["v"])
    whole = StemPlan.from_workload(w, score_mode=1)
    idx, cnt = _lists_of(whole, q, k, v)
    # the first chunk sees the tokens before q_start alone, the second one all keys
    parts = [(q[:q_start], q_start, 0), (q[q_start:], n, q_start)]
    row = 0
    for q_chunk, kv_len, start in parts:
        wc = wl.small("ad_chunk", seqlens=(kv_len,), hq=hq, hkv=hkv, block=block, permille=100)
        plan = StemPlan.from_workload(wc, score_mode=1, q_starts=[start], total_lens=[n])
        idx_c, cnt_c = _lists_of(plan, q_chunk, k[:kv_len], v[:kv_len])
        rows = slice(row, row + plan.info.total_q_blocks)
        assert np.array_equal(cnt_c, cnt[:, rows])
        width = plan.info.k_max
        assert np.array_equal(idx_c, idx[:, rows, :width]) and (idx[:, rows, width:] == -1).all()
        row = rows.stop
        plan.close()
    assert row == whole.info.total_q_blocks
    whole.close()


@pytest.mark.parametrize("block,seqlens,hq,hkv", [
    (64, (64 * 100,) * 7 + (64 * 100 + 33,), 32, 8),      # eight parts, two heads to a CTA
    (64, (64 * 250, 64 * 300 + 1, 64 * 200, 64 * 384), 28, 4),  # three parts, an odd group
    (128, (128 * 100 + 100, 128 * 260, 128 * 390), 32, 8),  # all three kinds of sums
])
def test_parts_of_a_batch_that_fills_the_sms(block, seqlens, hq, hkv):
    # A CTA adds up the parts of a tile where the batch fills the SMs (no room for sums then): the bits of each sequence alone.
    n = sum(seqlens)
    gen = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn((n, h, 128), generator=gen, device="cuda").to(torch.bfloat16) for h in (hq, hkv, hkv))

    def scores(lens, q, k, v):
        plan = StemPlan(lens, hq, hkv, block=block, budget_permille=50, score_mode=1)
        M = torch.full((hq, plan.info.metric_elems), float("nan"), dtype=torch.float32, device="cuda")
        binding.stem_score(plan, q, k, v, M)
        idx, cnt = _lists_of(plan, q, k, v)
        plan.close()
        return M.nan_to_num(7e30), idx, cnt, plan.info

    M, idx, cnt, info = scores(seqlens, q, k, v)
    tok = off = row = 0
    for length in seqlens:
        part = slice(tok, tok + length)
        M1, idx1, cnt1, info1 = scores((length,), q[part], k[part], v[part])
        rows = slice(row, row + info1.total_q_blocks)
        assert torch.equal(M1, M[:, off:off + info1.metric_elems])
        assert np.array_equal(idx1, idx[:, rows, :info1.k_max]) and (idx[:, rows, info1.k_max:] == -1).all()
        assert np.array_equal(cnt1, cnt[:, rows])
        tok, off, row = part.stop, off + info1.metric_elems, rows.stop
