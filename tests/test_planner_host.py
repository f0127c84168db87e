"""CPU-only checks of the planner's attention work lists and of the skewed K split (host logic behind the kernels'
work decomposition): every key of every decode sequence is covered exactly once per KV head, the queue order is
longest first, partial slots follow key order, group mode is chosen for small batches only; prefill items cover every
new token once per KV head; the K splits tile the K range without gaps or empty splits."""
import numpy as np
import pytest

from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl


def _stage_and_batch(dims, q_len, ctx_len):
    batch = wl.BatchSpec(list(q_len), list(ctx_len))
    num_pages = wl.pages_needed(batch) + 4
    mpps = max(-(-t // 16) for t in batch.total_len())
    cfg = B.make_config(dims, num_pages, batch.n_tokens, batch.n_seqs, mpps, max(batch.total_len()), device=-1)
    stage = B.hs_stage_create(cfg, None, 0, 0)
    tables = np.full((batch.n_seqs, mpps), -1, dtype=np.int32)
    for s, t in enumerate(batch.total_len()):
        pages = B.hs_kv_alloc(stage, s, t, mpps)
        tables[s, : len(pages)] = pages
    return stage, B.Batch(batch.q_len, batch.ctx_len, tables, 16, 16), batch


def _check_decode(dims, batch, items, group):
    dec_rows = [(s, c) for s, (q, c) in enumerate(zip(batch.q_len, batch.ctx_len)) if q == 1]
    cover = {(s, hk): np.zeros(c + 1, dtype=np.int32) for s, c in dec_rows for hk in range(dims.n_kv_heads)}
    for it in items:
        drow, hk, k0, k1, seq, tok = (int(v) for v in it[:6])
        assert dec_rows[drow][0] == seq and 0 <= hk < dims.n_kv_heads
        assert 0 <= k0 <= k1 <= dec_rows[drow][1] + 1 and (k0 % 16 == 0 or k0 == k1) and k1 - k0 <= 512
        assert group or k1 > k0
        cover[(seq, hk)][k0:k1] += 1
    for c in cover.values():
        assert np.all(c == 1)                      # every key exactly once per KV head
    if group:
        assert len(items) == 8 * len(cover)
        for g in range(len(cover)):                # a group's eight slices are consecutive and in key order
            blk = items[8 * g: 8 * g + 8]
            assert len({(int(r[4]), int(r[1])) for r in blk}) == 1
            assert all(int(blk[w][3]) == int(blk[w + 1][2]) for w in range(7)) and int(blk[0][2]) == 0
    else:
        keys = items[:, 3] - items[:, 2]
        assert np.all(keys[:-1] >= keys[1:])       # the queue hands the items out longest first
        slots = {}
        for it in items:                           # partial slots of a group: consecutive, in key order
            first, splits, idx = int(it[6]), int(it[7]) & 0xffff, int(it[7]) >> 16
            slots.setdefault((int(it[4]), int(it[1])), []).append((int(it[2]), first + idx, first, splits))
        used = []
        for lst in slots.values():
            lst.sort()
            assert len({(f, n) for _, _, f, n in lst}) == 1 and lst[0][3] == len(lst)
            assert [s for _, s, _, _ in lst] == list(range(lst[0][2], lst[0][2] + len(lst)))
            used += [s for _, s, _, _ in lst]
        assert sorted(used) == list(range(len(items)))     # no two groups share a slot


CASES = {
    "talker": ("c4_talker", None),
    "c2": ("c2_shared", None),
    "c3": ("c3_7b", None),
    "one_long": ("c3_7b", ([1], [16000])),
    "many_short": ("c4_talker", ([1] * 200, [3 + 7 * i for i in range(200)])),
    "mixed_runs": ("c3_7b", ([1] * 64 + [300], [127, 128, 129, 255, 256, 257, 383, 384, 385, 511, 512, 513] * 5 + [4000] * 4 + [0])),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_attention_work_lists_cover_every_key_and_token_once(name):
    wname, custom = CASES[name]
    dims = wl.DIMS[wname]
    if custom is None:
        b0 = wl.make_batch(wname, {"c4_talker": 3, "c2_shared": 1, "c3_7b": 2}[wname])
        q_len, ctx_len = b0.q_len, b0.ctx_len
    else:
        q_len, ctx_len = custom
    stage, batch_c, batch = _stage_and_batch(dims, q_len, ctx_len)
    try:
        dec, group, pre = B.hs_stage_plan_attention(stage, batch_c)
        _check_decode(dims, batch, dec, group)
        # group mode only where every group can have a block (148 SMs without a device) and no slice exceeds 32 pages
        n_groups = sum(1 for q in batch.q_len if q == 1) * dims.n_kv_heads
        if group:
            assert n_groups <= 148 and max(c + 1 for q, c in zip(batch.q_len, batch.ctx_len) if q == 1) <= 4096
        if name in ("c3", "one_long", "many_short"):
            assert not group
        if name in ("talker", "c2"):
            assert group
        # prefill items: every new token of a prefill sequence once per KV head, at most two tiles, longest first
        G = dims.n_q_heads // dims.n_kv_heads
        mt = max(8, (128 // G) & ~7)
        seen = {(s, hk): np.zeros(q, dtype=np.int32) for s, q in enumerate(batch.q_len) if q > 1 for hk in range(dims.n_kv_heads)}
        tok0 = np.concatenate([[0], np.cumsum(batch.q_len)[:-1]])
        for it in pre:
            s, hk, t0, nt, ctx, row0, qn = (int(v) for v in it[:7])
            assert 1 <= nt <= 2 * mt and ctx == batch.ctx_len[s] and qn == batch.q_len[s] and row0 == tok0[s]
            seen[(s, hk)][t0: t0 + nt] += 1
        for c in seen.values():
            assert np.all(c == 1)
        cost = [int(it[4]) + int(it[2]) + int(it[3]) for it in pre]
        assert cost == sorted(cost, reverse=True)
    finally:
        B.hs_stage_destroy(stage)


@pytest.mark.parametrize("name,ctx,keys", [("c3_7b", [4096], 256), ("c3_7b", [16000], 256), ("c3_7b", [8000, 7963], 256), ("c2_shared", [6000], 256),
                                           ("c4_talker", [7999, 7000, 6000, 5000], 256)])
def test_items_of_long_sequences_are_no_finer_than_one_warp_can_merge(name, ctx, keys):
    """A stage of the size of the batch: room for slices of small batches is not taken for items of single warps."""
    stage, batch_c, batch = _stage_and_batch(wl.DIMS[name], [1] * len(ctx), ctx)
    try:
        items, group, _ = B.hs_stage_plan_attention(stage, batch_c)
        _check_decode(wl.DIMS[name], batch, items, group)
        assert not group and int((items[:, 3] - items[:, 2]).max()) == keys
    finally:
        B.hs_stage_destroy(stage)


def test_k_splits_tile_the_k_range():
    for k_blocks in list(range(1, 70)) + [112, 148, 296, 1000]:
        for ks in range(1, 9):
            b = [B.hs_op_gemm_split_begin(k_blocks, ks, i) for i in range(ks + 1)]
            assert b[0] == 0 and b[-1] == k_blocks and all(x <= y for x, y in zip(b, b[1:]))
            lens = [y - x for x, y in zip(b, b[1:])]
            if k_blocks >= 10 * ks * (ks - 1) // 2 + 10 * ks and ks > 1:
                # long enough for the skew: each split ten blocks longer than the one before, the last takes the remainder
                assert all(lens[i + 1] - lens[i] == 10 for i in range(ks - 2)) and lens[-1] - lens[-2] >= 10
                assert min(lens) >= 10
            else:
                assert max(lens) - min(l for l in lens if l > 0) <= max(lens)      # equal runs (the tail may be short or empty)
                assert lens == sorted(lens, reverse=True)
    assert B.hs_op_gemm_split_begin(0, 1, 0) == -1 and B.hs_op_gemm_split_begin(10, 0, 0) == -1
    assert B.hs_op_gemm_split_begin(10, 2, 3) == -1
    # the down-projection of a 64-row step at 7B dimensions: 296 K blocks in 5 splits
    assert [B.hs_op_gemm_split_begin(296, 5, i) for i in range(6)] == [0, 39, 88, 147, 216, 296]


# Residual GEMMs (rows, width, contraction length) for which partial sums measured slower than the GEMM without them: few rows
# on the weight-streaming kernel, many rows whose partial sums cost more traffic than the splits save, rows that fill pairs
# of SMs; and such for which they measured clearly faster.
@pytest.mark.parametrize("M,N,K", [(17, 1024, 1024), (17, 1024, 2816), (32, 1024, 2816), (24, 2048, 2048),
                                   (1024, 1024, 1024), (1280, 1024, 2816), (1536, 1024, 2816), (2048, 1024, 2816),
                                   (3072, 1024, 2816), (1280, 2048, 5632), (3000, 2048, 5632), (600, 3584, 18944),
                                   (1450, 3584, 18944), (2112, 3584, 18944)])
def test_partial_sums_are_not_taken_where_they_are_slower(M, N, K):
    assert B.hs_op_gemm_part_splits(M, N, K) == 0


@pytest.mark.parametrize("M,N,K", [(17, 3584, 18944), (29, 3584, 3584), (64, 3584, 18944), (64, 2048, 5632), (65, 1024, 2816),
                                   (128, 2048, 2048),
                                   (256, 1024, 2816), (1024, 1024, 2816), (401, 3584, 18944), (512, 3584, 18944)])
def test_partial_sums_are_taken_where_they_are_faster(M, N, K):
    assert 2 <= B.hs_op_gemm_part_splits(M, N, K) <= 10


def test_partial_sums_at_the_edges_of_their_range():
    assert B.hs_op_gemm_part_splits(64, 16392, 4096) == 0            # wider than the norm kernel that adds them
    assert B.hs_op_gemm_part_splits(9, 3584, 3584) == 0              # the small-step fold
    assert B.hs_op_gemm_part_splits(0, 1024, 1024) == -1 and B.hs_op_gemm_part_splits(8, 1020, 1024) == -1
    assert B.hs_op_gemm_part_splits(8, 1024, 40) == -1


# Gate/up projections (rows, width, contraction length, SMs) -> the tile width whose step measured fastest, or within a
# hundredth of it.
@pytest.mark.parametrize("M,N,K,sms,widths", [
    (5, 18944, 3584, 24, (112, 128)), (24, 18944, 3584, 28, (112, 128)), (5, 18944, 3584, 64, (112,)), (29, 18944, 3584, 96, (96, 112)),
    (24, 18944, 3584, 120, (80,)), (100, 18944, 3584, 130, (80,)), (5, 18944, 3584, 148, (128,)), (24, 5632, 2048, 148, (48,))])
def test_width_of_the_gate_up_tiles(M, N, K, sms, widths):
    assert B.hs_op_gate_up_width(M, N, K, sms) in widths


# Residual projections (rows, width, contraction length, SMs) -> weight rows per block whose step measured fastest: units of 16
# rows where they are one round or all that occupies the device, not five rounds of them.
@pytest.mark.parametrize("M,N,K,sms,rows", [
    (1, 3584, 18944, 52, (48,)), (2, 3584, 18944, 52, (48,)), (5, 3584, 18944, 52, (48,)), (1, 3584, 18944, 148, (32,)),
    (1, 1024, 2816, 148, (16,)), (16, 1024, 1024, 96, (16,)), (8, 1024, 2816, 52, (32,))])
def test_weight_rows_of_a_weight_streaming_block(M, N, K, sms, rows):
    assert B.hs_op_weight_streaming_rows(M, N, K, sms) in rows
    assert B.hs_op_weight_streaming_rows(65, N, K, sms) == B.hs_op_weight_streaming_rows(M, N + 8, K, sms) == -1


def test_width_of_the_gate_up_tiles_at_the_edges():
    # a further round costs what it does whatever the length of K: the shorter K, the fewer rounds are worth having
    assert B.hs_op_gate_up_width(32, 2816, 1024, 20) > 48
    rounds = [-(-2816 // B.hs_op_gate_up_width(32, 2816, k, 20)) for k in (64, 256, 1024, 4096)]
    assert rounds == sorted(rounds)
    assert B.hs_op_gate_up_width(129, 18944, 3584, 96) == 128
    assert all(B.hs_op_gate_up_width(m, n, k, s) == -1 for m, n, k, s in ((0, 1024, 64, 1), (1, 56, 64, 1), (1, 1024, 0, 1), (1, 1024, 64, 0)))
    for sms in range(1, 149):
        w = B.hs_op_gate_up_width(64, 18944, 3584, sms)
        assert w % 16 == 0 and 48 <= w <= 128


# dims, prefill chunks, cached tokens of the chunks, decode contexts -> items at budget, from the forms that measured faster
SHARES = {
    "denoise_2": ("c6_dit", [256] * 2, [0] * 2, [], {148: 64, 74: 64, 52: 32, 37: 32}),
    "denoise_4": ("c6_dit", [256] * 4, [0] * 4, [], {148: 128, 96: 64, 37: 64}),
    "denoise_5": ("c6_dit", [256] * 5, [0] * 5, [], {148: 80}),
    "chunk_100": ("c3_7b", [100], [1000], [300, 700, 1500, 2200, 2600, 2900, 999], {148: 28, 96: 28, 48: 16}),
    "chunk_394": ("c3_7b", [394], [1000], [300, 700, 1500, 2200, 2600, 2900, 999], {148: 100, 96: 52, 48: 52}),
}


@pytest.mark.parametrize("name", sorted(SHARES))
def test_prefill_items_of_one_tile_only_where_each_has_an_sm_of_the_kernels_share(name):
    wname, q, c, dec, want = SHARES[name]
    dims = wl.DIMS[wname]
    stage, batch_c, batch = _stage_and_batch(dims, q + [1] * len(dec), c + dec)
    mt = max(8, (128 // (dims.n_q_heads // dims.n_kv_heads)) & ~7)
    singles = sum(-(-n // mt) for n in q) * dims.n_kv_heads
    doubles = sum(-(-n // (2 * mt)) for n in q) * dims.n_kv_heads
    try:
        for budget in sorted({1, 2, 15, 16, 17, 147} | set(want)):
            n, sms = B.hs_stage_plan_shares(stage, batch_c, budget)
            assert n in (singles, doubles)
            assert sms == 0 or (dec and 4 <= sms <= budget - 4 and budget >= 16)
            if n == singles != doubles:
                assert n <= budget - sms
            if budget in want:
                assert n == want[budget], (budget, n)
        for budget in (0, 149):
            with pytest.raises(B.HsError):
                B.hs_stage_plan_shares(stage, batch_c, budget)
    finally:
        B.hs_stage_destroy(stage)
