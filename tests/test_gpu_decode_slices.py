"""Decode attention of small batches: groups cut into slices of several blocks, the last of which merges them.  Against the
oracle and bit for bit across budgets; the slices themselves on the CPU."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

# name: dims, cached tokens.  One long sequence; the longest that is taken; lengths around a page and a slice's end, sequences
# of one key beside long ones; few KV heads and many; both head sizes.
CASES = {
    "one_long": (wl.StageDims(1, 256, 8, 2, 64, 512), [3001]),
    "longest": (wl.StageDims(1, 256, 4, 4, 128, 256), [4095, 2000]),
    "ragged": (wl.StageDims(1, 256, 4, 2, 128, 256), [0, 15, 16, 1023, 1024, 1025, 3777]),
    "nine": (wl.StageDims(2, 256, 4, 2, 64, 256), [3723, 3612, 3450, 3578, 761, 3419, 3888, 1449, 1119]),
}


def _plan(dims, ctx_len, q_len=None):
    batch = wl.BatchSpec([1] * len(ctx_len) if q_len is None else list(q_len), list(ctx_len))
    mpps = max(-(-t // 16) for t in batch.total_len())
    cfg = B.make_config(dims, wl.pages_needed(batch) + 4, batch.n_tokens, batch.n_seqs, mpps, max(batch.total_len()), device=-1)
    stage = B.hs_stage_create(cfg, None, 0, 0)
    try:
        tables = np.full((batch.n_seqs, mpps), -1, dtype=np.int32)
        for s, t in enumerate(batch.total_len()):
            pages = B.hs_kv_alloc(stage, s, t, mpps)
            tables[s, : len(pages)] = pages
        return B.hs_stage_plan_attention(stage, B.Batch(batch.q_len, batch.ctx_len, tables, 16, 16))
    finally:
        B.hs_stage_destroy(stage)


@pytest.mark.parametrize("name", sorted(CASES))
def test_slices_cover_every_key_once_and_have_a_block_each(name):
    dims, ctx_len = CASES[name]
    items, group, _ = _plan(dims, ctx_len)
    assert group and len(items) % 8 == 0 and len(items) // 8 <= 148
    cover = {(s, h): np.zeros(c + 1, dtype=np.int32) for s, c in enumerate(ctx_len) for h in range(dims.n_kv_heads)}
    slots, several = [], 0
    for i in range(0, len(items), 8):
        blk = items[i: i + 8]
        seq, hk, first, n, idx = int(blk[0][4]), int(blk[0][1]), int(blk[0][6]), int(blk[0][7]) & 0xffff, int(blk[0][7]) >> 16
        assert len({(int(r[4]), int(r[1]), int(r[6]), int(r[7])) for r in blk}) == 1 and 0 <= idx < n
        for w, r in enumerate(blk):
            assert int(r[2]) <= int(r[3]) and int(r[3]) - int(r[2]) <= 512 and (int(r[2]) % 16 == 0 or r[2] == r[3])
            assert w == 0 or int(blk[w - 1][3]) == int(r[2])
            cover[(seq, hk)][int(r[2]): int(r[3])] += 1
        slots.append(first + idx)
        several += n > 1
    assert all(np.all(c == 1) for c in cover.values()) and sorted(slots) == list(range(len(items) // 8))
    assert several > 0


def test_short_batches_and_batches_with_prefill_keep_one_slice_per_group():
    dims = wl.DIMS["c4_talker"]
    items, group, _ = _plan(dims, [100, 50])
    assert group and len(items) == 8 * 2 * dims.n_kv_heads
    for name in ("one_long", "nine"):                  # cut alone (above), whole beside a chunk
        dims, ctx_len = CASES[name]
        items, group, chunk = _plan(dims, [0] + ctx_len, [40] + [1] * len(ctx_len))
        assert group and len(chunk) and len(items) == 8 * len(ctx_len) * dims.n_kv_heads
        assert all(int(r[7]) == 1 for r in items)


def test_sequences_beyond_4096_keys_are_items_of_single_warps():
    """A warp keeps a page id per lane, so eight warps hold 256 pages: the longest slice of a group that is not cut."""
    dims = wl.DIMS["c3_7b"]
    for ctx, want in ((4094, True), (4095, True), (4096, False), (4097, False)):
        items, group, _ = _plan(dims, [ctx, 700])
        keys = sum(int(r[3]) - int(r[2]) for r in items if int(r[4]) == 0)
        assert group == want and keys == dims.n_kv_heads * (ctx + 1)
        assert all(int(r[3]) - int(r[2]) <= 512 for r in items)


# Batches (stage, rows, cached tokens from .. to) that measured faster with one slice per group, over the budgets or on most of
# them, and such that measured faster cut, at every budget: slices of the longest group, at least .. at most.
@pytest.mark.parametrize("name,rows,lo,hi,least,most", [
    ("c2_shared", 32, 256, 2048, 1, 1), ("c2_shared", 16, 256, 2048, 1, 2), ("c2_shared", 8, 256, 2048, 2, 3), ("c3_7b", 14, 512, 4096, 1, 2),
    ("c4_talker", 4, 128, 1024, 1, 1), ("c4_talker", 11, 128, 1500, 1, 1), ("c3_7b", 1, 4000, 4001, 5, 8), ("c3_7b", 3, 512, 4096, 3, 6),
    ("c2_shared", 1, 1500, 1501, 4, 8)])
def test_groups_are_cut_where_that_measured_faster(name, rows, lo, hi, least, most):
    ctx_len = np.random.default_rng(rows * 1000 + hi).integers(lo, hi, rows).tolist()
    items, group, _ = _plan(wl.DIMS[name], ctx_len)
    assert group and least <= max(int(r[7]) & 0xffff for r in items) <= most


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BF16_ACTIVATIONS])
@pytest.mark.parametrize("name", sorted(CASES))
def test_slices_match_the_oracle_at_every_budget(name, flags):
    dims, ctx_len = CASES[name]
    q_len = [1] * len(ctx_len)
    case = make_case(dims, wl.BatchSpec(q_len, list(ctx_len)), seed=61, kv_fill=True)
    y_ref = Oracle("f32").step(case.cfg, case.weights, case.kv_pool.copy(), q_len, ctx_len, case.block_tables, case.x)
    st = make_stage(case, flags=flags)
    try:
        first = None
        for budget in (148, 60, 7, 1):
            for _ in range(2):                         # (the counters of a launch are left ready for the next)
                st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
                out = run_step(st, case, budget)
                first = out if first is None else first
                assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        assert rel_err(first[0], y_ref) <= 2e-2        # the rule of every parity test (16-bit operands)
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1, -1])
def test_saturated_outputs_of_merged_slices_are_counted_once(scale):
    """Values beyond fp16's range in the cache: every element of a long sequence's attention output is clamped and counted by the
    block that merges the group's slices, none of a sequence whose values are ordinary."""
    dims, ctx_len = wl.StageDims(1, 256, 8, 2, 64, 512), [3001, 2500, 40]
    items, group, _ = _plan(dims, ctx_len)
    assert group and max(int(r[7]) & 0xffff for r in items) > 1
    case = make_case(dims, wl.BatchSpec([1] * 3, ctx_len), seed=67, kv_fill=True)
    pool = wl.bits_to_bf16_tensor(case.kv_pool).view(wl.kv_pool_shape(dims, case.cfg.num_pages))
    for s in (0, 1):
        for page in case.block_tables[s][: -(-(ctx_len[s] + 1) // 16)]:
            pool[0, 1, int(page)] = scale * 1.0e5
    st = make_stage(case, weights=[dict(lw, w_o=lw["w_o"] * 0) for lw in case.weights_t])      # (nothing behind it leaves the range)
    try:
        for i, budget in enumerate((148, 60, 1)):
            st.kv_pool.copy_(pool.reshape(-1))
            run_step(st, case, budget, expect_saturation=True)
            assert st.saturation_count() == (i + 1) * 2 * dims.q_dim, budget
            assert bool((st.debug_tensor("o")[:2].float() == scale * 65504).all())
    finally:
        st.close()
