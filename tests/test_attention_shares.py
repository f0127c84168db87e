"""How the planner shares the SMs out between the two attention kernels of a step with both kinds of work."""
import numpy as np
import pytest

from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl


def _shares(dims, q_len, ctx_len, budgets):
    batch = wl.BatchSpec(list(q_len), list(ctx_len))
    mpps = max(-(-t // 16) for t in batch.total_len())
    cfg = B.make_config(dims, wl.pages_needed(batch) + 4, batch.n_tokens, batch.n_seqs, mpps, max(batch.total_len()), device=-1)
    stage = B.hs_stage_create(cfg, None, 0, 0)
    try:
        tables = np.full((batch.n_seqs, mpps), -1, dtype=np.int32)
        for s, t in enumerate(batch.total_len()):
            pages = B.hs_kv_alloc(stage, s, t, mpps)
            tables[s, : len(pages)] = pages
        b = B.Batch(batch.q_len, batch.ctx_len, tables, 16, 16)
        return {n: B.hs_stage_plan_shares(stage, b, n) for n in budgets}
    finally:
        B.hs_stage_destroy(stage)


def test_a_chunk_and_a_full_decode_batch_are_balanced():
    """The prefill kernel pays per item as well as per block: it gets about half of the device, not two fifths."""
    for n, (items, sms) in _shares(wl.DIMS["c3_7b"], [2048] + [1] * 64, [0] + [512 + 56 * i for i in range(64)], (148, 120)).items():
        assert items == 256 and 0.42 * n <= sms <= 0.55 * n, (n, sms)


@pytest.mark.parametrize("rows,longest", [(32, 2000), (32, 1000), (20, 1500), (8, 700)])
def test_the_decode_kernel_gets_whole_rounds_of_its_blocks(rows, longest):
    """Group mode: rows x KV heads blocks; with one SM fewer they would need a round more."""
    dims = wl.DIMS["c2_shared"]
    groups = rows * dims.n_kv_heads
    for n, (items, sms) in _shares(dims, [700] * 8 + [1] * rows, [0] * 8 + [longest - 3 * i for i in range(rows)], (148, 112, 74)).items():
        assert items == 8 * 22 * dims.n_kv_heads and 4 <= sms <= n - 4
        assert sms == 4 or -(-groups // (sms - 1)) > -(-groups // sms), (n, sms)


# Batches on items of single warps (more than 148 groups, or a sequence beyond 4096 keys) -> what the prefill kernel takes
# beside them, of its time alone.
@pytest.mark.parametrize("name,q,c,dec,beside", [
    ("c2_shared", [300] * 2, [0] * 2, [900] * 7 + [4200], 1.0), ("c2_shared", [700] * 8, [0] * 8, [1500] * 80, 1.0),
    ("c3_7b", [394], [1000], [900] * 6 + [4200], 1.0), ("c3_7b", [1024], [0], [2500] * 64, 1.3), ("c3_7b", [2048], [0], [1999] * 40, 1.3)])
def test_the_shares_of_a_batch_without_groups_follow_the_bytes_it_streams(name, q, c, dec, beside):
    """The balance written out: 9 + beside * (5.6 us an item + 1.13 us a block) against 12 us + bytes at 42 GB/s per SM, at most
    5.5 TB/s; the smallest share of the least larger time."""
    dims = wl.DIMS[name]
    tokens = 2 * max(8, (128 // (dims.n_q_heads // dims.n_kv_heads)) & ~7)
    blocks = [-(-(x + min(t + tokens, n)) // 64) for n, x in zip(q, c) for t in range(0, n, tokens)]
    n_items, n_blocks, longest = len(blocks) * dims.n_kv_heads, sum(blocks) * dims.n_kv_heads, max(blocks)
    kv = sum(k + 1 for k in dec) * 4 * dims.kv_dim
    for n, (items, sms) in _shares(dims, q + [1] * len(dec), c + dec, (148, 112, 96)).items():
        if items != n_items or sms == 0:                # one-tile items, or the two in turn
            continue
        def us(b):
            return max(9 + beside * max(5.6 + 1.13 * longest, (5.6 * n_items + 1.13 * n_blocks) / (n - b)), 12 + kv / min(5.5e6, 42e3 * b))
        assert us(sms) <= min(us(b) for b in range(4, n - 3)) + 1e-6, (n, sms)
