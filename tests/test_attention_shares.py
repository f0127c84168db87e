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
