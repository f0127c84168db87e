"""Prefill attention items of one and of two Q tiles: the same bits whichever the budget brings about, and two-tile items
(more than one round of single tiles on the device) against the oracle, causal and bidirectional."""
import dataclasses

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import bits_to_f32, make_stage, run_step
from tests.helpers import make_case, rel_err

TOL = 2e-2        # max|err| / RMS, the rule of every parity test (16-bit operands)

# name: dims, new tokens, cached tokens, budgets, whether one-tile items occur among them.  Query heads per KV head 1, 7, 8
# and 16 (tiles of 128, 16, 16 and 8 tokens); short and absent second tiles; cached context; decode rows beside chunks.
CASES = {
    "g1": (wl.StageDims(2, 256, 4, 4, 64, 256), [256, 130, 129], [0, 40, 0], (148, 12, 3, 1), True),
    "g7": (wl.StageDims(2, 256, 14, 2, 64, 256), [100, 37], [0, 70], (148, 13, 1), True),
    "g8_decode": (wl.StageDims(2, 256, 16, 2, 64, 256), [200, 17, 1, 1], [33, 0, 300, 5], (148, 24, 16, 2), True),
    "g16_dh128": (wl.StageDims(2, 256, 16, 1, 128, 256), [61, 9, 8], [5, 100, 0], (148, 7, 1), True),
    "g1_many": (wl.StageDims(1, 256, 32, 32, 64, 256), [300, 340], [0, 20], (148, 37), False),
    "g7_many": (wl.StageDims(1, 256, 28, 4, 64, 256), [601], [50], (148, 37), False),
    "g8_many": (wl.StageDims(1, 256, 32, 4, 64, 256), [330, 290], [0, 9], (148, 37), False),
    "g16_many": (wl.StageDims(1, 256, 32, 2, 64, 256), [610], [0], (148, 37), False),
}


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BIDIRECTIONAL])
@pytest.mark.parametrize("name", sorted(CASES))
def test_items_of_one_and_of_two_tiles_give_the_same_bits(name, flags):
    dims, q_len, ctx_len, budgets, both = CASES[name]
    batch = wl.BatchSpec(list(q_len), list(ctx_len))
    case = make_case(dims, batch, seed=23, kv_fill=True)
    cfg = dataclasses.replace(case.cfg, bidirectional=bool(flags))
    y_ref = Oracle("f32").step(cfg, case.weights, case.kv_pool.copy(), batch.q_len, batch.ctx_len, case.block_tables, case.x)
    G = dims.n_q_heads // dims.n_kv_heads
    mt = max(8, (128 // G) & ~7)
    singles = sum(-(-n // mt) for n in q_len if n > 1) * dims.n_kv_heads
    st = make_stage(case, flags=flags)
    try:
        first, forms = None, set()
        x = case.x_t.to(st.device).contiguous()
        for budget in budgets:
            b = st.make_batch(batch.q_len, batch.ctx_len, case.block_tables, x, x.float())
            forms.add(B.hs_stage_plan_shares(st.handle, b, budget)[0] == singles)
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        assert forms == ({True, False} if both else {False})
        err = rel_err(first[0], y_ref)
        print(f"prefill items, {name}, flags {flags}: max|err|/RMS = {err:.2e}")
        assert err <= TOL
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["g1", "g7", "g16_dh128"])
def test_a_row_that_is_not_finite_spreads_alike_in_both_forms(name):
    dims, q_len, ctx_len, budgets, _ = CASES[name]
    batch = wl.BatchSpec(list(q_len), list(ctx_len))
    case = make_case(dims, batch, seed=29, kv_fill=True)
    case.x_t[q_len[0] // 2 + 3] = float("nan")
    st = make_stage(case)
    try:
        outs = []
        for budget in budgets:
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            y, pool = run_step(st, case, budget, expect_saturation=True)
            outs.append((y, bits_to_f32(pool)))
        assert np.isnan(outs[0][0]).any() and not np.isnan(outs[0][0]).all()
        for y, pool in outs[1:]:
            assert np.array_equal(y, outs[0][0], equal_nan=True) and np.array_equal(pool, outs[0][1], equal_nan=True)
    finally:
        st.close()
