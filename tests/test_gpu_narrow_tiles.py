"""Gate/up GEMM of small steps on single blocks: the width of its tiles follows the budget; the results do not."""
import numpy as np
import pytest
import torch

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from paper_2608_01785_b200.stage import Stage
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

BUDGETS = (148, 140, 120, 112, 96, 64, 48, 37, 28, 19, 1)

# More than 64 rows, so that the projection is on the tiled kernel: a full row tile and a ragged one, widths that no tile
# width divides (4648 = 96 * 48 + 40), a single tile column.
CASES = {
    "100_rows": (wl.StageDims(2, 256, 4, 2, 64, 4640), [97, 1, 2], [0, 30, 5]),
    "128_rows_ragged": (wl.StageDims(1, 264, 4, 2, 64, 4648), [128], [0]),
    "65_rows_one_tile": (wl.StageDims(1, 256, 4, 2, 64, 104), [65], [7]),
}


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BF16_ACTIVATIONS])
@pytest.mark.parametrize("name", sorted(CASES))
def test_tile_width_does_not_reach_the_output(name, flags):
    dims, q_len, ctx_len = CASES[name]
    assert len({B.hs_op_gate_up_width(sum(q_len), dims.d_ffn, dims.d_model, n) for n in BUDGETS}) > (2 if dims.d_ffn > 128 else 0)
    case = make_case(dims, wl.BatchSpec(q_len, ctx_len), seed=71, kv_fill=True)
    y_ref = Oracle("f32").step(case.cfg, case.weights, case.kv_pool.copy(), q_len, ctx_len, case.block_tables, case.x)
    st = make_stage(case, flags=flags)
    try:
        first = None
        for budget in BUDGETS:
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        assert rel_err(first[0], y_ref) <= 2e-2        # the rule of every parity test (16-bit operands)
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["100_rows", "128_rows_ragged"])
def test_saturated_values_are_counted_once_at_every_width(name):
    """Gate and up weights scaled such that some of the products leave fp16's range: a tile's last chunk of 32 columns has columns
    of the up projection behind the tile's own, which are as large and must not count."""
    dims, q_len, ctx_len = CASES[name]
    case = make_case(dims, wl.BatchSpec(q_len, ctx_len), seed=73, kv_fill=True)
    weights = [dict(lw, w_gate=lw["w_gate"] * 512, w_up=lw["w_up"] * 512) for lw in case.weights_t]
    st = make_stage(case, weights=weights)
    try:
        first, counts, before = None, [], 0
        for budget in BUDGETS:
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget, expect_saturation=True)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]), budget
            counts.append(st.saturation_count() - before)
            before += counts[-1]
        assert len(set(counts)) == 1 and counts[0] > 0
        if dims.n_layers == 1:                         # (the count is of all layers; 65504 is also what some smaller values round to)
            assert counts[0] <= int((st.debug_tensor("act")[: sum(q_len)].float().abs() == 65504).sum())
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [9, 29, 64])
def test_decode_steps_at_7b_dimensions_give_the_same_bits_at_every_width(rows):
    """Boxes of 32 and 64 activation rows; the norm folded into the neighbours (9 rows) and not."""
    dims = wl.replace(wl.DIMS["c3_7b"], n_layers=1)
    dev = torch.device("cuda:0")
    batch = wl.BatchSpec([1] * rows, [20 + i for i in range(rows)])
    total = batch.total_len()
    st = Stage(dims, wl.make_weights(dims, 3, dev, "depth_scaled"), wl.pages_needed(batch) + 2, rows, rows, max(-(-t // 16) for t in total),
               max(total), 0, 0)
    try:
        st.kv_pool_view().zero_()
        tables = st.block_table_array([st.kv_alloc(s, t) for s, t in enumerate(total)])
        x = wl.make_x(rows, dims.d_model, 3, dev)
        first = None
        for budget in BUDGETS[:-1]:
            y = torch.full((rows, dims.d_model), float("nan"), device=dev)
            st.step(st.make_batch(batch.q_len, batch.ctx_len, tables, x, y), budget)
            torch.cuda.synchronize()
            assert st.status() == 0 and st.saturation_count() == 0
            first = y if first is None else first
            assert torch.equal(y, first), budget
        assert bool(torch.isfinite(first).all())
    finally:
        st.close()
