"""Gate/up GEMM of more than 128 rows: the width of its tiles follows the budget, on pairs of SMs and on single blocks; the results do not."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

BUDGETS = (148, 120, 113, 112, 96, 74, 52, 48, 37, 28, 9, 2, 1)

# Row tiles with a few rows and full ones, widths that no tile width divides, a single tile column; the norms folded into the pairs' GEMMs
# (512 rows of d = 512 and wide projections are on pairs throughout) and not.
CASES = {
    "pairs_401_rows": (wl.StageDims(1, 256, 4, 2, 64, 5640), [300, 100, 1], [0, 30, 5]),
    "pairs_256_rows": (wl.StageDims(1, 512, 8, 2, 64, 4864), [256], [0]),
    "pairs_folded": (wl.StageDims(2, 2048, 16, 16, 128, 2816), [1025], [3]),
    "singles_256_rows": (wl.StageDims(2, 256, 4, 2, 64, 2824), [255, 1], [0, 40]),
    "singles_129_rows": (wl.StageDims(1, 264, 4, 2, 64, 1400), [129], [0]),
    "singles_one_tile": (wl.StageDims(1, 256, 4, 2, 64, 104), [130], [7]),
}


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BF16_ACTIVATIONS])
@pytest.mark.parametrize("name", sorted(CASES))
def test_tile_width_does_not_reach_the_output(name, flags):
    dims, q_len, ctx_len = CASES[name]
    assert len({B.hs_op_gate_up_tile(sum(q_len), dims.d_ffn, n) for n in BUDGETS}) > (1 if dims.d_ffn > 128 else 0)
    case = make_case(dims, wl.BatchSpec(q_len, ctx_len), seed=79, kv_fill=True)
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
