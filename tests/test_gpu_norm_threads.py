"""RMSNorm with many threads per row where the number of them is no power of two."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

# Rows that leave three (160 threads each, 444 the last of them) and five (96) to a block; widths of one to six groups of four
# columns per thread, the last group ragged.
CASES = {
    "297_rows": (wl.StageDims(2, 2568, 8, 2, 64, 1024), [290, 7], [0, 30]),
    "444_rows": (wl.StageDims(1, 3208, 8, 2, 64, 512), [444], [3]),
    "600_rows": (wl.StageDims(1, 1544, 8, 2, 64, 512), [600], [0]),
    "400_rows_narrow": (wl.StageDims(2, 520, 8, 2, 64, 512), [399, 1], [0, 9]),
}


@pytest.mark.gpu
@pytest.mark.parametrize("conditioned", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_norm_with_any_multiple_of_32_threads_per_row(name, conditioned):
    dims, q_len, ctx_len = CASES[name]
    batch = wl.BatchSpec(q_len, ctx_len)
    case = make_case(dims, batch, seed=83, kv_fill=True)
    mod = wl.make_modulation(dims, batch.n_seqs, 83) if conditioned else None
    weights = [dict(lw, mod=mod[l].numpy()) for l, lw in enumerate(case.weights)] if conditioned else case.weights
    y_ref = Oracle("f32").step(case.cfg, weights, case.kv_pool.copy(), q_len, ctx_len, case.block_tables, case.x)
    st = make_stage(case)
    try:
        if conditioned:
            st.set_modulation(mod.to(st.device).contiguous())
        first = None
        for budget in (st.sm_count, 61, 1):
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        assert rel_err(first[0], y_ref) <= 2e-2        # the rule of every parity test (16-bit operands)
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("d,T", [(2568, 297), (3208, 444), (1032, 297)])
def test_a_rows_sum_does_not_depend_on_the_threads_that_work_on_it(d, T):
    """T rows leave three to a block, 160 threads each; 592 leave four, 128 each: the keys and values of the first T, made from
    the norm of the same input, are the same bits (QKV's sums are, whatever the number of rows)."""
    dims = wl.StageDims(1, d, 8, 2, 64, 512)
    x = wl.make_x(592, d, 89)
    pools = []
    for n in (T, 592):
        case = make_case(dims, wl.BatchSpec([n], [0]), seed=89, mpps=37, num_pages=40)
        st = make_stage(case)
        try:
            pool = run_step(st, case, st.sm_count, x_t=x[:n])[1].reshape(2, 40, 2, 16, 64)[:, case.block_tables[0][: -(-n // 16)]]
            pools.append(pool.transpose(0, 1, 3, 2, 4).reshape(2, -1, 2, 64)[:, :T])
        finally:
            st.close()
    assert np.array_equal(pools[0], pools[1])
