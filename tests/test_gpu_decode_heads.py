"""Decode attention over the number of query heads per KV head: up to eight they are the columns of its tensor-core tiles, beyond the
rows.  Against the oracle, in group mode and as items of single warps (a sequence beyond 4096 keys), with pages that end anywhere."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

CONTEXTS = {"groups": [0, 1, 14, 15, 16, 37, 130, 511], "items": [4170, 2, 15, 129]}


@pytest.mark.gpu
@pytest.mark.parametrize("contexts", sorted(CONTEXTS))
@pytest.mark.parametrize("heads,head_dim", [(1, 64), (3, 128), (5, 64), (7, 128), (8, 64), (8, 128), (9, 64), (16, 128)])
def test_every_number_of_heads_in_a_group(heads, head_dim, contexts):
    dims = wl.StageDims(1, 256, 2 * heads, 2, head_dim, 512)
    ctx = CONTEXTS[contexts]
    case = make_case(dims, wl.BatchSpec([1] * len(ctx), ctx), seed=91, kv_fill=True)
    st = make_stage(case)
    try:
        y, pool = run_step(st, case, st.sm_count)
        st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
        y_b, pool_b = run_step(st, case, 7)
        assert np.array_equal(y_b, y) and np.array_equal(pool_b, pool)
        y_ref = Oracle("f32").step(case.cfg, case.weights, case.kv_pool.copy(), case.batch.q_len, ctx, case.block_tables, case.x)
        assert rel_err(y, y_ref) <= 2e-2
    finally:
        st.close()
