"""Steps whose residual GEMMs leave the partial sums of their K splits to the norm kernel behind them: against the oracle,
and bit for bit across budgets."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

TOL = 2e-2        # max|err| / RMS, the rule of every parity test (16-bit operands)

# name: dims, new tokens, cached tokens.  Row counts around the edges of the 32-row boxes and of the 128- and 256-row
# tiles, widths that leave a ragged tile column and a ragged K block, one row per block and many.
CASES = {
    "17_rows": (wl.StageDims(2, 1024, 16, 4, 64, 3072), [1] * 17, list(range(5, 600, 35))[:17]),
    "33_rows_wide_k": (wl.StageDims(2, 520, 8, 2, 64, 4104), [33], [0]),
    "65_rows": (wl.StageDims(2, 512, 8, 2, 64, 1408), [60, 1, 4], [0, 300, 12]),
    "128_rows": (wl.StageDims(2, 768, 12, 4, 64, 2048), [127, 1], [9, 40]),
    "129_rows": (wl.StageDims(2, 1032, 8, 2, 128, 2056), [129], [0]),
    "300_rows": (wl.StageDims(2, 1024, 8, 2, 128, 2816), [280] + [1] * 20, [33] + list(range(20, 400, 19))),
    # few rows of a long K (ten splits); norm threads that hold four groups and more splits than they request at a time, the
    # same with eight groups, and eight groups of rows wider than a round of them
    "24_rows_long_k": (wl.StageDims(1, 1024, 8, 2, 64, 8192), [20, 1, 1, 1, 1], [0, 300, 12, 5, 77]),
    "300_rows_d1032": (wl.StageDims(2, 1032, 8, 2, 128, 2816), [300], [0]),
    "594_rows_d1032": (wl.StageDims(2, 1032, 8, 2, 64, 2048), [594], [0]),
    "300_rows_d2056": (wl.StageDims(1, 2056, 8, 2, 64, 2048), [290, 1, 9], [0, 60, 3]),
}
# residual GEMMs whose splits add into the output in turn: two splits of 22 K blocks
ORDERED = {
    "300_rows_d2560": (wl.StageDims(1, 2560, 8, 2, 64, 1408), [299, 1], [0, 40]),
    "600_rows_d1032": (wl.StageDims(2, 1032, 8, 2, 64, 1408), [600], [0]),
}


def _check(dims, q_len, ctx_len, conditioned, name):
    batch = wl.BatchSpec(list(q_len), list(ctx_len))
    case = make_case(dims, batch, seed=41, kv_fill=True)
    mod = wl.make_modulation(dims, batch.n_seqs, 41) if conditioned else None
    weights = [dict(lw, mod=mod[l].numpy()) for l, lw in enumerate(case.weights)] if conditioned else case.weights
    y_ref = Oracle("f32").step(case.cfg, weights, case.kv_pool.copy(), batch.q_len, batch.ctx_len, case.block_tables, case.x)
    st = make_stage(case)
    try:
        if conditioned:
            st.set_modulation(mod.to(st.device).contiguous())
        first = None
        for budget in (st.sm_count, 52, 2, 1):
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        err = rel_err(first[0], y_ref)
        print(f"residual sums, {name}, conditioned {conditioned}: max|err|/RMS = {err:.2e}")
        assert err <= TOL
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("conditioned", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_partial_sums_of_the_residual_gemms(name, conditioned):
    _check(*CASES[name], conditioned, name)


@pytest.mark.gpu
@pytest.mark.parametrize("conditioned", [False, True])
@pytest.mark.parametrize("name", sorted(ORDERED))
def test_ordered_sums_of_the_residual_gemms(name, conditioned):
    _check(*ORDERED[name], conditioned, name)


def test_the_cases_reach_the_forms_they_are_named_for():
    splits = {n: B.hs_op_gemm_part_splits(sum(q), d.d_model, d.d_ffn) for n, (d, q, _) in {**CASES, **ORDERED}.items()}
    assert splits["24_rows_long_k"] > 8 and splits["300_rows_d1032"] > 4
    assert splits["594_rows_d1032"] > 2 and splits["300_rows_d2056"] > 2
    assert all(splits[n] >= 2 for n in CASES if n not in ("17_rows", "33_rows_wide_k", "129_rows"))
    assert all(splits[n] == 0 for n in ORDERED)
