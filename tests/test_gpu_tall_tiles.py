"""GEMMs of more than 64 rows whose tiles' width follows the budget -- gate/up and QKV, on pairs of SMs and on single blocks -- while the
results do not."""
import numpy as np
import pytest
import torch

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


# QKV on pairs and (the last three) on single blocks: heads of 64 and of 128, tiles that end inside a head and a projection, a last tile of one or two units of three, a ragged
# row tile; with biases and behind a folded norm.
QKV_CASES = {
    "dh128_split_heads": (wl.StageDims(1, 256, 28, 4, 128, 256), [600], [0], False),
    "dh128_bias_ragged": (wl.StageDims(1, 264, 22, 2, 128, 264), [500, 77, 1], [0, 30, 5], True),
    "dh64_projections_inside_a_tile": (wl.StageDims(1, 256, 40, 4, 64, 256), [1000, 1], [0, 9], True),
    "dh128_folded": (wl.StageDims(2, 2048, 16, 4, 128, 2816), [1025], [3], False),
    "singles_dh64_200_rows": (wl.StageDims(1, 256, 24, 4, 64, 256), [199, 1], [0, 20], True),
    "singles_dh128_70_rows": (wl.StageDims(1, 264, 7, 1, 128, 264), [70], [5], True),
    "singles_decode_65_rows": (wl.StageDims(1, 512, 8, 2, 64, 512), [1] * 65, [i % 19 for i in range(65)], False),
}


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BF16_ACTIVATIONS])
@pytest.mark.parametrize("name", sorted(QKV_CASES))
def test_qkv_tile_width_does_not_reach_the_output(name, flags):
    dims, q_len, ctx_len, bias = QKV_CASES[name]
    n = (dims.n_q_heads + 2 * dims.n_kv_heads) * dims.head_dim
    assert {B.hs_op_qkv_tile(sum(q_len), n, k) for k in BUDGETS} == ({64, 128} if name.startswith("singles") else {192, 256})
    case = make_case(dims, wl.BatchSpec(q_len, ctx_len), seed=83, kv_fill=True)
    st = make_stage(case, flags=flags)
    try:
        weights = case.weights
        if bias:
            g = torch.Generator().manual_seed(7)
            for l in range(dims.n_layers):
                b = [(torch.randn(k * dims.head_dim, generator=g) * 0.5).to(torch.bfloat16) for k in (dims.n_q_heads, dims.n_kv_heads, dims.n_kv_heads)]
                st.set_qkv_bias(l, *[t.to(st.device) for t in b])
                weights = weights[:l] + [dict(weights[l], **{k: t.float().numpy() for k, t in zip(("b_q", "b_k", "b_v"), b)})] + weights[l + 1:]
        y_ref = Oracle("f32").step(case.cfg, weights, case.kv_pool.copy(), q_len, ctx_len, case.block_tables, case.x)
        first = None
        for budget in BUDGETS:
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            out = run_step(st, case, budget)
            first = out if first is None else first
            assert np.array_equal(out[0], first[0]) and np.array_equal(out[1], first[1]), budget
        assert rel_err(first[0], y_ref) <= 2e-2        # the rule of every parity test (16-bit operands)
    finally:
        st.close()


def test_few_rows_keep_whole_qkv_tiles():
    """A tile of 64 columns behind an A box of fewer than 128 rows would be a stage shorter than what an MMA reads of it."""
    for n in (1536, 4608, 6144):
        for rows in (1, 20, 32, 33, 50, 64):
            assert {B.hs_op_qkv_tile(rows, n, k) for k in BUDGETS} == {128}, (rows, n)
        assert B.hs_op_qkv_tile(65, n, 148) == 64
    assert B.hs_op_qkv_tile(0, 1536, 148) == B.hs_op_qkv_tile(65, 64, 148) == B.hs_op_qkv_tile(65, 1536, 0) == -1
