"""Weight-streaming GEMM: the width of a block's unit follows the budget; the results do not.  Against a float64 product, and
whole steps bit for bit across budgets that take different widths."""
import numpy as np
import pytest
import torch

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

BUDGETS = (148, 112, 96, 64, 52, 37, 20, 9, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("f16", [True, False])
@pytest.mark.parametrize("M,N,K", [(1, 1024, 1024), (16, 3584, 512), (9, 1056, 2816), (16, 4640, 256), (17, 1024, 1056), (32, 3616, 512),
                                   (33, 1024, 512), (64, 2080, 1024), (5, 32, 32)])
def test_width_of_the_units_does_not_reach_the_output(M, N, K, f16):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(M * 7 + N + K)
    dt = torch.float16 if f16 else torch.bfloat16
    a = torch.randn(M, K, generator=gen, device=dev).to(dt)
    w = (torch.randn(N, K, generator=gen, device=dev) * 0.05).to(dt)
    r = torch.randn(M, N, generator=gen, device=dev)
    status = torch.zeros(2, dtype=torch.int32, device=dev)
    first = None
    for budget in BUDGETS:
        out = r.clone()
        B.hs_op_gemm_bf16(a.data_ptr(), w.data_ptr(), out.data_ptr(), out.data_ptr(), M, N, K, budget, status.data_ptr(), a_is_f16=f16)
        torch.cuda.synchronize()
        first = out if first is None else first
        assert torch.equal(out, first), budget
    ref = r.double() + a.double() @ w.double().T
    # products of 16-bit operands are exact in fp32: K + 8 additions of it, each within an ulp of the sum of the sizes
    bound = (K + 8) * 2.0 ** -23 * (r.double().abs() + a.double().abs() @ w.double().abs().T)
    assert bool(((first.double() - ref).abs() <= bound).all())
    assert int(status[0]) == 0


# Widths that three pairs of tiles do not divide (2832 / 24, 688 / 24), heads of both sizes, one row, a full row tile and
# two row tiles.
STEPS = {
    "one_row": (wl.StageDims(2, 1024, 16, 4, 64, 2832), [1], [300]),
    "11_rows": (wl.StageDims(2, 1024, 16, 4, 64, 2816), [1] * 11, [31 * i + 2 for i in range(11)]),
    "16_rows_dh128": (wl.StageDims(2, 512, 8, 2, 128, 688), [1] * 16, [17 * i for i in range(16)]),
    "29_rows_dh128": (wl.StageDims(2, 512, 8, 2, 128, 1408), [1] * 27 + [2], [40] * 27 + [0]),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(STEPS))
def test_steps_on_the_weight_streaming_kernel_at_every_width(name):
    dims, q_len, ctx_len = STEPS[name]
    case = make_case(dims, wl.BatchSpec(q_len, ctx_len), seed=52, kv_fill=True)
    y_ref = Oracle("f32").step(case.cfg, case.weights, case.kv_pool.copy(), q_len, ctx_len, case.block_tables, case.x)
    st = make_stage(case)
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
