"""Decode attention over the number of query heads per KV head: up to eight they are the columns of its tensor-core tiles, beyond the
rows.  Against the oracle, in group mode and as items of single warps (a sequence beyond 4096 keys), with pages that end anywhere."""
import numpy as np
import pytest
import torch

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


@pytest.mark.gpu
@pytest.mark.parametrize("heads,head_dim", [(1, 64), (4, 64), (5, 128), (8, 64), (8, 128)])
def test_a_head_gives_the_bits_of_a_larger_group(heads, head_dim):
    """Scores, weights and outputs are rounded and added alike whether heads are columns (at most eight in a group) or rows (here
    twelve).  Items that are a whole sequence."""
    hkv, many = 2, 12
    lens = [k - i % 3 if k > 3 else k for k in (1, 2, 9, 16, 17, 100, 201, 256) for i in range(64)]
    n, pages = len(lens), [-(-k // 16) for k in lens]
    tables = np.full((n, max(pages)), -1, dtype=np.int32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(17)
    for s, k in enumerate(pages):
        tables[s, :k] = np.arange(sum(pages[:s]), sum(pages[:s]) + k)
    pool = torch.randn(1, 2, sum(pages), hkv, 16, head_dim, generator=gen, device="cuda").to(torch.bfloat16)
    q = torch.randn(n, hkv, many, head_dim, generator=gen, device="cuda").to(torch.bfloat16)

    def attend(g, first, last):
        part = q[first:last, :, :g].contiguous()
        o = torch.full_like(part, float("nan"))
        B.hs_op_decode_attention_noalloc(part.data_ptr(), pool.data_ptr(), 1, 0, sum(pages), hkv * g, hkv, head_dim, lens[first:last],
                                         tables[first:last], o.data_ptr(), 148)
        torch.cuda.synchronize()
        assert B.hs_op_decode_attention_noalloc_status() == B.HS_OK
        return o
    for first in range(0, n, 64):
        want, got = attend(many, first, first + 64), attend(heads, first, first + 64)
        assert torch.isfinite(got).all() and torch.equal(got, want[:, :, :heads])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 24])                    # groups in slices, and whole ones
@pytest.mark.parametrize("head_dim", [64, 128])
def test_a_stage_s_head_gives_the_bits_of_a_larger_group(head_dim, n):
    ctx = [37 * i + 380 * (i % 9) for i in range(n)] if n > 2 else [3900, 2500]
    outs = []
    for heads in (24, 16):                                 # twelve and eight per KV head, the eight being the first of the twelve
        case = make_case(wl.StageDims(1, 256, heads, 2, head_dim, 256), wl.BatchSpec([1] * n, ctx), seed=92, kv_fill=True)
        w = make_case(wl.StageDims(1, 256, 24, 2, head_dim, 256), case.batch, seed=92).weights_t
        w_q = w[0]["w_q"].view(2, 12, head_dim, 256)[:, :heads // 2].reshape(-1, 256).contiguous()
        w_o = w[0]["w_o"].view(256, 2, 12, head_dim)[:, :, :heads // 2].reshape(256, -1).contiguous()
        st = make_stage(case, weights=[dict(w[0], w_q=w_q, w_o=w_o)])
        try:
            run_step(st, case, st.sm_count)
            outs.append([st.debug_tensor(k)[:n].clone().view(n, 2, -1, head_dim)[:, :, :8] for k in ("q", "o")])
        finally:
            st.close()
    assert torch.equal(outs[0][0], outs[1][0])              # (the same queries, or the comparison says nothing)
    assert torch.isfinite(outs[0][1].float()).all() and torch.equal(outs[0][1], outs[1][1])
