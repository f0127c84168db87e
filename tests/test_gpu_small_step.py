"""Small decode-only steps in one cooperative launch: against the oracle, and bit for bit -- outputs, cache and the stage's own
buffers -- against the chain of launches that a profiled step is, at every budget."""
import numpy as np
import pytest
import torch

from oracle.oracle import Oracle
from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from paper_2608_01785_b200.stage import Stage
from tests.gpu_helpers import make_stage, run_step
from tests.helpers import make_case, rel_err

D = wl.StageDims
# name: dims, cached tokens.  Two K steps per warp, a copy's four, one more, the most; heads per KV head from one to eight; rows of
# one tile and of two, a tile full and one row more; new tokens at the first and the last place of a page; groups cut into
# slices, more slices than blocks at the smaller budgets; one layer, and more than the three exchange buffers.
CASES = {
    "one_row": (D(4, 1024, 16, 4, 64, 2816), [300]),
    "one_row_sliced": (D(2, 1024, 16, 4, 64, 2816), [4079]),
    "sliced_beside_whole": (D(3, 1024, 16, 2, 64, 1536), [4079, 33, 2500]),
    "odd_slices": (D(2, 1024, 16, 4, 64, 1536), [3000, 3900, 100, 4000, 2000]),
    "first_token": (D(5, 512, 8, 2, 64, 512), [0]),
    "page_edges": (D(3, 768, 12, 4, 64, 2048), [0, 14, 15, 16, 31, 32, 1023]),
    "eight_heads_a_group": (D(3, 1024, 16, 2, 64, 1536), [700, 33, 255, 256, 1023, 5, 64, 300]),
    "nine_rows": (D(4, 1024, 16, 2, 64, 3072), [31 * i + 2 for i in range(9)]),
    "sixteen_rows": (D(2, 1024, 16, 4, 64, 2816), [61 * i + 15 for i in range(16)]),
    "wide": (D(2, 2048, 32, 8, 64, 3072), [90, 17, 400]),
    "one_head_a_group": (D(1, 1280, 20, 20, 64, 1280), [40, 200, 7]),
}

SLICED = {"one_row_sliced": {8}, "sliced_beside_whole": {1, 5, 8}, "odd_slices": {1, 3, 4, 5}}      # slices of its groups, else one


def _budgets(n, dims, sms):
    return [b for b in (sms, 96, 52, 33, 5, 1) if B.hs_op_one_launch_step(n, dims, b) == 1]


def _step(st, case, budget):
    st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
    y, pool = run_step(st, case, budget)
    n = case.batch.n_seqs
    return y, pool, *[st.debug_tensor(k)[:n].float().cpu().numpy() for k in ("h", "q", "o", "act")]


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, B.HS_FLAG_BF16_ACTIVATIONS])
@pytest.mark.parametrize("name", sorted(CASES))
def test_one_launch_gives_the_bits_of_the_chain(name, flags):
    dims, ctx = CASES[name]
    case = make_case(dims, wl.BatchSpec([1] * len(ctx), ctx), seed=61, kv_fill=True)
    st = make_stage(case, flags=flags)
    try:
        bias = [torch.randn(k, device=st.device).mul_(0.1).to(torch.bfloat16) for k in (dims.q_dim, dims.kv_dim, dims.kv_dim)]
        budgets = _budgets(len(ctx), dims, st.sm_count)
        assert budgets
        items, group, _ = B.hs_stage_plan_attention(st.handle, st.make_batch([1] * len(ctx), ctx, case.block_tables, case.x_t.to(st.device),
                                                                             torch.empty(len(ctx), dims.d_model, device=st.device)))
        assert group == 1 and set(items[:, 7] & 0xffff) == SLICED.get(name, {1})
        for biased in (False, True):
            if biased:
                st.set_qkv_bias(dims.n_layers - 1, *bias)
            B.hs_stage_profile_enable(st.handle, True)
            want = _step(st, case, st.sm_count)
            assert B.hs_stage_profile_read(st.handle)["gemm_qkv"][1] == dims.n_layers
            assert B.hs_stage_last_step_one_launch(st.handle) == 0
            B.hs_stage_profile_enable(st.handle, False)
            for budget in budgets:
                for a, b in zip(_step(st, case, budget), want):
                    assert np.array_equal(a, b), (budget, biased)
                assert B.hs_stage_last_step_one_launch(st.handle) == 1
            if not biased:
                y_ref = Oracle("f32").step(case.cfg, case.weights, case.kv_pool.copy(), case.batch.q_len, case.batch.ctx_len, case.block_tables, case.x)
                assert rel_err(want[0], y_ref) <= 2e-2
    finally:
        st.close()


@pytest.mark.gpu
def test_steps_of_other_sizes_leave_nothing_behind_for_the_next():
    """Rows come and go between steps of one stage, and NaN is a result like another: what a step finds in the exchange buffers
    must not matter."""
    dims = D(4, 1024, 16, 4, 64, 2816)
    ctx = [100 + 37 * i for i in range(16)]
    case = make_case(dims, wl.BatchSpec([1] * 16, ctx), seed=62, kv_fill=True)
    st = make_stage(case)
    try:
        def step(n, x):
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            return run_step(st, case, st.sm_count, [1] * n, ctx[:n], x[:n], case.block_tables[:n])[0]
        first = {n: step(n, case.x_t) for n in (16, 3, 9, 1)}
        bad = case.x_t.clone()
        bad[0] = float("nan")
        y = step(9, bad)
        assert np.isnan(y[0]).all() and np.array_equal(y[1:], first[9][1:])
        for n in (3, 16, 1, 9):
            assert np.array_equal(step(n, case.x_t), first[n]), n
    finally:
        st.close()


@pytest.mark.gpu
def test_a_second_stage_in_the_same_workspace_streams_its_own_weights():
    """The weights' tensor maps lie in the workspace.  (With bf16 activations the stages read the caller's tensors, so the two sets of
    maps differ; both sets of weights stay allocated.)"""
    dims = D(3, 1024, 16, 4, 64, 2816)
    ctx = [100, 37, 260]
    cases = [make_case(dims, wl.BatchSpec([1] * 3, ctx), seed=k, kv_fill=True) for k in (64, 65)]
    stages = [make_stage(c, flags=B.HS_FLAG_BF16_ACTIVATIONS) for c in cases]
    try:
        shared = stages[0]
        want = [_step(st, cases[0], shared.sm_count) for st in stages]
        assert not np.array_equal(want[0][0], want[1][0])
        for i in (1, 0, 1):
            B.hs_stage_destroy(shared.handle)
            shared.handle = 0
            ptrs = [{k: v.data_ptr() for k, v in lw.items()} for lw in stages[i].weights]
            shared.handle = B.hs_stage_create(shared.cfg, ptrs, shared.kv_pool.data_ptr(), shared.workspace.data_ptr())
            for a, b in zip(_step(shared, cases[0], shared.sm_count), want[i]):
                assert np.array_equal(a, b), i
    finally:
        for st in stages:
            st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("where", ["g_attn", "g_mlp", "w_up", "kv"])
def test_clamped_values_are_counted_as_the_chain_counts_them(where):
    """Beyond fp16's range: a first or a later norm's h, gate/up's act, the attention's output."""
    dims = D(3, 768, 12, 4, 64, 1024)
    ctx = [0, 14, 15, 16, 31, 130, 1023, 300, 77]
    case = make_case(dims, wl.BatchSpec([1] * 9, ctx), seed=67, kv_fill=True)
    weights = case.weights_t
    if where != "kv":
        weights = [dict(w, **{where: w[where] * (3e4 if where != "w_up" else 2e5)}) for w in weights]
    st = make_stage(case, weights=weights)
    try:
        pool = wl.bits_to_bf16_tensor(case.kv_pool, st.device) * (1e6 if where == "kv" else 1)

        def step(budget):
            before = st.saturation_count()
            st.kv_pool.copy_(pool)
            y = run_step(st, case, budget, expect_saturation=True)[0]
            return y, st.saturation_count() - before
        for n, budgets in ((9, (148, 52)), (4, (148, 5))):
            case.x_t, case.batch, case.block_tables = case.x_t[:n], wl.BatchSpec([1] * n, ctx[:n]), case.block_tables[:n]
            B.hs_stage_profile_enable(st.handle, True)
            want, count = step(st.sm_count)
            B.hs_stage_profile_enable(st.handle, False)
            assert count > 0
            for budget in budgets:
                y, got = step(budget)
                assert B.hs_stage_last_step_one_launch(st.handle) == 1
                assert got == count and np.array_equal(y, want, equal_nan=True), budget
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("budget", [148, 52, 3])
def test_one_launch_steps_and_chains_follow_each_other_without_a_wait(budget):
    """Steps of one stage of other rows and sequences in one stream, one-launch steps among chains (a prompt, more rows than sixteen), none
    waited for."""
    dims = D(4, 1024, 16, 4, 64, 2816)
    specs = [([1], [300]), ([1] * 16, [61 * i + 15 for i in range(16)]), ([1] * 3, [5, 700, 64]), ([20, 1], [0, 40]), ([1] * 8, [31 * i for i in range(8)]),
             ([1] * 17, [9 * i for i in range(17)]), ([1] * 2, [15, 2000]), ([1] * 9, [100 + i for i in range(9)])]
    batches = [wl.BatchSpec(q, c) for q, c in specs]
    mpps = max(-(-t // 16) for b in batches for t in b.total_len())
    tables, n_pages = [], 0
    for b in batches:                             # pages of its own for every batch: its step gives the same whenever it runs
        t = np.full((b.n_seqs, mpps), -1, dtype=np.int32)
        for s, total in enumerate(b.total_len()):
            k = -(-total // 16)
            t[s, :k] = np.arange(n_pages, n_pages + k)
            n_pages += k
        tables.append(t)
    st = Stage(dims, wl.make_weights(dims, 71, "cpu", "n002"), n_pages, max(b.n_tokens for b in batches), max(b.n_seqs for b in batches), mpps,
               max(t for b in batches for t in b.total_len()))
    try:
        gen = torch.Generator(device=st.device)
        gen.manual_seed(72)
        st.kv_pool.normal_(generator=gen)
        xs = [wl.make_x(b.n_tokens, dims.d_model, 73 + i, st.device) for i, b in enumerate(batches)]

        def step(i, sms):
            y = torch.full((batches[i].n_tokens, dims.d_model), float("nan"), device=st.device)
            st.step(st.make_batch(batches[i].q_len, batches[i].ctx_len, tables[i], xs[i], y), sms)
            return y
        B.hs_stage_profile_enable(st.handle, True)             # (chains)
        want = [step(i, st.sm_count) for i in range(len(batches))]
        torch.cuda.synchronize()
        B.hs_stage_profile_enable(st.handle, False)
        forms = []
        for i in range(len(batches)):
            step(i, budget)
            forms.append(B.hs_stage_last_step_one_launch(st.handle))
        assert forms == [B.hs_op_one_launch_step(len(q), dims, budget) if max(q) == 1 else 0 for q, _ in specs] and {0, 1} == set(forms)
        got = [(i, step(i, budget)) for i in [0, 1, 2, 3, 4, 5, 6, 7, 1, 0, 5, 2, 7, 4, 3, 6, 0, 0, 1, 1, 6, 2] * 3]
        torch.cuda.synchronize()
        assert st.status() == 0
        for i, y in got:
            assert torch.isfinite(y).all() and torch.equal(y, want[i]), i
    finally:
        st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["one_row_sliced", "first_token", "eight_heads_a_group", "sixteen_rows"])
def test_every_way_out_of_the_one_launch(name):
    """A launch that the context refuses becomes the chain.  A step whose wait runs out ends by itself and stores nothing that it has not got:
    no block leaves the first barrier, so neither the output nor the cache is touched.  What such a step leaves does not reach the
    next one."""
    dims, ctx = CASES[name]
    case = make_case(dims, wl.BatchSpec([1] * len(ctx), ctx), seed=66, kv_fill=True)
    st = make_stage(case)
    try:
        for budget in _budgets(len(ctx), dims, st.sm_count)[:3]:
            want = _step(st, case, budget)
            assert B.hs_stage_last_step_one_launch(st.handle) == 1
            B.hs_stage_one_launch_fault(st.handle, B.HS_FAULT_REFUSED)
            for a, b in zip(_step(st, case, budget), want):
                assert np.array_equal(a, b), budget
            assert B.hs_stage_last_step_one_launch(st.handle) == 0
            B.hs_stage_one_launch_fault(st.handle, B.HS_FAULT_GAVE_UP)
            for _ in range(3):
                _step(st, case, budget)
            B.hs_stage_one_launch_fault(st.handle, B.HS_FAULT_NONE)
            for a, b in zip(_step(st, case, budget), want):
                assert np.array_equal(a, b), budget
        x = case.x_t.to(st.device)
        for budget in _budgets(len(ctx), dims, st.sm_count)[:3]:      # (from here on the stage's status says what happened)
            st.kv_pool.copy_(wl.bits_to_bf16_tensor(case.kv_pool, st.device))
            y = torch.full((len(ctx), dims.d_model), -7.0, device=st.device)
            b = st.make_batch([1] * len(ctx), ctx, case.block_tables, x, y)
            B.hs_stage_one_launch_fault(st.handle, B.HS_FAULT_MISSING, 2_000_000)
            t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            t[0].record()
            st.step(b, budget)
            t[1].record()
            torch.cuda.synchronize()
            assert st.status() == B.HS_ERR_TIMEOUT and 2.0 <= t[0].elapsed_time(t[1]) < 50.0
            assert (y == -7.0).all() and np.array_equal(wl.bf16_bits_numpy(st.kv_pool).reshape(-1), case.kv_pool)
            B.hs_stage_one_launch_fault(st.handle, B.HS_FAULT_NONE)
            st.step(b, budget)
            torch.cuda.synchronize()
            assert np.array_equal(y.cpu().numpy(), want[0]) and np.array_equal(wl.bf16_bits_numpy(st.kv_pool).reshape(-1), want[1])
        for bad in ((-1, 1000), (4, 1000), (B.HS_FAULT_MISSING, 10), (B.HS_FAULT_MISSING, 10**9)):
            with pytest.raises(B.HsError):
                B.hs_stage_one_launch_fault(st.handle, *bad)
    finally:
        st.close()


def test_the_rule_that_takes_the_one_launch():
    t = wl.DIMS["c4_talker"]
    assert [B.hs_op_one_launch_step(n, t, 148) for n in (1, 8, 9, 16, 17)] == [1, 1, 1, 1, 0]
    assert [B.hs_op_one_launch_step(8, t, b) for b in (1, 52)] == [1, 1] and [B.hs_op_one_launch_step(9, t, b) for b in (31, 32)] == [0, 1]
    for dims in (D(33, 1024, 16, 4, 64, 2816), D(2, 1024, 8, 4, 128, 2816), D(2, 1024, 16, 1, 64, 2816), D(2, 1088, 16, 4, 64, 2816),
                 D(2, 1024, 16, 4, 64, 2832), D(2, 1024, 16, 4, 64, 3328), D(2, 2304, 16, 4, 64, 2816), wl.DIMS["c3_7b"], wl.DIMS["c2_shared"]):
        assert B.hs_op_one_launch_step(4, dims, 148) == 0, dims
    assert B.hs_op_one_launch_step(9, D(2, 1280, 16, 4, 64, 2816), 148) == 0 and B.hs_op_one_launch_step(0, t, 148) == -1
