"""Steps enqueued one behind the other without a wait between them: each one finds its own metadata (work lists, positions, block
tables), which the device fetches from the stage's few pinned blocks while the host already plans the next steps."""
import numpy as np
import pytest
import torch

from paper_2608_01785_b200 import workloads as wl
from paper_2608_01785_b200.stage import Stage

DIMS = wl.StageDims(2, 512, 8, 2, 64, 1408)
# new and cached tokens of the sequences: blocks that end at different words, one row and many, with and without prefill chunks
BATCHES = [([1], [7]), ([1, 1, 1], [300, 17, 33]), ([40], [0]), ([130, 1, 1], [50, 20, 260]), ([1] * 20, [11 * i for i in range(20)]), ([2, 1], [15, 15])]


@pytest.mark.gpu
@pytest.mark.parametrize("budget,pages", [(148, 0), (40, 0), (1, 0), (148, 4096), (16, 4096), (3, 4096), (1, 4096)])
def test_back_to_back_steps_find_their_own_metadata(budget, pages):
    """`pages`: width of the block tables, if more than the longest sequence takes: 320 KB of them are one or several rounds of the
    kernel that fetches them, or a copy."""
    batches = [wl.BatchSpec(list(q), list(c)) for q, c in BATCHES]
    mpps = max(pages, max(-(-t // 16) for b in batches for t in b.total_len()))
    tables, n_pages = [], 0                       # every batch has pages of its own: its step gives the same whenever it runs
    for b in batches:
        t = np.full((b.n_seqs, mpps), -1, dtype=np.int32)
        for s, total in enumerate(b.total_len()):
            k = -(-total // 16)
            t[s, :k] = np.arange(n_pages, n_pages + k)
            n_pages += k
        tables.append(t)
    st = Stage(DIMS, wl.make_weights(DIMS, 71, "cpu", "n002"), n_pages, max(b.n_tokens for b in batches), max(b.n_seqs for b in batches), mpps,
               max(t for b in batches for t in b.total_len()))
    try:
        gen = torch.Generator(device=st.device)
        gen.manual_seed(72)
        st.kv_pool.normal_(generator=gen)
        xs = [wl.make_x(b.n_tokens, DIMS.d_model, 73 + i, st.device) for i, b in enumerate(batches)]

        def step(i):
            y = torch.full((batches[i].n_tokens, DIMS.d_model), float("nan"), device=st.device)
            st.step(st.make_batch(batches[i].q_len, batches[i].ctx_len, tables[i], xs[i], y), budget)
            return y
        want = []
        for i in range(len(batches)):
            want.append(step(i))
            torch.cuda.synchronize()
        got = [(i, step(i)) for i in [0, 1, 2, 3, 4, 5, 4, 0, 3, 1, 5, 2] * 3]
        torch.cuda.synchronize()
        assert st.status() == 0
        for i, y in got:
            assert torch.isfinite(y).all() and torch.equal(y, want[i]), i
        # five steps are enqueued without a wait on the host, behind whatever the stream is doing
        ys, busy = [torch.empty_like(want[i]) for i in range(5)], torch.cuda.Event()
        args = [st.make_batch(batches[i].q_len, batches[i].ctx_len, tables[i], xs[i], ys[i]) for i in range(5)]
        torch.cuda._sleep(1_000_000_000)
        busy.record()
        for a in args:
            st.step(a, budget)
        assert not busy.query()
        torch.cuda.synchronize()
        assert all(torch.equal(y, want[i]) for i, y in enumerate(ys))
    finally:
        st.close()
