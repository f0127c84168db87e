"""Greedy sampling in the vocabulary GEMM's epilogue: the token is the first maximum of the logits the call wrote, at the
edges of its column tiles and row boxes, in call after call, and for rows without a maximum."""
import numpy as np
import pytest
import torch

from paper_2608_01785_b200 import binding as B


@pytest.mark.gpu
@pytest.mark.parametrize("V,n", [(8, 1), (264, 33), (1032, 65), (40008, 128)])
def test_tokens_are_the_first_maximum_of_the_logits(V, n):
    dev = torch.device("cuda:0")
    d = 256
    g = torch.Generator().manual_seed(V + n)
    gain = torch.ones(d, dtype=torch.bfloat16, device=dev)
    w = (0.02 * torch.randn(V, d, generator=g)).to(torch.bfloat16)
    w[V // 2:V // 2 + 2] = w[:2]                      # exact ties
    w = w.to(dev)
    cfg = B.make_head_config(d, V, 1e-6, 128)
    ws = torch.empty(B.hs_head_workspace_bytes(cfg), dtype=torch.uint8, device=dev)
    head = B.hs_head_create(cfg, gain.data_ptr(), w.data_ptr(), ws.data_ptr())
    try:
        rows = torch.arange(n, dtype=torch.int32, device=dev)
        for rep, budget in enumerate((148, 148, 5, 1)):
            y = torch.randn(n, d, generator=g)
            if rep == 1:
                y[n - 1] = float("inf")               # its logits are NaN: no maximum, and no trace in the next call
            y = y.to(dev)
            logits = torch.empty(n, V, device=dev)
            tokens = torch.full((n,), -7, dtype=torch.int32, device=dev)
            B.hs_head_step(head, y.data_ptr(), rows.data_ptr(), n, logits.data_ptr(), tokens.data_ptr(), budget)
            torch.cuda.synchronize()
            want = np.argmax(logits.cpu().numpy(), axis=1).astype(np.int32)
            if rep == 1:
                assert bool(torch.isnan(logits[n - 1]).all())
                want[n - 1] = 0x7fffffff
            assert np.array_equal(tokens.cpu().numpy(), want)
    finally:
        B.hs_head_destroy(head)


@pytest.mark.gpu
@pytest.mark.parametrize("budget", [148, 52])
def test_a_step_sees_gains_written_right_in_front_of_it(budget):
    """The gains are borrowed, not constant: a caller's kernel that rewrites them on the stream is ordered before the
    step, with no synchronisation between them."""
    dev = torch.device("cuda:0")
    d, V, n = 3584, 2048, 65
    g = torch.Generator(device=dev).manual_seed(3)
    w = torch.empty(V, d, dtype=torch.bfloat16, device=dev).normal_(0.0, 0.02, generator=g)
    gains = [torch.full((d,), float(v), dtype=torch.bfloat16, device=dev) for v in (1, 2, 4, 8)]     # exact factors
    gain = gains[0].clone()
    y = torch.randn(n, d, generator=g, device=dev)
    rows = torch.arange(n, dtype=torch.int32, device=dev)
    cfg = B.make_head_config(d, V, 1e-6, 128)
    ws = torch.empty(B.hs_head_workspace_bytes(cfg), dtype=torch.uint8, device=dev)
    head = B.hs_head_create(cfg, gain.data_ptr(), w.data_ptr(), ws.data_ptr())
    try:
        tokens = torch.empty(n, dtype=torch.int32, device=dev)
        logits = torch.empty(17, n, V, device=dev)
        scratch = torch.empty(1 << 24, device=dev)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream(device=dev)
        with torch.cuda.stream(stream):
            for i in range(17):
                scratch.fill_(float(i))              # the device is busy when the update is enqueued
                gain.copy_(gains[i % 4])
                B.hs_head_step(head, y.data_ptr(), rows.data_ptr(), n, logits[i].data_ptr(), tokens.data_ptr(), budget,
                               stream.cuda_stream)
        torch.cuda.synchronize()
        for i in range(17):                          # powers of two: every rounding of the step scales with the gain
            assert torch.equal(logits[i], logits[0] * float(gains[i % 4][0])), i
    finally:
        B.hs_head_destroy(head)


@pytest.mark.gpu
def test_the_first_maximum_of_rows_of_infinities_and_zeros():
    """Infinite logits of either sign, beside NaN ones too (never the maximum), and rows that underflow to zeros."""
    dev = torch.device("cuda:0")
    d, V, n = 256, 1032, 6
    g = torch.Generator().manual_seed(8)
    w = (0.02 * torch.randn(V, d, generator=g)).to(torch.bfloat16)
    w[:, 0] = 0.0
    w[700:, 0] = float("-inf")                    # logits -inf or +inf by the sign of the row's first element, NaN where it is 0
    y = torch.randn(n, d, generator=g)
    y[0, 0], y[1, 0], y[2, 0] = 1.0, -1.0, 0.0
    for budget, everywhere, scale in ((148, False, 1.0), (5, True, 1.0), (148, False, 2.0 ** -120)):
        if everywhere:
            w[:, 0] = float("-inf")
        if scale != 1.0:                          # gain and weights so small that every product underflows
            w = (torch.randn(V, d, generator=g) * scale).to(torch.bfloat16)
        wd, yd = w.to(dev), y.to(dev)
        gain = torch.full((d,), scale, dtype=torch.bfloat16, device=dev)
        cfg = B.make_head_config(d, V, 1e-6, 128)
        ws = torch.empty(B.hs_head_workspace_bytes(cfg), dtype=torch.uint8, device=dev)
        head = B.hs_head_create(cfg, gain.data_ptr(), wd.data_ptr(), ws.data_ptr())
        try:
            rows = torch.arange(n, dtype=torch.int32, device=dev)
            logits = torch.empty(n, V, device=dev)
            tokens = torch.full((n,), -7, dtype=torch.int32, device=dev)
            B.hs_head_step(head, yd.data_ptr(), rows.data_ptr(), n, logits.data_ptr(), tokens.data_ptr(), budget)
            torch.cuda.synchronize()
            lg, got = logits.cpu().numpy(), tokens.cpu().numpy()
            for r in range(n):
                if np.isnan(lg[r]).all():
                    assert got[r] == 0x7fffffff
                else:
                    assert got[r] == int(np.flatnonzero(lg[r] == np.nanmax(lg[r]))[0]), r
            if scale != 1.0:
                assert not lg.any() and not got.any()
            elif everywhere:
                assert np.isneginf(lg[0]).all() and np.isposinf(lg[1]).all() and got[0] == 0 and got[1] == 0
        finally:
            B.hs_head_destroy(head)
