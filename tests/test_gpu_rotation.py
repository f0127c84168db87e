"""The rotation of q and k rounds alike in every kernel that rotates: lo = fma(a, cos, -(b sin)), hi = fma(a, sin, b cos)."""
import numpy as np
import pytest
import torch

from paper_2608_01785_b200 import workloads as wl
from paper_2608_01785_b200.stage import Stage


def _bf16(v):
    """Nearest-even bf16 of float32 values, as float32."""
    u = v.astype(np.float32).view(np.uint32)
    return ((u + 0x7fff + ((u >> 16) & 1)) & np.uint32(0xffff0000)).view(np.float32)


def _cancelling(ratio):
    """a, b in 1 .. 2 of eight bits each (and b's power of two and sign) with a * ratio - b as small as they can make it."""
    m = np.arange(128, 256, dtype=np.float64) / 128
    r = m * abs(ratio)
    e = np.floor(np.log2(r))
    b = np.rint(r / 2 ** e * 128) / 128 * 2 ** e
    i = int(np.argmin(np.abs(r - b) / r))
    return m[i], b[i] * np.sign(ratio)


# rows, model width, query heads, KV heads, head_dim: weight streaming of one, two and four row tiles, single blocks of the tiled
# kernel, pairs of them.
CASES = {
    "9_rows": (9, 1024, 4, 4, 64),
    "16_rows_dh128": (16, 1024, 4, 4, 128),
    "31_rows": (31, 1024, 4, 4, 64),
    "33_rows_dh128": (33, 1024, 4, 4, 128),
    "64_rows": (64, 1024, 4, 4, 64),
    "65_rows": (65, 256, 4, 4, 64),
    "100_rows_dh128": (100, 256, 4, 4, 128),
    "1300_rows_dh128": (1300, 512, 12, 4, 128),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CASES))
def test_rotation_rounds_alike(name):
    """Rows of ones and weights with one value per row of k's projection, so that k before its rotation is that value exactly;
    values that nearly cancel in lo or in hi at some row's position, where the roundings inside show in the bf16 result."""
    T, d, hq, hk, dh = CASES[name]
    half = dh // 2
    dims = wl.StageDims(1, d, hq, hk, dh, 256, rms_eps=0.0)
    rng = np.random.default_rng(T)
    theta = np.power(float(dims.rope_base), -2.0 * np.arange(half) / dh)
    ang = np.arange(T, dtype=np.float64)[:, None] * theta
    cos, sin = np.cos(ang).astype(np.float32).astype(np.float64), np.sin(ang).astype(np.float32).astype(np.float64)
    k = np.zeros((hk, dh))
    for h in range(hk):
        for i in range(half):
            p = int(rng.integers(1, T))
            k[h, i], k[h, i + half] = _cancelling(cos[p, i] / sin[p, i] if i & 1 else -sin[p, i] / cos[p, i])
    lim = 2.0 ** 8                                       # (fp16 and fp32 hold them exactly)
    k = np.clip(k, -lim, lim)
    w_k = np.zeros((hk * dh, d), dtype=np.float32)
    w_k[np.arange(hk * dh), rng.integers(0, d, hk * dh)] = k.reshape(-1)
    dev = torch.device("cuda:0")
    weights = wl.make_layer_weights(dims, 5, 0)
    weights["g_attn"] = torch.ones(d, dtype=torch.bfloat16)
    weights["w_k"] = torch.from_numpy(w_k).to(torch.bfloat16)
    assert np.array_equal(weights["w_k"].float().numpy(), w_k)
    mpps = -(-T // 16)
    st = Stage(dims, [{n: v.to(dev) for n, v in weights.items()}], mpps + 1, T, 1, mpps, T)
    try:
        tables = st.block_table_array([st.kv_alloc(0, T)])
        x = torch.ones(T, d, dtype=torch.bfloat16, device=dev)
        y = torch.empty(T, d, device=dev)
        st.step(st.make_batch([T], [0], tables, x, y), st.sm_count)
        torch.cuda.synchronize()
        assert st.status() == 0
        got = st.kv_pool_view()[0, 0].float().cpu().numpy()[tables[0]]          # [page][head][16][dh]
        got = got.transpose(0, 2, 1, 3).reshape(-1, hk, dh)[:T]
    finally:
        st.close()
    a, b = k[None, :, :half], k[None, :, half:]
    c, s = cos[:, None, :], sin[:, None, :]
    f32 = lambda v: v.astype(np.float32).astype(np.float64)
    lo, hi = _bf16(a * c - f32(b * s)), _bf16(a * s + f32(b * c))
    other = np.mean(_bf16(f32(a * c) - b * s) != lo), np.mean(_bf16(f32(a * s) + b * c) != hi)
    assert min(other) > 0                                # (the roundings the other way do show)
    assert np.array_equal(got[..., :half], lo) and np.array_equal(got[..., half:], hi)
