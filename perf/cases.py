"""The workloads whose speed this repository looks after, through its public entry points (`Stage`, `binding`).

A case is one tick of a serving loop: a step of a stage (prefill chunks and decode rows together, as the scheduler admits
them), a denoising step, the sampling head behind a step, or a backbone step with talker steps beside it on the rest of
the SMs.  Dimensions, sequence lengths and SM budgets are those of `paper_2608_01785_b200/workloads.py`, of the trace
replay and of `bench.py`.  Fields of a stage case:

  dims        name in workloads.DIMS; `layers` of it are built (0 = all).  A layer's time does not depend on the depth,
              so the 7B-class cases beside the two full-depth ones keep four layers, like c2_shared
  prefill     number of prefill chunks, of chunk_lo .. chunk_hi new tokens behind 0 .. chunk_ctx cached ones
  decode      number of decode rows, with ctx_lo .. ctx_hi cached tokens each
  lens        seed of those lengths
  budget      SMs given to the step (a stage with a neighbour gets a part of the 148)
  bf16        activations in bf16 (HS_FLAG_BF16_ACTIVATIONS) instead of fp16
  bias        q / k / v biases, as in a 7B-class checkpoint
"""
import math

import numpy as np
import torch

from paper_2608_01785_b200 import binding as B
from paper_2608_01785_b200 import workloads as wl
from paper_2608_01785_b200.stage import Stage

VOCAB = 152064
PAGE = 16
FULL = 148


def _step(name, dims, layers=0, prefill=0, chunk_lo=0, chunk_hi=0, chunk_ctx=0, decode=0, ctx_lo=0, ctx_hi=0, lens=1,
          budget=FULL, bf16=False, bias=False):
    c = {"kind": "step", "dims": dims, "layers": layers, "prefill": prefill, "chunk_lo": chunk_lo, "chunk_hi": chunk_hi,
         "chunk_ctx": chunk_ctx, "decode": decode, "ctx_lo": ctx_lo, "ctx_hi": ctx_hi, "lens": lens, "budget": budget,
         "bf16": bf16, "bias": bias}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one voice request alone on the GPU: the talker decodes a single row, the smallest call there is
        _step("talker_1", "c4_talker", decode=1, ctx_lo=128, ctx_hi=1024, lens=11),
        # the talker's ordinary batch while the backbone is idle
        _step("talker_16", "c4_talker", decode=16, ctx_lo=128, ctx_hi=1024, lens=3),
        # the same stage beside a backbone that holds 96 SMs; an odd batch
        _step("talker_11_sm52", "c4_talker", decode=11, ctx_lo=128, ctx_hi=1500, lens=12, budget=52),
        # image generation: a conditioned denoising step over four images of 256 latent tokens
        {"name": "dit_4x256", "kind": "dit", "images": 4, "tokens": 256, "budget": FULL},
        # greedy sampling behind a full tick (65 sequences), and the lookup of the tokens it yields
        {"name": "head_65", "kind": "head", "rows": 65, "budget": FULL},
        # text decoding of a few requests, checkpoint-like: q / k / v biases, activations in bf16
        _step("7b_decode_9_bf16", "c3_7b", layers=4, decode=9, ctx_lo=512, ctx_hi=4096, lens=13, bf16=True, bias=True),
        # a decode-only tick of a full batch, whole depth
        _step("7b_decode_64", "c3_decode", decode=64, ctx_lo=512, ctx_hi=4096, lens=2),
        # a half-full decode tick while a downstream stage holds 52 SMs
        _step("7b_decode_29_sm96", "c3_7b", layers=4, decode=29, ctx_lo=300, ctx_hi=4000, lens=14, budget=96),
        # the last, ragged chunk of a chunked prefill with some decode rows beside it
        _step("7b_chunk_ragged", "c3_7b", layers=4, prefill=1, chunk_lo=300, chunk_hi=400, chunk_ctx=2048, decode=7,
              ctx_lo=200, ctx_hi=3000, lens=15),
        # eight prompts and 32 decode rows on a small shared backbone
        _step("shared_mixed", "c2_shared", prefill=8, chunk_lo=128, chunk_hi=1024, decode=32, ctx_lo=256, ctx_hi=2048,
              lens=1),
        # spatial sharing: the same backbone on 96 SMs, four talker steps beside it on the other 52
        {"name": "corun_96_52", "kind": "corun", "prefill": 8, "decode": 32, "lens": 16, "budget": 96, "talkers": 16,
         "talker_steps": 4},
        # the headline step: a full 2048-token chunk and 64 decode rows, 28 layers
        _step("7b_mixed", "c3_7b", prefill=1, chunk_lo=2048, chunk_hi=2048, decode=64, ctx_lo=512, ctx_hi=4096, lens=2),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))


def draw(rng):
    budget = FULL if rng.random() < 0.5 else rng.choice([120, 112, 96, 74, 52, 48, 37, rng.randint(28, 147)])
    lens = rng.randrange(1, 1 << 20)
    kind = rng.choice(["talker", "talker", "decode", "decode", "shared", "mixed", "dit", "head", "corun"])
    if kind == "talker":
        return _step("", "c4_talker", decode=rng.randint(1, 16), ctx_lo=64, ctx_hi=_log(rng, 128, 1500), lens=lens,
                     budget=budget)
    if kind == "decode":
        return _step("", "c3_7b", layers=4, decode=_log(rng, 1, 64), ctx_lo=64, ctx_hi=_log(rng, 256, 4096), lens=lens,
                     budget=budget, bf16=rng.random() < 0.25, bias=rng.random() < 0.5)
    if kind == "shared":
        hi = _log(rng, 32, 1024)
        return _step("", "c2_shared", prefill=rng.randint(1, 8), chunk_lo=max(1, hi // 8), chunk_hi=hi,
                     chunk_ctx=rng.choice([0, 0, 700]), decode=rng.randint(0, 32), ctx_lo=64, ctx_hi=_log(rng, 256, 2048),
                     lens=lens, budget=budget, bf16=rng.random() < 0.25)
    if kind == "mixed":
        n = _log(rng, 32, 2048)
        return _step("", "c3_7b", layers=4, prefill=1, chunk_lo=n, chunk_hi=n, chunk_ctx=rng.choice([0, 0, 2048]),
                     decode=rng.randint(0, 64), ctx_lo=64, ctx_hi=_log(rng, 256, 4096), lens=lens, budget=budget,
                     bf16=rng.random() < 0.25, bias=rng.random() < 0.5)
    if kind == "dit":
        return {"kind": "dit", "images": rng.randint(1, 4), "tokens": _log(rng, 64, 256), "budget": budget}
    if kind == "head":
        return {"kind": "head", "rows": _log(rng, 1, 128), "budget": budget}
    backbone = rng.choice([120, 112, 96, 74])
    return {"kind": "corun", "prefill": rng.randint(1, 8), "decode": rng.randint(1, 32), "lens": lens, "budget": backbone,
            "talkers": rng.randint(1, 16), "talker_steps": rng.randint(2, 5)}


# --- shapes of a case ---------------------------------------------------------------------------------------------
def _dims(case):
    d = wl.DIMS[case["dims"]]
    return wl.replace(d, n_layers=case["layers"]) if case["layers"] else d


def _batch(case):
    r = np.random.Generator(np.random.PCG64(case["lens"]))
    q = r.integers(case["chunk_lo"], case["chunk_hi"] + 1, case["prefill"]).tolist() if case["prefill"] else []
    c = r.integers(0, case["chunk_ctx"] + 1, case["prefill"]).tolist() if case["prefill"] else []
    ctx = r.integers(case["ctx_lo"], case["ctx_hi"] + 1, case["decode"]).tolist() if case["decode"] else []
    return wl.BatchSpec(q + [1] * len(ctx), c + ctx)


def _parts(case):
    """The stage steps of one pass: (step case, flags, conditioned, how often)."""
    if case["kind"] == "step":
        return [(case, B.HS_FLAG_BF16_ACTIVATIONS if case["bf16"] else 0, False, 1)]
    if case["kind"] == "dit":
        n = case["tokens"]
        c = _step("", "c6_dit", prefill=case["images"], chunk_lo=n, chunk_hi=n, budget=case["budget"])
        return [(c, B.HS_FLAG_BIDIRECTIONAL, True, 1)]
    a = _step("", "c2_shared", prefill=case["prefill"], chunk_lo=128, chunk_hi=1024, decode=case["decode"], ctx_lo=256,
              ctx_hi=2048, lens=case["lens"], budget=case["budget"])
    b = _step("", "c4_talker", decode=case["talkers"], ctx_lo=128, ctx_hi=1024, lens=case["lens"] + 1,
              budget=FULL - case["budget"])
    return [(a, 0, False, 1), (b, 0, False, case["talker_steps"])]


# --- state ---------------------------------------------------------------------------------------------------------
class _StageState:
    """A stage with weights, a cache that earlier steps have filled, the block tables and the next tick's rows."""

    def __init__(self, case, flags, conditioned, seed):
        dev = torch.device("cuda", torch.cuda.current_device())
        dims, batch = _dims(case), _batch(case)
        total = batch.total_len()
        mpps = max(-(-t // PAGE) for t in total)
        self.stage = Stage(dims, wl.make_weights(dims, seed, dev, "depth_scaled"), wl.pages_needed(batch) + 8,
                           batch.n_tokens, batch.n_seqs, mpps, max(total), dev.index, flags)
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed + 1)
        for layer in self.stage.kv_pool_view():
            layer.normal_(generator=gen)
        for s, t in enumerate(batch.ctx_len):           # pages of the context first, the new tokens' behind them
            if t:
                self.stage.kv_alloc(s, t)
        self.tables = self.stage.block_table_array([self.stage.kv_alloc(s, t) for s, t in enumerate(total)])
        if conditioned:
            self.stage.set_modulation(wl.make_modulation(dims, batch.n_seqs, seed, dev))
        if case["bias"]:
            for l in range(dims.n_layers):
                b = [(0.1 * torch.randn(n, generator=gen, device=dev)).to(torch.bfloat16)
                     for n in (dims.q_dim, dims.kv_dim, dims.kv_dim)]
                self.stage.set_qkv_bias(l, *b)
        self.batch, self.budget = batch, min(case["budget"], self.stage.sm_count)
        self.x = wl.make_x(batch.n_tokens, dims.d_model, seed, dev)
        self.y = torch.empty(batch.n_tokens, dims.d_model, dtype=torch.float32, device=dev)
        self.out = [self.y, *self.stage.kv_pool_view().unbind(0)]      # the cache layer by layer

    def step(self, stream=None):
        b = self.stage.make_batch(self.batch.q_len, self.batch.ctx_len, self.tables, self.x, self.y)
        self.stage.step(b, self.budget, stream)


class _HeadState:
    def __init__(self, case, seed):
        dev = torch.device("cuda", torch.cuda.current_device())
        d, n = wl.DIMS["c3_7b"].d_model, case["rows"]
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        self.n, self.d, self.budget = n, d, case["budget"]
        self.y = torch.randn(2048 + n, d, generator=gen, device=dev)
        self.rows = torch.arange(2048, 2048 + n, dtype=torch.int32, device=dev)
        self.gain = (1.0 + 0.02 * torch.randn(d, generator=gen, device=dev)).to(torch.bfloat16)
        self.w = torch.empty(VOCAB, d, dtype=torch.bfloat16, device=dev).normal_(0.0, 0.02, generator=gen)
        cfg = B.make_head_config(d, VOCAB, 1e-6, 128, dev.index)
        self.ws = torch.empty(B.hs_head_workspace_bytes(cfg), dtype=torch.uint8, device=dev)
        self.head = B.hs_head_create(cfg, self.gain.data_ptr(), self.w.data_ptr(), self.ws.data_ptr())
        self.logits = torch.empty(n, VOCAB, dtype=torch.float32, device=dev)
        self.tokens = torch.empty(n, dtype=torch.int32, device=dev)
        self.x = torch.empty(n, d, dtype=torch.bfloat16, device=dev)
        self.status = torch.zeros(1, dtype=torch.int32, device=dev)
        self.out = [self.logits, self.tokens, self.x]

    def __del__(self):
        if getattr(self, "head", 0):
            B.hs_head_destroy(self.head)


def prepare(case, seed):
    if case["kind"] == "head":
        return case, _HeadState(case, seed)
    parts = [_StageState(c, flags, cond, seed + 7919 * i) for i, (c, flags, cond, _) in enumerate(_parts(case))]
    if case["kind"] == "corun":
        return case, parts, [torch.cuda.Stream(), torch.cuda.Stream()], [t for p in parts for t in p.out]
    return case, parts[0]


def run(state):
    case = state[0]
    if case["kind"] == "head":
        s = state[1]
        stream = torch.cuda.current_stream().cuda_stream
        B.hs_head_step(s.head, s.y.data_ptr(), s.rows.data_ptr(), s.n, s.logits.data_ptr(), s.tokens.data_ptr(), s.budget,
                       stream)
        B.hs_op_embed(s.tokens.data_ptr(), s.n, s.w.data_ptr(), VOCAB, s.d, s.x.data_ptr(), s.budget,
                      s.status.data_ptr(), stream)
        return s.out
    if case["kind"] == "corun":
        (a, b), (sa, sb), out = state[1:]
        here = torch.cuda.current_stream()
        sa.wait_stream(here)
        sb.wait_stream(here)
        a.step(sa)
        for _ in range(case["talker_steps"]):
            b.step(sb)
        here.wait_stream(sa)
        here.wait_stream(sb)
        return out
    state[1].step()
    return state[1].out


# --- the same outputs in 64 bits, in plain torch ------------------------------------------------------------------------
def _rms(x, gain, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain


def _rope(v, pos, base):                                   # [tokens, heads, Dh], rotate-half pairs (i, i + Dh / 2)
    half = v.shape[-1] // 2
    theta = torch.pow(base, -torch.arange(half, dtype=torch.float64, device=v.device) / half)
    ang = pos.double()[:, None, None] * theta
    a, b, cos, sin = v[..., :half], v[..., half:], ang.cos(), ang.sin()
    return torch.cat((a * cos - b * sin, b * cos + a * sin), -1)


def _pages(batch):
    """Every sequence's pages: handed out in order, the contexts' first, then the ones the new tokens grow into."""
    nxt, tables = 0, [[] for _ in batch.q_len]
    for lens in (batch.ctx_len, batch.total_len()):
        for s, t in enumerate(lens):
            while len(tables[s]) * PAGE < t:
                tables[s].append(nxt)
                nxt += 1
    return tables


def _exact_step(case, flags, conditioned, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    dims, batch = _dims(case), _batch(case)
    Hq, Hk, Dh = dims.n_q_heads, dims.n_kv_heads, dims.head_dim
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed + 1)
    shape = wl.kv_pool_shape(dims, wl.pages_needed(batch) + 8)[1:]
    pool = [torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen) for _ in range(dims.n_layers)]
    bias = [[(0.1 * torch.randn(n, generator=gen, device=dev)).to(torch.bfloat16).double()
             for n in (dims.q_dim, dims.kv_dim, dims.kv_dim)] if case["bias"] else None for _ in range(dims.n_layers)]
    mod = wl.make_modulation(dims, batch.n_seqs, seed, dev).double() if conditioned else None
    seq = torch.repeat_interleave(torch.arange(batch.n_seqs), torch.tensor(batch.q_len)).to(dev)
    pos = torch.cat([torch.arange(c, c + q) for q, c in zip(batch.q_len, batch.ctx_len)]).to(dev)
    pages = [torch.tensor(t, device=dev) for t in _pages(batch)]
    slot = torch.cat([pages[s][torch.arange(c, c + q, device=dev) // PAGE] * PAGE
                      for s, (q, c) in enumerate(zip(batch.q_len, batch.ctx_len))]) + pos % PAGE
    x = wl.make_x(batch.n_tokens, dims.d_model, seed, dev).double()
    out = []
    for l in range(dims.n_layers):
        w = {k: v.double() for k, v in wl.make_layer_weights(dims, seed, l, dev, "depth_scaled").items()}

        def norm(v, gain, first):
            h = _rms(v, gain, dims.rms_eps)
            return h if mod is None else h * (1.0 + mod[l, seq, first + 1]) + mod[l, seq, first]

        def gated(v, which):
            return v if mod is None else v * mod[l, seq, which]

        h = norm(x, w["g_attn"], 0)
        q, k, v = (h @ w[n].T + (bias[l][i] if bias[l] else 0.0) for i, n in enumerate(("w_q", "w_k", "w_v")))
        q = _rope(q.view(-1, Hq, Dh), pos, dims.rope_base)
        k, v = _rope(k.view(-1, Hk, Dh), pos, dims.rope_base), v.view(-1, Hk, Dh)
        whole = pool[l].double()                           # a new key or value is read back in the cache's bf16
        for i, t in enumerate((k, v)):
            whole[i, slot // PAGE, :, slot % PAGE] = t
        pool[l] = None
        o, row = torch.empty_like(q), 0
        for s, (n, c) in enumerate(zip(batch.q_len, batch.ctx_len)):
            keys, vals = (whole[i, pages[s]].to(torch.bfloat16).double().permute(1, 0, 2, 3).reshape(Hk, -1, Dh)[:, :n + c]
                          for i in (0, 1))
            qs = q[row:row + n].view(n, Hk, Hq // Hk, Dh).permute(1, 2, 0, 3)                  # [Hk, G, n, Dh]
            sc = qs @ keys[:, None].transpose(-1, -2) / math.sqrt(Dh)
            if not flags & B.HS_FLAG_BIDIRECTIONAL:
                sc.masked_fill_(torch.arange(n + c, device=dev) > pos[row:row + n, None], -math.inf)
            o[row:row + n] = (sc.softmax(-1) @ vals[:, None]).permute(2, 0, 1, 3).reshape(n, Hq, Dh)
            row += n
        x = x + gated(o.view(-1, dims.q_dim) @ w["w_o"].T, 2)
        h = norm(x, w["g_mlp"], 3)
        x = x + gated((torch.nn.functional.silu(h @ w["w_gate"].T) * (h @ w["w_up"].T)) @ w["w_down"].T, 5)
        out.append(whole)
    return [x, *out]


def exact(case, seed):
    if case["kind"] == "head":
        s = _HeadState(case, seed)
        h = _rms(s.y[s.rows.long()].double(), s.gain.double(), 1e-6)
        return [torch.cat([h @ w.double().T for w in s.w.split(16384)], -1), None, None]
    return [t for i, (c, flags, cond, _) in enumerate(_parts(case)) for t in _exact_step(c, flags, cond, seed + 7919 * i)]


# --- what a pass cannot do without ---------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "head":
        d, n = wl.DIMS["c3_7b"].d_model, case["rows"]
        return {"bytes": VOCAB * d * 2 + n * d * (4 + 2 + 2) + d * 2 + n * VOCAB * 4 + n * 4, "flops": 2.0 * n * d * VOCAB}
    total_bytes = total_flops = 0.0
    for c, flags, cond, times in _parts(case):
        dims, batch = _dims(c), _batch(c)
        T, L = batch.n_tokens, dims.n_layers
        per_key = 2 * dims.kv_dim * 2
        moved = L * (dims.params_per_layer() + 2 * dims.d_model) * 2 + T * dims.d_model * (2 + 4)
        moved += L * per_key * sum(batch.total_len())          # cached keys read once, new ones written once
        if cond:
            moved += L * batch.n_seqs * 6 * dims.d_model * 4
        if flags & B.HS_FLAG_BIDIRECTIONAL:
            pairs = sum(n * (n + x) for n, x in zip(batch.q_len, batch.ctx_len))
        else:
            pairs = sum(x * n + n * (n + 1) / 2.0 for n, x in zip(batch.q_len, batch.ctx_len))
        flops = L * (2.0 * T * dims.params_per_layer() + 4.0 * dims.q_dim * pairs)
        total_bytes += times * moved
        total_flops += times * flops
    return {"bytes": total_bytes, "flops": total_flops}


def tolerance(case):
    """About four times the distance from the same path in float64, over the listed cases: fp16 activations rel 8e-4,
    largest 1.2e-2 (one bf16 step of a cached value, or a few); bf16 activations rel 4e-3, largest 1.7e-2; logits rel
    1.7e-3, largest 8e-3, and two logits closer than that may swap places."""
    if case["kind"] == "head":
        return {"rel": 0.007, "max": 0.035, "differ": 0.01}
    if case.get("bf16"):
        return {"rel": 0.016, "max": 0.08}
    return {"rel": 0.003, "max": 0.05}
