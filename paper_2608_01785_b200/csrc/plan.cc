// Host-only logic of the stage: configuration checks, the page allocator, and the per-step planner
// that turns a batch descriptor into the integer metadata the kernels consume.  Nothing that a result depends on
// depends on the SM budget, which is what keeps results identical across budgets; only how many (independent) Q tiles a
// prefill item carries and the two attention kernels' shares of the budget do.
#include <algorithm>
#include <numeric>

#include "hs_internal.h"

namespace hs {

hs_status_t validate_config(const hs_stage_config_t& c) {
  if (c.abi_version != HS_ABI_VERSION || (c.flags & ~(HS_FLAG_BF16_ACTIVATIONS | HS_FLAG_BIDIRECTIONAL)) != 0) return HS_ERR_INVALID_ARG;
  if (c.n_layers < 1 || c.d_model < 64 || c.n_q_heads < 1 || c.n_kv_heads < 1 || c.d_ffn < 64) return HS_ERR_INVALID_ARG;
  if (c.num_pages < 1 || c.max_tokens < 1 || c.max_seqs < 1 || c.max_pages_per_seq < 1 || c.max_position < 1)
    return HS_ERR_INVALID_ARG;
  if (c.max_seqs > c.max_tokens) return HS_ERR_INVALID_ARG;
  if (!(c.rms_eps >= 0.f) || !(c.rope_base > 1.f)) return HS_ERR_INVALID_ARG;
  if (c.page_size != kPage) return HS_ERR_UNSUPPORTED_SHAPE;
  if (c.head_dim != 64 && c.head_dim != 128) return HS_ERR_UNSUPPORTED_SHAPE;
  if (c.n_q_heads % c.n_kv_heads != 0 || c.n_q_heads / c.n_kv_heads > 16) return HS_ERR_UNSUPPORTED_SHAPE;
  // A 128-wide half of a GEMM tile must lie inside one of q / k / v
  if ((c.n_q_heads * c.head_dim) % 128 != 0 || (c.n_kv_heads * c.head_dim) % 128 != 0) return HS_ERR_UNSUPPORTED_SHAPE;
  // 16-byte rows for tiled copies and vector stores
  if (c.d_model % 8 != 0 || c.d_ffn % 8 != 0) return HS_ERR_UNSUPPORTED_SHAPE;
  // total rows of the pool as seen by a tiled copy must fit a 32-bit coordinate
  const int64_t rows = int64_t(c.n_layers) * 2 * c.num_pages * c.n_kv_heads * kPage;
  if (rows >= (int64_t(1) << 31)) return HS_ERR_UNSUPPORTED_SHAPE;
  return HS_OK;
}

// ------------------------------------------------------------------ pages --
PageAllocator::PageAllocator(int num_pages) {
  free_.resize(num_pages);
  for (int i = 0; i < num_pages; ++i) free_[i] = num_pages - 1 - i;
}

hs_status_t PageAllocator::grow(int64_t seq, int total_tokens, const std::vector<int32_t>** table) {
  auto it = owned_.find(seq);
  const int have = it == owned_.end() ? 0 : static_cast<int>(it->second.size());
  const int need = ceil_div(total_tokens, kPage) - have;
  if (need > static_cast<int>(free_.size())) return HS_ERR_OUT_OF_PAGES;
  std::vector<int32_t>& pages = owned_[seq];
  for (int i = 0; i < need; ++i) {
    pages.push_back(free_.back());
    free_.pop_back();
  }
  *table = &pages;
  return HS_OK;
}

hs_status_t PageAllocator::release(int64_t seq) {
  auto it = owned_.find(seq);
  if (it == owned_.end()) return HS_ERR_UNKNOWN_SEQ;
  for (auto p = it->second.rbegin(); p != it->second.rend(); ++p) free_.push_back(*p);
  owned_.erase(it);
  return HS_OK;
}

// --------------------------------------------------------- step metadata --
MetaLayout make_meta_layout(const hs_stage_config_t& c) {
  MetaLayout m{};
  const int G = c.n_q_heads / c.n_kv_heads;
  m.max_prefill_items = c.n_kv_heads * (c.max_tokens / prefill_tokens_per_item(G) + c.max_seqs);
  // a decode sequence of n keys has at most n / kDecodeSplit whole runs and kDecodeSplitMax / kDecodeTail pieces of a
  // last, incomplete one; cached keys are bounded by the pool.  (At least eight items for each SM of the device, so that a
  // small batch may be cut into slices finely; not into items of single warps, whose partial results one warp merges, 0.4 us
  // each: with that room a few sequences beyond 4096 keys were runs of 128 keys instead of 256, at 7B dimensions, 2 layers, one
  // of 8000 keys 257 -> 274 us per step, of 32000 351 -> 458.)
  m.max_warp_items = c.n_kv_heads * (c.max_seqs * 2 * (kDecodeSplitMax / kDecodeTail) + int((int64_t(c.num_pages) * kPage) / kDecodeSplit) + 1);
  m.max_decode_items = std::max(kMaxDecodeSlices * kDecodeWarps, m.max_warp_items);
  int off = 0;
  auto take = [&](int n) {
    int o = off;
    off += (n + 3) & ~3;   // keep every array 16-byte aligned
    return o;
  };
  m.tok_pos = take(c.max_tokens);
  m.tok_slot = take(c.max_tokens);
  m.tok_seq = take(c.max_tokens);
  m.seq_tok0 = take(c.max_seqs);
  m.seq_ctx = take(c.max_seqs);
  m.seq_qlen = take(c.max_seqs);
  m.block_tables = take(c.max_seqs * c.max_pages_per_seq);
  m.decode_rows = take(c.max_seqs * 4);
  m.counters = take(c.n_layers * 2);
  m.group_done = take(c.max_seqs * c.n_kv_heads);
  m.prefill_items = take(m.max_prefill_items * 8);    // (last: only what a step has of them travels)
  m.decode_items = take(m.max_decode_items * 8);
  m.total = off;
  return m;
}

int decode_items_of(int keys, int split) { return keys / split + ceil_div(keys % split, kDecodeTail); }

int pick_decode_split(const hs_stage_config_t& c, const hs_batch_t& b, int sm_count, int max_items) {
  // Every warp of the decode kernel works through whole items, longest first.  In units of the time a warp needs for
  // one page an item costs its pages + 8 (queue, record, page ids, first bytes, partial result, its share of the
  // merge), the whole runs are handed out in rounds -- a short last round leaves most warps idle for a whole item --
  // and the pieces of the incomplete runs fill what the last round leaves free, or add rounds of their own:
  //   cost = rounds x (pages per run + 8) + further rounds of pieces x (pages per piece + 8),
  //   rounds = ceil(whole runs / (0.97 x warps of the device)).
  // Measured on B200, 64 sequences of 512..4096 keys, 4 KV heads (model in brackets): 256 keys 72.6 us (72), 384 keys
  // 67.1 (64), 512 keys 77.8 (80); 16 sequences of 300..800 keys: 128 keys 17 us, 256 keys 21 us.
  const int64_t W = int64_t((sm_count > 0 ? sm_count : 148) * kDecodeWarps) * 97 / 100;
  const int piece_cost = kDecodeTail / kPage + 8;
  int best = kDecodeSplit;
  double best_cost = 1e30;
  for (int split = kDecodeTail; split <= kDecodeSplitMax; split += 128) {
    int64_t whole = 0, pieces = 0;
    for (int s = 0; s < b.n_seqs; ++s)
      if (b.q_len[s] == 1) {
        const int keys = b.ctx_len[s] + 1;
        whole += int64_t(c.n_kv_heads) * (keys / split);
        pieces += int64_t(c.n_kv_heads) * ceil_div(keys % split, kDecodeTail);
      }
    if (whole + pieces == 0) return kDecodeSplit;
    if (whole + pieces > max_items) continue;          // (only the smallest size can exceed the buffers)
    const int run_cost = split / kPage + 8;
    const int64_t rounds = (whole + W - 1) / W;
    const int64_t absorbed = (rounds * W - whole) * (run_cost / piece_cost);
    const int64_t left = pieces > absorbed ? pieces - absorbed : 0;
    const double cost = double(rounds * run_cost + (left + W - 1) / W * piece_cost);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = split;
    }
  }
  return best;
}

namespace {
// Work of the prefill attention with one or two Q tiles per item: items, 64-key blocks over all of them, longest item.
struct PrefillWork { int64_t items = 0, blocks = 0; int longest = 0; };
PrefillWork prefill_work(const hs_stage_config_t& c, const hs_batch_t& b, int item_tokens) {
  PrefillWork w;
  for (int s = 0; s < b.n_seqs; ++s) {
    const int n = b.q_len[s], ctx = b.ctx_len[s];
    if (n < 2) continue;
    for (int t0 = 0; t0 < n; t0 += item_tokens) {
      const int keys = (c.flags & HS_FLAG_BIDIRECTIONAL) ? ctx + n : ctx + std::min(t0 + item_tokens, n), blocks = ceil_div(keys, 64);
      w.items += c.n_kv_heads;
      w.blocks += int64_t(c.n_kv_heads) * blocks;
      w.longest = std::max(w.longest, blocks);
    }
  }
  return w;
}

// Split of the SM budget between the two attention kernels when a step has both kinds of work (decode_sms = 0: one after
// the other).  The decode kernel is bound by the K / V bytes it streams, the prefill kernel by its key blocks; with the
// rates measured on B200 (about 42 GB/s per SM up to 5.5 TB/s; 1.15 us per block of an item; 12 us per launch)
//   t_decode(b) = 12 + bytes / min(5.5e6, 42e3 b)    t_prefill(b) = 12 + 1.15 max(longest item, blocks / b)   [us]
// and the split is the one with the smallest larger time, taken only if that beats running them in turn by 8 %.
// Items of one tile (`singles`) take 2 us less but load their key blocks for one tile only, so they are taken only where
// every one has an SM of the kernel's share to itself.
// It moves work between SMs, never between results: both kernels give the same bits at any grid size.
struct AttnSplit { int decode_sms; double us; };
// Two-tile items: the choice between side by side and in turn stands, but the SMs are then shared out by what the kernels
// take beyond that -- the prefill kernel 5.6 us an item beside its 1.13 us a block; the decode kernel in group mode
// (`groups` blocks) whole rounds of its longest group, 0.85 us per page of a warp.  Beside items of single warps that stream
// more than 150 MB a layer, and so from the HBM for as long as they run, not from the L2, the prefill kernel takes 1.3 of that.
// Measured on B200, us per step without -> with the 1.3: 302 MB (64 decode rows at 7B dimensions, 4 layers) beside 2048 new
// tokens on 148 / 120 SMs 3568 -> 3472, 4745 -> 4642, beside 1024 on 112 / 74 2855 -> 2816, 3163 -> 3093; 188 MB (40 rows) beside
// 394 on 148 / 74 1078 -> 1074, 1620 -> 1609; 123 MB (80 rows of a small backbone) beside 5600 on 112 2485 -> 2519; 12 MB (8 rows,
// one of them of 4200 keys) beside 600 on 112 626 -> 644.
AttnSplit split_attention(const PrefillWork& w, bool singles, int64_t decode_kv_bytes, int budget, bool side_by_side, int groups,
                          int longest_pages) {
  auto t_dec = [&](int b) { return decode_kv_bytes > 0 ? 12.0 + double(decode_kv_bytes) / std::min(5.5e6, 42e3 * b) : 0.0; };
  auto t_pre = [&](int b) {
    if (singles) return w.items <= b ? 10.0 + 1.15 * w.longest : 1e30;
    return 12.0 + 1.15 * std::max(double(w.longest), double(w.blocks) / b);
  };
  const double in_turn = t_dec(budget) + t_pre(budget);
  AttnSplit r{0, in_turn};
  if (decode_kv_bytes == 0 || w.items == 0 || budget < 16 || !side_by_side) return r;
  double best = 0.92 * in_turn;
  for (int b = 4; b <= budget - 4; ++b) {
    const double t = std::max(t_dec(b), t_pre(budget - b));
    if (t < best) { best = t; r = AttnSplit{b, t}; }
  }
  if (r.decode_sms > 0 && !singles) {
    const double beside = groups == 0 && decode_kv_bytes > int64_t(150) * 1000000 ? 1.3 : 1.0;
    best = 1e30;
    for (int b = 4; b <= budget - 4; ++b) {
      const double pre = 9.0 + beside * std::max(5.6 + 1.13 * w.longest, (5.6 * double(w.items) + 1.13 * double(w.blocks)) / (budget - b));
      const double dec = groups ? 4.0 + ceil_div(groups, b) * (2.0 + 0.85 * ceil_div(longest_pages, kDecodeWarps)) : t_dec(b);
      if (std::max(pre, dec) < best - 1e-9) { best = std::max(pre, dec); r.decode_sms = b; }
    }
  }
  return r;
}
// Pages per slice of the decode attention's group mode, 0 = items of single warps instead.  One slice per group where every
// group has a block of its own and 128-key items would leave warps idle; in a decode-only step more, all with a block of
// their own on the device, where that is expected to be faster.  Modelled time of a launch: rounds of one slice per SM, each
// Dh / 16 - 2 us, a step of Dh / 272 us per page of a warp and 1.9 us where a group's slices are merged (fitted to steps of 1 to
// 32 rows of three stages, 1 to 8 cuts, 28 to 148 SMs); on the whole device and, with a weight of 0.1 each, on 13/16, 3/4,
// 13/20, 1/2, 7/20 and 1/4 of it, since the results depend on the cut and it must not depend on the budget; a cut has to gain a
// twenty-fifth.  Measured on B200, us per step on 148 / 74 / 37 SMs, one slice -> the cut taken: a row of 4000 keys at 7B
// dimensions, 2 layers, 242 -> 220, 289 -> 266, 425 -> 402; five of up to 3142 241 -> 232, 289 -> 279, 424 -> 434; nine of up to
// 3747 252 -> 241, 301 -> 314, 440 -> 472 (the one step of these where the whole device has the better of it); on a small
// backbone eight of up to 1931 192 -> 183, 248 -> 235, 357 -> 343, cut four times 180, 232 and 377; 32 of them stay whole (cut in
// two 258 for 257, 370 for 332, 509 for 481).  Never for sequences longer than eight warps' 32 pages: those are so many keys
// that items of single warps fill the device.
int pick_decode_slice(const hs_stage_config_t& c, const hs_batch_t& b, int sm_count, int split) {
  const int sms = std::min(sm_count > 0 ? sm_count : 148, kMaxDecodeSlices);
  int longest = 0, rows = 0;
  for (int s = 0; s < b.n_seqs; ++s)
    if (b.q_len[s] == 1) { ++rows; longest = std::max(longest, ceil_div(b.ctx_len[s] + 1, kPage)); }
  if (split != kDecodeTail || rows == 0 || rows * c.n_kv_heads > sms || longest > kDecodeWarps * 32) return 0;
  int best = longest;
  double best_us = 1e30;
  for (int cuts = 1; cuts <= (rows < b.n_seqs ? 1 : 8); ++cuts) {
    const int pages = ceil_div(longest, cuts);
    int n = 0;
    for (int s = 0; s < b.n_seqs; ++s)
      if (b.q_len[s] == 1) n += c.n_kv_heads * ceil_div(ceil_div(b.ctx_len[s] + 1, kPage), pages);
    if (n > sms) break;
    double us = 0.0;
    const double round_us = c.head_dim / 16.0 - 2.0 + ceil_div(pages, kDecodeWarps) * c.head_dim / 272.0 + (cuts > 1 ? 1.9 : 0.0);
    for (const int eightieths : {80, 65, 60, 52, 40, 28, 20})
      us += (eightieths == 80 ? 1.0 : 0.1) * ceil_div(n, std::max(1, sms * eightieths / 80)) * round_us;
    if (us < best_us * (cuts > 1 ? 0.96 : 1.0)) { best_us = us; best = pages; }
  }
  return best;
}
}  // namespace

hs_status_t plan_step(const hs_stage_config_t& c, const MetaLayout& ml, const hs_batch_t& b, int sm_count, int sm_budget,
                      bool side_by_side, std::vector<int32_t>& page_stamp, int32_t stamp, int32_t* meta,
                      int32_t* tok_seq, StepPlan* plan) {
  if (!b.q_len || !b.ctx_len || !b.block_tables) return HS_ERR_INVALID_ARG;
  if (b.n_seqs < 1 || b.n_seqs > c.max_seqs || b.n_tokens < 1 || b.n_tokens > c.max_tokens) return HS_ERR_INVALID_ARG;
  const int mpps = c.max_pages_per_seq;
  int64_t total = 0;
  for (int s = 0; s < b.n_seqs; ++s) {
    if (b.q_len[s] < 1 || b.ctx_len[s] < 0) return HS_ERR_INVALID_ARG;
    if (int64_t(b.ctx_len[s]) + b.q_len[s] > c.max_position) return HS_ERR_INVALID_ARG;
    total += b.q_len[s];
  }
  if (total != b.n_tokens) return HS_ERR_INVALID_ARG;
  // block tables: enough pages, ids in range, no page named twice in this step
  for (int s = 0; s < b.n_seqs; ++s) {
    const int need = ceil_div(b.ctx_len[s] + b.q_len[s], kPage);
    if (need > mpps) return HS_ERR_BAD_BLOCK_TABLE;
    for (int i = 0; i < need; ++i) {
      const int32_t pg = b.block_tables[size_t(s) * mpps + i];
      if (pg < 0 || pg >= c.num_pages) return HS_ERR_BAD_BLOCK_TABLE;
      if (page_stamp[pg] == stamp) return HS_ERR_BAD_BLOCK_TABLE;
      page_stamp[pg] = stamp;
    }
  }

  const int G = c.n_q_heads / c.n_kv_heads;
  const int Mt = prefill_tokens_per_item(G);
  int split = pick_decode_split(c, b, sm_count, ml.max_decode_items);
  // Group mode of the decode attention: in a batch small enough, every group = (sequence, KV head) is cut into equal
  // slices of whole pages such that all slices have a block of their own on the device; a block's eight warps share a
  // slice, and the block that delivers a group's last slice merges the group's (attention_decode.cuh).  A function of the
  // batch and the device's SM count, never of the budget.
  const int slice_pages = pick_decode_slice(c, b, sm_count, split);
  const bool group_mode = slice_pages > 0;
  if (!group_mode) split = pick_decode_split(c, b, sm_count, ml.max_warp_items);
  StepPlan p;
  p.n_tokens = b.n_tokens;
  p.n_seqs = b.n_seqs;
  // Tokens per prefill item: two Q tiles that share their key blocks, or one.  An item's tiles are independent rows, so the
  // results are the same bits (every budget sweep of the GPU tests crosses the line) and the choice may look at the
  // budget: it is the form whose attention is expected to end first with the SMs the prefill kernel gets.  Measured on
  // B200, two tiles -> one (us per step): denoising stage, 12 layers, 128 items of one tile, on 148 SMs 1009 -> 998, on 96
  // 1140 -> 1167, on 37 1870 -> 1925; at 7B dimensions, 2 layers, 7 decode rows beside a chunk of 394 tokens (100 items) on
  // 148 SMs 470 -> 466, on 96 662 -> 687, beside one of 100 tokens (28 items) on 148 304 -> 298, on 48 492 -> 519.
  int item_tokens = 2 * Mt;
  {
    for (int s = 0; s < b.n_seqs; ++s)
      if (b.q_len[s] == 1) p.decode_kv_bytes += int64_t(b.ctx_len[s] + 1) * 2 * c.n_kv_heads * c.head_dim * 2;
    const PrefillWork one = prefill_work(c, b, Mt), two = prefill_work(c, b, 2 * Mt);
    const AttnSplit with_one = split_attention(one, true, p.decode_kv_bytes, sm_budget, side_by_side, 0, 0);
    int groups = 0;                                   // (beside prefill work a group is one slice)
    for (int s = 0; s < b.n_seqs; ++s) groups += group_mode && b.q_len[s] == 1 ? c.n_kv_heads : 0;
    const AttnSplit with_two = split_attention(two, false, p.decode_kv_bytes, sm_budget, side_by_side, groups, slice_pages);
    if (with_one.us < with_two.us) item_tokens = Mt;
    p.decode_sms = item_tokens == Mt ? with_one.decode_sms : with_two.decode_sms;
  }

  struct Item { int32_t v[8]; int32_t cost; };
  std::vector<Item> pre;
  struct DecItem { int32_t v[8]; int32_t keys; };
  std::vector<DecItem> dec;
  int n_dec_items = 0, n_dec_rows = 0;
  int t = 0;
  for (int s = 0; s < b.n_seqs; ++s) {
    const int n = b.q_len[s], ctx = b.ctx_len[s];
    if (meta) {
      meta[ml.seq_tok0 + s] = t;
      meta[ml.seq_ctx + s] = ctx;
      meta[ml.seq_qlen + s] = n;
      for (int i = 0; i < mpps; ++i) meta[ml.block_tables + s * mpps + i] = b.block_tables[size_t(s) * mpps + i];
    }
    for (int j = 0; j < n; ++j) {
      const int pos = ctx + j;
      const int slot = b.block_tables[size_t(s) * mpps + pos / kPage] * kPage + pos % kPage;
      if (meta) {
        meta[ml.tok_pos + t + j] = pos;
        meta[ml.tok_slot + t + j] = slot;
        meta[ml.tok_seq + t + j] = s;
      }
      if (tok_seq) tok_seq[t + j] = s;
    }
    if (n == 1 && group_mode) {
      // decode, group mode: per KV head `slices` slices of the sequence's pages, each dealt evenly to eight warps (the last
      // of which may have none)
      const int keys = ctx + 1, pages = ceil_div(keys, kPage), slices = ceil_div(pages, slice_pages);
      if (meta) {
        int32_t* row = meta + ml.decode_rows + n_dec_rows * 4;
        row[0] = s; row[1] = t; row[2] = n_dec_items; row[3] = slices * kDecodeWarps;
      }
      for (int hk = 0; hk < c.n_kv_heads; ++hk)
        for (int i = 0; i < slices; ++i) {
          const int p0 = pages * i / slices, p1 = pages * (i + 1) / slices, per = ceil_div(p1 - p0, kDecodeWarps);
          for (int w = 0; w < kDecodeWarps; ++w) {
            const int k0 = std::min(keys, std::min(p1, p0 + w * per) * kPage), k1 = std::min(keys, std::min(p1, p0 + (w + 1) * per) * kPage);
            dec.push_back(DecItem{{n_dec_rows, hk, k0, k1, s, t, n_dec_items / kDecodeWarps + hk * slices, slices | (i << 16)}, 0});
          }
        }
      n_dec_items += c.n_kv_heads * slices * kDecodeWarps;
      if (slices > 1) p.decode_sliced = 1;
      ++n_dec_rows;
    } else if (n == 1) {
      // decode: keys 0..ctx cut into whole runs of `split` keys and the rest into pieces of kDecodeTail keys; the items
      // of a (sequence, KV head) group keep consecutive partial-result slots in key order, whatever the order the
      // queue hands them out in
      const int keys = ctx + 1, small = kDecodeTail;
      const int n_big = keys / split;
      const int splits = decode_items_of(keys, split);
      if (splits > 0x7fff) return HS_ERR_INVALID_ARG;      // the item record keeps the index within the group in 15 bits
      if (meta) {
        int32_t* row = meta + ml.decode_rows + n_dec_rows * 4;
        row[0] = s; row[1] = t; row[2] = n_dec_items; row[3] = splits;
      }
      for (int hk = 0; hk < c.n_kv_heads; ++hk)
        for (int j = 0; j < splits; ++j) {
          const int k0 = j < n_big ? j * split : n_big * split + (j - n_big) * small;
          const int k1 = j < n_big ? k0 + split : std::min(keys, k0 + small);
          dec.push_back(DecItem{{n_dec_rows, hk, k0, k1, s, t, n_dec_items + hk * splits, splits | (j << 16)}, k1 - k0});
        }
      n_dec_items += c.n_kv_heads * splits;
      ++n_dec_rows;
    } else {
      // a prefill item covers one or two Q tiles of Mt tokens each (the last one may be short)
      for (int t0 = 0; t0 < n; t0 += item_tokens)
        for (int hk = 0; hk < c.n_kv_heads; ++hk) {
          const int nt = std::min(item_tokens, n - t0);
          pre.push_back(Item{{s, hk, t0, nt, ctx, t, n, 0}, ctx + t0 + nt});
        }
    }
    t += n;
  }
  if (int(pre.size()) > ml.max_prefill_items || n_dec_items > ml.max_decode_items) return HS_ERR_INVALID_ARG;
  // longest first, so that the dynamic queue finishes evenly; ties keep batch order
  std::stable_sort(pre.begin(), pre.end(), [](const Item& a, const Item& b2) { return a.cost > b2.cost; });
  // decode items likewise: the long runs first, the short ones fill the end of the kernel
  if (!group_mode) std::stable_sort(dec.begin(), dec.end(), [](const DecItem& a, const DecItem& b2) { return a.keys > b2.keys; });
  if (meta) {
    for (size_t i = 0; i < dec.size(); ++i)
      for (int k = 0; k < 8; ++k) meta[ml.decode_items + int(i) * 8 + k] = dec[i].v[k];
    for (size_t i = 0; i < pre.size(); ++i)
      for (int k = 0; k < 8; ++k) meta[ml.prefill_items + int(i) * 8 + k] = pre[i].v[k];
    for (int i = 0; i < c.n_layers * 2; ++i) meta[ml.counters + i] = 0;
    for (int i = 0; i < c.max_seqs * c.n_kv_heads; ++i) meta[ml.group_done + i] = 0;
  }
  p.n_prefill_items = int(pre.size());
  p.n_decode_items = n_dec_items;
  p.decode_group = group_mode && n_dec_items > 0 ? 1 : 0;
  p.n_decode_rows = n_dec_rows;
  p.meta_words = n_dec_items > 0 ? ml.decode_items + n_dec_items * 8 : ml.prefill_items + int(pre.size()) * 8;
  if (plan) *plan = p;
  return HS_OK;
}

}  // namespace hs
