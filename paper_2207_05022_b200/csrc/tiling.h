// How a layer's four GEMMs are cut for a call of so many tokens, where its decoded matrices stand in the working buffer, and
// how many planes of partial sums follow.  Host arithmetic only, also compiled by the tests.
//
// Every rule sees a call's token count rounded up to whole tiles of kTileM: all calls of a step take the same planes, so what
// the largest call of each step needs (partial_rows) is enough for every call.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace sti {

constexpr int kTileM = 128;                 // tokens per MMA tile
constexpr int kChunkK = 64;                 // one TMA box = 64 columns = one 128-byte swizzle row; a stage holds 1, 2 or 4 boxes
constexpr int kBoxBytes = kTileM * kChunkK * 2;     // 16 KB
// header = barriers (256 B) + bias (512 B) + one 128-byte centroid table per warp; stages start 1024-aligned after it
constexpr int kHeaderBytes = 3072;

inline size_t gemm_weight_bytes(uint32_t n_rows, uint32_t k_total) { return static_cast<size_t>(n_rows) * k_total * 2; }

// Ring shape for a weight tile of `w_bytes` and a K range of `k_total`: boxes per stage and stages.
// Fewer, larger stages mean fewer waits for the MMA-issuing warp; at least ~64 KB stay in flight.
inline bool gemm_pick_ring(uint32_t w_bytes, uint32_t k_total, uint32_t hdr_bytes, uint32_t* n_stages, uint32_t* bps) {
  const long room = 227L * 1024 - static_cast<long>(hdr_bytes) - static_cast<long>(w_bytes);
  if (room < 3L * kBoxBytes) return false;           // the tile does not fit
  const uint32_t n_boxes = k_total / kChunkK;
  if (n_boxes <= 8 && room >= 2L * 4 * kBoxBytes) { *bps = 4; *n_stages = 2; return true; }   // a tile's K in <= 2 stages
  if (room >= 3L * 2 * kBoxBytes) { *bps = 2; *n_stages = static_cast<uint32_t>(room / (2 * kBoxBytes) > 4 ? 4 : room / (2 * kBoxBytes)); return true; }
  *bps = 1;
  *n_stages = static_cast<uint32_t>(room / kBoxBytes > 6 ? 6 : room / kBoxBytes);
  return true;
}

// Whether a weight tile of n rows x k columns leaves room for a ring of four boxes.
inline bool tile_fits(int n, int k) {
  uint32_t st = 0, bp = 0;
  return gemm_pick_ring(static_cast<uint32_t>(gemm_weight_bytes(n, k)), k, kHeaderBytes, &st, &bp) && st * bp >= 4;
}

struct Tuning {
  int qkv_n = 32, f1_n = 64, o_n = 64, o_group = 4, f2_n = 64;
  int f2_group = 0;                    // FFN slices per K group of FFN2: 0 = chosen per layer and token count (pick_f2_group)
  int cta_budget = 148;                // (replaced by the device's SM count in parse_tuning) CTAs a GEMM launch may use when it splits the token tiles over CTAs
  int wide_min_tokens = -1;            // weights decoded into the working buffer, GEMMs over it: -1 = by the rule of use_wide, 0 = never, else from this many tokens on
  int f2_one_plane_min_tokens = 4096;  // there, FFN2's K range in one piece (one output plane) from this many tokens on (0 = by cost)
  int wide_nt = 0, wide_splits = 0;    // there, features per tile and K splits: 0 = chosen by pick_wide
  int attn_tc_min_items = -1;          // tensor-core attention: -1 = by the rule of tc_attention, 0 = never, else from this many (sequence, kept head) pairs on, whatever their length
};

// What the rules go by besides a layer's kept units and a call's tokens.
struct Tiling {
  int hidden = 0, slice = 0;           // columns of the model and of an FFN slice
  size_t attn_weights = 0, ffn_weights = 0;   // of a unit
  long long max_tokens = 0;            // of the context
  bool fused_only = false;             // products on the plain ALUs: no working buffer
  Tuning tune;
};

inline long long whole_tiles(long long tokens) { return (tokens + kTileM - 1) / kTileM * kTileM; }

// From how many tokens on a layer goes through the working buffer: the fused kernels' time grows with every 128-token tile, that
// of the GEMMs over the buffer with every two and with the weights they fetch; a layer of BERT-large's size is ahead from
// four tiles on, a smaller one from five (us per layer in a model / in a call by itself, fused against buffer: BERT-large 1 x 256
// 38.6 / - against 40.5, 5 x 77 48.8 / 49.5 against 44.9 / 48.1, 4 x 128 50.1 / 50.7 against 46.1 / 49.3, 5 x 128 55.2 / 57.5
// against 50.6 / 55.2; BERT-base 5 x 77 37.7 / 38.8 against 37.4 / 42.7, 4 x 128 37.7 / 38.9 against 38.1 / 42.7, 5 x 128
// 41.9 / 45.2 against 40.5 / 43.2, 8 x 128 51.2 / 53.4 against 45.2 / 49.3).
constexpr int kWideTokens = 513, kWideTokensLarge = 385;
constexpr size_t kWideLargeWeights = 8u << 20;

// Token counts are told apart in tiles of 128, and no further than where the working buffer takes over.
inline int f2_tiles(const Tiling& t, long long tokens) {
  long long most = t.max_tokens;
  if (t.tune.wide_min_tokens != 0) most = std::min<long long>(most, t.tune.wide_min_tokens > 0 ? t.tune.wide_min_tokens : kWideTokens);
  return static_cast<int>(whole_tiles(std::max(1LL, std::min(tokens, most))) / kTileM);
}

// FFN slices per K group of FFN2 in a layer that keeps `ns` of them, for calls of `n_mtiles` token tiles.  More slices per group:
// fewer fp32 planes written and read back by the LayerNorm (8 bytes per element at 5 TB/s), but a longer MMA chain per CTA
// (0.7 us per 256 columns and 128-token tile) and a longer decode, of which
// other kernels leave about 1.4 us per 256 columns in the open; and a launch that fills every SM delays its neighbours (1 us).
// Groups of more than 1024 columns leave the ring too little: five slices of 256 took 57.0 -> 61.6 us (a BERT-base layer of
// 9 slices, 1536 tokens).  Fitted to 91 timings with 1 to 6 slices per group, 6 to 16 slices kept, 64 to 4000 tokens: its choice
// is 0.5 % above the best one in the mean, 4.2 % at most (us per layer with 2 / 3 / 4 slices: BERT-large, 16 slices, 256 tokens
// 38.6 / 37.2 / 38.7, 1024 68.4 / 69.2 / 64.1; 12 slices, 256 tokens 35.0 / 37.0 / 36.0; BERT-base, 128 tokens 27.3 / 27.7 / 28.3).
inline int pick_f2_group(const Tiling& tiling, int ns, int n_mtiles) {
  const Tuning& t = tiling.tune;
  if (t.f2_group > 0) return t.f2_group;
  const int f = tiling.slice;
  int best = 1;                        // also where no more than one slice fits in shared memory
  double best_cost = -1.0;
  for (int g = std::max(1, std::min(2, ns)); g <= ns; ++g) {
    if (g > 1 && (g * f > 1024 || !tile_fits(t.f2_n, g * f))) break;
    const int planes = (ns + g - 1) / g, widest = (ns + planes - 1) / planes, jobs = planes * (tiling.hidden / t.f2_n);
    const int m_ctas = std::max(1, std::min(n_mtiles, t.cta_budget / jobs)), tiles = (n_mtiles + m_ctas - 1) / m_ctas;
    const double filled = static_cast<double>(jobs) * m_ctas / t.cta_budget;
    const double cost = std::max(1.0, filled) * widest * (f / 256.0) * (tiles * 0.7 + 1.4) +
                        planes * 128.0 * n_mtiles * tiling.hidden * 8.0 / 5.0e6 + std::min(1.0, filled);
    if (best_cost < 0.0 || cost < best_cost) { best = g; best_cost = cost; }
  }
  return best;
}

// Calls of many tokens: decode the layer into the working buffer, then GEMMs over it.
inline bool use_wide(const Tiling& t, int heads, int slices, long long tokens) {
  if (t.tune.wide_min_tokens == 0 || t.fused_only) return false;
  if (t.tune.wide_min_tokens > 0) return tokens >= t.tune.wide_min_tokens;
  const size_t weights = static_cast<size_t>(heads) * t.attn_weights + static_cast<size_t>(slices) * t.ffn_weights;
  return tokens >= (weights >= kWideLargeWeights ? kWideTokensLarge : kWideTokens);
}

// One of a layer's weight matrices in the working buffer (expand.cu).
struct WideMatrix {
  uint32_t row0 = 0;                   // first 128-byte row
  uint32_t n = 0, k_chunks = 0;        // features, chunks of 64 columns
};

// Tiles of a GEMM over the working buffer: cycles of the chunks of every wave, of the last tile's epilogue and of the fp32 planes
// that K splits add (written, and read by the LayerNorm).  Fitted to 22 shapes of 256 to 4096 tokens, both models, one to four splits;
// within 2 % of the best of them (us per BERT-large layer with 256-wide tiles and 1 / 2 / 3 / 4 splits: 1024 tokens 69.1 / 59.5 / 57.4 /
// 56.4, picked 57.2; 2048 tokens 83.9 / 75.2 / 82.1 / 81.1, picked 74.4; with 128-wide ones 64.2 / 58.2 / 62.1 / 61.2 and 82.3 / 85.5 /
// 88.9 / 92.3; 512 tokens, 128 wide, 59.5 / 52.3 / 49.8 / 49.7, picked 51.1).
struct WideChoice { uint32_t nt, splits, clusters; };
inline WideChoice pick_wide(const Tiling& tiling, long long call_tokens, const WideMatrix& m, bool may_split) {
  const Tuning& t = tiling.tune;
  const long long tokens = whole_tiles(call_tokens);      // the planes' cost by the step, too: see above
  const uint32_t pairs = static_cast<uint32_t>((tokens + 255) / 256), held = static_cast<uint32_t>(std::max(1, t.cta_budget / 2));
  WideChoice best{256, 1, 1};
  double best_cost = -1.0;
  for (uint32_t nt = 256; nt >= 128; nt /= 2) {
    if (t.wide_nt > 0 && nt != static_cast<uint32_t>(t.wide_nt)) continue;
    for (uint32_t splits = 1; splits <= (may_split ? 4u : 1u) && splits <= m.k_chunks; ++splits) {
      if (may_split && t.wide_splits > 0 && splits != std::min(static_cast<uint32_t>(t.wide_splits), m.k_chunks)) continue;
      const uint32_t tiles = pairs * ((m.n + nt - 1) / nt) * splits, waves = (tiles + held - 1) / held;
      const double cost = waves * ((m.k_chunks + splits - 1) / splits * (nt == 256 ? 540.0 : 400.0) + 500.0) + (nt == 256 ? 1500.0 : 1000.0) +
                          (splits - 1) * 8.0 * tokens * m.n / 2500.0;
      if (best_cost < 0.0 || cost < best_cost) { best = {nt, splits, std::min(tiles, held)}; best_cost = cost; }
    }
  }
  return best;
}
// FFN2 and the O projection write fp32 planes, one per K split.
inline WideChoice pick_wide_f2(const Tiling& t, long long tokens, const WideMatrix& m) {
  return pick_wide(t, tokens, m, !(t.tune.f2_one_plane_min_tokens > 0 && whole_tiles(tokens) >= t.tune.f2_one_plane_min_tokens));
}

// Sizes and places of a layer's matrices (QKV, O, FFN1, FFN2) in its working buffer; the buffer's rows of 128 bytes.  A matrix has
// one place in all of a plan's layers, as large as the widest of them needs (`most_heads`, `most_slices`): the warps that decode
// ahead write while the kernel before theirs may still read, and what that one reads is never the same matrix (gemm_wide.cu).
inline uint32_t place_wide(const Tiling& t, int heads, int slices, int most_heads, int most_slices, WideMatrix (&wide)[4]) {
  const uint32_t d = static_cast<uint32_t>(t.hidden);
  uint32_t row = 0;
  for (int m = 0; m < 4; ++m) {
    auto features = [&](int h, int s) { return m == 0 ? 192u * h : m == 2 ? static_cast<uint32_t>(t.slice * s) : d; };
    auto columns = [&](int h, int s) { return m == 1 ? 64u * h : m == 3 ? static_cast<uint32_t>(t.slice * s) : d; };
    wide[m] = {row, features(heads, slices), columns(heads, slices) / 64};
    row += (features(most_heads, most_slices) + 255) / 256 * 256 * (columns(most_heads, most_slices) / 64);       // whole tiles of 256 features
  }
  return row;
}

// Planes of partial sums that the O projection and FFN2 of a layer write in a call of `tokens` tokens.
struct SumPlanes { int o, f2; };
inline SumPlanes sum_planes(const Tiling& t, int heads, int slices, long long tokens) {
  if (use_wide(t, heads, slices, tokens)) {
    WideMatrix wide[4];
    (void)place_wide(t, heads, slices, heads, slices, wide);
    return {heads > 0 ? static_cast<int>(pick_wide(t, tokens, wide[1], true).splits) : 0,
            slices > 0 ? static_cast<int>(pick_wide_f2(t, tokens, wide[3]).splits) : 0};
  }
  const int group = pick_f2_group(t, slices, f2_tiles(t, tokens));
  return {(heads + t.tune.o_group - 1) / t.tune.o_group, (slices + group - 1) / group};
}

// Rows of `hidden` partial sums that the calls of a context need at most for this layer.  Within a step of kTileM tokens only
// the way through the working buffer or not can change, once: the step's first and last call show both, and the last one's tokens
// bound every call's.
inline size_t partial_rows(const Tiling& t, int heads, int slices) {
  size_t rows = 1;
  for (long long first = 1; first <= t.max_tokens; first += kTileM) {
    const long long last = std::min<long long>(first + kTileM - 1, t.max_tokens);
    for (long long tokens : {first, last}) {
      const SumPlanes p = sum_planes(t, heads, slices, tokens);
      rows = std::max(rows, static_cast<size_t>(last) * static_cast<size_t>(std::max(p.o, p.f2)));
    }
  }
  return rows;
}

}  // namespace sti
