// Shard quantizer on the device (Section 6: Gaussian outlier-aware dictionary quantization).
//
// Two kernels produce the same output.  quantize_select_kernel (further down, the default) never sorts: the
// clusters are equal-population slices of the sorted order, so all it needs are the 2^k - 1 elements that sit at
// the slice boundaries, which it finds by rank selection.  Units it cannot handle (zero variance, more than
// kSelMaxSeg weights in one selection bin, an inlier range whose ends it does not find, no inlier) are marked and done by
// quantize_units_kernel, the sorting kernel:
//
// One CTA of 1024 threads per shard unit runs the paper's steps in order on the unit's flat fp32 array:
//   1. maximum-likelihood fit of one Gaussian (mean, 1/n variance; fp64 block reductions);
//   2. outliers = weights whose log-likelihood is below -4: their (offset, value) pairs are written in
//      ascending offset order by a stable compaction; the other weights become (sortable key, offset) pairs;
//   3. a least-significant-digit radix sort (4 passes of 8 bits, stable, so equal weights keep their
//      original order) of the pairs between two workspace buffers, 4096 elements per step: every thread
//      holds one element of each of four consecutive 1024-element stripes, ranks come from warp match
//      masks plus a per-(stripe, warp, digit) count table in shared memory;
//   4. 2^k clusters of equal population over the sorted order, cluster c = [floor(c n'/2^k), floor((c+1) n'/2^k)),
//      centroid = arithmetic mean (fp64 sum, rounded once to fp32);
//   5. every weight gets its cluster's k-bit index; an outlier's slot gets the nearest centroid's index
//      (lower index on a tie);
//   6. the indexes are packed into the upload format: index i at stream bits [i k, i k + k), LSB first.
// All decisions that yield integers (outlier test, sort order, cluster of a rank, nearest centroid) are taken
// in fp64 / exact integer arithmetic.  Units are independent: the grid is the number of units.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>
#include <type_traits>

#include "../../include/sti_quantize.h"
#include "outlier_range.h"
#include "sti_device.cuh"

namespace {

namespace cg = cooperative_groups;
using sti::is_outlier;
using sti::pdl_launch_dependents;
using sti::pdl_wait;

constexpr int kQThreads = 1024;
constexpr int kQWarps = kQThreads / 32;

constexpr int kItems = 4;             // elements per thread and chunk; a chunk is 4 stripes of 1024 consecutive elements
constexpr int kSlots = kItems * kQWarps;   // (stripe, warp) pairs of a chunk, in element order

struct QuantShared {
  double red[kQWarps];
  uint32_t hist[256];
  uint32_t base[2][256];
  uint8_t wcount[kSlots][256];       // per chunk: elements of digit d held by (stripe, warp) slot q
  uint16_t woff[kSlots][256];        // per chunk: elements of digit d held by the slots before q
  uint32_t wcnt_in[kSlots], wcnt_out[kSlots];
  uint32_t tot_in, tot_out;
  uint16_t stripe_tot[kItems][256];  // per chunk: elements of digit d in stripe j
  uint32_t bounds[65];
  float cents[64];
};

__device__ __forceinline__ double block_sum(double v, double* red, int tid) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < kQWarps; ++w) t += red[w];
  __syncthreads();
  return t;
}

// Maximum-likelihood mean and 1/n variance in fp64 (n is a multiple of 4; four 16-byte loads in flight per thread).
__device__ __forceinline__ void fit_gaussian(const float* w, uint32_t n, double* red, int tid, double& mu, double& var) {
  double s = 0.0;
  for (uint32_t i0 = 4u * tid; i0 < n; i0 += 16u * kQThreads) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t i = i0 + u * 4u * kQThreads;
      v[u] = i < n ? *reinterpret_cast<const float4*>(w + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      s += (static_cast<double>(v[u].x) + static_cast<double>(v[u].y)) + (static_cast<double>(v[u].z) + static_cast<double>(v[u].w));
  }
  mu = block_sum(s, red, tid) / static_cast<double>(n);
  double q = 0.0;
  for (uint32_t i0 = 4u * tid; i0 < n; i0 += 16u * kQThreads) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t i = i0 + u * 4u * kQThreads;
      v[u] = i < n ? *reinterpret_cast<const float4*>(w + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i0 + u * 4u * kQThreads >= n) continue;
      const double d0 = static_cast<double>(v[u].x) - mu, d1 = static_cast<double>(v[u].y) - mu;
      const double d2 = static_cast<double>(v[u].z) - mu, d3 = static_cast<double>(v[u].w) - mu;
      q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
    }
  }
  var = block_sum(q, red, tid) / static_cast<double>(n);
}

// Order-preserving map of an fp32 bit pattern to an unsigned key (-0 sorts as +0).
__device__ __forceinline__ uint32_t sort_key(float x) {
  uint32_t u = __float_as_uint(x);
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// Lanes of the warp that hold the same 8-bit digit (valid lanes only): eight ballots, a fixed cost whatever
// the number of distinct digits (a hardware match instruction walks the distinct values one by one).
__device__ __forceinline__ uint32_t same_digit_lanes(uint32_t d, bool valid) {
  uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool bit = (d >> b) & 1u;
    const uint32_t bal = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? bal : ~bal;
  }
  return peers;
}
__global__ void __launch_bounds__(kQThreads, 1)
quantize_units_kernel(const float* w_all, uint32_t n, int bits, uint32_t* codes_all, float* cent_all, uint32_t* ooff_all,
                      float* oval_all, uint32_t max_out, uint32_t* n_out_all, uint8_t* ws_all, size_t ws_per_unit,
                      const uint8_t* only_marked) {
  extern __shared__ __align__(16) uint8_t q_smem[];
  QuantShared& sm = *reinterpret_cast<QuantShared*>(q_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t unit = blockIdx.x;
  pdl_wait();                                                         // for the selection kernel's marks
  if (only_marked[unit] == 0) return;                                 // it has done this unit
  const uint32_t K = 1u << bits;
  const float* w = w_all + static_cast<size_t>(unit) * n;
  uint32_t* codes = codes_all + static_cast<size_t>(unit) * (static_cast<size_t>(n) * bits / 32);
  float* cent = cent_all + static_cast<size_t>(unit) * K;
  uint32_t* ooff = ooff_all + static_cast<size_t>(unit) * max_out;
  float* oval = oval_all + static_cast<size_t>(unit) * max_out;
  uint8_t* ws = ws_all + static_cast<size_t>(unit) * ws_per_unit;
  uint32_t* key[2] = {reinterpret_cast<uint32_t*>(ws), reinterpret_cast<uint32_t*>(ws) + 2 * static_cast<size_t>(n)};
  uint32_t* idx[2] = {key[0] + n, key[1] + n};
  uint8_t* codes8 = ws + 16 * static_cast<size_t>(n);

  // ---- 1. Gaussian fit
  double mu, var;
  fit_gaussian(w, n, sm.red, tid, mu, var);
  const double c0 = -0.5 * log(2.0 * 3.14159265358979323846 * var);
  const double inv2var = 1.0 / (2.0 * var);

  // ---- 2. outliers out (ascending offsets), the rest as (key, offset) pairs, both by stable compaction
  uint32_t n_in = 0, n_out = 0;
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (uint32_t start = 0; start < n; start += kItems * kQThreads) {
    float x[kItems];
    bool in[kItems], out[kItems];
    uint32_t m_in[kItems], m_out[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const uint32_t i = start + j * kQThreads + tid;
      x[j] = i < n ? w[i] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const uint32_t i = start + j * kQThreads + tid;
      out[j] = i < n && is_outlier(x[j], mu, inv2var, c0);
      in[j] = i < n && !out[j];
      m_in[j] = __ballot_sync(0xffffffffu, in[j]);
      m_out[j] = __ballot_sync(0xffffffffu, out[j]);
      if (lane == 0) { sm.wcnt_in[j * kQWarps + warp] = __popc(m_in[j]); sm.wcnt_out[j * kQWarps + warp] = __popc(m_out[j]); }
    }
    __syncthreads();
    // exclusive prefix of the 128 slot counts in element order: warp 0, four slots per lane, one shuffle scan
    if (warp == 0) {
      uint32_t a[4], b[4], sa = 0, sb = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) { a[e] = sm.wcnt_in[4 * lane + e]; b[e] = sm.wcnt_out[4 * lane + e]; sa += a[e]; sb += b[e]; }
      uint32_t ia = sa, ib = sb;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ta = __shfl_up_sync(0xffffffffu, ia, o), tb = __shfl_up_sync(0xffffffffu, ib, o);
        if (lane >= o) { ia += ta; ib += tb; }
      }
      uint32_t ea = ia - sa, eb = ib - sb;
#pragma unroll
      for (int e = 0; e < 4; ++e) { sm.wcnt_in[4 * lane + e] = ea; sm.wcnt_out[4 * lane + e] = eb; ea += a[e]; eb += b[e]; }
      if (lane == 31) { sm.tot_in = ia; sm.tot_out = ib; }
    }
    __syncthreads();
    const uint32_t run_in = sm.tot_in, run_out = sm.tot_out;
    uint32_t pre_in[kItems], pre_out[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) { pre_in[j] = sm.wcnt_in[j * kQWarps + warp]; pre_out[j] = sm.wcnt_out[j * kQWarps + warp]; }
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const uint32_t i = start + j * kQThreads + tid;
      if (in[j]) {
        const uint32_t dst = n_in + pre_in[j] + __popc(m_in[j] & lt_mask);
        key[0][dst] = sort_key(x[j]);
        idx[0][dst] = i;
      }
      if (out[j]) {
        const uint32_t dst = n_out + pre_out[j] + __popc(m_out[j] & lt_mask);
        if (dst < max_out) { ooff[dst] = i; oval[dst] = x[j]; }
      }
    }
    n_in += run_in;
    n_out += run_out;
    __syncthreads();
  }
  if (tid == 0) n_out_all[unit] = n_out;

  // ---- 3. stable LSD radix sort of the n_in pairs, 8 bits per pass
  int cur = 0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 8 * pass;
    const uint32_t* ksrc = key[cur];
    const uint32_t* isrc = idx[cur];
    uint32_t* kdst = key[cur ^ 1];
    uint32_t* idst = idx[cur ^ 1];
    if (tid < 256) sm.hist[tid] = 0;
    __syncthreads();
    // one shared-memory atomic per distinct digit of a warp (the high digits of weights fall into a few bins)
    const uint32_t n_in_up = (n_in + 31u) & ~31u;          // whole warps take every iteration (match is warp-wide)
    for (uint32_t i0 = tid; i0 < n_in_up; i0 += 8 * kQThreads) {
      uint32_t kv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { const uint32_t i = i0 + u * kQThreads; kv[u] = i < n_in ? ksrc[i] : 0u; }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t i = i0 + u * kQThreads;
        const uint32_t dg = (kv[u] >> shift) & 255u;
        const uint32_t pm = same_digit_lanes(dg, i < n_in);
        if (i < n_in && (pm & lt_mask) == 0) atomicAdd(&sm.hist[dg], static_cast<uint32_t>(__popc(pm)));
      }
    }
    __syncthreads();
    // exclusive prefix of the histogram -> first destination of every digit
    if (tid < 256) sm.base[0][tid] = sm.hist[tid];
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {
      uint32_t v = 0;
      if (tid < 256 && tid >= o) v = sm.base[0][tid - o];
      __syncthreads();
      if (tid < 256) sm.base[0][tid] += v;
      __syncthreads();
    }
    if (tid < 256) sm.base[0][tid] -= sm.hist[tid];
    __syncthreads();
    int bsel = 0;
    for (uint32_t start = 0; start < n_in; start += kItems * kQThreads) {
      uint32_t kk[kItems], ii[kItems], d[kItems], peers[kItems];
      bool valid[kItems];
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        const uint32_t i = start + j * kQThreads + tid;
        valid[j] = i < n_in;
        kk[j] = valid[j] ? ksrc[i] : 0u;
        ii[j] = valid[j] ? isrc[i] : 0u;
      }
      for (int z = tid; z < kSlots * 256 / 4; z += kQThreads) reinterpret_cast<uint32_t*>(&sm.wcount[0][0])[z] = 0u;
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        d[j] = (kk[j] >> shift) & 255u;
        peers[j] = same_digit_lanes(d[j], valid[j]);
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kItems; ++j)
        if (valid[j] && (peers[j] & lt_mask) == 0) sm.wcount[j * kQWarps + warp][d[j]] = static_cast<uint8_t>(__popc(peers[j]));
      __syncthreads();
      {
        // thread (stripe sj, digit sd): prefix over the stripe's 32 warps; the four stripes run side by side
        const int sj = tid >> 8, sd = tid & 255;
        uint32_t pre = 0;
        for (int ww = 0; ww < kQWarps; ++ww) {
          sm.woff[sj * kQWarps + ww][sd] = static_cast<uint16_t>(pre);
          pre += sm.wcount[sj * kQWarps + ww][sd];
        }
        sm.stripe_tot[sj][sd] = static_cast<uint16_t>(pre);
      }
      __syncthreads();
      if (tid < 256) {
        uint32_t t = 0;
#pragma unroll
        for (int j = 0; j < kItems; ++j) t += sm.stripe_tot[j][tid];
        sm.base[bsel ^ 1][tid] = sm.base[bsel][tid] + t;
      }
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        if (valid[j]) {
          uint32_t dst = sm.base[bsel][d[j]] + sm.woff[j * kQWarps + warp][d[j]] + __popc(peers[j] & lt_mask);
#pragma unroll
          for (int jj = 0; jj < kItems; ++jj)
            if (jj < j) dst += sm.stripe_tot[jj][d[j]];
          kdst[dst] = kk[j];
          idst[dst] = ii[j];
        }
      }
      bsel ^= 1;
      __syncthreads();
    }
    cur ^= 1;
  }
  const uint32_t* ks = key[cur];
  const uint32_t* is = idx[cur];

  // ---- 4. equal-population clusters, centroid = mean
  if (tid <= static_cast<int>(K))
    sm.bounds[tid] = static_cast<uint32_t>(static_cast<uint64_t>(tid) * n_in / K);
  __syncthreads();
  for (uint32_t c = warp; c < K; c += kQWarps) {
    const uint32_t lo = sm.bounds[c], hi = sm.bounds[c + 1];
    double acc = 0.0;
    for (uint32_t r = lo + lane; r < hi; r += 32) acc += static_cast<double>(key_value(ks[r]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      const float m = hi > lo ? static_cast<float>(acc / static_cast<double>(hi - lo)) : 0.f;
      sm.cents[c] = m;
      cent[c] = m;
    }
  }
  __syncthreads();

  // ---- 5. indexes: the cluster of a weight's rank; for an outlier the nearest centroid
  for (uint32_t r0 = tid; r0 < n_in; r0 += 8 * kQThreads) {
    uint32_t dst[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { const uint32_t r = r0 + u * kQThreads; dst[u] = r < n_in ? is[r] : 0u; }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t r = r0 + u * kQThreads;
      if (r >= n_in) continue;
      uint32_t c = r * K / n_in;             // r < 2^26 and K <= 2^6: the product fits 32 bits
      while (c + 1 < K && sm.bounds[c + 1] <= r) ++c;
      while (c > 0 && sm.bounds[c] > r) --c;
      codes8[dst[u]] = static_cast<uint8_t>(c);
    }
  }
  if (n_out > 0) {
    for (uint32_t i0 = tid; i0 < n; i0 += 8 * kQThreads) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { const uint32_t i = i0 + u * kQThreads; v[u] = i < n ? w[i] : 0.f; }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t i = i0 + u * kQThreads;
        if (i >= n || !is_outlier(v[u], mu, inv2var, c0)) continue;
        uint32_t best = 0;
        double bd = fabs(static_cast<double>(v[u]) - static_cast<double>(sm.cents[0]));
        for (uint32_t c = 1; c < K; ++c) {
          const double dd = fabs(static_cast<double>(v[u]) - static_cast<double>(sm.cents[c]));
          if (dd < bd) { bd = dd; best = c; }
        }
        codes8[i] = static_cast<uint8_t>(best);
      }
    }
  }
  __syncthreads();

  // ---- 6. the index stream: 32 consecutive indexes are exactly `bits` words; a thread reads them as two 16-byte
  //         loads and shifts them into a 64-bit window, emitting a word whenever 32 bits are complete
  const uint32_t n_groups = n / 32;
  for (uint32_t gidx = tid; gidx < n_groups; gidx += kQThreads) {
    const uint4 a = *reinterpret_cast<const uint4*>(codes8 + static_cast<size_t>(gidx) * 32);
    const uint4 b = *reinterpret_cast<const uint4*>(codes8 + static_cast<size_t>(gidx) * 32 + 16);
    const uint32_t src[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint64_t window = 0;
    uint32_t fill = 0, out_w = gidx * bits;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const uint32_t code = (src[e >> 2] >> (8 * (e & 3))) & 255u;
      window |= static_cast<uint64_t>(code) << fill;
      fill += bits;
      if (fill >= 32u) {
        codes[out_w++] = static_cast<uint32_t>(window);
        window >>= 32;
        fill -= 32u;
      }
    }
  }
}


// ---------------------------------------------------------------------------------------------------------------
// Selection kernel.  The stable sorted order of the inliers is the lexicographic order of (key, offset) pairs, and
// cluster c starts at sorted rank floor(c n'/2^k).  So a weight's index is the number of boundary elements (the
// elements at those ranks, c = 1 .. 2^k - 1) whose pair is not above its own, and nothing has to be sorted but the
// few weights that share a value bin with a boundary.  A cluster of C CTAs (C = 1 .. 16, chosen by the number of units
// in the call) works on one unit:
//   1. 256 of its weights say about where the others lie: equal-width value bins over a little more than the
//      inliers' range (the bin is a monotone function of the value, so bins partition the sorted order), and from
//      where on a weight may be an outlier;
//   2. ONE pass: fp64 moments, a histogram of all weights over the bins, one per CTA, and a list of the tails;
//   3. the moments give the outlier test, which the listed tails are put to; the histograms are added up through
//      distributed shared memory, and the prefix gives the bin and the in-bin rank of every boundary (the outliers
//      below the mean come first);
//   4. a second pass gives every weight outside the boundary bins its index (bin -> number of boundaries in lower
//      bins), adds the cluster sums and packs the stream; the weights of boundary bins are set aside as pairs, their
//      indexes left zero in the stream, and so are the outliers', which only lie in special bins, too;
//   5. a warp per boundary bin ranks its pairs by counting, ORs their indexes into the stream and adds their values to
//      the sums in rank order; then the centroids and the outliers' indexes.
// Every warp owns one contiguous run of the unit in both passes (a lane reads four consecutive weights at a time), so
// outlier lists come out in ascending offsets from per-warp counts alone.  Cluster sums are plain fp64 additions in a
// fixed order (every cell of a shared-memory table has one writing thread or threads that take turns, columns and
// CTAs are added in a fixed tree), so the output is deterministic.  What 256 weights say only decides how long things take:
// should outliers lie further in than the listed tails, the tails are listed again; should a boundary lie in a bin
// with outliers, or a bin hold too many weights, the unit is sorted.
//
// The fp64 outlier test is monotone on either side of the mean, so it is taken once per unit, to find the smallest and
// the largest fp32 value that pass it; a weight is then an inlier if it lies between these two.
//
// Two CTAs of 512 threads share an SM: while one waits at a cluster barrier or for memory the other has the pipes.
// That leaves 64 registers: what pass 4 does not need is kept in shared memory meanwhile, because a spilled value comes back
// from L2 (the streamed weights push it out of the first-level cache): three of them cost a small call 1.2 of 28 us.
//
// Bound: with few units the chain of six or seven cluster barriers and the table passes between them (22 of the 30 us that
// 12 units of 196,608 weights take at 4 bits); with many the shared-memory pipe and the latency of the chains through
// it: pass 2 takes 11.6 cycles per 32 weights, the histogram's atomics (3.9 wavefronts each); pass 4 15.5, the table
// lookup, the fp64 read-modify-write of the sums and the staging of the stream.  Moments, histogram and indexes as three
// passes, with the inliers looked for in each: 384 units of 524,288 weights at 3 bits 624 -> 494 us, 200 at 4 bits 345 ->
// 267, 384 at 6 bits 928 -> 819, 40 of 100,096 at 3 bits 43.1 -> 39.5, 12 of 196,608 at 4 bits 31.5 -> 30.4.

constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelMaxCluster = 16;
constexpr int kSelBins = 16384;            // most value bins; half of them for units of at most 2^18 weights
constexpr int kSelMaxSeg = 1024;           // weights of one boundary bin that are ranked by counting
constexpr int kSelSmemSeg = 256;           // ... in shared memory; more than that from the workspace
constexpr int kSelGroups = 4;              // groups of 128 consecutive weights (four per lane) a warp classifies per step
constexpr int kSelStep = kSelGroups * 128; // weights of one step of one warp
constexpr uint32_t kSelTails = 32;         // weights of a warp's tails that are listed in shared memory; more of them in the workspace
constexpr int kAccCells = 8192;            // fp64 cells of the cluster-sum table: 2^k clusters x columns

struct SelTail { uint32_t offset; float value; };

struct SelShared {
  double red[2][kSelWarps];
  double moments[2][kSelMaxCluster][2];    // of every CTA of the cluster: sum and sum of squares (the second set: the repeated pass)
  double part[kSelMaxCluster][64];         // cluster sums of every CTA
  double extra_lo[64], extra_hi[64];       // sums of cluster c's weights from the bin of its lower / only of its upper boundary
  uint32_t warp_out[kSelWarps];            // outliers of each warp's run -> their exclusive prefix
  uint32_t warp_in[kSelWarps];             // weights in each warp's run of bins -> their exclusive prefix
  uint32_t cta_out[kSelMaxCluster], cta_low[kSelMaxCluster];    // of every CTA: outliers found, those below the mean among them
  uint32_t range_in[kSelMaxCluster];       // of every CTA: weights in its range of bins
  uint32_t low;
  uint32_t bounds[65];
  uint32_t bnd_bin[64], bnd_rho[64], seg_len[64];   // of boundary c: its bin, its rank in the bin, the bin's population
  uint32_t seg_start[64];                  // where the pairs of the bin that boundary c is the first of begin
  uint32_t seg_count[64];                  // 2 and 3 bits: pairs in that list so far (the first CTA's copy counts for the cluster);
                                           // above: the next free place of this CTA in the list
  uint32_t longest;
  float cents[64];
  alignas(16) uint8_t binfo[kSelBins];     // boundaries in lower bins (6 bits) | kInfoBoundary: holds one | kInfoSpecial: look closer
  SelTail tails[kSelWarps][kSelTails];     // the first entries of each warp's list of tails
  // What the end of the kernel needs again, kept here and not in registers: a spilled one would come back from L2.
  uint32_t n_tails[kSelWarps], n_in, n_out;
  float least, most;
  alignas(16) uint32_t stage[kSelWarps][2 * 128 * 6 / 32];       // the packed indexes of two groups
  union alignas(16) {
    uint32_t hist[kSelBins];               // this CTA's histogram; in its own range of bins the cluster's, then its prefix
    double acc[kAccCells];                 // later the cluster sums
    unsigned long long pairs[kSelWarps][2][kSelSmemSeg];         // and last the boundary bins: as gathered, their keys in order
  } u;
};
static_assert(2 * (sizeof(SelShared) + 1024) <= 228 * 1024, "two CTAs on an SM");
static_assert(4 * kSelSmemSeg >= kSelMaxSeg, "the longest bin's keys in a warp's pairs");
static_assert(sti::kEndCandidates == 16, "half a warp");
static_assert(kSelBins / kSelMaxCluster / kSelWarps <= 64, "eight of the cluster's CTAs per lane");

// A weight of a special bin is looked at by itself: the bin holds a boundary, or an end of the inliers' range, or lies outside it.
constexpr uint32_t kInfoSpecial = 0x80u, kInfoBoundary = 0x40u;

// What classifies a weight of a unit.
struct SelUnit {
  float least, most;                       // the inliers' range
  float inv, off;                          // place of a value between the ends of the bins: 0 .. 1
  float last;                              // the last bin's number times 2^-149, the smallest fp32 number
  __device__ __forceinline__ bool inlier(float x) const { return x >= least && x <= most; }
  // The nearest integer of a clamped value in [0, last bin], monotone in x: as a multiple of 2^-149 it is its own bit pattern.
  // NaN goes to bin 0.
  __device__ __forceinline__ uint32_t bin(float x) const { return __float_as_uint(__fmul_rn(__saturatef(fmaf(x, inv, off)), last)); }
};

__device__ __forceinline__ float4 load4(const float* w, uint32_t i, uint32_t n) {
  return i < n ? *reinterpret_cast<const float4*>(w + i) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// A thread's sum and sum of squares -> the cluster's, in fp64 and in a fixed order.
__device__ __forceinline__ void cluster_sums(cg::cluster_group& cluster, SelShared& sm, int set, double a, double b, int tid, double& sum,
                                             double& squares) {
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); b += __shfl_xor_sync(0xffffffffu, b, o); }
  if (lane == 0) { sm.red[0][warp] = a; sm.red[1][warp] = b; }
  __syncthreads();
  if (set == 0) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");      // the cluster's CTAs have all started
  const int n_ctas = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  if (tid < n_ctas) {                      // thread t hands this CTA's sums to CTA t
    a = b = 0.0;
    for (int v = 0; v < kSelWarps; ++v) { a += sm.red[0][v]; b += sm.red[1][v]; }
    double* to = cluster.map_shared_rank(&sm.moments[set][rank][0], tid);
    to[0] = a; to[1] = b;
  }
  cluster.sync();
  sum = squares = 0.0;
  for (int r = 0; r < n_ctas; ++r) { sum += sm.moments[set][r][0]; squares += sm.moments[set][r][1]; }
}

// The first step of a warp's run, for for_each_group to begin with.
__device__ __forceinline__ void load_step(const float* w, uint32_t n, uint32_t base, float4 (&next)[kSelGroups]) {
#pragma unroll
  for (int u = 0; u < kSelGroups; ++u) next[u] = load4(w, base + u * 128u, n);
}
// Calls f(first offset of the lane's four, the four weights, whether they exist) for every group of 128 weights of a warp's run,
// in order, all lanes together.  The next step's loads are issued together before this one is worked on (spread over the step,
// each into the registers just used, they took 84 instead of 50 us for the first pass over 384 units of 524,288 weights).
template <typename F>
__device__ __forceinline__ void for_each_group(const float* w, uint32_t n, uint32_t base, uint32_t part, float4 (&next)[kSelGroups], F f) {
  for (uint32_t e0 = 0; e0 < part; e0 += kSelStep) {
    float4 x[kSelGroups];
#pragma unroll
    for (int u = 0; u < kSelGroups; ++u) {
      x[u] = next[u];
      if (e0 + kSelStep < part) next[u] = load4(w, base + e0 + kSelStep + u * 128u, n);
    }
#pragma unroll
    for (int u = 0; u < kSelGroups; ++u) f(base + e0 + u * 128u, x[u], base + e0 + u * 128u < n);
  }
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float y;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// A warp's list of weights below `lo` or above `hi`, by ascending offsets.
struct SelTails {
  SelTail* near;                           // the first kSelTails of them
  SelTail* far;                            // the others: places kSelTails .. of this array
  uint32_t n;
  __device__ __forceinline__ SelTail& at(uint32_t k) const { return k < kSelTails ? near[k] : far[k]; }
  // Those of one group of 128 weights, all lanes together.  One group in eight of Gaussian weights has one; with heavier tails (a
  // deviation near 1, where the outliers' share grows, or a scale that varies inside the unit) most have several.  Lane after lane
  // took 206 us for 16 units of 524,288 weights of deviation 5 at 6 bits and 280 for 64 at 3 bits with half of the weights ten times
  // smaller, now 121 and 224; a vote per weight instead of per bit of the count spills (384 Gaussian ones at 6 bits 803 -> 831).
  __device__ __forceinline__ void add(uint32_t i0, const float4& x, bool exists, float lo, float hi) {
    const float most = max3(fmaxf(x.x, x.y), x.z, x.w), least = min3(fminf(x.x, x.y), x.z, x.w);
    const bool any = exists && (most > hi || least < lo);
    if (!__any_sync(0xffffffffu, any)) return;
    const float v[4] = {x.x, x.y, x.z, x.w};
    uint32_t count = 0;
    if (any) {
#pragma unroll
      for (int j = 0; j < 4; ++j) count += v[j] < lo || v[j] > hi ? 1u : 0u;
    }
    const uint32_t lt_mask = (1u << (threadIdx.x & 31u)) - 1u;
    uint32_t k = n;                        // this lane's first place: the counts of the lanes before it, 0 to 4, added up bit by bit
#pragma unroll
    for (int bit = 0; bit < 3; ++bit) {
      const uint32_t all = __ballot_sync(0xffffffffu, (count >> bit & 1u) != 0u);
      k += __popc(all & lt_mask) << bit;
      n += __popc(all) << bit;
    }
    if (any) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v[j] < lo || v[j] > hi) at(k++) = {i0 + j, v[j]};
    }
  }
};

template <int BITS>      // the index width is a compile-time constant: the packing and the table addressing unroll to immediates
__global__ void __launch_bounds__(kSelThreads, 2)
quantize_select_kernel(const float* w_all, uint32_t n, uint32_t n_bins, uint32_t* codes_all, float* cent_all, uint32_t* ooff_all,
                       float* oval_all, uint32_t max_out, uint32_t* n_out_all, uint8_t* ws_all, size_t ws_per_unit,
                       uint8_t* marks) {
  extern __shared__ __align__(16) uint8_t q_smem[];
  SelShared& sm = *reinterpret_cast<SelShared*>(q_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_ctas = cluster.num_blocks(), rank = cluster.block_rank(), unit = blockIdx.x / n_ctas;
  constexpr uint32_t bits = BITS, K = 1u << BITS;
  const float* w = w_all + static_cast<size_t>(unit) * n;
  uint32_t* codes = codes_all + static_cast<size_t>(unit) * (static_cast<size_t>(n) * bits / 32);
  float* cent = cent_all + static_cast<size_t>(unit) * K;
  uint32_t* ooff = ooff_all + static_cast<size_t>(unit) * max_out;
  float* oval = oval_all + static_cast<size_t>(unit) * max_out;
  unsigned long long* cand = reinterpret_cast<unsigned long long*>(ws_all + static_cast<size_t>(unit) * ws_per_unit);
  const uint32_t lt_mask = (1u << lane) - 1u;
  pdl_launch_dependents();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");         // waited for before the first remote access

  // the warp's run: whole steps
  const uint32_t steps = (n + kSelStep - 1u) / kSelStep, n_warps = n_ctas * kSelWarps;
  const uint32_t part = ((steps + n_warps - 1u) / n_warps) * kSelStep;
  const uint32_t base = (rank * kSelWarps + static_cast<uint32_t>(warp)) * part + 4u * lane;     // the lane's first weight

  for (uint32_t i = tid; i < n_bins / 4; i += kSelThreads) reinterpret_cast<uint4*>(sm.u.hist)[i] = make_uint4(0u, 0u, 0u, 0u);

  // ---- 1. Where the bins go and what may be an outlier, from 256 weights spread over the unit: a Gaussian of their mean absolute
  //         deviation, which a few outliers hardly change.  Every warp of the cluster looks at the same ones by itself.  A poor
  //         guess costs time only: bins that are too wide, or the tails listed a second time.
  SelUnit un;
  float tail_lo, tail_hi;
  float4 ahead[kSelGroups];
  {
    float4 x[2];
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u)
      x[u] = *reinterpret_cast<const float4*>(w + static_cast<size_t>(static_cast<uint64_t>(n / 4u) * (32u * u + lane) / 64u) * 4u);
    load_step(w, n, base, ahead);
    float s = ((x[0].x + x[0].y) + (x[0].z + x[0].w)) + ((x[1].x + x[1].y) + (x[1].z + x[1].w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float centre = s * (1.f / 256.f);
    s = 0.f;
#pragma unroll
    for (int u = 0; u < 2; ++u) s += (fabsf(x[u].x - centre) + fabsf(x[u].y - centre)) + (fabsf(x[u].z - centre) + fabsf(x[u].w - centre));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float deviation = s * (1.25331414f / 256.f);                 // a Gaussian's is sqrt(pi / 2) mean absolute deviations; within 5 %
    const float c = 4.f - 0.918938533f - logf(deviation);              // radius of the inliers of such a Gaussian: sqrt(2 c) deviations
    const float radius = deviation * (c > 0.f ? sqrtf(2.f * c) : 4.f);
    un.inv = 1.f / (2.7f * radius);
    un.off = 0.5f - centre * un.inv;
    if (!(un.inv < 1.0e34f) || !(fabsf(un.off) < 1.0e34f)) { un.inv = 0.f; un.off = 0.5f; }
    un.last = __uint_as_float(n_bins - 1u);
    tail_lo = centre - 0.88f * radius;
    tail_hi = centre + 0.88f * radius;
  }
  if (tid < 64) { sm.seg_count[tid] = 0u; sm.extra_lo[tid] = sm.extra_hi[tid] = 0.0; }
  if (tid == 0) sm.low = 0u;
  __syncthreads();                         // the histogram is all zeros

  // ---- 2. one pass: Gaussian fit, histogram, list of the tails.  Squares about zero: should the mean be far off, so that they
  //         cancel, a second pass about the mean found.
  auto tails_far = [&](uint32_t run_start) { return reinterpret_cast<SelTail*>(cand + n) + run_start; };      // the workspace's second half
  SelTails tails = {sm.tails[warp], tails_far(base - 4u * lane), 0u};
  double s[2] = {0.0, 0.0}, q[2] = {0.0, 0.0};
  for_each_group(w, n, base, part, ahead, [&](uint32_t i0, const float4& x, bool exists) {
    if (exists) {
      const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double d = static_cast<double>(v[j]);
        s[j & 1] += d;
        q[j & 1] = fma(d, d, q[j & 1]);
        atomicAdd(&sm.u.hist[un.bin(v[j])], 1u);
      }
    }
    tails.add(i0, x, exists, tail_lo, tail_hi);
  });
  const double count = static_cast<double>(n);
  double sum, squares;
  cluster_sums(cluster, sm, 0, s[0] + s[1], q[0] + q[1], tid, sum, squares);
  // the cluster's histogram: CTA r adds up range r of the bins, in its own copy, and forms the prefix inside each warp's
  // run of it
  const uint32_t range = n_bins / n_ctas, range0 = rank * range, run = range / kSelWarps;
  {
    uint32_t* mine = sm.u.hist + range0 + warp * run;
    // A lane reads four bins from every `groups`-th CTA, all in flight together (at most eight: 16 CTAs have runs of 64 bins or
    // 32); the groups' sums are added up by shuffles.
    const uint32_t vec = run < 128u ? run / 4u : 32u, groups = 32u / vec, group = lane / vec;
    for (uint32_t i = 4u * (lane % vec); i < run; i += 128) {
      uint4 r[8], t = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (uint32_t q = 0; q < 8; ++q) {
        const uint32_t from = group + q * groups;
        r[q] = from < n_ctas ? *cluster.map_shared_rank(reinterpret_cast<const uint4*>(mine + i), (rank + from) & (n_ctas - 1u)) : t;
      }
#pragma unroll
      for (uint32_t q = 0; q < 8; ++q) { t.x += r[q].x; t.y += r[q].y; t.z += r[q].z; t.w += r[q].w; }
      for (uint32_t o = vec; o < 32u; o <<= 1) {
        t.x += __shfl_xor_sync(0xffffffffu, t.x, o); t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
        t.z += __shfl_xor_sync(0xffffffffu, t.z, o); t.w += __shfl_xor_sync(0xffffffffu, t.w, o);
      }
      if (group == 0u) *reinterpret_cast<uint4*>(mine + i) = t;
    }
    __syncwarp();
    uint32_t before = 0;
    for (uint32_t i = lane; i < run; i += 32) {
      const uint32_t t = mine[i];
      uint32_t inc = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const uint32_t s = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += s; }
      mine[i] = before + inc - t;
      before += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) sm.warp_in[warp] = before;
  }
  double mu = sum / count;
  double var = squares / count - mu * mu;
  if (!(mu * mu <= 4.0 * var)) {                                       // the same in every thread of the cluster
    const double shift = mu;
    s[0] = s[1] = q[0] = q[1] = 0.0;
    load_step(w, n, base, ahead);
    for_each_group(w, n, base, part, ahead, [&](uint32_t, const float4& x, bool exists) {
      if (!exists) return;
      const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double d = static_cast<double>(v[j]) - shift;
        s[j & 1] += d;
        q[j & 1] = fma(d, d, q[j & 1]);
      }
    });
    cluster_sums(cluster, sm, 1, s[0] + s[1], q[0] + q[1], tid, sum, squares);
    var = squares / count - (sum / count) * (sum / count);
    mu += sum / count;
  }
  const double c0 = -0.5 * log(2.0 * 3.14159265358979323846 * var);
  const double inv2var = 1.0 / (2.0 * var);
  const double radius = sqrt(2.0 * var * (c0 + 4.0));                  // inliers satisfy (x - mu)^2 <= 2 var (c0 + 4)
  // Others may still be reading this CTA's histogram: a CTA that leaves before the next barrier waits for them.
  auto leave_to_the_sort = [&]() {
    if (rank == 0 && tid == 0) marks[unit] = 1;                        // every thread of the cluster leaves
    cluster.sync();
  };
  if (!(var > 0.0) || !(radius > 0.0)) {
    leave_to_the_sort();
    return;
  }
  {
    // half a warp's lanes each around the lower and the upper threshold
    const int sign = lane < sti::kEndCandidates ? -1 : 1;
    const float x = sti::end_candidate(static_cast<float>(mu + sign * radius), lane % sti::kEndCandidates, sign);
    const uint32_t in = __ballot_sync(0xffffffffu, !is_outlier(x, mu, inv2var, c0));
    const int least = sti::end_index(in & 0xffffu), most = sti::end_index(in >> 16);
    if (least < 0 || most < 0) {
      leave_to_the_sort();
      return;
    }
    un.least = __shfl_sync(0xffffffffu, x, least);
    un.most = __shfl_sync(0xffffffffu, x, sti::kEndCandidates + most);
  }

  // ---- 3. the outliers among the tails
  if (!(un.least <= tail_lo && un.most >= tail_hi)) {                  // some lie further in: list exactly them
    tails.n = 0;
    load_step(w, n, base, ahead);
    for_each_group(w, n, base, part, ahead, [&](uint32_t i0, const float4& x, bool exists) { tails.add(i0, x, exists, un.least, un.most); });
  }
  __syncwarp();
  uint32_t my_out = 0, my_low = 0;
  for (uint32_t k = lane; k < tails.n; k += 32) {
    const float x = tails.at(k).value;
    my_out += un.inlier(x) ? 0u : 1u;
    my_low += x < un.least ? 1u : 0u;
  }
  my_out = __reduce_add_sync(0xffffffffu, my_out);
  my_low = __reduce_add_sync(0xffffffffu, my_low);
  if (lane == 0) {
    sm.warp_out[warp] = my_out;
    if (my_low != 0u) atomicAdd(&sm.low, my_low);
  }
  __syncthreads();
  if (warp == 0) {
    const uint32_t mine = lane < kSelWarps ? sm.warp_out[lane] : 0u;
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < kSelWarps; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    if (lane < kSelWarps) sm.warp_out[lane] = inc - mine;
    const uint32_t total = __shfl_sync(0xffffffffu, inc, kSelWarps - 1);
    if (lane < static_cast<int>(n_ctas)) {
      *cluster.map_shared_rank(&sm.cta_out[rank], lane) = total;
      *cluster.map_shared_rank(&sm.cta_low[rank], lane) = sm.low;
    }
  }

  __syncthreads();
  if (warp == 0) {
    const uint32_t mine = lane < kSelWarps ? sm.warp_in[lane] : 0u;
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < kSelWarps; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    if (lane < kSelWarps) sm.warp_in[lane] = inc - mine;
    const uint32_t total = __shfl_sync(0xffffffffu, inc, kSelWarps - 1);
    if (lane < static_cast<int>(n_ctas)) *cluster.map_shared_rank(&sm.range_in[rank], lane) = total;
  }
  cluster.sync();

  // ---- the boundary ranks, among all weights (the outliers below the mean come before every inlier): the CTA whose range of
  //      bins holds one finds its bin and tells the others
  uint32_t n_out = 0, n_low = 0, out_before = 0, in_before = 0;
  for (uint32_t r = 0; r < n_ctas; ++r) {
    if (r < rank) { out_before += sm.cta_out[r]; in_before += sm.range_in[r]; }
    n_out += sm.cta_out[r];
    n_low += sm.cta_low[r];
  }
  const uint32_t least_bin = un.bin(un.least), most_bin = un.bin(un.most);       // outliers are in these or beyond
  const uint32_t n_in = n - n_out;
  if (n_in == 0) {                         // no rank to look for: nothing below would be written before it is read
    if (rank == 0 && tid == 0) marks[unit] = 1;                        // every thread of the cluster leaves
    return;
  }
  if (tid <= static_cast<int>(K)) {
    sm.bounds[tid] = static_cast<uint32_t>(static_cast<uint64_t>(tid) * n_in / K);
    const uint32_t r = n_low + sm.bounds[tid];
    if (tid >= 1 && tid < static_cast<int>(K) && r >= in_before && r - in_before < sm.range_in[rank]) {
      const uint32_t at = r - in_before;
      uint32_t v = 0;                                                  // the last run, then bin, whose prefix is <= the rank holds it
      for (uint32_t step = kSelWarps / 2; step > 0; step >>= 1) if (sm.warp_in[v + step] <= at) v += step;
      const uint32_t* bins = sm.u.hist + range0 + v * run;
      const uint32_t in_run = at - sm.warp_in[v];
      uint32_t b = 0;
      for (uint32_t step = run / 2; step > 0; step >>= 1) if (bins[b + step] <= in_run) b += step;
      const uint32_t run_end = (v + 1 < kSelWarps ? sm.warp_in[v + 1] : sm.range_in[rank]) - sm.warp_in[v];
      const uint32_t bin = range0 + v * run + b;
      uint32_t len = (b + 1 < run ? bins[b + 1] : run_end) - bins[b];
      if (bin <= least_bin || bin >= most_bin) len = ~0u;              // outliers among its weights: too long for a list
      for (uint32_t q = 0; q < n_ctas; ++q) {
        *cluster.map_shared_rank(&sm.bnd_bin[tid], q) = bin;
        *cluster.map_shared_rank(&sm.bnd_rho[tid], q) = in_run - bins[b];
        *cluster.map_shared_rank(&sm.seg_len[tid], q) = len;
      }
    }
  }
  __syncthreads();                                                     // this CTA's histogram has been searched
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  // Where a CTA's pairs go in the cluster's lists: with few boundaries every pair asks the first CTA, which takes as long as a
  // read of its memory; with many - a special bin in most groups of 128 weights - the CTAs before this one are asked how
  // many weights they have in a boundary's bin, which takes another cluster barrier (us asking for every pair / ahead: 384 units of
  // 524,288 weights at 3 bits 493 / 496, 2 of 262,144 27.2 / 29.1; 200 of 524,288 at 4 bits 284 / 267, 12 of 196,608 31.4 / 30.4; 16
  // of 262,144 at 5 bits 53.7 / 51.8; 384 of 524,288 at 6 bits 877 / 819).
  constexpr bool kAskAhead = BITS >= 4;
  // meanwhile: pass 4's first loads, its table, the outlier lists
  float4 next[2] = {load4(w, base, n), load4(w, base + 128u, n)};
  if constexpr (!kAskAhead)
    for (int i = tid; i < kAccCells / 2; i += kSelThreads) reinterpret_cast<uint4*>(sm.u.acc)[i] = make_uint4(0u, 0u, 0u, 0u);
  uint32_t run_out = out_before + sm.warp_out[warp];
  for (uint32_t k0 = 0; k0 < tails.n; k0 += 32) {
    const SelTail t = k0 + lane < tails.n ? tails.at(k0 + lane) : SelTail{0u, un.least};
    const uint32_t all = __ballot_sync(0xffffffffu, !un.inlier(t.value)), dst = run_out + __popc(all & lt_mask);
    if (!un.inlier(t.value) && dst < max_out) { ooff[dst] = t.offset; oval[dst] = t.value; }
    run_out += __popc(all);
  }
  if (lane == 0) sm.n_tails[warp] = tails.n;
  if (tid == 0) { sm.n_in = n_in; sm.n_out = n_out; sm.least = un.least; sm.most = un.most; }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // lists of the boundary bins' pairs: the first boundary of a bin owns its list, in which the CTAs' pairs follow one another
  auto owns = [&](uint32_t c) { return c == 1u || sm.bnd_bin[c] != sm.bnd_bin[c - 1]; };
  if (warp == kSelWarps - 1) {
    uint32_t start = 0, longest = 0;
    for (uint32_t c0 = 0; c0 < K; c0 += 32) {
      const uint32_t c = c0 + lane;
      const uint32_t len = c >= 1u && c < K && owns(c) ? sm.seg_len[c] : 0u;
      uint32_t inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
      if (c < K) sm.seg_start[c] = start + inc - len;
      start += __shfl_sync(0xffffffffu, inc, 31);
      longest = max(longest, __reduce_max_sync(0xffffffffu, len));
    }
    if (lane == 0) sm.longest = longest;
  }
  uint32_t fill = 0;                                                   // what the CTAs before this one put into boundary tid's bin
  if constexpr (kAskAhead) {
    if (tid >= 1 && tid < static_cast<int>(K) && owns(tid)) {
      const uint32_t b = sm.bnd_bin[tid], holder = b / range;          // the holder's own count made way for the cluster's
      uint32_t others = 0, t[kSelMaxCluster];
#pragma unroll
      for (uint32_t r = 0; r < kSelMaxCluster; ++r)                    // all in flight together
        t[r] = r < n_ctas && r != holder ? *cluster.map_shared_rank(&sm.u.hist[b], r) : 0u;
#pragma unroll
      for (uint32_t r = 0; r < kSelMaxCluster; ++r) {
        others += t[r];
        if (r < rank) fill += t[r];
      }
      if (holder < rank) fill += sm.seg_len[tid] - others;
    }
  }
  for (uint32_t i = tid; i < n_bins / 16; i += kSelThreads) {          // sixteen bins a thread
    uint32_t below = 0, packed[4];                                     // boundaries 1 .. below sit in lower bins (their bins ascend)
#pragma unroll
    for (uint32_t step = K >> 1; step > 0; step >>= 1)
      if (sm.bnd_bin[below + step] < 16u * i) below += step;
    uint32_t next = below + 1 < K ? sm.bnd_bin[below + 1] : 0xffffffffu;
    if (next > 16u * i + 15u && 16u * i > least_bin && 16u * i + 15u < most_bin) {       // none of them is special
      const uint32_t four = below * 0x01010101u;
      reinterpret_cast<uint4*>(sm.binfo)[i] = make_uint4(four, four, four, four);
      continue;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      packed[q] = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t b = 16u * i + 4 * q + e;
        while (next < b) { ++below; next = below + 1 < K ? sm.bnd_bin[below + 1] : 0xffffffffu; }
        const uint32_t info = next == b ? kInfoBoundary | kInfoSpecial : b <= least_bin || b >= most_bin ? kInfoSpecial : 0u;
        packed[q] |= (below | info) << (8 * e);
      }
    }
    reinterpret_cast<uint4*>(sm.binfo)[i] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
  }
  if constexpr (kAskAhead) cluster.sync();                             // nobody looks at another CTA's histogram any more
  else __syncthreads();
  if (sm.longest > static_cast<uint32_t>(kSelMaxSeg)) {
    if (rank == 0 && tid == 0) marks[unit] = 1;
    return;
  }
  if constexpr (kAskAhead) {
    if (tid < static_cast<int>(K)) sm.seg_count[tid] = sm.seg_start[tid] + fill;
    for (int i = tid; i < kAccCells / 2; i += kSelThreads) reinterpret_cast<uint4*>(sm.u.acc)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }

  // ---- 4. indexes, cluster sums, the packed stream
  // The cluster-sum table has one column per `share` neighbouring lanes (1, 2 or 4: 2^k columns of 512 cells do not
  // fit above 16 clusters); the lanes of such a group add one after the other, so every cell sees a fixed order of
  // additions.  A weight without an index yet adds a zero to cluster 0.
  constexpr uint32_t acc_cols = (kAccCells >> BITS) < kSelThreads ? (kAccCells >> BITS) : kSelThreads;
  constexpr uint32_t share = kSelThreads / acc_cols;
  double* column = sm.u.acc + static_cast<uint32_t>(tid) / share;
  for (uint32_t e0 = 0; e0 < part; e0 += 256u) {
    if (base - 4u * lane + e0 >= n) break;                             // the whole warp
    const float4 x[2] = {next[0], next[1]};
    uint32_t packed[2];
    next[0] = load4(w, base + e0 + 256u, n);                           // at the end of the run: the next warp's first, unused
    next[1] = load4(w, base + e0 + 384u, n);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t i0 = base + e0 + u * 128u;
      float v[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
      uint32_t code[4], flags = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        code[j] = sm.binfo[un.bin(v[j])];
        flags |= code[j];
      }
      if ((flags & kInfoSpecial) != 0u || i0 >= n) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool boundary = (code[j] & kInfoBoundary) != 0u;       // such bins hold inliers only
          const bool later = i0 >= n || boundary || !un.inlier(v[j]);  // no index yet
          code[j] &= 63u;
          if (i0 < n && boundary) {
            uint32_t pos;
            if constexpr (kAskAhead) pos = atomicAdd(&sm.seg_count[code[j] + 1u], 1u);
            else pos = sm.seg_start[code[j] + 1u] + atomicAdd(cluster.map_shared_rank(&sm.seg_count[code[j] + 1u], 0), 1u);
            cand[pos] = (static_cast<unsigned long long>(sort_key(v[j])) << 32) | (i0 + j);
          }
          if (later) { code[j] = 0u; v[j] = 0.f; }
        }
      }
      packed[u] = code[0] | (code[1] << bits) | (code[2] << (2 * bits)) | (code[3] << (3 * bits));
#pragma unroll
      for (uint32_t q = 0; q < share; ++q) {
        if (share == 1u || (lane & (share - 1u)) == q) {
#pragma unroll
          for (int j = 0; j < 4; ++j) column[code[j] * acc_cols] += static_cast<double>(v[j]);
        }
        if (share > 1u) __syncwarp();
      }
    }
    // The stream: the lanes of a pair exchange so that each has the indexes of eight consecutive weights of one group,
    // `bits` whole bytes (even lanes of the first group, odd ones of the second); the bytes go through shared memory.
    uint8_t* stage = reinterpret_cast<uint8_t*>(sm.stage[warp]);
    {
      const bool odd = (lane & 1) != 0;
      const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? packed[0] : packed[1], 1);
      const uint32_t first = odd ? got : packed[0], second = odd ? packed[1] : got;
      const uint64_t eight = first | (static_cast<uint64_t>(second) << (4 * bits));
      uint8_t* to = stage + (lane & 1) * 16u * bits + (static_cast<uint32_t>(lane) >> 1) * bits;
      if constexpr (BITS == 4) {
        *reinterpret_cast<uint32_t*>(to) = static_cast<uint32_t>(eight);
      } else if constexpr (BITS % 2 == 0) {
#pragma unroll
        for (int h = 0; h < BITS / 2; ++h) reinterpret_cast<uint16_t*>(to)[h] = static_cast<uint16_t>(eight >> (16 * h));
      } else {
#pragma unroll
        for (int h = 0; h < BITS; ++h) to[h] = static_cast<uint8_t>(eight >> (8 * h));
      }
    }
    __syncwarp();
    const uint32_t word0 = (base - 4u * lane + e0) / 32u * bits, n_words = n / 32u * bits;
#pragma unroll
    for (uint32_t i = lane; i < 8u * bits; i += 32)
      if (word0 + i < n_words) codes[word0 + i] = sm.stage[warp][i];
    __syncwarp();
  }
  __syncthreads();
  for (uint32_t c = warp; c < K; c += kSelWarps) {                     // the columns of a cluster in a fixed order
    double acc = 0.0;
    for (uint32_t t = lane; t < acc_cols; t += 32) acc += sm.u.acc[c * acc_cols + t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane < static_cast<int>(n_ctas)) *cluster.map_shared_rank(&sm.part[rank][c], lane) = acc;
  }
  cluster.sync();                                                      // pairs and streams are complete as well

  // ---- 5. the boundary bins, a warp each: a pair's rank is the number of smaller pairs of its bin (all are distinct)
  // The lists' address is worked out again, from a unit number that the compiler does not know: kept over pass 4 it makes
  // another value there come back from L2 (384 units of 524,288 weights at 3 bits 487 -> 520 us, 200 at 4 bits 270 -> 286).  The
  // cluster's number is the unit's; block number over cluster size took 12 units of 196,608 at 4 bits 29.0 -> 29.8.
  uint32_t same_unit;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(same_unit));
  const unsigned long long* lists = reinterpret_cast<const unsigned long long*>(ws_all + static_cast<size_t>(same_unit) * ws_per_unit);
  for (uint32_t c = 1u + warp * n_ctas + rank; c < K; c += n_warps) {       // neighbours on different SMs
    if (!owns(c)) continue;
    const uint32_t m = sm.seg_len[c], bin = sm.bnd_bin[c];
    uint32_t last = c;                                                 // the bin's boundaries: c .. last
    while (last + 1u < K && sm.bnd_bin[last + 1u] == bin) ++last;
    const unsigned long long* from = lists + sm.seg_start[c];
    // The keys in order, which is all that the sums need: behind the pairs, or where a longer bin's would have been (the unit's
    // workspace has no room for them: its second half holds the tails beyond the warps' lists).
    uint32_t* sorted = reinterpret_cast<uint32_t*>(sm.u.pairs[warp][0]) + (m <= static_cast<uint32_t>(kSelSmemSeg) ? 2 * kSelSmemSeg : 0);
    if (m <= static_cast<uint32_t>(kSelSmemSeg)) {
      for (uint32_t j = lane; j < m; j += 32) sm.u.pairs[warp][0][j] = from[j];
      if (lane == 0 && (m & 1u) != 0u) sm.u.pairs[warp][0][m] = ~0ull;
      from = sm.u.pairs[warp][0];
      __syncwarp();
    }
    for (uint32_t j0 = 0; j0 < m; j0 += 128) {
      unsigned long long mine[4];
      uint32_t smaller[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int e = 0; e < 4; ++e) mine[e] = j0 + 32 * e + lane < m ? from[j0 + 32 * e + lane] : 0ull;
      if (m <= static_cast<uint32_t>(kSelSmemSeg)) {
        const ulonglong2* two = reinterpret_cast<const ulonglong2*>(sm.u.pairs[warp][0]);
        auto rank_by_counting = [&](auto lists) {
#pragma unroll 4
          for (uint32_t t = 0; t < (m + 1) / 2; ++t) {                 // the list is padded with a largest pair
            const ulonglong2 other = two[t];
#pragma unroll
            for (int e = 0; e < decltype(lists)::value; ++e)
              smaller[e] += (other.x < mine[e] ? 1u : 0u) + (other.y < mine[e] ? 1u : 0u);
          }
        };
        const uint32_t left = m - j0;
        if (left <= 32) rank_by_counting(std::integral_constant<int, 1>());
        else if (left <= 64) rank_by_counting(std::integral_constant<int, 2>());
        else if (left <= 96) rank_by_counting(std::integral_constant<int, 3>());
        else rank_by_counting(std::integral_constant<int, 4>());
      } else {
        for (uint32_t t = 0; t < m; ++t) {
          const unsigned long long other = from[t];
#pragma unroll
          for (int e = 0; e < 4; ++e) smaller[e] += other < mine[e] ? 1u : 0u;
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (j0 + 32 * e + lane >= m) continue;
        sorted[smaller[e]] = static_cast<uint32_t>(mine[e] >> 32);
        uint32_t code = c - 1u;
        while (code + 1u <= last && sm.bnd_rho[code + 1u] <= smaller[e]) ++code;
        const uint64_t bit = (mine[e] & 0xffffffffull) * bits;
        const uint32_t sh = static_cast<uint32_t>(bit & 31u);
        atomicOr(&codes[bit >> 5], code << sh);
        if (sh + bits > 32u) atomicOr(&codes[(bit >> 5) + 1], code >> (32u - sh));
      }
    }
    __syncwarp();
    for (uint32_t k = c - 1u; k <= last; ++k) {                        // the bin's share of clusters c - 1 .. last
      const uint32_t lo = k == c - 1u ? 0u : sm.bnd_rho[k], hi = k == last ? m : sm.bnd_rho[k + 1u];
      double acc = 0.0;
      for (uint32_t t = lo + lane; t < hi; t += 32) acc += static_cast<double>(key_value(sorted[t]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      double* to = k == c - 1u ? &sm.extra_hi[k] : &sm.extra_lo[k];
      if (lane < static_cast<int>(n_ctas)) *cluster.map_shared_rank(to, lane) = acc;
    }
    __syncwarp();                                                      // the buffers are free for the warp's next bin
  }
  cluster.sync();                                                      // the last access to another CTA's shared memory
  if (tid < static_cast<int>(K)) {
    double acc = sm.extra_lo[tid] + sm.extra_hi[tid];
    for (uint32_t r = 0; r < n_ctas; ++r) acc += sm.part[r][tid];
    const uint32_t members = sm.bounds[tid + 1] - sm.bounds[tid];
    const float m = members > 0 ? static_cast<float>(acc / static_cast<double>(members)) : 0.f;
    sm.cents[tid] = m;
    if (rank == 0) cent[tid] = m;
  }
  if (rank == 0 && tid == 0) { n_out_all[unit] = sm.n_out; marks[unit] = 0; }
  __syncthreads();

  // an outlier's slot gets the nearest centroid's index (its bits in the stream are still zero)
  const float least = sm.least, most = sm.most;
  const uint32_t n_mine = sm.n_tails[warp], inliers = sm.n_in;
  for (uint32_t k = lane; k < n_mine; k += 32) {
    const SelTail t = k < kSelTails ? sm.tails[warp][k] : tails_far(base - 4u * lane)[k];
    if (t.value >= least && t.value <= most) continue;
    auto distance = [&](uint32_t c) { return fabs(static_cast<double>(t.value) - static_cast<double>(sm.cents[c])); };
    uint32_t best = 0;
    if (inliers >= K) {          // no empty cluster: the centroids ascend between the outliers of either side
      if (t.value > most) for (best = K - 1u; best > 0u && distance(best - 1u) == distance(K - 1u);) --best;
    } else {
      for (uint32_t c = 1; c < K; ++c)
        if (distance(c) < distance(best)) best = c;
    }
    const uint64_t bit = static_cast<uint64_t>(t.offset) * bits;
    const uint32_t sh = static_cast<uint32_t>(bit & 31u);
    atomicOr(&codes[bit >> 5], best << sh);
    if (sh + bits > 32u) atomicOr(&codes[(bit >> 5) + 1], best >> (32u - sh));
  }
}


// How many CTAs share a unit.  What an SM spends on its CTAs, in thousands of cycles: on a pair of CTAs 0.75 per
// thousand weights of each and 10 + 1.3 C per CTA for the table passes and barriers of a cluster of C (more CTAs, more
// remote reads); on a CTA that has the SM to itself 0.84 per thousand weights and 36 + 0.5 C, with nothing to fill its
// waits.  Summed over the waves of clusters the device holds at a time.  Fitted to calls of 1 to 384 units of 32,768 to
// 524,288 weights, whose fastest C it picks or comes within 4 % of; e.g. 12 units of 196,608 weights at 4 bits take
// 93 / 59 / 40 / 32 / 36 us with C = 1 / 2 / 4 / 8 / 16, 384 of 524,288 at 3 bits 504 / 507 / 528 / 707 / 1155.
uint32_t pick_cluster(uint32_t n_units, uint32_t n, int sm_count, const int (&resident)[5]) {
  const uint32_t steps = (n + kSelStep - 1u) / kSelStep;
  uint32_t best = 1;
  double best_cost = -1.0;
  for (int e = 0; e < 5; ++e) {
    const uint32_t c = 1u << e;
    if (e > 0 && (resident[e] < 1 || steps < c * kSelWarps)) break;    // at least a step for every warp
    const uint32_t held = resident[e] > 0 ? static_cast<uint32_t>(resident[e]) : 1u;
    const uint32_t full = (n_units - 1u) / held, last = n_units - full * held;     // full waves, clusters of the last one
    const double weights = n / 1000.0 / c, paired = 0.75 * weights + 10.0 + 1.3 * c, alone = 0.84 * weights + 36.0 + 0.5 * c;
    const double cost = 2.0 * full * paired + (last * c <= static_cast<uint32_t>(sm_count) ? alone : 2.0 * paired);
    if (best_cost < 0.0 || cost < best_cost) { best = c; best_cost = cost; }
  }
  return best;
}

// What a device's launches need to know, looked up once per device: the kernels' attributes are set then, too.
struct QuantDevice {
  bool ready = false;
  int sm_count = 0;
  int resident[5] = {0, 0, 0, 0, 0};       // clusters of 1, 2, 4, 8, 16 selection CTAs the device holds at a time
};
constexpr int kQuantMaxDevices = 64;

cudaLaunchConfig_t select_config(uint32_t n_units, uint32_t n_ctas, cudaStream_t cs, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_units * n_ctas);
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = sizeof(SelShared);
  cfg.stream = cs;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = n_ctas; attr->val.clusterDim.y = 1; attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int BITS>
cudaError_t select_configure_one(QuantDevice* d) {
  cudaError_t e = cudaFuncSetAttribute(quantize_select_kernel<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sizeof(SelShared)));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(quantize_select_kernel<BITS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < 5 && BITS == 2; ++k) {                           // the widths' kernels have the same footprint
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = select_config(1, 1u << k, nullptr, &attr);
    if (cudaOccupancyMaxActiveClusters(&d->resident[k], quantize_select_kernel<BITS>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      d->resident[k] = 0;
    }
  }
  return cudaSuccess;
}

// nullptr: the device cannot run the kernels.  The caller has made `device` current.
const QuantDevice* quant_device(int device) {
  static QuantDevice devices[kQuantMaxDevices];
  static std::mutex lock;
  if (device >= kQuantMaxDevices) return nullptr;
  std::lock_guard<std::mutex> hold(lock);
  QuantDevice& d = devices[device];
  if (d.ready) return &d;
  if (cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || d.sm_count < 1 ||
      cudaFuncSetAttribute(quantize_units_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(QuantShared))) != cudaSuccess ||
      select_configure_one<2>(&d) != cudaSuccess || select_configure_one<3>(&d) != cudaSuccess ||
      select_configure_one<4>(&d) != cudaSuccess || select_configure_one<5>(&d) != cudaSuccess ||
      select_configure_one<6>(&d) != cudaSuccess)
    return nullptr;
  d.ready = true;
  return &d;
}

template <typename... Args>
cudaError_t launch_select(int bits, const cudaLaunchConfig_t& cfg, Args... args) {
  switch (bits) {
    case 2: return cudaLaunchKernelEx(&cfg, quantize_select_kernel<2>, args...);
    case 3: return cudaLaunchKernelEx(&cfg, quantize_select_kernel<3>, args...);
    case 4: return cudaLaunchKernelEx(&cfg, quantize_select_kernel<4>, args...);
    case 5: return cudaLaunchKernelEx(&cfg, quantize_select_kernel<5>, args...);
    default: return cudaLaunchKernelEx(&cfg, quantize_select_kernel<6>, args...);
  }
}

size_t ws_per_unit_bytes(uint32_t n) { return (17 * static_cast<size_t>(n) + 255) & ~static_cast<size_t>(255); }
size_t marks_bytes(uint32_t n_units) { return (static_cast<size_t>(n_units) + 255) & ~static_cast<size_t>(255); }

}  // namespace

extern "C" {

size_t sti_quantize_workspace_bytes(uint32_t n_units, uint32_t n_weights) {
  return static_cast<size_t>(n_units) * ws_per_unit_bytes(n_weights) + marks_bytes(n_units);
}

sti_status sti_quantize_units_by(int device, void* stream, const float* w_dev, uint32_t n_units, uint32_t n_weights, int bits,
                                 uint32_t* codes_dev, float* centroids_dev, uint32_t* outlier_off_dev, float* outlier_val_dev,
                                 uint32_t max_outliers, uint32_t* n_outliers_dev, void* workspace_dev, size_t workspace_bytes,
                                 int method, uint8_t* sorted_units_dev) {
  if (!w_dev || !codes_dev || !centroids_dev || !outlier_off_dev || !outlier_val_dev || !n_outliers_dev || !workspace_dev)
    return STI_ERR_ARG;
  if (method != STI_QUANTIZE_SELECT && method != STI_QUANTIZE_SORT) return STI_ERR_ARG;
  if (bits < 2 || bits > 6) return STI_ERR_BITS;
  if (n_units == 0 || n_units > 65535 || n_weights == 0 || n_weights % 32 != 0 || n_weights > (1u << 26) || max_outliers == 0)
    return STI_ERR_SHAPE;
  if (workspace_bytes < sti_quantize_workspace_bytes(n_units, n_weights)) return STI_ERR_SIZE;
  if ((reinterpret_cast<uintptr_t>(workspace_dev) & 15) != 0 || (reinterpret_cast<uintptr_t>(w_dev) & 15) != 0) return STI_ERR_ARG;
  int prev = 0;
  if (device < 0 || cudaGetDevice(&prev) != cudaSuccess || (prev != device && cudaSetDevice(device) != cudaSuccess)) {
    (void)cudaGetLastError();
    return STI_ERR_CUDA;
  }
  sti_status st = STI_OK;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace_dev);
  const size_t per_unit = ws_per_unit_bytes(n_weights);
  uint8_t* marks = ws + static_cast<size_t>(n_units) * per_unit;
  const QuantDevice* dev = quant_device(device);
  if (dev == nullptr) {
    (void)cudaGetLastError();
    st = STI_ERR_CUDA;
  }
  // the sorting kernel follows at once (it leaves the units the selection has done) and is launched while the selection
  // still runs
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t sort_cfg = {};
  sort_cfg.gridDim = dim3(n_units);
  sort_cfg.blockDim = dim3(kQThreads);
  sort_cfg.dynamicSmemBytes = sizeof(QuantShared);
  sort_cfg.stream = cs;
  if (st == STI_OK) {
    if (method == STI_QUANTIZE_SELECT) {
      cudaLaunchAttribute attr;
      const cudaLaunchConfig_t cfg = select_config(n_units, pick_cluster(n_units, n_weights, dev->sm_count, dev->resident), cs, &attr);
      const uint32_t n_bins = n_weights > (1u << 18) ? kSelBins : kSelBins / 2;      // about a hundred weights in a bin
      if (launch_select(bits, cfg, w_dev, n_weights, n_bins, codes_dev, centroids_dev, outlier_off_dev, outlier_val_dev,
                        max_outliers, n_outliers_dev, ws, per_unit, marks) != cudaSuccess)
        st = STI_ERR_CUDA;
      sort_cfg.attrs = &early;
      sort_cfg.numAttrs = 1;
    } else if (cudaMemsetAsync(marks, 1, n_units, cs) != cudaSuccess) {
      st = STI_ERR_CUDA;
    }
  }
  if (st == STI_OK &&
      cudaLaunchKernelEx(&sort_cfg, quantize_units_kernel, w_dev, n_weights, bits, codes_dev, centroids_dev, outlier_off_dev,
                         outlier_val_dev, max_outliers, n_outliers_dev, ws, per_unit, static_cast<const uint8_t*>(marks)) != cudaSuccess)
    st = STI_ERR_CUDA;
  if (st == STI_OK && sorted_units_dev != nullptr &&
      cudaMemcpyAsync(sorted_units_dev, marks, n_units, cudaMemcpyDeviceToDevice, cs) != cudaSuccess)
    st = STI_ERR_CUDA;
  if (prev != device) (void)cudaSetDevice(prev);
  return st;
}

sti_status sti_quantize_units(int device, void* stream, const float* w_dev, uint32_t n_units, uint32_t n_weights, int bits,
                              uint32_t* codes_dev, float* centroids_dev, uint32_t* outlier_off_dev, float* outlier_val_dev,
                              uint32_t max_outliers, uint32_t* n_outliers_dev, void* workspace_dev, size_t workspace_bytes) {
  return sti_quantize_units_by(device, stream, w_dev, n_units, n_weights, bits, codes_dev, centroids_dev, outlier_off_dev,
                               outlier_val_dev, max_outliers, n_outliers_dev, workspace_dev, workspace_bytes,
                               STI_QUANTIZE_SELECT, nullptr);
}

}  // extern "C"
