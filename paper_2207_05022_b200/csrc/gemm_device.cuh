// Device-side pieces of the fused dequant-GEMM that more than one kernel uses: tile constants, the
// shared-memory header with the mbarriers, the weight-tile decode (Section 4.2 decompression: index
// unpack -> per-unit centroid table -> outlier patch), TMA / descriptor helpers and the epilogue maths.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include "sti_device.cuh"
#include "sti_kernels.h"
#include "tiling.h"

namespace sti {
namespace {

constexpr int kThreads = 512;               // warp 0: TMA producer, warp 1: MMA issuer, warps 4-11: epilogue; all 16 decode
constexpr int kWarps = kThreads / 32;
constexpr int kMaxStages = 8;
constexpr int kTableStride = 64;            // bf16 entries of a warp's centroid table
constexpr int kEpilogueWarp0 = 4;             // epilogue warps 4..11: two per TMEM lane quadrant
constexpr int kEpilogueWarps = 8;

struct SmemHeader {
  uint64_t full[kMaxStages];     // activation chunk landed (TMA transaction bytes)
  uint64_t empty[kMaxStages];    // the MMAs that read the chunk have completed
  uint64_t acc_full[2];          // accumulator buffer complete
  uint64_t acc_empty[2];         // accumulator buffer drained by the epilogue warps
  uint64_t drain;                // failure path only: all issued MMAs have completed
  uint32_t tmem_base;
  volatile uint32_t abort;       // a bounded wait ran out somewhere in the CTA
};

// ---------------------------------------------------------------------------------------
// Weight-tile decode (Section 4.2 decompression), one task of 4096 weights per warp at a time.
//
// Bound: latency, then the integer pipe.  A warp's chain is descriptor -> (planes, table, outliers) -> unpack -> its own
// outliers, with no barrier of the CTA inside.  Up to 4 bits the table is looked up with byte permutes on registers
// (2 to 2.6 integer instructions per weight; the shared-memory lookup took 3.5 and a shared-memory access each), 5 and 6
// bits look up a table in shared memory.
// Measured from a CTA's start to its decoded tile: 64 x 768 weights at 4 bits 4.5 -> 3.2 us, 64 x 1024 at 2..6 bits
// 5.5 -> 4.0 (segment descriptors with divisions, a search for each thread's outlier and a CTA barrier before the
// outliers came first); BERT-base, 385 tokens 50.5 -> 43.8 us per layer, BERT-large, 256 tokens 48.0 -> 46.2.
// ---------------------------------------------------------------------------------------
struct TaskLoads {               // a task's loads in flight
  uint32_t w[24];                // lane's 128 indexes: `bits` planes of four words
  float c0, c1;                  // centroids lane and lane + 32
  uint32_t rc;                   // outlier number `lane`
  float val;
};

__device__ __forceinline__ DecodeTask load_task(const DecodeTask* p) {
  const uint4 a = __ldg(reinterpret_cast<const uint4*>(p)), b = __ldg(reinterpret_cast<const uint4*>(p) + 1);
  DecodeTask t;
  t.codes = reinterpret_cast<const uint8_t*>(static_cast<uint64_t>(a.x) | (static_cast<uint64_t>(a.y) << 32));
  t.table = a.z; t.out_rc = a.w; t.out_val = b.x;
  t.n_out = static_cast<uint16_t>(b.y); t.bits = static_cast<uint8_t>(b.y >> 16); t.narrow = static_cast<uint8_t>(b.y >> 24);
  t.row0 = static_cast<uint16_t>(b.z); t.kcore0 = static_cast<uint16_t>(b.z >> 16);
  t.origin = b.w;
  return t;
}

// All loads of a task back to back.  Six planes whatever `bits` is - a plane number beyond it re-reads the last plane,
// a cache hit - so that none waits for another.
__device__ __forceinline__ void issue_loads(const DecodeTask& t, uint32_t lane, TaskLoads& f) {
  if (t.bits == 0 || t.bits > 6) return;
  const uint4* src = reinterpret_cast<const uint4*>(t.codes) + lane;
  uint4 v[6];
#pragma unroll
  for (uint32_t p = 0; p < 6; ++p) v[p] = __ldg(src + (p < t.bits ? p : t.bits - 1u) * 32u);
  const float* table = reinterpret_cast<const float*>(t.codes + t.table);
  const uint32_t n_entries = 1u << t.bits;
  f.c0 = lane < n_entries ? __ldg(table + lane) : 0.f;
  f.c1 = lane + 32 < n_entries ? __ldg(table + lane + 32) : 0.f;
  f.rc = 0u;
  f.val = 0.f;
  if (lane < t.n_out) {
    f.rc = __ldg(reinterpret_cast<const uint32_t*>(t.codes + t.out_rc) + lane);
    f.val = __ldg(reinterpret_cast<const float*>(t.codes + t.out_val) + lane);
  }
#pragma unroll
  for (int p = 0; p < 6; ++p) { f.w[4 * p + 0] = v[p].x; f.w[4 * p + 1] = v[p].y; f.w[4 * p + 2] = v[p].z; f.w[4 * p + 3] = v[p].w; }
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// 32 indexes of at most 4 bits -> four words of eight 4-bit fields.
template <int BITS>
__device__ __forceinline__ void spread_to_nibbles(const uint32_t (&w)[BITS], uint32_t (&sel)[4]) {
  static_assert(BITS >= 2 && BITS <= 4, "one byte permute takes a 3-bit index");
  if constexpr (BITS == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sel[i] = w[i];
  } else {
    uint32_t x[4];             // eight indexes each, in the low bits
    if constexpr (BITS == 3) {
      x[0] = w[0]; x[1] = __funnelshift_r(w[0], w[1], 24); x[2] = __funnelshift_r(w[1], w[2], 16); x[3] = w[2] >> 8;
    } else {
      x[0] = w[0]; x[1] = w[0] >> 16; x[2] = w[1]; x[3] = w[1] >> 16;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {      // halves apart, quarters apart, eighths apart; what is in between is masked last
      uint32_t y = (x[i] & 0x0000ffffu) | ((x[i] << (16 - 4 * BITS)) & 0xffff0000u);
      y = (y & 0x00ff00ffu) | ((y << (8 - 2 * BITS)) & 0xff00ff00u);
      y = (y & 0x0f0f0f0fu) | ((y << (4 - BITS)) & 0xf0f0f0f0u);
      sel[i] = y & (BITS == 3 ? 0x77777777u : 0x33333333u);
    }
  }
}

// The table in registers, low and high bytes of the bf16 entries apart, four entries to a word.
template <int BITS>
struct ByteTable {
  static constexpr int kWords = BITS == 2 ? 1 : (1 << BITS) / 4;
  uint32_t lo[kWords], hi[kWords];
  __device__ __forceinline__ void load(const uint16_t* tab) {
#pragma unroll
    for (int i = 0; i < kWords; ++i) {
      const uint2 e = *reinterpret_cast<const uint2*>(tab + 4 * i);
      lo[i] = prmt(e.x, e.y, 0x6420u);
      hi[i] = prmt(e.x, e.y, 0x7531u);
    }
  }
  // bf16 values of the four indexes in the low 16 bits of `sel`, in order
  __device__ __forceinline__ void four(uint32_t sel, uint32_t upper, uint32_t& w0, uint32_t& w1) const {
    uint32_t l, h;
    if constexpr (BITS <= 3) {
      l = prmt(lo[0], lo[kWords - 1], sel);
      h = prmt(hi[0], hi[kWords - 1], sel);
    } else {                   // entries 0-7 and 8-15 side by side, then byte j from the side that index j's top bit names
      l = prmt(prmt(lo[0], lo[1], sel), prmt(lo[2], lo[3], sel), upper);
      h = prmt(prmt(hi[0], hi[1], sel), prmt(hi[2], hi[3], sel), upper);
    }
    w0 = prmt(l, h, 0x5140u);
    w1 = prmt(l, h, 0x7362u);
  }
};

// Where the decoded weights of a task go.  `piece(base, grp, ss)`: eight columns (ss of four) of index group grp (of four) of
// the lane's row; `element(row, col)`: byte offset of a weight of the task, for outliers and uncompressed units.
// The tile of a GEMM CTA: K-major core matrices, (row, k) at ((k / 8) * n_rows + row) * 16 + (k % 8) * 2.
struct TilePlace {
  uint8_t* wsm;
  uint32_t n_rows, row0, kcore0, narrow;
  __device__ __forceinline__ TilePlace(uint8_t* w, uint32_t rows, const DecodeTask& t)
      : wsm(w), n_rows(rows), row0(t.row0), kcore0(t.kcore0), narrow(t.narrow) {}
  __device__ __forceinline__ uint8_t* group(uint32_t grp, uint32_t lane) const {
    uint8_t* dst0 = wsm + (static_cast<size_t>(kcore0) * n_rows + row0 + lane) * 16;
    return dst0 + (narrow ? (grp & 1) * 4 * (n_rows * 16) + (grp >> 1) * 512 : grp * 4 * (n_rows * 16));
  }
  __device__ __forceinline__ uint8_t* piece(uint8_t* group_base, uint32_t, uint32_t ss, uint32_t) const {
    return group_base + ss * (n_rows * 16);                       // from eight columns to the next eight
  }
  __device__ __forceinline__ uint8_t* element(uint32_t row, uint32_t col) const {
    return wsm + (static_cast<size_t>(kcore0 + (col >> 3)) * n_rows + row0 + row) * 16 + (col & 7) * 2;
  }
};
// A task by itself: two blocks of 32 rows x 64 columns in the 128-byte-swizzled K-major layout that TMA and the tensor core
// know (a row is 128 bytes, its eight 16-byte pieces permuted by the row's number modulo 8).  Wide tasks: the block's
// columns 0-63 and 64-127; narrow ones: rows 0-31 and 32-63.
struct SwizzledPlace {
  uint8_t* wsm;
  uint32_t narrow;
  __device__ __forceinline__ SwizzledPlace(uint8_t* w, const DecodeTask& t) : wsm(w), narrow(t.narrow) {}
  __device__ __forceinline__ uint8_t* group(uint32_t grp, uint32_t lane) const { return wsm + (grp >> 1) * 4096 + lane * 128; }
  __device__ __forceinline__ uint8_t* piece(uint8_t* group_base, uint32_t grp, uint32_t ss, uint32_t lane) const {
    return group_base + ((((grp & 1) * 4 + ss) ^ (lane & 7)) << 4);
  }
  __device__ __forceinline__ uint8_t* element(uint32_t row, uint32_t col) const {
    const uint32_t block = narrow ? row >> 5 : col >> 6, c = col & 63;
    return wsm + block * 4096 + (row & 31) * 128 + (((c >> 3) ^ (row & 7)) << 4) + (c & 7) * 2;
  }
};

// Index unpack -> table lookup -> 16-byte stores.  Each lane holds 128 consecutive
// indexes of its own row (narrow tasks: of rows l and l + 32).  `half`: 0 = the whole quantum (four groups of 32 indexes),
// 1 / 2 = its first / second two groups only (two warps share a task when a tile has few; both hold the task's planes).
// 32 indexes are exactly BITS words: the loop is rolled over the four groups and always reads w[0 .. BITS), the words
// moving down after each group - the decode runs once per CTA, so its code is fetched cold and its size is what it costs.
template <int BITS, typename Place>
__device__ __forceinline__ void unpack_task(const uint32_t (&planes)[24], const Place& place, const uint16_t* __restrict__ tab,
                                            uint32_t lane, uint32_t half) {
  uint32_t w[4 * BITS];
#pragma unroll
  for (int i = 0; i < 4 * BITS; ++i) w[i] = planes[i];
  if (half == 2) {
#pragma unroll
    for (int i = 0; i < 2 * BITS; ++i) w[i] = planes[i + 2 * BITS];
  }
  const uint32_t grp0 = half == 2 ? 2 : 0, grp1 = half == 1 ? 2 : 4;
  ByteTable<BITS <= 4 ? BITS : 2> table;
  if constexpr (BITS <= 4) table.load(tab);
#pragma unroll 1
  for (uint32_t grp = grp0; grp < grp1; ++grp) {
    uint32_t lo[BITS];
#pragma unroll
    for (int i = 0; i < BITS; ++i) lo[i] = w[i];
    uint8_t* dst = place.group(grp, lane);
    if constexpr (BITS <= 4) {
      uint32_t sel[4];
      spread_to_nibbles<BITS>(lo, sel);
#pragma unroll
      for (int ss = 0; ss < 4; ++ss) {
        const uint32_t low = BITS == 4 ? sel[ss] & 0x77777777u : sel[ss];
        const uint32_t upper = BITS == 4 ? ((sel[ss] >> 1) & 0x44444444u) | 0x32103210u : 0u;
        uint4 v;
        table.four(low, upper, v.x, v.y);
        table.four(low >> 16, upper >> 16, v.z, v.w);
        *reinterpret_cast<uint4*>(place.piece(dst, grp, ss, lane)) = v;
      }
    } else {
#pragma unroll
      for (int ss = 0; ss < 4; ++ss) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t c0 = extract_index_words<BITS>(lo, 8 * ss + 2 * e);
          const uint32_t c1 = extract_index_words<BITS>(lo, 8 * ss + 2 * e + 1);
          pk[e] = static_cast<uint32_t>(tab[c0]) | (static_cast<uint32_t>(tab[c1]) << 16);
        }
        *reinterpret_cast<uint4*>(place.piece(dst, grp, ss, lane)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
#pragma unroll
    for (int i = 0; i + BITS < 4 * BITS; ++i) w[i] = w[i + BITS];
  }
}

// Uncompressed (32-bit) version of a unit: rows are plain fp32, rounded to bf16 on the way in.  A load covers four rows x
// 32 columns, four whole lines (a lane per row would touch 32 lines with every load: 9 us for a tile of 64 x 1024);
// sixteen loads in flight.
template <typename Place>
__device__ __forceinline__ void unpack_raw(const DecodeTask& t, const Place& place, uint32_t lane, uint32_t half) {
#pragma unroll 1
  for (uint32_t first = half == 2 ? 16 : 0; first < (half == 1 ? 16u : 32u); first += 16) {
    float4 v[16];
    const uint32_t r = lane >> 3, c = (lane & 7) * 4;
    // of load i: its rows and columns (wide tasks: eight row groups of a 32-column strip, then the next strip)
    auto row = [&](uint32_t i) { return (t.narrow ? i >> 1 : i & 7) * 4 + r; };
    auto col = [&](uint32_t i) { return (t.narrow ? i & 1 : i >> 3) * 32 + c; };
#pragma unroll
    for (uint32_t i = 0; i < 16; ++i)
      v[i] = __ldg(reinterpret_cast<const float4*>(t.codes + static_cast<size_t>(row(first + i)) * t.out_val + col(first + i) * 4));
#pragma unroll
    for (uint32_t i = 0; i < 16; ++i)
      *reinterpret_cast<uint2*>(place.element(row(first + i), col(first + i))) =
          make_uint2(pack_bf16x2(v[i].x, v[i].y), pack_bf16x2(v[i].z, v[i].w));
  }
}

// The task (or half of it) to its place; the warp's own 128 bytes at `tab` take the table, rounded once to bf16
// (round-to-nearest-even).  Outliers (Section 6: they keep their original value) follow, the warp's own only.
template <typename Place>
__device__ __forceinline__ void finish_task(const DecodeTask& t, const TaskLoads& f, uint16_t* tab, const Place& place,
                                            uint32_t lane, uint32_t half) {
  if (t.bits == 32) { unpack_raw(t, place, lane, half); return; }
  if (t.bits == 0) return;
  tab[lane] = bf16_bits(f.c0);
  tab[lane + 32] = bf16_bits(f.c1);
  __syncwarp();
  switch (t.bits) {
    case 2: unpack_task<2>(f.w, place, tab, lane, half); break;
    case 3: unpack_task<3>(f.w, place, tab, lane, half); break;
    case 4: unpack_task<4>(f.w, place, tab, lane, half); break;
    case 5: unpack_task<5>(f.w, place, tab, lane, half); break;
    case 6: unpack_task<6>(f.w, place, tab, lane, half); break;
    default: break;
  }
  __syncwarp();                        // the slots below are written; the table may be overwritten by the next task
  uint32_t rc = f.rc;
  float val = f.val;
  for (uint32_t o = lane; o < t.n_out;) {
    uint32_t row, col;
    const bool inside = outlier_place(t, rc, row, col);
    const bool second = t.narrow ? row >= 32 : col >= 64;
    if (inside && (half == 0 || second == (half == 2))) *reinterpret_cast<uint16_t*>(place.element(row, col)) = bf16_bits(val);
    o += 32;
    if (o < t.n_out) {
      rc = __ldg(reinterpret_cast<const uint32_t*>(t.codes + t.out_rc) + o);
      val = __ldg(reinterpret_cast<const float*>(t.codes + t.out_val) + o);
    }
  }
}

// A decoded task (SwizzledPlace, 8 KB at `tile`) to its place in the working buffer `dst` (see expand.cu).  One lane; the caller
// has fenced the writes to the tile.  The copy is a bulk group of its own.
__device__ __forceinline__ void store_expanded(const DecodeTask& t, const uint8_t* tile, uint8_t* dst) {
  uint8_t* to = dst + static_cast<size_t>(expanded_at(t)) * 4096;
  const uint32_t from = smem_addr(tile), apart = t.narrow ? 4096u : 16384u;     // the block's next 32 rows, or the next 64 columns
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], 4096;" ::"l"(to), "r"(from) : "memory");
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], 4096;" ::"l"(to + apart), "r"(from + 4096) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// ---------------------------------------------------------------------------------------
// TMA / mbarrier helpers local to this kernel
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// [128 rows x 64 columns] box at (column k0, row m0); rows past the tensor's extent arrive as zeros.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int k0, int m0, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(k0), "r"(m0), "r"(bar)
      : "memory");
}
// K-major, 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;                 // leading byte offset: unused for this layout
  d |= static_cast<uint64_t>(1024 >> 4) << 32;         // stride byte offset
  d |= static_cast<uint64_t>(1) << 46;                 // descriptor version for sm_100
  d |= static_cast<uint64_t>(2) << 61;                 // layout type: 128-byte swizzle
  return d;
}

// ---------------------------------------------------------------------------------------
// Thread-block clusters: rank, barrier, the other CTA's barriers
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {     // every thread of both CTAs
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t rank) {   // same offset in CTA `rank`
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// An arrival with release semantics at CTA scope only: enough where it hands over tensor memory (ordered by the tcgen05
// fences), and it does not wait for the thread's earlier global stores to reach the cluster's point of coherence, which
// the cluster-scope form does.
__device__ __forceinline__ void mbar_arrive_cluster_cta_scope(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// two floats per instruction
__device__ __forceinline__ uint64_t pack_f32x2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// erf-GELU of two values.  erf through the rational approximation 7.1.26 of Abramowitz & Stegun (absolute error
// below 1.5e-7, three orders of magnitude under the bf16 rounding of the result) with the hardware
// exponential; the epilogue runs it for every element of the FFN1 output.
// With t = 1 / (1 + p |v| / sqrt 2) and q(t) the polynomial:  gelu(v) = max(v, 0) - |v| t q(t) / 2 exp(-v^2 / 2).
// All but the two special functions work on pairs (their unit takes 16 lanes a cycle, so a 128 x 256 tile's GELU is 4096 cycles of
// it; one reciprocal for a pair took FFN1 no less time, and other bits).
__device__ __forceinline__ uint64_t gelu_erf_x2(uint64_t v) {
  const auto both = [](float c) { return pack_f32x2(c, c); };
  float d0, d1, t0, t1, e0, e1, v0, v1;
  unpack_f32x2(v, v0, v1);
  const uint64_t abs_v = pack_f32x2(fminf(fabsf(v0), 1e30f), fminf(fabsf(v1), 1e30f));     // finite: t is 0 for an infinite v
  unpack_f32x2(fma_f32x2(abs_v, both(0.3275911f * 0.70710678118654752440f), both(1.0f)), d0, d1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t0) : "f"(d0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t1) : "f"(d1));
  const uint64_t t = pack_f32x2(t0, t1);
  uint64_t q = fma_f32x2(t, both(0.5f * 1.061405429f), both(0.5f * -1.453152027f));
  q = fma_f32x2(q, t, both(0.5f * 1.421413741f));
  q = fma_f32x2(q, t, both(0.5f * -0.284496736f));
  q = fma_f32x2(q, t, both(0.5f * 0.254829592f));
  unpack_f32x2(mul_f32x2(mul_f32x2(v, v), both(-0.72134752044448170368f)), e0, e1);     // exp(-v^2 / 2) = 2^(v^2 * (-log2(e) / 2))
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(e0));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(e1));
  const uint64_t minus_tail = mul_f32x2(mul_f32x2(abs_v, t), q) ^ 0x8000000080000000ull;
  return fma_f32x2(minus_tail, pack_f32x2(e0, e1), pack_f32x2(fmaxf(v0, 0.f), fmaxf(v1, 0.f)));
}

// 16 accumulator columns + bias (16-byte aligned), erf-GELU if asked for.
template <bool GELU>
__device__ __forceinline__ void bias_act16(const uint32_t (&r)[16], const float* bias_sm, float (&v)[16]) {
#pragma unroll
  for (int i = 0; i < 16; i += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bias_sm + i);
    uint64_t lo = add_f32x2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), pack_f32x2(b.x, b.y));
    uint64_t hi = add_f32x2(pack_f32x2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), pack_f32x2(b.z, b.w));
    if constexpr (GELU) { lo = gelu_erf_x2(lo); hi = gelu_erf_x2(hi); }
    unpack_f32x2(lo, v[i], v[i + 1]);
    unpack_f32x2(hi, v[i + 2], v[i + 3]);
  }
}

// 16 output columns of the warp's 32 rows: every lane comes with its own row's values, and the lanes of a group of G (two
// for bf16, four for fp32) exchange 16-byte pieces so that a store covers whole 32- or 64-byte runs of fewer rows.  A lane
// per row touches 32 lines with every store, and the load/store unit takes a cycle for each: 4096 cycles for a 128 x 128
// fp32 tile, as long as 64 of its MMAs take.
// `first` = row (lane - lane % G) of the output at the block's first column; rows_left = how many rows from there exist.
template <typename OutT>
__device__ __forceinline__ void store_block16(const float (&v)[16], OutT* first, int ldo, int rows_left, uint32_t lane) {
  constexpr uint32_t G = sizeof(OutT) == 2 ? 2 : 4;
  uint4 c[G];
#pragma unroll
  for (uint32_t i = 0; i < G; ++i) {
    if constexpr (sizeof(OutT) == 2)
      c[i] = make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                        pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
    else
      c[i] = make_uint4(__float_as_uint(v[4 * i]), __float_as_uint(v[4 * i + 1]), __float_as_uint(v[4 * i + 2]), __float_as_uint(v[4 * i + 3]));
  }
#pragma unroll
  for (uint32_t step = 1; step < G; step <<= 1) {      // piece i of lane j <-> piece j of lane i, a bit at a time
    const bool up = (lane & step) != 0;
#pragma unroll
    for (uint32_t i = 0; i < G; ++i) {
      if (i & step) continue;
      uint4 &lo = c[i], &hi = c[i | step];
      const uint4 give = up ? lo : hi;
      uint4 got;
      got.x = __shfl_xor_sync(0xffffffffu, give.x, step); got.y = __shfl_xor_sync(0xffffffffu, give.y, step);
      got.z = __shfl_xor_sync(0xffffffffu, give.z, step); got.w = __shfl_xor_sync(0xffffffffu, give.w, step);
      if (up) lo = got; else hi = got;
    }
  }
  OutT* dst = first + (lane & (G - 1)) * (16 / sizeof(OutT));
#pragma unroll
  for (uint32_t i = 0; i < G; ++i)
    if (static_cast<int>(i) < rows_left) *reinterpret_cast<uint4*>(dst + static_cast<size_t>(i) * ldo) = c[i];
}
// The first row of the lane's exchange group.
template <typename OutT>
__device__ __forceinline__ int group_row(int t, uint32_t lane) { return t - static_cast<int>(lane & (sizeof(OutT) == 2 ? 1u : 3u)); }

struct PrefetchRanges {
  const uint8_t* ptr[4];
  uint32_t bytes[4];
};

// Pulls [ptr, ptr + bytes) into L2, one 128-byte line per instruction, the range shared out over
// `n_threads` threads of which this is number `t`.  Packed shards are read once per forward, so without
// this every decode starts with address translation and DRAM latency on its critical path.
__device__ __forceinline__ void prefetch_range_l2(const uint8_t* ptr, uint32_t bytes, uint32_t t, uint32_t n_threads) {
  // plain loads whose values are dropped: unlike a prefetch hint they also bring the translation in
  uint32_t sink = 0;
  for (uint32_t off = t * 128u; off < bytes; off += n_threads * 128u) {
    uint32_t v;
    asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(v) : "l"(ptr + off) : "memory");
    sink |= v;
  }
  asm volatile("" ::"r"(sink));
}

// ---------------------------------------------------------------------------------------
// Decode of one job's weight tile by all warps of the CTA.  The first task's loads are issued by `begin`, as early as
// the caller can; `finish` ends with the tile visible to the tensor core (proxy fence + CTA barrier).
// ---------------------------------------------------------------------------------------
struct TileDecode {
  DecodeTask task;
  TaskLoads loads;
  uint32_t unit, half;
  // a tile with at most half as many tasks as the CTA has warps: two warps share a task (half the decode latency)
  static __device__ __forceinline__ bool split(uint32_t task_stride) { return 2 * task_stride <= kWarps; }
  __device__ __forceinline__ void begin(const DecodeTask* tasks, uint32_t task_stride, uint32_t tid) {
    const uint32_t lane = tid & 31, warp = tid >> 5;
    unit = split(task_stride) ? warp >> 1 : warp;
    half = split(task_stride) ? 1 + (warp & 1) : 0;
    task.bits = 0;
    if (unit < task_stride) {
      task = load_task(tasks + unit);
      issue_loads(task, lane, loads);
    }
  }
  __device__ __forceinline__ void finish(const DecodeTask* tasks, uint32_t task_stride, uint16_t* warp_tables, uint8_t* wsm,
                                         uint32_t n_rows, uint32_t tid) {
    const uint32_t lane = tid & 31, warp = tid >> 5;
    uint16_t* tab = warp_tables + warp * kTableStride;
    while (unit < task_stride) {
      finish_task(task, loads, tab, TilePlace(wsm, n_rows, task), lane, half);
      unit += split(task_stride) ? kWarps / 2 : kWarps;
      if (unit < task_stride) {
        task = load_task(tasks + unit);
        issue_loads(task, lane, loads);
      }
    }
    fence_proxy_async_smem();
    __syncthreads();
  }
};

// ---------------------------------------------------------------------------------------
// Two-CTA (cta_group::2) forms of the tensor-memory, TMA and MMA helpers
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t n_cols) {     // one warp in each CTA
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(n_cols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t n_cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(n_cols) : "memory");
}
// Own tile into own shared memory, completion bytes credited to the barrier at `bar_cluster_addr` (CTA 0's).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int k0, int m0,
                                                 uint32_t bar_cluster_addr) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(k0), "r"(m0), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_ss_x4_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t a_step,
                                                     uint32_t b_step, uint32_t idesc, uint32_t accumulate_first) {
  asm volatile(
      "{\n\t.reg .pred p0, p1;\n\t.reg .b64 a1, a2, a3, b1, b2, b3, as, bs;\n\t"
      "setp.ne.b32 p0, %6, 0;\n\t"
      "setp.eq.b32 p1, 0, 0;\n\t"
      "cvt.u64.u32 as, %3;\n\t"
      "cvt.u64.u32 bs, %4;\n\t"
      "add.u64 a1, %1, as;\n\tadd.u64 a2, a1, as;\n\tadd.u64 a3, a2, as;\n\t"
      "add.u64 b1, %2, bs;\n\tadd.u64 b2, b1, bs;\n\tadd.u64 b3, b2, bs;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %5, p0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %5, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %5, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %5, p1;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(a_step), "r"(b_step), "r"(idesc), "r"(accumulate_first)
      : "memory");
}
// Completion of all MMAs issued so far -> the barrier at this offset in both CTAs.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(static_cast<uint16_t>(3)) : "memory");
}

}  // namespace
}  // namespace sti
