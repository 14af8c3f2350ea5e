// GEMM over decoded weights for calls of many tokens: Y[T, N] = X[T, K] W[N, K]^T, W in the working buffer that expand.cu
// fills (bf16, blocks of 128 features x 64 columns, already swizzled).
//
// Persistent pairs of CTAs (cta_group::2), one CTA per SM.  A pair takes tiles of 256 tokens x NT features (256 or 128): each
// CTA loads its own 128 tokens and its half of the features, 64 columns at a time, into a ring of stages; CTA 0 issues
// the MMAs (M = 256, N = NT) into one of two accumulators in tensor memory (at NT = 256 all of it) while eight epilogue warps of
// each CTA drain the other: tcgen05.ld -> bias / erf-GELU -> shared memory -> bulk tensor store.  fp32 outputs may be split
// along K; every split writes a plane of its own, which the LayerNorm after it adds up.
//
//   warp 0      producer: TMA boxes of activations and weights, both CTAs' bytes reported to CTA 0's `full` barriers
//   warp 1      MMA issuer (CTA 0)
//   warps 2-3   decode the same matrix of the next layer into the other working buffer (expand.cu): it is ready a layer ahead;
//               at NT = 128 warps 12-13 as well
//   warps 4-11  epilogue, two per tensor-memory lane quadrant, half of the tile's features each
//
// Bound: the MMAs, as long as a launch has several waves of tiles: a chunk of 64 columns takes 540 cycles at NT = 256 (the tensor
// core's 512) and 395 at 128 (24 KB written to and 24 KB read from shared memory: 384).  With one wave as much goes
// into what is around them: 2.3 us until the first chunk is there, 2.3 (erf-GELU 4.3) for the last tile's epilogue, 0.75 to end.
// BERT-large, us per launch, fused two-CTA kernels with one decoded tile per CTA -> this one: QKV, O, FFN1, FFN2 of 4096 tokens
// 28 / 12 / 39 / 42 -> 21 / 11 / 28 / 25, of 16,384 tokens 95 / 42 / 143 / 145 -> 80 / 38 / 110 / 111 (power cap), of 1024 tokens
// 14.6 / 9.4 / 18.0 / 13.8 -> 10.5 / 8.7 / 12.9 / 13.3.
//
// Every wait is bounded (see mbar_wait_bounded).
#include <type_traits>

#include "gemm_device.cuh"

namespace sti {
namespace {

constexpr uint32_t kWideMaxStages = 8;
// Shared memory: barriers, a bias slice per epilogue warp and a table per decoding warp; then, 1024-aligned, the stages, the
// epilogue warps' output tiles and the decoding warps' tasks.
constexpr uint32_t kWideBiasOffset = 512, kWideBiasPerWarp = 128, kWideTableOffset = kWideBiasOffset + kEpilogueWarps * kWideBiasPerWarp * 4;
constexpr uint32_t kWideMaxDecodeWarps = 4;
constexpr uint32_t kWideHeaderBytes = 6144;
constexpr uint32_t kWideDecodeWarp0 = 2, kWideLateDecodeWarp0 = kEpilogueWarp0 + kEpilogueWarps;      // 2, 3, then 12, 13
constexpr uint32_t kOutTileBytes = 4096;                 // 32 rows of 128 bytes

struct WideHeader {
  uint64_t full[kWideMaxStages];   // CTA 0: both CTAs' boxes of the stage have landed
  uint64_t empty[kWideMaxStages];  // both CTAs: the MMAs that read the stage have completed
  uint64_t acc_full[2];            // both CTAs: the accumulator is complete
  uint64_t acc_empty[2];           // CTA 0: both CTAs' epilogue warps have read it
  uint64_t drain;                  // failure path only
  uint32_t tmem_base;
};
static_assert(sizeof(WideHeader) <= kWideBiasOffset, "barriers before the bias slices");
static_assert(kWideTableOffset + kWideMaxDecodeWarps * kTableStride * 2 <= kWideHeaderBytes && kWideHeaderBytes % 1024 == 0, "header");

template <uint32_t NT>
struct Wide {
  static constexpr uint32_t kStageBytes = kBoxBytes + NT / 2 * 128;       // 128 tokens and NT / 2 features, 64 columns each
  static constexpr uint32_t kDecodeWarps = NT == 256 ? 2 : 4;             // many tokens leave them time, few leave the shared memory
  static constexpr uint32_t kThreads = 32 * (kWideLateDecodeWarp0 + kDecodeWarps - 2);
  static constexpr uint32_t kOutTiles = NT == 256 ? 1 : 2;                // per epilogue warp
  static constexpr uint32_t kOutBytes = kEpilogueWarps * kOutTiles * kOutTileBytes, kDecodeBytes = kDecodeWarps * 8192;
  static constexpr uint32_t kFit = (227u * 1024 - kWideHeaderBytes - kOutBytes - kDecodeBytes) / kStageBytes;
  static constexpr uint32_t kStages = kFit < kWideMaxStages ? kFit : kWideMaxStages;
  static constexpr uint32_t kSmemBytes = kWideHeaderBytes + kStages * kStageBytes + kOutBytes + kDecodeBytes;
};

// Tiles of a launch, features first, then token pairs, then K splits: the pairs that run together share activations.
struct WideTile { uint32_t n, m, c0, c1, split; };
__device__ __forceinline__ WideTile wide_tile(const WideShape& s, uint32_t index) {
  WideTile t;
  t.n = index % s.n_tiles;
  const uint32_t rest = index / s.n_tiles;
  t.m = rest % s.m_pairs;
  t.split = rest / s.m_pairs;
  t.c0 = t.split * s.k_chunks / s.splits;
  t.c1 = (t.split + 1) * s.k_chunks / s.splits;
  return t;
}

// The chunks of 64 columns that a pair walks, tile after tile.
struct WideWalk {
  const WideShape& s;
  uint32_t index, step, n_all, kc;
  WideTile tile;
  __device__ __forceinline__ WideWalk(const WideShape& shape, uint32_t first, uint32_t n_clusters)
      : s(shape), index(first), step(n_clusters), n_all(shape.n_tiles * shape.m_pairs * shape.splits) { enter(); }
  __device__ __forceinline__ bool done() const { return index >= n_all; }
  __device__ __forceinline__ void enter() {
    tile = wide_tile(s, index);
    kc = tile.c0;
  }
  __device__ __forceinline__ void next() {
    if (++kc == tile.c1) { index += step; enter(); }
  }
};

// 32 rows x 128 bytes at (column, row, plane); rows past the tensor's end are left out.  A bulk group of its own.
__device__ __forceinline__ void store_out_tile(const CUtensorMap* map, uint32_t src, int col, int row, int plane) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];\n\tcp.async.bulk.commit_group;"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(col), "r"(row), "r"(plane), "r"(src) : "memory");
}

// A warp's part of an accumulator: `n_cols` columns (a multiple of 64) of its 32 token rows -> bias / erf-GELU -> 128-byte rows in
// shared memory (swizzled: lanes hold consecutive rows) -> bulk tensor store, so that whole lines leave the SM.  The loop
// over 16 columns is rolled and loads one step ahead.  `flush(col)` stores the tile that ends before column `col`; it returns
// where the next one goes.  `handed_over` runs once the accumulator has been read.
template <bool GELU, typename OutT, typename Flush, typename Done>
__device__ __forceinline__ void drain(uint32_t taddr, uint32_t n_cols, const float* bias_sm, uint8_t* tile, uint32_t lane, Flush flush, Done handed_over) {
  constexpr uint32_t kTileCols = 128 / sizeof(OutT), kPieces = sizeof(OutT);       // 16-byte pieces that 16 columns make: 2 or 4
  uint32_t next[16];
  tmem_ld_32x32b_x16(taddr, next);
  tc_wait_ld_x16(next);
#pragma unroll 1
  for (uint32_t col = 0; col < n_cols; col += 16) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = next[i];
    if (col + 16 < n_cols) tmem_ld_32x32b_x16(taddr + col + 16, next);
    float v[16];
    bias_act16<GELU>(r, bias_sm + col, v);
    const uint32_t piece0 = (col % kTileCols) / 16 * kPieces;
#pragma unroll
    for (uint32_t i = 0; i < kPieces; ++i) {
      uint4 c;
      if constexpr (sizeof(OutT) == 2)
        c = make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                       pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
      else
        c = make_uint4(__float_as_uint(v[4 * i]), __float_as_uint(v[4 * i + 1]), __float_as_uint(v[4 * i + 2]), __float_as_uint(v[4 * i + 3]));
      *reinterpret_cast<uint4*>(tile + lane * 128 + (((piece0 + i) ^ (lane & 7)) << 4)) = c;
    }
    tc_wait_ld_x16(next);
    if (col + 32 >= n_cols && col + 16 < n_cols) handed_over();      // the last 16 columns are in registers
    if ((col + 16) % kTileCols == 0) tile = flush(col + 16);
  }
}

// One kernel for every GEMM of a layer: the output kind is a launch parameter, so that the code stays in the instruction caches
// from launch to launch.
template <uint32_t NT>
__global__ void __launch_bounds__(Wide<NT>::kThreads, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap omap,
                 const WideShape s, int kind, int weights_ready, const float* __restrict__ bias, const int32_t* __restrict__ bias_off,
                 int* __restrict__ err, const DecodeTask* __restrict__ tasks, uint32_t n_tasks, uint8_t* __restrict__ expanded,
                 unsigned long long* stamps) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr uint32_t kStages = Wide<NT>::kStages, kStageBytes = Wide<NT>::kStageBytes, kTmemCols = 2 * NT;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // uniform to the compiler
  if (tid == 0) { stamp_min(stamps, STAMP_FIRST_START); stamp_max(stamps, STAMP_LAST_START); }
  const uint32_t rank = cluster_ctarank(), cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  WideHeader* hdr = reinterpret_cast<WideHeader*>(smem);
  const uint32_t ring = smem_addr(smem) + kWideHeaderBytes;
  if (tid == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&xmap)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&wmap)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&omap)) : "memory");
  }
  if (tid == 0) {
    for (uint32_t i = 0; i < kStages; ++i) {
      mbar_init(smem_addr(&hdr->full[i]), 1);
      mbar_init(smem_addr(&hdr->empty[i]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_addr(&hdr->acc_full[b]), 1);
      mbar_init(smem_addr(&hdr->acc_empty[b]), 2 * kEpilogueWarps);
    }
    mbar_init(smem_addr(&hdr->drain), 1);
    mbar_fence_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_addr(&hdr->tmem_base), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = hdr->tmem_base;
  cluster_sync_all();                  // all barriers of the pair are initialised
  const uint32_t n_all = s.n_tiles * s.m_pairs * s.splits;
  const bool decoder = warp == kWideDecodeWarp0 || warp == kWideDecodeWarp0 + 1 || warp >= kWideLateDecodeWarp0;
  bool failed = false;
  // this CTA's half of a tile's features, one chunk: a whole block of 128 features, or half of one
  auto load_weights = [&](const WideWalk& at, uint32_t stage) {
    const uint32_t block = NT == 256 ? 2 * at.tile.n + rank : at.tile.n;
    const uint32_t row = s.w_row0 + (block * s.k_chunks + at.kc) * 128 + (NT == 256 ? 0 : 64 * rank);
    if (rank == 0) mbar_expect_tx(smem_addr(&hdr->full[stage]), 2 * kStageBytes);
    tma_load_2d_pair(ring + stage * kStageBytes + kBoxBytes, &wmap, 0, static_cast<int>(row), map_to_cta(smem_addr(&hdr->full[stage]), 0));
  };
  auto load_tokens = [&](const WideWalk& at, uint32_t stage) {
    tma_load_2d_pair(ring + stage * kStageBytes, &xmap, static_cast<int>(at.kc * kChunkK), static_cast<int>((2 * at.tile.m + rank) * kTileM),
                     map_to_cta(smem_addr(&hdr->full[stage]), 0));
  };
  // weights that are in place already fill the ring's first round before the preceding kernel has finished
  uint32_t early = 0;
  if (warp == 0 && weights_ready)
    for (WideWalk at(s, cluster, n_clusters); !at.done() && early < kStages; at.next(), ++early) {
      if (elect_one()) load_weights(at, early);
      __syncwarp();
    }
  if (!decoder) {                      // decoding depends on no kernel before this one
    pdl_wait();
    // Not before the wait: by this a kernel that has started knows that everything before the last GEMM over the working buffer
    // has finished (the kernels in between release their successors at once).  Its decoders write the place of their own matrix,
    // which all layers share and which that last GEMM, being another of the four, does not read: of QKV and O, or FFN1 and FFN2,
    // the second follows whenever the first is run, and a layer that decodes ahead has all four.
    pdl_launch_dependents();
  }
  if (tid == 0) stamp_min(stamps, STAMP_RELEASE);

  if (warp == 0) {
    // The whole warp walks the loop converged, one elected lane issues: a loop that one lane runs alone took 560 cycles a chunk.
    uint32_t c = 0, stage = 0, phase = 0;
    for (WideWalk at(s, cluster, n_clusters); !at.done(); at.next(), ++c) {
      if (c >= kStages && !__all_sync(0xffffffffu, mbar_wait_bounded(smem_addr(&hdr->empty[stage]), phase))) { failed = true; break; }
      if (elect_one()) {
        if (c >= early) load_weights(at, stage);
        load_tokens(at, stage);
      }
      __syncwarp();
      if (++stage == kStages) { stage = 0; if (c >= kStages) phase ^= 1; }
    }
    // give the copies in flight a bounded chance to land (CTA 0's barriers count both CTAs' bytes, CTA 1 leaves with it)
    if (failed && rank == 0)
      for (uint32_t k = c > kStages ? c - kStages : 0; k < c; ++k)
        if (!mbar_wait_bounded(smem_addr(&hdr->full[k % kStages]), (k / kStages) & 1)) break;
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((NT >> 3) << 17) | ((256u >> 4) << 24);
      const uint64_t a_desc0 = umma_smem_desc_sw128(ring), b_desc0 = umma_smem_desc_sw128(ring + kBoxBytes);
      uint32_t total = 0;              // chunks this pair walks
      for (uint32_t i = cluster; i < n_all; i += n_clusters) { const WideTile t = wide_tile(s, i); total += t.c1 - t.c0; }
      uint32_t c = 0, stage = 0, phase = 0, ti = 0;
      for (uint32_t i = cluster; i < n_all && !failed; i += n_clusters, ++ti) {
        const WideTile t = wide_tile(s, i);
        const uint32_t buf = ti & 1;
        if (ti >= 2 && !__all_sync(0xffffffffu, mbar_wait_bounded(smem_addr(&hdr->acc_empty[buf]), ((ti >> 1) - 1) & 1))) {
          failed = true;
          break;
        }
        for (uint32_t kc = t.c0; kc < t.c1; ++kc, ++c) {
          if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_addr(&hdr->full[stage]), phase))) { failed = true; break; }
          tc_fence_after_sync();
          if (elect_one()) {
            const uint64_t step = stage * (kStageBytes >> 4);
            umma_bf16_ss_x4_pair(tmem_base + buf * NT, a_desc0 + step, b_desc0 + step, 2, 2, idesc, kc != t.c0 ? 1u : 0u);
            if (c + kStages < total) umma_commit_pair(smem_addr(&hdr->empty[stage]));      // only if the stage is refilled
            if (kc + 1 == t.c1) umma_commit_pair(smem_addr(&hdr->acc_full[buf]));
          }
          __syncwarp();
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
      if (failed && c > 0) {           // outstanding MMAs: one more bounded chance before tensor memory is freed
        if (elect_one()) umma_commit_pair(smem_addr(&hdr->drain));
        __syncwarp();
        (void)mbar_wait_bounded(smem_addr(&hdr->drain), 0);
      }
    }
  } else if (decoder) {
    const uint32_t index = warp < kEpilogueWarp0 ? warp - kWideDecodeWarp0 : warp - kWideLateDecodeWarp0 + 2;
    const uint32_t stride = gridDim.x * Wide<NT>::kDecodeWarps;
    uint8_t* tile = smem + kWideHeaderBytes + kStages * kStageBytes + Wide<NT>::kOutBytes + index * 8192;
    uint16_t* table = reinterpret_cast<uint16_t*>(smem + kWideTableOffset) + index * kTableStride;
    uint32_t next = blockIdx.x + index * gridDim.x;
    if (next < n_tasks) {
      DecodeTask task = load_task(tasks + next);
      TaskLoads loads;
      issue_loads(task, lane, loads);
      while (true) {
        next += stride;
        const bool more = next < n_tasks;
        DecodeTask task2;
        TaskLoads loads2;
        if (more) { task2 = load_task(tasks + next); issue_loads(task2, lane, loads2); }     // under this task's unpacking
        finish_task(task, loads, table, SwizzledPlace(tile, task), lane, 0);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          store_expanded(task, tile, expanded);
          if (more) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          else asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        if (!more) break;
        task = task2;
        loads = loads2;
      }
    }
  } else {
    const uint32_t q = warp & 3, half = (warp - kEpilogueWarp0) >> 2;      // tensor-memory lane quadrant, half of the tile's columns
    float* bias_sm = reinterpret_cast<float*>(smem + kWideBiasOffset) + (warp - kEpilogueWarp0) * kWideBiasPerWarp;
    uint8_t* const tiles = smem + kWideHeaderBytes + kStages * kStageBytes + (warp - kEpilogueWarp0) * Wide<NT>::kOutTiles * kOutTileBytes;
    uint32_t ti = 0, slot = 0;
    for (uint32_t i = cluster; i < n_all; i += n_clusters, ++ti) {
      const WideTile t = wide_tile(s, i);
      const uint32_t buf = ti & 1, n0 = t.n * NT + half * (NT / 2);
      __syncwarp();
      for (uint32_t k = lane; k < NT / 2; k += 32) {
        const uint32_t n = n0 + k;
        bias_sm[k] = bias != nullptr && n < s.n ? __ldg(bias + __ldg(bias_off + (n >> 6)) + (n & 63)) : 0.f;
      }
      __syncwarp();
      uint32_t ok = 1;
      if (lane == 0) ok = mbar_wait_bounded(smem_addr(&hdr->acc_full[buf]), (ti >> 1) & 1) ? 1u : 0u;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) { failed = true; break; }
      tc_fence_after_sync();
      const int row = static_cast<int>((2 * t.m + rank) * kTileM + q * 32);
      const uint32_t taddr = tmem_base + ((q * 32) << 16) + buf * NT + half * (NT / 2);
      auto handed_over = [&]() {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_cta_scope(map_to_cta(smem_addr(&hdr->acc_empty[buf]), 0));
      };
      auto run = [&](auto out, auto gelu) {
        using Out = decltype(out);
        constexpr uint32_t kTileCols = 128 / sizeof(Out);
        auto flush = [&](uint32_t end) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            const uint32_t n = n0 + end - kTileCols;
            // the next tile's place must have been read by the store before this one
            if (n < s.n && row < static_cast<int>(s.T)) {
              store_out_tile(&omap, smem_addr(tiles + slot * kOutTileBytes), static_cast<int>(s.plane64 ? 0 : n), row,
                             static_cast<int>(s.plane64 ? n >> 6 : t.split));
              asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(Wide<NT>::kOutTiles - 1) : "memory");
            } else {
              asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            }
          }
          __syncwarp();
          slot = (slot + 1) % Wide<NT>::kOutTiles;
          return tiles + slot * kOutTileBytes;
        };
        drain<decltype(gelu)::value, Out>(taddr, NT / 2, bias_sm, tiles + slot * kOutTileBytes, lane, flush, handed_over);
      };
      if (kind == GEMM_BF16_TO_F32) run(0.f, std::false_type());
      else if (kind == GEMM_BF16_TO_BF16_GELU) run(__nv_bfloat16(), std::true_type());
      else run(__nv_bfloat16(), std::false_type());
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  if (failed && lane == 0) atomicCAS(err, ERR_NONE, ERR_WAIT_TIMEOUT);
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();      // neither CTA frees tensor memory or exits while the pair's MMAs may still use it
  if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
  if (tid == 0) stamp_max(stamps, STAMP_LAST_END);
}

template <uint32_t NT>
cudaError_t launch_t(GemmKind kind, const WideLaunch& p, cudaStream_t s) {
  return launch_kernel_cluster(gemm_wide_kernel<NT>, dim3(2 * p.clusters), dim3(Wide<NT>::kThreads), Wide<NT>::kSmemBytes, s, p.pdl, 2u,
                               p.xmap, p.wmap, p.omap, p.shape, static_cast<int>(kind), p.weights_ready ? 1 : 0, p.bias, p.bias_off, p.err,
                               p.beside.tasks, p.beside.n_tasks, p.beside.dst, p.stamps);
}

}  // namespace

cudaError_t gemm_wide_configure() {
  cudaError_t e = cudaFuncSetAttribute(gemm_wide_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, Wide<256>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_wide_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Wide<128>::kSmemBytes);
  return e;
}

cudaError_t launch_gemm_wide(GemmKind kind, const WideLaunch& p, cudaStream_t s) {
  return p.nt == 256 ? launch_t<256>(kind, p, s) : launch_t<128>(kind, p, s);
}

}  // namespace sti
