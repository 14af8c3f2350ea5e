// Per-head scaled-dot-product attention over the kept heads (Section 2.1: each attention head
// independently contributes one representation; Section 4.2: any subset of heads executes), for short sequences and
// small batches (attention_tc.cu: long sequences of many heads).
//
// One CTA = (tile of 16 QW queries, kept head, sequence) with QW x KS warps: warp (qg, ks) has 16 query rows and every KS-th
// block of KB keys.  K and V of the sequence (<= 512 keys, padded keys as zeros) come into shared memory with cp.async,
// K first, so that the scores start while V is under way; scores and the probability-value product run on mma.sync
// m16n8k16 bf16 with fp32 accumulation and ldmatrix fragments, softmax online in registers with shuffles over the four
// lanes that share a row.  With KS > 1 the splits' (max, sum, output) triples meet in shared memory (where K and V were),
// and each split finishes its share of the output columns.
//
// Bound: latency.  With few CTAs a CTA's serial chain is what counts - its load, one or two key blocks, the merge - so the
// keys are split; with many the loads of K and V and the exponentials, so that more warps share them.
// Measured per launch inside a layer, end to end of the kernels around it: 1 x 256 tokens of 16 heads 7.0 -> 4.3 us,
// 1 x 128 of 12 5.6 -> 3.1, 8 x 128 of 16 10.4 -> 4.5, 3 x 441 of 10 17.2 -> 10.0 (4-byte fragment loads and stores, K and V
// awaited together, CTAs piled onto few SMs).
#include <algorithm>

#include <cuda_bf16.h>

#include "sti_device.cuh"
#include "sti_kernels.h"

namespace sti {
namespace {

constexpr int kHeadDim = 64;
constexpr int kKStride = 64 + 8;      // bf16 per K / V row in shared memory: ldmatrix rows fall on different banks
constexpr int kMergeWords = 36;       // a warp's triple: two maxima, two sums, 32 outputs per lane

struct AttnArgs {
  const uint16_t* qkv;      // [(kept head * 3 + {Q,K,V})][T][64] bf16
  uint16_t* out;            // [T][n_kept * 64] bf16
  const int32_t* seq_lens;  // optional, per sequence
  int n_kept, batch, seq;
  unsigned long long* stamps;   // profiling record or null
};

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ float exp2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <int QW, int KS, int KB>      // eight warps per CTA come in large grids: two to an SM
__global__ void __launch_bounds__(32 * QW * KS, QW == 8 ? 2 : 0)
attention_kernel(AttnArgs p) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int kThreads = 32 * QW * KS;
  const int qt = blockIdx.x, hi = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int qg = warp % QW, ks = warp / QW;
  const int g = lane >> 2, t4 = lane & 3;
  const int L = p.seq, T = p.batch * L;

  pdl_launch_dependents();
  if (tid == 0) { stamp_min(p.stamps, STAMP_FIRST_START); stamp_max(p.stamps, STAMP_LAST_START); }
  const uint16_t* Qg = p.qkv + (static_cast<size_t>(hi * 3 + 0) * T + static_cast<size_t>(b) * L) * kHeadDim;
  const uint16_t* Kg = p.qkv + (static_cast<size_t>(hi * 3 + 1) * T + static_cast<size_t>(b) * L) * kHeadDim;
  const uint16_t* Vg = p.qkv + (static_cast<size_t>(hi * 3 + 2) * T + static_cast<size_t>(b) * L) * kHeadDim;
  pdl_wait();          // q, k, v (and possibly seq_lens) come from the preceding kernels
  if (tid == 0) stamp_min(p.stamps, STAMP_RELEASE);
  int valid = L;
  if (p.seq_lens != nullptr) {
    valid = p.seq_lens[b];
    valid = valid < 0 ? 0 : (valid > L ? L : valid);
  }
  const int n_blocks = (valid + KB - 1) / KB, rows = n_blocks * KB;

  const uint32_t qs_addr = smem_addr(smem), ks_addr = qs_addr + QW * 16 * kKStride * 2;
  const uint32_t vs_addr = ks_addr + static_cast<uint32_t>((L + KB - 1) / KB * KB * kKStride * 2);
  // rows first .. first + n of `src` (those from `end` on as zeros)
  auto load_rows = [&](uint32_t dst, const uint16_t* src, int first, int n, int end) {
    for (int idx = tid; idx < n * 8; idx += kThreads) {
      const int row = idx >> 3, piece = idx & 7;
      const bool ok = first + row < end;
      cp_async16(dst + static_cast<uint32_t>(row * kKStride + piece * 8) * 2,
                 src + static_cast<size_t>(ok ? first + row : 0) * kHeadDim + piece * 8, ok ? 16u : 0u);
    }
  };
  load_rows(qs_addr, Qg, qt * QW * 16, QW * 16, L);
  load_rows(ks_addr, Kg, 0, rows, valid);
  asm volatile("cp.async.commit_group;" ::: "memory");
  load_rows(vs_addr, Vg, 0, rows, valid);
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();

  // query fragments of this warp's 16 rows: matrices rows 0-7 and 8-15 for eight dimensions, then for the next eight
  const int q0 = (qt * QW + qg) * 16;
  const uint32_t my_q = qs_addr + static_cast<uint32_t>(qg * 16 * kKStride) * 2;
  uint32_t qa[4][4];
#pragma unroll
  for (int kk = 0; kk < 4; ++kk)
    ldmatrix_x4(my_q + static_cast<uint32_t>((lane & 15) * kKStride + kk * 16 + (lane >> 4) * 8) * 2, qa[kk]);

  const float scale_log2 = 0.125f * 1.4426950408889634f;     // 1/sqrt(64) * log2(e)
  float o[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
  float m_run[2] = {-INFINITY, -INFINITY};                   // of the raw scores
  float l_run[2] = {0.f, 0.f};
  for (int kb0 = 0; kb0 < n_blocks; kb0 += KS) {
    const int kb = kb0 + ks;
    const bool mine = KS == 1 || kb < n_blocks;              // the whole warp
    float s[KB / 8][4];
    if (mine) {
#pragma unroll
      for (int j = 0; j < KB / 8; ++j) {
        s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
        // matrix lane / 8 of a load: the eight dimensions from 8 (lane / 8) on of keys 8 j ..
        const uint32_t krow = ks_addr + static_cast<uint32_t>((kb * KB + j * 8 + (lane & 7)) * kKStride + (lane >> 3) * 8) * 2;
        uint32_t lo[4], hi4[4];
        ldmatrix_x4(krow, lo);
        ldmatrix_x4(krow + 64, hi4);
        mma_bf16_16816(s[j], qa[0], lo[0], lo[1]);
        mma_bf16_16816(s[j], qa[1], lo[2], lo[3]);
        mma_bf16_16816(s[j], qa[2], hi4[0], hi4[1]);
        mma_bf16_16816(s[j], qa[3], hi4[2], hi4[3]);
      }
      if ((kb + 1) * KB > valid) {
#pragma unroll
        for (int j = 0; j < KB / 8; ++j) {
          const int key = kb * KB + j * 8 + 2 * t4;
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (key + (c & 1) >= valid) s[j][c] = -INFINITY;
        }
      }
      float alpha[2], m_scaled[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float m = m_run[r];
#pragma unroll
        for (int j = 0; j < KB / 8; ++j) m = fmaxf(m, fmaxf(s[j][2 * r], s[j][2 * r + 1]));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));      // finite: the block holds a valid key
        m_scaled[r] = m * scale_log2;
        alpha[r] = exp2_ftz(fmaf(m_run[r], scale_log2, -m_scaled[r]));
        m_run[r] = m;
        l_run[r] *= alpha[r];
      }
#pragma unroll
      for (int j = 0; j < KB / 8; ++j) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          s[j][c] = exp2_ftz(fmaf(s[j][c], scale_log2, -m_scaled[c >> 1]));
          l_run[c >> 1] += s[j][c];
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[j][c] *= alpha[c >> 1];
    }
    if (kb0 == 0) {                                          // V has arrived, every thread's pieces of it
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
    }
    if (!mine) continue;
#pragma unroll
    for (int kk = 0; kk < KB / 16; ++kk) {
      uint32_t pa[4];
      pa[0] = pack_bf16x2(s[2 * kk][0], s[2 * kk][1]);
      pa[1] = pack_bf16x2(s[2 * kk][2], s[2 * kk][3]);
      pa[2] = pack_bf16x2(s[2 * kk + 1][0], s[2 * kk + 1][1]);
      pa[3] = pack_bf16x2(s[2 * kk + 1][2], s[2 * kk + 1][3]);
      // matrices of a load: keys 0-7 and 8-15 of this step for eight dimensions, then for the next eight
      const uint32_t vrow = vs_addr + static_cast<uint32_t>((kb * KB + kk * 16 + (lane & 15)) * kKStride + (lane >> 4) * 8) * 2;
#pragma unroll
      for (int jd = 0; jd < 8; jd += 2) {
        uint32_t v4[4];
        ldmatrix_x4_trans(vrow + jd * 16, v4);
        mma_bf16_16816(o[jd], pa, v4[0], v4[1]);
        mma_bf16_16816(o[jd + 1], pa, v4[2], v4[3]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {        // the four lanes of a row hold disjoint keys
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
  }
  const int ldo = p.n_kept * kHeadDim;
  if constexpr (KS == 1) {
    // through the warp's own query rows in shared memory, so that a store covers whole lines
    uint8_t* stage = smem + static_cast<size_t>(qg) * 16 * kKStride * 2;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float inv = l_run[r] > 0.f ? 1.f / l_run[r] : 0.f;
#pragma unroll
      for (int jd = 0; jd < 8; ++jd)
        *reinterpret_cast<uint32_t*>(stage + ((g + 8 * r) * kKStride + jd * 8 + 2 * t4) * 2) = pack_bf16x2(o[jd][2 * r] * inv, o[jd][2 * r + 1] * inv);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = i * 4 + (lane >> 3), piece = lane & 7;
      if (q0 + row < L)
        *reinterpret_cast<uint4*>(p.out + (static_cast<size_t>(b) * L + q0 + row) * ldo + hi * kHeadDim + piece * 8) =
            *reinterpret_cast<const uint4*>(stage + (row * kKStride + piece * 8) * 2);
    }
  } else {
    auto store = [&](int jd, int r, float x, float y) {
      const int row = q0 + g + 8 * r;
      if (row < L)
        *reinterpret_cast<uint32_t*>(p.out + (static_cast<size_t>(b) * L + row) * ldo + hi * kHeadDim + 2 * t4 + jd * 8) = pack_bf16x2(x, y);
    };
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                   // K and V have been read for the last time
    float* merge = reinterpret_cast<float*>(smem);           // [KS][QW][36][32]
    float* mine = merge + (static_cast<size_t>(ks) * QW + qg) * kMergeWords * 32 + lane;
    mine[0 * 32] = m_run[0]; mine[1 * 32] = m_run[1]; mine[2 * 32] = l_run[0]; mine[3 * 32] = l_run[1];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) mine[(4 + j * 4 + c) * 32] = o[j][c];
    __syncthreads();
    float f[KS][2], inv[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      float m = -INFINITY, l = 0.f;
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        f[k][r] = merge[(static_cast<size_t>(k) * QW + qg) * kMergeWords * 32 + r * 32 + lane];
        m = fmaxf(m, f[k][r]);
      }
      const float m_use = m == -INFINITY ? 0.f : m;
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        f[k][r] = exp2_ftz((f[k][r] - m_use) * scale_log2);
        l = fmaf(merge[(static_cast<size_t>(k) * QW + qg) * kMergeWords * 32 + (2 + r) * 32 + lane], f[k][r], l);
      }
      inv[r] = l > 0.f ? 1.f / l : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8 / KS; ++i) {
      const int jd = ks * (8 / KS) + i;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < KS; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          acc[c] = fmaf(merge[((static_cast<size_t>(k) * QW + qg) * kMergeWords + 4 + jd * 4 + c) * 32 + lane], f[k][c >> 1], acc[c]);
      store(jd, 0, acc[0] * inv[0], acc[1] * inv[0]);
      store(jd, 1, acc[2] * inv[1], acc[3] * inv[1]);
    }
  }
  if (p.stamps != nullptr) {
    __syncthreads();
    if (tid == 0) stamp_max(p.stamps, STAMP_LAST_END);
  }
}

template <int QW, int KS, int KB>
size_t attn_smem_bytes(int L) {
  const size_t kv = (static_cast<size_t>((L + KB - 1) / KB * KB) * 2 + QW * 16) * kKStride * 2;
  const size_t merge = KS > 1 ? static_cast<size_t>(KS) * QW * kMergeWords * 32 * 4 : 0;
  return kv > merge ? kv : merge;
}
constexpr size_t kSmSmem = 228 * 1024, kCtaReserved = 1024;
template <int QW, int KS, int KB>
cudaError_t configure_one() {
  return cudaFuncSetAttribute(attention_kernel<QW, KS, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmSmem - kCtaReserved));
}
// A grid that leaves SMs to spare is spread over all of them by asking for as much shared memory as keeps further CTAs off
// an SM: left to itself the hardware puts CTAs onto the same SM while others stay empty (128 CTAs of eight warps, 128 keys:
// 6.4 against 4.6 us).
template <int QW, int KS, int KB>
cudaError_t launch_one(const AttnArgs& a, int sm_count, cudaStream_t s, bool pdl) {
  const dim3 grid((a.seq + 16 * QW - 1) / (16 * QW), a.n_kept, a.batch);
  const size_t n_ctas = static_cast<size_t>(grid.x) * grid.y * grid.z, per_sm = (n_ctas + sm_count - 1) / sm_count;
  size_t smem = attn_smem_bytes<QW, KS, KB>(a.seq);
  if (per_sm <= 4) {
    const size_t too_many = (kSmSmem / (per_sm + 1)) / 1024 * 1024;         // per_sm + 1 CTAs of this size would not fit ...
    const size_t fits = (kSmSmem / per_sm - kCtaReserved) / 1024 * 1024;    // ... and per_sm do
    smem = std::max(smem, std::min(too_many, fits));
  }
  return launch_kernel(attention_kernel<QW, KS, KB>, grid, dim3(32 * QW * KS), smem, s, pdl, a);
}

}  // namespace

cudaError_t attention_configure() {
  cudaError_t e;
  if ((e = configure_one<2, 1, 32>()) != cudaSuccess) return e;
  if ((e = configure_one<2, 2, 64>()) != cudaSuccess) return e;
  if ((e = configure_one<2, 4, 64>()) != cudaSuccess) return e;
  if ((e = configure_one<4, 1, 32>()) != cudaSuccess) return e;
  if ((e = configure_one<4, 1, 64>()) != cudaSuccess) return e;
  if ((e = configure_one<4, 2, 64>()) != cudaSuccess) return e;
  if ((e = configure_one<8, 1, 32>()) != cudaSuccess) return e;
  return configure_one<8, 1, 64>();
}

cudaError_t launch_attention(const uint16_t* qkv, uint16_t* out, int n_kept, int batch, int seq,
                             const int32_t* seq_lens, int sm_count, int next_ctas, cudaStream_t s, bool pdl,
                             unsigned long long* stamps) {
  if (n_kept <= 0) return cudaSuccess;
  const AttnArgs a{qkv, out, seq_lens, n_kept, batch, seq, stamps};
  const auto ctas = [&](int rows) { return static_cast<long>((seq + rows - 1) / rows) * n_kept * batch; };
  // Few CTAs: the smallest query tiles that still find an SM each, and the keys of more than two blocks split over warps
  // (one sequence of 256 keys, 16 heads: 32 queries x 4 splits 4.2 us, 64 x 2 5.3, 128 x 1 6.8) - on the SMs that the O
  // projection after it does not want: its CTAs start meanwhile and decode their weights (the same sequence with 128 CTAs
  // 263 us for six layers, with 64 246).  Where even tiles of 128 queries leave it too few SMs, all of them.
  // Then tiles of 128 queries: fewer reads of K and V.
  // Blocks of 32 keys where they save half a block of padding (43 x 91: 12.1 against 14.8 us), and up to 32 keys.
  const long limit = ctas(128) <= sm_count - next_ctas ? sm_count - next_ctas : sm_count;
  const bool pad32 = (seq - 1) % 64 < 32;
  if (seq <= 32) return launch_one<2, 1, 32>(a, sm_count, s, pdl);
  if (seq > 64) {
    if (ctas(32) <= limit) return seq > 128 ? launch_one<2, 4, 64>(a, sm_count, s, pdl) : launch_one<2, 2, 64>(a, sm_count, s, pdl);
    if (seq > 128 && ctas(64) <= limit) return launch_one<4, 2, 64>(a, sm_count, s, pdl);
    if (seq > 128 || ctas(64) > limit)
      return pad32 ? launch_one<8, 1, 32>(a, sm_count, s, pdl) : launch_one<8, 1, 64>(a, sm_count, s, pdl);
  }
  return pad32 ? launch_one<4, 1, 32>(a, sm_count, s, pdl) : launch_one<4, 1, 64>(a, sm_count, s, pdl);
}

}  // namespace sti
