// Per-head attention on the tcgen05 tensor cores for long sequences (Section 2.1: softmax(Q K^T / sqrt 64) V per kept head;
// padded keys get probability exactly 0).
//
// One CTA per two query tiles of 128 of a (sequence, kept head): two groups of four warps, ONE thread per query row, so a row's
// maximum and sum never leave the thread, and one warp per group that issues its loads and MMAs.  Two CTAs share an SM (113 KB,
// half the tensor memory each), which puts four softmax warps on every scheduler: while one waits for a tensor-core result,
// reads scores or reduces, the others keep the special-function units busy.
//
// Per 32-key step a group's warps take the row's scores into registers (tcgen05.ld), the maximum, the exponentials and their
// sum, and put the bf16 probabilities back into tensor memory over the scores; O += P V (P is the tensor-memory operand)
// follows.  There are two score buffers, so S = Q K^T of the next step is computed during this step's exponentials (and 32 keys
// are what two buffers leave room for: with one buffer of 64 keys a step took 2,500 cycles, 1,300 of them waiting for P V and S
// in turn).  Keys and values stream through a ring of five 64-key chunks read by both groups; the group that finishes a chunk
// last refills its place, so nobody waits for a producer.
//
// O stays in tensor memory for the whole tile.  The maximum used for the exponentials moves only when a step's maximum exceeds
// it by more than 2^8 (then O and the sum are rescaled); the sum and O are in fp32 and the division by the sum at the end takes
// any common factor out, so nothing is lost by a maximum that lags behind.
//
// Bound: the exponentials.  32 x 128 of them take 256 cycles of an SM's special-function units, 34 us for 32 x 512 tokens of 16
// heads; measured 60 us, the units 54 % busy, issue slots 47 % (K and V of a sequence resident, one CTA per SM, probabilities
// through shared memory, O in registers: 117 us; persistent CTAs with a producer and 128-key steps: 74 us).
//
// Tensor memory of group g: S and P of even / odd steps at column 128 g / 128 g + 32, O at 128 g + 64.  Waits are bounded; a
// role that gives up sets the abort flag and the status word, the others see the flag or run out of their own waits.
#include <cuda_bf16.h>

#include "gemm_device.cuh"
#include "sti_kernels.h"

namespace sti {
namespace {

constexpr int kTcGroups = 2, kTcGroupWarps = 4, kTcMmaWarp = kTcGroups * kTcGroupWarps, kTcThreads = 32 * (kTcMmaWarp + kTcGroups);
constexpr int kTcQTile = 128, kTcChunk = 64, kTcStep = 32, kTcHead = 64, kTcRing = 5;
constexpr int kTcMaxSeq = 512;
constexpr uint32_t kTcBox = kTcChunk * kTcHead * 2;              // 8 KB: 64 rows x 64 bf16, one TMA box
constexpr uint32_t kTcOffQ = 1024;                               // a query tile per group; its output tile in the end
constexpr uint32_t kTcOffKV = kTcOffQ + kTcGroups * 2 * kTcBox;  // ring: keys and values of a chunk
constexpr uint32_t kTcSmem = kTcOffKV + kTcRing * 2 * kTcBox;
static_assert(2 * (kTcSmem + 1024) <= 228 * 1024, "two CTAs per SM");
constexpr uint32_t kTcTmemCols = 256;

struct TcBarriers {
  uint64_t k_full[kTcRing], v_full[kTcRing];
  uint64_t q_full[kTcGroups];
  uint64_t s_full[kTcGroups][2];   // the group's scores of an even / odd step are complete in tensor memory
  uint64_t p_full[kTcGroups][2];   // its probabilities are
  uint64_t o_full[kTcGroups];      // its P V of a step has completed
  uint64_t o_last[kTcGroups];      // ... of the last step
  uint64_t tail_zeroed;            // the rows of V past the valid keys are zeros (if there are any: see zero_tail)
  uint64_t drain[kTcGroups];
  int readers_done[kTcMaxSeq / kTcChunk];      // groups that have finished with a chunk
  int requested;                   // chunks asked for so far
  int tail_taken;                  // a group has taken on the zeroing
  uint32_t tmem_base;
  volatile uint32_t abort;
};
static_assert(sizeof(TcBarriers) <= kTcOffQ, "header");

__device__ __forceinline__ uint64_t umma_smem_desc_sw128_mn(uint32_t saddr) {    // V: keys are rows, the 64 features contiguous
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// D[128 x N] += A[128 x 16] B[N x 16]^T with A (bf16 pairs, lane = row) in tensor memory
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(tmem_d), "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
               "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
               : "memory");
}
// One 32 x 64 tile of the output (128-byte swizzle in shared memory) as a bulk group of its own.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n\tcp.async.bulk.commit_group;"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// tcgen05.wait::ld that names the registers of one earlier 32-column load as read-write operands: the compiler then
// keeps those values where the load put them until here and orders every later use after the wait, so the load may
// stay in flight while the thread works on other registers.
__device__ __forceinline__ void tmem_wait_ld_x32(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}

__device__ __forceinline__ void tmem_wait_ld_x16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// Whole warp; the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, uint32_t lane, volatile uint32_t* abort) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  uint32_t ok = 1;
  if (lane == 0) ok = *abort ? 0u : (mbar_wait_bounded(bar, parity) ? 1u : 0u);
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

__global__ void __launch_bounds__(kTcThreads, 2)
attention_tc_kernel(const __grid_constant__ CUtensorMap qkv_map, const __grid_constant__ CUtensorMap out_map,
                    uint16_t* __restrict__ out, const int32_t* __restrict__ seq_lens, int n_kept, int batch, int L,
                    int* __restrict__ err, unsigned long long* stamps) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) { stamp_min(stamps, STAMP_FIRST_START); stamp_max(stamps, STAMP_LAST_START); }
  TcBarriers* bar = reinterpret_cast<TcBarriers*>(smem);
  const uint32_t sbase = smem_addr(smem);
  if ((sbase & 1023u) != 0 || L < 1 || L > kTcMaxSeq) {
    if (tid == 0) atomicCAS(err, ERR_NONE, ERR_BAD_JOB);
    return;
  }
  if (tid == kTcMmaWarp * 32) {
    for (int c = 0; c < kTcRing; ++c) { mbar_init(smem_addr(&bar->k_full[c]), 1); mbar_init(smem_addr(&bar->v_full[c]), 1); }
    for (int g = 0; g < kTcGroups; ++g) {
      mbar_init(smem_addr(&bar->q_full[g]), 1);
      for (int e = 0; e < 2; ++e) {
        mbar_init(smem_addr(&bar->s_full[g][e]), 1);
        mbar_init(smem_addr(&bar->p_full[g][e]), kTcGroupWarps);
      }
      mbar_init(smem_addr(&bar->o_full[g]), 1);
      mbar_init(smem_addr(&bar->o_last[g]), 1);
      mbar_init(smem_addr(&bar->drain[g]), 1);
    }
    mbar_init(smem_addr(&bar->tail_zeroed), 1);
    for (int c = 0; c < kTcMaxSeq / kTcChunk; ++c) bar->readers_done[c] = 0;
    bar->tail_taken = 0;
    bar->requested = 0;
    bar->abort = 0;
    mbar_fence_init();
    fence_proxy_async_smem();
    tma_prefetch_map(&qkv_map);
    tma_prefetch_map(&out_map);
  }
  if (warp == kTcMmaWarp) {
    tmem_alloc(smem_addr(&bar->tmem_base), kTcTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = bar->tmem_base;
  pdl_launch_dependents();
  pdl_wait();
  if (tid == 0) stamp_min(stamps, STAMP_RELEASE);

  const int hi = blockIdx.y, b = blockIdx.z, T = batch * L;
  int valid = L;
  if (seq_lens != nullptr) valid = min(max(__ldg(seq_lens + b), 0), L);
  const int nc = (valid + kTcChunk - 1) / kTcChunk;              // chunks and steps with at least one valid key
  const int ns = (valid + kTcStep - 1) / kTcStep;
  const uint32_t g = warp < kTcMmaWarp ? warp >> 2 : warp - kTcMmaWarp, quad = warp & 3;
  const int tile0 = static_cast<int>(blockIdx.x) * kTcGroups;    // the CTA's first query tile
  const int n_groups = min(kTcGroups, (L + kTcQTile - 1) / kTcQTile - tile0);
  const uint32_t q_sm = sbase + kTcOffQ + g * 2 * kTcBox, kv_sm = sbase + kTcOffKV;
  bool failed = false, issued = false;
  auto wait = [&](uint64_t* m, uint32_t parity) { return warp_wait(smem_addr(m), parity & 1, lane, &bar->abort); };
  // one thread: chunk c of the keys and values into its place of the ring
  auto load_keys = [&](int c, bool values) {
    const uint32_t full = smem_addr(values ? &bar->v_full[c % kTcRing] : &bar->k_full[c % kTcRing]);
    mbar_expect_tx(full, kTcBox);
    tma_load_2d(kv_sm + (2 * (c % kTcRing) + (values ? 1 : 0)) * kTcBox, &qkv_map, 0, (hi * 3 + (values ? 2 : 1)) * T + b * L + c * kTcChunk,
                full);
  };
  const uint32_t col = tmem + g * 128;

  if (static_cast<int>(g) >= n_groups) {
    // the second group of a sequence's last, single tile
  } else if (nc == 0) {
    // no valid key: the head contributes nothing, and the rows that exist are written all the same
    if (warp < kTcMmaWarp) {
      const int q0 = (tile0 + static_cast<int>(g)) * kTcQTile + static_cast<int>(quad * 32), ldo = n_kept * kTcHead;
      uint16_t* dst = out + (static_cast<size_t>(b) * L + q0) * ldo + hi * kTcHead + (lane & 7) * 8;
      for (int r = static_cast<int>(lane >> 3); r < min(32, L - q0); r += 4)
        *reinterpret_cast<uint4*>(dst + static_cast<size_t>(r) * ldo) = make_uint4(0u, 0u, 0u, 0u);
    }
  } else if (warp >= kTcMmaWarp) {
    // ---- the group's loads and MMAs
    if (lane == 0) {
      if (g == 0) load_keys(0, false);
      const uint32_t full = smem_addr(&bar->q_full[g]);
      mbar_expect_tx(full, 2 * kTcBox);
      for (int h = 0; h < 2; ++h)
        tma_load_2d(q_sm + h * kTcBox, &qkv_map, 0, hi * 3 * T + b * L + (tile0 + static_cast<int>(g)) * kTcQTile + h * kTcChunk, full);
      if (g == 0) {
        load_keys(0, true);
        for (int c = 1; c < nc && c < kTcRing; ++c) { load_keys(c, false); load_keys(c, true); }
        atomicMax(&bar->requested, min(nc, kTcRing));
      }
    }
    __syncwarp();
    const uint32_t idesc_s = umma_idesc_bf16_m128(kTcStep);
    const uint32_t idesc_o = umma_idesc_bf16_m128(kTcHead) | (1u << 16);         // B (V) is MN-major
    const uint64_t q_desc = umma_smem_desc_sw128(q_sm), k_desc0 = umma_smem_desc_sw128(kv_sm);
    const uint64_t v_desc0 = umma_smem_desc_sw128_mn(kv_sm + kTcBox);
    auto issue_scores = [&](int c) -> bool {
      const int st = (c >> 1) % kTcRing;
      if ((c & 1) == 0 && !wait(&bar->k_full[st], (c >> 1) / kTcRing)) return false;
      tc_fence_after_sync();
      if (elect_one()) {
        umma_bf16_ss_x4(col + (c & 1) * kTcStep, q_desc, k_desc0 + st * (2 * kTcBox >> 4) + (c & 1) * (kTcBox / 2 >> 4), 2, 2, idesc_s, 0u);
        umma_commit(smem_addr(&bar->s_full[g][c & 1]));
      }
      __syncwarp();
      issued = true;
      return true;
    };
    // The last 16 keys of P V may hold fewer valid ones.  The others' probabilities are 0, but their rows of V are padding or
    // the next sequence's, and 0 x Inf and 0 x NaN are NaN: zeros take their place, at most 15 rows of the last chunk, which
    // nobody has multiplied by yet.  Whichever group comes first does it for both (the swizzle moves pieces inside a row only).
    auto zero_tail = [&](int st) -> bool {
      int taken = 0;
      if (lane == 0) taken = atomicExch(&bar->tail_taken, 1);
      if (__shfl_sync(0xffffffffu, taken, 0) != 0) return wait(&bar->tail_zeroed, 0);
      uint4* rows = reinterpret_cast<uint4*>(smem + kTcOffKV + (2 * st + 1) * kTcBox + (valid % kTcChunk) * (kTcHead * 2));
      const int n_pieces = (16 - valid % 16) * (kTcHead * 2 / 16);
      for (int i = static_cast<int>(lane); i < n_pieces; i += 32) rows[i] = make_uint4(0u, 0u, 0u, 0u);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&bar->tail_zeroed));
      return true;
    };
    failed = !wait(&bar->q_full[g], 0) || !issue_scores(0) || (ns > 1 && !issue_scores(1));
    for (int c = 0; c < ns && !failed; ++c) {
      // O += P V; the step's second 16 keys are left out if none of them is valid
      const int chunk = c >> 1, st = chunk % kTcRing;
      if ((c & 1) == 0 && !wait(&bar->v_full[st], chunk / kTcRing)) { failed = true; break; }
      if (c + 1 == ns && valid % 16 != 0 && !zero_tail(st)) { failed = true; break; }
      if (!wait(&bar->p_full[g][c & 1], c >> 1)) { failed = true; break; }
      tc_fence_after_sync();
      if (elect_one()) {
        const uint64_t vd = v_desc0 + st * (2 * kTcBox >> 4) + (c & 1) * (kTcBox / 2 >> 4);
        const uint32_t p_col = col + (c & 1) * kTcStep;
        umma_bf16_ts(col + 64, p_col, vd, idesc_o, c > 0 ? 1u : 0u);
        if (valid - c * kTcStep > 16) umma_bf16_ts(col + 64, p_col + 8, vd + (2048 >> 4), idesc_o, 1u);
        umma_commit(smem_addr(&bar->o_full[g]));
        if (c + 1 == ns) umma_commit(smem_addr(&bar->o_last[g]));
      }
      __syncwarp();
      issued = true;
      if (c + 2 < ns) {                                          // scores of the step after next go where this step's P is
        if (!wait(&bar->o_full[g], c) || !issue_scores(c + 2)) { failed = true; break; }
        if (lane == 0 && (c & 1) != 0 && chunk + kTcRing < nc) { // this group has finished with the chunk
          __threadfence_block();
          if (atomicAdd(&bar->readers_done[chunk], 1) == n_groups - 1) {
            __threadfence_block();
            load_keys(chunk + kTcRing, false);
            load_keys(chunk + kTcRing, true);
            atomicMax(&bar->requested, chunk + kTcRing + 1);
          }
        }
        __syncwarp();
      }
    }
    if (!failed) failed = !wait(&bar->o_last[g], 0);
  } else {
    // ---- softmax: thread = query row
    const uint32_t t_lane = (quad * 32) << 16;
    const uint32_t s_addr = col + t_lane, o_addr = s_addr + 64;
    const float scale = 0.125f * 1.4426950408889634f;            // 1/sqrt(64) * log2(e)
    const int q0 = (tile0 + static_cast<int>(g)) * kTcQTile + static_cast<int>(quad * 32);
    const bool idle = q0 >= L;                                   // rows past the sequence: only the barriers
    float m = -INFINITY, l = 0.f;
    for (int c = 0; c < ns && !failed; ++c) {
      if (!wait(&bar->s_full[g][c & 1], c >> 1)) { failed = true; break; }
      tc_fence_after_sync();
      const uint32_t buf = s_addr + (c & 1) * kTcStep;
      uint32_t s[32];
      if (!idle) {
        const int n_valid = valid - c * kTcStep;                 // keys of this step at and past it are padding
        tmem_ld_32x32b_x32(buf, s);
        tmem_wait_ld_x32(s);
        if (n_valid < kTcStep) {
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (k >= n_valid) s[k] = 0xff800000u;                // -inf
        }
        float mx[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          mx[e] = max3(__uint_as_float(s[e]), __uint_as_float(s[e + 2]), __uint_as_float(s[e + 4]));
#pragma unroll
          for (int k = 6; k < 30; k += 4) mx[e] = max3(mx[e], __uint_as_float(s[e + k]), __uint_as_float(s[e + k + 2]));
        }
        const float mc = max3(fmaxf(mx[0], mx[1]), __uint_as_float(s[30]), __uint_as_float(s[31])) * scale;   // finite: a valid key
        if (c == 0) {
          m = mc;
        } else if (__any_sync(0xffffffffu, mc > m + 8.f)) {
          if (!wait(&bar->o_full[g], c - 1)) { failed = true; break; }     // P V of step c - 2 came before these scores
          tc_fence_after_sync();
          const float m_new = fmaxf(m, mc), alpha = fast_exp2(m - m_new);
          m = m_new;
          l *= alpha;
#pragma unroll 1
          for (int e = 0; e < 4; ++e) {
            uint32_t r[16];
            tmem_ld_32x32b_x16(o_addr + e * 16, r);
            tmem_wait_ld_x16(r);
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * alpha);
            tmem_st_32x32b_x16(o_addr + e * 16, r);
          }
        }
      }
      if (!idle) {
        const uint64_t scale2 = pack_f32x2(scale, scale), minus_m2 = pack_f32x2(-m, -m);
        uint64_t sum2[2] = {0u, 0u};
        uint32_t pk[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          float p0, p1;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * k]), __uint_as_float(s[2 * k + 1])), scale2, minus_m2), p0, p1);
          p0 = fast_exp2(p0);
          p1 = fast_exp2(p1);
          sum2[k & 1] = add_f32x2(sum2[k & 1], pack_f32x2(p0, p1));
          pk[k] = pack_bf16x2(p0, p1);
        }
        tmem_st_32x32b_x16(buf, pk);
        float l0, l1;
        unpack_f32x2(add_f32x2(sum2[0], sum2[1]), l0, l1);
        l += l0 + l1;
        tc_wait_st();
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&bar->p_full[g][c & 1]));
    }
    if (!failed) failed = !wait(&bar->o_last[g], 0);
    if (!failed && !idle) {
      tc_fence_after_sync();
      const float inv = 1.0f / l;                                // at least one valid key: l > 0
      // through the query tile's shared memory (its last reader was S) and a bulk store
      uint8_t* stage = smem + kTcOffQ + g * 2 * kTcBox + quad * 4096;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        uint32_t o[32];
        tmem_ld_32x32b_x32(o_addr + e * 32, o);
        tmem_wait_ld_x32(o);
        auto two = [&](int k) { return pack_bf16x2(__uint_as_float(o[k]) * inv, __uint_as_float(o[k + 1]) * inv); };
#pragma unroll
        for (int k = 0; k < 32; k += 8)
          *reinterpret_cast<uint4*>(stage + lane * 128 + (((e * 4 + k / 8) ^ (lane & 7)) << 4)) =
              make_uint4(two(k), two(k + 2), two(k + 4), two(k + 6));
      }
      if (q0 + 32 <= L) {
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&out_map, smem_addr(stage), hi * kTcHead, b * L + q0);
          bulk_wait_read();
        }
      } else {                                                   // the sequence ends inside: the rows that exist, four at a time
        __syncwarp();
        const int ldo = n_kept * kTcHead;
        uint16_t* dst = out + (static_cast<size_t>(b) * L + q0) * ldo + hi * kTcHead + (lane & 7) * 8;
        for (int r = static_cast<int>(lane >> 3); r < L - q0; r += 4)
          *reinterpret_cast<uint4*>(dst + static_cast<size_t>(r) * ldo) =
              *reinterpret_cast<const uint4*>(stage + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
      }
      __syncwarp();
    }
  }
  if (failed) {
    bar->abort = 1;
    if (lane == 0) atomicCAS(err, ERR_NONE, ERR_WAIT_TIMEOUT);
    if (issued) {                                // outstanding MMAs: one more bounded chance before tensor memory is freed
      if (elect_one()) umma_commit(smem_addr(&bar->drain[g]));
      __syncwarp();
      (void)mbar_wait_bounded(smem_addr(&bar->drain[g]), 0);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kTcMmaWarp) {
    if (bar->abort && lane == 0 && nc > 0) {     // copies that nobody waited for: a bounded chance to land before the CTA exits
      for (int r = max(0, bar->requested - kTcRing); r < bar->requested; ++r) {
        (void)mbar_wait_bounded(smem_addr(&bar->k_full[r % kTcRing]), (r / kTcRing) & 1);
        (void)mbar_wait_bounded(smem_addr(&bar->v_full[r % kTcRing]), (r / kTcRing) & 1);
      }
      for (int t = 0; t < n_groups; ++t) (void)mbar_wait_bounded(smem_addr(&bar->q_full[t]), 0);
    }
    __syncwarp();
    tmem_dealloc(tmem, kTcTmemCols);
  }
  if (tid == 0) stamp_max(stamps, STAMP_LAST_END);
}

}  // namespace

cudaError_t attention_tc_configure() {
  return cudaFuncSetAttribute(attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kTcSmem));
}

// `qkv_map`: TMA view of qkv as [3 * n_kept * T rows, 64 columns] bf16, boxes of 64 rows, 128-byte swizzle;
// `out_map`: of out as [T rows, 64 n_kept columns], boxes of 32 rows, the same swizzle.
cudaError_t launch_attention_tc(const CUtensorMap& qkv_map, const CUtensorMap& out_map, uint16_t* out, int n_kept, int batch, int seq,
                                 const int32_t* seq_lens, int* err, cudaStream_t s, bool pdl, unsigned long long* stamps) {
  if (n_kept <= 0 || batch <= 0) return cudaSuccess;
  if (seq < 1 || seq > kTcMaxSeq || batch > 65535) return cudaErrorInvalidValue;
  const int tile_pairs = (seq + kTcGroups * kTcQTile - 1) / (kTcGroups * kTcQTile);
  return launch_kernel(attention_tc_kernel, dim3(tile_pairs, n_kept, batch), dim3(kTcThreads), kTcSmem, s, pdl, qkv_map, out_map, out,
                       seq_lens, n_kept, batch, seq, err, stamps);
}

}  // namespace sti
