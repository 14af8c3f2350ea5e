// Residual + bias + LayerNorm over the split-K partial sums of the O projection and of FFN2
// (Section 2.1; Section 6: biases and layernorm parameters stay in fp32).
// Below 2048 rows of at most 1024: 128 threads to a row.  From there: a
// warp per row.  Wider rows: one CTA per row, one float4 per thread.
#include <cuda_bf16.h>

#include "sti_device.cuh"
#include "sti_kernels.h"

namespace sti {
namespace {

__device__ __forceinline__ float block_sum(float v, float* red, int tid, int n_warps) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  float t = 0.f;
#pragma unroll 1
  for (int w = 0; w < n_warps; ++w) t += red[w];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(512)
layernorm_kernel(LnLaunch p) {
  __shared__ float red[16];
  const int tid = threadIdx.x;
  const int n_warps = blockDim.x >> 5;
  const size_t row = static_cast<size_t>(blockIdx.x) * p.d;
  const int c = tid * 4;
  pdl_launch_dependents();
  if (tid == 0) { stamp_min(p.stamps, STAMP_FIRST_START); stamp_max(p.stamps, STAMP_LAST_START); }
  float4 a = __ldg(reinterpret_cast<const float4*>(p.bias + c));      // parameters: not written by any kernel
  const float4 g = __ldg(reinterpret_cast<const float4*>(p.gamma + c));
  const float4 b = __ldg(reinterpret_cast<const float4*>(p.beta + c));
  pdl_wait();                                                          // residual and partial sums are
  if (tid == 0) stamp_min(p.stamps, STAMP_RELEASE);                    // the preceding kernels' output
  if (p.resid_bf16) {
    const uint2 r = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p.resid) + row + c));
    a.x += __uint_as_float(r.x << 16); a.y += __uint_as_float(r.x & 0xffff0000u);
    a.z += __uint_as_float(r.y << 16); a.w += __uint_as_float(r.y & 0xffff0000u);
  } else {
    const float4 r = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(p.resid) + row + c));
    a.x += r.x; a.y += r.y; a.z += r.z; a.w += r.w;
  }
  const size_t pstride = static_cast<size_t>(p.T) * p.d;
  int q = 0;
#pragma unroll 1
  for (; q + 4 <= p.n_partial; q += 4) {          // four independent loads at a time
    const float4 s0 = __ldg(reinterpret_cast<const float4*>(p.partial + (q + 0) * pstride + row + c));
    const float4 s1 = __ldg(reinterpret_cast<const float4*>(p.partial + (q + 1) * pstride + row + c));
    const float4 s2 = __ldg(reinterpret_cast<const float4*>(p.partial + (q + 2) * pstride + row + c));
    const float4 s3 = __ldg(reinterpret_cast<const float4*>(p.partial + (q + 3) * pstride + row + c));
    a.x += (s0.x + s1.x) + (s2.x + s3.x); a.y += (s0.y + s1.y) + (s2.y + s3.y);
    a.z += (s0.z + s1.z) + (s2.z + s3.z); a.w += (s0.w + s1.w) + (s2.w + s3.w);
  }
#pragma unroll 1
  for (; q < p.n_partial; ++q) {
    const float4 s = __ldg(reinterpret_cast<const float4*>(p.partial + q * pstride + row + c));
    a.x += s.x; a.y += s.y; a.z += s.z; a.w += s.w;
  }
  const float mean = block_sum(a.x + a.y + a.z + a.w, red, tid, n_warps) / static_cast<float>(p.d);
  const float dx = a.x - mean, dy = a.y - mean, dz = a.z - mean, dw = a.w - mean;
  const float var = block_sum(dx * dx + dy * dy + dz * dz + dw * dw, red, tid, n_warps) / static_cast<float>(p.d);
  const float rstd = rsqrtf(var + p.eps);
  float4 y;
  y.x = dx * rstd * g.x + b.x; y.y = dy * rstd * g.y + b.y;
  y.z = dz * rstd * g.z + b.z; y.w = dw * rstd * g.w + b.w;
  if (p.out_f32) *reinterpret_cast<float4*>(p.out_f32 + row + c) = y;
  if (p.out_bf16)
    *reinterpret_cast<uint2*>(p.out_bf16 + row + c) = make_uint2(pack_bf16x2(y.x, y.y), pack_bf16x2(y.z, y.w));
  if (p.stamps != nullptr) {
    __syncthreads();
    if (tid == 0) stamp_max(p.stamps, STAMP_LAST_END);
  }
}

// Up to 2048 rows of at most 1024: a CTA of 128 threads per row, two float4 each.
// Bound: latency.  Residual and the first P partial-sum planes (four, or eight where there are more) are in flight together, gamma and beta while the row is
// reduced: two memory round trips and two exchanges between four warps per row (one float4 per thread and one plane at a
// time took five trips; BERT-large, 256 tokens 5.1 -> 3.7 and 6.5 -> 5.9 us, 1024 tokens 5.6 -> 3.4 and 7.1 -> 6.1,
// BERT-base, 128 tokens 2.8 -> 2.1 and 3.8 -> 3.1; eight planes at once 4.7 -> 4.1 at BERT-large, 256 tokens, 5.6 -> 4.1 at 384).
// Small CTAs also leave an SM sooner: the next GEMM's CTAs, which need a
// whole one and decode their weights meanwhile, start earlier than with rows packed into large CTAs on fewer SMs.
constexpr uint32_t kLnGroup = 128;
constexpr int kLnGroupMaxHidden = 1024;
template <int P>
__global__ void __launch_bounds__(kLnGroup)
layernorm_group_kernel(LnLaunch p) {
  __shared__ float red[8];
  const uint32_t gt = threadIdx.x, row = blockIdx.x;
  pdl_launch_dependents();
  if (gt == 0) { stamp_min(p.stamps, STAMP_FIRST_START); stamp_max(p.stamps, STAMP_LAST_START); }
  const uint32_t lane = gt & 31, w = gt >> 5, n4 = static_cast<uint32_t>(p.d) / 4;
  const size_t base = static_cast<size_t>(row) * p.d, pstride = static_cast<size_t>(p.T) * p.d;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool on[2] = {gt < n4, gt + kLnGroup < n4};
  auto plane = [&](int q, int v) {
    return on[v] && q < p.n_partial ? *reinterpret_cast<const float4*>(p.partial + q * pstride + base + 4 * (gt + kLnGroup * v)) : zero;
  };
  auto add4 = [](float4& a, const float4 (&s)[4]) {
    a.x += (s[0].x + s[1].x) + (s[2].x + s[3].x); a.y += (s[0].y + s[1].y) + (s[2].y + s[3].y);
    a.z += (s[0].z + s[1].z) + (s[2].z + s[3].z); a.w += (s[0].w + s[1].w) + (s[2].w + s[3].w);
  };
  float4 bias[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) bias[v] = on[v] ? __ldg(reinterpret_cast<const float4*>(p.bias) + gt + kLnGroup * v) : zero;
  pdl_wait();
  if (gt == 0) stamp_min(p.stamps, STAMP_RELEASE);
  float4 a[2];
  {
    float4 r[2] = {zero, zero}, s[2][P / 4][4];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const uint32_t c = gt + kLnGroup * v;
      if (on[v]) {
        if (p.resid_bf16) {
          const uint2 t = *reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p.resid) + base + 4 * c);
          r[v] = make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u), __uint_as_float(t.y << 16), __uint_as_float(t.y & 0xffff0000u));
        } else {
          r[v] = *reinterpret_cast<const float4*>(static_cast<const float*>(p.resid) + base + 4 * c);
        }
      }
#pragma unroll
      for (int q = 0; q < P; ++q) s[v][q / 4][q % 4] = plane(q, v);
    }
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      a[v] = make_float4(bias[v].x + r[v].x, bias[v].y + r[v].y, bias[v].z + r[v].z, bias[v].w + r[v].w);
#pragma unroll
      for (int q = 0; q < P / 4; ++q) add4(a[v], s[v][q]);
    }
  }
#pragma unroll 1
  for (int q0 = P; q0 < p.n_partial; q0 += 4) {
    float4 s[2][4];
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int q = 0; q < 4; ++q) s[v][q] = plane(q0 + q, v);
#pragma unroll
    for (int v = 0; v < 2; ++v) add4(a[v], s[v]);
  }
  float4 gamma[2], beta[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    gamma[v] = on[v] ? __ldg(reinterpret_cast<const float4*>(p.gamma) + gt + kLnGroup * v) : zero;
    beta[v] = on[v] ? __ldg(reinterpret_cast<const float4*>(p.beta) + gt + kLnGroup * v) : zero;
  }
  auto row_sum = [&](float v, float* slot) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) slot[w] = v;
    __syncthreads();
    return (slot[0] + slot[1]) + (slot[2] + slot[3]);
  };
  const float inv_d = 1.f / static_cast<float>(p.d);
  const float mean = __fmul_rn(row_sum(((a[0].x + a[0].y) + (a[0].z + a[0].w)) + ((a[1].x + a[1].y) + (a[1].z + a[1].w)), red), inv_d);
  float sq = 0.f;
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    a[v].x -= mean; a[v].y -= mean; a[v].z -= mean; a[v].w -= mean;
    if (on[v]) sq = fmaf(a[v].x, a[v].x, fmaf(a[v].y, a[v].y, fmaf(a[v].z, a[v].z, fmaf(a[v].w, a[v].w, sq))));
  }
  const float rstd = rsqrtf(fmaf(row_sum(sq, red + 4), inv_d, p.eps));
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    if (!on[v]) continue;
    const uint32_t c = gt + kLnGroup * v;
    float4 y;
    y.x = fmaf(__fmul_rn(a[v].x, rstd), gamma[v].x, beta[v].x); y.y = fmaf(__fmul_rn(a[v].y, rstd), gamma[v].y, beta[v].y);
    y.z = fmaf(__fmul_rn(a[v].z, rstd), gamma[v].z, beta[v].z); y.w = fmaf(__fmul_rn(a[v].w, rstd), gamma[v].w, beta[v].w);
    if (p.out_f32) *reinterpret_cast<float4*>(p.out_f32 + base + 4 * c) = y;
    if (p.out_bf16) *reinterpret_cast<uint2*>(p.out_bf16 + base + 4 * c) = make_uint2(pack_bf16x2(y.x, y.y), pack_bf16x2(y.z, y.w));
  }
  if (p.stamps != nullptr) {
    __syncthreads();
    if (gt == 0) stamp_max(p.stamps, STAMP_LAST_END);
  }
}

// A whole line of scratch that nobody will read: its L2 copy is dropped, not written to memory.
__device__ __forceinline__ void discard_line(const float* p) { asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory"); }

// Many tokens: a warp per row, lane l holding float4 number l, l + 32, ... of it (V = d / 128 of them).  Every load of
// a row - residual and one partial-sum plane at a time - is issued before the first use, and the two
// reductions are warp shuffles: no barrier, and enough bytes in flight per SM to keep the memory system busy.
// The more registers, the more of a row is in flight, but the fewer warps are resident, and a second wave costs more than either:
// three builds, each for the rows that it does in one wave.  Two CTAs of eight rows per SM (up to 127 registers) take 2368 rows:
// with four planes 8.1 -> 6.4 us at 2048 rows of 1024.  Three such CTAs, 3552 rows: 10.1 us at 3072 rows, 10.6 with two per SM.
// From 4096 rows on (one plane) seven CTAs of four rows (72 registers): 8.4 -> 6.4 us at 4096 rows, 31.7 -> 25.8 at 16,384
// with the planes discarded; with four planes that build loses (11.7 us at 3072 rows).
// Tried instead: the residual and the first plane asked for together (86 registers, two CTAs per SM instead of three: 31.6 ->
// 34.4 us at 16,384 rows of 1024), persistent warps that ask for their next row ahead (level there, 27.9 -> 31.5 with fp32
// residuals at 10,240 rows).
constexpr int kLnWarpMinRows = 2048, kLnFewPlanesMinRows = 4096;
template <int V, int ROWS, int CTAS>
__global__ void __launch_bounds__(ROWS * 32, CTAS == 3 ? 0 : CTAS)      // 3 come without asking, and without spills
layernorm_warp_kernel(LnLaunch p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x * ROWS + warp;
  pdl_launch_dependents();
  if (threadIdx.x == 0) { stamp_min(p.stamps, STAMP_FIRST_START); stamp_max(p.stamps, STAMP_LAST_START); }
  float4 a[V];
#pragma unroll
  for (int v = 0; v < V; ++v) a[v] = __ldg(reinterpret_cast<const float4*>(p.bias + (lane + v * 32) * 4));
  pdl_wait();
  if (threadIdx.x == 0) stamp_min(p.stamps, STAMP_RELEASE);
  if (r < p.T) {
    const size_t row = static_cast<size_t>(r) * p.d;
    if (p.resid_bf16) {
      uint2 rr[V];
#pragma unroll
      for (int v = 0; v < V; ++v)
        rr[v] = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p.resid) + row + (lane + v * 32) * 4));
#pragma unroll
      for (int v = 0; v < V; ++v) {
        a[v].x += __uint_as_float(rr[v].x << 16); a[v].y += __uint_as_float(rr[v].x & 0xffff0000u);
        a[v].z += __uint_as_float(rr[v].y << 16); a[v].w += __uint_as_float(rr[v].y & 0xffff0000u);
      }
    } else {
      float4 rr[V];
#pragma unroll
      for (int v = 0; v < V; ++v)
        rr[v] = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(p.resid) + row + (lane + v * 32) * 4));
#pragma unroll
      for (int v = 0; v < V; ++v) { a[v].x += rr[v].x; a[v].y += rr[v].y; a[v].z += rr[v].z; a[v].w += rr[v].w; }
    }
    const size_t pstride = static_cast<size_t>(p.T) * p.d;
#pragma unroll 1
    for (int q = 0; q < p.n_partial; ++q) {
      float4 s[V];
#pragma unroll
      for (int v = 0; v < V; ++v)
        s[v] = __ldg(reinterpret_cast<const float4*>(p.partial + q * pstride + row + (lane + v * 32) * 4));
#pragma unroll
      for (int v = 0; v < V; ++v) { a[v].x += s[v].x; a[v].y += s[v].y; a[v].z += s[v].z; a[v].w += s[v].w; }
    }
    float part = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) part += (a[v].x + a[v].y) + (a[v].z + a[v].w);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float mean = part / static_cast<float>(p.d);
    if constexpr (ROWS == 4) {
      if (p.discard) {                 // every lane's loads have returned
        for (int q = 0; q < p.n_partial; ++q)
          for (int line = lane; line < V * 4; line += 32) discard_line(p.partial + q * pstride + row + line * 32);
      }
    }
    part = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      a[v].x -= mean; a[v].y -= mean; a[v].z -= mean; a[v].w -= mean;
      part += (a[v].x * a[v].x + a[v].y * a[v].y) + (a[v].z * a[v].z + a[v].w * a[v].w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float rstd = rsqrtf(part / static_cast<float>(p.d) + p.eps);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int c = (lane + v * 32) * 4;
      const float4 g = __ldg(reinterpret_cast<const float4*>(p.gamma + c));
      const float4 b = __ldg(reinterpret_cast<const float4*>(p.beta + c));
      float4 y;
      y.x = a[v].x * rstd * g.x + b.x; y.y = a[v].y * rstd * g.y + b.y;
      y.z = a[v].z * rstd * g.z + b.z; y.w = a[v].w * rstd * g.w + b.w;
      if (p.out_f32) *reinterpret_cast<float4*>(p.out_f32 + row + c) = y;
      if (p.out_bf16)
        *reinterpret_cast<uint2*>(p.out_bf16 + row + c) = make_uint2(pack_bf16x2(y.x, y.y), pack_bf16x2(y.z, y.w));
    }
  }
  if (p.stamps != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) stamp_max(p.stamps, STAMP_LAST_END);
  }
}

template <int V>
cudaError_t launch_warp_rows(const LnLaunch& p, cudaStream_t s, bool pdl) {
  const dim3 grid4((p.T + 3) / 4), grid8((p.T + 7) / 8);
  if (p.T >= kLnFewPlanesMinRows) return launch_kernel(layernorm_warp_kernel<V, 4, 7>, grid4, dim3(128), 0, s, pdl, p);
  if (p.T > 2 * 8 * p.sm_count) return launch_kernel(layernorm_warp_kernel<V, 8, 3>, grid8, dim3(256), 0, s, pdl, p);
  return launch_kernel(layernorm_warp_kernel<V, 8, 2>, grid8, dim3(256), 0, s, pdl, p);
}

__global__ void cast_bf16_kernel(const float* __restrict__ in, uint16_t* __restrict__ out, size_t n4,
                                 unsigned long long* stamps) {
  const size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  pdl_launch_dependents();
  if (threadIdx.x == 0) { stamp_min(stamps, STAMP_FIRST_START); stamp_max(stamps, STAMP_LAST_START); }
  pdl_wait();
  if (threadIdx.x == 0) stamp_min(stamps, STAMP_RELEASE);
  if (i < n4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(in) + i);
    reinterpret_cast<uint2*>(out)[i] = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
  }
  if (stamps != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) stamp_max(stamps, STAMP_LAST_END);
  }
}

}  // namespace

cudaError_t launch_layernorm(const LnLaunch& p, cudaStream_t s, bool pdl) {
  if (p.T <= 0) return cudaSuccess;
  if (p.d % 128 != 0 || p.d > 2048) return cudaErrorInvalidValue;     // d / 4 threads, whole warps
  if (p.T >= kLnWarpMinRows && p.d <= 1024) {      // thousands of rows: a warp per row
    switch (p.d / 128) {
      case 1: return launch_warp_rows<1>(p, s, pdl);
      case 2: return launch_warp_rows<2>(p, s, pdl);
      case 3: return launch_warp_rows<3>(p, s, pdl);
      case 4: return launch_warp_rows<4>(p, s, pdl);
      case 5: return launch_warp_rows<5>(p, s, pdl);
      case 6: return launch_warp_rows<6>(p, s, pdl);
      case 7: return launch_warp_rows<7>(p, s, pdl);
      case 8: return launch_warp_rows<8>(p, s, pdl);
      default: break;
    }
  }
  if (p.d <= kLnGroupMaxHidden)
    return p.n_partial > 4 ? launch_kernel(layernorm_group_kernel<8>, dim3(p.T), dim3(kLnGroup), 0, s, pdl, p)
                           : launch_kernel(layernorm_group_kernel<4>, dim3(p.T), dim3(kLnGroup), 0, s, pdl, p);
  return launch_kernel(layernorm_kernel, dim3(p.T), dim3(p.d / 4), 0, s, pdl, p);
}

cudaError_t launch_cast_bf16(const float* in, uint16_t* out, size_t n, cudaStream_t s, bool pdl, unsigned long long* stamps) {
  if (n == 0) return cudaSuccess;
  if (n % 4) return cudaErrorInvalidValue;
  const size_t n4 = n / 4;
  return launch_kernel(cast_bf16_kernel, dim3(static_cast<unsigned>((n4 + 255) / 256)), dim3(256), 0, s, pdl, in, out, n4, stamps);
}

}  // namespace sti
