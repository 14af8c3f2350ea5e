// Internal interface between the host runtime (api.cu) and the sm_100a kernels.
// Nothing here is part of the public ABI.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "decode_task.h"

namespace sti {

// One weight-stationary tile: n_rows output features x k_total input features.
struct Job {
  uint32_t task_begin, n_tasks;
  uint32_t n_rows;          // 32, 64 or 128 (multiple of 64 when the matrices have 64 in-features)
  uint32_t k_total;         // multiple of 64
  uint32_t x_koff;          // first column of the activation operand
  uint32_t out_mat;         // output element (t, c) goes to out[(out_mat*T + t)*ldo + out_col + c]
  uint32_t out_col;
  int32_t bias_off;         // index of the tile's first bias element, -1 = no bias
};

enum GemmKind : int {
  GEMM_BF16_TO_BF16 = 1,      // bf16 in, bf16 out (+bias)                     : QKV
  GEMM_BF16_TO_BF16_GELU = 2, // bf16 in, bf16 out, +bias, erf-GELU            : FFN1
  GEMM_BF16_TO_F32 = 3        // bf16 in, fp32 partial sums out, no bias       : O projection, FFN2
};

struct GemmLaunch {
  const Job* jobs;
  const DecodeTask* tasks;
  int n_jobs;
  int m_ctas;               // CTAs along the token dimension (each loops over its M tiles)
  CUtensorMap xmap;         // TMA descriptor of x: [T rows, ldx columns] bf16, box 64 x 128, 128-byte swizzle
  const void* x;            // [T, ldx] bf16
  int ldx;
  int T;
  void* out;
  int ldo;
  const float* bias;
  int* err;                 // device status word
  size_t smem_bytes;        // header + w_bytes + n_stages activation stages
  uint32_t n_stages;        // stages in the activation ring
  uint32_t bps;             // 16 KB boxes (64 columns) per stage: 1, 2 or 4
  uint32_t w_bytes;         // shared memory reserved for the weight tile (largest job)
  uint32_t hdr_bytes;       // barriers + bias + per-warp centroid tables
  uint32_t task_stride;     // the tasks of job j start at tasks[j * task_stride], unused ones have bits == 0
  const uint8_t* pf_ptr[4]; // what the next layer reads first (packed shards, tile descriptors, dense parameters):
  uint32_t pf_bytes[4];     // pulled into L2 by this launch's idle warps
  bool simt_debug;          // compute the products on the plain ALUs instead of the tensor cores
  bool pdl;                 // launch with programmatic dependent launch
  unsigned long long* stamps;   // this launch's profiling record (see sti_device.cuh), or null
};

size_t gemm_smem_bytes(uint32_t w_bytes, uint32_t n_stages, uint32_t bps, uint32_t hdr_bytes);
cudaError_t gemm_configure();   // opt in to large dynamic shared memory (once per device)
cudaError_t launch_gemm(GemmKind kind, const GemmLaunch& p, cudaStream_t s);

// A layer's weights decoded into the working buffer (expand.cu): task i's two 4 KB pieces, the first one at expanded_at(task).
struct ExpandLaunch {
  const DecodeTask* tasks;
  uint32_t n_tasks;
  uint8_t* dst;
  bool pdl;
};
cudaError_t launch_expand(const ExpandLaunch& p, cudaStream_t s);

// GEMM over the working buffer (gemm_wide.cu).
struct WideShape {
  uint32_t T, n;            // tokens, output features (a multiple of 64)
  uint32_t n_tiles, m_pairs, splits, k_chunks;      // tiles of NT features, of 256 tokens, planes, chunks of 64 columns
  uint32_t w_row0;          // first 128-byte row of the matrix in the working buffer
  uint32_t plane64;         // 1: features 64 i .. 64 i + 63 are plane i of the output; 0: planes are K splits
};
struct WideLaunch {
  WideShape shape;
  uint32_t nt;              // features per tile: 256 or 128
  uint32_t clusters;        // CTA pairs
  CUtensorMap xmap;         // x: [T rows, K columns] bf16, boxes of 128 rows x 64 columns, 128-byte swizzle
  CUtensorMap wmap;         // working buffer as rows of 64 elements, boxes of nt / 2 rows, not swizzled (it is already)
  CUtensorMap omap;         // output as [planes][T][columns], boxes of 32 rows x 128 bytes, 128-byte swizzle
  const float* bias;        // null: none
  const int32_t* bias_off;  // per 64 features: where their bias begins
  bool weights_ready;       // decoded by a kernel that has finished before this one can start: read without waiting
  ExpandLaunch beside;      // decoded beside it by otherwise idle warps (n_tasks 0: nothing), the same matrix of another layer: no kernel in flight reads its place
  int* err;
  bool pdl;
  unsigned long long* stamps;
};
cudaError_t gemm_wide_configure();
cudaError_t launch_gemm_wide(GemmKind kind, const WideLaunch& p, cudaStream_t s);

// Per-head attention over kept heads.  qkv: [(kept*3 + which)][T][64] bf16; out: [T][n_kept*64] bf16.
// sm_count (the device's multiprocessor count) and next_ctas (the CTAs of the O projection that follows) pick the CTA shape.
cudaError_t attention_configure();
cudaError_t launch_attention(const uint16_t* qkv, uint16_t* out, int n_kept, int batch, int seq,
                             const int32_t* seq_lens, int sm_count, int next_ctas, cudaStream_t s, bool pdl,
                             unsigned long long* stamps);

// The same attention on the tcgen05 tensor cores, one CTA per two tiles of 128 queries of a (sequence, kept head), for
// many tokens (attention_tc.cu).
// `qkv_map`: TMA view of qkv as [3 * n_kept * T rows, 64 columns] bf16, boxes of 64 rows x 64 columns, 128-byte swizzle;
// `out_map`: of out as [T rows, 64 n_kept columns], boxes of 32 rows x 64 columns, the same swizzle.
cudaError_t attention_tc_configure();
cudaError_t launch_attention_tc(const CUtensorMap& qkv_map, const CUtensorMap& out_map, uint16_t* out, int n_kept, int batch, int seq,
                                const int32_t* seq_lens, int* err, cudaStream_t s, bool pdl, unsigned long long* stamps);

// out = LayerNorm(sum_p partial[p] + bias + resid) * gamma + beta.
struct LnLaunch {
  const float* partial;     // [n_partial][T][d]
  int n_partial;
  const float* bias;        // [d]
  const void* resid;        // [T][d], fp32 or bf16
  int resid_bf16;
  const float* gamma;
  const float* beta;
  float eps;
  int T, d;
  float* out_f32;           // optional
  uint16_t* out_bf16;       // optional
  int sm_count;
  int discard;              // the planes are not needed after this launch: it may drop them from L2 unwritten
  unsigned long long* stamps;   // profiling record or null
};
cudaError_t launch_layernorm(const LnLaunch& p, cudaStream_t s, bool pdl);

// fp32 -> bf16 (round-to-nearest-even) copy of the activations the first GEMM reads.
cudaError_t launch_cast_bf16(const float* in, uint16_t* out, size_t n, cudaStream_t s, bool pdl, unsigned long long* stamps);

// Stand-alone decode of one matrix (inspection / parity).
struct DecodeLaunch {
  const uint4* codes;       // re-tiled stream of the matrix (raw fp32 when bits == 32)
  const float* table;
  const uint32_t* out_rc;   // the matrix's outliers: row << 16 | column
  const float* out_val;
  uint32_t n_out;
  uint32_t bits, rows, kc;
  float* w;                 // optional outputs
  uint8_t* codes_out;
  uint16_t* wbf16;
};
cudaError_t launch_decode(const DecodeLaunch& p, cudaStream_t s);

// Launch with or without the programmatic-dependent-launch attribute (every kernel of the layer calls
// pdl_wait before it reads what its predecessor wrote, so consecutive kernels may overlap their prologues).
// `cluster_x` > 1 groups that many consecutive CTAs along x into one thread-block cluster.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                         bool pdl, unsigned cluster_x, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (cluster_x > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster_x; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool pdl,
                                 Args... args) {
  return launch_kernel_cluster(kernel, grid, block, smem, s, pdl, 1u, args...);
}

constexpr int ERR_NONE = 0;
constexpr int ERR_WAIT_TIMEOUT = 1;   // a bounded mbarrier wait ran out
constexpr int ERR_BAD_JOB = 2;        // a job descriptor failed the kernel's own checks

}  // namespace sti
