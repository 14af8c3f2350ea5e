// A layer's weights decoded once into bf16 (Section 4.2 decompression into a working buffer), for calls of many tokens.
//
// The fused dequant-GEMM (dqgemm.cu) decodes a weight tile in the CTA that multiplies with it and keeps it in shared memory.
// That is the better way as long as a weight meets few token tiles; with many, the tile takes the shared memory that a deep
// ring of both operands needs, and 64 features per CTA keep the tensor cores waiting for activations (gemm_wide.cu has the
// figures).  Here one warp decodes one task of 4096 weights with the same routine and writes it, already in the layout the
// tensor core reads from shared memory, to the working buffer; the GEMMs then fetch both operands by TMA.
//
// Working buffer of a matrix of N features and K columns: blocks of 128 features x 64 columns, 16 KB each, block
// (n, k) at (n * K / 64 + k) * 16 KB; inside a block a feature's 64 columns are 128 bytes, their 16-byte pieces permuted by
// the feature's number modulo 8 (the 128-byte swizzle of shared-memory operands).  A task is two pieces of 4 KB of it.
//
// One task per warp, no loop: 3072 tasks of a BERT-large layer are 768 CTAs of four warps, all on the device at once.  Bound by
// latency (descriptor, planes, unpacking, store): about 7 us for such a layer.  It runs where nothing can hide it, ahead of a
// forward's first layer and of streamed ones; the others are decoded beside the layer before (gemm_wide.cu).
#include "gemm_device.cuh"

namespace sti {
namespace {

constexpr int kExpandWarps = 4;

struct alignas(1024) ExpandShared {
  uint8_t tile[kExpandWarps][8192];
  uint16_t table[kExpandWarps][kTableStride];
};

// Nothing is stored before the preceding kernel on the stream has finished: it may still read the buffer.
__global__ void __launch_bounds__(kExpandWarps * 32, 6)
expand_kernel(const DecodeTask* __restrict__ tasks, uint32_t n_tasks, uint8_t* __restrict__ dst) {
  __shared__ ExpandShared sm;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, index = blockIdx.x * kExpandWarps + warp;
  const bool mine = index < n_tasks;
  DecodeTask task;
  pdl_launch_dependents();
  if (mine) {
    task = load_task(tasks + index);
    TaskLoads loads;
    issue_loads(task, lane, loads);
    finish_task(task, loads, sm.table[warp], SwizzledPlace(sm.tile[warp], task), lane, 0);
    fence_proxy_async_smem();
  }
  pdl_wait();
  __syncwarp();
  if (mine && lane == 0) {
    store_expanded(task, sm.tile[warp], dst);
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
}

}  // namespace

cudaError_t launch_expand(const ExpandLaunch& p, cudaStream_t s) {
  const unsigned ctas = (p.n_tasks + kExpandWarps - 1) / kExpandWarps;
  return launch_kernel(expand_kernel, dim3(ctas), dim3(kExpandWarps * 32), 0, s, p.pdl, p.tasks, p.n_tasks, p.dst);
}

}  // namespace sti
