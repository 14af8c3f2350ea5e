// Functions that kernels, the host runtime and host-compiled tests share.
#pragma once

#if defined(__CUDACC__)
#define STI_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define STI_HOST_DEVICE inline
#endif
