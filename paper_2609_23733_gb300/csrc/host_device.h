// Functions that the kernels and the host evaluate alike.
#pragma once

#ifdef __CUDACC__
#define VP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define VP_HOST_DEVICE inline
#endif
