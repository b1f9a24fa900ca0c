// For small functions that host code compiles too (their tests do).
#pragma once

#ifdef __CUDACC__
#define RELEARN_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define RELEARN_HOST_DEVICE inline
#endif
