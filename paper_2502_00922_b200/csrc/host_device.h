// Functions that the kernels and the host, tests included, compile alike.
#pragma once

#ifdef __CUDACC__
#define HUFFLLM_HD __host__ __device__ __forceinline__
#else
#define HUFFLLM_HD inline
#endif
