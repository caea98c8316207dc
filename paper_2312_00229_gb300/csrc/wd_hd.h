// Functions of headers that also compile for the host alone, without nvcc.
#pragma once

#ifdef __CUDACC__
#define WD_HD __host__ __device__ __forceinline__
#else
#define WD_HD inline
#endif
