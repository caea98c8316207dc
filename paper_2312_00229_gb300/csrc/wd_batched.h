// Internal launch interface of the persistent batched forward kernel.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "wd_common.cuh"
#include "wdweno.h"

namespace wdweno {

struct BatchedArgs {
  int count;
  const weno_image* in;   // device array
  const weno_image* out;  // device array
  int in_dtype, out_dtype, out_mode;
  int64_t rows_per_band;  // 0: the setup kernel chooses from the images' sizes
  int sms;                // SMs of the device (for that choice)
  int threads;            // CTA width: 256 or 128 (one column per thread), 128 or 64 (two)
  int cols;               // coarse columns per thread: 1 or 2
  void* workspace;        // >= batched_workspace_bytes(count), 16-byte aligned
};

size_t batched_workspace_bytes(int count);

// CTA shape where the caller leaves the strip width open: two-column strips of
// 118 for the kernels with storage types fixed at compile time (the best or
// within 3% of it over 25 batches), one-column strips of 119 for the others
// (different types, beta != 2: mostly 5 to 20% less time than 118; images about
// 64 wide 15 to 20% more).
void batched_default_shape(int bmode, int in_t, int out_t, int* threads, int* cols);

cudaError_t launch_zoom2x_batched(const BatchedArgs& a, const MethodConsts& k, int bmode,
                                  cudaStream_t stream);

}  // namespace wdweno
