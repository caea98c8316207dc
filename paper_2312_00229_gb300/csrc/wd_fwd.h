// Internal launch interface of the forward kernel (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "wd_common.cuh"
#include "wd_fwd_model.h"

namespace wdweno {

struct FwdArgs {
  const void* in;
  void* out;
  int in_dtype, out_dtype;
  int64_t n, m, planes;          // coarse rows, columns, channels
  int64_t in_sc, in_sh, in_sw;   // element strides
  int64_t out_sc, out_sh, out_sw;
  int64_t orows, ocols;          // output extent (2n or 2n-1, ...)
  int64_t rows_per_band;
  int out_vec;                   // unit column stride and 2-element aligned rows
  int out_vec4;                  // unit column stride and 4-element aligned rows
  int threads;                   // CTA width: 256 or 128 (one column), 128, 96 or 64 (two)
  int cols;                      // coarse columns per thread: 1, or 2 (paired tile)
};

// How output elements of `esz` bytes can be stored together.
__host__ __device__ inline void set_store_modes(FwdArgs& a, int64_t esz) {
  const uint64_t base = reinterpret_cast<uint64_t>(a.out);
  a.out_vec = a.out_sw == 1 && a.out_sh % 2 == 0 && a.out_sc % 2 == 0 &&
              base % (uint64_t)(2 * esz) == 0;
  a.out_vec4 = a.out_sw == 1 && a.out_sh % 4 == 0 && a.out_sc % 4 == 0 &&
               base % (uint64_t)(4 * esz) == 0;
}

// fwd_find_plan (wd_fwd_model.h), the last plans remembered.
FwdPlan fwd_plan_for(int64_t n, int64_t m, int64_t planes, int sms, int threads, int cols,
                     int64_t rows);

int tile_width_fwd();
int threads_fwd();
cudaError_t launch_zoom2x_fwd(const FwdArgs& a, const MethodConsts& k, int bmode,
                              cudaStream_t stream);
// Abandoned bounded waits counted by the forward kernels of each translation
// unit (summed; optionally reset).
cudaError_t fwd_wait_timeouts(unsigned int* count, bool reset);
cudaError_t fwd_wait_timeouts_typed(unsigned int* count, bool reset);
cudaError_t fwd_wait_timeouts_batched(unsigned int* count, bool reset);

}  // namespace wdweno
