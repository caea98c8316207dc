// Forward kernels with the storage types fixed at compile time and beta = 1: the
// same-type pairs.
// (The run-time-typed kernels of wd_fwd.cu issue 484 instructions a px-ch, these 353,
// FP32, 118-column strips, bands of 16 rows: 1x1025x1025 on the 2n-1 grid 34.4 -> 19.4
// us, and with the run-time-typed kernels' best strips, 119, 26.1.)
#include "wd_fwd_kernels.cuh"

namespace wdweno {

cudaError_t launch_fwd_typed_b1(const FwdArgs& a, const MethodConsts& k, cudaStream_t stream,
                                  bool* handled) {
  using fwd_kernels::launch_fwd;
  using fwd_tile::TypedIO;
  *handled = a.in_dtype == a.out_dtype;
  if (!*handled) return cudaSuccess;
  switch (a.in_dtype) {
    case DT_U8: return launch_fwd<B1, TypedIO<uint8_t, uint8_t>>(a, k, stream);
    case DT_F16: return launch_fwd<B1, TypedIO<__half, __half>>(a, k, stream);
    case DT_BF16:
      return launch_fwd<B1, TypedIO<__nv_bfloat16, __nv_bfloat16>>(a, k, stream);
    default: return launch_fwd<B1, TypedIO<float, float>>(a, k, stream);
  }
}

}  // namespace wdweno
