// Forward 2x zoom, one launch per image (all planes): grid = strips x bands x
// planes, one CTA per tile.  The tile body is in wd_fwd_tile.cuh.  Storage
// types are compile-time parameters for the common pairs (wd_fwd_typed*.cu);
// any other pair, and beta = 0, goes through the run-time-typed kernels here.
#include "wd_cascade.h"
#include "wd_fwd_kernels.cuh"
#include "wd_fwd_model.h"

namespace wdweno {

cudaError_t launch_fwd_typed(const FwdArgs& a, const MethodConsts& k, int bmode,
                             cudaStream_t stream, bool* handled);
cudaError_t launch_fwd_typed_b1(const FwdArgs& a, const MethodConsts& k, cudaStream_t stream,
                                bool* handled);
cudaError_t launch_fwd_typed_bgen(const FwdArgs& a, const MethodConsts& k, cudaStream_t stream,
                                  bool* handled);

int tile_width_fwd() { return fwd_tile::TILE_W; }
int threads_fwd() { return fwd_tile::THREADS; }

namespace {

// A plan is a function of its key alone, so the last ones are remembered (per
// thread, a direct-mapped table): finding one scans some hundred candidates,
// about 10 us of host time.
struct PlanKey {
  int64_t n, m, planes, rows;
  int sms, threads, cols;
  bool operator==(const PlanKey& o) const {
    return n == o.n && m == o.m && planes == o.planes && rows == o.rows && sms == o.sms &&
           threads == o.threads && cols == o.cols;
  }
};
struct PlanSlot {
  bool used;
  PlanKey key;
  FwdPlan plan;
};

}  // namespace

FwdPlan fwd_plan_for(int64_t n, int64_t m, int64_t planes, int sms, int threads, int cols,
                     int64_t rows) {
  const PlanKey key{n, m, planes, rows, sms > 0 ? sms : 152, threads, cols};
  static thread_local PlanSlot table[64];
  const uint64_t h = (uint64_t)(n * 1000003 + m * 10007 + planes * 101 + rows * 7 + threads + cols);
  PlanSlot& slot = table[(h ^ (h >> 17)) & 63];
  if (!slot.used || !(slot.key == key))
    slot = PlanSlot{true, key, fwd_find_plan(n, m, planes, key.sms, threads, cols, rows)};
  return slot.plan;
}

cudaError_t launch_zoom2x_fwd(const FwdArgs& a, const MethodConsts& k, int bmode,
                              cudaStream_t stream) {
  using fwd_tile::DynIO;
  if (bmode == B2 || bmode == B2R) {
    bool handled = false;
    cudaError_t e = launch_fwd_typed(a, k, bmode, stream, &handled);
    if (handled) return e;
    if (bmode == B2R) return fwd_kernels::launch_fwd<B2R, DynIO>(a, k, stream);
    return fwd_kernels::launch_fwd<B2, DynIO>(a, k, stream);
  }
  if (bmode == BGEN) {
    bool handled = false;
    cudaError_t e = k.beta == 1.f ? launch_fwd_typed_b1(a, k, stream, &handled)
                                  : launch_fwd_typed_bgen(a, k, stream, &handled);
    if (handled) return e;
  }
  if (bmode == B0) return fwd_kernels::launch_fwd<B0, DynIO>(a, k, stream);
  return fwd_kernels::launch_fwd<BGEN, DynIO>(a, k, stream);
}

cudaError_t fwd_wait_timeouts(unsigned int* count, bool reset) {
  unsigned int a = 0, b = 0, c = 0, d = 0;
  cudaError_t e = fwd_tile::read_wait_timeouts(&a, reset);
  if (e == cudaSuccess) e = fwd_wait_timeouts_typed(&b, reset);
  if (e == cudaSuccess) e = fwd_wait_timeouts_batched(&c, reset);
  if (e == cudaSuccess) e = fwd_wait_timeouts_cascade(&d, reset);
  *count = a + b + c + d;
  return e;
}

}  // namespace wdweno
