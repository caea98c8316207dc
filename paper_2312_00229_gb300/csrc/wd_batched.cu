// Batched forward 2x zoom: many images of independent sizes in one
// persistent launch fed by a device-side tile queue.
//
// Workspace (caller-owned, no initialisation needed):
//   [0]   unsigned long long  head, next tile
//   [8]   unsigned long long  total, tiles of all images; rows per band in the
//                             top 16 bits
//   [16]  unsigned long long  prefix[count + 1], the exclusive prefix sum of
//                             the tiles of each image (a malformed image has
//                             none)
// The setup kernel fills it from the device-resident descriptors, so a
// stream capture of the call replays correctly with new pixel data.  The
// persistent kernel is in wd_batched_kernel.cuh; this unit instantiates it
// with one coarse column per thread, wd_batched2.cu with two.
#include "wd_batched_kernel.cuh"
#include "wd_fwd_model.h"

namespace wdweno {

cudaError_t launch_batched_paired(const BatchedArgs& a, const MethodConsts& k, int bmode,
                                  cudaStream_t stream);

namespace {

using batched::Queue;
using batched::strip_width;

constexpr int SETUP_THREADS = 1024;

__device__ bool descriptor_ok(const weno_image& in, const weno_image& out, int out_mode) {
  if (!in.data || !out.data) return false;
  if (in.height < 1 || in.width < 1 || in.channels < 1 || in.channels >= 65536) return false;
  if (in.height >= (int64_t(1) << 31) || in.width >= (int64_t(1) << 31)) return false;
  if (in.stride_c < 1 || in.stride_h < 1 || in.stride_w < 1) return false;
  if (out.stride_c < 1 || out.stride_h < 1 || out.stride_w < 1) return false;
  const int64_t d = out_mode == WENO_OUT_2N_MINUS_1 ? 1 : 0;
  return out.height == 2 * in.height - d && out.width == 2 * in.width - d &&
         out.channels == in.channels;
}

// Tiles of one image with bands of at most `rows` rows and strips of `tw`
// columns.
__device__ unsigned long long image_tiles(const weno_image& in, int64_t rows, int tw) {
  const unsigned long long strips = ((unsigned long long)in.width + tw - 1) / tw;
  const int64_t r = batched::even_band(in.height, rows);
  const unsigned long long bands = (unsigned long long)((in.height + r - 1) / r);
  return strips * bands * (unsigned long long)in.channels;
}

// Band heights the setup kernel chooses from.
constexpr int CANDS = BATCHED_CANDS;
__constant__ BatchedHeights g_heights = BATCHED_HEIGHTS;

__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One CTA: validates the descriptors, chooses the band height where the
// caller left it open, and writes the exclusive prefix sum of tiles.
//
// The choice takes the band height with the least modelled time (batched_us of
// wd_fwd_model.h).  Against the fixed default before any choice, 128 rows and
// one-column strips of 247, uint8 unless said, graph replay: 5 images of sides 48..96 104
// -> 23 us; 16 of 100..400 110 -> 50; 30 BF16 planes of 64..512 114 -> 66; 64 FP16 images
// of 64..1024 706 -> 560; 1100 of 16..24 1101 -> 134; one of 1080x1920 106 -> 76, of
// 2000x2000 159 -> 129.  About 8 us of a launch is the choice itself, on one CTA.
__global__ void __launch_bounds__(SETUP_THREADS) batched_setup_kernel(BatchedArgs a,
                                                                      FwdShape shape) {
  Queue* q = static_cast<Queue*>(a.workspace);
  __shared__ unsigned long long part[SETUP_THREADS / 32];
  __shared__ float c_tiles[CANDS], c_steps[CANDS];
  __shared__ int c_longest[CANDS];
  __shared__ int s_rows;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int tw = strip_width(a.threads, a.cols);
  const int chunk = (a.count + SETUP_THREADS - 1) / SETUP_THREADS;
  const int lo = min(a.count, t * chunk), hi = min(a.count, lo + chunk);
  int64_t rows = a.rows_per_band;
  if (rows <= 0) {
    if (t < CANDS) {
      c_tiles[t] = c_steps[t] = 0.f;
      c_longest[t] = 0;
    }
    __syncthreads();
    BatchedCost c[CANDS];
#pragma unroll
    for (int j = 0; j < CANDS; ++j) c[j] = BatchedCost{0.f, 0.f, 0.f};
    for (int i = lo; i < hi; ++i) {
      const weno_image in = a.in[i], out = a.out[i];
      if (!descriptor_ok(in, out, a.out_mode)) continue;
      const float strips = float((in.width + tw - 1) / tw) * float(in.channels);
#pragma unroll
      for (int j = 0; j < CANDS; ++j)
        batched_add(c[j], (int)in.height, strips, g_heights.rows[j]);
    }
    if (warp * 32 * chunk < a.count) {  // warps with images
#pragma unroll
      for (int j = 0; j < CANDS; ++j) {
        const float tiles = warp_sum(c[j].tiles), steps = warp_sum(c[j].steps);
        const float longest = warp_max(c[j].longest);
        if (lane == 0) {
          atomicAdd(&c_tiles[j], tiles);
          atomicAdd(&c_steps[j], steps);
          atomicMax(&c_longest[j], (int)longest);
        }
      }
    }
    __syncthreads();
    if (warp == 0) {
      float us = 3.0e38f;
      if (lane < CANDS && c_tiles[lane] > 0.f)
        us = batched_us(shape, a.sms,
                        BatchedCost{c_tiles[lane], c_steps[lane], float(c_longest[lane])});
      int best = lane;
      for (int o = 16; o; o >>= 1) {
        const float v = __shfl_xor_sync(0xffffffffu, us, o);
        const int w = __shfl_xor_sync(0xffffffffu, best, o);
        if (v < us || (v == us && w < best)) {
          us = v;
          best = w;
        }
      }
      if (lane == 0) s_rows = g_heights.rows[best < CANDS ? best : 0];
    }
    __syncthreads();
    rows = s_rows;
  }
  unsigned long long sum = 0ULL;
  for (int i = lo; i < hi; ++i) {
    const weno_image in = a.in[i], out = a.out[i];
    if (descriptor_ok(in, out, a.out_mode)) sum += image_tiles(in, rows, tw);
  }
  // inclusive scan over the threads: within warps, then over their totals
  unsigned long long scan = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(0xffffffffu, scan, o);
    if (lane >= o) scan += v;
  }
  if (lane == 31) part[warp] = scan;
  __syncthreads();
  if (warp == 0) {
    unsigned long long v = part[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    part[lane] = v;
  }
  __syncthreads();
  if (warp > 0) scan += part[warp - 1];
  unsigned long long run = scan - sum;  // exclusive start
  for (int i = lo; i < hi; ++i) {
    q->prefix[i] = run;
    const weno_image in = a.in[i], out = a.out[i];
    if (descriptor_ok(in, out, a.out_mode)) run += image_tiles(in, rows, tw);
  }
  if (t == SETUP_THREADS - 1) {
    q->prefix[a.count] = scan;
    q->total = scan | ((unsigned long long)rows << batched::ROWS_SHIFT);
    q->head = 0ULL;
  }
}

}  // namespace

size_t batched_workspace_bytes(int count) {
  size_t b = 16 + 8 * (size_t(count) + 1);
  return (b + 15) & ~size_t(15);
}

void batched_default_shape(int bmode, int in_t, int out_t, int* threads, int* cols) {
  // (launch_typed of wd_batched_kernel.cuh)
  const bool fixed = in_t == out_t && (bmode == B2 || (bmode == B2R && in_t != DT_BF16));
  *threads = fixed ? 64 : 128;
  *cols = fixed ? 2 : 1;
}

cudaError_t launch_zoom2x_batched(const BatchedArgs& a, const MethodConsts& k, int bmode,
                                  cudaStream_t stream) {
  FwdShape shape = FWD_SHAPES[0];
  for (const FwdShape& s : FWD_SHAPES)
    if (s.threads == a.threads && s.cols == a.cols) shape = s;
  batched_setup_kernel<<<1, SETUP_THREADS, 0, stream>>>(a, shape);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (a.cols == 2) return launch_batched_paired(a, k, bmode, stream);
  return batched::launch_typed<1>(a, k, bmode, stream);
}

cudaError_t fwd_wait_timeouts_batched(unsigned int* count, bool reset) {
  return fwd_tile::read_wait_timeouts(count, reset);
}

}  // namespace wdweno
