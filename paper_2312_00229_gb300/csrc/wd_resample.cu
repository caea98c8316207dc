// Tensor-product WENO resampling to an arbitrary size (arXiv 2312.00229,
// Sec. 3.3, Eq. tensor), the second stage of the arbitrary-scale zoom.
//
// The 1-D WENO interpolant of Sec. 2 on the cell [x_i, x_{i+1}], t in [0, 1],
// with samples v0..v3 at x_{i-1..i+2}: writing g = v2 - v1,
// sL = v0 - 2 v1 + v2 and sR = v1 - 2 v2 + v3, the two quadratics are
//     p_i(t)     = v1 + g t + sL (t^2 - t) / 2
//     p_{i+1}(t) = v1 + g t + sR (t^2 - t) / 2
// (Eq. Tocnost), their indicators (Sec. 2) are g^2 + 13/12 sL^2 and
// g^2 + 13/12 sR^2, and the linear weights that recover the cubic (Eq.
// PolinomZaVelikiStencil) are C_0 = (2 - t)/3, C_1 = (1 + t)/3, so
//     u = v1 + g t + (t^2 - t)/2 (alpha_0 sL + alpha_1 sR) / (alpha_0 + alpha_1),
//     alpha_s = C_s / (eps_h + SI_s)^beta                     (Eq. IzrazOmega).
// Inputs outside the image are clamped to the edge.
//
// Everything of an interpolant but C_s and the powers of t belongs to its
// cell, not to t: g, sL, sR and the weights' powers of the indicators are
// formed once per cell (Cell2) and evaluated at each output inside (eval2).
#include <atomic>
#include <type_traits>

#include "wd_common.cuh"
#include "wd_packed.cuh"
#include "wd_resample.h"
#include "wd_resample_plan.h"
#include "wd_resample_window.h"

namespace wdweno {

namespace {

// Two cells at once on Blackwell's packed two-lane FP32 instructions (pk_*
// helpers of wd_packed.cuh).  wL, wR: the indicators' part of the weights
// alpha_0 : alpha_1 = C_0 eR^beta : C_1 eL^beta.
struct Cell2 {
  f2 v1, g, sL, sR, wL, wR;
};

template <int BMODE>
__device__ __forceinline__ Cell2 cell2(f2 v0, f2 v1, f2 v2, f2 v3, float eps, float beta) {
  Cell2 c;
  c.v1 = v1;
  c.g = pk_sub(v2, v1);
  c.sL = pk_fma(pk_bc(-2.f), v1, pk_add(v0, v2));
  c.sR = pk_fma(pk_bc(-2.f), v2, pk_add(v1, v3));
  if (BMODE == B0) return c;
  const f2 k2 = pk_bc(13.f / 12.f), e = pk_bc(eps);
  const f2 eL = pk_fma(c.g, c.g, pk_fma(pk_mul(k2, c.sL), c.sL, e));
  const f2 eR = pk_fma(c.g, c.g, pk_fma(pk_mul(k2, c.sR), c.sR, e));
  if (BMODE == B2R) {
    // the squares as written; the host picks this form only where the storage
    // type bounds the data so that every square, their sum and the numerator
    // of eval2 are normal FP32 numbers
    c.wL = pk_mul(eL, eL);
    c.wR = pk_mul(eR, eR);
  } else {
    // both indicators divided by the larger one, so no power over- or
    // underflows.  eps is at least 1e-30 (host side), so the larger indicator
    // is a normal number.
    const f2 inv = pk_rcp(make_float2(fmaxf(eL.x, eR.x), fmaxf(eL.y, eR.y)));
    c.wL = pk_mul(eL, inv);
    c.wR = pk_mul(eR, inv);
    if (BMODE != B2) {
      const f2 b = pk_bc(beta);
      const f2 lR = pk_mul(b, make_float2(lg2_approx(c.wR.x), lg2_approx(c.wR.y)));
      const f2 lL = pk_mul(b, make_float2(lg2_approx(c.wL.x), lg2_approx(c.wL.y)));
      c.wR = make_float2(ex2_approx(lR.x), ex2_approx(lR.y));
      c.wL = make_float2(ex2_approx(lL.x), ex2_approx(lL.y));
    }
  }
  return c;
}

// The interpolants at offset t: C0 = (2 - t)/3, h = (t^2 - t)/2.
template <int BMODE>
__device__ __forceinline__ f2 eval2(const Cell2& c, f2 t, f2 C0, f2 h) {
  const f2 C1 = pk_sub(pk_bc(1.f), C0);
  f2 a0, a1;
  if (BMODE == B0) {
    a0 = C0;
    a1 = C1;
  } else if (BMODE == B2) {
    a0 = pk_mul(pk_mul(C0, c.wR), c.wR);
    a1 = pk_mul(pk_mul(C1, c.wL), c.wL);
  } else {
    a0 = pk_mul(C0, c.wR);
    a1 = pk_mul(C1, c.wL);
  }
  // a0 + a1 >= 1/3 in the scaled forms: one ratio is 1 and both C_s are at
  // least 1/3
  const f2 mix = pk_mul(pk_fma(a0, c.sL, pk_mul(a1, c.sR)), pk_rcp(pk_add(a0, a1)));
  return pk_fma(h, mix, pk_fma(c.g, t, c.v1));
}

__device__ __forceinline__ float pos_c0(float t) { return (2.f - t) * (1.f / 3.f); }
__device__ __forceinline__ float pos_h(float t) { return 0.5f * fmaf(t, t, -t); }

// Cell index and offset of output index j on the endpoint-aligned grid of
// n_out points over 0..n-1: i = floor(j (n-1) / (n_out-1)) exactly (by
// multiply-high when the numerator fits 32 bits), t = remainder / (n_out-1).
// WIDE: larger numerators (products of sides from 2^32 on) by a quotient in FP64,
// at most one off as it is below 2^31, in place of a 64-bit integer division
// (a line of 10^6 samples -> 3 10^6 57 -> 29 us; in the other kernels, which
// find fewer positions, the longer code costs 1 to 2% at every size).
template <bool WIDE = false>
__device__ __forceinline__ void grid_pos(int j, int n, int n_out, const AxisDiv& d, int& i,
                                         float& t) {
  if (n <= 1 || n_out <= 1) { i = 0; t = 0.f; return; }
  const int den = n_out - 1;
  if (d.fast) {
    const uint32_t num = (uint32_t)j * (uint32_t)(n - 1);
    const uint32_t t1 = __umulhi(d.mag, num);
    const uint32_t q = (t1 + ((num - t1) >> d.sh1)) >> d.sh2;
    i = (int)q;
    t = (float)(int)(num - q * (uint32_t)den) * d.inv;
  } else {
    const int64_t num = (int64_t)j * (n - 1);
    int64_t q, rest;
    if (WIDE) {
      q = (int64_t)((double)num * d.inv64);
      rest = num - q * den;
      if (rest < 0) {
        --q;
        rest += den;
      } else if (rest >= den) {
        ++q;
        rest -= den;
      }
    } else {
      q = num / den;
      rest = num - q * den;
    }
    i = (int)q;
    t = (float)rest * d.inv;
  }
  if (i > n - 2) { i = n - 2; t = 1.f; }  // last sample: t = 1 on the last cell
}

__device__ __forceinline__ int clamp_idx(int v, int n) { return v < 0 ? 0 : (v > n - 1 ? n - 1 : v); }

// Storage access: a concrete element type, or Dyn for the run-time type.
struct Dyn {};

// Storage bits of one element and their value (the loads of a group are all
// issued before any of them is converted).
template <class T>
__device__ __forceinline__ uint32_t rs_load_bits(const void* base, int64_t idx, int dt) {
  if constexpr (std::is_same<T, Dyn>::value) {
    return load_elem_bits(base, idx, dt);
  } else {
    return load_elem_bits(base, idx, DTypeOf<T>::value);
  }
}

template <class T>
__device__ __forceinline__ float rs_value(uint32_t b, int dt) {
  if constexpr (std::is_same<T, Dyn>::value) {
    return elem_bits_value(b, dt);
  } else {
    return elem_bits_value(b, DTypeOf<T>::value);
  }
}

template <class T>
__device__ __forceinline__ void rs_store(void* base, int64_t idx, float v, int dt, int clampf) {
  if constexpr (std::is_same<T, Dyn>::value) {
    store_elem(base, idx, v, dt, clampf);
  } else {
    store_typed<T>(base, idx, v, clampf);
  }
}

// An output from its 16 samples: all loads are issued before the first is used,
// columns are interpolated in packed pairs.
template <int BMODE, class TIn>
__device__ __forceinline__ float output_at(const ResampleArgs& a, int64_t plane, int i, float ty,
                                           int j, float tx, float eps, float beta) {
  const int n = (int)a.n, m = (int)a.m;
  int64_t row[4], col[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    row[p] = plane * a.in_sc + (int64_t)clamp_idx(i - 1 + p, n) * a.in_sh;
    col[p] = (int64_t)clamp_idx(j - 1 + p, m) * a.in_sw;
  }
  uint32_t b[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) b[p][q] = rs_load_bits<TIn>(a.in, row[p] + col[q], a.in_dtype);
  f2 z[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    f2 v[4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
      v[p] = make_float2(rs_value<TIn>(b[p][2 * q], a.in_dtype),
                         rs_value<TIn>(b[p][2 * q + 1], a.in_dtype));
    z[q] = n > 1 ? eval2<BMODE>(cell2<BMODE>(v[0], v[1], v[2], v[3], eps, beta), pk_bc(ty),
                                pk_bc(pos_c0(ty)), pk_bc(pos_h(ty)))
                 : v[1];
  }
  float u = z[0].y;
  if (m > 1)
    u = eval2<BMODE>(cell2<BMODE>(pk_bc(z[0].x), pk_bc(z[0].y), pk_bc(z[1].x), pk_bc(z[1].y), eps,
                                  beta),
                     pk_bc(tx), pk_bc(pos_c0(tx)), pk_bc(pos_h(tx)))
            .x;
  return u;
}

// The interpolant at cell i, offset t of a line of n samples `stride` apart.
template <int BMODE, class TIn>
__device__ __forceinline__ float line_at(const ResampleArgs& a, int64_t base, int64_t stride,
                                         int i, int n, float t, float eps, float beta) {
  if (n == 1) return rs_value<TIn>(rs_load_bits<TIn>(a.in, base, a.in_dtype), a.in_dtype);
  uint32_t b[4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
    b[p] = rs_load_bits<TIn>(a.in, base + (int64_t)clamp_idx(i - 1 + p, n) * stride, a.in_dtype);
  f2 v[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) v[p] = pk_bc(rs_value<TIn>(b[p], a.in_dtype));
  return eval2<BMODE>(cell2<BMODE>(v[0], v[1], v[2], v[3], eps, beta), pk_bc(t), pk_bc(pos_c0(t)),
                      pk_bc(pos_h(t)))
      .x;
}

// One thread per output, for reductions beyond 1/2 (little to share between
// neighbouring outputs).  1080p -> 480x270 uint8: 9.2 us with run-time types and 64-bit
// positions, now 6.8.
template <int BMODE, class TIn, class TOut>
__global__ void __launch_bounds__(256) resample_kernel(ResampleArgs a, float eps, float beta) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t r = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
  if (r >= a.n_out || c >= a.m_out) return;
  const int64_t plane = blockIdx.z;
  const int n = (int)a.n, m = (int)a.m;
  int i, j;
  float ty, tx;
  grid_pos((int)r, n, (int)a.n_out, a.div_y, i, ty);
  grid_pos((int)c, m, (int)a.m_out, a.div_x, j, tx);
  const float u = output_at<BMODE, TIn>(a, plane, i, ty, j, tx, eps, beta);
  rs_store<TOut>(a.out, plane * a.out_sc + r * a.out_sh + c * a.out_sw, u, a.out_dtype,
                 a.clamp_float);
}

// Single-sample axes, where one interpolant makes an output, and fewer rows than
// a tile has warps, where most of a tile's warps would idle: one thread per
// output column and `span` output rows, blockDim.y apart, or, of a single input
// column, per output row and `span` columns, blockDim.x apart.  What the outputs of
// a thread share is formed once: the column's position, and the output itself
// where the input has one row or one column.  uint8, us, by one thread per output and
// now: 1x1000 -> 1000x3000 26 and 5.3, 1x10^6 -> 8x10^6 97 and 12 (bound by the
// positions and the stores), 400000x1 -> 500000x1 225 and 7.0, 500x1 -> 500x3000 17 and
// 3.5; 4x10^6 -> 7x700000, 16 loads an output, 55 and 53.
template <int BMODE, class TIn, class TOut>
__global__ void __launch_bounds__(256)
    resample_lines_kernel(ResampleArgs a, float eps, float beta, int span) {
  const int n = (int)a.n, m = (int)a.m;
  const bool along_x = m == 1 && n > 1;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x * (along_x ? span : 1) + threadIdx.x;
  int64_t r = (int64_t)blockIdx.y * blockDim.y * (along_x ? 1 : span) + threadIdx.y;
  if (r >= a.n_out || c >= a.m_out) return;
  const int64_t plane = blockIdx.z, base = plane * a.in_sc;
  int64_t o = plane * a.out_sc + r * a.out_sh + c * a.out_sw;
  const int64_t step = along_x ? blockDim.x * a.out_sw : blockDim.y * a.out_sh;
  // outputs of this thread
  const int64_t left = along_x ? (a.m_out - c - 1) / blockDim.x : (a.n_out - r - 1) / blockDim.y;
  const int count = left < span ? (int)left + 1 : span;
  int i, j;
  float ty, tx;
  if (along_x)
    grid_pos<true>((int)r, n, (int)a.n_out, a.div_y, i, ty);
  else
    grid_pos<true>((int)c, m, (int)a.m_out, a.div_x, j, tx);
  if (n == 1 || m == 1) {  // (uniform)
    const float u = along_x ? line_at<BMODE, TIn>(a, base, a.in_sh, i, n, ty, eps, beta)
                            : line_at<BMODE, TIn>(a, base, a.in_sw, j, m, tx, eps, beta);
    for (int k = 0; k < count; ++k, o += step)
      rs_store<TOut>(a.out, o, u, a.out_dtype, a.clamp_float);
  } else {
    for (int k = 0; k < count; ++k, o += step, r += blockDim.y) {
      grid_pos<true>((int)r, n, (int)a.n_out, a.div_y, i, ty);
      rs_store<TOut>(a.out, o, output_at<BMODE, TIn>(a, plane, i, ty, j, tx, eps, beta),
                     a.out_dtype, a.clamp_float);
    }
  }
}

// ---- the tiled forms (sizes: wd_resample_plan.h) -------------------------------------
constexpr int RS_THREADS = 32 * RS_WARPS;
constexpr int RS_REG_OUT = 4;  // outputs of a cell with constants in registers

template <class T>
__device__ __forceinline__ int elem_bytes(int dt) {
  if constexpr (std::is_same<T, Dyn>::value)
    return dt == DT_U8 ? 1 : (dt == DT_F32 ? 4 : 2);
  else
    return (int)sizeof(T);
}

// A warp copies a row of `nc` encoded elements from shared memory to `out`, in
// words of four elements where the output's rows allow that.
template <class E, class V>
__device__ __forceinline__ void flush_as(char* out, int64_t sw, int vec4,
                                         const unsigned char* stage, int nc, int lane) {
  int done = 0;
  if (vec4) {
    const int words = nc >> 2;
    V* dst = reinterpret_cast<V*>(out) + lane;
    const V* src = reinterpret_cast<const V*>(stage) + lane;
#pragma unroll
    for (int w = 0; w < RS_TC_MAX / 128 + 1; ++w) {
      if (32 * w >= words) break;  // (uniform)
      if (lane + 32 * w < words) dst[32 * w] = src[32 * w];
    }
    done = words * 4;
    if (done == nc) return;
  }
  E* dst = reinterpret_cast<E*>(out);
  const E* src = reinterpret_cast<const E*>(stage);
  for (int c = done + lane; c < nc; c += 32) dst[c * sw] = src[c];
}

template <class T>
__device__ __forceinline__ void rs_flush(char* out, int64_t sw, int vec4,
                                         const unsigned char* stage, int nc, int lane, int dt) {
  const int esz = elem_bytes<T>(dt);
  if (esz == 1)
    flush_as<uint8_t, uint32_t>(out, sw, vec4, stage, nc, lane);
  else if (esz == 4)
    flush_as<float, float4>(out, sw, vec4, stage, nc, lane);
  else
    flush_as<uint16_t, uint2>(out, sw, vec4, stage, nc, lane);
}

// Separable tiled form for output/input spacing ratios down to 1/2 on both
// axes.  A CTA of 8 warps owns a tile of output columns and 8 `rows` output
// rows of one plane; a warp owns `rows` consecutive ones and never waits for
// another after the position tables:
//   pass 1   the column interpolants z(r, k) = w(A(:, k), y_r) (Eq. tensor,
//            first factor) of its rows at the tile's window columns, from the
//            input rows straight to registers (all loads in flight before the
//            first is used); an input cell's indicators serve every output
//            row inside it
//   pass 2   the row interpolants across the z values (second factor)
// Per output this is 1 + (in/out column ratio) + halo 1-D interpolants
// instead of the 5 of the direct form.
//
// The forms differ in the tile and in pass 2 (which one runs: wd_resample_plan.h):
//   RS_CELLS    magnified columns: the tile is as wide as fits 64 window columns,
//               two per lane, and pass 2 gives a lane two cells of the row,
//               whose indicators serve all of their outputs (three at 3x)
//   RS_OUTPUTS  the outputs of 128 window columns, 128 at most, and up to eight
//               rows a warp; pass 2 gives a lane up to four outputs, each with
//               its cell's indicators formed anew
//   RS_REDUCED  128 outputs, four rows a warp, up to 264 window columns; pass 2
//               by outputs
// The encoded outputs go through a staging row in shared memory to whole-word
// stores.
//
// What bounds it: instruction issue (71% of slots at 3x uint8; FMA pipe 46%, LSU
// 44%), a quarter of it address arithmetic.  Against the form before (a decoded
// window in shared memory, every output's indicators formed anew, 4-byte
// stores from four outputs per lane with strided z reads), us:
//     1080p uint8 -> 3x 124 -> 75, -> 2x 77 -> 45, -> 1.33x 39.9 -> 31.6, 1x 33 -> 24.5
//     4317x7677 FP32 -> 3240x5760 uint8 353 -> 214; 1080p FP32 -> 900x1600 26 -> 19.4
// (79, 48, 33.5, 26, 224 and 20 before windows inside the image took their rows one
// stride apart without the clamped offsets, and the rows of each cell were
// counted once per warp).
// Small outputs are bound by the launch and one warp's chain: 64x64 -> 100x100 4.7
// -> 3.3 us.  Packed constants pinned in registers, scalar instead of packed
// arithmetic, and two or four CTAs per SM measured slower.
template <int FORM>
struct RsShared {
  static constexpr int TC = FORM == RS_CELLS ? RS_TC_MAX : RS_TC_DOWN;
  static constexpr int WZ =
      FORM == RS_CELLS ? RS_WC_UP + 4 : (FORM == RS_OUTPUTS ? RS_WC_OUT : RS_WC_DOWN);
  static constexpr int ROWS = FORM == RS_REDUCED ? RS_DOWN_ROWS : RS_MAX_ROWS;  // a warp, at most
  float4 row_a[RS_WARPS * RS_MAX_ROWS];  // (t, t, C0, C0) of each output row
  float2 row_h[RS_WARPS * RS_MAX_ROWS];  // (h, h)
  int64_t in_off[RS_MAX_IN];             // byte offset of each (clamped) input row
  int row_i[RS_WARPS * RS_MAX_ROWS];     // its cell
  int col_j[TC];
  float col_t[TC];
  int start[RS_WC_UP + 1];               // first output column of each cell (RS_CELLS)
  float z[RS_WARPS][ROWS][WZ];
  // encoded outputs of a row, and a spare element
  __align__(16) unsigned char stage[RS_WARPS][4 * TC + 16];
};

// Pass 1 of a warp: z of its output rows (tile rows q0 ..) at window columns
// k0 + lane and k0 + lane + 32 (those past the window are not used).  rows_in:
// input rows they read; rows_of: output rows in each cell, four bits a cell;
// in_base: input row of in_off[0].
template <int BMODE, class TIn, class SH>
__device__ __forceinline__ void column_pass(const ResampleArgs& a, SH& sh, int warp, int lane,
                                            int q0, int rows_in, uint32_t rows_of, int in_base,
                                            int kfirst, int wc,
                                            int k0, const char* plane, int esz, float eps,
                                            float beta) {
  const int ka = k0 + lane, kb = ka + 32;
  const int first = sh.row_i[q0];
  uint32_t ba[RS_PRE], bb[RS_PRE];
  if (a.in_sw == 1 && window_inside(kfirst, k0, (int)a.m, first, rows_in, (int)a.n)) {
    // (uniform) nothing to clamp: rows one stride apart, columns at fixed offsets
    const char* p0 =
        plane + (int64_t)(first - 1) * a.in_sh * esz + column_bytes(kfirst, ka, esz);
    const int64_t step = a.in_sh * esz;
#pragma unroll
    for (int p = 0; p < RS_PRE; ++p) {
      if (p < rows_in) {
        ba[p] = rs_load_bits<TIn>(p0, 0, a.in_dtype);
        bb[p] = rs_load_bits<TIn>(p0, 32, a.in_dtype);
        p0 += step;
      }
    }
  } else {
    const char* pa =
        plane + (int64_t)clamp_idx(kfirst + min(ka, wc - 1), (int)a.m) * a.in_sw * esz;
    const char* pb =
        plane + (int64_t)clamp_idx(kfirst + min(kb, wc - 1), (int)a.m) * a.in_sw * esz;
    const int64_t* off = sh.in_off + (first - 1 - in_base);
#pragma unroll
    for (int p = 0; p < RS_PRE; ++p) {
      if (p < rows_in) {  // (uniform)
        ba[p] = rs_load_bits<TIn>(pa + off[p], 0, a.in_dtype);
        bb[p] = rs_load_bits<TIn>(pb + off[p], 0, a.in_dtype);
      }
    }
  }
  f2 v[RS_PRE];
#pragma unroll
  for (int p = 0; p < RS_PRE; ++p)
    if (p < rows_in)
      v[p] = make_float2(rs_value<TIn>(ba[p], a.in_dtype), rs_value<TIn>(bb[p], a.in_dtype));
  const bool in_a = ka < SH::WZ, in_b = kb < SH::WZ;
  float* z = &sh.z[warp][0][0] + k0 + lane;
  const float4* ra = sh.row_a + q0;
  const float2* rh = sh.row_h + q0;
#pragma unroll
  for (int p = 0; p < RS_MAX_CELLS; ++p) {
    int rows = (rows_of >> (4 * p)) & 15;  // output rows in cell p
    if (rows) {
      const Cell2 c = cell2<BMODE>(v[p], v[p + 1], v[p + 2], v[p + 3], eps, beta);
#pragma unroll 1
      do {
        const float4 ta = *ra++;
        const float2 th = *rh++;
        const f2 zz = eval2<BMODE>(c, make_float2(ta.x, ta.y), make_float2(ta.z, ta.w), th);
        if (in_a) z[0] = zz.x;
        if (in_b) z[32] = zz.y;
        z += SH::WZ;
      } while (--rows);
    }
  }
}

// Pass 2 of a warp by cells: of at most NJ outputs, whose
// positions are kept in registers (with NJ = RS_REG_OUT cells may have more,
// which read theirs from the tables).
template <int BMODE, class TOut, int NJ, class SH>
__device__ __forceinline__ void row_pass_up(const ResampleArgs& a, SH& sh, int warp, int lane,
                                            int nq, int nc, int cells, int most, char* out,
                                            int64_t row_bytes, float eps, float beta) {
  // cells `lane` and `lane + 32`: their output columns and positions; outputs
  // a cell does not have go to a spare element after the row
  const int sa = lane < cells ? sh.start[lane] : 0;
  const int na = lane < cells ? sh.start[lane + 1] - sa : 0;
  const int sb = lane + 32 < cells ? sh.start[lane + 32] : 0;
  const int nb = lane + 32 < cells ? sh.start[lane + 33] - sb : 0;
  f2 t[NJ], C0[NJ], h[NJ];
  int ia[NJ], ib[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    ia[j] = j < na ? sa + j : RS_TC_MAX;
    ib[j] = j < nb ? sb + j : RS_TC_MAX;
    t[j] = make_float2(sh.col_t[j < na ? sa + j : 0], sh.col_t[j < nb ? sb + j : 0]);
    C0[j] = make_float2(pos_c0(t[j].x), pos_c0(t[j].y));
    h[j] = make_float2(pos_h(t[j].x), pos_h(t[j].y));
  }
  unsigned char* stage = sh.stage[warp];
  const float* zr = sh.z[warp][0] + lane;
#pragma unroll 1
  for (int q = 0; q < nq; ++q, out += row_bytes, zr += SH::WZ) {
    const Cell2 c = cell2<BMODE>(make_float2(zr[0], zr[32]), make_float2(zr[1], zr[33]),
                                 make_float2(zr[2], zr[34]), make_float2(zr[3], zr[35]), eps,
                                 beta);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const f2 u = eval2<BMODE>(c, t[j], C0[j], h[j]);
      rs_store<TOut>(stage, ia[j], u.x, a.out_dtype, a.clamp_float);
      rs_store<TOut>(stage, ib[j], u.y, a.out_dtype, a.clamp_float);
    }
    if (NJ == RS_REG_OUT) {
#pragma unroll 1
      for (int j = NJ; j < most; ++j) {
        const f2 tt = make_float2(sh.col_t[j < na ? sa + j : 0], sh.col_t[j < nb ? sb + j : 0]);
        const f2 u = eval2<BMODE>(c, tt, make_float2(pos_c0(tt.x), pos_c0(tt.y)),
                                  make_float2(pos_h(tt.x), pos_h(tt.y)));
        rs_store<TOut>(stage, j < na ? sa + j : RS_TC_MAX, u.x, a.out_dtype, a.clamp_float);
        rs_store<TOut>(stage, j < nb ? sb + j : RS_TC_MAX, u.y, a.out_dtype, a.clamp_float);
      }
    }
    __syncwarp();
    rs_flush<TOut>(out, a.out_sw, a.out_vec4, stage, nc, lane, a.out_dtype);
    __syncwarp();
  }
}

// Pass 2 of a warp by outputs: outputs lane, lane + 32, .. of the row
// (consecutive lanes read z values at most 2 apart), two in a packed pair.
template <int BMODE, class TOut, class SH>
__device__ __forceinline__ void row_pass_outputs(const ResampleArgs& a, SH& sh, int warp, int lane,
                                              int nq, int nc, int kfirst, char* out,
                                              int64_t row_bytes, float eps, float beta) {
  constexpr bool FORM_OUT = SH::ROWS != RS_DOWN_ROWS;
  const float* z[4];
  f2 t[2], C0[2], h[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int ca = min(lane + 64 * q, nc - 1), cb = min(lane + 64 * q + 32, nc - 1);
    z[2 * q] = sh.z[warp][0] + (sh.col_j[ca] - 1 - kfirst);
    z[2 * q + 1] = sh.z[warp][0] + (sh.col_j[cb] - 1 - kfirst);
    t[q] = make_float2(sh.col_t[ca], sh.col_t[cb]);
    C0[q] = make_float2(pos_c0(t[q].x), pos_c0(t[q].y));
    h[q] = make_float2(pos_h(t[q].x), pos_h(t[q].y));
  }
  unsigned char* stage = sh.stage[warp];
#pragma unroll
  for (int r = 0; r < SH::ROWS; ++r, out += row_bytes) {
    if (r >= nq) break;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (FORM_OUT && q == 1 && nc <= 64) break;  // (uniform)
      const float* za = z[2 * q] + r * SH::WZ;
      const float* zb = z[2 * q + 1] + r * SH::WZ;
      const f2 u = eval2<BMODE>(
          cell2<BMODE>(make_float2(za[0], zb[0]), make_float2(za[1], zb[1]),
                       make_float2(za[2], zb[2]), make_float2(za[3], zb[3]), eps, beta),
          t[q], C0[q], h[q]);
      // columns past the tile repeat its last and land after the row
      rs_store<TOut>(stage, lane + 64 * q, u.x, a.out_dtype, a.clamp_float);
      rs_store<TOut>(stage, lane + 64 * q + 32, u.y, a.out_dtype, a.clamp_float);
    }
    __syncwarp();
    rs_flush<TOut>(out, a.out_sw, a.out_vec4, stage, nc, lane, a.out_dtype);
    __syncwarp();
  }
}

template <int BMODE, class TIn, class TOut, int FORM>
__global__ void __launch_bounds__(RS_THREADS, 3)
    resample_tiled_kernel(const __grid_constant__ ResampleArgs a, float eps, float beta) {
  using SH = RsShared<FORM>;
  __shared__ SH sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)a.n, m = (int)a.m;
  const int tc = a.tile_cols, tr = RS_WARPS * a.warp_rows;
  const int c0 = (int)blockIdx.x * tc, r0 = (int)blockIdx.y * tr;
  const int64_t plane = blockIdx.z;
  const int nc = min((int)a.m_out - c0, tc);
  const int nr = min((int)a.n_out - r0, tr);
  // every output column's and row's cell and offset; the first and last of
  // them bound the input window
  for (int c = tid; c < nc; c += RS_THREADS)
    grid_pos(c0 + c, m, (int)a.m_out, a.div_x, sh.col_j[c], sh.col_t[c]);
  if (tid < nr) {
    float t;
    grid_pos(r0 + tid, n, (int)a.n_out, a.div_y, sh.row_i[tid], t);
    const float C0 = pos_c0(t), h = pos_h(t);
    sh.row_a[tid] = make_float4(t, t, C0, C0);
    sh.row_h[tid] = make_float2(h, h);
  }
  __syncthreads();
  const int kfirst = sh.col_j[0] - 1, in_base = sh.row_i[0] - 1;
  const int wc = sh.col_j[nc - 1] + 2 - kfirst + 1;  // <= the form's window (host)
  const int wr = sh.row_i[nr - 1] + 2 - in_base + 1; // <= RS_MAX_IN (host)
  const int esz = elem_bytes<TIn>(a.in_dtype);
  for (int r = tid; r < wr; r += RS_THREADS)
    sh.in_off[r] = (int64_t)clamp_idx(in_base + r, n) * a.in_sh * esz;
  if (FORM == RS_CELLS) {
    for (int c = tid; c < nc; c += RS_THREADS)
      if (c == 0 || sh.col_j[c] != sh.col_j[c - 1]) sh.start[sh.col_j[c] - 1 - kfirst] = c;
    if (tid == 0) sh.start[wc - 3] = nc;
  }
  __syncthreads();
  const int q0 = warp * a.warp_rows;
  const int nq = min(nr - q0, a.warp_rows);
  if (nq <= 0) return;
  const char* in_plane = static_cast<const char*>(a.in) + plane * a.in_sc * esz;
  // lane q holds the cell of row q, counted from the first row's
  const int rel = lane < nq ? sh.row_i[q0 + lane] - sh.row_i[q0] : -1;
  const int rows_in = __shfl_sync(0xffffffffu, rel, nq - 1) + 4;
  uint32_t rows_of = rel >= 0 ? 1u << (4 * rel) : 0u;
  rows_of = __reduce_add_sync(0xffffffffu, rows_of);
  for (int k0 = 0; k0 < wc; k0 += 64)
    column_pass<BMODE, TIn>(a, sh, warp, lane, q0, rows_in, rows_of, in_base, kfirst, wc, k0, in_plane, esz, eps,
                            beta);
  __syncwarp();
  const int osz = elem_bytes<TOut>(a.out_dtype);
  char* out = static_cast<char*>(a.out) +
              (plane * a.out_sc + (int64_t)(r0 + q0) * a.out_sh + (int64_t)c0 * a.out_sw) * osz;
  const int64_t row_bytes = a.out_sh * osz;
  if constexpr (FORM == RS_CELLS) {
    const int cells = wc - 3;
    int most = 0;  // outputs of the fullest cell
    for (int k = lane; k < cells; k += 32) most = max(most, sh.start[k + 1] - sh.start[k]);
    most = __reduce_max_sync(0xffffffffu, most);
    if (most <= 2)
      row_pass_up<BMODE, TOut, 2>(a, sh, warp, lane, nq, nc, cells, most, out, row_bytes, eps, beta);
    else if (most == 3)
      row_pass_up<BMODE, TOut, 3>(a, sh, warp, lane, nq, nc, cells, most, out, row_bytes, eps, beta);
    else
      row_pass_up<BMODE, TOut, 4>(a, sh, warp, lane, nq, nc, cells, most, out, row_bytes, eps, beta);
  } else {
    row_pass_outputs<BMODE, TOut>(a, sh, warp, lane, nq, nc, kfirst, out, row_bytes, eps, beta);
  }
}

template <int BMODE, class TIn, class TOut>
cudaError_t launch_form(const ResampleArgs& a, float eps, float beta, cudaStream_t stream) {
  if (a.form == RS_DIRECT) {
    const dim3 block(32, 8);
    const dim3 grid((unsigned)((a.m_out + 31) / 32), (unsigned)((a.n_out + 7) / 8),
                    (unsigned)a.planes);
    resample_kernel<BMODE, TIn, TOut><<<grid, block, 0, stream>>>(a, eps, beta);
    return cudaGetLastError();
  }
  if (a.form == RS_LINES) {
    const bool along_x = a.m == 1 && a.n > 1;
    const int64_t bx = a.tile_cols, by = 256 / bx, span = a.warp_rows;
    const int64_t cols = bx * (along_x ? span : 1), rows = by * (along_x ? 1 : span);
    const dim3 grid((unsigned)((a.m_out + cols - 1) / cols), (unsigned)((a.n_out + rows - 1) / rows),
                    (unsigned)a.planes);
    resample_lines_kernel<BMODE, TIn, TOut>
        <<<grid, dim3((unsigned)bx, (unsigned)by), 0, stream>>>(a, eps, beta, (int)span);
    return cudaGetLastError();
  }
  const int tr = RS_WARPS * a.warp_rows;
  const dim3 grid((unsigned)((a.m_out + a.tile_cols - 1) / a.tile_cols),
                  (unsigned)((a.n_out + tr - 1) / tr), (unsigned)a.planes);
  if (a.form == RS_CELLS)
    resample_tiled_kernel<BMODE, TIn, TOut, RS_CELLS><<<grid, RS_THREADS, 0, stream>>>(a, eps, beta);
  else if (a.form == RS_OUTPUTS)
    resample_tiled_kernel<BMODE, TIn, TOut, RS_OUTPUTS><<<grid, RS_THREADS, 0, stream>>>(a, eps, beta);
  else
    resample_tiled_kernel<BMODE, TIn, TOut, RS_REDUCED><<<grid, RS_THREADS, 0, stream>>>(a, eps, beta);
  return cudaGetLastError();
}

template <class TIn, class TOut>
cudaError_t launch_beta(const ResampleArgs& a, float eps, float beta, int bmode,
                              cudaStream_t stream) {
  switch (bmode) {
    case B2: return launch_form<B2, TIn, TOut>(a, eps, beta, stream);
    case B2R: return launch_form<B2R, TIn, TOut>(a, eps, beta, stream);
    case B0: return launch_form<B0, TIn, TOut>(a, eps, beta, stream);
    default: return launch_form<BGEN, TIn, TOut>(a, eps, beta, stream);
  }
}

}  // namespace

static int resample_sms() {
  static std::atomic<int> known[64];
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  v = known[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 152;
  known[dev].store(v, std::memory_order_relaxed);
  return v;
}

static AxisDiv axis_div(int64_t n, int64_t n_out) {
  AxisDiv d{1u, 0, 0, 0, 0.f, 0.0};
  if (n <= 1 || n_out <= 1) return d;
  const uint64_t den = (uint64_t)(n_out - 1);
  d.inv64 = 1.0 / (double)den;
  d.inv = (float)d.inv64;
  // the largest numerator is (n_out - 1)(n - 1)
  if (den >= (1ull << 32) || (uint64_t)(n - 1) >= (1ull << 32) ||
      den * (uint64_t)(n - 1) >= (1ull << 32))
    return d;
  int l = 0;
  while ((1ull << l) < den) ++l;
  d.mag = (uint32_t)(((1ull << 32) * ((1ull << l) - den)) / den + 1);
  d.sh1 = l < 1 ? l : 1;
  d.sh2 = l > 1 ? l - 1 : 0;
  d.fast = 1;
  return d;
}

cudaError_t launch_resample(const ResampleArgs& a_in, float eps, float beta, int bmode,
                            cudaStream_t stream) {
  ResampleArgs a = a_in;
  a.div_y = axis_div(a.n, a.n_out);
  a.div_x = axis_div(a.m, a.m_out);
  const RsPlan plan = rs_plan(
      RsShape{a.n, a.m, a.planes, a.n_out, a.m_out,
              a.out_dtype == DT_U8 ? 1 : (a.out_dtype == DT_F32 ? 4 : 2)},
      resample_sms());
  a.form = plan.form;
  a.tile_cols = plan.cols;
  a.warp_rows = plan.rows;
  const int i = a.in_dtype, o = a.out_dtype;
  if (i == DT_U8 && o == DT_U8) return launch_beta<uint8_t, uint8_t>(a, eps, beta, bmode, stream);
  if (i == DT_F16 && o == DT_F16) return launch_beta<__half, __half>(a, eps, beta, bmode, stream);
  if (i == DT_BF16 && o == DT_BF16)
    return launch_beta<__nv_bfloat16, __nv_bfloat16>(a, eps, beta, bmode, stream);
  if (i == DT_F32 && o == DT_F32) return launch_beta<float, float>(a, eps, beta, bmode, stream);
  if (i == DT_U8 && o == DT_F32) return launch_beta<uint8_t, float>(a, eps, beta, bmode, stream);
  if (i == DT_F32 && o == DT_U8) return launch_beta<float, uint8_t>(a, eps, beta, bmode, stream);
  return launch_beta<Dyn, Dyn>(a, eps, beta, bmode, stream);
}

}  // namespace wdweno
