// How a resampling call runs, from its sizes and output type alone: kernel form,
// tile and rows.  Host code in a header of its own, so that every plan's bounds can be
// checked on the CPU.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace wdweno {

// Three forms of the tiled kernel, one thread per output, and one per line of
// outputs (wd_resample.cu).
enum RsForm { RS_REDUCED = 0, RS_CELLS = 1, RS_OUTPUTS = 2, RS_DIRECT = 3, RS_LINES = 4 };

constexpr int RS_WARPS = 8;
constexpr int RS_MAX_ROWS = 8;                 // output rows per warp, at most
constexpr int RS_DOWN_ROWS = 4;                // the same, where the rows are reduced
constexpr int RS_MAX_CELLS = 8;                // input cells a warp's rows span, at most
constexpr int RS_PRE = RS_MAX_CELLS + 3;       // input rows
constexpr int RS_TC_DOWN = 128;                // output columns of a tile, at most
constexpr int RS_TC_MAX = 480;                 // the same, RS_CELLS
constexpr int RS_WC_UP = 64;                   // window columns, RS_CELLS
constexpr int RS_WC_DOWN = 2 * RS_TC_DOWN + 8; // RS_REDUCED (>= 2 (RS_TC_DOWN - 1) + 5)
constexpr int RS_WC_OUT = 128;                 // RS_OUTPUTS
constexpr int RS_MAX_IN = 2 * RS_WARPS * RS_DOWN_ROWS + 8;  // input rows of a tile, at most

struct RsShape {
  int64_t n, m, planes;  // input rows, columns, channels
  int64_t n_out, m_out;  // output rows, columns
  int out_bytes;         // of an output element
};

struct RsPlan {
  int form;
  int cols;      // output columns of a tile (RS_LINES: of a block)
  int rows;      // output rows per warp (RS_LINES: outputs per thread)
  int64_t ctas;  // of the tiled kernel, with at least two rows per warp
};

// Tile of a form: output columns, as many as its window serves (a span of d
// input spacings touches at most ceil(d) + 4 samples) in whole words, and rows
// per warp.  Each warp loads 3 rows more than its cells, so more rows cost less
// as long as about every SM gets a CTA (reduced rows: three in four SMs, as
// halving 4 rows there doubles the halo's share).  Magnified rows go down to 2
// while three CTAs an SM, the most that fit, still hold them all, which shortens
// every CTA's chain: 200x300 -> 800x1200 9.5 -> 8.3 us, 100x1000 -> 800x8000
// 14.0 -> 11.8.
inline RsPlan rs_plan_tile(const RsShape& s, int form, int sms) {
  int64_t tc = RS_TC_DOWN;
  if (form != RS_REDUCED && s.m_out > 1) {
    const int64_t span = (form == RS_CELLS ? RS_WC_UP : RS_WC_OUT) - 4;
    tc = span * (s.m_out - 1) / (s.m - 1) + 1;
    tc = std::min<int64_t>(tc, form == RS_CELLS ? RS_TC_MAX : RS_TC_DOWN) & ~int64_t(3);
  }
  const bool up = s.n_out >= s.n;
  const int64_t strips = (s.m_out + tc - 1) / tc * s.planes;
  auto count = [&](int rows) {
    return strips * ((s.n_out + RS_WARPS * rows - 1) / (RS_WARPS * rows));
  };
  int rows = up && form != RS_REDUCED ? RS_MAX_ROWS : RS_DOWN_ROWS;
  while (rows > 2 && RS_WARPS * (rows / 2) >= s.n_out) rows >>= 1;  // (no warp without rows)
  while (rows > 1 && (count(rows) < (up ? sms : 3 * sms / 4) ||
                      (up && rows > 2 && count(rows / 2) <= 3 * sms)))
    rows >>= 1;
  return RsPlan{form, (int)tc, rows, count(std::max(rows, 2))};
}

// Lines of outputs: a block's columns, and outputs per thread, more than one
// once there are threads enough for every SM.
inline RsPlan rs_plan_lines(const RsShape& s, int sms) {
  const bool along_x = s.m == 1 && s.n > 1;
  int cols = 1;
  while (cols < (along_x ? 32 : 256) && cols < s.m_out) cols *= 2;
  const int64_t by = 256 / cols;
  const double outputs = double(s.m_out) * double(s.n_out) * double(s.planes);
  int64_t span = std::max<int64_t>(1, int64_t(std::min(8.0, outputs / (1024.0 * sms))));
  // (blocks along y fit the grid; along_x there are eight rows a block)
  if (!along_x) span = std::max<int64_t>(span, (s.n_out + 65535 * by - 1) / (65535 * by));
  return RsPlan{RS_LINES, cols, (int)span, 0};
}

inline RsPlan rs_plan(const RsShape& s, int sms) {
  const int64_t dx = s.m - 1, dx_out = s.m_out - 1, dy = s.n - 1, dy_out = s.n_out - 1;
  // spacing ratios beyond 2: little to share between neighbouring outputs
  if ((dx_out > 0 && 2 * dx_out < dx) || (dy_out > 0 && 2 * dy_out < dy))
    return RsPlan{RS_DIRECT, 0, 0, 0};
  if (s.n == 1 || s.m == 1 || s.n_out < RS_WARPS) return rs_plan_lines(s, sms);
  if (s.m_out < s.m) {
    // Reduced columns: 128 outputs with the window they need, or, where the rows
    // are magnified or the columns reduced by less than 1.12, the outputs of 128
    // window columns (eight rows a warp where they are magnified, and two column
    // passes in place of three).  540x960 -> 1080x900 16.2 -> 11.3 us, 222x987 ->
    // 206x914 8.2 -> 6.8; but 2160x3840 -> 1270x2258 47.5 against 53.6 by outputs.
    const bool near = 100 * dx < 112 * dx_out;
    return rs_plan_tile(s, s.n_out >= s.n || near ? RS_OUTPUTS : RS_REDUCED, sms);
  }
  // A few rows of magnified columns: a tile is little work, so few tiles
  // (8x200000 -> 8x300000 33 -> 20 us).
  if (dx_out < 2 * dx && s.n_out <= 2 * RS_WARPS) return rs_plan_tile(s, RS_OUTPUTS, sms);
  const RsPlan c = rs_plan_tile(s, RS_CELLS, sms), o = rs_plan_tile(s, RS_OUTPUTS, sms);
  const int64_t c_strips = (s.m_out + c.cols - 1) / c.cols;
  const int64_t o_strips = (s.m_out + o.cols - 1) / o.cols;
  if (2 * dx_out < 5 * dx) {
    // Magnified less than 2.5 times: by cells (540x960 -> 1080x1920 14.4 us, 18.8 by
    // outputs), but at about the same spacing 64 window columns serve no more
    // outputs, and tiles by outputs are twice as wide (540x960 -> 600x1000 10.7 ->
    // 8.2 us).
    const bool by_outputs =
        100 * dx_out < 115 * dx && s.n_out >= s.n && 8 * o_strips < 5 * c_strips;
    return by_outputs ? o : c;
  }
  // Magnified more.  By cells, pass 2 of a row costs a strip 4 units and one per
  // output of a cell, or a quarter of one per lane whose output meets in the same
  // shared-memory bank; by outputs, 5 units 128 columns, 5.5 in FP32.  Below some two
  // CTAs an SM either costs more.  (Fitted to 3x to 64x of 8x8 to 1080x1920, three
  // types.)  A strip by cells is 480 outputs at most, so from 8x on it has fewer
  // and fewer cells for its 64 places: us by cells and by outputs, 540x960 uint8 4x
  // 35 and 43, 8x 112 and 159, 12x 311 and 349, 16x 800 and 614; 64x64 8x 6.3 and 4.9,
  // 16x 12.5 and 8.6, 64x 356 and 85; 3x3 -> 4000x4000 949 and 30.
  const int64_t f = (2 * dx_out + dx) / (2 * dx);  // outputs per cell
  int64_t banks = 1;                               // gcd(words from cell to cell, 32)
  if (f * s.out_bytes % 4 == 0)
    while (banks < 32 && (f * s.out_bytes / 4) % (2 * banks) == 0) banks *= 2;
  auto idle = [&](int64_t ctas) {
    return double(std::max<int64_t>(ctas, 21 * sms / 10)) / double(ctas);
  };
  const double by_cells =
      double(c_strips * (4 + f * std::max<int64_t>(1, banks / 4))) * idle(c.ctas);
  const double by_outputs = double(o_strips) * (s.out_bytes == 4 ? 5.5 : 5.0) * idle(o.ctas);
  return by_outputs <= by_cells ? o : c;
}

}  // namespace wdweno
