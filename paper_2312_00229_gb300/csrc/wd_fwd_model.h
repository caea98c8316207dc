// Time model of the forward tiles, shared by the one-launch plan (host) and
// the batched launch's setup kernel (device).
//
// A CTA sweeps its band of `rows` coarse rows in rows + FILL steps (the halo
// and the pipeline's fill count FILL: idle stages make them shorter).  One
// step takes, with k CTAs of a shape on an SM, sqrt(lat^2 + (k issue)^2): the
// dependent chain of a step when few CTAs share the SM, the issue slots of
// all of them when many do.  Fitted to 680 launches over 48x64 .. 2160x3840,
// 1 and 3 planes, uint8 to FP32, bands of 3 to 192 rows (rms error 4.4%).
// Bands short enough to fill the GPU in one wave pay on small images, where
// the sweep is a serial chain: 3x48x64 uint8 14.0 -> 5.9 us (rows 16 -> 3),
// 3x256x256 FP32 15.2 -> 9.2 us, 1x300x700 FP16 14.4 -> 8.3 us, 3x512x512
// 17.9 -> 15.9 us; from 1024x1024 on the plans are those of the rule before
// (two-column strips, bands balancing the waves), or 182-column strips.
#pragma once

#include <math.h>
#include <stdint.h>

#include "wd_hd.h"

namespace wdweno {

struct FwdShape {
  int threads, cols;  // CTA
  int per_sm;         // CTAs resident per SM
  float lat, issue;   // us
};

constexpr float FWD_FILL = 6.3f;  // steps

// Strips of 118, 246, 182, 119 and 247 output columns.  (182 is the library's
// own choice only: it covers 512 columns with 576 thread columns where 118 takes
// 640 and 246 takes 768, 96x512x512 FP32 279 -> 247 us, 3x512x512 uint8 15.9 -> 14.3,
// 3x480x854 18.7 -> 17.9; on a tie 118 is kept, 1-2% faster.)
constexpr FwdShape FWD_SHAPES[5] = {{64, 2, 6, 0.5365f, 0.1250f},
                                    {128, 2, 3, 0.4970f, 0.2580f},
                                    {96, 2, 4, 0.5365f, 0.1915f},
                                    {128, 1, 4, 0.3846f, 0.1481f},
                                    {256, 1, 2, 0.3840f, 0.3031f}};

constexpr int fwd_strip(const FwdShape& s) {
  return s.cols == 2 ? 2 * s.threads - 10 : s.threads - 9;
}

// Tile shape of a one-launch forward: `threads` per CTA, `cols` coarse columns
// per thread (1: 256 or 128 threads, 247 or 119 output columns per strip; 2:
// 128, 96 or 64 threads, 246, 182 or 118) and coarse rows per band.
struct FwdPlan {
  int threads, cols;
  int64_t rows;
};

// The plan with the least modelled time for `planes` planes of n x m samples
// on a GPU of `sms` SMs; threads (with cols) and rows are taken as given where
// they are not 0.
inline FwdPlan fwd_find_plan(int64_t n, int64_t m, int64_t planes, int sms, int threads, int cols,
                             int64_t given_rows) {
  const auto step_us = [](const FwdShape& s, int64_t k) {
    return sqrt(double(s.lat) * s.lat + double(k) * k * s.issue * s.issue);
  };
  FwdPlan best{256, 1, given_rows > 0 ? given_rows : n};
  double best_us = 1e300;
  for (const FwdShape& s : FWD_SHAPES) {
    if (threads != 0 && (s.threads != threads || s.cols != cols)) continue;
    const int64_t base = (m + fwd_strip(s) - 1) / fwd_strip(s) * planes;
    const int64_t slots = (int64_t)sms * s.per_sm;
    const double full = step_us(s, s.per_sm);
    int64_t last = -1;
    for (int64_t bands = 1; bands <= n && bands <= 4096; ++bands) {
      const int64_t rows = given_rows > 0 ? given_rows : (n + bands - 1) / bands;
      if (rows == last) continue;
      // bands below 16 rows only up to two waves of CTAs
      if (bands > 1 && (rows < 2 || (rows < 16 && base * bands > 2 * slots))) break;
      last = rows;
      const int64_t ctas = base * ((n + rows - 1) / rows);
      const int64_t rest = ctas % slots;
      double t = double(ctas / slots) * full;
      if (rest) t += step_us(s, (rest + sms - 1) / sms);
      t *= double(rows < n ? rows : n) + FWD_FILL;
      if (t < best_us - 1e-9) {
        best_us = t;
        best = FwdPlan{s.threads, s.cols, rows};
      }
      if (given_rows > 0) break;
    }
  }
  return best;
}

// ---- the batched launch ---------------------------------------------------------
// Bands below this height are as high as the caller or the choice says; higher
// ones are as even as their count allows (wd_batched_kernel.cuh: even_band).
constexpr int BATCHED_EVEN_FROM = 48;
// Band heights the choice is made from.
constexpr int BATCHED_CANDS = 13;
struct BatchedHeights {
  int rows[BATCHED_CANDS];
};
constexpr BatchedHeights BATCHED_HEIGHTS = {{3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192}};
// Steps of a queue's tile beyond its rows: the fill, the ring clearing, the
// ticket and the descriptor.
constexpr float BATCHED_FILL = 10.f;

// What a band height would cost, summed over images.
struct BatchedCost {
  float tiles, steps, longest;
};

// Adds an image of n rows and `strips` strips (of all planes) in bands of at
// most `rows` rows.
WD_HD void batched_add(BatchedCost& c, int n, float strips, int rows) {
  const int b0 = (n - 1) / rows + 1;
  const int r = rows < BATCHED_EVEN_FROM ? (rows < n ? rows : n) : (n - 1) / b0 + 1;
  const float bands = float((n - 1) / r + 1);
  c.tiles += strips * bands;
  c.steps += strips * (float(n) + bands * BATCHED_FILL);
  c.longest = fmaxf(c.longest, float(r));
}

WD_HD float batched_step_us(const FwdShape& s, float k) {
  return sqrtf(s.lat * s.lat + k * k * s.issue * s.issue);
}

// Modelled time of a queue of such tiles: whole waves of resident CTAs at the
// mean tile's length and a last one as long as the longest tile, with as few
// CTAs an SM as it fills.  (The model before spread the steps evenly over the
// CTAs, which holds for many tiles of mixed lengths; of a few large images of
// one wave and a half it chose heights that start a second wave: 1500x1500
// uint8 137 -> 102 us, 2000x2000 196 -> 129.)
WD_HD float batched_us(const FwdShape& s, int sms, const BatchedCost& c) {
  const float slots = float(sms) * float(s.per_sm);
  const float full = floorf(c.tiles / slots), rest = c.tiles - full * slots;
  const float one = c.longest + BATCHED_FILL;
  float us = full * (c.steps / c.tiles) * batched_step_us(s, float(s.per_sm));
  if (rest > 0.f) us += one * batched_step_us(s, ceilf(rest / float(sms)));
  const float k = fminf(float(s.per_sm), ceilf(c.tiles / float(sms)));
  return fmaxf(us, one * batched_step_us(s, k));
}

}  // namespace wdweno
