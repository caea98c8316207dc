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
// the sweep is a serial chain: 3x48x64 uint8 14.0 -> 6.2 us (rows 16 -> 3),
// 3x256x256 FP32 15.2 -> 9.2 us, 1x300x700 FP16 14.4 -> 8.3 us, 3x512x512
// 17.9 -> 15.9 us; from 1024x1024 on the plans are those of the rule before
// (two-column strips, bands balancing the waves), or 182-column strips.
#pragma once

#include <stdint.h>

namespace wdweno {

struct FwdShape {
  int threads, cols;  // CTA
  int per_sm;         // CTAs resident per SM
  float lat, issue;   // us
};

constexpr float FWD_FILL = 6.3f;    // steps
constexpr float FWD_LAUNCH = 2.2f;  // us

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

}  // namespace wdweno
