// Window arithmetic of the tiled resampling kernel, in a header of its own so
// that it can be checked on the host at widths no test image has.  Sides go up
// to 2^31 - 1: sums of an index and a window's length, and byte offsets of a
// column, do not fit 32 bits there.
#pragma once

#include <stdint.h>

#include "wd_hd.h"

namespace wdweno {

// Whether window columns kfirst + k0 .. + 63 and input rows first - 1 ..
// first - 2 + rows_in all lie inside an n x m image, so that nothing is clamped.
WD_HD bool window_inside(int kfirst, int k0, int m, int first, int rows_in, int n) {
  return kfirst >= 0 && kfirst <= m - 64 - k0 && first >= 1 && first - 1 <= n - rows_in;
}

// Byte offset of window column k (relative to kfirst) of a row with unit
// column stride.
WD_HD int64_t column_bytes(int kfirst, int k, int esz) { return ((int64_t)kfirst + k) * esz; }

}  // namespace wdweno
