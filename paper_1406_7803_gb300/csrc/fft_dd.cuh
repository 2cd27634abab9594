// fft_dd.cuh -- the double-float axis passes of one group of lengths (fft2.cuh): the strided y pass
// (split values in and out), the strided x pass (joined into FP64 on the way out, or the high parts
// alone into an FP32 grid) and the contiguous z pass (split on the way in).  A translation unit defines FDE_DD_SIDES, FDE_DD_LINES
// and FDE_DD_AXIS, the name of its entry point.
#pragma once

#include "fft3.cuh"

#define FDE_NO_SIDES(X)

namespace fde {

namespace {
FDE_AXIS_LAUNCHERS(FDE_DD_SIDES, FDE_DD_LINES)
}

// axis 3: z, 2: y, 1: x (FP64 in place), 0: x with the high parts into `out` (FP32); false when n is not
// of this group.
bool FDE_DD_AXIS(int axis, int n, long long nlines, int stride, void* data, void* out, const ddc* tw, int sign,
                 cudaStream_t st) {
  if (axis == 3) return contig_axis<dd, AsF64, AsIs>(n, nlines, data, tw, sign, st);
  if (axis == 2) return strided_axis<dd, AsIs, AsIs>(n, nlines, stride, data, data, tw, sign, st);
  if (axis == 1) return strided_axis<dd, AsIs, AsF64>(n, nlines, stride, data, data, tw, sign, st);
  return strided_axis<dd, AsIs, AsHigh>(n, nlines, stride, data, out, tw, sign, st);
}

}  // namespace fde
