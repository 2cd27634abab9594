// fft_dd.cu -- full-grid 3D transforms of FP64 grids in double-float arithmetic (dd.cuh).
//
// The two-step axis passes (fft3.cuh) on the double-float type: each value is two floats, so the
// arithmetic runs on the FP32 pipes (64x the FP64 rate on this part) at about 48 significant
// bits.  The first axis pass reads the FP64 grid and splits each value, the middle pass keeps the
// split form in global memory (the same 16 bytes per complex value), and the last pass adds the
// parts back into FP64 -- or, for values that are used in FP32 alone (the gradients of the pointwise
// functionals), writes the high parts to an FP32 grid: an FP64 addition a value and half the traffic less.
#include "fft3.cuh"

namespace fde {

using DdAxis = bool(int axis, int n, long long nlines, int stride, void* data, void* out, const ddc* tw, int sign,
                    cudaStream_t st);
DdAxis dd_axis_0, dd_axis_1, dd_axis_2, dd_axis_3, dd_axis_4, dd_axis_5;

bool launch_fft3d_dd(double2* data, const GridDims& g, const FftPlans<dd>& fp, int sign, cudaStream_t st,
                     float2* high) {
  if (!grid_ok(g)) return false;
  ProfScope prof_("k_fft_axis_dd", st);
  const long long nr = (long long)g.n1 * g.n2 * g.n3;
  DdAxis* const groups[] = {dd_axis_0, dd_axis_1, dd_axis_2, dd_axis_3, dd_axis_4, dd_axis_5};
  const auto pass = [&](int axis, int n, int stride, const ddc* tw) {
    for (DdAxis* f : groups)
      if (f(axis, n, nr / n, stride, data, high, tw, sign, st)) return;
  };
  pass(3, g.n3, 1, fp.p3.tw);
  pass(2, g.n2, g.n3, fp.p2.tw);
  pass(high ? 0 : 1, g.n1, g.n2 * g.n3, fp.p1.tw);
  return true;
}

}  // namespace fde
