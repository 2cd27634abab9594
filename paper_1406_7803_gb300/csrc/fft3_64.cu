// fft3_64.cu -- double grids' 3D transforms (fft3.cuh).
#include "fft3.cuh"

namespace fde {

namespace {
FDE_AXIS_LAUNCHERS(FDE_PLANE_SIDES, FDE_SPLIT_LINES)
}

template <>
bool launch_fft3d_two_step<double>(cplx<double>* data, const GridDims& g, const FftPlans<double>& fp, int sign, cudaStream_t st) {
  if (!grid_ok(g)) return false;
  ProfScope prof_("k_fft_axis_f64", st);
  const long long nr = (long long)g.n1 * g.n2 * g.n3;
  contig_axis<double, AsIs, AsIs>(g.n3, nr / g.n3, data, fp.p3.tw, sign, st);
  strided_axis<double, AsIs, AsIs>(g.n2, nr / g.n2, g.n3, data, data, fp.p2.tw, sign, st);
  strided_axis<double, AsIs, AsIs>(g.n1, nr / g.n1, g.n2 * g.n3, data, data, fp.p1.tw, sign, st);
  return true;
}

}  // namespace fde
