// hpsi2_p64.cu -- double instantiations of the plane pass (hpsi2_p.cuh).
#include "hpsi2_p.cuh"

namespace fde {

template bool two_step_grid<double>(const GridDims&, const SphereDev&);
template int plane_group<double>(const GridDims&, const HpsiItemDesc<double>*, int, int);
template cudaError_t launch_plane_pass<double>(const GridDims&, unsigned, const HpsiBatch<double>&, const FftPlans<double>&,
                                             cudaStream_t);
template cudaError_t launch_plane_density<double>(const GridDims&, const cplx<double>*, const SphereDev&, int, const double*,
                                                double*, double*, int, const FftPlans<double>&, cudaStream_t);

}  // namespace fde
