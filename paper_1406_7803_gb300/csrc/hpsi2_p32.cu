// hpsi2_p32.cu -- float instantiations of the plane pass (hpsi2_p.cuh).
#include "hpsi2_p.cuh"

namespace fde {

template bool two_step_grid<float>(const GridDims&, const SphereDev&);
template int plane_group<float>(const GridDims&, const HpsiItemDesc<float>*, int, int);
template cudaError_t launch_plane_pass<float>(const GridDims&, unsigned, const HpsiBatch<float>&, const FftPlans<float>&,
                                             cudaStream_t);
template cudaError_t launch_plane_density<float>(const GridDims&, const cplx<float>*, const SphereDev&, int, const double*,
                                                double*, double*, int, const FftPlans<float>&, cudaStream_t);

}  // namespace fde
