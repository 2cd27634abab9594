// hpsi2_z64.cu -- double instantiations of the z passes (hpsi2_z.cuh).
#include "hpsi2_z.cuh"

namespace fde {

template void launch_zinv_cols<double>(int, unsigned, const HpsiBatch<double>&, const cplx<double>*, cudaStream_t);
template void launch_zfwd_cols<double>(int, unsigned, const HpsiBatch<double>&, double, const cplx<double>*, cudaStream_t);

}  // namespace fde
