// hpsi2_z32.cu -- float instantiations of the z passes (hpsi2_z.cuh).
#include "hpsi2_z.cuh"

namespace fde {

template void launch_zinv_cols<float>(int, unsigned, const HpsiBatch<float>&, const cplx<float>*, cudaStream_t);
template void launch_zfwd_cols<float>(int, unsigned, const HpsiBatch<float>&, float, const cplx<float>*, cudaStream_t);

}  // namespace fde
