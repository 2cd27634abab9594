// hpsi2_z.cuh -- launches of the z passes (hpsi2.cuh) for every two-step length.
#pragma once

#include "hpsi2.cuh"

namespace fde {

template <typename T>
void launch_zinv_cols(int n3, unsigned blocks, const HpsiBatch<T>& B, const cplx<T>* tw, cudaStream_t st) {
  switch (n3) {
#define FDE_CASE(N, R1, R2)                                                        \
  case N:                                                                          \
    count_launches(1);                                                             \
    k_zinv_cols<T, R1, R2><<<blocks, z_threads<T, R1, R2>(), 0, st>>>(B, tw);     \
    break;
    FDE_SPLIT_LINES(FDE_CASE)
#undef FDE_CASE
  }
}
template <typename T>
void launch_zfwd_cols(int n3, unsigned blocks, const HpsiBatch<T>& B, T inv_nr, const cplx<T>* tw, cudaStream_t st) {
  switch (n3) {
#define FDE_CASE(N, R1, R2)                                                               \
  case N:                                                                                 \
    count_launches(1);                                                                    \
    k_zfwd_cols<T, R1, R2><<<blocks, z_threads<T, R1, R2>(), 0, st>>>(B, inv_nr, tw);    \
    break;
    FDE_SPLIT_LINES(FDE_CASE)
#undef FDE_CASE
  }
}

}  // namespace fde
