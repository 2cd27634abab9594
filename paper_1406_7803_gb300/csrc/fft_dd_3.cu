// fft_dd_3.cu -- double-float axis passes of one group of lengths (fft_dd.cuh).
#define FDE_DD_SIDES FDE_PLANE_SIDES3
#define FDE_DD_LINES FDE_SPLIT_SIDES3
#define FDE_DD_AXIS dd_axis_3
#include "fft_dd.cuh"
