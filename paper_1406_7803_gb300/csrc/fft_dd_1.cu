// fft_dd_1.cu -- double-float axis passes of one group of lengths (fft_dd.cuh).
#define FDE_DD_SIDES FDE_PLANE_SIDES1
#define FDE_DD_LINES FDE_SPLIT_SIDES1
#define FDE_DD_AXIS dd_axis_1
#include "fft_dd.cuh"
