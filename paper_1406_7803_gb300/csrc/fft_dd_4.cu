// fft_dd_4.cu -- double-float axis passes of one group of lengths (fft_dd.cuh).
#define FDE_DD_SIDES FDE_NO_SIDES
#define FDE_DD_LINES FDE_SPLIT_LONG0
#define FDE_DD_AXIS dd_axis_4
#include "fft_dd.cuh"
