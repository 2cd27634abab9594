// fft_dd_5.cu -- double-float axis passes of one group of lengths (fft_dd.cuh).
#define FDE_DD_SIDES FDE_NO_SIDES
#define FDE_DD_LINES FDE_SPLIT_LONG1
#define FDE_DD_AXIS dd_axis_5
#include "fft_dd.cuh"
