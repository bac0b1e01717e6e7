// Fixed-point plane-phase kernels of one group of transform lengths.
#include "tc_fx_kernels.cuh"

FX_INSTANTIATE(c, FX_LENGTHS_C)
