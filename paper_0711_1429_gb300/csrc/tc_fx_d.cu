// Fixed-point plane-phase kernels of one group of transform lengths.
#include "tc_fx_kernels.cuh"

FX_INSTANTIATE(d, FX_LENGTHS_D)
