// Fixed-point plane-phase kernels of one group of transform lengths.
#include "tc_fx_kernels.cuh"

FX_INSTANTIATE(a, FX_LENGTHS_A)
