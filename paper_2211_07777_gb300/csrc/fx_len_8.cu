// Fixed-point passes of the lengths of FX_SHARD_8.
#include "fx_kernels.cuh"

FX_UNIT(8)
