// Fixed-point passes of the lengths of FX_SHARD_5.
#include "fx_kernels.cuh"

FX_UNIT(5)
