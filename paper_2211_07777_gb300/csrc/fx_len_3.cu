// Fixed-point passes of the lengths of FX_SHARD_3.
#include "fx_kernels.cuh"

FX_UNIT(3)
