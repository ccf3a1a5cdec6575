// FP32 lane-pair passes of the lengths of FX_SHARD_10.
#include "f2_kernels.cuh"

F2_UNIT(10)
