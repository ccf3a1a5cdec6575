// FP32 lane-pair passes of the lengths of FX_SHARD_5.
#include "f2_kernels.cuh"

F2_UNIT(5)
