// Dispatch of the FP32 lane-pair passes to the translation unit of their length.
#include <cuda_runtime.h>

#include "fx_plan.cuh"
#include "passes.cuh"

namespace flups {

#define F2_DECL(i)                                                                                             \
  cudaError_t launch_f2_##i(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st); \
  cudaError_t limit_f2_##i(int kind, int P);
F2_DECL(0)
F2_DECL(1)
F2_DECL(2)
F2_DECL(3)
F2_DECL(4)
F2_DECL(5)
F2_DECL(6)
F2_DECL(7)
F2_DECL(8)
F2_DECL(9)
F2_DECL(10)
F2_DECL(11)

cudaError_t launch_f2(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
  switch (p.P) {
#define F2_CASE(P) case P:
    FX_SHARD_0(F2_CASE) return launch_f2_0(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_1(F2_CASE) return launch_f2_1(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_2(F2_CASE) return launch_f2_2(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_3(F2_CASE) return launch_f2_3(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_4(F2_CASE) return launch_f2_4(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_5(F2_CASE) return launch_f2_5(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_6(F2_CASE) return launch_f2_6(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_7(F2_CASE) return launch_f2_7(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_8(F2_CASE) return launch_f2_8(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_9(F2_CASE) return launch_f2_9(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_10(F2_CASE) return launch_f2_10(kind, p, grid, nthr, smem, st);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_11(F2_CASE) return launch_f2_11(kind, p, grid, nthr, smem, st);
#undef F2_CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t limit_f2(int kind, int P) {
  switch (P) {
#define F2_CASE(P) case P:
    FX_SHARD_0(F2_CASE) return limit_f2_0(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_1(F2_CASE) return limit_f2_1(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_2(F2_CASE) return limit_f2_2(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_3(F2_CASE) return limit_f2_3(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_4(F2_CASE) return limit_f2_4(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_5(F2_CASE) return limit_f2_5(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_6(F2_CASE) return limit_f2_6(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_7(F2_CASE) return limit_f2_7(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_8(F2_CASE) return limit_f2_8(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_9(F2_CASE) return limit_f2_9(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_10(F2_CASE) return limit_f2_10(kind, P);
#undef F2_CASE
#define F2_CASE(P) case P:
    FX_SHARD_11(F2_CASE) return limit_f2_11(kind, P);
#undef F2_CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace flups
