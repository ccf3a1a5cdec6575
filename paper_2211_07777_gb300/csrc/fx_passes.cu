// Dispatch of the fixed-point passes to the translation unit of their length.
#include <cuda_runtime.h>

#include "fx_plan.cuh"
#include "passes.cuh"

namespace flups {

#define FX_DECL(i)                                                                                             \
  cudaError_t launch_fx_##i(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st); \
  cudaError_t limit_fx_##i(int kind, int P);
FX_DECL(0)
FX_DECL(1)
FX_DECL(2)
FX_DECL(3)
FX_DECL(4)
FX_DECL(5)
FX_DECL(6)
FX_DECL(7)
FX_DECL(8)
FX_DECL(9)
FX_DECL(10)
FX_DECL(11)

cudaError_t launch_fx(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
  switch (p.P) {
#define FX_CASE(P) case P:
    FX_SHARD_0(FX_CASE) return launch_fx_0(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_1(FX_CASE) return launch_fx_1(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_2(FX_CASE) return launch_fx_2(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_3(FX_CASE) return launch_fx_3(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_4(FX_CASE) return launch_fx_4(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_5(FX_CASE) return launch_fx_5(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_6(FX_CASE) return launch_fx_6(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_7(FX_CASE) return launch_fx_7(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_8(FX_CASE) return launch_fx_8(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_9(FX_CASE) return launch_fx_9(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_10(FX_CASE) return launch_fx_10(kind, p, grid, nthr, smem, st);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_11(FX_CASE) return launch_fx_11(kind, p, grid, nthr, smem, st);
#undef FX_CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t limit_fx(int kind, int P) {
  switch (P) {
#define FX_CASE(P) case P:
    FX_SHARD_0(FX_CASE) return limit_fx_0(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_1(FX_CASE) return limit_fx_1(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_2(FX_CASE) return limit_fx_2(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_3(FX_CASE) return limit_fx_3(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_4(FX_CASE) return limit_fx_4(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_5(FX_CASE) return limit_fx_5(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_6(FX_CASE) return limit_fx_6(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_7(FX_CASE) return limit_fx_7(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_8(FX_CASE) return limit_fx_8(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_9(FX_CASE) return limit_fx_9(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_10(FX_CASE) return limit_fx_10(kind, P);
#undef FX_CASE
#define FX_CASE(P) case P:
    FX_SHARD_11(FX_CASE) return limit_fx_11(kind, P);
#undef FX_CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace flups
