// Lengths of the fixed-point passes, their radices, and the translation units that compile them.
#pragma once

namespace flups {

// Lengths and their radices, fewest stages first, then the cheapest split by operations per value and
// threads left idle; equal even radices first and last, whose stores have the widest strides (FxRows).
#define FX_LENGTHS(X) \
  X(4, 2, 2, 2, 1, 1) \
  X(6, 2, 3, 2, 1, 1) \
  X(8, 2, 4, 2, 1, 1) \
  X(9, 2, 3, 3, 1, 1) \
  X(12, 2, 4, 3, 1, 1) \
  X(16, 2, 4, 4, 1, 1) \
  X(18, 2, 6, 3, 1, 1) \
  X(24, 2, 8, 3, 1, 1) \
  X(27, 3, 3, 3, 3, 1) \
  X(32, 2, 8, 4, 1, 1) \
  X(36, 2, 6, 6, 1, 1) \
  X(48, 2, 12, 4, 1, 1) \
  X(54, 2, 9, 6, 1, 1) \
  X(64, 2, 8, 8, 1, 1) \
  X(72, 2, 12, 6, 1, 1) \
  X(81, 2, 9, 9, 1, 1) \
  X(96, 2, 12, 8, 1, 1) \
  X(108, 3, 6, 3, 6, 1) \
  X(128, 2, 16, 8, 1, 1) \
  X(144, 2, 12, 12, 1, 1) \
  X(162, 3, 9, 9, 2, 1) \
  X(192, 2, 16, 12, 1, 1) \
  X(216, 3, 6, 6, 6, 1) \
  X(243, 4, 9, 3, 3, 3) \
  X(256, 2, 16, 16, 1, 1) \
  X(288, 3, 12, 2, 12, 1) \
  X(324, 3, 9, 9, 4, 1) \
  X(384, 3, 16, 8, 3, 1) \
  X(432, 3, 6, 12, 6, 1) \
  X(486, 4, 9, 9, 3, 2) \
  X(512, 3, 8, 8, 8, 1) \
  X(576, 3, 12, 4, 12, 1) \
  X(648, 4, 6, 6, 3, 6) \
  X(729, 3, 9, 9, 9, 1) \
  X(768, 3, 16, 3, 16, 1) \
  X(864, 3, 12, 6, 12, 1) \
  X(972, 4, 9, 9, 4, 3) \
  X(1024, 3, 8, 16, 8, 1) \
  X(1152, 3, 12, 8, 12, 1) \
  X(1296, 4, 6, 6, 6, 6) \
  X(1458, 4, 9, 9, 9, 2) \
  X(1536, 4, 8, 8, 3, 8) \
  X(1728, 3, 12, 12, 12, 1) \
  X(1944, 4, 6, 9, 6, 6) \
  X(2048, 3, 16, 8, 16, 1) \
  X(2187, 4, 9, 9, 9, 3) \
  X(2304, 3, 12, 16, 12, 1) \
  X(2592, 4, 6, 12, 6, 6) \
  X(2916, 4, 9, 9, 9, 4) \
  X(3072, 4, 8, 16, 3, 8) \
  X(3456, 4, 12, 12, 2, 12) \
  X(3888, 4, 6, 12, 9, 6) \
  X(4096, 3, 16, 16, 16, 1)


// The lengths by translation unit (fx_len_<i>.cu), balanced by compile time.
#define FX_SHARD_0(X) X(4) X(12) X(27) X(256) X(1296) X(2187)
#define FX_SHARD_1(X) X(6) X(8) X(81) X(972) X(4096)
#define FX_SHARD_2(X) X(9) X(24) X(162) X(288) X(2304)
#define FX_SHARD_3(X) X(16) X(18) X(384) X(512) X(3072)
#define FX_SHARD_4(X) X(32) X(144) X(1152) X(1458)
#define FX_SHARD_5(X) X(36) X(432) X(864) X(2916)
#define FX_SHARD_6(X) X(48) X(96) X(1536) X(3456)
#define FX_SHARD_7(X) X(54) X(128) X(192) X(3888)
#define FX_SHARD_8(X) X(64) X(324) X(729) X(1728)
#define FX_SHARD_9(X) X(72) X(243) X(1944) X(2048)
#define FX_SHARD_10(X) X(108) X(486) X(1024) X(2592)
#define FX_SHARD_11(X) X(216) X(576) X(648) X(768)

// Words per lane behind the renormalisations: three per direction of a four-stage transform, before and after the
// Green product.
constexpr int kFxSlots = 8;

struct FxPlan {
  int n, r[4];
};
__host__ __device__ constexpr FxPlan fx_plan(int P) {
  switch (P) {
#define FX_ROW(P, n, a, b, c, d) \
  case P: return FxPlan{n, {a, b, c, d}};
    FX_LENGTHS(FX_ROW)
#undef FX_ROW
  }
  return FxPlan{0, {1, 1, 1, 1}};
}
// butterflies of radix R a thread takes: up to 18 values in registers
__host__ __device__ constexpr int fx_nb(int R) { return R == 9 || R == 6 ? 2 : (R == 3 ? 5 : (R > 8 ? 1 : 16 / R)); }
// values per thread that every stage of the plan can take: a block has at least P W / fx_ept(P) threads
__host__ __device__ constexpr int fx_ept(int P) {
  int e = 18;
  for (int s = 0; s < fx_plan(P).n; ++s) {
    const int R = fx_plan(P).r[s], v = R * fx_nb(R);
    if (v < e) e = v;
  }
  return e;
}
// Lanes of a full tile and the stride of its rows: about 2048 complex values per CTA (32 KB, 128-192 threads of up
// to 128 registers, so that four CTAs share an SM), 4096 in the fused complex pass, whose code is the longest:
// warps of one CTA run the same stretch of it and share its instruction fetches (unbounded 128^3 197 -> 186 us,
// 192^3 895 -> 840; the other passes 0-8% slower with 4096, all 10-30% slower with 8192).  At least 4 lanes
// (64 contiguous bytes along x) up to P = 1024.
// FX_CURL: the Biot-Savart pass, which holds three components, about 1024 values each.
enum FxTileClass : int { FX_PLAIN = 0, FX_FUSED_C2C = 1, FX_CURL = 2 };
__host__ __device__ constexpr int fx_width(int cls, int P) {
  int W = 1;
  while (W < 32 && 2 * W * P <= (cls == FX_FUSED_C2C ? 4096 : (cls == FX_CURL ? 1024 : 2048))) W *= 2;
  if (cls == FX_CURL) return W;
  const int wmin = P <= 1024 ? 4 : (P <= 2048 ? 2 : 1);
  return W < wmin ? wmin : W;
}
// Rows of the tile in shared memory (16-byte values, W of them a row).  With 8 lanes a row is one 128-byte
// wavefront of a quarter warp and no access conflicts; with fewer, a quarter warp touches 8 / W consecutive rows
// (contiguous), except in the stores of a transform's first stage, whose rows are R apart: a gap of one row after
// every B = R rows (R even) puts those on different banks.
template <int P, int CLS> struct FxRows {
  static constexpr int W = fx_width(CLS, P);
  static constexpr int B = W < 8 && fx_plan(P).r[0] % 2 == 0 ? fx_plan(P).r[0] : 0;
  static constexpr int size = (P + (B ? (P - 1) / (B ? B : 1) : 0)) * W;
  __host__ __device__ static constexpr int at(int i) { return (B ? i + i / (B ? B : 1) : i) * W; }
  // at(j + r n) = at(j) + at(r n) for every j
  __host__ __device__ static constexpr bool linear(int n) { return !B || n % (B ? B : 1) == 0; }
};
__host__ __device__ constexpr int fx_tile_values(int cls, int P) {
  const int W = fx_width(cls, P), r0 = fx_plan(P).r[0];
  return (P + (W < 8 && r0 % 2 == 0 ? (P - 1) / r0 : 0)) * W;
}
__host__ __device__ constexpr int fx_prod(int P, int s0, int s1) {
  int n = 1;
  for (int s = s0; s < s1; ++s) n *= fx_plan(P).r[s];
  return n;
}

// ---------------------------------------------------------------------------
// Plans of the FP32 lane-pair passes.  Their kernels wait for memory rather than for arithmetic, so a thread takes one
// butterfly of at most 9 values: half the registers of the plans above, twice the warps per SM (unbounded 192^3 447 ->
// 372 us, channel 256^3 338 -> 300).  Lengths that would need a fourth stage keep the plans above (768 points
// 60 us against 80), and so does the Biot-Savart pass, whose three tiles fill the SM (256 points 101 against 130).
// ---------------------------------------------------------------------------
#define F2_LENGTHS(X) \
  X(4, 2, 2, 2, 1, 1, 1) \
  X(6, 2, 3, 2, 1, 1, 1) \
  X(8, 2, 4, 2, 1, 1, 1) \
  X(9, 2, 3, 3, 1, 1, 1) \
  X(12, 2, 4, 3, 1, 1, 1) \
  X(16, 2, 8, 2, 1, 1, 1) \
  X(18, 2, 9, 2, 1, 1, 1) \
  X(24, 2, 8, 3, 1, 1, 1) \
  X(27, 2, 9, 3, 1, 1, 1) \
  X(32, 2, 8, 4, 1, 1, 1) \
  X(36, 2, 6, 6, 1, 1, 1) \
  X(48, 2, 8, 6, 1, 1, 1) \
  X(54, 2, 9, 6, 1, 1, 1) \
  X(64, 2, 8, 8, 1, 1, 1) \
  X(72, 2, 9, 8, 1, 1, 1) \
  X(81, 2, 9, 9, 1, 1, 1) \
  X(96, 3, 8, 4, 3, 1, 1) \
  X(108, 3, 9, 4, 3, 1, 1) \
  X(128, 3, 8, 2, 8, 1, 1) \
  X(144, 3, 9, 8, 2, 1, 1) \
  X(162, 3, 9, 9, 2, 1, 1) \
  X(192, 3, 8, 3, 8, 1, 1) \
  X(216, 3, 6, 6, 6, 1, 1) \
  X(243, 3, 9, 9, 3, 1, 1) \
  X(256, 3, 8, 4, 8, 1, 1) \
  X(288, 3, 9, 8, 4, 1, 1) \
  X(324, 3, 9, 9, 4, 1, 1) \
  X(384, 3, 8, 6, 8, 1, 1) \
  X(432, 3, 9, 8, 6, 1, 1) \
  X(486, 3, 9, 9, 6, 1, 1) \
  X(512, 3, 8, 8, 8, 1, 1) \
  X(576, 3, 8, 9, 8, 1, 1) \
  X(648, 3, 9, 9, 8, 1, 1) \
  X(729, 3, 9, 9, 9, 1, 1) \
  X(768, 3, 16, 3, 16, 1, 1) \
  X(864, 3, 12, 6, 12, 1, 1) \
  X(972, 4, 9, 9, 4, 3, 1) \
  X(1024, 3, 8, 16, 8, 1, 1) \
  X(1152, 3, 12, 8, 12, 1, 1) \
  X(1296, 4, 6, 6, 6, 6, 1) \
  X(1458, 4, 9, 9, 9, 2, 1) \
  X(1536, 4, 8, 8, 3, 8, 1) \
  X(1728, 3, 12, 12, 12, 1, 1) \
  X(1944, 4, 6, 9, 6, 6, 1) \
  X(2048, 3, 16, 8, 16, 1, 1) \
  X(2187, 4, 9, 9, 9, 3, 1) \
  X(2304, 3, 12, 16, 12, 1, 1) \
  X(2592, 4, 9, 9, 8, 4, 1) \
  X(2916, 4, 9, 9, 9, 4, 1) \
  X(3072, 4, 8, 16, 3, 8, 1) \
  X(3456, 4, 12, 12, 2, 12, 1) \
  X(3888, 4, 6, 12, 9, 6, 1) \
  X(4096, 3, 16, 16, 16, 1, 1)

struct F2Plan {
  int n, r[5];
};
__host__ __device__ constexpr F2Plan f2_plan(int P) {
  switch (P) {
#define F2_ROW(P, n, a, b, c, d, e) \
  case P: return F2Plan{n, {a, b, c, d, e}};
    F2_LENGTHS(F2_ROW)
#undef F2_ROW
  }
  return F2Plan{0, {1, 1, 1, 1, 1}};
}
__host__ __device__ constexpr F2Plan f2_plan_of(int cls, int P) {
  if (cls != FX_CURL) return f2_plan(P);
  const FxPlan f = fx_plan(P);
  return F2Plan{f.n, {f.r[0], f.r[1], f.r[2], f.r[3], 1}};
}
// butterflies of radix R a thread takes: one of the small plans' butterflies, as many as in fx_nb in the others
__host__ __device__ constexpr int f2_nb(int cls, int P, int R) {
  const F2Plan f = f2_plan_of(cls, P);
  const bool small = cls != FX_CURL && f.n <= 3 && f.r[0] <= 9 && f.r[1] <= 9 && f.r[2] <= 9;
  return !small ? fx_nb(R) : (R == 4 ? 2 : (R == 3 ? 3 : (R == 2 ? 4 : 1)));
}
__host__ __device__ constexpr int f2_ept(int cls, int P) {
  int e = 18;
  for (int s = 0; s < f2_plan_of(cls, P).n; ++s) {
    const int R = f2_plan_of(cls, P).r[s], v = R * f2_nb(cls, P, R);
    if (v < e) e = v;
  }
  return e;
}
// threads of a full tile of the Biot-Savart pass; within a CTA's 512, else the length runs on the kernels of curl.cu
__host__ __device__ constexpr int f2_curl_threads(int P) {
  return 3 * (((P * fx_width(FX_CURL, P) + f2_ept(FX_CURL, P) - 1) / f2_ept(FX_CURL, P) + 31) / 32 * 32);
}
// What the lane pairs take: complex passes of powers of two stay on the column kernels (use_f2).
__host__ __device__ constexpr bool f2_complex(int P) { return (P & (P - 1)) != 0; }
__host__ __device__ constexpr bool f2_curl(int P) { return f2_curl_threads(P) <= 512; }
template <int P, int CLS> struct F2Rows {
  static constexpr int W = fx_width(CLS, P);
  static constexpr F2Plan plan = f2_plan_of(CLS, P);
  static constexpr int B = W < 8 && plan.r[0] % 2 == 0 ? plan.r[0] : 0;
  static constexpr int size = (P + (B ? (P - 1) / (B ? B : 1) : 0)) * W;
  __host__ __device__ static constexpr int at(int i) { return (B ? i + i / (B ? B : 1) : i) * W; }
  __host__ __device__ static constexpr bool linear(int n) { return !B || n % (B ? B : 1) == 0; }
  __host__ __device__ static constexpr int nb(int R) { return f2_nb(CLS, P, R); }
  __host__ __device__ static constexpr int prod(int s0, int s1) {
    int n = 1;
    for (int s = s0; s < s1; ++s) n *= f2_plan_of(CLS, P).r[s];
    return n;
  }
};
__host__ __device__ constexpr int f2_tile_values(int cls, int P) {
  const int W = fx_width(cls, P), r0 = f2_plan_of(cls, P).r[0];
  return (P + (W < 8 && r0 % 2 == 0 ? (P - 1) / r0 : 0)) * W;
}

}  // namespace flups
