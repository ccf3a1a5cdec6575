// Host-side check of the fixed-point arithmetic (csrc/fx64.cuh, compiled for the CPU; no device code runs):
// prints the largest errors, in units of the last place, of the register DFTs against long double sums of
// their definition, of the products against long double products, and of the FP64 decoding; inputs reach the bounds
// the header states.  One "name value" pair per line.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <random>

#include "fx64.cuh"
#include "fx_plan.cuh"

using namespace flups;
using ld = long double;
using C = std::complex<ld>;

static std::mt19937_64 gen(11);
static const ld kPi = 3.141592653589793238462643383279502884L;
static ld uni() { return std::uniform_real_distribution<double>(-1.0, 1.0)(gen); }

template <int R, bool INV> static ld dft_error() {
  ld worst = 0;
  for (int t = 0; t < 64; ++t) {
    cfx v[16];
    C x[16];
    for (int i = 0; i < R; ++i) {
      // bound of a decoded pair; t = 0: every part at it, t = 1: one value only
      const ld a = t == 0 ? 1 : uni(), b = t == 0 ? -1 : uni();
      const ld s = t == 1 && i != 1 ? 0 : 0x1.6ap57L;
      v[i].x = (long long)(a * s);
      v[i].y = (long long)(b * s);
      x[i] = C(v[i].x, v[i].y);
    }
    fx_dft<R, INV>(v);
    for (int k = 0; k < R; ++k) {
      C s = 0;
      for (int i = 0; i < R; ++i) s += x[i] * std::polar((ld)1, (INV ? 2 : -2) * kPi * (ld)(i * k % R) / R);
      worst = std::fmax(worst, std::abs(s - C(v[k].x, v[k].y)));
    }
  }
  return worst;
}
template <int R> static void dft_line() {
  std::printf("dft%d %.3Lg\ndft%d_inv %.3Lg\n", R, dft_error<R, false>(), R, dft_error<R, true>());
}

int main() {
  dft_line<2>(); dft_line<3>(); dft_line<4>(); dft_line<6>(); dft_line<8>(); dft_line<9>(); dft_line<12>(); dft_line<16>();
  ld wc = 0, wm = 0, wd = 0;
  for (int t = 0; t < 20000; ++t) {
    const ld a = kPi * uni(), ph = kPi * uni(), r = std::pow((ld)2, t % 2 ? 62.5L : 40 + 20 * uni());
    const long long wr = llroundl(ldexpl(cosl(a), kFxTwBits)), wi = llroundl(ldexpl(-sinl(a), kFxTwBits));
    const fxw w = {fx_hi(wr), fx_lo(wr), fx_hi(wi), fx_lo(wi)};
    const cfx x = fx_make((long long)(r * cosl(ph) * 0.999L), (long long)(r * sinl(ph) * 0.999L));
    const cfx p = fx_cmul<false>(x, w), q = fx_cmul<true>(x, w);
    wc = std::fmax(wc, std::abs(C(x.x, x.y) * C(wr, wi) / 0x1p64L - C(p.x, p.y)));
    wc = std::fmax(wc, std::abs(C(x.x, x.y) * C(wr, -wi) / 0x1p64L - C(q.x, q.y)));
    wm = std::fmax(wm, std::fabs((ld)x.x * wr / 0x1p64L - fx_mul(x.x, w.xh, w.xl)));
    const double d = std::ldexp((double)uni(), (int)(70 * uni()));
    const int E = 1023 + 70;
    unsigned long long b;
    std::memcpy(&b, &d, 8);
    wd = std::fmax(wd, std::fabs(ldexpl(d, kFxBias - E) - (ld)fx_decode(b, E)));
    if ((ld)fx_hi(x.x) * 0x1p32L + fx_lo(x.x) != (ld)x.x) return 1;
  }
  std::printf("cmul %.3Lg\nmul %.3Lg\ndecode %.4Lg\n", wc, wm, wd);
  // Mean decoding error of positive values 2^-d below the lane's largest, beyond the ties' bias of half a unit of the
  // value's own precision, and of values uniform up to the lane's largest: a one-sign field's errors must not add up.
  ld worst = 0, all = 0;
  for (int up = kFxUp; up <= kFxUp + kFxTwShift; up += kFxTwShift)
    for (int d = 0; d <= 48; ++d) {
      ld sum = 0;
      const int n = 100000;
      for (int i = 0; i < n; ++i) {
        unsigned long long b = ((unsigned long long)(1000 - d) << 52) | (gen() >> 12);
        double v;
        std::memcpy(&v, &b, 8);
        if (d == 0) {
          v = (double)ldexpl((ld)gen() + ldexpl((ld)gen(), -64), 1000 - 1023 - 64);
          std::memcpy(&b, &v, 8);
        }
        const ld e = fx_decode(b, 1000, up) - ldexpl(v, 1075 + up - 1000);
        sum += e;
        wd = std::fmax(wd, std::fabs(e));
      }
      if (d == 0) all = std::fmax(all, std::fabs(sum) / n);
      else worst = std::fmax(worst, std::fabs(sum) / n - (d > up ? ldexpl(0.5L, up - d) : 0));
    }
  std::printf("decode_all %.4Lg\ndecode_mean %.3Lg\ndecode_binade %.3Lg\n", wd, all, worst);
  // double-float values below the lane's largest (2^20): both floats rounded
  ld wdf = 0;
  for (int t = 0; t < 100000; ++t) {
    const double v = std::ldexp((double)uni(), 20 - (t % 60));
    const float hi = (float)v, lo = (float)(v - (double)hi);
    unsigned wh, wl;
    std::memcpy(&wh, &hi, 4);
    std::memcpy(&wl, &lo, 4);
    const int E = 1023 + 19;
    const unsigned long long b = ((unsigned long long)wl << 32) | wh;
    wdf = std::fmax(wdf, std::fabs(ldexpl((ld)hi + lo, kFxBias - E) - (ld)fx_decode_df(b, E)));
    if (fx_float_exp(wh & 0x7fffffffu) > E) return 13;
  }
  // subnormal floats: 2^-126 as the lane's largest beside 2^-140 and 2^-149
  if (fx_float_exp(0x00400000u) != 897 || fx_decode_df(0x00000001u, 897) != 1LL << (kFxUp + 29) ||
      fx_decode_df(0x8000020000800000ull, 897) != (1LL << (kFxUp + 52)) - (1LL << (kFxUp + 38)))
    return 17;
  if (fx_decode_df(0, kFxMinE) != 0 || fx_float_exp(0) != 0 || fx_float_exp(0x7f800000u) != 2047) return 14;
  std::printf("decode_df %.3Lg\n", wdf);
  // Green products: factors over 60 binary orders with modes over 60, the larger product of a pair aligned to 57 bits
  ld wg = 0, wa = 0;
  for (int t = 0; t < 100000; ++t) {
    cfx p[2];
    ld want[2];
    int d[2], T = 0;
    const int ref = 1023;
    for (int i = 0; i < 2; ++i) {
      const double g = std::ldexp((double)uni(), (int)(30 * uni()) - 40);
      const long long x = (long long)(0x1.69p62L * uni() * std::pow((ld)2, 30 * (uni() - 1)));
      unsigned long long b;
      std::memcpy(&b, &g, 8);
      const fxg q = fx_green(fx_green_pack(b, ref));
      if (ldexpl((ld)q.h * 0x1p32L + q.l, ref - q.d - 1075 - kFxGreenUp) != (ld)g) return 7;
      p[i] = fx_make(fx_mul(x, q.h, q.l), fx_mul(-x / 2, q.h, q.l));
      d[i] = q.d;
      want[i] = (ld)x * g;
      wg = std::fmax(wg, std::fabs(ldexpl(want[i], 1075 + kFxGreenUp - 64 - ref + d[i]) - p[i].x));
      const int b2 = fx_top_bit(p[i], d[i]);
      T = b2 > T ? b2 : T;
    }
    cfx a[2];
    for (int i = 0; i < 2; ++i) {
      a[i] = fx_align(p[i], d[i], T);
      // error of the alignment alone, in units of the aligned values
      wa = std::fmax(wa, std::fabs(ldexpl((ld)p[i].x, kFxAligned + kFxGreenRange - d[i] - T) - a[i].x));
      if (std::fabs(ldexpl(want[i], -fx_align_exp(T, ref)) - a[i].x) > 0x1p26L) return 12;  // a unit of a 31-bit product at most
      if (std::llabs(a[i].x) > 1LL << kFxAligned || std::llabs(a[i].y) > 1LL << kFxAligned) return 8;
    }
    // a product of 33 bits or more reaches the top
    if (std::llabs(p[0].x) >= 1LL << 33 && std::llabs(p[1].x) >= 1LL << 33 && std::llabs(a[0].x) < 1LL << (kFxAligned - 2) &&
        std::llabs(a[1].x) < 1LL << (kFxAligned - 2))
      return 9;
  }
  const fxg z = fx_green(fx_green_pack(0, 1000)), sb = fx_green(fx_green_pack(0x800fffffffffffffull, 1000));
  if (z.h || z.l || sb.h || sb.l || z.d != kFxGreenRange) return 10;
  if (fx_align(fx_make(0, 0), 0, fx_top_bit(fx_make(0, 0), 0)).x != 0) return 11;
  std::printf("green %.3Lg\nalign %.3Lg\n", wg, wa);
  std::printf("zero %lld\nsubnormal %lld\n", fx_decode(0, kFxMinE), fx_decode(0x800fffffffffffffull, kFxMinE));
  std::printf("shr_even %lld\n", fx_shr(24, 4) * 100 + fx_shr(8, 4) * 10 + fx_shr(7, 0));  // 1.5 -> 2, 0.5 -> 0, 7
  // every plan multiplies to its length within the block limits
#define CHECK(P, N, r0, r1, r2, r3) \
  if (r0 * r1 * r2 * r3 != P || fx_prod(P, 0, fx_plan(P).n) != P || N < 2 || fx_ept(P) < 12 || fx_ept(P) > 18) return 2;
  FX_LENGTHS(CHECK)
  // the tile's rows are distinct and inside the size that the planner allots
#define ROWS(P, N, r0, r1, r2, r3)                                                                            \
  if (FxRows<P, FX_PLAIN>::size != fx_tile_values(FX_PLAIN, P) || FxRows<P, FX_CURL>::size != fx_tile_values(FX_CURL, P)) return 3; \
  for (int i = 0; i < P; ++i)                                                                                 \
    if (FxRows<P, FX_PLAIN>::at(i) + FxRows<P, FX_PLAIN>::W > (i + 1 < P ? FxRows<P, FX_PLAIN>::at(i + 1) : FxRows<P, FX_PLAIN>::size)) return 4;
  FX_LENGTHS(ROWS)
#define ROWS2(P, N, r0, r1, r2, r3, r4)                                                                           \
  if (F2Rows<P, FX_PLAIN>::size != f2_tile_values(FX_PLAIN, P) || F2Rows<P, FX_CURL>::size != f2_tile_values(FX_CURL, P)) \
    return 5;                                                                                                     \
  if (r0 * r1 * r2 * r3 * r4 != P || F2Rows<P, FX_PLAIN>::prod(0, N) != P || f2_ept(FX_PLAIN, P) < 6) return 6;
  F2_LENGTHS(ROWS2)
  return 0;
}
