// 64-bit block fixed-point arithmetic of the FP64-class passes.
//
// GB300 has 2 FP64 lanes per SM and clock, but 64 lanes of 32-bit integer adds (ALU pipe) and 64 of
// 32 x 32 -> 64-bit integer multiply-adds (FMA pipe): measured 38 64-bit adds and 55 wide
// multiply-adds against 1.9 FP64 operations per SM and clock.  A 1D transform only adds and rotates,
// so it can run on integers that share one exponent: the FP64 values of a lane (one pencil, or the two
// real pencils packed in a lane) are aligned to the lane's largest exponent, transformed in 64-bit
// fixed point, and rounded once to FP64 at the end.
//
// Headroom.  Decoded parts are below 2^57, so a complex value is below 2^57.5 (2^58.5 for the sum of
// two packed pencils).  A radix-R butterfly grows the modulus by at most R <= 16; the twiddles of
// every following stage carry a factor 2^-4 (tables scaled by 2^60 against a product shifted by 64),
// so no value passes 2^62.5, and none 2^61.5 where two values are added before the next scaling.  The unit in
// the last place is 2^-57 of the lane's largest input: 16 times finer than the FP64 spacing at that value;
// lanes whose values do not grow are shifted up between stages (fx_kernels.cuh), so the coarsest rounding is
// the final one to FP64.  Values below 2^-4 of the lane's largest input hold less than FP64's 53 bits, and what lies below
// 2^-58 of it is lost: an error of each pass against its lane's largest value, where FP64's sums may also cancel
// exactly.  Infinite or NaN inputs make every value of their lane NaN.
//
// Products.  x = xh 2^32 + xl with both halves signed (|xl| <= 2^31), w likewise; (x w) >> 64 takes
// xh wh and the upper part of xh wl + xl wh and drops xl wl, which is below one unit.  |xh wl| <= 2^30.5 2^31
// and |xl wh| <= 2^31 2^28 (wh < 2^28 in the 2^60 tables), so the four middle products of a complex
// product stay below 2^63; the constants inside the butterflies multiply values below 2^60.5 by fractions
// whose magnitudes add up to at most 0.6, where the same sum is below 2^62.8.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace flups {

struct __align__(16) cfx {
  long long x, y;
};
// twiddle cos - i sin scaled by 2^60: high and low signed halves of both parts
struct __align__(16) fxw {
  int xh, xl, yh, yl;
};

#define FXD __host__ __device__ __forceinline__

FXD long long fx_mulw(int a, int b) { return (long long)a * b; }
// a b + c, one wide multiply-add
FXD long long fx_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)((unsigned long long)fx_mulw(a, b) + (unsigned long long)c);
#endif
}
// a K + c with an immediate factor
template <int K> FXD long long fx_madk(int a, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "n"(K), "l"(c));
  return r;
#else
  return (long long)((unsigned long long)fx_mulw(a, K) + (unsigned long long)c);
#endif
}
// c + (m >> 32): the upper half joins on the multiply pipe, sign extension included
FXD long long fx_top(long long m, long long c) { return fx_madk<1>((int)(m >> 32), c); }
// x = fx_hi(x) 2^32 + fx_lo(x), both signed
FXD int fx_lo(long long x) { return (int)(unsigned)(unsigned long long)x; }
FXD int fx_hi(long long x) {
  return (int)((unsigned)((unsigned long long)x >> 32) + ((unsigned)(unsigned long long)x >> 31));
}

FXD cfx fx_make(long long x, long long y) { cfx c; c.x = x; c.y = y; return c; }
FXD cfx fx_add(cfx a, cfx b) { return fx_make(a.x + b.x, a.y + b.y); }
FXD cfx fx_sub(cfx a, cfx b) { return fx_make(a.x - b.x, a.y - b.y); }
// times -i (forward) or +i (inverse)
template <bool INV> FXD cfx fx_mi(cfx a) { return INV ? fx_make(-a.y, a.x) : fx_make(a.y, -a.x); }

// Every shift rounds to nearest, decoding too: a truncation's mean error of half a unit is the same at every position, and
// a constant over the modes is a peak P times higher at the first point after the inverse transform (measured
// with truncation at 256^3: 1.3e-12 relative instead of 4e-16).  The half unit starts the multiply-add chain.
constexpr long long kFxHalf32 = 1LL << 31;
// t / 2, the half of an odd t rounded up or down by the lowest bit of r (no preferred direction)
FXD long long fx_half(long long t, long long r) { return (t + (r & 1)) >> 1; }
// x 2^-s rounded to nearest, ties to even
FXD long long fx_shr(long long x, int s) {
  const int one = s > 0 ? 1 : 0;
  return (x + (((1LL << s) >> 1) - one) + ((x >> s) & one)) >> s;
}

// Shifts by any count: 64 and more leave 0 or the sign (what PTX's shifts do; a clamp would cost an instruction).
FXD unsigned long long fx_lsr(unsigned long long x, int s) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s > 63 ? 0 : x >> s;
#endif
}
FXD long long fx_asr(long long x, int s) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return x >> (s > 63 ? 63 : s);
#endif
}

// round(x w 2^-64), w = wh 2^32 + wl
FXD long long fx_mul(long long x, int wh, int wl) {
  const int xh = fx_hi(x), xl = fx_lo(x);
  return fx_top(fx_mad(xl, wh, fx_mad(xh, wl, kFxHalf32)), fx_mulw(xh, wh));
}
// a w 2^-4 (w a table entry), or a conj(w) 2^-4
template <bool CONJ> FXD cfx fx_cmul(cfx a, fxw w) {
  const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
  const int nh = -w.yh, nl = -w.yl;
  const int ph = CONJ ? nh : w.yh, pl = CONJ ? nl : w.yl;   // imaginary part of the factor
  const int mh = CONJ ? w.yh : nh, ml = CONJ ? w.yl : nl;   // and its negative
  const long long mr = fx_mad(yl, mh, fx_mad(yh, ml, fx_mad(xl, w.xh, fx_mad(xh, w.xl, kFxHalf32))));
  const long long mi = fx_mad(xl, ph, fx_mad(xh, pl, fx_mad(yl, w.xh, fx_mad(yh, w.xl, kFxHalf32))));
  return fx_make(fx_top(mr, fx_mad(yh, mh, fx_mulw(xh, w.xh))), fx_top(mi, fx_mad(xh, ph, fx_mulw(yh, w.xh))));
}

// Constants of the butterflies: c = n + f 2^-64, n the nearest integer, so that x n starts the multiply-add
// chain and |f| <= 2^63 needs no doubling.
struct FX_C45 { static constexpr int n = 1; static constexpr long long f = -5402926248376769404LL; };  // cos(pi/4)
struct FX_C8 { static constexpr int n = 1; static constexpr long long f = -1404174782535421627LL; };  // cos(pi/8)
struct FX_S8 { static constexpr int n = 0; static constexpr long long f = 7059263338087549767LL; };  // sin(pi/8)
struct FX_S60 { static constexpr int n = 1; static constexpr long long f = -2471395088767036514LL; };  // sqrt(3)/2
struct FX_C40 { static constexpr int n = 1; static constexpr long long f = -4315718282406409839LL; };  // cos(2 pi/9)
struct FX_S40 { static constexpr int n = 1; static constexpr long long f = -6589405544070453923LL; };  // sin(2 pi/9)
struct FX_C80 { static constexpr int n = 0; static constexpr long long f = 3203243492287910726LL; };  // cos(4 pi/9)
struct FX_S80 { static constexpr int n = 1; static constexpr long long f = -280247492088382768LL; };  // sin(4 pi/9)
struct FX_C160 { static constexpr int n = -1; static constexpr long long f = 1112474790118499113LL; };  // cos(8 pi/9)
struct FX_S160 { static constexpr int n = 0; static constexpr long long f = 6309158051982071155LL; };  // sin(8 pi/9)
template <class C> struct FxNeg { static constexpr int n = -C::n; static constexpr long long f = -C::f; };
template <class C> struct FxHalves {
  static constexpr int l = (int)(unsigned)((unsigned long long)C::f & 0xffffffffull);
  static constexpr int h = (int)((C::f - l) >> 32);
};
template <int N> FXD long long fx_nx(long long x) { return N == 0 ? 0 : (N > 0 ? x : -x); }
// round(x c)
template <class C> FXD long long fx_mulc(long long x) {
  using K = FxHalves<C>;
  const int xh = fx_hi(x), xl = fx_lo(x);
  return fx_top(fx_madk<K::h>(xl, fx_madk<K::l>(xh, kFxHalf32)), fx_madk<K::h>(xh, fx_nx<C::n>(x)));
}
// round(x c + y s)
template <class C, class S> FXD long long fx_dot(long long x, int xh, int xl, long long y, int yh, int yl) {
  using K = FxHalves<C>;
  using L = FxHalves<S>;
  const long long m = fx_madk<L::h>(yl, fx_madk<L::l>(yh, fx_madk<K::h>(xl, fx_madk<K::l>(xh, kFxHalf32))));
  return fx_top(m, fx_madk<L::h>(yh, fx_madk<K::h>(xh, fx_nx<C::n>(x) + fx_nx<S::n>(y))));
}
// a (C - i S) (forward) or a (C + i S) (inverse)
template <bool INV, class C, class S> FXD cfx fx_rot(cfx a) {
  const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
  using P = std::conditional_t<INV, FxNeg<S>, S>;   // re = C x + P y
  using M = std::conditional_t<INV, S, FxNeg<S>>;   // im = C y + M x
  return fx_make(fx_dot<C, P>(a.x, xh, xl, a.y, yh, yl), fx_dot<C, M>(a.y, yh, yl, a.x, xh, xl));
}
// a W8 and a W8^3 (forward), or their conjugates
template <bool INV> FXD cfx fx_rot8_1(cfx a) {
  return INV ? fx_make(fx_mulc<FX_C45>(a.x - a.y), fx_mulc<FX_C45>(a.x + a.y))
             : fx_make(fx_mulc<FX_C45>(a.x + a.y), fx_mulc<FX_C45>(a.y - a.x));
}
template <bool INV> FXD cfx fx_rot8_3(cfx a) {
  return INV ? fx_make(fx_mulc<FxNeg<FX_C45>>(a.x + a.y), fx_mulc<FX_C45>(a.x - a.y))
             : fx_make(fx_mulc<FX_C45>(a.y - a.x), fx_mulc<FxNeg<FX_C45>>(a.x + a.y));
}

// ---------------------------------------------------------------------------
// Register DFTs (forward exp(-2 pi i q r / R)), natural order in and out.
// ---------------------------------------------------------------------------
template <bool INV> FXD void fx_dft2(cfx& a, cfx& b) {
  const cfx t = a;
  a = fx_add(t, b);
  b = fx_sub(t, b);
}
template <bool INV> FXD void fx_dft3(cfx& a, cfx& b, cfx& c) {
  const cfx t1 = fx_add(b, c), d = fx_sub(b, c);
  const cfx t2 = fx_make(a.x - fx_half(t1.x, a.x), a.y - fx_half(t1.y, a.y));
  const cfx t3 = fx_mi<INV>(fx_make(fx_mulc<FX_S60>(d.x), fx_mulc<FX_S60>(d.y)));
  a = fx_add(a, t1);
  b = fx_add(t2, t3);
  c = fx_sub(t2, t3);
}
template <bool INV> FXD void fx_dft4(cfx& a, cfx& b, cfx& c, cfx& d) {
  const cfx t0 = fx_add(a, c), t1 = fx_sub(a, c), t2 = fx_add(b, d), u = fx_sub(b, d);
  a = fx_add(t0, t2);
  c = fx_sub(t0, t2);
  // t1 -+ i u without forming the rotated value
  const cfx p = fx_make(t1.x + u.y, t1.y - u.x), m = fx_make(t1.x - u.y, t1.y + u.x);
  b = INV ? m : p;
  d = INV ? p : m;
}
template <bool INV> FXD void fx_dft8(cfx* v) {
  cfx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  fx_dft4<INV>(e0, e1, e2, e3);
  fx_dft4<INV>(o0, o1, o2, o3);
  o1 = fx_rot8_1<INV>(o1);
  o3 = fx_rot8_3<INV>(o3);
  v[0] = fx_add(e0, o0);
  v[4] = fx_sub(e0, o0);
  v[1] = fx_add(e1, o1);
  v[5] = fx_sub(e1, o1);
  const cfx p = fx_make(e2.x + o2.y, e2.y - o2.x), m = fx_make(e2.x - o2.y, e2.y + o2.x);  // e2 -+ i o2
  v[2] = INV ? m : p;
  v[6] = INV ? p : m;
  v[3] = fx_add(e3, o3);
  v[7] = fx_sub(e3, o3);
}
template <bool INV> FXD void fx_dft16(cfx* v) {
  // 4 x 4: columns n2 hold x[4 n1 + n2]; twiddles W16^(n2 k1); rows k1
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) fx_dft4<INV>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
  v[5] = fx_rot<INV, FX_C8, FX_S8>(v[5]);
  v[6] = fx_rot8_1<INV>(v[6]);
  v[7] = fx_rot<INV, FX_S8, FX_C8>(v[7]);
  v[9] = fx_rot8_1<INV>(v[9]);
  v[10] = fx_mi<INV>(v[10]);
  v[11] = fx_rot8_3<INV>(v[11]);
  v[13] = fx_rot<INV, FX_S8, FX_C8>(v[13]);
  v[14] = fx_rot8_3<INV>(v[14]);
  v[15] = fx_rot<INV, FxNeg<FX_C8>, FxNeg<FX_S8>>(v[15]);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) fx_dft4<INV>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
  cfx t[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) t[i] = v[i];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = t[4 * k1 + k2];
}
// coprime factors need no twiddles: input n = 3 n1 + 2 n2 (6), 4 n1 + 3 n2 (12), output by the
// Chinese remainder theorem k = 3 k1 + 4 k2 (6), 4 k1 + 9 k2 (12)
template <bool INV> FXD void fx_dft6(cfx* v) {
  cfx a[3], b[3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    a[n2] = v[(2 * n2) % 6];
    b[n2] = v[(3 + 2 * n2) % 6];
    fx_dft2<INV>(a[n2], b[n2]);
  }
  fx_dft3<INV>(a[0], a[1], a[2]);
  fx_dft3<INV>(b[0], b[1], b[2]);
#pragma unroll
  for (int k2 = 0; k2 < 3; ++k2) {
    v[(4 * k2) % 6] = a[k2];
    v[(3 + 4 * k2) % 6] = b[k2];
  }
}
template <bool INV> FXD void fx_dft12(cfx* v) {
  cfx t[3][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) t[n1][n2] = v[(4 * n1 + 3 * n2) % 12];
    fx_dft3<INV>(t[0][n2], t[1][n2], t[2][n2]);
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    fx_dft4<INV>(t[k1][0], t[k1][1], t[k1][2], t[k1][3]);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[(4 * k1 + 9 * k2) % 12] = t[k1][k2];
  }
}
template <bool INV> FXD void fx_dft9(cfx* v) {
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) fx_dft3<INV>(v[n2], v[3 + n2], v[6 + n2]);
  v[4] = fx_rot<INV, FX_C40, FX_S40>(v[4]);
  v[5] = fx_rot<INV, FX_C80, FX_S80>(v[5]);
  v[7] = fx_rot<INV, FX_C80, FX_S80>(v[7]);
  v[8] = fx_rot<INV, FX_C160, FX_S160>(v[8]);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) fx_dft3<INV>(v[3 * k1], v[3 * k1 + 1], v[3 * k1 + 2]);
  cfx t[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) t[i] = v[i];
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[3 * k1 + k2];
}
template <int R, bool INV> FXD void fx_dft(cfx* v) {
  if constexpr (R == 2) fx_dft2<INV>(v[0], v[1]);
  else if constexpr (R == 3) fx_dft3<INV>(v[0], v[1], v[2]);
  else if constexpr (R == 4) fx_dft4<INV>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 6) fx_dft6<INV>(v);
  else if constexpr (R == 8) fx_dft8<INV>(v);
  else if constexpr (R == 9) fx_dft9<INV>(v);
  else if constexpr (R == 12) fx_dft12<INV>(v);
  else fx_dft16<INV>(v);
}

// ---------------------------------------------------------------------------
// FP64 <-> lane fixed point.  E is the lane's largest biased exponent (kFxMinE .. 2046; 2047 marks a lane
// with an infinite or NaN input): value = fixed 2^(E - kFxBias).  With E at least 64, a zero's or subnormal's
// shift empties the word, so the implicit bit needs no test (lanes below 1e-289 lose bits towards FP64's own
// underflow).
// ---------------------------------------------------------------------------
constexpr int kFxUp = 4;                  // bits below the FP64 unit of the lane's largest value
constexpr int kFxBias = 1075 + kFxUp;
constexpr int kFxMinE = 80;
constexpr int kFxTwBits = 60;             // scale of the twiddle tables
constexpr int kFxTwShift = 64 - kFxTwBits;  // every twiddled stage divides by 2^4

// up: bits below the FP64 unit of the largest value (at most 8).  The word is aligned one bit higher and rounded to
// nearest by that bit.  Ties go away from zero: that adds at most half a unit of the value's own FP64 precision, and only where
// one bit of it is dropped (2^-54 of the value), so one-sign inputs gain no error that FP64 would not have; a
// truncation has half a unit of the lane's largest value instead.  (Rounding costs about 2% of a solve; to nearest even,
// from the dropped bits' carry, 7-10%: open 128^3 326 us, periodic 1024^3 44.5 ms, truncated 294 and 41.1.)
FXD long long fx_decode(unsigned long long bits, int E, int up = kFxUp) {
  const int hi = (int)(unsigned)(bits >> 32);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << (up + 1);
  const int s = E - e, sg = hi >> 31;
  const long long t = (long long)fx_lsr(m, s);
  return ((t ^ sg) + 1) >> 1;
}

// The same for a double-float value hi + lo (hi in the lower word): both floats aligned and rounded to nearest.
FXD long long fx_decode_float(unsigned w, int E, int up) {
  const int e = (int)(w >> 23) & 255, sg = (int)w >> 31, s = E - (e ? e : 1) - 896;
  const unsigned long long m = (unsigned long long)((w & 0x7fffffu) | (e ? 0x800000u : 0)) << (30 + up);
  const long long t = (long long)fx_lsr(m, s);
  return ((t ^ sg) + 1) >> 1;
}
FXD long long fx_decode_df(unsigned long long bits, int E, int up = kFxUp) {
  return fx_decode_float((unsigned)bits, E, up) + fx_decode_float((unsigned)(bits >> 32), E, up);
}
// FP64's biased exponent of the larger float of a double-float value, from its bits without the sign
FXD int fx_float_exp(unsigned w) {
  const int e = (int)(w >> 23);
  return w == 0 ? 0 : (e == 255 ? 2047 : (e ? e : 1) + 896);
}

// Green factors keep FP64's 53 bits and an exponent each: a pencil's factors fall by many orders of magnitude (1/k^2,
// Gaussians), and modes under large factors decide the solution.  Word: the factor at 2^61 <= |g| < 2^62 in signed
// halves, and in the low half's 9 zero bits the binary orders below the spectrum's largest exponent (`ref`); a
// factor 2^-511 below it is zero.  The products round(x g 2^-64) of parts |x| < 2^62.5 stay below 2^60.5 (xl gh + xh gl
// below 2^62.4) and are aligned one by one to the lane's largest.  (With factors in one fixed point per pencil and
// products rounded at the scale of the largest factor times the largest mode, a periodic field with a mean had an
// error of 1.1e-13 instead of 1.2e-15 at 1024 points.)
struct fxg {
  int h, l, d;
};
constexpr int kFxGreenUp = 9, kFxGreenRange = (1 << kFxGreenUp) - 1;
FXD unsigned long long fx_green_pack(unsigned long long bits, int ref) {
  const int hi = (int)(unsigned)(bits >> 32), sg = hi >> 31, e = (hi >> 20) & 0x7ff, d = ref - e;
  if (e == 0 || d >= kFxGreenRange) return kFxGreenRange;
  const long long m = (long long)(((bits & 0xfffffffffffffull) | 0x10000000000000ull) << kFxGreenUp), v = (m ^ sg) - sg;
  return ((unsigned long long)(unsigned)fx_hi(v) << 32) | (unsigned)fx_lo(v) | (unsigned)d;
}
FXD fxg fx_green(unsigned long long word) {
  const int lo = (int)(unsigned)word;
  fxg g;
  g.h = (int)(unsigned)(word >> 32);
  g.l = lo & ~kFxGreenRange;
  g.d = lo & kFxGreenRange;
  return g;
}
// Top bit (from the upper words; at least 32) of a product with a factor d orders down.
FXD int fx_top_bit(cfx p, int d) {
  const int x = (int)(p.x >> 32), y = (int)(p.y >> 32);
  const unsigned m = (unsigned)((x ^ (x >> 31)) | (y ^ (y >> 31)));
#ifdef __CUDA_ARCH__
  const int z = __clz((int)m);
#else
  const int z = m ? __builtin_clz(m) : 32;
#endif
  return 64 + kFxGreenRange - z - d;
}
// The product at the lane's scale, where the largest one (top bit T) has 57 bits; rounded to nearest (a tie goes up,
// which happens to values whose own last bit is the dropped one).
constexpr int kFxAligned = 57;
FXD long long fx_align1(long long p, int l, int r) { return (fx_asr(p << l, r) + 1) >> 1; }
FXD cfx fx_align(cfx p, int d, int T) {
  const int n = kFxAligned + kFxGreenRange - T - d;
  const int l = n < 0 ? 1 : n + 1, r = n < 0 ? -n : 0;
  return fx_make(fx_align1(p.x, l, r), fx_align1(p.y, l, r));
}
// x g = aligned value times 2 to this
FXD int fx_align_exp(int T, int ref) { return T - kFxAligned - kFxGreenRange + ref - (1075 + kFxGreenUp - 64); }

}  // namespace flups
