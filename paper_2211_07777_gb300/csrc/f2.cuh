// Pairs of FP32 transforms in packed arithmetic (sm_100+: one instruction adds, multiplies or multiply-adds two
// floats held in a 64-bit register pair).
//
// A value holds the same position of two independent complex sequences: x = (re0, re1), y = (im0, im1).  Every
// step of a transform then costs half the instructions per value, and twiddles and addresses are shared by the
// two; the FP32 passes were bound by instruction issue, not by the FP32 lanes.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace flups {

using f2 = unsigned long long;  // (low, high) floats
struct __align__(16) cf2 {
  f2 x, y;
};
// twiddle c - i s, each part twice
struct __align__(16) f2w {
  f2 c, s;
};

#define F2D __device__ __forceinline__

F2D f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
F2D float2 f2_get(f2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
F2D f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
F2D f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
F2D f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
F2D f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }
F2D f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
F2D f2 f2_dup(float a) { return f2_pack(a, a); }

F2D cf2 f2_make(f2 x, f2 y) { cf2 c; c.x = x; c.y = y; return c; }
F2D cf2 operator+(cf2 a, cf2 b) { return f2_make(f2_add(a.x, b.x), f2_add(a.y, b.y)); }
F2D cf2 operator-(cf2 a, cf2 b) { return f2_make(f2_sub(a.x, b.x), f2_sub(a.y, b.y)); }
F2D cf2 f2_scale(cf2 a, f2 s) { return f2_make(f2_mul(a.x, s), f2_mul(a.y, s)); }
// a (c - i s), or a (c + i s) with CONJ
template <bool CONJ> F2D cf2 f2_cmul(cf2 a, f2 c, f2 s) {
  const f2 tx = f2_mul(a.x, s), ty = f2_mul(a.y, s);
  return CONJ ? f2_make(f2_sub(f2_mul(a.x, c), ty), f2_fma(a.y, c, tx))
              : f2_make(f2_fma(a.x, c, ty), f2_sub(f2_mul(a.y, c), tx));
}
// a (C - i S) for constants, forward, or its conjugate
template <bool INV> F2D cf2 f2_rot(cf2 a, float C, float S) {
  const f2 c = f2_dup(C), s = f2_dup(INV ? -S : S), n = f2_dup(INV ? S : -S);
  return f2_make(f2_fma(a.y, s, f2_mul(a.x, c)), f2_fma(a.x, n, f2_mul(a.y, c)));
}
template <bool INV> F2D cf2 f2_mi(cf2 a) { return INV ? f2_make(f2_neg(a.y), a.x) : f2_make(a.y, f2_neg(a.x)); }
// a W8 and a W8^3 (forward), or their conjugates
template <bool INV> F2D cf2 f2_rot8_1(cf2 a) {
  const f2 r = f2_dup(0.70710678118654752440f);
  const f2 p = f2_add(a.x, a.y), m = INV ? f2_sub(a.x, a.y) : f2_sub(a.y, a.x);
  return INV ? f2_make(f2_mul(m, r), f2_mul(p, r)) : f2_make(f2_mul(p, r), f2_mul(m, r));
}
template <bool INV> F2D cf2 f2_rot8_3(cf2 a) {
  const f2 r = f2_dup(0.70710678118654752440f), n = f2_dup(-0.70710678118654752440f);
  const f2 p = f2_add(a.x, a.y), m = INV ? f2_sub(a.x, a.y) : f2_sub(a.y, a.x);
  return INV ? f2_make(f2_mul(p, n), f2_mul(m, r)) : f2_make(f2_mul(m, r), f2_mul(p, n));
}

// ---------------------------------------------------------------------------
// Register DFTs (forward exp(-2 pi i q r / R)), natural order in and out.
// ---------------------------------------------------------------------------
template <bool INV> F2D void f2_dft2(cf2& a, cf2& b) {
  const cf2 t = a;
  a = t + b;
  b = t - b;
}
// p -+ i u (forward minus), and its conjugate partner
template <bool INV> F2D void f2_pm(cf2 p, cf2 u, cf2& lo, cf2& hi) {
  const cf2 a = f2_make(f2_add(p.x, u.y), f2_sub(p.y, u.x)), b = f2_make(f2_sub(p.x, u.y), f2_add(p.y, u.x));
  lo = INV ? b : a;
  hi = INV ? a : b;
}
template <bool INV> F2D void f2_dft3(cf2& a, cf2& b, cf2& c) {
  const cf2 t1 = b + c, d = b - c;
  const f2 h = f2_dup(-0.5f);
  const cf2 t2 = f2_make(f2_fma(t1.x, h, a.x), f2_fma(t1.y, h, a.y));
  const cf2 u = f2_scale(d, f2_dup(0.86602540378443864676f));
  a = a + t1;
  f2_pm<INV>(t2, u, b, c);
}
template <bool INV> F2D void f2_dft4(cf2& a, cf2& b, cf2& c, cf2& d) {
  const cf2 t0 = a + c, t1 = a - c, t2 = b + d, u = b - d;
  a = t0 + t2;
  c = t0 - t2;
  f2_pm<INV>(t1, u, b, d);
}
template <bool INV> F2D void f2_dft8(cf2* v) {
  cf2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  f2_dft4<INV>(e0, e1, e2, e3);
  f2_dft4<INV>(o0, o1, o2, o3);
  o1 = f2_rot8_1<INV>(o1);
  o3 = f2_rot8_3<INV>(o3);
  v[0] = e0 + o0;
  v[4] = e0 - o0;
  v[1] = e1 + o1;
  v[5] = e1 - o1;
  f2_pm<INV>(e2, o2, v[2], v[6]);
  v[3] = e3 + o3;
  v[7] = e3 - o3;
}
template <bool INV> F2D void f2_dft16(cf2* v) {
  // 4 x 4: columns n2 hold x[4 n1 + n2]; twiddles W16^(n2 k1); rows k1
  constexpr float c8 = 0.92387953251128675613f, s8 = 0.38268343236508977173f;
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) f2_dft4<INV>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
  v[5] = f2_rot<INV>(v[5], c8, s8);
  v[6] = f2_rot8_1<INV>(v[6]);
  v[7] = f2_rot<INV>(v[7], s8, c8);
  v[9] = f2_rot8_1<INV>(v[9]);
  v[10] = f2_mi<INV>(v[10]);
  v[11] = f2_rot8_3<INV>(v[11]);
  v[13] = f2_rot<INV>(v[13], s8, c8);
  v[14] = f2_rot8_3<INV>(v[14]);
  v[15] = f2_rot<INV>(v[15], -c8, -s8);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) f2_dft4<INV>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
  cf2 t[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) t[i] = v[i];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = t[4 * k1 + k2];
}
// coprime factors need no twiddles: input n = 3 n1 + 2 n2 (6), 4 n1 + 3 n2 (12), output by the
// Chinese remainder theorem k = 3 k1 + 4 k2 (6), 4 k1 + 9 k2 (12)
template <bool INV> F2D void f2_dft6(cf2* v) {
  cf2 a[3], b[3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    a[n2] = v[(2 * n2) % 6];
    b[n2] = v[(3 + 2 * n2) % 6];
    f2_dft2<INV>(a[n2], b[n2]);
  }
  f2_dft3<INV>(a[0], a[1], a[2]);
  f2_dft3<INV>(b[0], b[1], b[2]);
#pragma unroll
  for (int k2 = 0; k2 < 3; ++k2) {
    v[(4 * k2) % 6] = a[k2];
    v[(3 + 4 * k2) % 6] = b[k2];
  }
}
template <bool INV> F2D void f2_dft12(cf2* v) {
  cf2 t[3][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) t[n1][n2] = v[(4 * n1 + 3 * n2) % 12];
    f2_dft3<INV>(t[0][n2], t[1][n2], t[2][n2]);
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    f2_dft4<INV>(t[k1][0], t[k1][1], t[k1][2], t[k1][3]);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[(4 * k1 + 9 * k2) % 12] = t[k1][k2];
  }
}
template <bool INV> F2D void f2_dft9(cf2* v) {
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) f2_dft3<INV>(v[n2], v[3 + n2], v[6 + n2]);
  v[4] = f2_rot<INV>(v[4], 0.76604444311897803520f, 0.64278760968653932632f);
  v[5] = f2_rot<INV>(v[5], 0.17364817766693034885f, 0.98480775301220805937f);
  v[7] = f2_rot<INV>(v[7], 0.17364817766693034885f, 0.98480775301220805937f);
  v[8] = f2_rot<INV>(v[8], -0.93969262078590838405f, 0.34202014332566873304f);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) f2_dft3<INV>(v[3 * k1], v[3 * k1 + 1], v[3 * k1 + 2]);
  cf2 t[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) t[i] = v[i];
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[3 * k1 + k2];
}
template <int R, bool INV> F2D void f2_dft(cf2* v) {
  if constexpr (R == 2) f2_dft2<INV>(v[0], v[1]);
  else if constexpr (R == 3) f2_dft3<INV>(v[0], v[1], v[2]);
  else if constexpr (R == 4) f2_dft4<INV>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 6) f2_dft6<INV>(v);
  else if constexpr (R == 8) f2_dft8<INV>(v);
  else if constexpr (R == 9) f2_dft9<INV>(v);
  else if constexpr (R == 12) f2_dft12<INV>(v);
  else f2_dft16<INV>(v);
}

}  // namespace flups
