// FP64-class passes (FP64 arrays in and out) in 64-bit block fixed point (fx64.cuh): all five of a Poisson solve, the
// four around the curl of a Biot-Savart solve (whose own array is double-float on FP64E), and the DCT-I of every
// precision's Green spectrum.  One kernel per pass kind and length P = 2^a 3^b, for every axis and tile width.
//
// A CTA holds W lanes (pencils; two packed real pencils per lane for real data) x P complex values
// in shared memory and transforms them in place: a thread takes whole butterflies of up to 18 values in
// registers, the block synchronises, and the values go back.  Complex passes read the first stage's
// inputs from HBM into registers and store the last stage's outputs from registers, as do the real
// passes of periodic and unbounded directions; symmetric directions build their extension in shared
// memory.  Each length has its plan of radices 16, 12, 9, 8, 6, 4, 3, 2 at compile time (fx_plan), so the
// factor 3 costs no separate engine; the tile width stays a run-time value, one integer operation per access.
#pragma once
#include <cuda_runtime.h>

#include "fx64.cuh"
#include "fx_plan.cuh"
#include "green.cuh"
#include "pass_common.cuh"
#include "passes.cuh"

namespace flups {

namespace {

// A tile's shared memory after the 128-byte block of its mbarrier: S, then lane exponents and Green
// offsets, then the staged Green slice (128-byte aligned).
// renormalisation slots: second to fourth stage forward (and before the Green product, one more), the products' top
// bit, second to fourth stage inverse
constexpr int kFxSlotFwd = 0, kFxSlotGain = 4, kFxSlotInv = 5;

struct FxSmem {
  cfx* S;
  int* emax;          // W lane exponents
  unsigned* words;    // kFxSlots x W magnitudes (upper words ORed) behind the lanes' renormalisations
  long long* goff;    // 2 W Green offsets
  unsigned long long* mbar;
  unsigned long long* G;  // staged slice: factors by folded mode and pencil
};

__device__ __forceinline__ FxSmem fx_smem(unsigned char* smraw, int W, int rows) {
  FxSmem m;
  unsigned char* base = smraw + ((128u - (smem_u32(smraw) & 127u)) & 127u);
  m.mbar = reinterpret_cast<unsigned long long*>(base);
  m.S = reinterpret_cast<cfx*>(base + 128);
  m.goff = reinterpret_cast<long long*>(base + 128 + (size_t)rows * sizeof(cfx));
  m.emax = reinterpret_cast<int*>(m.goff + 2 * W);
  m.words = reinterpret_cast<unsigned*>(m.emax + W);
  unsigned char* g = reinterpret_cast<unsigned char*>(m.words + kFxSlots * W);
  m.G = reinterpret_cast<unsigned long long*>(g + ((128u - (smem_u32(g) & 127u)) & 127u));
  return m;
}

__device__ __forceinline__ unsigned abs_hi(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
__device__ __forceinline__ long long dec(double d, int E, int up = kFxUp) {
  return fx_decode((unsigned long long)__double_as_longlong(d), E, up);
}
// a double-float value's bits; out of line, so that the passes' code stays short
__device__ __noinline__ long long dec_df(double d, int E, int up) {
  return fx_decode_df((unsigned long long)__double_as_longlong(d), E, up);
}
// FP64 value of x 2^q rounded to nearest, for results in FP64's normal range.  The conversion runs on the FP64
// pipe (measured 1.9 per SM and clock), which is otherwise idle, and the scale joins the exponent field;
// normalising in integers took 3 times the instructions.
__device__ __forceinline__ double enc(long long x, int q) {
  const double d = __ll2double_rn(x);
  const int h = __double2hiint(d);
  return __hiloint2double(h ? h + (q << 20) : 0, __double2loint(d));
}
// the same for any scale (kind 1), or NaN (kind 2); out of line, so that the passes' code stays short
__device__ __noinline__ double enc_slow(long long x, int q, int kind) {
  return kind == 1 ? scalbn(__ll2double_rn(x), q) : __longlong_as_double(0x7ff8000000000000ll);
}
// the same as a double-float value (kind 3: the array of the double-float curl), hi in the lower word.  Conversions
// between 32-bit integers and floats: the value is shifted up to 62 bits, hi takes the upper word's 24 leading bits, lo
// the rest, at most 2^38, in steps of 2^8 (conversions of 64-bit integers run at 4.5 per SM and clock: forward pass
// beside the curl, open 128^3, 161 us)
__device__ __forceinline__ double enc_df(long long x, int q) {
  const int h0 = (int)(x >> 32), z = max(__clz(h0 ^ (h0 >> 31)) - 2, 0);
  x <<= z;
  const int xh = fx_hi(x), xl = fx_lo(x);
  const float a = __int2float_rn(xh);
  const long long r = (((long long)(xh - __float2int_rz(a)) << 32) + xl + 128) >> 8;
  const int s = min(max(q - z, -250), 190), s1 = s >> 1, s2 = s - s1;
  const float sa = __int_as_float((s1 + 127) << 23), sb = __int_as_float((s2 + 127) << 23);
  return __hiloint2double(__float_as_int(__int2float_rn((int)r) * sa * 256.f * sb), __float_as_int(a * sa * 4294967296.f * sb));
}
__device__ __forceinline__ double enc_any(long long x, int q, int kind) {
  if (__builtin_expect(kind == 0, 1)) return enc(x, q);
  return kind == 3 ? enc_df(x, q) : enc_slow(x, q, kind);
}
// 0: every |x| < 2^63 scales to a normal number (or 0); 1: not so; 2: NaN lane
__device__ __forceinline__ int fx_out_kind(int E, int q) { return E >= 2047 ? 2 : (q > -1020 && q < 950 ? 0 : 1); }

__device__ __forceinline__ int fx_store_kind(const PassParams& p, int E, int q) {
  const int kind = fx_out_kind(E, q);
  return (p.fx_df & 2) && kind != 2 ? 3 : kind;
}

// Largest magnitude (upper words) of the lane's inputs over the CTA, as a biased exponent; a thread's
// inputs belong to lane `lane` = tid mod W.
__device__ __forceinline__ void lane_max(int* emax, unsigned m, int W, int lane, int tid) {
  for (int o = W; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) < W) atomicMax(&emax[lane], (int)(m >> 20));
}

__device__ __forceinline__ fxw fx_twiddle(const fxw* tw, int i) {
  const int4 q = __ldg(reinterpret_cast<const int4*>(tw + i));
  fxw w;
  w.xh = q.x;
  w.xl = q.y;
  w.yh = q.z;
  w.yl = q.w;
  return w;
}

template <int N> using ic = std::integral_constant<int, N>;

struct FxTile {
  cfx* S;
  int W, lw, tid, nt;
  const fxw* tw;
  bool df;  // FX_RAW_DF: the input array holds double-float values
};
// Rows of the tile are a compile-time number of values apart (FxRows), so that a butterfly's accesses are offsets
// from one address; narrower tiles of small grids keep the stride.
// Values j + r nbf of a butterfly from the tile, and its outputs o + r Ns into it
template <class RW> struct FxFromS {
  const cfx* S;
  template <int R, int nbf> __device__ __forceinline__ void operator()(ic<R>, ic<nbf>, int j, int l, cfx* v) const {
    const cfx* s = S + RW::at(j) + l;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (RW::linear(nbf)) v[r] = s[RW::at(r * nbf)];
      else v[r] = S[RW::at(j + r * nbf) + l];
    }
  }
};
template <class RW> struct FxToS {
  cfx* S;
  template <int R, int Ns> __device__ __forceinline__ void operator()(ic<R>, ic<Ns>, int o, int l, const cfx* v) const {
    cfx* s = S + RW::at(o) + l;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (RW::linear(Ns) || (Ns == 1 && R == RW::B)) s[RW::at(r * Ns)] = v[r];
      else S[RW::at(o + r * Ns) + l] = v[r];
    }
  }
};

// Lane renormalisation.  The fixed factor 2^-4 of a twiddled stage is what the worst case needs; a lane whose
// values did not grow (a spectrum of a few modes) would lose those bits at every stage.  From the second stage
// of a transform on, and before the Green product, the lane's values are therefore shifted up to the bound
// again: the stage before ORs the magnitudes of its outputs' upper words per lane, the next one shifts by
// the free bits, eight integer operations per value.  (The Green products are aligned one by one, fx_align.)  (Relative error against a 64-bit solution, mixed 256^3: 1e-13
// to 1.7e-12 with the fixed factors alone, 4e-16 to 5e-15 with the shift from the third stage on.)
enum FxSrc : int { FX_TILE = 0, FX_RAW = 1, FX_GAIN = 2, FX_RAW_DF = 3 };
__device__ __forceinline__ int fx_free_tw(unsigned w) { return max(__clz(w) - 3, 0); }    // parts below 2^61
__device__ __forceinline__ unsigned fx_mag(long long x) {
  const int h = (int)(x >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned fx_mag_df(long long bits) {
  return max((unsigned)bits & 0x7fffffffu, (unsigned)((unsigned long long)bits >> 32) & 0x7fffffffu);
}
__device__ __forceinline__ void lane_or(unsigned* word, unsigned m, int W, int lane, int tid) {
  for (int o = W; o < 32; o <<= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
  if ((tid & 31) < W) atomicOr(&word[lane], m);
}
// Largest top bit of the lane's products.
__device__ __forceinline__ void lane_top(unsigned* word, int m, int W, int lane, int tid) {
  for (int o = W; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) < W) atomicMax(reinterpret_cast<int*>(&word[lane]), m);
}
// Shift that the renormalisations of lane l added: forward and inverse transforms of the plan, before the product.
template <int P>
__device__ __forceinline__ int fx_shifted(const unsigned* words, int W, int l, bool fwd, bool gain, bool inv) {
  constexpr int n = fx_plan(P).n;
  int e = gain ? fx_free_tw(words[(kFxSlotFwd + n - 1) * W + l]) : 0;
#pragma unroll
  for (int s = 1; s < n; ++s) {
    if (fwd) e += fx_free_tw(words[(kFxSlotFwd + s - 1) * W + l]);
    if (inv) e += fx_free_tw(words[(kFxSlotInv + s - 1) * W + l]);
  }
  return e;
}

// One stage of radix R after a product Ns of earlier radices.  SRC: FX_RAW, In gives FP64 bits, aligned to the
// lane's exponent (maxima in `lanes`) here, FX_RAW_DF the same or double-float values; FX_GAIN, In gives Green products (FxGained) and aligns them to the lane's
// largest (`lanes`).  words: the transform's slots; every stage but the first is renormalised.  In and Out move whole butterflies: values
// at positions j + r P/R, outputs at o + r Ns.
template <int P, int R, int Ns, bool INV, int SRC, bool TO_S, int s, bool SCAN_LAST = false, class In, class Out>
__device__ __forceinline__ void fx_stage(const FxTile& t, unsigned* lanes, unsigned* words, In in, Out out) {
  constexpr int NB = fx_nb(R), nbf = P / R;
  constexpr bool TW = s > 0, SCAN = SCAN_LAST || s < fx_plan(P).n - 1;
  static_assert((s > 0) == (Ns > 1), "stage and product of earlier radices");
  const int total = nbf * t.W;
  const int lane = t.tid & (t.W - 1);
  cfx v[NB][R];
  int top = 0;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int idx = t.tid + b * t.nt, j = idx >> t.lw;
    if (idx < total) {
      if constexpr (SRC == FX_GAIN) top = max(top, in.products(ic<R>(), ic<nbf>(), j, lane, v[b]));
      else in(ic<R>(), ic<nbf>(), j, lane, v[b]);
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = fx_make(0, 0);
    }
  }
  if constexpr (SRC == FX_RAW || SRC == FX_RAW_DF) {
    const bool df = SRC == FX_RAW_DF && t.df;
    unsigned m = 0;
    if (df) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r)
          m = max(m, max(fx_mag_df(v[b][r].x), fx_mag_df(v[b][r].y)));
      m = (unsigned)fx_float_exp(m) << 20;
    } else {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r)
          m = max(m, max((unsigned)(v[b][r].x >> 32) & 0x7fffffffu, (unsigned)(v[b][r].y >> 32) & 0x7fffffffu));
    }
    lane_max(reinterpret_cast<int*>(lanes), m, t.W, lane, t.tid);
    __syncthreads();
    const int E = max((int)lanes[lane], kFxMinE);
    if (df) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = fx_make(fx_decode_df(v[b][r].x, E), fx_decode_df(v[b][r].y, E));
    } else {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = fx_make(fx_decode(v[b][r].x, E), fx_decode(v[b][r].y, E));
    }
  } else if constexpr (SRC == FX_GAIN) {
    lane_top(lanes, top, t.W, lane, t.tid);
    __syncthreads();
    const int T = (int)lanes[lane];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int idx = t.tid + b * t.nt, j = idx >> t.lw;
      if (idx < total) in.align(ic<R>(), ic<nbf>(), j, T, v[b]);
    }
  } else if constexpr (TO_S) {
    __syncthreads();  // every input is in registers before the tile is overwritten
  }
  if constexpr (TW) {
    const int n = fx_free_tw(words[(s - 1) * t.W + lane]);
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = fx_make(v[b][r].x << n, v[b][r].y << n);
  }
  unsigned mo = 0;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int idx = t.tid + b * t.nt, j = idx >> t.lw;
    if (idx < total) {
      const int k = TW ? j % Ns : 0;
      if constexpr (TW) {
        constexpr int tstep = (2 * P) / (Ns * R);
        v[b][0] = fx_make(fx_shr(v[b][0].x, kFxTwShift), fx_shr(v[b][0].y, kFxTwShift));
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = fx_cmul<INV>(v[b][r], fx_twiddle(t.tw, r * k * tstep));
      }
      fx_dft<R, INV>(v[b]);
      out(ic<R>(), ic<Ns>(), (j - k) * R + k, lane, v[b]);
      if constexpr (SCAN) {
#pragma unroll
        for (int r = 0; r < R; ++r) mo |= fx_mag(v[b][r].x) | fx_mag(v[b][r].y);
      }
    }
  }
  if constexpr (SCAN) lane_or(words + s * t.W, mo, t.W, lane, t.tid);
  if constexpr (TO_S) __syncthreads();
}

// Stages [s, s1) of the plan inside the tile (REV: radices in reverse order); words: the transform's slots.
// SCAN_LAST: the last stage's outputs are scanned too.
template <int P, class RW, bool INV, bool REV, int s, int s1, bool SCAN_LAST = false>
__device__ __forceinline__ void fx_mid_stages(const FxTile& t, unsigned* words) {
  if constexpr (s < s1) {
    constexpr FxPlan pl = fx_plan(P);
    constexpr int R = pl.r[REV ? pl.n - 1 - s : s], Ns = REV ? fx_prod(P, pl.n - s, pl.n) : fx_prod(P, 0, s);
    fx_stage<P, R, Ns, INV, FX_TILE, true, s, SCAN_LAST>(t, nullptr, words, FxFromS<RW>{t.S}, FxToS<RW>{t.S});
    fx_mid_stages<P, RW, INV, REV, s + 1, s1, SCAN_LAST>(t, words);
  }
}

// Green offset (axis term excluded) of pencil q, or, of a spectrum that is not stored, its partial |k|^2 (bits of a
// double); 0 past the last pencil.
__device__ __forceinline__ long long fx_green_base(const PassParams& p, int q, int o) {
  const FusedGreen& g = p.g;
  if (q >= p.npen) return 0;
  int c[3];
  if (p.axis == 0) { c[1] = q % g.dims1; c[2] = q / g.dims1; c[0] = 0; }
  else if (p.axis == 1) { c[0] = q; c[2] = o; c[1] = 0; }
  else { c[0] = q; c[1] = o; c[2] = 0; }
  const long long st[3] = {1, (long long)g.gpitch, (long long)g.gpitch * g.gext[1]};
  long long off = 0;
  double k2 = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d == p.axis) continue;
    int gi = c[d];
    if (g.fold[d]) gi = min(gi, g.fold[d] - gi);
    off += gi * st[d];
    if (!g.stored) k2 += ((const double*)g.tab[d])[gi];
  }
  return g.stored ? off : __double_as_longlong(k2);
}
// The tile's slice of a spectrum that is not stored: factors by folded mode, n pencils a row.
__device__ __noinline__ void fx_green_eval(const FusedGreen& g, int axis, const long long* base, unsigned long long* G,
                                           int n, int tid, int nt) {
  const double* tab = (const double*)g.tab[axis];
  for (int i = tid; i < g.gext[axis] * n; i += nt)
    G[i] = fx_green_pack((unsigned long long)__double_as_longlong(green_spectral(
                             __longlong_as_double(base[i % n]) + tab[i / n], g.kernel, g.eps2_half, g.scale)), g.ref);
}

// Green products of a complex lane in the first inverse stage: u^ = G^ f^.  g: the lane's factors by folded mode, gs
// apart, in the staged slice or in the stored spectrum; up: the modes' renormalisation.
template <int P, class RW> struct FxGained {
  const cfx* S;
  const unsigned long long* g;
  long long gs;
  int up;
  // factor of position j + r nbf: its own mode in the lower half, the mirrored one in the upper
  template <int R, int nbf, class F> __device__ __forceinline__ void each(int j, F f) const {
    const unsigned long long *lo = g + j * gs, *hi = g + (P - j) * gs;
    const long long step = nbf * gs;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool low = 2 * (r + 1) <= R || (2 * r < R && 2 * (j + r * nbf) <= P);
      f(r, low ? lo + r * step : hi - r * step);
    }
  }
  template <int R, int nbf> __device__ __forceinline__ int products(ic<R>, ic<nbf>, int j, int l, cfx* v) const {
    FxFromS<RW>{S}(ic<R>(), ic<nbf>(), j, l, v);
    int top = 0;
    each<R, nbf>(j, [&](int r, const unsigned long long* f) {
      const fxg q = fx_green(*f);
      v[r] = fx_make(fx_mul(v[r].x << up, q.h, q.l), fx_mul(v[r].y << up, q.h, q.l));
      top = max(top, fx_top_bit(v[r], q.d));
    });
    return top;
  }
  // (the orders are read again: kept, they would take a register per value)
  template <int R, int nbf> __device__ __forceinline__ void align(ic<R>, ic<nbf>, int j, int T, cfx* v) const {
    each<R, nbf>(j, [&](int r, const unsigned long long* f) {
      v[r] = fx_align(v[r], *reinterpret_cast<const int*>(f) & kFxGreenRange, T);
    });
  }
};

// Load of real data pairs whose extension is built in the tile (symmetric and semi-unbounded directions, and
// every real pass on pinned host arrays): items (lane, i < n_data), at most U per thread.  Values that the extension
// has no place for (odd node faces, the duplicate periodic node) count as 0 before the lane's exponent is taken.
template <int P, class RW, int U>
__device__ __forceinline__ void fx_load_ext(const PassParams& p, const FxTile& t, int type, const double* in, int q0,
                                            int* emax) {
  const int W = t.W, N = p.N, nd = p.n_data, tot = nd * W;
  const int bt = base_type(type);
  const bool rev = is_reversed(type), node = p.center == C_NODE;
  const int z0 = node && (bt == T_OO || bt == T_OE || bt == T_OU) ? 0 : -1;
  const int zN = node && (bt == T_OO || bt == T_EO || bt == T_PER) ? N : -1;
  cfx* S = t.S;
  double a[U], b[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int idx = t.tid + u * t.nt;
    a[u] = b[u] = 0.0;
    if (idx < tot) {
      const int l = p.fx_host ? idx / nd : idx & (W - 1), i = p.fx_host ? idx % nd : idx >> t.lw;
      const int qa = q0 + 2 * l;
      const long long off = (long long)qa * p.ai.ls + (long long)i * p.ai.js;
      const int dix = rev ? nd - 1 - i : i;
      const bool used = dix != z0 && dix != zN;
      if (used && qa < p.npen) a[u] = in[off];
      if (used && qa + 1 < p.npen) b[u] = in[off + p.ai.ls];
      if (p.fx_host) atomicMax(&emax[l], (int)(max(abs_hi(a[u]), abs_hi(b[u])) >> 20));
    }
  }
  // zero padding and odd faces
  int lo[3], hi[3];
  const int nz = zero_ranges(bt, p.center, N, lo, hi);
  for (int z = 0; z < nz; ++z)
    for (int idx = t.tid; idx < (min(hi[z], P) - lo[z]) * W; idx += t.nt)
      S[RW::at(lo[z] + (idx >> t.lw)) + (idx & (W - 1))] = fx_make(0, 0);
  if (!p.fx_host) {
    unsigned m = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) m = max(m, max(abs_hi(a[u]), abs_hi(b[u])));
    lane_max(emax, m, W, t.tid & (W - 1), t.tid);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int idx = t.tid + u * t.nt;
    if (idx >= tot) continue;
    const int l = p.fx_host ? idx / nd : idx & (W - 1), i = p.fx_host ? idx % nd : idx >> t.lw;
    const int E = max(emax[l], kFxMinE);
    const cfx v = fx_make(dec(a[u], E), dec(b[u], E));
    const int dix = rev ? nd - 1 - i : i;
    int pos[4], sg[4];
    const int n = images(bt, p.center, N, dix, pos, sg);
    for (int k = 0; k < n; ++k) S[RW::at(pos[k]) + l] = sg[k] > 0 ? v : fx_make(-v.x, -v.y);
  }
  __syncthreads();
}

// Forward transform of real data into the tile: pairs (row q0 + 2l, row q0 + 2l + 1).
template <int P, class RW, bool SCAN_LAST>
__device__ __forceinline__ void fx_forward_real(const PassParams& p, const FxTile& t, int type, const double* in,
                                                int q0, int* emax, unsigned* words) {
  constexpr FxPlan pl = fx_plan(P);
  if ((type == T_PER || type == T_UNB) && !p.fx_host) {
    // no images: the first stage reads its positions from memory
    const int nu = p.n_use, npen = p.npen;
    const long long ls = p.ai.ls, js = p.ai.js;
    fx_stage<P, pl.r[0], 1, false, FX_RAW, true, 0>(
        t, reinterpret_cast<unsigned*>(emax), words,
        [=](auto R, auto nbf, int j, int l, cfx* v) {
          const int qa = q0 + 2 * l;
          const double* r = in + (long long)qa * ls + (long long)j * js;
          const long long step = (long long)nbf.value * js;
          const int la = qa < npen ? nu - j : 0, lb = qa + 1 < npen ? nu - j : 0;
#pragma unroll
          for (int k = 0; k < R.value; ++k, r += step)
            v[k] = fx_make(k * nbf.value < la ? __double_as_longlong(r[0]) : 0,
                           k * nbf.value < lb ? __double_as_longlong(r[ls]) : 0);
        },
        FxToS<RW>{t.S});
  } else {
    if (p.n_data * t.W <= 9 * t.nt) fx_load_ext<P, RW, 9>(p, t, type, in, q0, emax);
    else fx_load_ext<P, RW, 19>(p, t, type, in, q0, emax);
    fx_stage<P, pl.r[0], 1, false, FX_TILE, true, 0>(t, nullptr, words, FxFromS<RW>{t.S}, FxToS<RW>{t.S});
  }
  fx_mid_stages<P, RW, false, false, 1, pl.n, SCAN_LAST>(t, words);
}

// Store of real data from the tile's last inverse stage; lane_q(l, &q, &kind): scale of lane l's values.
template <int P, class RW, class Q>
__device__ __forceinline__ void fx_store_real(const PassParams& p, const FxTile& t, int type, double* out, int q0,
                                              unsigned* words, Q lane_q) {
  constexpr FxPlan pl = fx_plan(P);
  constexpr int R = pl.r[pl.n - 1], Ns = P / R;
  const int nd = p.n_data, N = p.N;
  const int bt = base_type(type);
  const bool rev = is_reversed(type);
  const bool node = p.center == C_NODE;
  const bool odd0 = node && (bt == T_OO || bt == T_OE || bt == T_OU), oddN = node && (bt == T_OO || bt == T_EO);
  const bool dup = bt == T_PER && node && nd > N;
  const long long ls = p.ao.ls, js = p.ao.js;
  const int npen = p.npen;
  if (!p.fx_host) {
    fx_stage<P, R, Ns, true, FX_TILE, false, pl.n - 1>(
        t, nullptr, words, FxFromS<RW>{t.S}, [&](auto R_, auto Ns_, int o, int l, const cfx* v) {
          const int qa = q0 + 2 * l;
          if (qa >= npen) return;
          int q, kind;
          lane_q(l, &q, &kind);
          const bool two = qa + 1 < npen;
          double* d = out + (long long)qa * ls + (long long)(rev ? nd - 1 - o : o) * js;
          const long long step = (rev ? -(long long)Ns_.value : (long long)Ns_.value) * js;
          if (dup && o == 0) {  // phi_N := phi_0
            d[(long long)N * js] = enc_any(v[0].x, q, kind);
            if (two) d[(long long)N * js + ls] = enc_any(v[0].y, q, kind);
          }
          const int lim = (dup ? N : nd) - o;
          // odd node faces hold 0
          const int z0 = odd0 ? -o : -1, zN = oddN ? N - o : -1;
          if (kind == 0) {
#pragma unroll
            for (int r = 0; r < R_.value; ++r, d += step) {
              if (r * Ns_.value >= lim) continue;
              const bool z = r * Ns_.value == z0 || r * Ns_.value == zN;
              d[0] = z ? 0.0 : enc(v[r].x, q);
              if (two) d[ls] = z ? 0.0 : enc(v[r].y, q);
            }
          } else {
#pragma unroll
            for (int r = 0; r < R_.value; ++r, d += step) {
              if (r * Ns_.value >= lim) continue;
              const bool z = r * Ns_.value == z0 || r * Ns_.value == zN;
              d[0] = z ? 0.0 : enc_slow(v[r].x, q, kind);
              if (two) d[ls] = z ? 0.0 : enc_slow(v[r].y, q, kind);
            }
          }
        });
    return;
  }
  fx_stage<P, R, Ns, true, FX_TILE, true, pl.n - 1>(t, nullptr, words, FxFromS<RW>{t.S}, FxToS<RW>{t.S});
  for (int idx = t.tid; idx < nd * t.W; idx += t.nt) {
    const int l = idx / nd, i = idx % nd, qa = q0 + 2 * l;
    if (qa >= npen) continue;
    const int pos = dup && i == N ? 0 : (rev ? nd - 1 - i : i);
    const bool zero = (odd0 && pos == 0) || (oddN && pos == N);
    const cfx v = t.S[RW::at(pos) + l];
    int q, kind;
    lane_q(l, &q, &kind);
    double* d = out + (long long)qa * ls + (long long)i * js;
    d[0] = zero ? 0.0 : enc_any(v.x, q, kind);
    if (qa + 1 < npen) d[ls] = zero ? 0.0 : enc_any(v.y, q, kind);
  }
}

template <int KIND, int P>
__global__ void __launch_bounds__(512, 1) k_fx(const __grid_constant__ PassParams p) {
  pass_entry(p);
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr bool REAL = KIND == K_FWD_REAL || KIND == K_INV_REAL || KIND == K_FUSED_REAL;
  constexpr bool FUSED = KIND == K_FUSED_REAL || KIND == K_FUSED_C2C;
  using RW = FxRows<P, (KIND == K_FUSED_C2C ? FX_FUSED_C2C : FX_PLAIN)>;
  const FxSmem m = fx_smem(smraw, p.W, RW::size);
  const int tid = threadIdx.x, nt = blockDim.x;
  FxTile t;
  t.S = m.S;
  t.W = p.W;
  t.lw = p.lw;
  t.tid = tid;
  t.nt = nt;
  t.tw = (const fxw*)p.tw;
  t.df = p.fx_df & 1;
  constexpr FxPlan pl = fx_plan(P);
  constexpr int ns = pl.n, half = P / 2, R0 = pl.r[0], RL = pl.r[ns - 1];
  const int W = p.W;
  cfx* S = m.S;
  const int q0 = blockIdx.x * (REAL ? 2 * W : W);
  // fused pass: rows o and n - o share a Green slice and run back to back
  int o = blockIdx.y;
  if (KIND == K_FUSED_C2C && o > 0) o = (blockIdx.y & 1) ? (o + 1) / 2 : (int)gridDim.y - o / 2;
  const long long bi = (long long)o * p.ai.os + (long long)blockIdx.z * p.ai.cs;
  const long long bo = (long long)o * p.ao.os + (long long)blockIdx.z * p.ao.cs;
  const int type = comp_type(p, blockIdx.z);
  if (tid < W) m.emax[tid] = 0;
  for (int i = tid; i < kFxSlots * W; i += nt) m.words[i] = 0;
  unsigned* wf = m.words + kFxSlotFwd * W;
  unsigned* wi = m.words + kFxSlotInv * W;
  unsigned* wg = m.words + kFxSlotGain * W;
  unsigned* emax = reinterpret_cast<unsigned*>(m.emax);
  const bool tma_g = FUSED && p.gpre && p.gmap, eval_g = FUSED && !p.g.stored;
  if constexpr (FUSED) {
    for (int l = tid; l < (REAL ? 2 * W : W); l += nt) m.goff[l] = fx_green_base(p, q0 + l, o);
    if (tma_g && tid == 0) mbar_init(m.mbar, 1);
  }
  __syncthreads();
  if constexpr (FUSED) {
    if (eval_g) fx_green_eval(p.g, p.axis, m.goff, m.G, REAL ? 2 * W : W, tid, nt);
  }
  if (tma_g && tid == 0) {
    const FusedGreen& g = p.g;
    const int od = p.axis == 2 ? 1 : 2;  // the direction o runs along
    const int go = g.fold[od] ? min(o, g.fold[od] - o) : o;
    const char* maps = (const char*)p.gmap;
    mbar_expect_tx(m.mbar, (unsigned)((half + 1) * W * sizeof(long long)));
    for (int r0 = 0; r0 < half; r0 += p.gbox) {
      if (p.axis == 2) tma_load_3d(m.G + (size_t)r0 * W, maps, q0, go, r0, m.mbar);
      else tma_load_3d(m.G + (size_t)r0 * W, maps, q0, r0, go, m.mbar);
    }
    if (p.axis == 2) tma_load_3d(m.G + (size_t)half * W, maps + 128, q0, go, half, m.mbar);
    else tma_load_3d(m.G + (size_t)half * W, maps + 128, q0, half, go, m.mbar);
  }
  // exponent of a fixed-point value of lane l after the forward (or a single inverse) transform
  constexpr int shift = kFxTwShift * (ns - 1) - kFxBias;
  const FxFromS<RW> from_s{S};
  const FxToS<RW> to_s{S};

  if constexpr (KIND == K_FWD_REAL) {
    fx_forward_real<P, RW, false>(p, t, type, (const double*)p.in + bi, q0, m.emax, wf);
    const int bt = base_type(type);
    const bool cplx = bt == T_PER || bt == T_UNB, quarter = is_quarter(bt), oddo = is_odd_origin(bt);
    const bool cell = p.center == C_CELL;
    const int nm = p.n_modes, l = tid & (W - 1), qa = q0 + 2 * l;
    const int E = max(m.emax[l], kFxMinE);
    // the split leaves twice the modes; a phase costs 2^4, a quarter-wave type halves
    const int q = E + shift - fx_shifted<P>(m.words, W, l, true, false, false) - 1 + (cplx || !cell ? 0 : kFxTwShift) - (quarter ? 1 : 0);
    const int kind = fx_store_kind(p, E, q);
    if (qa < p.npen) {
      const bool two = qa + 1 < p.npen;
      for (int k = tid >> p.lw; k < nm; k += nt >> p.lw) {
        const int kk = quarter ? 2 * k + 1 : k, km = kk == 0 ? 0 : P - kk;
        const cfx zk = S[RW::at(kk) + l], zm = S[RW::at(km) + l];
        cfx A = fx_make(zk.x + zm.x, zk.y - zm.y), B = fx_make(zk.y + zm.y, zm.x - zk.x);
        const long long off = bo + (long long)qa * p.ao.ls + (long long)k * p.ao.js;
        if (cplx) {
          double2* out = (double2*)p.out;
          out[off] = make_double2(enc_any(A.x, q, kind), enc_any(A.y, q, kind));
          if (two) out[off + p.ao.ls] = make_double2(enc_any(B.x, q, kind), enc_any(B.y, q, kind));
        } else {
          double* out = (double*)p.out;
          if (cell) {
            const fxw w = fx_twiddle(t.tw, kk);
            A = fx_cmul<false>(A, w);
            B = fx_cmul<false>(B, w);
          }
          out[off] = enc_any(oddo ? -A.y : A.x, q, kind);
          if (two) out[off + p.ao.ls] = enc_any(oddo ? -B.y : B.x, q, kind);
        }
      }
    }
  } else if constexpr (KIND == K_INV_REAL) {
    const int bt = base_type(type);
    const bool cplx = bt == T_PER || bt == T_UNB, quarter = is_quarter(bt), oddo = is_odd_origin(bt);
    const bool cell = p.center == C_CELL;
    const int nm = p.n_modes, l = tid & (W - 1), qa = q0 + 2 * l;
    const bool ra = qa < p.npen, rb = qa + 1 < p.npen;
    // stored modes of both pencils: at most 10 per thread (the host sizes the block)
    constexpr int U = 10;
    double ax[U], ay[U], bx[U], by[U];
    const long long offl = bi + (long long)qa * p.ai.ls;
    unsigned mx = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = (tid + u * nt) >> p.lw;
      ax[u] = ay[u] = bx[u] = by[u] = 0.0;
      if (k < nm) {
        const long long off = offl + (long long)k * p.ai.js;
        if (cplx) {
          const double2* in = (const double2*)p.in;
          const bool real_mode = k == 0 || 2 * k == P;
          if (ra) {
            const double2 c = in[off];
            ax[u] = c.x;
            ay[u] = real_mode ? 0.0 : c.y;
          }
          if (rb) {
            const double2 c = in[off + p.ai.ls];
            bx[u] = c.x;
            by[u] = real_mode ? 0.0 : c.y;
          }
        } else {
          const double* in = (const double*)p.in;
          if (ra) ax[u] = in[off];
          if (rb) bx[u] = in[off + p.ai.ls];
        }
      }
      if (!t.df) mx = max(max(mx, max(abs_hi(ax[u]), abs_hi(ay[u]))), max(abs_hi(bx[u]), abs_hi(by[u])));
    }
    if (t.df) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        mx = max(max(mx, max(fx_mag_df(__double_as_longlong(ax[u])), fx_mag_df(__double_as_longlong(ay[u])))),
                 max(fx_mag_df(__double_as_longlong(bx[u])), fx_mag_df(__double_as_longlong(by[u]))));
      mx = (unsigned)fx_float_exp(mx) << 20;
    }
    lane_max(m.emax, mx, W, l, tid);
    if (quarter)  // even modes of the quarter-wave types are zero
      for (int idx = tid; idx < half * W; idx += nt) S[RW::at(2 * (idx >> p.lw)) + (idx & (W - 1))] = fx_make(0, 0);
    __syncthreads();
    const int E = max(m.emax[l], kFxMinE);
    // the half-sample phase divides by 2^4: such coefficients keep 4 more bits
    const int up = kFxUp + (cplx || !cell ? 0 : kFxTwShift);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = (tid + u * nt) >> p.lw;
      if (k >= nm) continue;
      const int kk = quarter ? 2 * k + 1 : k;
      cfx A, B;
      if (t.df) {
        A = fx_make(dec_df(ax[u], E, up), dec_df(ay[u], E, up));
        B = fx_make(dec_df(bx[u], E, up), dec_df(by[u], E, up));
      } else {
        A = fx_make(dec(ax[u], E, up), dec(ay[u], E, up));
        B = fx_make(dec(bx[u], E, up), dec(by[u], E, up));
      }
      if (!cplx) {
        if (oddo) {
          A = fx_make(0, -A.x);
          B = fx_make(0, -B.x);
        }
        if (cell) {
          const fxw w = fx_twiddle(t.tw, kk);
          A = fx_cmul<true>(A, w);
          B = fx_cmul<true>(B, w);
        }
      }
      S[RW::at(kk) + l] = fx_make(A.x - B.y, A.y + B.x);
      if (kk != 0 && 2 * kk != P) S[RW::at(P - kk) + l] = fx_make(A.x + B.y, B.x - A.y);
    }
    __syncthreads();
    fx_stage<P, R0, 1, true, FX_TILE, true, 0>(t, nullptr, wi, from_s, to_s);
    fx_mid_stages<P, RW, true, false, 1, ns - 1>(t, wi);
    const int add = shift + (quarter ? 1 : 0);
    fx_store_real<P, RW>(p, t, type, (double*)p.out + bo, q0, wi, [&](int lane, int* q, int* kind) {
      const int Ee = max(m.emax[lane], kFxMinE);
      *q = Ee + add - fx_shifted<P>(m.words, W, lane, false, false, true);
      *kind = fx_out_kind(Ee, *q);
    });
  } else if constexpr (KIND == K_FUSED_REAL) {
    fx_forward_real<P, RW, true>(p, t, type, (const double*)p.in + bi, q0, m.emax, wf);
    const bool quarter = is_quarter(base_type(type));
    {
      // the two pencils' products in place of the packed modes k and P - k, then, aligned, packed again
      const int l = tid & (W - 1), upx = fx_free_tw(wf[(ns - 1) * W + l]);
      const long long st3 = p.axis == 0 ? 1 : (p.axis == 1 ? (long long)p.g.gpitch : (long long)p.g.gpitch * p.g.gext[1]);
      const unsigned long long* Ga = eval_g ? m.G + 2 * l : (const unsigned long long*)p.g.stored + m.goff[2 * l];
      const unsigned long long* Gb = eval_g ? Ga + 1 : (const unsigned long long*)p.g.stored + m.goff[2 * l + 1];
      const long long gs = eval_g ? 2 * W : st3;
      int top = 0;
      for (int k = tid >> p.lw; k <= half; k += nt >> p.lw) {
        if (quarter && !(k & 1)) continue;
        const int km = k == 0 ? 0 : P - k;
        cfx zk = S[RW::at(k) + l], zm = S[RW::at(km) + l];
        zk = fx_make(zk.x << upx, zk.y << upx);
        zm = fx_make(zm.x << upx, zm.y << upx);
        const long long o3 = (quarter ? (k - 1) >> 1 : k) * gs;
        const fxg fa = fx_green(Ga[o3]), fb = fx_green(Gb[o3]);
        const cfx A = fx_make(fx_mul(zk.x + zm.x, fa.h, fa.l), fx_mul(zk.y - zm.y, fa.h, fa.l));
        const cfx B = fx_make(fx_mul(zk.y + zm.y, fb.h, fb.l), fx_mul(zm.x - zk.x, fb.h, fb.l));
        top = max(top, max(fx_top_bit(A, fa.d), fx_top_bit(B, fb.d)));
        // modes 0 and P/2 are real
        if (km == k) {
          S[RW::at(k) + l] = fx_make(A.x, B.x);
        } else {
          S[RW::at(k) + l] = A;
          S[RW::at(km) + l] = B;
        }
      }
      lane_top(wg, top, W, l, tid);
      __syncthreads();
      const int T = (int)wg[l];
      for (int k = tid >> p.lw; k <= half; k += nt >> p.lw) {
        const int km = k == 0 ? 0 : P - k;
        cfx A = fx_make(0, 0), B = A;
        if (!quarter || (k & 1)) {
          const long long o3 = (quarter ? (k - 1) >> 1 : k) * gs;
          A = S[RW::at(k) + l];
          if (km == k) {
            B.x = A.y;
            A.y = 0;
          } else {
            B = S[RW::at(km) + l];
          }
          A = fx_align(A, (int)Ga[o3] & kFxGreenRange, T);
          B = fx_align(B, (int)Gb[o3] & kFxGreenRange, T);
        }
        S[RW::at(k) + l] = fx_make(A.x - B.y, A.y + B.x);
        if (km != k) S[RW::at(km) + l] = fx_make(A.x + B.y, B.x - A.y);
      }
    }
    __syncthreads();
    fx_stage<P, R0, 1, true, FX_TILE, true, 0>(t, nullptr, wi, from_s, to_s);
    fx_mid_stages<P, RW, true, false, 1, ns - 1>(t, wi);
    fx_store_real<P, RW>(p, t, type, (double*)p.out + bo, q0, wi, [&](int lane, int* q, int* kind) {
      const int Ee = max(m.emax[lane], kFxMinE);
      *q = Ee - fx_shifted<P>(m.words, W, lane, true, true, true) + 2 * shift + kFxBias - 1 +
           fx_align_exp((int)wg[lane], p.g.gref ? *p.g.gref : p.g.ref);
      *kind = fx_out_kind(Ee, *q);
    });
  } else {
    // complex passes
    const double2* in = (const double2*)p.in + bi;
    double2* out = (double2*)p.out + bo;
    const int npen = p.npen, n_in = KIND == K_INV_C2C ? P : p.n_use;
    const long long ils = p.ai.ls, ijs = p.ai.js, ols = p.ao.ls, ojs = p.ao.js;
    auto load = [=](auto R, auto nbf, int j, int l, cfx* v) {
      const longlong2* c = reinterpret_cast<const longlong2*>(in) + (long long)(q0 + l) * ils + (long long)j * ijs;
      const long long step = (long long)nbf.value * ijs;
      const int lim = q0 + l < npen ? n_in - j : 0;
#pragma unroll
      for (int r = 0; r < R.value; ++r, c += step) {
        longlong2 x = make_longlong2(0, 0);
        if (r * nbf.value < lim) x = *c;
        v[r] = fx_make(x.x, x.y);
      }
    };
    const int l0 = tid & (W - 1);
    const int n_out = KIND == K_FWD_C2C ? P : p.n_data;
    // node-centred periodic: phi_N := phi_0
    const int dup = (KIND != K_FWD_C2C && p.type == T_PER && p.center == C_NODE && p.n_data > p.N) ? p.N : -1;
    int q = 0, kind = 0;
    bool store_ok = true;
    auto store = [&](auto R, auto Ns, int o, int l, const cfx* v) {
      if (q0 + l >= npen || !store_ok) return;
      double2* d = out + (long long)(q0 + l) * ols + (long long)o * ojs;
      const long long step = (long long)Ns.value * ojs;
      const int lim = n_out - o;
      if (dup >= 0 && o == 0) d[(long long)dup * ojs] = make_double2(enc_any(v[0].x, q, kind), enc_any(v[0].y, q, kind));
      if (kind == 0) {
#pragma unroll
        for (int r = 0; r < R.value; ++r, d += step)
          if (r * Ns.value < lim) *d = make_double2(enc(v[r].x, q), enc(v[r].y, q));
      } else if (KIND == K_FWD_C2C && kind == 3) {
#pragma unroll
        for (int r = 0; r < R.value; ++r, d += step)
          if (r * Ns.value < lim) *d = make_double2(enc_df(v[r].x, q), enc_df(v[r].y, q));
      } else {
#pragma unroll
        for (int r = 0; r < R.value; ++r, d += step)
          if (r * Ns.value < lim) *d = make_double2(enc_slow(v[r].x, q, kind), enc_slow(v[r].y, q, kind));
      }
    };
    if constexpr (KIND == K_FUSED_C2C) {
      fx_stage<P, R0, 1, false, FX_RAW, true, 0>(t, emax, wf, load, to_s);
      fx_mid_stages<P, RW, false, false, 1, ns, true>(t, wf);
      // u^ = G^ f^ in the first inverse stage (radices reversed)
      if (tma_g) {
        if (!mbar_wait_bounded(m.mbar, p.errflag, 1, p.dbg_wait & 1)) store_ok = false;
      }
      const long long go = m.goff[l0];
      const long long st3 = p.axis == 0 ? 1 : (p.axis == 1 ? (long long)p.g.gpitch : (long long)p.g.gpitch * p.g.gext[1]);
      const bool staged = tma_g || eval_g;
      const FxGained<P, RW> gained{S, staged ? m.G + l0 : (const unsigned long long*)p.g.stored + go,
                                   staged ? (long long)W : st3, fx_free_tw(wf[(ns - 1) * W + l0])};
      fx_stage<P, RL, 1, true, FX_GAIN, true, 0>(t, wg, wi, gained, to_s);
      fx_mid_stages<P, RW, true, true, 1, ns - 1>(t, wi);
      const int E = max(m.emax[l0], kFxMinE);
      q = E - fx_shifted<P>(m.words, W, l0, true, true, true) + 2 * shift + kFxBias + 
          fx_align_exp((int)wg[l0], p.g.gref ? *p.g.gref : p.g.ref);
      kind = fx_out_kind(E, q);
      fx_stage<P, R0, P / R0, true, FX_TILE, false, ns - 1>(t, nullptr, wi, from_s, store);
    } else {
      constexpr bool INV = KIND == K_INV_C2C;
      fx_stage<P, R0, 1, INV, INV ? FX_RAW_DF : FX_RAW, true, 0>(t, emax, wf, load, to_s);
      fx_mid_stages<P, RW, INV, false, 1, ns - 1>(t, wf);
      const int E = max(m.emax[l0], kFxMinE);
      q = E + shift - fx_shifted<P>(m.words, W, l0, true, false, false);
      kind = INV ? fx_out_kind(E, q) : fx_store_kind(p, E, q);
      fx_stage<P, RL, P / RL, INV, FX_TILE, false, ns - 1>(t, nullptr, wf, from_s, store);
    }
  }
}

}  // namespace

template <int KIND, int P>
cudaError_t fx_launch(const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)nthr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = p.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_fx<KIND, P>, p);
}

template <int P>
cudaError_t fx_launch_kind(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
  switch (kind) {
    case K_FWD_REAL: return fx_launch<K_FWD_REAL, P>(p, grid, nthr, smem, st);
    case K_INV_REAL: return fx_launch<K_INV_REAL, P>(p, grid, nthr, smem, st);
    case K_FWD_C2C: return fx_launch<K_FWD_C2C, P>(p, grid, nthr, smem, st);
    case K_INV_C2C: return fx_launch<K_INV_C2C, P>(p, grid, nthr, smem, st);
    case K_FUSED_REAL: return fx_launch<K_FUSED_REAL, P>(p, grid, nthr, smem, st);
    case K_FUSED_C2C: return fx_launch<K_FUSED_C2C, P>(p, grid, nthr, smem, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int KIND, int P> cudaError_t fx_limit() {
  return cudaFuncSetAttribute(k_fx<KIND, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}
template <int P> cudaError_t fx_limit_kind(int kind) {
  switch (kind) {
    case K_FWD_REAL: return fx_limit<K_FWD_REAL, P>();
    case K_INV_REAL: return fx_limit<K_INV_REAL, P>();
    case K_FWD_C2C: return fx_limit<K_FWD_C2C, P>();
    case K_INV_C2C: return fx_limit<K_INV_C2C, P>();
    case K_FUSED_REAL: return fx_limit<K_FUSED_REAL, P>();
    case K_FUSED_C2C: return fx_limit<K_FUSED_C2C, P>();
    default: return cudaErrorInvalidValue;
  }
}

#define FX_LAUNCH_CASE(P) \
  case P: return fx_launch_kind<P>(kind, p, grid, nthr, smem, st);
#define FX_LIMIT_CASE(P) \
  case P: return fx_limit_kind<P>(kind);
// Launcher and shared-memory limits of the lengths of FX_SHARD_<i>.
#define FX_UNIT(i)                                                                                              \
  namespace flups {                                                                                             \
  cudaError_t launch_fx_##i(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) { \
    switch (p.P) { FX_SHARD_##i(FX_LAUNCH_CASE) }                                                               \
    return cudaErrorInvalidValue;                                                                               \
  }                                                                                                             \
  cudaError_t limit_fx_##i(int kind, int P) {                                                                   \
    switch (P) { FX_SHARD_##i(FX_LIMIT_CASE) }                                                                  \
    return cudaErrorInvalidValue;                                                                               \
  }                                                                                                             \
  }

}  // namespace flups
