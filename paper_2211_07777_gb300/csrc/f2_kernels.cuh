// FP32 passes on pairs of lanes in packed arithmetic (f2.cuh): one kernel per pass kind and length
// P = 2^a 3^b (plans of fx_plan.cuh), for every axis and tile width.
//
// A CTA holds W lanes x P values of 16 bytes in shared memory, a value being one position of two complex
// sequences: two neighbouring pencils of a complex pass, or four real pencils q .. q + 3 packed as
// q + i (q + 2) and (q + 1) + i (q + 3).  The tile is transformed in place, whole butterflies in registers between two
// barriers (one of up to 9 values a thread where three such stages make the length, else, and in the Biot-Savart pass,
// up to 18 values: fx_plan.cuh); complex passes and the real passes of periodic and unbounded directions
// read the first stage's inputs from memory and store the last stage's outputs from registers.
#pragma once
#include <cuda_runtime.h>

#include "f2.cuh"
#include "fx_plan.cuh"
#include "pass_common.cuh"
#include "passes.cuh"

namespace flups {

namespace {

// Threads a kernel is compiled for: the block of a full tile, rounded up (small grids take at most 256)
template <int P> struct F2Block {
  static constexpr int n = (P * fx_width(FX_PLAIN, P) + f2_ept(FX_PLAIN, P) - 1) / f2_ept(FX_PLAIN, P);
  static constexpr int threads = n <= 256 ? 256 : (n <= 512 ? 512 : 768);
  static_assert(n <= 768, "threads of a tile");
};

template <int N> using ic2 = std::integral_constant<int, N>;

// A tile's shared memory: the 128-byte block of its mbarrier, the tile, the pencils' Green offsets and partial
// |k|^2, then the staged Green slice (128-byte aligned).
struct F2Smem {
  cf2* S;
  long long* goff;   // 4 W
  float* k2p;        // 4 W
  unsigned long long* mbar;
  float* G;          // (P/2 + 1) x 2 W
};
__device__ __forceinline__ F2Smem f2_smem(unsigned char* smraw, int W, int rows) {
  F2Smem m;
  unsigned char* base = smraw + ((128u - (smem_u32(smraw) & 127u)) & 127u);
  m.mbar = reinterpret_cast<unsigned long long*>(base);
  m.S = reinterpret_cast<cf2*>(base + 128);
  m.goff = reinterpret_cast<long long*>(base + 128 + (size_t)rows * sizeof(cf2));
  m.k2p = reinterpret_cast<float*>(m.goff + 4 * W);
  unsigned char* g = reinterpret_cast<unsigned char*>(m.k2p + 4 * W);
  m.G = reinterpret_cast<float*>(g + ((128u - (smem_u32(g) & 127u)) & 127u));
  return m;
}

struct F2Tile {
  cf2* S;
  int W, lw, tid, nt;
  const f2w* tw;
};
__device__ __forceinline__ f2w f2_twiddle(const f2w* tw, int i) {
  const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2*>(tw + i));
  f2w w;
  w.c = q.x;
  w.s = q.y;
  return w;
}
// Values j + r nbf of a butterfly from the tile, and its outputs o + r Ns into it
template <class RW> struct F2FromS {
  const cf2* S;
  template <int R, int nbf> __device__ __forceinline__ void operator()(ic2<R>, ic2<nbf>, int j, int l, cf2* v) const {
    const cf2* s = S + RW::at(j) + l;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (RW::linear(nbf)) v[r] = s[RW::at(r * nbf)];
      else v[r] = S[RW::at(j + r * nbf) + l];
    }
  }
};
template <class RW> struct F2ToS {
  cf2* S;
  template <int R, int Ns> __device__ __forceinline__ void operator()(ic2<R>, ic2<Ns>, int o, int l, const cf2* v) const {
    cf2* s = S + RW::at(o) + l;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (RW::linear(Ns) || (Ns == 1 && R == RW::B)) s[RW::at(r * Ns)] = v[r];
      else S[RW::at(o + r * Ns) + l] = v[r];
    }
  }
};

// One stage of radix R after a product Ns of earlier radices.  FROM_S: the inputs are the tile, which TO_S
// overwrites.
template <int P, class RW, int R, int Ns, bool INV, bool FROM_S, bool TO_S, class In, class Out>
__device__ __forceinline__ void f2_stage(const F2Tile& t, In in, Out out) {
  constexpr int NB = RW::nb(R), nbf = P / R;
  const int total = nbf * t.W;
  const int lane = t.tid & (t.W - 1);
  cf2 v[NB][R];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int idx = t.tid + b * t.nt, j = idx >> t.lw;
    if (idx < total) in(ic2<R>(), ic2<nbf>(), j, lane, v[b]);
  }
  if constexpr (FROM_S && TO_S) __syncthreads();
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int idx = t.tid + b * t.nt, j = idx >> t.lw;
    if (idx < total) {
      const int k = Ns > 1 ? j % Ns : 0;
      if constexpr (Ns > 1) {
        constexpr int tstep = (2 * P) / (Ns * R);
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const f2w w = f2_twiddle(t.tw, r * k * tstep);
          v[b][r] = f2_cmul<INV>(v[b][r], w.c, w.s);
        }
      }
      f2_dft<R, INV>(v[b]);
      out(ic2<R>(), ic2<Ns>(), (j - k) * R + k, lane, v[b]);
    }
  }
  if constexpr (TO_S) __syncthreads();
}

// Stages [s, s1) of the plan inside the tile (REV: radices in reverse order).
template <int P, class RW, bool INV, bool REV, int s, int s1>
__device__ __forceinline__ void f2_mid_stages(const F2Tile& t) {
  if constexpr (s < s1) {
    constexpr F2Plan pl = RW::plan;
    constexpr int R = pl.r[REV ? pl.n - 1 - s : s], Ns = REV ? RW::prod(pl.n - s, pl.n) : RW::prod(0, s);
    f2_stage<P, RW, R, Ns, INV, true, true>(t, F2FromS<RW>{t.S}, F2ToS<RW>{t.S});
    f2_mid_stages<P, RW, INV, REV, s + 1, s1>(t);
  }
}

// Four real values of pencils q .. q + 3 (zero past the last pencil).  vec: the array's pencils are adjacent and
// groups of four are 16-byte aligned and inside its rows.
__device__ __forceinline__ cf2 f2_load4(const float* in, long long ls, int q, int npen, bool vec) {
  float a[4];
  if (vec) {
    const float4 f = *reinterpret_cast<const float4*>(in);
    a[0] = f.x;
    a[1] = q + 1 < npen ? f.y : 0.f;
    a[2] = q + 2 < npen ? f.z : 0.f;
    a[3] = q + 3 < npen ? f.w : 0.f;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = q + i < npen ? in[i * ls] : 0.f;
  }
  return f2_make(f2_pack(a[0], a[1]), f2_pack(a[2], a[3]));
}
__device__ __forceinline__ void f2_store4(float* out, long long ls, int q, int npen, bool vec, cf2 v) {
  const float2 a = f2_get(v.x), b = f2_get(v.y);
  if (vec && q + 3 < npen) {
    *reinterpret_cast<float4*>(out) = make_float4(a.x, a.y, b.x, b.y);
  } else {
    out[0] = a.x;
    if (q + 1 < npen) out[ls] = a.y;
    if (q + 2 < npen) out[2 * ls] = b.x;
    if (q + 3 < npen) out[3 * ls] = b.y;
  }
}
// Two complex values of pencils q, q + 1
__device__ __forceinline__ cf2 f2_load2(const float2* in, long long ls, int q, int npen, bool vec) {
  float2 a = make_float2(0.f, 0.f), b = a;
  if (vec) {
    const float4 f = *reinterpret_cast<const float4*>(in);
    a = make_float2(f.x, f.y);
    b = make_float2(f.z, f.w);
  } else {
    a = in[0];
  }
  if (q + 1 >= npen) b = make_float2(0.f, 0.f);
  else if (!vec) b = in[ls];
  return f2_make(f2_pack(a.x, b.x), f2_pack(a.y, b.y));
}
__device__ __forceinline__ void f2_store2(float2* out, long long ls, int q, int npen, bool vec, cf2 v) {
  const float2 x = f2_get(v.x), y = f2_get(v.y);
  if (vec && q + 1 < npen) {
    *reinterpret_cast<float4*>(out) = make_float4(x.x, y.x, x.y, y.y);
  } else {
    out[0] = make_float2(x.x, y.x);
    if (q + 1 < npen) out[ls] = make_float2(x.y, y.y);
  }
}

// Real data of symmetric and semi-unbounded directions (and of every direction on pinned host arrays): the
// periodic extension is built in the tile.
template <int P, class RW>
__device__ __forceinline__ void f2_load_ext(const PassParams& p, const F2Tile& t, int type, const float* in, int q0) {
  const int W = t.W, N = p.N, nd = p.n_data, tot = nd * W;
  const int bt = base_type(type);
  const bool rev = is_reversed(type);
  cf2* S = t.S;
  int lo[3], hi[3];
  const int nz = zero_ranges(bt, p.center, N, lo, hi);
  for (int z = 0; z < nz; ++z)
    for (int idx = t.tid; idx < (min(hi[z], P) - lo[z]) * W; idx += t.nt)
      S[RW::at(lo[z] + (idx >> t.lw)) + (idx & (W - 1))] = f2_make(0, 0);
  constexpr int U = 4;
  for (int base = t.tid; base < tot; base += U * t.nt) {
    cf2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * t.nt;
      if (idx >= tot) continue;
      const int l = p.fx_host ? idx / nd : idx & (W - 1), i = p.fx_host ? idx % nd : idx >> t.lw;
      const int q = q0 + 4 * l;
      v[u] = f2_make(0, 0);
      if (q < p.npen) v[u] = f2_load4(in + (long long)q * p.ai.ls + (long long)i * p.ai.js, p.ai.ls, q, p.npen, p.f2_vec & 1);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * t.nt;
      if (idx >= tot) continue;
      const int l = p.fx_host ? idx / nd : idx & (W - 1), i = p.fx_host ? idx % nd : idx >> t.lw;
      const int dix = rev ? nd - 1 - i : i;
      int pos[4], sg[4];
      const int n = images(bt, p.center, N, dix, pos, sg);
      for (int k = 0; k < n; ++k) S[RW::at(pos[k]) + l] = sg[k] > 0 ? v[u] : f2_make(f2_neg(v[u].x), f2_neg(v[u].y));
    }
  }
  __syncthreads();
}

// Forward transform of real data into the tile.
template <int P, class RW>
__device__ __forceinline__ void f2_forward_real(const PassParams& p, const F2Tile& t, int type, const float* in, int q0) {
  constexpr F2Plan pl = RW::plan;
  if ((type == T_PER || type == T_UNB) && !p.fx_host) {
    const int nu = p.n_use, npen = p.npen;
    const long long ls = p.ai.ls, js = p.ai.js;
    const bool vec = p.f2_vec & 1;
    f2_stage<P, RW, pl.r[0], 1, false, false, true>(
        t,
        [=](auto R, auto nbf, int j, int l, cf2* v) {
          const int q = q0 + 4 * l;
          const float* r = in + (long long)q * ls + (long long)j * js;
          const long long step = (long long)nbf.value * js;
          const int lim = q < npen ? nu - j : 0;
#pragma unroll
          for (int k = 0; k < R.value; ++k, r += step) {
            v[k] = f2_make(0, 0);
            if (k * nbf.value < lim) v[k] = f2_load4(r, ls, q, npen, vec);
          }
        },
        F2ToS<RW>{t.S});
  } else {
    f2_load_ext<P, RW>(p, t, type, in, q0);
    f2_stage<P, RW, pl.r[0], 1, false, true, true>(t, F2FromS<RW>{t.S}, F2ToS<RW>{t.S});
  }
  f2_mid_stages<P, RW, false, false, 1, pl.n>(t);
}

// Store of real data from the tile's last inverse stage.
template <int P, class RW>
__device__ __forceinline__ void f2_store_real(const PassParams& p, const F2Tile& t, int type, float* out, int q0) {
  constexpr F2Plan pl = RW::plan;
  constexpr int R = pl.r[pl.n - 1], Ns = P / R;
  const int nd = p.n_data, N = p.N;
  const int bt = base_type(type);
  const bool rev = is_reversed(type);
  const bool node = p.center == C_NODE;
  const bool odd0 = node && (bt == T_OO || bt == T_OE || bt == T_OU), oddN = node && (bt == T_OO || bt == T_EO);
  const bool dup = bt == T_PER && node && nd > N;
  const long long ls = p.ao.ls, js = p.ao.js;
  const int npen = p.npen;
  const bool vec = p.f2_vec & 2;
  if (!p.fx_host) {
    f2_stage<P, RW, R, Ns, true, true, false>(
        t, F2FromS<RW>{t.S}, [&](auto R_, auto Ns_, int o, int l, const cf2* v) {
          const int q = q0 + 4 * l;
          if (q >= npen) return;
          float* d = out + (long long)q * ls + (long long)(rev ? nd - 1 - o : o) * js;
          const long long step = (rev ? -(long long)Ns_.value : (long long)Ns_.value) * js;
          if (dup && o == 0) f2_store4(d + (long long)N * js, ls, q, npen, vec, v[0]);  // phi_N := phi_0
          const int lim = (dup ? N : nd) - o;
          const int z0 = odd0 ? -o : -1, zN = oddN ? N - o : -1;  // odd node faces hold 0
#pragma unroll
          for (int r = 0; r < R_.value; ++r, d += step) {
            if (r * Ns_.value >= lim) continue;
            const bool z = r * Ns_.value == z0 || r * Ns_.value == zN;
            f2_store4(d, ls, q, npen, vec, z ? f2_make(0, 0) : v[r]);
          }
        });
    return;
  }
  f2_stage<P, RW, R, Ns, true, true, true>(t, F2FromS<RW>{t.S}, F2ToS<RW>{t.S});
  for (int idx = t.tid; idx < nd * t.W; idx += t.nt) {
    const int l = idx / nd, i = idx % nd, q = q0 + 4 * l;
    if (q >= npen) continue;
    const int pos = dup && i == N ? 0 : (rev ? nd - 1 - i : i);
    const bool zero = (odd0 && pos == 0) || (oddN && pos == N);
    f2_store4(out + (long long)q * ls + (long long)i * js, ls, q, npen, false, zero ? f2_make(0, 0) : t.S[RW::at(pos) + l]);
  }
}

// G^ of two pencils at folded mode g3: stored spectrum or closed form
__device__ __forceinline__ f2 f2_green2(const FusedGreen& g, int axis, const long long* goff, const float* k2p, int g3,
                                        long long st3) {
  float a, b;
  if (g.stored) {
    const float* G = (const float*)g.stored;
    a = __ldg(&G[goff[0] + g3 * st3]);
    b = __ldg(&G[goff[1] + g3 * st3]);
  } else {
    const float t3 = ((const float*)g.tab[axis])[g3];
    float k[2] = {k2p[0] + t3, k2p[1] + t3};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float k2 = k[i], sc = (float)g.scale;
      float v = 0.f;
      if (k2 > 0.f) {
        v = -sc / k2;
        if (g.kernel != 0 && g.kernel != 100) {
          const float s = k2 * (float)g.eps2_half;
          float acc = 1.f, term = 1.f;
          for (int m = 1; m < g.kernel / 2; ++m) {
            term = term * s / (float)m;
            acc += term;
          }
          v = -sc * expf(-s) * acc / k2;
        }
      }
      k[i] = v;
    }
    a = k[0];
    b = k[1];
  }
  return f2_pack(a, b);
}

// Green offset (axis term excluded) and partial |k|^2 of pencil q; zeros past the last pencil.
__device__ __forceinline__ void f2_green_base(const PassParams& p, int q, int o, long long* goff, float* k2p) {
  const FusedGreen& g = p.g;
  long long off = 0;
  float k2 = 0.f;
  if (q < p.npen) {
    int c[3];
    if (p.axis == 0) { c[1] = q % g.dims1; c[2] = q / g.dims1; c[0] = 0; }
    else if (p.axis == 1) { c[0] = q; c[2] = o; c[1] = 0; }
    else { c[0] = q; c[1] = o; c[2] = 0; }
    const long long st[3] = {1, (long long)g.gpitch, (long long)g.gpitch * g.gext[1]};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (d == p.axis) continue;
      int gi = c[d];
      if (g.fold[d]) gi = min(gi, g.fold[d] - gi);
      off += gi * st[d];
      if (!g.stored) k2 += ((const float*)g.tab[d])[gi];
    }
  }
  *goff = off;
  *k2p = k2;
}

// Spectra of the pencils packed in the real and imaginary parts, from modes k and P - k: twice their values
__device__ __forceinline__ void f2_split(cf2 zk, cf2 zm, cf2& A, cf2& B) {
  A = f2_make(f2_add(zk.x, zm.x), f2_sub(zk.y, zm.y));
  B = f2_make(f2_add(zk.y, zm.y), f2_sub(zm.x, zk.x));
}

template <int KIND, int P>
__global__ void __launch_bounds__(F2Block<P>::threads, 768 / F2Block<P>::threads) k_f2(const __grid_constant__ PassParams p) {
  pass_entry(p);
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr bool REAL = KIND == K_FWD_REAL || KIND == K_INV_REAL || KIND == K_FUSED_REAL;
  constexpr bool FUSED = KIND == K_FUSED_REAL || KIND == K_FUSED_C2C;
  using RW = F2Rows<P, FX_PLAIN>;
  constexpr F2Plan pl = RW::plan;
  constexpr int ns = pl.n, half = P / 2, R0 = pl.r[0], RL = pl.r[ns - 1];
  const int W = p.W;
  const F2Smem m = f2_smem(smraw, W, RW::size);
  const int tid = threadIdx.x, nt = blockDim.x;
  const F2Tile t{m.S, W, p.lw, tid, nt, (const f2w*)p.tw};
  cf2* S = m.S;
  const int q0 = blockIdx.x * (REAL ? 4 * W : 2 * W);
  // fused pass: rows o and n - o share a Green slice and run back to back
  int o = blockIdx.y;
  if (KIND == K_FUSED_C2C && o > 0) o = (blockIdx.y & 1) ? (o + 1) / 2 : (int)gridDim.y - o / 2;
  const long long bi = (long long)o * p.ai.os + (long long)blockIdx.z * p.ai.cs;
  const long long bo = (long long)o * p.ao.os + (long long)blockIdx.z * p.ao.cs;
  const int type = comp_type(p, blockIdx.z);
  const bool tma_g = FUSED && p.gpre && p.gmap;
  if constexpr (FUSED) {
    for (int l = tid; l < (REAL ? 4 * W : 2 * W); l += nt) f2_green_base(p, q0 + l, o, &m.goff[l], &m.k2p[l]);
    if (tma_g && tid == 0) mbar_init(m.mbar, 1);
    __syncthreads();
    if (tma_g && tid == 0) {
      const FusedGreen& g = p.g;
      const int od = p.axis == 2 ? 1 : 2;  // the direction o runs along
      const int go = g.fold[od] ? min(o, g.fold[od] - o) : o;
      const char* maps = (const char*)p.gmap;
      const int GW = 2 * W;
      mbar_expect_tx(m.mbar, (unsigned)((half + 1) * GW * sizeof(float)));
      for (int r0 = 0; r0 < half; r0 += p.gbox) {
        if (p.axis == 2) tma_load_3d(m.G + (size_t)r0 * GW, maps, q0, go, r0, m.mbar);
        else tma_load_3d(m.G + (size_t)r0 * GW, maps, q0, r0, go, m.mbar);
      }
      if (p.axis == 2) tma_load_3d(m.G + (size_t)half * GW, maps + 128, q0, go, half, m.mbar);
      else tma_load_3d(m.G + (size_t)half * GW, maps + 128, q0, half, go, m.mbar);
    }
  }
  const F2FromS<RW> from_s{S};
  const F2ToS<RW> to_s{S};
  const long long st3 = !FUSED || p.axis == 0 ? 1 : (p.axis == 1 ? (long long)p.g.gpitch : (long long)p.g.gpitch * p.g.gext[1]);

  if constexpr (KIND == K_FWD_REAL) {
    f2_forward_real<P, RW>(p, t, type, (const float*)p.in + bi, q0);
    const int bt = base_type(type);
    const bool cplx = bt == T_PER || bt == T_UNB, quarter = is_quarter(bt), oddo = is_odd_origin(bt);
    const bool cell = p.center == C_CELL, vec = p.f2_vec & 2;
    const int nm = p.n_modes, l = tid & (W - 1), q = q0 + 4 * l;
    if (q < p.npen) {
      const f2 h = f2_dup(quarter ? 0.25f : 0.5f);  // the split leaves twice the modes; a quarter-wave type halves
      for (int k = tid >> p.lw; k < nm; k += nt >> p.lw) {
        const int kk = quarter ? 2 * k + 1 : k, km = kk == 0 ? 0 : P - kk;
        cf2 A, B;
        f2_split(S[RW::at(kk) + l], S[RW::at(km) + l], A, B);
        A = f2_scale(A, h);
        B = f2_scale(B, h);
        const long long off = bo + (long long)q * p.ao.ls + (long long)k * p.ao.js;
        if (cplx) {
          float2* out = (float2*)p.out + off;
          f2_store2(out, p.ao.ls, q, p.npen, vec, A);
          if (q + 2 < p.npen) f2_store2(out + 2 * p.ao.ls, p.ao.ls, q + 2, p.npen, vec, B);
        } else {
          if (cell) {
            const f2w w = f2_twiddle(t.tw, kk);
            A = f2_cmul<false>(A, w.c, w.s);
            B = f2_cmul<false>(B, w.c, w.s);
          }
          f2_store4((float*)p.out + off, p.ao.ls, q, p.npen, vec,
                    oddo ? f2_make(f2_neg(A.y), f2_neg(B.y)) : f2_make(A.x, B.x));
        }
      }
    }
  } else if constexpr (KIND == K_INV_REAL) {
    const int bt = base_type(type);
    const bool cplx = bt == T_PER || bt == T_UNB, quarter = is_quarter(bt), oddo = is_odd_origin(bt);
    const bool cell = p.center == C_CELL, vec = p.f2_vec & 1;
    const int nm = p.n_modes, l = tid & (W - 1), q = q0 + 4 * l, npen = p.npen;
    const long long offl = bi + (long long)q * p.ai.ls;
    if (quarter)  // even modes of the quarter-wave types are zero
      for (int idx = tid; idx < half * W; idx += nt) S[RW::at(2 * (idx >> p.lw)) + (idx & (W - 1))] = f2_make(0, 0);
    constexpr int U = 4;
    for (int k0 = tid >> p.lw; k0 < nm; k0 += U * (nt >> p.lw)) {
      cf2 Av[U], Bv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * (nt >> p.lw);
        Av[u] = Bv[u] = f2_make(0, 0);
        if (k >= nm || q >= npen) continue;
        const long long off = offl + (long long)k * p.ai.js;
        if (cplx) {
          const float2* in = (const float2*)p.in + off;
          Av[u] = f2_load2(in, p.ai.ls, q, npen, vec);
          if (q + 2 < npen) Bv[u] = f2_load2(in + 2 * p.ai.ls, p.ai.ls, q + 2, npen, vec);
        } else {
          const cf2 c = f2_load4((const float*)p.in + off, p.ai.ls, q, npen, vec);
          Av[u].x = c.x;
          Bv[u].x = c.y;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * (nt >> p.lw);
        if (k >= nm) continue;
        const int kk = quarter ? 2 * k + 1 : k;
        cf2 A = Av[u], B = Bv[u];
        if (cplx) {
          if (kk == 0 || 2 * kk == P) A.y = B.y = 0;  // DC and Nyquist of a real signal are real
        } else {
          if (quarter) {
            const f2 two = f2_dup(2.f);
            A.x = f2_mul(A.x, two);
            B.x = f2_mul(B.x, two);
          }
          if (oddo) {
            A = f2_make(0, f2_neg(A.x));
            B = f2_make(0, f2_neg(B.x));
          }
          if (cell) {
            const f2w w = f2_twiddle(t.tw, kk);
            A = f2_cmul<true>(A, w.c, w.s);
            B = f2_cmul<true>(B, w.c, w.s);
          }
        }
        S[RW::at(kk) + l] = f2_make(f2_sub(A.x, B.y), f2_add(A.y, B.x));
        if (kk != 0 && 2 * kk != P) S[RW::at(P - kk) + l] = f2_make(f2_add(A.x, B.y), f2_sub(B.x, A.y));
      }
    }
    __syncthreads();
    f2_stage<P, RW, R0, 1, true, true, true>(t, from_s, to_s);
    f2_mid_stages<P, RW, true, false, 1, ns - 1>(t);
    f2_store_real<P, RW>(p, t, type, (float*)p.out + bo, q0);
  } else if constexpr (KIND == K_FUSED_REAL) {
    f2_forward_real<P, RW>(p, t, type, (const float*)p.in + bi, q0);
    const bool quarter = is_quarter(base_type(type));
    {
      const int l = tid & (W - 1);
      const f2 h = f2_dup(0.5f);
      for (int k = tid >> p.lw; k <= half; k += nt >> p.lw) {
        const int km = k == 0 ? 0 : P - k;
        cf2 A = f2_make(0, 0), B = A;
        if (!quarter || (k & 1)) {
          f2_split(S[RW::at(k) + l], S[RW::at(km) + l], A, B);
          const int g3 = quarter ? (k - 1) >> 1 : k;
          A = f2_scale(A, f2_mul(h, f2_green2(p.g, p.axis, &m.goff[4 * l], &m.k2p[4 * l], g3, st3)));
          B = f2_scale(B, f2_mul(h, f2_green2(p.g, p.axis, &m.goff[4 * l + 2], &m.k2p[4 * l + 2], g3, st3)));
        }
        S[RW::at(k) + l] = f2_make(f2_sub(A.x, B.y), f2_add(A.y, B.x));
        if (k != 0 && 2 * k != P) S[RW::at(km) + l] = f2_make(f2_add(A.x, B.y), f2_sub(B.x, A.y));
      }
    }
    __syncthreads();
    f2_stage<P, RW, R0, 1, true, true, true>(t, from_s, to_s);
    f2_mid_stages<P, RW, true, false, 1, ns - 1>(t);
    f2_store_real<P, RW>(p, t, type, (float*)p.out + bo, q0);
  } else {
    // complex passes
    const int l0 = tid & (W - 1), ql = q0 + 2 * l0, npen = p.npen;
    const long long ils = p.ai.ls, ijs = p.ai.js, ols = p.ao.ls, ojs = p.ao.js;
    const float2* in = (const float2*)p.in + bi + (long long)ql * ils;
    float2* out = (float2*)p.out + bo + (long long)ql * ols;
    const int n_in = KIND == K_INV_C2C ? P : p.n_use, n_out = KIND == K_FWD_C2C ? P : p.n_data;
    const bool vin = p.f2_vec & 1, vout = p.f2_vec & 2;
    auto load = [=](auto R, auto nbf, int j, int, cf2* v) {
      const float2* c = in + (long long)j * ijs;
      const long long step = (long long)nbf.value * ijs;
      const int lim = ql < npen ? n_in - j : 0;
#pragma unroll
      for (int r = 0; r < R.value; ++r, c += step) {
        v[r] = f2_make(0, 0);
        if (r * nbf.value < lim) v[r] = f2_load2(c, ils, ql, npen, vin);
      }
    };
    // node-centred periodic: phi_N := phi_0
    const int dup = (KIND != K_FWD_C2C && p.type == T_PER && p.center == C_NODE && p.n_data > p.N) ? p.N : -1;
    bool store_ok = ql < npen;
    auto store = [&](auto R, auto Ns, int o_, int, const cf2* v) {
      if (!store_ok) return;
      float2* d = out + (long long)o_ * ojs;
      const long long step = (long long)Ns.value * ojs;
      const int lim = n_out - o_;
      if (dup >= 0 && o_ == 0) f2_store2(d + (long long)dup * ojs, ols, ql, npen, vout, v[0]);
#pragma unroll
      for (int r = 0; r < R.value; ++r, d += step)
        if (r * Ns.value < lim) f2_store2(d, ols, ql, npen, vout, v[r]);
    };
    if constexpr (KIND == K_FUSED_C2C) {
      f2_stage<P, RW, R0, 1, false, false, true>(t, load, to_s);
      f2_mid_stages<P, RW, false, false, 1, ns>(t);
      // u^ = G^ f^ in the first inverse stage (radices reversed)
      if (tma_g) {
        if (!mbar_wait_bounded(m.mbar, p.errflag, 1, p.dbg_wait & 1)) store_ok = false;
      }
      const long long* goff = &m.goff[2 * l0];
      const float* k2p = &m.k2p[2 * l0];
      const float* Gs = m.G;
      auto gained = [&](auto R, auto nbf, int j, int l, cf2* v) {
        from_s(R, nbf, j, l, v);
#pragma unroll
        for (int r = 0; r < R.value; ++r) {
          const int i = j + r * nbf.value, g3 = min(i, P - i);
          const f2 g = tma_g ? *reinterpret_cast<const f2*>(&Gs[g3 * 2 * W + 2 * l])
                             : f2_green2(p.g, p.axis, goff, k2p, g3, st3);
          v[r] = f2_scale(v[r], g);
        }
      };
      f2_stage<P, RW, RL, 1, true, true, true>(t, gained, to_s);
      f2_mid_stages<P, RW, true, true, 1, ns - 1>(t);
      f2_stage<P, RW, R0, P / R0, true, true, false>(t, from_s, store);
    } else {
      constexpr bool INV = KIND == K_INV_C2C;
      f2_stage<P, RW, R0, 1, INV, false, true>(t, load, to_s);
      f2_mid_stages<P, RW, INV, false, 1, ns - 1>(t);
      f2_stage<P, RW, RL, P / RL, INV, true, false>(t, from_s, store);
    }
  }
}

// ---------------------------------------------------------------------------
// Fused last direction of the Biot-Savart solve: each third of the CTA transforms one component's tile in shared
// memory, u^ = G^ (i w x f^) is taken point by point over the three (the derivative factors of curl.cu), and
// each third transforms one result back.
// ---------------------------------------------------------------------------
struct F2Curl {       // per lane: the factors of the two non-axis directions, per source component
  cf2 fac[2][3];
};

// Derivative factor along direction d of source component c at the pencil's mode: real for r2r coefficients
// (sine-type sources +, cosine-type -), imaginary otherwise.
__device__ __forceinline__ float2 f2_factor(const FusedGreen& g, int d, int c, int mode) {
  const int kk = (g.role[d] == 0 && g.quarter[d]) ? 2 * mode + 1 : mode;
  const float s = ((const float*)g.dsym[d])[kk];
  if (g.role[d] == 0) return make_float2(((g.srcodd[d] >> c) & 1) ? s : -s, 0.f);
  return make_float2(0.f, s);
}
// product of complex pairs
__device__ __forceinline__ cf2 f2_mulc(cf2 a, cf2 b) {
  return f2_make(f2_sub(f2_mul(a.x, b.x), f2_mul(a.y, b.y)), f2_fma(a.x, b.y, f2_mul(a.y, b.x)));
}
// u_c = G (D_a f_b - D_b f_a), (a, b) = (c + 1, c + 2); s3: symbol along the axis
__device__ __forceinline__ void f2_curl(int axis, const F2Curl& f, f2 s3, f2 G, const cf2* F, cf2* U) {
  const int d0 = axis == 0 ? 1 : 0;  // directions of fac[0], fac[1]
  auto term = [&](int d, int c) {    // D_d f_c
    if (d == axis) return f2_make(f2_neg(f2_mul(F[c].y, s3)), f2_mul(F[c].x, s3));
    return f2_mulc(f.fac[d == d0 ? 0 : 1][c], F[c]);
  };
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int a = (c + 1) % 3, b = (c + 2) % 3;
    U[c] = f2_scale(term(a, b) - term(b, a), G);
  }
}

template <bool REAL, int P>
__global__ void __launch_bounds__(512, 1) k_f2_curl(const __grid_constant__ PassParams p) {
  pass_entry(p);
  extern __shared__ __align__(16) unsigned char smraw[];
  using RW = F2Rows<P, FX_CURL>;
  constexpr F2Plan pl = RW::plan;
  constexpr int ns = pl.n, half = P / 2, R0 = pl.r[0], RL = pl.r[ns - 1];
  constexpr int per = REAL ? 4 : 2, NP = REAL ? 2 : 1;  // pencils and pencil pairs of a lane
  const int W = p.W, tid = threadIdx.x, nt = blockDim.x, axis = p.axis;
  cf2* S0 = reinterpret_cast<cf2*>(smraw);
  F2Curl* fac = reinterpret_cast<F2Curl*>(S0 + 3 * RW::size);       // NP per lane
  long long* goff = reinterpret_cast<long long*>(fac + NP * W);      // per lane: per
  float* k2p = reinterpret_cast<float*>(goff + per * W);
  const int q0 = blockIdx.x * per * W, o = blockIdx.y, npen = p.npen;
  const long long bi = (long long)o * p.ai.os, bo = (long long)o * p.ao.os;
  const FusedGreen& g = p.g;
  for (int i = tid; i < per * W; i += nt) {
    const int q = q0 + i;
    f2_green_base(p, q, o, &goff[i], &k2p[i]);
    // pencil i of the block: lane i / per; real lanes pair (q, q + 1) and (q + 2, q + 3)
    float* dst = reinterpret_cast<float*>(&fac[(i / per) * NP + (i % per) / 2]);
    int crd[3];
    if (axis == 0) { crd[1] = q % g.dims1; crd[2] = q / g.dims1; crd[0] = 0; }
    else if (axis == 1) { crd[0] = q; crd[2] = o; crd[1] = 0; }
    else { crd[0] = q; crd[1] = o; crd[2] = 0; }
    int e = 0;
    for (int d = 0; d < 3; ++d) {
      if (d == axis) continue;
      for (int c = 0; c < 3; ++c) {
        const float2 v = q < npen ? f2_factor(g, d, c, crd[d]) : make_float2(0.f, 0.f);
        dst[(e * 3 + c) * 4 + (i & 1)] = v.x;
        dst[(e * 3 + c) * 4 + 2 + (i & 1)] = v.y;
      }
      ++e;
    }
  }
  __syncthreads();
  const long long st3 = axis == 0 ? 1 : (axis == 1 ? (long long)g.gpitch : (long long)g.gpitch * g.gext[1]);
  const float* sym3 = (const float*)g.dsym[axis];
  const int l = tid & (W - 1);  // of the thread's transforms too: a third is a multiple of W threads
  const int ql = q0 + per * l;
  const long long ils = p.ai.ls, ijs = p.ai.js, ols = p.ao.ls, ojs = p.ao.js;
  const int ntc = nt / 3, mine = tid / ntc;  // threads and number of this thread's component
  const F2Tile t{S0 + mine * RW::size, W, p.lw, tid - mine * ntc, ntc, (const f2w*)p.tw};
  {
    if constexpr (REAL) {
      f2_forward_real<P, RW>(p, t, comp_type(p, mine), (const float*)p.in + bi + mine * p.ai.cs, q0);
    } else {
      const float2* in = (const float2*)p.in + bi + mine * p.ai.cs + (long long)ql * ils;
      const int n_in = p.n_use;
      const bool vin = p.f2_vec & 1;
      f2_stage<P, RW, R0, 1, false, false, true>(
          t,
          [=](auto R, auto nbf, int j, int, cf2* v) {
            const float2* s = in + (long long)j * ijs;
            const long long step = (long long)nbf.value * ijs;
            const int lim = ql < npen ? n_in - j : 0;
#pragma unroll
            for (int r = 0; r < R.value; ++r, s += step) {
              v[r] = f2_make(0, 0);
              if (r * nbf.value < lim) v[r] = f2_load2(s, ils, ql, npen, vin);
            }
          },
          F2ToS<RW>{t.S});
      f2_mid_stages<P, RW, false, false, 1, ns>(t);
    }
  }
  if constexpr (REAL) {
    const bool quarter = is_quarter(base_type(comp_type(p, 0)));
    const f2 h = f2_dup(0.5f);
#pragma unroll 1
    for (int k = tid >> p.lw; k <= half; k += nt >> p.lw) {
      const int km = k == 0 ? 0 : P - k;
      const bool live = !quarter || (k & 1);
      const int g3 = quarter ? max(k - 1, 0) >> 1 : k;
      const f2 s3 = f2_dup(sym3[k]);
      cf2 A[3], B[3], UA[3], UB[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const cf2* S = S0 + c * RW::size;
        f2_split(S[RW::at(k) + l], S[RW::at(km) + l], A[c], B[c]);
        UA[c] = UB[c] = f2_make(0, 0);
      }
      if (live) {
        f2_curl(axis, fac[2 * l], s3, f2_mul(h, f2_green2(g, axis, &goff[4 * l], &k2p[4 * l], g3, st3)), A, UA);
        f2_curl(axis, fac[2 * l + 1], s3, f2_mul(h, f2_green2(g, axis, &goff[4 * l + 2], &k2p[4 * l + 2], g3, st3)), B, UB);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        cf2* S = S0 + c * RW::size;
        S[RW::at(k) + l] = f2_make(f2_sub(UA[c].x, UB[c].y), f2_add(UA[c].y, UB[c].x));
        if (k != 0 && 2 * k != P) S[RW::at(km) + l] = f2_make(f2_add(UA[c].x, UB[c].y), f2_sub(UB[c].x, UA[c].y));
      }
    }
  } else {
#pragma unroll 1
    for (int k = tid >> p.lw; k < P; k += nt >> p.lw) {
      cf2 F[3], U[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) F[c] = S0[c * RW::size + RW::at(k) + l];
      f2_curl(axis, fac[l], f2_dup(sym3[k]), f2_green2(g, axis, &goff[2 * l], &k2p[2 * l], min(k, P - k), st3), F, U);
#pragma unroll
      for (int c = 0; c < 3; ++c) S0[c * RW::size + RW::at(k) + l] = U[c];
    }
  }
  __syncthreads();
  {
    const F2FromS<RW> from_s{t.S};
    if constexpr (REAL) {
      f2_stage<P, RW, R0, 1, true, true, true>(t, from_s, F2ToS<RW>{t.S});
      f2_mid_stages<P, RW, true, false, 1, ns - 1>(t);
      f2_store_real<P, RW>(p, t, (g.utypes >> (4 * mine)) & 15, (float*)p.out + bo + mine * p.ao.cs, q0);
    } else {
      f2_stage<P, RW, RL, 1, true, true, true>(t, from_s, F2ToS<RW>{t.S});
      f2_mid_stages<P, RW, true, true, 1, ns - 1>(t);
      float2* out = (float2*)p.out + bo + mine * p.ao.cs + (long long)ql * ols;
      const int dup = (p.type == T_PER && p.center == C_NODE && p.n_data > p.N) ? p.N : -1;
      const int n_out = p.n_data;
      const bool vout = p.f2_vec & 2;
      f2_stage<P, RW, R0, P / R0, true, true, false>(t, from_s, [=](auto R, auto Ns, int o_, int, const cf2* v) {
        if (ql >= npen) return;
        float2* d = out + (long long)o_ * ojs;
        const long long step = (long long)Ns.value * ojs;
        const int lim = n_out - o_;
        if (dup >= 0 && o_ == 0) f2_store2(d + (long long)dup * ojs, ols, ql, npen, vout, v[0]);
#pragma unroll
        for (int r = 0; r < R.value; ++r, d += step)
          if (r * Ns.value < lim) f2_store2(d, ols, ql, npen, vout, v[r]);
      });
    }
  }
}

}  // namespace

template <int KIND, int P> constexpr bool f2_has() {
  if (KIND == K_FWD_C2C || KIND == K_INV_C2C || KIND == K_FUSED_C2C) return f2_complex(P);
  return KIND >= K_CURL_REAL ? f2_curl(P) : true;
}
// The kernel of a kind and length (nullptr: the planner sends no such pass here).
template <int KIND, int P> constexpr auto f2_kernel() {
  using Kernel = void (*)(PassParams);
  if constexpr (!f2_has<KIND, P>()) return Kernel(nullptr);
  else if constexpr (KIND >= K_CURL_REAL) return Kernel(k_f2_curl<KIND == K_CURL_REAL, P>);
  else return Kernel(k_f2<KIND, P>);
}
template <int KIND, int P>
cudaError_t f2_launch(const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
  if constexpr (!f2_has<KIND, P>()) {
    return cudaErrorInvalidValue;
  } else {
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
    return cudaLaunchKernelEx(&cfg, f2_kernel<KIND, P>(), p);
  }
}
template <int KIND, int P> cudaError_t f2_limit() {
  if constexpr (!f2_has<KIND, P>()) return cudaErrorInvalidValue;
  else return cudaFuncSetAttribute(f2_kernel<KIND, P>(), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}
#define F2_KINDS(DO)                   \
  switch (kind) {                      \
    case K_FWD_REAL: DO(K_FWD_REAL);   \
    case K_INV_REAL: DO(K_INV_REAL);   \
    case K_FWD_C2C: DO(K_FWD_C2C);     \
    case K_INV_C2C: DO(K_INV_C2C);     \
    case K_FUSED_REAL: DO(K_FUSED_REAL); \
    case K_FUSED_C2C: DO(K_FUSED_C2C); \
    case K_CURL_REAL: DO(K_CURL_REAL); \
    case K_CURL_C2C: DO(K_CURL_C2C);   \
    default: return cudaErrorInvalidValue; \
  }
template <int P>
cudaError_t f2_launch_kind(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) {
#define F2_DO(K) return f2_launch<K, P>(p, grid, nthr, smem, st)
  F2_KINDS(F2_DO)
#undef F2_DO
}
template <int P> cudaError_t f2_limit_kind(int kind) {
#define F2_DO(K) return f2_limit<K, P>()
  F2_KINDS(F2_DO)
#undef F2_DO
}

#define F2_LAUNCH_CASE(P) \
  case P: return f2_launch_kind<P>(kind, p, grid, nthr, smem, st);
#define F2_LIMIT_CASE(P) \
  case P: return f2_limit_kind<P>(kind);
// Launcher and shared-memory limits of the lengths of FX_SHARD_<i>.
#define F2_UNIT(i)                                                                                              \
  namespace flups {                                                                                             \
  cudaError_t launch_f2_##i(int kind, const PassParams& p, dim3 grid, int nthr, size_t smem, cudaStream_t st) { \
    switch (p.P) { FX_SHARD_##i(F2_LAUNCH_CASE) }                                                               \
    return cudaErrorInvalidValue;                                                                               \
  }                                                                                                             \
  cudaError_t limit_f2_##i(int kind, int P) {                                                                   \
    switch (P) { FX_SHARD_##i(F2_LIMIT_CASE) }                                                                  \
    return cudaErrorInvalidValue;                                                                               \
  }                                                                                                             \
  }

}  // namespace flups
