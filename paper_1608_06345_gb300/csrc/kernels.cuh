// Device code of the fused pull-stream + BGK-collide step and its helpers.
//
// Per cell and time step (paper: Eq. (13)-(18), Tables I/II, Sec. V):
//   a1 pull     g~_i(x) = g*_i(x - c_i), h~_i(x) = h*_i(x - c_i)
//   a2 moments  rho = sum g~, rho u = sum xi g~, rho E = sum xi^2/2 g~ + sum h~,
//               T = (2E - u^2) / (D + delta)
//   a3 F_i      w_i rho [A0 + A1 s + A2 s^2 + s^3/6 + s^4/24], s = xi_i.u, the
//               fourth-order Hermite equilibrium of Eq. (18) regrouped in
//               powers of s; A0..A2 depend on the velocity group only, so a
//               (c, -c) pair shares the even part and flips the odd part.
//   a4 Fh_i     (delta/2) T F_i
//   a5 relax    g* = g~ + (F - g~)/tau_f,  h* = h~ + (Fh - h~)/tau_g; store.
//
// Representation: every population is held as its deviation from a fixed
// reference equilibrium of the instance, g_i = gref_i + dg_i with
// gref_i = F_i(rho0, u = 0, T0) and h_i = href_i + dh_i with
// href_i = (delta/2) T0 gref_i.  This is an exact change of variables (the
// scheme is linear in g, h given the moments, and the reference totals are
// known: sum gref = rho0, sum xi gref = 0, sum xi^2/2 gref = rho0 D T0 / 2,
// sum href = rho0 delta T0 / 2).  Working on the small dg, dh keeps FP32 and
// 16-bit storage from losing the momentum to cancellation in sum xi_i g_i.
//
// Storage: structure of arrays, cell index x + nx*(y + ny*z).  FP64/FP32:
// 2Q planes (0..Q-1 for g, Q..2Q-1 for h) of ps elements holding dg, dh.
// 16-bit: Q planes of ps 32-bit pairs, g_i in the low half and h_i in the
// high half, holding dg/gref and dh/hscale.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "lattice.h"
#include "pair_order.h"

namespace lbm {

constexpr int kPeriodic = 0;
constexpr int kZeroGradient = 1;

// ---------------------------------------------------------------------------
// compile-time helpers
// ---------------------------------------------------------------------------
template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<N, I + 1>(f);
  }
}

template <int LAT>
struct Lat {
  static constexpr int D = (LAT == 0) ? 2 : 3;
  static constexpr int Q = (LAT == 0) ? 37 : 107;
  static constexpr int G = (LAT == 0) ? 8 : 10;
  __host__ __device__ static constexpr int cx(int i) { return (LAT == 0 ? kD2Q37 : kD3Q107).c[i][0]; }
  __host__ __device__ static constexpr int cy(int i) { return (LAT == 0 ? kD2Q37 : kD3Q107).c[i][1]; }
  __host__ __device__ static constexpr int cz(int i) { return (LAT == 0 ? kD2Q37 : kD3Q107).c[i][2]; }
  __host__ __device__ static constexpr int grp(int i) { return (LAT == 0 ? kD2Q37 : kD3Q107).grp[i]; }
  __host__ __device__ static constexpr int c2(int i) { return cx(i) * cx(i) + cy(i) * cy(i) + cz(i) * cz(i); }
};

// ---------------------------------------------------------------------------
// start of a kernel that may be set up while its stream's previous kernel
// drains (launch_next): wait until that one has finished and its writes are
// visible, before touching global memory
// ---------------------------------------------------------------------------
__device__ __forceinline__ void wait_for_previous_kernel() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// per-instance constants, already converted to the compute type C on the host
// (a double->float conversion runs on the FP64 pipe, which is slow on GB300)
// ---------------------------------------------------------------------------
template <class C>
struct Args {
  int n[3];          // nx, ny, nz
  int bc[3];         // kPeriodic / kZeroGradient per axis
  long long ps;      // plane stride in elements
  C r;               // xi = r c
  C half_r2;         // r^2 / 2
  C Dd;              // D + delta
  C inv_Dd;          // 1 / (D + delta)
  C half_delta;      // delta / 2
  C omega_f;         // 1 / tau_f
  C omega_g;         // 1 / tau_g
  C rho0, T0, t0;    // reference state; t0 = T0 - 1
  C wg[10];          // group weights
  C x2g[10];         // group |xi|^2
  C gref[10];        // reference equilibrium per group, w rho0 A0(u = 0, t0)
  C pref[10];        // A0(u = 0, t0) - 1 per group
  // 16-bit storage codec: dg = gref * d, dh = hscale * e
  C inv_gref[10], hscale[10], inv_hscale[10];
  unsigned int* flag;  // error word: bit 0 = non-finite rho or T met, bit 1 = a wait gave up
  // FP64 relaxation (relax_put_k)
  C om1_f;           // 1 - 1 / tau_f
  C hd_fg;           // (delta / 2) tau_f / tau_g
  C wf[10];          // group weights / tau_f
};

// ---------------------------------------------------------------------------
// storage codec
// ---------------------------------------------------------------------------
template <class S>
struct IsS16 : std::integral_constant<bool, std::is_same<S, __half>::value ||
                                              std::is_same<S, __nv_bfloat16>::value> {};

template <class S>
__device__ __forceinline__ S ldg_s(const S* p) {
  if constexpr (std::is_same<S, __half>::value) {
    unsigned short v = __ldg(reinterpret_cast<const unsigned short*>(p));
    return __ushort_as_half(v);
  } else if constexpr (std::is_same<S, __nv_bfloat16>::value) {
    unsigned short v = __ldg(reinterpret_cast<const unsigned short*>(p));
    return __ushort_as_bfloat16(v);
  } else {
    return __ldg(p);
  }
}

template <class S>
__device__ __forceinline__ float s16_to_f(S v) {
  if constexpr (std::is_same<S, __half>::value) return __half2float(v);
  else return __bfloat162float(v);
}

template <class S>
__device__ __forceinline__ S f_to_s16(float v) {
  if constexpr (std::is_same<S, __half>::value) return __float2half_rn(v);
  else return __float2bfloat16_rn(v);
}

// decode a stored population of group g into its deviation (dg or dh);
// IS_H selects the h codec
template <class S, class C, bool IS_H>
__device__ __forceinline__ C decode(S v, int g, const Args<C>& a) {
  if constexpr (IsS16<S>::value) {
    const C d = static_cast<C>(s16_to_f(v));
    return IS_H ? a.hscale[g] * d : a.gref[g] * d;
  } else {
    return static_cast<C>(v);
  }
}

template <class S, class C, bool IS_H>
__device__ __forceinline__ S encode(C v, int g, const Args<C>& a) {
  if constexpr (IsS16<S>::value) {
    const C d = IS_H ? v * a.inv_hscale[g] : v * a.inv_gref[g];
    return f_to_s16<S>(static_cast<float>(d));
  } else {
    return static_cast<S>(v);
  }
}

// ---------------------------------------------------------------------------
// population addressing
//   FP64 / FP32 storage: plane p (0..Q-1 for g, Q..2Q-1 for h), element
//     p * ps + cell;
//   16-bit storage: g_i and h_i of a cell are adjacent, one 32-bit pair
//     (g in the low half): plane i holds ps pairs, pair i * ps + cell.  One
//     access moves both populations of a direction.
// ---------------------------------------------------------------------------
template <class S>
__device__ __forceinline__ void unpack16(unsigned v, float& lo, float& hi) {
  if constexpr (std::is_same<S, __half>::value) {
    lo = __half2float(__ushort_as_half((unsigned short)(v & 0xffffu)));
    hi = __half2float(__ushort_as_half((unsigned short)(v >> 16)));
  } else {  // bfloat16: the upper 16 bits of an FP32
    lo = __uint_as_float(v << 16);
    hi = __uint_as_float(v & 0xffff0000u);
  }
}

template <class S>
__device__ __forceinline__ unsigned pack16(float lo, float hi) {
  if constexpr (std::is_same<S, __half>::value)
    return (unsigned)__half_as_ushort(__float2half_rn(lo)) | ((unsigned)__half_as_ushort(__float2half_rn(hi)) << 16);
  else
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
           ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

// raw stored (g_i, h_i) of a cell (16-bit: the stored relative deviations)
template <int Q, class S, class C>
__device__ __forceinline__ void ld_gh(const S* __restrict__ src, int i, long long ps, size_t cell, C& g, C& h) {
  if constexpr (IsS16<S>::value) {
    float lo, hi;
    unpack16<S>(__ldg(reinterpret_cast<const unsigned*>(src) + ((size_t)i * ps + cell)), lo, hi);
    g = static_cast<C>(lo);
    h = static_cast<C>(hi);
  } else {
    g = static_cast<C>(__ldg(src + ((size_t)i * ps + cell)));
    h = static_cast<C>(__ldg(src + ((size_t)(Q + i) * ps + cell)));
  }
}

// store raw (g_i, h_i) (already in the stored scale)
template <int Q, class S, class C>
__device__ __forceinline__ void st_gh(S* __restrict__ dst, int i, long long ps, size_t cell, C g, C h) {
  if constexpr (IsS16<S>::value) {
    reinterpret_cast<unsigned*>(dst)[(size_t)i * ps + cell] = pack16<S>(static_cast<float>(g), static_cast<float>(h));
  } else {
    dst[(size_t)i * ps + cell] = static_cast<S>(g);
    dst[(size_t)(Q + i) * ps + cell] = static_cast<S>(h);
  }
}

// deviations (dg, dh) of a stored raw pair of group grp
template <class S, class C>
__device__ __forceinline__ void scale_gh(C& g, C& h, int grp, const Args<C>& a) {
  if constexpr (IsS16<S>::value) {
    g *= a.gref[grp];
    h *= a.hscale[grp];
  }
}

// ---------------------------------------------------------------------------
// read-only loads that stay where they are written: not merged with another of
// the same address, not moved past one another
__device__ __forceinline__ float ld_again(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_again(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_again(const double* p) {
  double v;
  asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ unsigned ld_again(const unsigned* p) {
  unsigned v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// ---------------------------------------------------------------------------
// two FP32 values in one 64-bit register; add and subtract work on both in one
// instruction, each rounded as the scalar one is
// ---------------------------------------------------------------------------
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack_f32x2(float a, float b) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ void unpack_f32x2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add_f32x2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 sub_f32x2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 neg_f32x2(f32x2 a) { return a ^ 0x8000000080000000ull; }

// ---------------------------------------------------------------------------
// equilibrium deviations (Eq. (18), regrouped by powers of s per group)
//
// With u2 = |u|^2, t = T - 1, x2 = |xi|^2 of the group:
//   F_i / (w rho) = A0 + A1 s + A2 s^2 + s^3/6 + s^4/24
//   A0 = 1 + P,  P = -u2/2 + t (x2 - D)/2 + u2^2/8 + t (D + 2 - x2) u2 / 4
//                    + t^2 [x2^2 - 2 (D + 2) x2 + D (D + 2)] / 8
//   A1 = 1 - u2/2 + t (x2 - D - 2)/2
//   A2 = 1/2 - u2/4 + t (x2 - D - 4)/4
// and the deviation from gref = w rho0 (1 + pref):
//   dF_i = w [drho (1 + P) + rho0 (P - pref)] + w rho [A1 s + A2 s^2 + ...]
//   dFh_i = (delta/2) (T dF_i + dT gref_i)
// ---------------------------------------------------------------------------
template <int LAT, class C>
struct EqCoef {
  // per-cell polynomials in the group's x2 (see above); the per-group
  // coefficients are formed just before that group's velocities are emitted
  C pa, pb, pc, be0, be1, ga0, ga1;
  C rho, drho;
  C ur[3];  // r u
  C T, dT;
};

template <int LAT, class C>
__device__ __forceinline__ void eq_coeffs(C drho, const C (&u)[3], C dT, const Args<C>& a, EqCoef<LAT, C>& k) {
  using L = Lat<LAT>;
  constexpr C D = C(L::D);
  k.rho = a.rho0 + drho;
  k.drho = drho;
  k.T = a.T0 + dT;
  k.dT = dT;
  const C t = a.t0 + dT;
  const C u2 = u[0] * u[0] + u[1] * u[1] + (L::D == 3 ? u[2] * u[2] : C(0));
  // P = pa + pb x2 + pc x2^2;  A1 = be0 + be1 x2;  A2 = ga0 + ga1 x2
  k.pa = -C(0.5) * u2 - C(0.5) * D * t + C(0.125) * u2 * u2 + C(0.25) * (D + C(2)) * t * u2 +
         C(0.125) * D * (D + C(2)) * t * t;
  k.pb = C(0.5) * t - C(0.25) * t * u2 - C(0.25) * (D + C(2)) * t * t;
  k.pc = C(0.125) * t * t;
  k.be0 = C(1) - C(0.5) * u2 - C(0.5) * (D + C(2)) * t;
  k.be1 = C(0.5) * t;
  k.ga0 = C(0.5) - C(0.25) * u2 - C(0.25) * (D + C(4)) * t;
  k.ga1 = C(0.25) * t;
  k.ur[0] = a.r * u[0];
  k.ur[1] = a.r * u[1];
  k.ur[2] = L::D == 3 ? a.r * u[2] : C(0);
}

// emit(I, dF_i) for every velocity i of [IB, IE): the rest velocity (when
// IB = 0), then the (c, -c) pairs sharing the even part of the polynomial in
// s.  Velocities are ordered by group, so a group's coefficients c0..c4 are
// formed once, at its first pair in the range, and are dead after its last.
// IB is 0 or odd, IE odd or Q (whole pairs only).
// RELAX: emits omega_f dF_i
template <int LAT, class C, int IB = 0, int IE = Lat<LAT>::Q, bool RELAX = false, class Emit>
__device__ __forceinline__ void eq_emit(const EqCoef<LAT, C>& k, const Args<C>& a, Emit&& emit) {
  using L = Lat<LAT>;
  C c0, c1, c2, c3, c4;
  auto group = [&](int g) {
    const C x2 = a.x2g[g];
    const C P = fma(x2, fma(x2, k.pc, k.pb), k.pa);
    const C W = (RELAX ? a.wf[g] : a.wg[g]) * k.rho;
    c0 = (RELAX ? a.wf[g] : a.wg[g]) * fma(k.drho, C(1) + P, a.rho0 * (P - a.pref[g]));
    c1 = W * fma(k.be1, x2, k.be0);
    c2 = W * fma(k.ga1, x2, k.ga0);
    c3 = W * C(1.0 / 6.0);
    c4 = W * C(1.0 / 24.0);
  };
  static_assert((IB == 0 || IB % 2 == 1) && (IE == L::Q || IE % 2 == 1) && IB < IE, "whole pairs only");
  if constexpr (IB == 0) {
    group(0);
    emit(std::integral_constant<int, 0>{}, c0);
  }
  static_for<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (i % 2 == 1 && i >= IB && i < IE) {
      constexpr int g = L::grp(i);
      if constexpr (i == IB || L::grp(i - 1) != g) group(g);
      constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
      C s = C(0);
      if constexpr (cx != 0) s = fma(C(cx), k.ur[0], s);
      if constexpr (cy != 0) s = fma(C(cy), k.ur[1], s);
      if constexpr (cz != 0) s = fma(C(cz), k.ur[2], s);
      const C s2 = s * s;
      const C e = fma(s2, fma(s2, c4, c2), c0);
      const C o = s * fma(s2, c3, c1);
      emit(std::integral_constant<int, i>{}, e + o);
      emit(std::integral_constant<int, i + 1>{}, e - o);
    }
  });
}

// dF and dFh of every velocity (used by the init kernel)
template <int LAT, class C, class Emit>
__device__ __forceinline__ void equilibrium_dev(C drho, const C (&u)[3], C dT, const Args<C>& a, Emit&& emit) {
  using L = Lat<LAT>;
  EqCoef<LAT, C> k;
  eq_coeffs<LAT, C>(drho, u, dT, a, k);
  const C hd = a.half_delta;
  eq_emit<LAT, C>(k, a, [&](auto I, C dF) {
    constexpr int g = L::grp(decltype(I)::value);
    emit(I, dF, hd * fma(k.T, dF, dT * a.gref[g]));
  });
}

// ---------------------------------------------------------------------------
// source coordinate of a pull along one axis (|c| <= 3)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int pull_coord(int p, int c, int n, int bc) {
  int q = p - c;
  if (bc == kPeriodic) {
    if (n >= 4) {  // one correction at most
      q = (q < 0) ? q + n : q;
      q = (q >= n) ? q - n : q;
    } else {  // n >= 1 and |c| <= 3: at most three corrections
      while (q < 0) q += n;
      while (q >= n) q -= n;
    }
  } else {
    q = q < 0 ? 0 : (q > n - 1 ? n - 1 : q);
  }
  return q;
}

// ---------------------------------------------------------------------------
// moments of a cell from the deviations (Eq. (14), (15)), taken over the
// (c, -c) pairs: sum and difference of the pair
//   drho = sum dg, rho = rho0 + drho, rho u = r sum c dg,
//   rho E = rho0 (D + delta) T0 / 2 + dK + dH with dK = r^2/2 sum c^2 dg, dH = sum dh,
//   T = (2E - u^2)/(D + delta) = T0 + dT,
//   dT = [2 (dK + dH) - rho u^2 - (D + delta) T0 drho] / (rho (D + delta))
// ---------------------------------------------------------------------------
// SCALED: the accessors return the stored 16-bit values d, e (dg = gref d,
// dh = hscale e); the group scales are folded into the sums' coefficients
// instead of decoding every value.
template <int LAT, class C, bool SCALED, class GetG, class GetH>
__device__ __forceinline__ void moments_raw(GetG&& getg, GetH&& geth, const Args<C>& a, C& drho, C (&u)[3],
                                            C& dT) {
  using L = Lat<LAT>;
  C m, H;
  if constexpr (SCALED) {
    m = a.gref[0] * getg(std::integral_constant<int, 0>{});
    H = a.hscale[0] * geth(std::integral_constant<int, 0>{});
  } else {
    m = getg(std::integral_constant<int, 0>{});
    H = geth(std::integral_constant<int, 0>{});
  }
  C jx = C(0), jy = C(0), jz = C(0), k2 = C(0);
  C s1 = C(1), s2 = C(2), s3 = C(3), sc2 = C(0), sh = C(1);  // group scale times 1, 2, 3, |c|^2; h scale
  static_for<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (i % 2 == 1) {
      constexpr int g = L::grp(i);
      if constexpr (SCALED && L::grp(i - 1) != g) {
        s1 = a.gref[g];
        s2 = C(2) * s1;
        s3 = C(3) * s1;
        sc2 = C(L::c2(i)) * s1;
        sh = a.hscale[g];
      }
      auto mul = [&](int c) -> C {  // the coefficient c * scale for |c| <= 3
        const int ac = c < 0 ? -c : c;
        const C v = ac == 1 ? s1 : (ac == 2 ? s2 : s3);
        return c < 0 ? -v : v;
      };
      const C gp = getg(I), gm = getg(std::integral_constant<int, i + 1>{});
      const C sp = gp + gm, df = gp - gm;
      const C hp = geth(I) + geth(std::integral_constant<int, i + 1>{});
      if constexpr (SCALED) {
        m = fma(s1, sp, m);
        if constexpr (L::cx(i) != 0) jx = fma(mul(L::cx(i)), df, jx);
        if constexpr (L::cy(i) != 0) jy = fma(mul(L::cy(i)), df, jy);
        if constexpr (L::cz(i) != 0) jz = fma(mul(L::cz(i)), df, jz);
        k2 = fma(sc2, sp, k2);
        H = fma(sh, hp, H);
      } else {
        m += sp;
        if constexpr (L::cx(i) != 0) jx = fma(C(L::cx(i)), df, jx);
        if constexpr (L::cy(i) != 0) jy = fma(C(L::cy(i)), df, jy);
        if constexpr (L::cz(i) != 0) jz = fma(C(L::cz(i)), df, jz);
        k2 = fma(C(L::c2(i)), sp, k2);
        H += hp;
      }
    }
  });
  (void)s2;
  (void)s3;
  const C rho = a.rho0 + m;
  const C inv = C(1) / rho;
  drho = m;
  u[0] = a.r * jx * inv;
  u[1] = a.r * jy * inv;
  u[2] = (L::D == 3) ? a.r * jz * inv : C(0);
  const C u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const C dE2 = C(2) * fma(a.half_r2, k2, H);
  dT = (dE2 - rho * u2 - a.Dd * a.T0 * m) * inv * a.inv_Dd;
}

template <int LAT, class C, class GetG, class GetH>
__device__ __forceinline__ void moments_dev(GetG&& getg, GetH&& geth, const Args<C>& a, C& drho, C (&u)[3],
                                            C& dT) {
  moments_raw<LAT, C, false>(getg, geth, a, drho, u, dT);
}

// the velocities in P parts of whole (c, -c) pairs
template <int LAT, int P>
struct Split {
  static constexpr int NP = (Lat<LAT>::Q - 1) / 2;  // (c, -c) pairs
  // part 0: the rest velocity and pairs [0, NP/P); part w: pairs [w NP/P, (w+1) NP/P)
  __host__ __device__ static constexpr int begin(int w) { return w == 0 ? 0 : 1 + 2 * (w * NP / P); }
  __host__ __device__ static constexpr int end(int w) { return 1 + 2 * ((w + 1) * NP / P); }
  __host__ __device__ static constexpr int kmax() {
    int m = 0;
    for (int w = 0; w < P; ++w) m = (end(w) - begin(w) > m) ? end(w) - begin(w) : m;
    return m;
  }
};

// The sums of moments_raw restricted to the velocities [IB, IE) (whole
// pairs): acc = {sum dg, sum c_x dg, sum c_y dg, sum c_z dg,
// r^2/2 sum c^2 dg + sum dh}.  Summing the parts of a partition gives the
// cell's sums (up to rounding order).
template <int LAT, class C, bool SCALED, int IB, int IE, class GetG, class GetH>
__device__ __forceinline__ void moments_partial(GetG&& getg, GetH&& geth, const Args<C>& a, C (&acc)[5]) {
  using L = Lat<LAT>;
  C m = C(0), H = C(0);
  if constexpr (IB == 0) {
    if constexpr (SCALED) {
      m = a.gref[0] * getg(std::integral_constant<int, 0>{});
      H = a.hscale[0] * geth(std::integral_constant<int, 0>{});
    } else {
      m = getg(std::integral_constant<int, 0>{});
      H = geth(std::integral_constant<int, 0>{});
    }
  }
  C jx = C(0), jy = C(0), jz = C(0), k2 = C(0), gs = C(0);
  C s1 = C(1), s2 = C(2), s3 = C(3), sc2 = C(0), sh = C(1);
  static_for<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (i % 2 == 1 && i >= IB && i < IE) {
      constexpr int g = L::grp(i);
      if constexpr (SCALED && (i == IB || L::grp(i - 1) != g)) {
        s1 = a.gref[g];
        s2 = C(2) * s1;
        s3 = C(3) * s1;
        sc2 = C(L::c2(i)) * s1;
        sh = a.hscale[g];
      }
      auto mul = [&](int c) -> C {
        const int ac = c < 0 ? -c : c;
        const C v = ac == 1 ? s1 : (ac == 2 ? s2 : s3);
        return c < 0 ? -v : v;
      };
      const C gp = getg(I), gm = getg(std::integral_constant<int, i + 1>{});
      const C sp = gp + gm, df = gp - gm;
      const C hp = geth(I) + geth(std::integral_constant<int, i + 1>{});
      if constexpr (SCALED) {
        m = fma(s1, sp, m);
        if constexpr (L::cx(i) != 0) jx = fma(mul(L::cx(i)), df, jx);
        if constexpr (L::cy(i) != 0) jy = fma(mul(L::cy(i)), df, jy);
        if constexpr (L::cz(i) != 0) jz = fma(mul(L::cz(i)), df, jz);
        k2 = fma(sc2, sp, k2);
        H = fma(sh, hp, H);
      } else {
        if constexpr (L::cx(i) != 0) jx = fma(C(L::cx(i)), df, jx);
        if constexpr (L::cy(i) != 0) jy = fma(C(L::cy(i)), df, jy);
        if constexpr (L::cz(i) != 0) jz = fma(C(L::cz(i)), df, jz);
        H += hp;
        if constexpr (std::is_same<C, double>::value) {  // the group first: one instruction less per pair
          constexpr bool first = i == IB || i - 2 < IB || L::grp(i - 2) != g;
          constexpr bool last = i + 2 >= IE || L::grp(i + 2 < L::Q ? i + 2 : i) != g;
          gs = first ? sp : gs + sp;
          if constexpr (last) {
            m += gs;
            k2 = fma(C(L::c2(i)), gs, k2);
          }
        } else {
          m += sp;
          k2 = fma(C(L::c2(i)), sp, k2);
        }
      }
    }
  });
  (void)s2;
  (void)s3;
  (void)gs;
  acc[0] = m;
  acc[1] = jx;
  acc[2] = jy;
  acc[3] = jz;
  acc[4] = fma(a.half_r2, k2, H);
}

// drho, u, dT of a cell from its summed partials (the closing lines of
// moments_raw with dK + dH = acc[4])
template <int LAT, class C>
__device__ __forceinline__ void moments_finish(const C (&acc)[5], const Args<C>& a, C& drho, C (&u)[3], C& dT) {
  using L = Lat<LAT>;
  const C m = acc[0];
  const C rho = a.rho0 + m;
  const C inv = C(1) / rho;
  drho = m;
  u[0] = a.r * acc[1] * inv;
  u[1] = a.r * acc[2] * inv;
  u[2] = (L::D == 3) ? a.r * acc[3] * inv : C(0);
  const C u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  dT = (C(2) * acc[4] - rho * u2 - a.Dd * a.T0 * m) * inv * a.inv_Dd;
}

// ---------------------------------------------------------------------------
// collide one cell given its pulled deviations and store the result:
//   g* = g~ + omega_f (dF - g~)
//   h* = h~ + omega_g (dFh - h~) = (omega_g hd T) dF + (1 - omega_g) h~ + omega_g hd dT gref
// ---------------------------------------------------------------------------
// For 16-bit storage the accessors return the stored d, e and the new values
// are formed directly in the stored scale:
//   d* = d + omega_f (dF / gref - d),  e* = (hA / hs) dF + (1 - omega_g) e + hb gref / hs
// FD: the finite-difference variant of Sec. III, which relaxes the cell's own
// values and subtracts the convection term conv(I) = {c_g, c_h} (in the
// stored scale) from the relaxed values.
// relax_store_k: the relaxation and store of the velocities [IB, IE) of a
// cell whose equilibrium coefficients k (formed from its moments by
// eq_coeffs) are known; cell is the element index within a plane (32 bits:
// below 2^32 cells per instance)
// relax_put_k: the same with put(I, g, h) receiving the new values (16-bit
// storage: before packing) instead of the store
template <int LAT, class S, class C, bool FD, int IB, int IE, class GetG, class GetH, class Conv, class Put>
__device__ __forceinline__ void relax_put_k(GetG&& getg, GetH&& geth, Conv&& conv, const Args<C>& a,
                                            const EqCoef<LAT, C>& k, Put&& put) {
  using L = Lat<LAT>;
  constexpr bool SCALED = IsS16<S>::value;
  const C om1 = C(1) - a.omega_g;
  const C hbs = a.omega_g * a.half_delta * k.dT;
  if constexpr (std::is_same<S, double>::value) {
    // FP64 is bound by its pipe, 2 instructions per SM and clock: with
    // omega_f in the group's weights g* = (1 - omega_f) g + omega_f dF is one
    // instruction instead of two (with the moments' sums by group: D2Q37
    // 1024^2 1101 -> 1035 us per step, D3Q107 256 x 128 x 128 12.7 -> 11.5 ms)
    const C hA = a.hd_fg * k.T;
    C hbg = C(0);
    eq_emit<LAT, C, IB, IE, true>(k, a, [&](auto I, C dFw) {
      constexpr int i = decltype(I)::value;
      if constexpr (i == IB || L::grp(i == 0 ? 0 : i - 1) != L::grp(i)) hbg = hbs * a.gref[L::grp(i)];
      C gn = fma(a.om1_f, getg(I), dFw);
      C hn = fma(hA, dFw, fma(om1, geth(I), hbg));
      if constexpr (FD) {
        const auto cv = conv(I);
        gn -= cv.g;
        hn -= cv.h;
      }
      put(I, gn, hn);
    });
    return;
  }
  const C hA = a.omega_g * a.half_delta * k.T;
  C ig = C(1), hAs = hA, hbg = C(0);  // per-group: 1/gref, hA/hs, hbs gref/hs (16-bit)
  eq_emit<LAT, C, IB, IE>(k, a, [&](auto I, C dF) {
    constexpr int i = decltype(I)::value;
    constexpr int g = L::grp(i);
    const C gi = getg(I), hi = geth(I);
    if constexpr (SCALED) {
      if constexpr (i == IB || L::grp(i == 0 ? 0 : i - 1) != g) {
        ig = a.inv_gref[g];
        hAs = hA * a.inv_hscale[g];
        hbg = hbs * a.gref[g] * a.inv_hscale[g];
      }
      C dn = fma(a.omega_f, fma(dF, ig, -gi), gi);
      C en = fma(hAs, dF, fma(om1, hi, hbg));
      if constexpr (FD) {
        const auto cv = conv(I);
        dn -= cv.g;
        en -= cv.h;
      }
      put(I, dn, en);
    } else {
      C gn = fma(a.omega_f, dF - gi, gi);
      C hn = fma(hA, dF, fma(om1, hi, hbs * a.gref[g]));
      if constexpr (FD) {
        const auto cv = conv(I);
        gn -= cv.g;
        hn -= cv.h;
      }
      put(I, gn, hn);
    }
  });
}

template <int LAT, class S, class C, bool IDX32, bool FD, int IB = 0, int IE = Lat<LAT>::Q, class GetG, class GetH,
          class Conv>
__device__ __forceinline__ void relax_store_k(GetG&& getg, GetH&& geth, Conv&& conv, const Args<C>& a,
                                              const EqCoef<LAT, C>& k, S* __restrict__ dst, long long ps,
                                              unsigned cell) {
  constexpr int Q = Lat<LAT>::Q;
  // IDX32: element index plane * ps + cell in unsigned 32 bits (the caller
  // checked that every element index is below 2^32); else plane base + the
  // cell's byte offset in 64 bits
  char* db = reinterpret_cast<char*>(dst) + (size_t)cell * sizeof(S);
  const size_t pb = (size_t)ps * sizeof(S);
  auto st = [&](int plane, S v) {
    if constexpr (IDX32) dst[(unsigned)plane * (unsigned)ps + cell] = v;
    else *reinterpret_cast<S*>(db + (size_t)plane * pb) = v;
  };
  relax_put_k<LAT, S, C, FD, IB, IE>(getg, geth, conv, a, k, [&](auto I, C gn, C hn) {
    constexpr int i = decltype(I)::value;
    if constexpr (IsS16<S>::value) {  // one 32-bit (g_i, h_i) pair
      unsigned* dp = reinterpret_cast<unsigned*>(dst);
      const unsigned pv = pack16<S>(static_cast<float>(gn), static_cast<float>(hn));
      if constexpr (IDX32) dp[(unsigned)i * (unsigned)ps + cell] = pv;
      else dp[(size_t)i * ps + cell] = pv;
    } else {
      st(i, static_cast<S>(gn));
      st(Q + i, static_cast<S>(hn));
    }
  });
}

// relax_store_k with the equilibrium coefficients formed from the moments
template <int LAT, class S, class C, bool IDX32, bool FD, int IB = 0, int IE = Lat<LAT>::Q, class GetG, class GetH,
          class Conv>
__device__ __forceinline__ void relax_store(GetG&& getg, GetH&& geth, Conv&& conv, const Args<C>& a, C drho,
                                            const C (&u)[3], C dT, S* __restrict__ dst, long long ps,
                                            unsigned cell) {
  EqCoef<LAT, C> k;
  eq_coeffs<LAT, C>(drho, u, dT, a, k);
  relax_store_k<LAT, S, C, IDX32, FD, IB, IE>(getg, geth, conv, a, k, dst, ps, cell);
}

// the moments of a cell as every one-thread-per-cell kernel sums them.  FP64:
// in the four parts of k_step_split, so that the FP64 shapes, and the row and
// the tile kernel of the finite-difference step, give the same bits
template <int LAT, class S, class C, class GetG, class GetH>
__device__ __forceinline__ void moments_cell(GetG&& getg, GetH&& geth, const Args<C>& a, C& drho, C (&u)[3], C& dT) {
  if constexpr (std::is_same<S, double>::value) {
    C sum[5];
    static_for<4>([&](auto W) {
      constexpr int w = decltype(W)::value;
      C acc[5];
      moments_partial<LAT, C, false, Split<LAT, 4>::begin(w), Split<LAT, 4>::end(w)>(getg, geth, a, acc);
#pragma unroll
      for (int k = 0; k < 5; ++k) sum[k] = w == 0 ? acc[k] : sum[k] + acc[k];
    });
    moments_finish<LAT, C>(sum, a, drho, u, dT);
  } else {
    moments_raw<LAT, C, IsS16<S>::value>(getg, geth, a, drho, u, dT);
  }
}

template <int LAT, class S, class C, bool IDX32, bool FD, class GetG, class GetH, class Conv>
__device__ __forceinline__ void collide_store_impl(GetG&& getg, GetH&& geth, Conv&& conv, const Args<C>& a,
                                                   S* __restrict__ dst, long long ps, unsigned cell) {
  C drho, u[3], dT;
  moments_cell<LAT, S, C>(getg, geth, a, drho, u, dT);
  if (!(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
  relax_store<LAT, S, C, IDX32, FD>(getg, geth, conv, a, drho, u, dT, dst, ps, cell);
}

template <class C>
struct ConvGH {
  C g, h;
};

// the stream-and-collide form: no convection term
template <int LAT, class S, class C, bool IDX32, class GetG, class GetH>
__device__ __forceinline__ void collide_store(GetG&& getg, GetH&& geth, const Args<C>& a, S* __restrict__ dst,
                                              long long ps, unsigned cell) {
  collide_store_impl<LAT, S, C, IDX32, false>(getg, geth, [](auto) { return ConvGH<C>{C(0), C(0)}; }, a, dst, ps,
                                              cell);
}

// raw value of a stored population in the compute type (16-bit: the stored
// relative deviation, not decoded)
template <class S, class C>
__device__ __forceinline__ C raw_value(S v) {
  if constexpr (IsS16<S>::value) return static_cast<C>(s16_to_f(v));
  else return static_cast<C>(v);
}

// ---------------------------------------------------------------------------
// the fused step of one cell
//   STAGE 0: the 2Q pulled values live in registers (D2Q37)
//   STAGE 1: they are staged in shared memory by 4/8-byte cp.async (D3Q107,
//            FP32/FP64 storage): no registers held while the loads fly
//   STAGE 3: g in registers, h staged in shared memory by cp.async (D3Q107,
//            FP32/FP64): half the shared memory per cell of STAGE 1
//   STAGE 6: 16-bit storage, the Q pulled (g_i, h_i) pairs held packed in
//            registers (one register per direction, half of STAGE 0's) and
//            unpacked where each pass uses them
//   STAGE 9: 16-bit storage, half the pairs packed in registers and the
//            other half staged in shared memory by cp.async (D3Q107)
// A block covers BX consecutive cells of a row (thread = cell).
// ---------------------------------------------------------------------------
// ROW: the block's row (y, z) lies at least 3 cells from every y and z face,
// so no pull of the row wraps or clamps along y or z: the source row of
// direction i is the cell's own row shifted by -(c_y nx + c_z nx ny), the same
// for every thread.  Only the x part of the pull differs between threads (a
// 7-entry table of byte offsets); plane and row shifts are uniform, and the
// stores address the cell through one per-thread pointer plus the uniform
// plane stride.  The arithmetic is that of the general path.
// UNI (with ROW, any row): the row shift of direction i is not -(c_y nx +
// c_z nx ny) but the block-uniform ysh[c_y + 3] + zsh[c_z + 3], the shifts
// of the pulled row and plane after the y and z rules; the rows within 3
// cells of a y or z face take the ROW path's code with these tables.
template <int LAT, class S, class C, int STAGE, int BX, bool IDX32 = false, bool ROW = false, bool UNI = false>
__device__ __forceinline__ void step_cell(const S* __restrict__ src, S* __restrict__ dst, const Args<C>& a, int x,
                                          int y, int z) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  if (x >= nx) return;
  constexpr size_t E = IsS16<S>::value ? 2 * sizeof(S) : sizeof(S);  // bytes per stored element (pair)
  // source offsets for lattice components c = -3..3 (index c + 3); ROW keeps
  // only xb, the byte offset of the pulled x in the cell's own row
  unsigned xo[ROW ? 1 : 7], yo[ROW ? 1 : 7], zo[ROW ? 1 : 7], xb[ROW ? 7 : 1];
  unsigned ysh[UNI ? 7 : 1], zsh[UNI ? 7 : 1];
  const unsigned rowcell = (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)z);
  if constexpr (UNI) {
    static_assert(ROW && IDX32, "uniform shift tables extend the 32-bit ROW path");
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      ysh[k] = (unsigned)(pull_coord(y, k - 3, ny, a.bc[1]) - y) * (unsigned)nx;
      zsh[k] = (L::D == 3) ? (unsigned)(pull_coord(z, k - 3, nz, a.bc[2]) - z) * ((unsigned)nx * (unsigned)ny) : 0u;
    }
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    if constexpr (ROW) {  // element index of the pulled x in the cell's own row (a byte offset without IDX32)
      xb[k] = (rowcell + (unsigned)pull_coord(x, k - 3, nx, a.bc[0])) * (IDX32 ? 1u : (unsigned)E);
    } else {
      xo[k] = (unsigned)pull_coord(x, k - 3, nx, a.bc[0]);
      yo[k] = (unsigned)pull_coord(y, k - 3, ny, a.bc[1]) * (unsigned)nx;
      zo[k] = (L::D == 3) ? (unsigned)pull_coord(z, k - 3, nz, a.bc[2]) * (unsigned)nx * (unsigned)ny : 0u;
    }
  }
  const unsigned cell = (unsigned)x + rowcell;
  const long long ps = a.ps;
  auto src_off = [&](auto I) -> unsigned {
    constexpr int i = decltype(I)::value;
    if constexpr (ROW) return 0u;  // not used on the ROW path
    else return zo[L::cz(i) + 3] + yo[L::cy(i) + 3] + xo[L::cx(i) + 3];
  };
  // addresses = plane base (uniform across the grid) + per-thread byte
  // offset; g_i and h_i share the offset of direction i
  const char* sb = reinterpret_cast<const char*>(src);
  const size_t pb = (size_t)ps * sizeof(S);
  auto ld = [&](auto I, int plane, size_t offb) -> S {
    return ldg_s(reinterpret_cast<const S*>(sb + (size_t)plane * pb + offb));
  };
  // address of the pulled element of direction I in plane `plane` (pair
  // index for 16-bit storage): IDX32 -- the launcher checked that every
  // element index of the buffer is below 2^32 -- in unsigned 32-bit element
  // arithmetic, else plane base + 64-bit byte offset
  auto pptr = [&](int plane, auto I) -> const char* {
    constexpr int i = decltype(I)::value;
    if constexpr (UNI) {
      const unsigned u = (unsigned)plane * (unsigned)ps + ysh[L::cy(i) + 3] + zsh[L::cz(i) + 3];
      return reinterpret_cast<const char*>(src) + (size_t)(u + xb[L::cx(i) + 3]) * E;
    } else if constexpr (ROW && IDX32) {
      // uniform part plane ps - c_y nx - c_z nx ny plus the thread's x index,
      // in unsigned 32-bit arithmetic: the sum is the element index, below 2^32
      const unsigned u = (unsigned)plane * (unsigned)ps - (unsigned)(L::cy(i) * nx) -
                         (unsigned)(L::cz(i)) * ((unsigned)nx * (unsigned)ny);
      return reinterpret_cast<const char*>(src) + (size_t)(u + xb[L::cx(i) + 3]) * E;
    } else if constexpr (ROW) {
      const long long shift = -((long long)L::cy(i) * nx + (long long)L::cz(i) * nx * ny) * (long long)E;
      return sb + ((long long)plane * ps * (long long)E + shift) + xb[L::cx(i) + 3];
    } else if constexpr (IDX32) {
      return reinterpret_cast<const char*>(src) + (size_t)((unsigned)plane * (unsigned)ps + src_off(I)) * E;
    } else {
      return sb + (size_t)plane * ((size_t)ps * E) + (size_t)src_off(I) * E;
    }
  };
  constexpr bool SIDX32 = IDX32;
  if constexpr (STAGE == 0) {
    C g[Q], h[Q];
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (ROW) {
        if constexpr (IsS16<S>::value) {
          float lo, hi;
          unpack16<S>(__ldg(reinterpret_cast<const unsigned*>(pptr(i, I))), lo, hi);
          g[i] = lo;
          h[i] = hi;
        } else {
          g[i] = raw_value<S, C>(ldg_s(reinterpret_cast<const S*>(pptr(i, I))));
          h[i] = raw_value<S, C>(ldg_s(reinterpret_cast<const S*>(pptr(Q + i, I))));
        }
      } else if constexpr (IsS16<S>::value) {  // one 32-bit pair holds g_i and h_i
        const unsigned* sp = reinterpret_cast<const unsigned*>(src);
        const unsigned v = IDX32 ? __ldg(sp + ((unsigned)i * (unsigned)ps + src_off(I)))
                                 : __ldg(sp + ((size_t)i * ps + src_off(I)));
        float lo, hi;
        unpack16<S>(v, lo, hi);
        g[i] = lo;
        h[i] = hi;
      } else if constexpr (IDX32) {
        const unsigned off = src_off(I);
        g[i] = raw_value<S, C>(ldg_s(src + ((unsigned)i * (unsigned)ps + off)));
        h[i] = raw_value<S, C>(ldg_s(src + ((unsigned)(Q + i) * (unsigned)ps + off)));
      } else {
        const size_t offb = (size_t)src_off(I) * sizeof(S);
        g[i] = raw_value<S, C>(ld(I, i, offb));
        h[i] = raw_value<S, C>(ld(I, Q + i, offb));
      }
    });
    collide_store<LAT, S, C, SIDX32>([&](auto I) { return g[decltype(I)::value]; },
                                     [&](auto I) { return h[decltype(I)::value]; }, a, dst, ps, cell);
  } else if constexpr (STAGE == 6) {
    static_assert(IsS16<S>::value, "packed pairs need 16-bit storage");
    unsigned pr[Q];
    static_for<Q>([&](auto I) {
      pr[decltype(I)::value] = __ldg(reinterpret_cast<const unsigned*>(pptr(decltype(I)::value, I)));
    });
    auto lo = [](unsigned v) -> C {
      float l, h;
      unpack16<S>(v, l, h);
      return static_cast<C>(l);
    };
    auto hi = [](unsigned v) -> C {
      float l, h;
      unpack16<S>(v, l, h);
      return static_cast<C>(h);
    };
    C drho, u[3], dT;
    moments_raw<LAT, C, true>([&](auto I) { return lo(pr[decltype(I)::value]); },
                              [&](auto I) { return hi(pr[decltype(I)::value]); }, a, drho, u, dT);
    if (!(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
    // an empty asm that claims to change each pair: the relaxation pass
    // unpacks again instead of the compiler keeping the moments pass's 2Q
    // unpacked values alive (it emits no instruction)
    static_for<Q>([&](auto I) { asm volatile("" : "+r"(pr[decltype(I)::value])); });
    relax_store<LAT, S, C, SIDX32, false>([&](auto I) { return lo(pr[decltype(I)::value]); },
                                         [&](auto I) { return hi(pr[decltype(I)::value]); },
                                         [](auto) { return ConvGH<C>{C(0), C(0)}; }, a, drho, u, dT, dst, ps, cell);
  } else if constexpr (STAGE == 9) {
    // 16-bit storage: the pairs of the first (Q + 1) / 2 directions held
    // packed in registers (as STAGE 6), the others staged in shared memory
    // slots [i - NR][thread] by 4-byte cp.async (as STAGE 3 stages h), so a
    // thread holds about half the registers of STAGE 6
    static_assert(IsS16<S>::value, "packed pairs need 16-bit storage");
    constexpr int NR = (Q + 1) / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned* sp = reinterpret_cast<unsigned*>(smem_raw);  // [Q - NR][BX]
    const int t = threadIdx.x;
    unsigned pr[NR];
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (i < NR) {
        pr[i] = __ldg(reinterpret_cast<const unsigned*>(pptr(i, I)));
      } else {
        const unsigned sa = (unsigned)__cvta_generic_to_shared(sp + (i - NR) * BX + t);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(pptr(i, I)));
      }
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    const volatile unsigned* spv = sp;
    auto word = [&](auto I) -> unsigned {
      constexpr int i = decltype(I)::value;
      if constexpr (i < NR) return pr[i];
      else return spv[(i - NR) * BX + t];
    };
    auto lo = [&](auto I) -> C {
      float l, h;
      unpack16<S>(word(I), l, h);
      return static_cast<C>(l);
    };
    auto hi = [&](auto I) -> C {
      float l, h;
      unpack16<S>(word(I), l, h);
      return static_cast<C>(h);
    };
    C drho, u[3], dT;
    moments_raw<LAT, C, true>(lo, hi, a, drho, u, dT);
    if (!(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
    // as STAGE 6: the relaxation pass unpacks the held pairs again
    static_for<NR>([&](auto I) { asm volatile("" : "+r"(pr[decltype(I)::value])); });
    relax_store<LAT, S, C, SIDX32, false>(lo, hi, [](auto) { return ConvGH<C>{C(0), C(0)}; }, a, drho, u, dT, dst,
                                         ps, cell);
  } else if constexpr (STAGE == 3) {
    static_assert(sizeof(S) == 4 || sizeof(S) == 8, "cp.async needs 4- or 8-byte elements");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* sh = reinterpret_cast<S*>(smem_raw);  // [Q][BX]: h only
    const int t = threadIdx.x;
    C g[Q];
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      const unsigned sa = (unsigned)__cvta_generic_to_shared(sh + i * BX + t);
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(pptr(Q + i, I)), "n"(sizeof(S)));
      g[i] = static_cast<C>(ldg_s(reinterpret_cast<const S*>(pptr(i, I))));
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    // volatile: the moments pass and the relaxation pass each read h_i from
    // shared memory, so the 107 h values are not all held in registers
    const volatile S* shv = sh;
    collide_store<LAT, S, C, SIDX32>([&](auto I) { return g[decltype(I)::value]; },
                                     [&](auto I) { return static_cast<C>(shv[decltype(I)::value * BX + t]); }, a,
                                     dst, ps, cell);
  } else {
    static_assert(STAGE == 1 && (sizeof(S) == 4 || sizeof(S) == 8), "cp.async needs 4- or 8-byte elements");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* sg = reinterpret_cast<S*>(smem_raw);  // [2Q][BX]
    const int t = threadIdx.x;
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      const unsigned sa0 = (unsigned)__cvta_generic_to_shared(sg + i * BX + t);
      const unsigned sa1 = (unsigned)__cvta_generic_to_shared(sg + (Q + i) * BX + t);
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa0), "l"(pptr(i, I)), "n"(sizeof(S)));
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa1), "l"(pptr(Q + i, I)), "n"(sizeof(S)));
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    // each thread reads back only the slots it filled itself; the reads are
    // volatile so that each pass re-reads shared memory instead of holding
    // every staged value in registers
    const volatile S* sgv = sg;
    collide_store<LAT, S, C, SIDX32>(
        [&](auto I) { return raw_value<S, C>(sgv[decltype(I)::value * BX + t]); },
        [&](auto I) { return raw_value<S, C>(sgv[(Q + decltype(I)::value) * BX + t]); }, a, dst, ps, cell);
  }
}

// Rows a launch of k_step covers:
//   kRowsAll:      every row (block (x, y, z)); a block whose row lies 3 or
//                  more cells from every y and z face takes the ROW
//                  addressing (the branch is uniform over the block), the
//                  others, and grids too small to have such rows, the
//                  general one.  One kernel, both code paths.
//   kRowsInterior: only those rows (block (x, y - 3, z - 3)), ROW addressing
//   kRowsBoundary: only the other rows of a 3D grid (block (x, k): the k-th
//                  row of the 3-cell z slabs, then of the 3-cell y slabs of
//                  the interior z), ROW addressing with block-uniform row
//                  shift tables (UNI)
//   kRowsUniform:  block (x, y, z) for every row of a 3D grid, all with the
//                  ROW path's code and block-uniform row shift tables (UNI)
// A 3D grid launches kRowsUniform (FP32 storage) or kRowsInterior then
// kRowsBoundary (16-bit storage), so each kernel carries one code path.
//   kRowsFlat:     the cells of a 2D grid in their order in memory (block
//                  (x)), whatever row they are in: where rows are no multiple
//                  of 32 cells, the stores of row-wise blocks straddle the
//                  32-byte sectors and their last block is partly empty.  The
//                  general addressing, one integer addition more per load.
constexpr int kRowsAll = 0, kRowsInterior = 1, kRowsBoundary = 2, kRowsUniform = 3, kRowsFlat = 4;

__device__ __forceinline__ void boundary_row(int k, int ny, int nz, int& y, int& z) {
  if (k < 6 * ny) {
    const int zz = k / ny;
    z = zz < 3 ? zz : nz - 6 + zz;
    y = k - zz * ny;
  } else {
    const int kk = k - 6 * ny;
    z = 3 + kk / 6;
    const int yy = kk - (kk / 6) * 6;
    y = yy < 3 ? yy : ny - 6 + yy;
  }
}

template <int LAT, class S, class C, int STAGE, int BX, int MINB = 1, bool IDX32 = false, int ROWS = kRowsAll>
__global__ void __launch_bounds__(BX, MINB) k_step(const S* __restrict__ src, S* __restrict__ dst, const Args<C> a) {
  wait_for_previous_kernel();
  const int x = blockIdx.x * BX + threadIdx.x;
  if constexpr (ROWS == kRowsFlat) {
    const int y = x / a.n[0];
    if (y < a.n[1]) step_cell<LAT, S, C, STAGE, BX, IDX32, false>(src, dst, a, x - y * a.n[0], y, 0);
  } else if constexpr (ROWS == kRowsInterior) {
    step_cell<LAT, S, C, STAGE, BX, IDX32, true>(src, dst, a, x, blockIdx.y + 3, blockIdx.z + 3);
  } else if constexpr (ROWS == kRowsUniform) {
    step_cell<LAT, S, C, STAGE, BX, true, true, true>(src, dst, a, x, blockIdx.y, blockIdx.z);
  } else if constexpr (ROWS == kRowsBoundary) {
    int y, z;
    boundary_row(blockIdx.y, a.n[1], a.n[2], y, z);
    // the ROW path's code with block-uniform row shifts (UNI), where element
    // indices fit 32 bits; else the general path
    if constexpr (IDX32) step_cell<LAT, S, C, STAGE, BX, true, true, true>(src, dst, a, x, y, z);
    else step_cell<LAT, S, C, STAGE, BX, IDX32, false>(src, dst, a, x, y, z);
  } else {
    const int y = blockIdx.y, z = blockIdx.z;
    // (the per-thread byte offsets of the ROW path are 32-bit: N E < 2^32)
    constexpr long long E = IsS16<S>::value ? 2 * (long long)sizeof(S) : (long long)sizeof(S);
    const bool row = y >= 3 && y < a.n[1] - 3 && (Lat<LAT>::D == 2 || (z >= 3 && z < a.n[2] - 3)) &&
                     (long long)a.n[0] * a.n[1] * a.n[2] * E < (1LL << 32);
    if (row)
      step_cell<LAT, S, C, STAGE, BX, IDX32, true>(src, dst, a, x, y, z);
    else
      step_cell<LAT, S, C, STAGE, BX, IDX32, false>(src, dst, a, x, y, z);
  }
}

// ---------------------------------------------------------------------------
// the velocity-split step (STAGE 4): a block of P warps covers 32 cells of a
// row; warp w pulls, sums and relaxes only its part [begin(w), end(w)) of the
// velocities.  The parts' five partial sums meet in shared memory and every
// warp adds them in the same order, so all parts use identical moments.
// Each thread holds 2 (end - begin) values instead of 2Q, which keeps the
// register count near that of the D2Q37 kernel for D3Q107.
// ---------------------------------------------------------------------------
// SHARE: warp 0 alone finishes the moments and forms the equilibrium
// coefficients, which the other warps read from shared memory after a second
// barrier (less arithmetic per cell; worth it where the FP64 pipe is the bound)
template <int LAT, class S, class C, int P, int MINB, bool SHARE = false>
__global__ void __launch_bounds__(32 * P, MINB) k_step_split(const S* __restrict__ src, S* __restrict__ dst,
                                                            const Args<C> a) {
  using L = Lat<LAT>;
  using SP = Split<LAT, P>;
  constexpr int Q = L::Q;
  constexpr int K = SP::kmax();
  constexpr bool SCALED = IsS16<S>::value;
  __shared__ C red[P][5][32];
  wait_for_previous_kernel();
  const int lane = threadIdx.x, w = threadIdx.y;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  const int x = blockIdx.x * 32 + lane, y = blockIdx.y, z = blockIdx.z;
  const bool active = x < nx;
  const int xs = active ? x : nx - 1;  // lanes past the row end pull from a valid cell and store nothing
  unsigned xo[7], yo[7], zo[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    xo[k] = (unsigned)pull_coord(xs, k - 3, nx, a.bc[0]);
    yo[k] = (unsigned)pull_coord(y, k - 3, ny, a.bc[1]) * (unsigned)nx;
    zo[k] = (L::D == 3) ? (unsigned)pull_coord(z, k - 3, nz, a.bc[2]) * (unsigned)nx * (unsigned)ny : 0u;
  }
  const unsigned cell = (unsigned)xs + (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)z);
  const long long ps = a.ps;
  const char* sb = reinterpret_cast<const char*>(src);
  const size_t pb = (size_t)ps * sizeof(S);
  C g[K], h[K];
  // phase 1: pull this warp's velocities and sum its partial moments
  static_for<P>([&](auto W) {
    constexpr int IB = SP::begin(decltype(W)::value), IE = SP::end(decltype(W)::value);
    if (w == decltype(W)::value) {
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (i >= IB && i < IE) {
          const unsigned off = zo[L::cz(i) + 3] + yo[L::cy(i) + 3] + xo[L::cx(i) + 3];
          if constexpr (SCALED) {
            const unsigned v = __ldg(reinterpret_cast<const unsigned*>(src) + ((size_t)i * ps + off));
            float lo, hi;
            unpack16<S>(v, lo, hi);
            g[i - IB] = lo;
            h[i - IB] = hi;
          } else {
            const size_t offb = (size_t)off * sizeof(S);
            g[i - IB] = static_cast<C>(ldg_s(reinterpret_cast<const S*>(sb + (size_t)i * pb + offb)));
            h[i - IB] = static_cast<C>(ldg_s(reinterpret_cast<const S*>(sb + (size_t)(Q + i) * pb + offb)));
          }
        }
      });
      C acc[5];
      moments_partial<LAT, C, SCALED, IB, IE>([&](auto I) { return g[decltype(I)::value - IB]; },
                                              [&](auto I) { return h[decltype(I)::value - IB]; }, a, acc);
#pragma unroll
      for (int k = 0; k < 5; ++k) red[w][k][lane] = acc[k];
    }
  });
  __syncthreads();
  auto finish = [&](EqCoef<LAT, C>& k) {  // sum the parts in a fixed order, then the cell's coefficients
    C acc[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      C v = red[0][q][lane];
#pragma unroll
      for (int p = 1; p < P; ++p) v += red[p][q][lane];
      acc[q] = v;
    }
    C drho, u[3], dT;
    moments_finish<LAT, C>(acc, a, drho, u, dT);
    if (w == 0 && active && !(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
    eq_coeffs<LAT, C>(drho, u, dT, a, k);
  };
  EqCoef<LAT, C> k;
  if constexpr (SHARE) {
    __shared__ EqCoef<LAT, C> shk[32];
    if (w == 0) {
      finish(k);
      shk[lane] = k;
    }
    __syncthreads();
    if (w != 0) k = shk[lane];
  } else {
    finish(k);
  }
  if (!active) return;
  // phase 2: relax and store this warp's velocities
  static_for<P>([&](auto W) {
    constexpr int IB = SP::begin(decltype(W)::value), IE = SP::end(decltype(W)::value);
    if (w == decltype(W)::value)
      relax_store_k<LAT, S, C, false, false, IB, IE>(
          [&](auto I) { return g[decltype(I)::value - IB]; }, [&](auto I) { return h[decltype(I)::value - IB]; },
          [](auto) { return ConvGH<C>{C(0), C(0)}; }, a, k, dst, ps, cell);
  });
}

// ---------------------------------------------------------------------------
// the mirror-pair step (STAGE 8): every cell is worked by two lanes of one
// warp, lane l and lane l ^ 16.  The lower half-warp (half 0, sign +1) takes
// the member c of each (c, -c) pair and the rest velocity; the upper half
// (half 1, sign -1) takes the member -c.  Both halves run one instruction
// stream:
//   - the pull of -c reads x + c, so the sign is folded into the 7-entry
//     offset tables of each axis, and the member -c lies one plane after c;
//   - s(-c; u) = s(c; -u): with u negated the pair's even part e(s^2) is the
//     same and the odd part flips, so each half stores e + o with its own
//     sign of u;
//   - the five moment sums of the halves meet by one __shfl_xor_sync each;
//     both lanes add (or subtract) the two halves' partial sums in the same
//     operand order, so they hold bitwise identical moments.
// A thread holds the (Q + 1) / 2 pulled (g, h) of its half instead of Q, so
// about twice the warps fit per SM; the pair's even and odd parts are formed
// by both lanes.  A block of BX threads covers BX / 2 cells of a row; lanes
// past the row end pull from a valid cell, take part in the shuffles and
// store nothing.
// ---------------------------------------------------------------------------
template <int LAT, class S, class C, int BX, int MINB, bool IDX32, bool HS>
__global__ void __launch_bounds__(BX, MINB) k_step_mirror(const S* __restrict__ src, S* __restrict__ dst,
                                                         const Args<C> a) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  constexpr int NP = (Q - 1) / 2;  // (c, -c) pairs; pair k is velocities 2k+1 (c) and 2k+2 (-c)
  constexpr bool SCALED = IsS16<S>::value;
  static_assert(BX % 32 == 0, "whole warps");
  static_assert(!(HS && SCALED), "16-bit pairs are held packed in registers");
  wait_for_previous_kernel();
  const int lane = threadIdx.x & 31;
  const int half = lane >> 4;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  const int x = blockIdx.x * (BX / 2) + (threadIdx.x >> 5) * 16 + (lane & 15);
  const int y = blockIdx.y, z = blockIdx.z;
  const bool active = x < nx;
  const int xs = active ? x : nx - 1;
  const int sg = half ? -1 : 1;
  // source offsets of the pull of sg * c for c = -3..3 (index c + 3)
  unsigned xo[7], yo[7], zo[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    xo[k] = (unsigned)pull_coord(xs, sg * (k - 3), nx, a.bc[0]);
    yo[k] = (unsigned)pull_coord(y, sg * (k - 3), ny, a.bc[1]) * (unsigned)nx;
    zo[k] = (L::D == 3) ? (unsigned)pull_coord(z, sg * (k - 3), nz, a.bc[2]) * (unsigned)nx * (unsigned)ny : 0u;
  }
  const unsigned cell = (unsigned)xs + (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)z);
  const long long ps = a.ps;
  // element index of this half's member in plane `plane` (pair index for
  // 16-bit storage) at cell offset off
  auto eidx = [&](int plane, unsigned off) -> size_t {
    if constexpr (IDX32) return (size_t)((unsigned)(plane + half) * (unsigned)ps + off);
    else return (size_t)(plane + half) * (size_t)ps + off;
  };
  // the pulled values: FP32/FP64 g in registers and h in registers or (HS)
  // in shared memory slots [k][thread] filled by cp.async; 16-bit storage
  // the packed (g, h) pairs in registers.  The rest velocity is pulled by
  // half 0 only (half 1 keeps zeros).
  C g0 = C(0), h0 = C(0);
  C g[SCALED ? 1 : NP];
  C h[(SCALED || HS) ? 1 : NP];
  unsigned pr[SCALED ? NP : 1];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S* shh = reinterpret_cast<S*>(smem_raw);  // HS: [NP][BX]
  if (half == 0) {
    if constexpr (SCALED) {
      float lo, hi;
      unpack16<S>(__ldg(reinterpret_cast<const unsigned*>(src) + (size_t)cell), lo, hi);
      g0 = lo;
      h0 = hi;
    } else {
      g0 = static_cast<C>(ldg_s(src + (size_t)cell));
      h0 = static_cast<C>(ldg_s(src + (size_t)Q * (size_t)ps + cell));
    }
  }
  static_for<NP>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int i = 2 * k + 1;
    const unsigned off = zo[L::cz(i) + 3] + yo[L::cy(i) + 3] + xo[L::cx(i) + 3];
    if constexpr (SCALED) {
      pr[k] = __ldg(reinterpret_cast<const unsigned*>(src) + eidx(i, off));
    } else {
      if constexpr (HS) {
        static_assert(sizeof(S) == 4 || sizeof(S) == 8, "cp.async needs 4- or 8-byte elements");
        const unsigned sa = (unsigned)__cvta_generic_to_shared(shh + k * BX + threadIdx.x);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(src + eidx(Q + i, off)),
                     "n"(sizeof(S)));
      } else {
        h[k] = static_cast<C>(ldg_s(src + eidx(Q + i, off)));
      }
      g[k] = static_cast<C>(ldg_s(src + eidx(i, off)));
    }
  });
  if constexpr (HS) asm volatile("cp.async.wait_all;\n" ::: "memory");
  // accessors of the pulled g, h of pair k (16-bit: the stored relative
  // deviations, unpacked where they are used; HS: h re-read from shared
  // memory by each pass)
  const volatile S* shv = shh;
  auto getg = [&](int k) -> C {
    if constexpr (SCALED) {
      float lo, hi;
      unpack16<S>(pr[k], lo, hi);
      return static_cast<C>(lo);
    } else {
      return g[k];
    }
  };
  auto geth = [&](int k) -> C {
    if constexpr (SCALED) {
      float lo, hi;
      unpack16<S>(pr[k], lo, hi);
      return static_cast<C>(hi);
    } else if constexpr (HS) {
      return static_cast<C>(shv[k * BX + threadIdx.x]);
    } else {
      return h[k];
    }
  };
  // this half's partial sums, with the member c's components (for half 1
  // the momentum sums are minus its share)
  C m, H, jx = C(0), jy = C(0), jz = C(0), k2 = C(0);
  if constexpr (SCALED) {
    m = a.gref[0] * g0;
    H = a.hscale[0] * h0;
  } else {
    m = g0;
    H = h0;
  }
  {
    C s1 = C(1), sc2 = C(0), sh = C(1);
    static_for<NP>([&](auto K) {
      constexpr int k = decltype(K)::value;
      constexpr int i = 2 * k + 1;
      constexpr int gr = L::grp(i);
      const C gk = getg(k), hk = geth(k);
      if constexpr (SCALED) {
        if constexpr (k == 0 || L::grp(i - 2) != gr) {
          s1 = a.gref[gr];
          sc2 = C(L::c2(i)) * s1;
          sh = a.hscale[gr];
        }
        const C gv = s1 * gk;
        m += gv;
        if constexpr (L::cx(i) != 0) jx = fma(C(L::cx(i)), gv, jx);
        if constexpr (L::cy(i) != 0) jy = fma(C(L::cy(i)), gv, jy);
        if constexpr (L::cz(i) != 0) jz = fma(C(L::cz(i)), gv, jz);
        k2 = fma(sc2, gk, k2);
        H = fma(sh, hk, H);
      } else {
        m += gk;
        if constexpr (L::cx(i) != 0) jx = fma(C(L::cx(i)), gk, jx);
        if constexpr (L::cy(i) != 0) jy = fma(C(L::cy(i)), gk, jy);
        if constexpr (L::cz(i) != 0) jz = fma(C(L::cz(i)), gk, jz);
        k2 = fma(C(L::c2(i)), gk, k2);
        H += hk;
      }
    });
    (void)s1;
    (void)sc2;
    (void)sh;
  }
  const C e4 = fma(a.half_r2, k2, H);
  // combine the halves: lower + upper for the even sums, lower - upper for
  // the momentum; both lanes evaluate the same operation on the same operands
  C acc[5];
  {
    const C own[5] = {m, jx, jy, jz, e4};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (q == 3 && L::D == 2) {
        acc[q] = C(0);
        continue;
      }
      const C other = __shfl_xor_sync(0xffffffffu, own[q], 16);
      const C lo = half ? other : own[q];
      const C up = half ? own[q] : other;
      acc[q] = (q >= 1 && q <= 3) ? lo - up : lo + up;
    }
  }
  C drho, u[3], dT;
  moments_finish<LAT, C>(acc, a, drho, u, dT);
  if (active && half == 0 && !(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
  if constexpr (SCALED) {
    // an empty asm that claims to change each pair: the relaxation pass
    // unpacks again instead of keeping the moments pass's unpacked values
    // alive (it emits no instruction)
    static_for<NP>([&](auto K) { asm volatile("" : "+r"(pr[decltype(K)::value])); });
  }
  EqCoef<LAT, C> kc;
  eq_coeffs<LAT, C>(drho, u, dT, a, kc);
  // this half's sign of u: s of the member -c is s(c) at -u
#pragma unroll
  for (int q = 0; q < 3; ++q) kc.ur[q] = half ? -kc.ur[q] : kc.ur[q];
  // relax and store
  const C hA = a.omega_g * a.half_delta * kc.T;
  const C om1 = C(1) - a.omega_g;
  const C hbs = a.omega_g * a.half_delta * kc.dT;
  auto store = [&](int i, unsigned plane_half, C gn, C hn) {
    // the stored plane is i + plane_half
    if constexpr (SCALED) {
      unsigned* dp = reinterpret_cast<unsigned*>(dst);
      const unsigned pv = pack16<S>(static_cast<float>(gn), static_cast<float>(hn));
      if constexpr (IDX32) dp[(unsigned)(i + plane_half) * (unsigned)ps + cell] = pv;
      else dp[(size_t)(i + plane_half) * ps + cell] = pv;
    } else {
      if constexpr (IDX32) {
        dst[(unsigned)(i + plane_half) * (unsigned)ps + cell] = static_cast<S>(gn);
        dst[(unsigned)(Q + i + plane_half) * (unsigned)ps + cell] = static_cast<S>(hn);
      } else {
        dst[(size_t)(i + plane_half) * ps + cell] = static_cast<S>(gn);
        dst[(size_t)(Q + i + plane_half) * ps + cell] = static_cast<S>(hn);
      }
    }
  };
  // per group: the equilibrium coefficients c0..c4 and the relaxation's
  // constants (ig = 1/gref, hAs = hA/hscale, hbg = hbs gref/hscale for
  // 16-bit storage; hAs = hA, hbg = hbs gref otherwise)
  C c0, c1, c2, c3, c4, ig, hAs, hbg;
  auto group = [&](int gr) {
    const C x2 = a.x2g[gr];
    const C P = fma(x2, fma(x2, kc.pc, kc.pb), kc.pa);
    const C W = a.wg[gr] * kc.rho;
    c0 = a.wg[gr] * fma(kc.drho, C(1) + P, a.rho0 * (P - a.pref[gr]));
    c1 = W * fma(kc.be1, x2, kc.be0);
    c2 = W * fma(kc.ga1, x2, kc.ga0);
    c3 = W * C(1.0 / 6.0);
    c4 = W * C(1.0 / 24.0);
    if constexpr (SCALED) {
      ig = a.inv_gref[gr];
      hAs = hA * a.inv_hscale[gr];
      hbg = hbs * a.gref[gr] * a.inv_hscale[gr];
    } else {
      ig = C(1);
      hAs = hA;
      hbg = hbs * a.gref[gr];
    }
  };
  auto relax = [&](C dF, C gv, C hv, C& gn, C& hn) {
    if constexpr (SCALED) gn = fma(a.omega_f, fma(dF, ig, -gv), gv);
    else gn = fma(a.omega_f, dF - gv, gv);
    hn = fma(hAs, dF, fma(om1, hv, hbg));
  };
  group(0);
  if (active && half == 0) {
    C gn, hn;
    relax(c0, g0, h0, gn, hn);
    store(0, 0u, gn, hn);
  }
  static_for<NP>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int i = 2 * k + 1;
    constexpr int gr = L::grp(i);
    if constexpr (k == 0 || L::grp(i - 2) != gr) group(gr);
    C s = C(0);
    if constexpr (L::cx(i) != 0) s = fma(C(L::cx(i)), kc.ur[0], s);
    if constexpr (L::cy(i) != 0) s = fma(C(L::cy(i)), kc.ur[1], s);
    if constexpr (L::cz(i) != 0) s = fma(C(L::cz(i)), kc.ur[2], s);
    const C s2 = s * s;
    const C e = fma(s2, fma(s2, c4, c2), c0);
    const C o = s * fma(s2, c3, c1);
    C gn, hn;
    relax(e + o, getg(k), geth(k), gn, hn);
    if (active) store(i, (unsigned)half, gn, hn);
  });
}

// ---------------------------------------------------------------------------
// two steps of a D2Q37 FP32 grid in one launch
//
// A single step of a large grid runs at the memory's copy rate (1433 us per
// 4096^2 step, 1.02 of it), so what is left is to move the state less often.
// A block marches down a strip of columns.  Two of its four groups of warps
// (A) do the first step, one row after the other, and put the new
// populations into shared memory; the other two (B) do the second step a few
// rows behind, from there, and store the result.  The state between the two
// steps never leaves the SM: a cell costs one read and one write of its
// populations per two steps.
//   Ring: the population of direction i of row r is pulled by row r + c_y,
// so it is kept until B has pulled that row: c_y + 5 rows, 5 on average over
// the lattice, 189 KB at 128 columns, one block per SM.  The directions of
// one c_y share a region [row slot][plane][column].
//   Order: A's groups take the even and the odd rows, B's likewise, so that
// one group's loads overlap the other's arithmetic (16 warps of 128
// registers).  A stores row t once B has pulled row t - 8 of the band, B
// pulls row q once A's rows up to q + 6 are stored; both wait on mbarriers, by
// the rules of pair_order.h, which says why no wait can miss its phase.
//   A's columns are the strip's w and 3 on each side, its rows the band's
// and 3 above and below, each mapped to a grid cell by the axis' rule
// (wrapped, or the edge cell's again at a zero-gradient end), so B pulls
// without any boundary case.  Neighbouring strips repeat those cells' first
// step.  Every cell's arithmetic is that of the single step, bit for bit.
//   Measured, us per step, single -> pair: 4096^2 1433 -> 1144, 2048^2 361 ->
// 284, 1024^2 92.6 -> 77.5, 2999 x 1777 519 -> 377.  It is bound by A's wait
// for its loads (5000 of a group's 10000 cycles per row).  Also built: one
// group each for A and B with the next row's loads in registers (255 of
// them) and a block barrier per row, 1521 us; A's loads by cp.async into
// shared memory two rows ahead, 96 columns, 12 warps, 1156; two columns per
// thread in f32x2 arithmetic, 0.64 of the instructions but 8 warps, 1387;
// rows brought to L2 ahead of the loads, 1400 - 1500.
// ---------------------------------------------------------------------------
struct PairRing {
  static constexpr int cy(int i) { return Lat<0>::cy(i); }
  static constexpr int depth(int k) { return k + 2; }  // rows kept of the directions with c_y = k - 3
  static constexpr int members(int k) {
    int n = 0;
    for (int i = 0; i < 37; ++i) n += cy(i) == k - 3;
    return n;
  }
  static constexpr int rank(int i) {
    int n = 0;
    for (int j = 0; j < i; ++j) n += cy(j) == cy(i);
    return n;
  }
  // words per column of one row slot, and the region's first word per column
  static constexpr int row(int k, int planes) { return members(k) * planes; }
  static constexpr int begin(int k, int planes) {
    int n = 0;
    for (int j = 0; j < k; ++j) n += row(j, planes) * depth(j);
    return n;
  }
  static constexpr size_t bytes(int planes) { return sizeof(unsigned) * kPairW * (size_t)begin(7, planes); }
};

__device__ __forceinline__ int map_coord(int q, int n, int bc) {
  if (bc == kPeriodic) {
    while (q < 0) q += n;
    while (q >= n) q -= n;
    return q;
  }
  return q < 0 ? 0 : (q > n - 1 ? n - 1 : q);
}

// mbarriers of the ring (one arrival per warp of a group); a wait gives up
// after a number of tries of about a microsecond each, so that no fault
// elsewhere can leave a block spinning (lbm_set_wait_limit)

__device__ __forceinline__ void bar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(b)), "r"(count));
}
__device__ __forceinline__ void bar_arrive(unsigned long long* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((unsigned)__cvta_generic_to_shared(b)) : "memory");
}
__device__ __forceinline__ bool bar_wait(unsigned long long* b, unsigned parity, int tries) {
  const unsigned at = (unsigned)__cvta_generic_to_shared(b);
  unsigned done = 0;
  for (int n = 0; n < tries && !done; ++n)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(at), "r"(parity)
        : "memory");
  return __all_sync(0xffffffffu, done != 0);
}

template <bool IDX32>
__global__ void __launch_bounds__(4 * kPairW, 1) k_step_pair(const float* __restrict__ src, float* __restrict__ dst,
                                                             const Args<float> a, int w, int tries) {
  using L = Lat<0>;
  using S = float;
  using C = float;
  constexpr int Q = L::Q, W = kPairW, NPL = 2, NB = kPairBars;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long stored[NB], pulled[NB];  // A's row t, B's row q (mod NB)
  wait_for_previous_kernel();
  S* ring = reinterpret_cast<S*>(smem_raw);
  const int nx = a.n[0], ny = a.n[1];
  const int x0 = blockIdx.x * w;
  const int y0 = (int)((long long)ny * blockIdx.y / gridDim.y), y1 = (int)((long long)ny * (blockIdx.y + 1) / gridDim.y);
  const int rows = y1 - y0;
  const long long ps = a.ps;
  const int j = threadIdx.x & (W - 1), group = threadIdx.x / W;  // 0, 1: A's even and odd rows; 2, 3: B's
  if (threadIdx.x < NB) {
    bar_init(stored + threadIdx.x, W / 32);
    bar_init(pulled + threadIdx.x, W / 32);
  }
  __syncthreads();
  auto arrive = [&](unsigned long long* b) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) bar_arrive(b);
  };
  auto wait = [&](unsigned long long* b, int n) {  // for row n's arrivals
    const bool ok = bar_wait(b + (n & (NB - 1)), (n / NB) & 1, tries);
    if (!ok) atomicOr(a.flag, 2u);
    return ok;
  };
  // first word (of column 0) of the slot of A's row t in the region of c_y = k - 3, and that two rows later
  auto slot_of = [](auto K, int t) {
    constexpr int k = decltype(K)::value;
    constexpr int step = PairRing::row(k, NPL) * W, first = PairRing::begin(k, NPL) * W, d = PairRing::depth(k);
    return first + (t % d) * step;
  };
  auto two_later = [](auto K, int s) {
    constexpr int k = decltype(K)::value;
    constexpr int step = PairRing::row(k, NPL) * W, end = PairRing::begin(k + 1, NPL) * W;
    s += 2 * step;
    return s >= end ? s - step * PairRing::depth(k) : s;
  };
  int slot[7];
  if (group < 2) {
    const bool active = j < w + 6;
    const int mine = rows + 6;  // the band's rows and 3 on each side
    unsigned xb[7];
    {
      const int x = map_coord(x0 - 3 + j, nx, a.bc[0]);
#pragma unroll
      for (int k = 0; k < 7; ++k) xb[k] = (unsigned)pull_coord(x, k - 3, nx, a.bc[0]);
    }
    static_for<7>([&](auto K) { slot[decltype(K)::value] = slot_of(K, group); });
    for (int t = group; t < mine; t += 2) {
      C g[Q], h[Q];
      if (active) {
        const int y = map_coord(y0 - 3 + t, ny, a.bc[1]);
        unsigned yo[7];
#pragma unroll
        for (int k = 0; k < 7; ++k) yo[k] = (unsigned)pull_coord(y, k - 3, ny, a.bc[1]) * (unsigned)nx;
        static_for<Q>([&](auto I) {
          constexpr int i = decltype(I)::value;
          auto at = [&](int plane) {
            if constexpr (IDX32) return src + (size_t)((unsigned)plane * (unsigned)ps + yo[L::cy(i) + 3] + xb[L::cx(i) + 3]);
            else return src + ((size_t)plane * (size_t)ps + yo[L::cy(i) + 3] + xb[L::cx(i) + 3]);
          };
          g[i] = __ldg(at(i));
          h[i] = __ldg(at(Q + i));
        });
      }
      auto getg = [&](auto I) { return g[decltype(I)::value]; };
      auto geth = [&](auto I) { return h[decltype(I)::value]; };
      EqCoef<0, C> k;
      if (active) {
        C drho, u[3], dT;
        moments_raw<0, C, false>(getg, geth, a, drho, u, dT);
        if (!(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
        eq_coeffs<0, C>(drho, u, dT, a, k);
      }
      if (pair_a_pulled(t) >= 0 && !wait(pulled, pair_a_pulled(t))) return;
      if (pair_a_stored(t) >= 0 && !wait(stored, pair_a_stored(t))) return;
      if (active)
        relax_put_k<0, S, C, false, 0, Q>(getg, geth, [](auto) { return ConvGH<C>{C(0), C(0)}; }, a, k,
                                          [&](auto I, C gn, C hn) {
                                            constexpr int i = decltype(I)::value, kc = L::cy(i) + 3;
                                            constexpr int pl = NPL * PairRing::rank(i);
                                            S* p = ring + slot[kc] + j;
                                            p[pl * W] = gn;
                                            p[(pl + 1) * W] = hn;
                                          });
      arrive(stored + (t & (NB - 1)));
      static_for<7>([&](auto K) { slot[decltype(K)::value] = two_later(K, slot[decltype(K)::value]); });
    }
  } else {
    const bool active = j < w && x0 + j < nx;
    // B's row q pulls direction i from A's row q + 3 - c_y
    static_for<7>([&](auto K) { slot[decltype(K)::value] = slot_of(K, group - 2 + 6 - decltype(K)::value); });
    for (int q = group - 2; q < rows; q += 2) {
      for (int n = pair_b_begin(q); n <= pair_b_end(q); ++n)
        if (!wait(stored, n)) return;
      C g[Q], h[Q];
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value, kc = L::cy(i) + 3;
        constexpr int pl = NPL * PairRing::rank(i);
        const S* p = ring + slot[kc] + (active ? j : 0) + 3 - L::cx(i);
        g[i] = p[pl * W];
        h[i] = p[(pl + 1) * W];
      });
      arrive(pulled + (q & (NB - 1)));
      if (active)
        collide_store<0, S, C, IDX32>([&](auto I) { return g[decltype(I)::value]; },
                                      [&](auto I) { return h[decltype(I)::value]; }, a, dst, ps,
                                      (unsigned)nx * (unsigned)(y0 + q) + (unsigned)(x0 + j));
      static_for<7>([&](auto K) { slot[decltype(K)::value] = two_later(K, slot[decltype(K)::value]); });
    }
  }
}

// ---------------------------------------------------------------------------
// the finite-difference variant of Sec. III (Eq. (16)/(17) with the
// convection term discretised along each axis by the third-order upwind
// difference; the printed g_j is read as g_i), lamr = lambda r, lambda = dt/dx:
//   q*_i = q_i - lambda xi_i . D(q_i) - omega (q_i - Q_eq,i)
//   D_a(q) at p for c_a > 0: [q(p-2) - 6 q(p-1) + 3 q(p) + 2 q(p+1)] / 6
//                 for c_a < 0: [-q(p+2) + 6 q(p+1) - 3 q(p) - 2 q(p-1)] / 6
// One thread per cell; the own 2Q values in registers, the upwind neighbours
// read per direction (their reuse across the block is served by L1/L2).
// ---------------------------------------------------------------------------
template <int LAT, class S, class C, int BX>
__global__ void __launch_bounds__(BX) k_step_fd(const S* __restrict__ src, S* __restrict__ dst, const Args<C> a,
                                                C lamr) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  wait_for_previous_kernel();
  const int x = blockIdx.x * BX + threadIdx.x;
  const int y = blockIdx.y, z = blockIdx.z;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  if (x >= nx) return;
  // positions p + k, k = -2..2 (index k + 2), after the boundary rule
  unsigned xp[5], yp[5], zp[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    xp[k] = (unsigned)pull_coord(x, 2 - k, nx, a.bc[0]);
    yp[k] = (unsigned)pull_coord(y, 2 - k, ny, a.bc[1]) * (unsigned)nx;
    zp[k] = (L::D == 3) ? (unsigned)pull_coord(z, 2 - k, nz, a.bc[2]) * (unsigned)nx * (unsigned)ny : 0u;
  }
  const unsigned cell = xp[2] + yp[2] + zp[2];
  const long long ps = a.ps;
  C g[Q], h[Q];
  static_for<Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    ld_gh<Q, S, C>(src, i, ps, cell, g[i], h[i]);
  });
  // upwind differences of g_i and h_i along one axis with position table
  // `pos` (the other two axes at the cell's own position `rest`)
  auto upwind = [&](int i, int sgn, const unsigned (&pos)[5], unsigned rest, C og, C oh, C& dg, C& dh) {
    C gm2, hm2, gm1, hm1, gp1, hp1;  // values at the upwind-2, upwind-1 and downwind-1 positions
    const int u2 = sgn > 0 ? 0 : 4, u1 = sgn > 0 ? 1 : 3, d1 = sgn > 0 ? 3 : 1;
    ld_gh<Q, S, C>(src, i, ps, pos[u2] + rest, gm2, hm2);
    ld_gh<Q, S, C>(src, i, ps, pos[u1] + rest, gm1, hm1);
    ld_gh<Q, S, C>(src, i, ps, pos[d1] + rest, gp1, hp1);
    const C sg = sgn > 0 ? C(1) : C(-1);
    dg = sg * (gm2 - C(6) * gm1 + C(3) * og + C(2) * gp1) * C(1.0 / 6.0);
    dh = sg * (hm2 - C(6) * hm1 + C(3) * oh + C(2) * hp1) * C(1.0 / 6.0);
  };
  auto conv = [&](auto I) {
    constexpr int i = decltype(I)::value;
    constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
    C cg = C(0), ch = C(0), dg, dh;
    if constexpr (cx != 0) {
      upwind(i, cx, xp, yp[2] + zp[2], g[i], h[i], dg, dh);
      cg = fma(C(cx), dg, cg);
      ch = fma(C(cx), dh, ch);
    }
    if constexpr (cy != 0) {
      upwind(i, cy, yp, xp[2] + zp[2], g[i], h[i], dg, dh);
      cg = fma(C(cy), dg, cg);
      ch = fma(C(cy), dh, ch);
    }
    if constexpr (cz != 0) {
      upwind(i, cz, zp, xp[2] + yp[2], g[i], h[i], dg, dh);
      cg = fma(C(cz), dg, cg);
      ch = fma(C(cz), dh, ch);
    }
    return ConvGH<C>{lamr * cg, lamr * ch};
  };
  collide_store_impl<LAT, S, C, false, true>([&](auto I) { return g[decltype(I)::value]; },
                                             [&](auto I) { return h[decltype(I)::value]; }, conv, a, dst, ps,
                                             cell);
}

// ---------------------------------------------------------------------------
// the same in two passes over a tile of BX x BY x BZ cells per block: the
// moments from the cell's own 2Q values, then for each direction the own
// value again, its upwind neighbours, the relaxation and the store; value by
// value the arithmetic of k_step_fd.  Nothing but the moments is held between
// the passes, so many more cells are in flight, and a tile's neighbours along
// y and z are mostly its own cells, found in L1.
//   Measured, us per step, against k_step_fd: D3Q107 (255 registers and
// spills, 8 warps per SM; the loads of 1460 neighbours per cell went to L2)
// 112 x 96 x 80 FP32 2069 -> 800, FP16 storage 940 -> 731; 256 x 128 x 128
// 9879 -> 3820 and 5543 -> 3488.  D2Q37 FP16 storage 4096^2 1789 -> 1537,
// FP32 2613 -> 2690, which keeps k_step_fd; D3Q107 FP64 256 x 128 x 128 33.8
// -> 30.2 ms.  Also tried: tiles of 32 x 4 x 4 and 32 x 2 x 4, 0 to 10% more;
// the second pass as a loop over the pairs with the next direction's loads
// ahead, 883 (112 x 96 x 80 FP32); that in f32x2 arithmetic, two cells per
// thread, 693, but with other roundings.
// ---------------------------------------------------------------------------
template <int LAT, class S, class C, int BX, int BY, int BZ, int MINB>
__global__ void __launch_bounds__(BX* BY* BZ, MINB) k_step_fd_tile(const S* __restrict__ src, S* __restrict__ dst,
                                                                    const Args<C> a, C lamr) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const int x = blockIdx.x * BX + threadIdx.x, y = blockIdx.y * BY + threadIdx.y;
  wait_for_previous_kernel();
  const int z = (L::D == 3) ? blockIdx.z * BZ + threadIdx.z : 0;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  if (x >= nx || y >= ny || z >= nz) return;
  const unsigned row = (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)z);
  const unsigned cell = (unsigned)x + row;
  // element index of the cell at p + k, k = -2, -1, 1, 2 along each axis, after the boundary rule
  unsigned at[3][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = j < 2 ? j - 2 : j - 1;
    at[0][j] = row + (unsigned)pull_coord(x, -k, nx, a.bc[0]);
    at[1][j] = (unsigned)x + (unsigned)nx * ((unsigned)pull_coord(y, -k, ny, a.bc[1]) + (unsigned)ny * (unsigned)z);
    at[2][j] = (L::D == 3) ? (unsigned)x + (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)pull_coord(z, -k, nz, a.bc[2])) : 0u;
  }
  const long long ps = a.ps;
  auto plane = [&](int i) {
    if constexpr (IsS16<S>::value) return reinterpret_cast<const unsigned*>(src) + (size_t)i * ps;
    else return src + (size_t)i * ps;
  };
  auto split = [&](auto v, C& g, C& h) {
    float lo, hi;
    unpack16<S>(v, lo, hi);
    g = static_cast<C>(lo);
    h = static_cast<C>(hi);
  };
  auto near = [&](int i, unsigned e, C& g, C& h) {
    if constexpr (IsS16<S>::value) {
      split(__ldg(plane(i) + e), g, h);
    } else {
      g = __ldg(plane(i) + e);
      h = __ldg(plane(Q + i) + e);
    }
  };
  C drho, u[3], dT;
  {
    C g, h;
    moments_cell<LAT, S, C>(
        [&](auto I) { near(decltype(I)::value, cell, g, h); return g; },
        [&](auto I) { near(decltype(I)::value, cell, g, h); return h; }, a, drho, u, dT);
  }
  if (!(isfinite(drho) && isfinite(dT))) atomicOr(a.flag, 1u);
  C g, h;  // the direction's own values
  auto own = [&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (IsS16<S>::value) {
      split(ld_again(plane(i) + cell), g, h);
    } else {
      g = ld_again(plane(i) + cell);
      h = ld_again(plane(Q + i) + cell);
    }
    return g;
  };
  auto conv = [&](auto I) {
    constexpr int i = decltype(I)::value;
    C cg = C(0), ch = C(0);
    auto axis = [&](int ax, int c) {
      if (c == 0) return;
      C gm2, hm2, gm1, hm1, gp1, hp1;  // the upwind-2, upwind-1 and downwind-1 values
      near(i, at[ax][c > 0 ? 0 : 3], gm2, hm2);
      near(i, at[ax][c > 0 ? 1 : 2], gm1, hm1);
      near(i, at[ax][c > 0 ? 2 : 1], gp1, hp1);
      const C sg = c > 0 ? C(1) : C(-1);
      const C dg = sg * (gm2 - C(6) * gm1 + C(3) * g + C(2) * gp1) * C(1.0 / 6.0);
      const C dh = sg * (hm2 - C(6) * hm1 + C(3) * h + C(2) * hp1) * C(1.0 / 6.0);
      cg = fma(C(c), dg, cg);
      ch = fma(C(c), dh, ch);
    };
    axis(0, L::cx(i));
    axis(1, L::cy(i));
    axis(2, L::cz(i));
    return ConvGH<C>{lamr * cg, lamr * ch};
  };
  relax_store<LAT, S, C, false, true>(own, [&](auto) { return h; }, conv, a, drho, u, dT, dst, ps, cell);
}

// ---------------------------------------------------------------------------
// batched step of a pool of independent instances (continuous batching)
//
// Every resident instance has a slot descriptor in device memory (its
// constants, its two buffers, which buffer is current and how many steps it
// still has to take) and contributes tiles of BX cells along a row to one
// flat tile list.  A persistent grid walks the list; tiles of instances with
// no steps left are skipped.  Each cell runs exactly the arithmetic of the
// single-instance kernel, so an instance's result does not depend on what
// else is resident.  k_pool_advance then decrements the step counters and
// flips the buffers (and stops an instance whose error word is set); a
// bundle of steps is a CUDA graph of these two kernels.
// ---------------------------------------------------------------------------
template <class C>
struct PoolSlot {
  Args<C> a;
  void* buf[2];
  int cur;         // buffer holding the current state
  int steps_left;  // steps still to take
};

template <int LAT, class S, class C, int STAGE, int BX, int MINB>
__global__ void __launch_bounds__(BX, MINB) k_pool_step(const PoolSlot<C>* __restrict__ slots,
                                                  const int4* __restrict__ tiles, const int* __restrict__ n_tiles) {
  wait_for_previous_kernel();
  const int nt = *n_tiles;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const int4 tl = tiles[t];  // slot, x0, y, z
    const PoolSlot<C>& sl = slots[tl.x];
    if (sl.steps_left <= 0) continue;
    const int c = sl.cur;
    step_cell<LAT, S, C, STAGE, BX>(static_cast<const S*>(sl.buf[c]), static_cast<S*>(sl.buf[c ^ 1]), sl.a,
                                    tl.y + (int)threadIdx.x, tl.z, tl.w);
  }
}

template <class C>
__global__ void k_pool_advance(PoolSlot<C>* __restrict__ slots, int nslots) {
  wait_for_previous_kernel();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nslots && slots[i].steps_left > 0) {
    if (*slots[i].a.flag) {
      slots[i].steps_left = 0;  // a non-finite instance takes no further steps
    } else {
      slots[i].steps_left -= 1;
      slots[i].cur ^= 1;
    }
  }
}

// ---------------------------------------------------------------------------
// init: g = F(rho, u, T), h = (delta/2) T F from FP64 device fields, stored
// as deviations from the reference equilibrium.  Arithmetic in the compute
// type C of the instance (FP64 only for FP64 instances); the differences
// rho - rho0 and T - T0 are taken in FP64 before rounding to C.
// ---------------------------------------------------------------------------
template <int LAT, class S, class C>
__global__ void k_init(S* __restrict__ dst, const double* __restrict__ rho, const double* __restrict__ u,
                       const double* __restrict__ T, long long N, const Args<C> a, double rho0, double T0) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= N) return;
  const C drho = static_cast<C>(rho[cell] - rho0), dT = static_cast<C>(T[cell] - T0);
  const C uu[3] = {static_cast<C>(u[cell]), static_cast<C>(u[N + cell]),
                   L::D == 3 ? static_cast<C>(u[2 * N + cell]) : C(0)};
  const long long ps = a.ps;
  equilibrium_dev<LAT, C>(drho, uu, dT, a, [&](auto I, C dF, C dFh) {
    constexpr int i = decltype(I)::value;
    if constexpr (IsS16<S>::value)
      st_gh<Q, S, C>(dst, i, ps, cell, dF * a.inv_gref[L::grp(i)], dFh * a.inv_hscale[L::grp(i)]);
    else
      st_gh<Q, S, C>(dst, i, ps, cell, dF, dFh);
  });
}

// ---------------------------------------------------------------------------
// moments of the stored state (rho, u, T out in FP64), arithmetic in the
// compute type C; rho0 + drho and T0 + dT are formed in FP64
// ---------------------------------------------------------------------------
template <int LAT, class S, class C>
__global__ void k_moments(const S* __restrict__ src, double* __restrict__ rho, double* __restrict__ u,
                          double* __restrict__ T, long long N, const Args<C> a, double rho0, double T0) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= N) return;
  const long long ps = a.ps;
  C g[Q], h[Q];
  static_for<Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    ld_gh<Q, S, C>(src, i, ps, cell, g[i], h[i]);
  });
  C drho, uu[3], dT;
  moments_raw<LAT, C, IsS16<S>::value>([&](auto I) { return g[decltype(I)::value]; },
                                       [&](auto I) { return h[decltype(I)::value]; }, a, drho, uu, dT);
  rho[cell] = rho0 + static_cast<double>(drho);
  u[cell] = static_cast<double>(uu[0]);
  u[N + cell] = static_cast<double>(uu[1]);
  if (L::D == 3) u[2 * N + cell] = static_cast<double>(uu[2]);
  T[cell] = T0 + static_cast<double>(dT);
}

// ---------------------------------------------------------------------------
// FP64 conservation sums of the deviations: per-block partials, then one
// fixed-order final pass; the host adds the reference totals N rho0 (mass)
// and N rho0 (D + delta) T0 / 2 (energy)
//
// The totals are bound by the FP64 pipe (2 instructions per SM and clock)
// long before HBM: a term-by-term FP64 sum takes about 5 FP64 instructions
// per direction (185 per D2Q37 cell, plus a conversion per value), and HBM
// delivers a cell's FP32 values every 26.  So FP32 and 16-bit storage sum on
// the FP32 pipe first: every accumulator is an unevaluated sum hi + lo, each
// addition to hi keeps its rounding error (Knuth's two-sum) and adds it to
// lo.  An addition to lo rounds too, by up to 2^-24 of lo, so over n terms
// the sum could be off by some n^2 2^-49 of its largest partial sum -- unless
// lo is exact.  It is where the terms are of like size: every error is a
// multiple of the last place of the smallest term and lo stays below 2^24 of
// those while n max|x| < 2^24 min|x| or so.  Hence the order of the sums: the
// directions of one velocity group, whose weights are equal, over up to
// kTotalsRun cells of a thread, with accumulators for g, h and, per axis, each
// |c_a|; then they are added up in FP64 with the factors c, |c|^2 (34 sums
// for D2Q37, 53 for D3Q107, 4 FP64 instructions each).  Sums of h over all groups in one
// accumulator were off by up to 1e-12 on uniform fields, where every thread
// makes the same error; these are within 2e-15 there and on random fields
// (tests/test_gpu_totals_exact.py), as term-by-term FP64 sums are.  A run
// with a sum that is not finite (values that are infinite or NaN, or too
// large to sum in FP32) is summed again term by term in FP64.  FP64 storage
// sums its pairs and groups in FP64.
//   Measured, k_conserve_partial alone, one accumulator for h -> these: D2Q37
// FP32 2048^2 247 -> 211 us, FP16 storage 186 -> 182, D3Q107 FP32 128 x 128 x
// 127 353 -> 377, FP16 storage 379 -> 336; D2Q37 FP32 300^2 20.6 -> 24.1 (four
// cells per thread carry all 34 FP64 additions).  Without the next group's
// first loads issued before the present group's FP64 additions 261, 218, 398,
// 370 us; runs of 16 cells 232, 199, 378, 341.  lbm_conserved_noalloc, 16
// cells per thread, the whole call: 296 -> 246, 200 -> 221, 397 -> 370, 503 ->
// 345.
// ---------------------------------------------------------------------------
constexpr int kRedMaxBlocks = 1024;  // partials an instance has room for
constexpr int kRedVals = 5;  // mass, momentum[3], energy
constexpr int kTotalsRun = 32;
template <class S>
constexpr int totals_load() { return sizeof(S) == 8 ? 1 : 4; }  // cells per load

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// hi + lo += x, the error of the addition to hi kept in lo
__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
  hi = s;
}
__device__ __forceinline__ void two_sum(f32x2& hi, f32x2& lo, f32x2 x) {
  const f32x2 s = add_f32x2(hi, x), b = sub_f32x2(s, hi);
  lo = add_f32x2(lo, add_f32x2(sub_f32x2(hi, sub_f32x2(s, b)), sub_f32x2(x, b)));
  hi = s;
}

// a velocity group in the totals: its directions [first, first + count), and
// the values that |c_a| takes in it (one or two besides 0)
template <int LAT, int GRP>
struct TotalsGroup {
  using L = Lat<LAT>;
  static constexpr int g = GRP;
  static constexpr int c2 = (LAT == 0 ? kD2Q37 : kD3Q107).c2[GRP];
  static constexpr int count = (LAT == 0 ? kD2Q37 : kD3Q107).members[GRP];
  static constexpr int begin() {
    int i = 0;
    while (L::grp(i) != GRP) ++i;
    return i;
  }
  static constexpr int first = begin();
  __host__ __device__ static constexpr int value(int k) {  // the (k + 1)-th of them in order of size, or 0
    for (int v = 1; v <= 3; ++v)
      for (int a = 0; a < L::D; ++a)
        if ((LAT == 0 ? kD2Q37 : kD3Q107).rep[GRP][a] == v) {
          if (k-- == 0) return v;
          break;
        }
    return 0;
  }
  static constexpr int batch = count % 4 == 0 ? 4 : (count % 3 == 0 ? 3 : 1);  // directions per batch of loads
  static constexpr int speeds = value(1) != 0 ? 2 : 1;
  __host__ __device__ static constexpr int speed(int v) { return v == value(0) ? 0 : 1; }
};

// the totals of the cells begin, begin + stride, ... below end, every term
// added in FP64
template <int LAT, class S>
__device__ __noinline__ void add_totals_by_term(const S* __restrict__ src, long long ps, long long begin,
                                                long long end, long long stride, double r, double half_r2,
                                                const Args<float>& af, double (&acc)[kRedVals]) {
  using L = Lat<LAT>;
  for (long long cell = begin; cell < end; cell += stride) {
    static_for<L::Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      float gf, hf;
      ld_gh<L::Q, S, float>(src, i, ps, cell, gf, hf);
      scale_gh<S, float>(gf, hf, L::grp(i), af);
      const double g = gf;
      acc[0] += g;
      if constexpr (L::cx(i) != 0) acc[1] += (r * L::cx(i)) * g;
      if constexpr (L::cy(i) != 0) acc[2] += (r * L::cy(i)) * g;
      if constexpr (L::cz(i) != 0) acc[3] += (r * L::cz(i)) * g;
      acc[4] += half_r2 * L::c2(i) * g + double(hf);
    });
  }
}

// adds the deviations' totals of the VEC cells from begin, from begin +
// stride, ... below end: acc = {mass, momentum[3], energy}.  VEC = 4 (FP32
// and 16-bit storage) reads 16 bytes at a time: src, ps, begin and stride
// are multiples of four elements, and so is end.
template <int LAT, class S, int VEC>
__device__ __forceinline__ void add_totals(const S* __restrict__ src, long long ps, long long begin, long long end,
                                           long long stride, double r, double half_r2, const Args<float>& af,
                                           double (&acc)[kRedVals]) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q, G = L::G, D = L::D;
  if constexpr (sizeof(S) == 8) {
    for (long long cell = begin; cell < end; cell += stride) {
      double g0, h0;
      ld_gh<Q, S, double>(src, 0, ps, cell, g0, h0);
      double mass = g0, hs = h0, k2 = 0.0, grp = 0.0, j[3] = {0.0, 0.0, 0.0};
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (i % 2 == 1) {  // the pair c, -c
          double gp, hp, gm, hm;
          ld_gh<Q, S, double>(src, i, ps, cell, gp, hp);
          ld_gh<Q, S, double>(src, i + 1, ps, cell, gm, hm);
          const double d = gp - gm;
          if constexpr (L::cx(i) != 0) j[0] = fma(double(L::cx(i)), d, j[0]);
          if constexpr (L::cy(i) != 0) j[1] = fma(double(L::cy(i)), d, j[1]);
          if constexpr (L::cz(i) != 0) j[2] = fma(double(L::cz(i)), d, j[2]);
          hs += hp + hm;
          grp += gp + gm;
          if constexpr (i + 2 >= Q || L::grp(i + 2 < Q ? i + 2 : i) != L::grp(i)) {  // the group's last pair
            mass += grp;
            k2 = fma(double(L::c2(i)), grp, k2);
            grp = 0.0;
          }
        }
      });
      acc[0] += mass;
#pragma unroll
      for (int a = 0; a < D; ++a) acc[1 + a] = fma(r, j[a], acc[1 + a]);
      acc[4] += fma(half_r2, k2, hs);
    }
  } else {
    // V cells per load (16 bytes per thread and load keep enough of them in
    // flight); the cells' values are summed in the two halves of f32x2
    constexpr int V = VEC;
    using W = typename std::conditional<V == 4, uint4, unsigned>::type;
    constexpr int NPL = IsS16<S>::value ? 1 : 2;
    while (begin < end) {
      const long long first = begin;
      begin = min(end, first + (kTotalsRun / V) * stride);
      double part[kRedVals] = {0.0, 0.0, 0.0, 0.0, 0.0};
      bool fine = true;
      // the batch of loads that is issued while the one before is summed, also
      // from one quad of cells and from one group to the next
      W next[4][NPL];
      auto fetch = [&](auto K, auto M, long long cell) {
        using R = TotalsGroup<LAT, decltype(K)::value>;
        static_for<R::batch>([&](auto J) {
          constexpr int i = R::first + decltype(M)::value * R::batch + decltype(J)::value;
#pragma unroll
          for (int q = 0; q < NPL; ++q)
            next[decltype(J)::value][q] = ld_again(reinterpret_cast<const W*>(
                reinterpret_cast<const unsigned*>(src) + ((size_t)(q * Q + i) * ps + cell)));
        });
      };
      fetch(std::integral_constant<int, 0>{}, std::integral_constant<int, 0>{}, first);
      static_for<G>([&](auto K) {
        using R = TotalsGroup<LAT, decltype(K)::value>;
        constexpr int NB = R::count / R::batch;
        f32x2 ghi = 0ull, glo = 0ull, hhi = 0ull, hlo = 0ull, jhi[D][R::speeds], jlo[D][R::speeds];
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int c = 0; c < R::speeds; ++c) jhi[a][c] = jlo[a][c] = 0ull;
        auto add = [&](auto I, f32x2 g, f32x2 h) {
          constexpr int i = decltype(I)::value;
          if constexpr (IsS16<S>::value) {  // the 16-bit codec in FP32, as the step evaluates it
            float a0, a1;
            unpack_f32x2(g, a0, a1);
            g = pack_f32x2(__fmul_rn(a0, af.gref[R::g]), __fmul_rn(a1, af.gref[R::g]));
            unpack_f32x2(h, a0, a1);
            h = pack_f32x2(__fmul_rn(a0, af.hscale[R::g]), __fmul_rn(a1, af.hscale[R::g]));
          }
          two_sum(ghi, glo, g);
          two_sum(hhi, hlo, h);
          auto axis = [&](int a, int c) {
            if (c > 0) two_sum(jhi[a][R::speed(c)], jlo[a][R::speed(c)], g);
            if (c < 0) two_sum(jhi[a][R::speed(-c)], jlo[a][R::speed(-c)], neg_f32x2(g));
          };
          axis(0, L::cx(i));
          axis(1, L::cy(i));
          if constexpr (D == 3) axis(2, L::cz(i));
        };
#pragma unroll 1
        for (long long cell = first; cell < begin; cell += stride) {
          static_for<NB>([&](auto M) {
            constexpr int m = decltype(M)::value;
            W now[R::batch][NPL];
            static_for<R::batch>([&](auto J) {
#pragma unroll
              for (int q = 0; q < NPL; ++q) now[decltype(J)::value][q] = next[decltype(J)::value][q];
            });
            if constexpr (m + 1 < NB) fetch(K, std::integral_constant<int, m + 1>{}, cell);
            else if (cell + stride < begin) fetch(K, std::integral_constant<int, 0>{}, cell + stride);
            else if constexpr (R::g + 1 < G)
              fetch(std::integral_constant<int, R::g + 1>{}, std::integral_constant<int, 0>{}, first);
            static_for<R::batch>([&](auto J) {
              constexpr int i = R::first + m * R::batch + decltype(J)::value;
              const W(&w)[NPL] = now[decltype(J)::value];
              auto two = [&](unsigned g0, unsigned g1, unsigned h0, unsigned h1) {
                if constexpr (IsS16<S>::value) {
                  float ga, ha, gb, hb;
                  unpack16<S>(g0, ga, ha);
                  unpack16<S>(g1, gb, hb);
                  add(std::integral_constant<int, i>{}, pack_f32x2(ga, gb), pack_f32x2(ha, hb));
                } else {
                  add(std::integral_constant<int, i>{}, pack_f32x2(__uint_as_float(g0), __uint_as_float(g1)),
                      pack_f32x2(__uint_as_float(h0), __uint_as_float(h1)));
                }
              };
              if constexpr (V == 4) {
                two(w[0].x, w[0].y, w[NPL - 1].x, w[NPL - 1].y);
                two(w[0].z, w[0].w, w[NPL - 1].z, w[NPL - 1].w);
              } else {
                two(w[0], 0u, w[NPL - 1], 0u);
              }
            });
          });
        }
        auto total = [&](f32x2 h2, f32x2 l2) {
          float hi, x, lo, y;
          unpack_f32x2(h2, hi, x);
          unpack_f32x2(l2, lo, y);
          two_sum(hi, lo, x);
          lo = __fadd_rn(lo, y);
          fine = fine && isfinite(hi) && isfinite(lo);
          return double(hi) + double(lo);
        };
        const double m = total(ghi, glo);
        part[0] += m;
        part[4] += fma(half_r2 * R::c2, m, total(hhi, hlo));
        static_for<D * R::speeds>([&](auto J) {
          constexpr int a = decltype(J)::value / R::speeds, c = decltype(J)::value % R::speeds;
          if constexpr (R::c2 != 0) part[1 + a] = fma(r * R::value(c), total(jhi[a][c], jlo[a][c]), part[1 + a]);
        });
      });
      if (!fine) {
#pragma unroll
        for (int k = 0; k < kRedVals; ++k) part[k] = 0.0;
        for (int v = 0; v < V; ++v)
          add_totals_by_term<LAT, S>(src, ps, first + v, begin, stride, r, half_r2, af, part);
      }
#pragma unroll
      for (int k = 0; k < kRedVals; ++k) acc[k] += part[k];
    }
  }
}

// the block's sum of acc, in warp order, into partial[blockIdx.x]
template <int THREADS>
__device__ __forceinline__ void store_block_totals(const double (&acc)[kRedVals], double* __restrict__ partial) {
  __shared__ double sh[THREADS / 32][kRedVals];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kRedVals; ++k) {
    const double v = warp_sum(acc[k]);
    if (lane == 0) sh[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kRedVals) {
    double s = 0.0;
    for (int w = 0; w < THREADS / 32; ++w) s += sh[w][threadIdx.x];
    partial[blockIdx.x * kRedVals + threadIdx.x] = s;
  }
}

template <int LAT, class S, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) k_conserve_partial(const S* __restrict__ src, long long N,
                                                                             const Args<double> a, const Args<float> af,
                                                                             double* __restrict__ partial) {
  double acc[kRedVals] = {0.0, 0.0, 0.0, 0.0, 0.0};
  // an instance's planes start on 256 bytes, so whole quads of cells can be
  // read at once; the last N mod 4 go to the first threads of the last block
  constexpr int V = totals_load<S>();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
  const long long whole = N / V * V;
  add_totals<LAT, S, V>(src, a.ps, t * V, whole, nt * V, a.r, a.half_r2, af, acc);
  if constexpr (V > 1) {
    if (blockIdx.x == gridDim.x - 1)
      add_totals<LAT, S, 1>(src, a.ps, whole + threadIdx.x, N, THREADS, a.r, a.half_r2, af, acc);
  }
  store_block_totals<THREADS>(acc, partial);
}


}  // namespace lbm
