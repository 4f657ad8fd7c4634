// ader_fixr.cuh -- the Rusanov flux of the interface kernels in the fixed-point
// arithmetic of ader_fix.h.
//
// What bounds it.  A Rusanov flux is ~40 FP64 operations (1D; 2D 55, 3D 70), 64 issue
// cycles of a scheduler each; the same in fixed point is ~340 integer and float
// instructions without any FP64 one.  Interface kernels, FP64 flux -> this one: 1D
// N = 5, 1e5 cells 63 -> 46 us, N = 7, 1e6 cells 577 -> 307, 2D N = 5, 160^2 141 -> 80,
// 3D N = 3, 48^3 2.5 -> 0.82 ms (1 to 3 % of it the bounds below and what they need: 1D N = 5
// in the present tiles 40.1 -> 41.4 us, N = 7 267 -> 272).
//
// Units: powers of two above the two states' largest rho, E and |m| (see ader_fix.cuh);
// fluxes at frac 57, off by 2^-56 of the units (FP64: 2^-53 of every operand).  The
// wave speed enters only as s (b - a): the FP32 speed where its error is well below FP64's
// rounding of the flux, else c = sqrt(gamma p / rho) refined by two Newton steps in integers,
// where that is enough.  Both errors are bounded from the state: p is a small part of the
// unit of E at high Mach number, where an absolute error of p counts 1 / c times.
// Everything else -- rho below 1/8 of the unit, p below 2^-25 of it or rho not positive, jumps
// beyond 2^-8 of the fluxes, units far from one, and what lies too far below its unit for
// frac 57: gamma below 9/8 (make_fx_gas), speeds below 3/16 of the unit, which only a fast
// flow along the face has -- is left to the FP64 form.
//
// Largest error of the 1D flux against quadruple precision in units of rho s, sqrt(rho E) s, E s
// (gamma = 1.4, jumps 1e-14 to 1e-2, tests/host_src/fixed_check.cpp), this form and FP64:
// Mach 1e-7 1.7 and 4.2e-16, Mach 1 2.0 and 4.9, Mach 10 3.3 and 9.1, Mach 100 3.8 and 10,
// Mach 1000 3.6 and 11.
#pragma once

#include "ader_fix.h"
#include "ader_ops.h"

namespace ader {

// x (|x| < 2^e) at frac 61 in units of 2^e, truncated
ADER_HD fxi fx_from_double(double x, int e) {
  const int hi = fx_dhi(x);
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = ex ? ((unsigned)hi & 0xfffffu) | 0x100000u : 0u;
  const unsigned ml = ex ? (unsigned)fx_dlo(x) : 0u;
  const unsigned long long m = (unsigned long long)fx_join(fx_funnel_l(ml, mh, 8), ml << 8);
  const int k = min(e + 1022 - ex, 63);
  const fxi v = (fxi)(m >> k);
  return hi < 0 ? -v : v;
}

// x in [0, 1] at frac 60, truncated
ADER_HD fxi fx_from_float(float x) {
  const unsigned b = fx_fbits(x);
  const int ex = (int)(b >> 23);
  const fxi m = ex ? (fxi)((b & 0x7fffffu) | 0x800000u) : 0;
  return ex >= 90 ? m << (ex - 90) : m >> min(90 - ex, 63);
}

// 2^k as a float (|k| < 126)
ADER_HD float fx_pow2f(int k) {
#ifdef __CUDA_ARCH__
  return __int_as_float((127 + k) << 23);
#else
  return ldexpf(1.0f, k);
#endif
}

// X 2^k rounded to nearest, on the integer pipe (|k| < 500)
ADER_HD double fx_to_double_int(fxi x, int k) {
  const unsigned long long a = (unsigned long long)(x < 0 ? -x : x);
  const int lz = fx_clz(a);
  if (lz > 62) return a ? (x < 0 ? -1.0 : 1.0) * fx_double((1023 + k) << 20, 0) : 0.0;
  const unsigned long long m = (((a << lz) >> 10) + 1) >> 1;  // 2^52 <= m <= 2^53
  const unsigned long long b =
      ((unsigned long long)(unsigned)(1022 + 63 - lz + k) << 52) + m;
  return fx_double((int)((b >> 32) | (x < 0 ? 0x80000000u : 0u)), (int)b);
}

// One side's flux in direction DIR at frac 57, its normal velocity (limbs, frac 60), p
// (frac 57) and 1 / rho (frac 28); as fx_fluxes.
template <int D, int DIR>
ADER_HD void fx_flux_dir(const fxi (&q)[D + 2], const FxGas& g, fxi (&F)[D + 2], Fx2& Un, fxi& p,
                         int& r1, unsigned& bad) {
  const Fx2 R = fx_split(q[0]);
  bad |= (unsigned)(R.h - 0x4100000) & 0x80000000u;
  const int r0 = fx_rint(fx_rcpf((float)R.h) * 0x1p57f);
  const int nh = (int)(0u - (unsigned)R.h);
  const fxi e = fx_madw(nh, r0, (fxi)1 << 57);
  const int es = (int)fx_funnel_l((unsigned)fx_lo(e), (unsigned)fx_hi(e), 24);
  r1 = r0 + (fx_hi(fx_madw(r0, es, (fxi)1 << 48)) >> 17);
  Fx2 M[D], U[D];
  unsigned m4[D];
  fxi W = q[D + 1] + q[D + 1], P[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const fxi m = q[1 + d];
    M[d] = fx_split(m);
    const fxi pu = fx_madw(M[d].h, r1, (fxi)1 << 28);
    bad |= ((unsigned)fx_hi(pu) + (1u << 26)) & 0xf8000000u;
    const int u0 = (int)fx_funnel_l((unsigned)fx_lo(pu), (unsigned)fx_hi(pu), 3);
    const fxi mr = m + 8;  // m to frac 57, rounded
    m4[d] = fx_funnel_l((unsigned)fx_lo(mr), (unsigned)fx_hi(mr), 28);
    if (d == DIR) F[0] = fx_join((unsigned)(fx_hi(mr) >> 4), m4[d]);
    const int rem = (int)(m4[d] + (unsigned)nh * (unsigned)u0 -
                          (unsigned)fx_hi(fx_madw(R.l, u0, (fxi)1 << 31)));
    const fxi us = fx_madw(rem, r1, (fxi)1 << 24);
    U[d] = fx_split(fx_join((unsigned)(fx_hi(us) >> 25),
                            fx_funnel_l((unsigned)fx_lo(us), (unsigned)fx_hi(us), 7)));
    U[d].h = (int)((unsigned)U[d].h + (unsigned)u0);
    FxAcc a = fx_zero<0>();
    fx_mac(a, M[d].h, M[d].l, U[d]);
    P[d] = fx_fold<0>(a);
    W -= P[d];
  }
  Un = U[DIR];
  const Fx2 Ws = fx_split(W);
  FxAcc a = fx_zero<2>();
  fx_mac(a, g.g2h, g.g2l, Ws);
  p = fx_fold<2>(a);
  const Fx2 H = fx_split(q[D + 1] + p);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    if (d == DIR) {
      F[1 + d] = P[d] + p;
    } else {
      a = fx_zero<0>();
      fx_mac(a, M[d].h, M[d].l, Un);
      F[1 + d] = fx_fold<0>(a);
    }
  }
  a = fx_zero<4>();
  fx_mac(a, H.h, H.l, Un);
  a.m += fx_hi(fx_madw(H.l, Un.l, (fxi)1 << 31));  // up to 2^-55: gas at rest shows it
  F[D + 1] = fx_fold<4>(a);
}

// c = sqrt(gamma p / rho) at frac 57 from its float value c0 (cell units): X = gamma p / rho
// as u in fx_fluxes, then c + (X - c^2) / (2 c) twice, the first time rounded to frac 28.
// The second correction is then at most 2^-29 (as a float good to 2^-50) and leaves its square
// over 2 c, 2^-59 / c.  X is within 2^-53 (p within 2^-56; 1 / rho is below 2.1 where the two
// sides of a face are as close as the caller asks), which makes 2^-54 / c.
ADER_HD fxi fx_sound_speed(fxi rho, fxi p57, int r1, float c0, const FxGas& g, unsigned& bad) {
  const Fx2 R = fx_split(rho);
  const fxi p = (fxi)((unsigned long long)p57 << 4);  // frac 61 (p < gamma - 1 <= 1)
  const int nh = (int)(0u - (unsigned)R.h);
  const fxi pu = fx_madw(fx_split(p).h, r1, (fxi)1 << 28);
  bad |= ((unsigned)fx_hi(pu) + (1u << 26)) & 0xf8000000u;  // p / rho < 2
  const int u0 = (int)fx_funnel_l((unsigned)fx_lo(pu), (unsigned)fx_hi(pu), 3);
  const int rem = (int)((unsigned)fx_lo(p57) + (unsigned)nh * (unsigned)u0 -
                        (unsigned)fx_hi(fx_madw(R.l, u0, (fxi)1 << 31)));
  const fxi us = fx_madw(rem, r1, (fxi)1 << 24);
  Fx2 Y = fx_split(us >> 25);
  Y.h = (int)((unsigned)Y.h + (unsigned)u0);  // p / rho at frac 60
  FxAcc a = fx_zero<1>();
  fx_mac(a, g.gh, g.gl, Y);
  const fxi X = fx_fold<1>(a);  // frac 57
  int ci = fx_rint(c0 * 0x1p28f);
  const float half = fx_rcpf(c0) * 0.5f;
  ci += fx_rint((float)(int)((X - 2 * ((fxi)ci * ci)) >> 8) * half * 0x1p-21f);
  const fxi d = X - 2 * ((fxi)ci * ci);  // below 2^30 (c < 2)
  return ((fxi)ci << 29) + fx_rint((float)(int)d * half);
}

// Twice the Rusanov flux between a (low side) and b in direction DIR.  False: not taken
// (G2 unset).  speed, where asked for: s (always the refined one: a further variable's jump
// has nothing to do with the Euler ones), the two normal velocities and the bound on the
// relative error of s, for further variables' fluxes.
template <int D, int DIR>
ADER_HD bool fx_rusanov2(const double* a, const double* b, double* G2, const FxGas& g,
                         double* speed = nullptr) {
  constexpr int M = D + 2;
  if (!g.ok) return false;
  auto field = [](double x) { return (fx_dhi(x) >> 20) & 0x7ff; };
  const int er = max(field(a[0]), field(b[0])), ee = max(field(a[M - 1]), field(b[M - 1]));
  int em = 0;
#pragma unroll
  for (int d = 0; d < D; ++d) em = max(em, max(field(a[1 + d]), field(b[1 + d])));
  const int ea = er - 1022, ec = max((ee - 1022 - ea + 1) >> 1, em - 1022 - ea);
  if (max(er, max(em, ee)) >= 1023 + 60 || abs(ea) > 30 || abs(ec) > 30) return false;
  fxi qa[M], qb[M], Fa[M], Fb[M], pa, pb;
  Fx2 Ua, Ub;
  int ra, rb;
  unsigned bad = 0u;
#pragma unroll
  for (int r = 0; r < M; ++r) {
    const int e = r == 0 ? ea : r < M - 1 ? ea + ec : ea + 2 * ec;
    qa[r] = fx_from_double(a[r], e);
    qb[r] = fx_from_double(b[r], e);
    if (r == M - 1) {
      qa[r] = (qa[r] + 8) >> 4;
      qb[r] = (qb[r] + 8) >> 4;
    }
  }
  fx_flux_dir<D, DIR>(qa, g, Fa, Ua, pa, ra, bad);
  fx_flux_dir<D, DIR>(qb, g, Fb, Ub, pb, rb, bad);
  if (bad || fx_hi(pa) <= 0 || fx_hi(pb) <= 0) return false;
  // FP32 speeds in the units' velocity
  const float fua = fabsf((float)Ua.h) * 0x1p-28f, fub = fabsf((float)Ub.h) * 0x1p-28f;
  auto pressure = [](fxi p) {  // both words: at Mach 100 the high one holds 12 bits
    return fmaf((float)fx_hi(p), 0x1p-25f, (float)(unsigned)fx_lo(p) * 0x1p-57f);
  };
  const float ca = sqrtf(g.gammaf * pressure(pa) * ((float)ra * 0x1p-28f));
  const float cb = sqrtf(g.gammaf * pressure(pb) * ((float)rb * 0x1p-28f));
  const float sf = fmaxf(fua + ca, fub + cb);
  if (!(sf >= 0.1875f)) return false;
  fxi d[M], S[M];
  float jf = 0.0f, ff = 0.0f;
#pragma unroll
  for (int r = 0; r < M; ++r) {
    d[r] = qb[r] - qa[r];
    S[r] = Fa[r] + Fb[r];
    const float j = fabsf(fmaf((float)fx_hi(d[r]), 0x1p32f, (float)(unsigned)fx_lo(d[r])));
    jf = fmaxf(jf, r < M - 1 ? j : 16.0f * j);
    ff = fmaxf(ff, fabsf((float)fx_hi(S[r])));
  }
  jf *= 0x1p-61f;
  ff *= 0x1p-25f;
  fxi sd[M];
  double s_out = 0.0;
  // the FP32 speed: c and the sum are within 2^-21 relative, u and si at their last bits
  float s_err = fmaf(0x1p-21f, sf, 0x1p-27f);
  if (!speed && s_err * jf <= 0x1p-54f * ff) {
    if (!(sf < 15.0f)) return false;
    const int si = fx_rint(sf * 0x1p27f);
#pragma unroll
    for (int r = 0; r < M; ++r) {
      const Fx2 x = fx_split(d[r]);
      const FxAcc t{fx_madw(si, x.h, 0), fx_madw(si, x.l, (fxi)1 << (r < M - 1 ? 30 : 26)), 0};
      sd[r] = r < M - 1 ? fx_fold<1>(t) : fx_fold<5>(t);
    }
  } else {
    // the refined one (fx_sound_speed): its error times the jump below FP64's rounding of the
    // flux, and the jump below 2^-8 of it
    s_err = fmaf(0x1p-53f, fx_rcpf(fminf(ca, cb)), 0x1p-49f * sf);
    if (!(fmaf(0x1p-45f, sf, s_err) * jf <= 1e-16f * ff) || !(sf < 7.0f)) return false;
    auto magnitude = [](const Fx2& u) {  // |u| at frac 57
      const fxi x = ((fxi)u.h << 32) + u.l;
      return (x < 0 ? -x : x) >> 3;
    };
    const fxi sa = magnitude(Ua) + fx_sound_speed(qa[0], pa, ra, ca, g, bad);
    const fxi sb = magnitude(Ub) + fx_sound_speed(qb[0], pb, rb, cb, g, bad);
    if (bad) return false;
    const fxi sm = sa > sb ? sa : sb;
    const Fx2 s = fx_split(sm);
#pragma unroll
    for (int r = 0; r < M; ++r) {
      FxAcc t = r < M - 1 ? fx_zero<3>() : fx_zero<4>();
      const Fx2 x = fx_split(r < M - 1 ? d[r] : d[r] * 8);
      fx_mac(t, s.h, s.l, x);
      if (r == M - 1) t.m += fx_hi(fx_madw(s.l, x.l, (fxi)1 << 31));
      sd[r] = r < M - 1 ? fx_fold<3>(t) : fx_fold<4>(t);
    }
    if (speed) s_out = fx_to_double_int(sm, ec - 57);
  }
#pragma unroll
  for (int r = 0; r < M; ++r) {
    const int e = ec + (r == 0 ? ea : r < M - 1 ? ea + ec : ea + 2 * ec);
    G2[r] = fx_to_double_int(S[r] - sd[r], e - 57);
  }
  if (speed) {
    speed[0] = s_out;
    speed[1] = fx_to_double_int(((fxi)Ua.h << 32) + Ua.l, ec - 60);
    speed[2] = fx_to_double_int(((fxi)Ub.h << 32) + Ub.l, ec - 60);
    speed[3] = (double)(s_err * fx_rcpf(sf) * 1.0001f);
  }
  return true;
}

}  // namespace ader
