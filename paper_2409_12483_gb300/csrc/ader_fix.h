// ader_fix.h -- 60-bit fixed-point arithmetic on 32-bit integer multipliers, the
// number form of the FP64 predictor's inner loop (ader_fix.cuh).
//
// GB300 issues 2 FP64 lanes per SM and clock against 32 lanes of 32 x 32 + 64-bit
// integer multiply-add (mad.wide, measured on data that varies), so a product of two
// two-limb integers (3 mad.wide) costs a fifth of one DFMA.  Inside one cell the
// scheme's contractions mix all nodes, so the rounding of a result is set by the
// largest value of the cell: a common exponent per cell and variable loses
// nothing against a floating-point significand, and 57 fraction bits below that
// exponent are more than the 53 of FP64.
//
// Numbers: a 64-bit integer X = x 2^f ("frac f"); limbs (h, l) with X = h 2^32 + l
// and l in [-2^31, 2^31), so that every partial product is a signed 32 x 32 one.
// A contraction sum_j c_j x_j keeps two 64-bit sums, hh = sum h h and
// m = sum (h l + l h); the l l terms (below 2^-2 of the last bit kept, of either
// sign) are left out.  The value of the sum is hh + m 2^-32 in units of 2^64.
// All functions also compile for the host (tests/host_src/fixed_check.cpp measures them there).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>

#ifdef __CUDACC__
#define ADER_HD __host__ __device__ __forceinline__
#else
#define ADER_HD inline
#endif

namespace ader {

#ifndef __CUDACC__
using std::abs;
using std::max;
using std::min;
#endif

typedef long long fxi;

struct Fx2 {
  int h, l;
};

// The device forms are PTX: written in C++, (fxi)(int)(x >> 32) becomes an arithmetic
// 64-bit shift and the product that uses it a 64 x 64-bit one (a flux took 135
// instructions instead of 75).
ADER_HD int fx_hi(fxi x) {
#ifdef __CUDA_ARCH__
  int h, l;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(x));
  return h;
#else
  return (int)(x >> 32);
#endif
}
ADER_HD int fx_lo(fxi x) {
#ifdef __CUDA_ARCH__
  int h, l;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(x));
  return l;
#else
  return (int)(uint32_t)(uint64_t)x;
#endif
}
ADER_HD fxi fx_join(unsigned h, unsigned l) {
#ifdef __CUDA_ARCH__
  fxi x;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(l), "r"(h));
  return x;
#else
  return (fxi)(((uint64_t)h << 32) | l);
#endif
}

// words of a double, floats and their bits, the float reciprocal within one unit in the
// last place (any x that is not far from one), leading zeros
ADER_HD int fx_dhi(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (int)(uint32_t)(b >> 32);
#endif
}
ADER_HD int fx_dlo(double x) {
#ifdef __CUDA_ARCH__
  return __double2loint(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (int)(uint32_t)b;
#endif
}
ADER_HD double fx_double(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const uint64_t b = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
ADER_HD unsigned fx_fbits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
ADER_HD int fx_rint(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return x >= 0x1p31f ? 0x7fffffff : x > -0x1p31f ? (int)lrintf(x) : (int)0x80000000u;
#endif
}
ADER_HD float fx_rcpf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
ADER_HD int fx_clz(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

ADER_HD Fx2 fx_split(fxi x) { return Fx2{fx_hi(x + 0x80000000LL), fx_lo(x)}; }

ADER_HD fxi fx_madw(int a, int b, fxi c) { return (fxi)a * (fxi)b + c; }
// (x << k) and (x >> k) of the 96-bit number x:lo, the words that stay
ADER_HD unsigned fx_funnel_l(unsigned lo, unsigned hi, int k) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, k);
#else
  return (k & 31) ? (hi << (k & 31)) | (lo >> (32 - (k & 31))) : hi;
#endif
}

// Sums of a contraction; SH: the left shift of its fold (rounds to nearest).  m is kept
// in two parts, so that no chain of multiply-adds is longer than the sum.
struct FxAcc {
  fxi hh, m, m2;
};
template <int SH>
ADER_HD FxAcc fx_zero() {
  return FxAcc{0, (fxi)1 << (31 - SH), 0};
}
ADER_HD void fx_mac(FxAcc& s, int ch, int cl, const Fx2& x) {
  s.hh = fx_madw(ch, x.h, s.hh);
  s.m = fx_madw(ch, x.l, s.m);
  s.m2 = fx_madw(cl, x.h, s.m2);
}
// (hh + m 2^-32) 2^SH
template <int SH>
ADER_HD fxi fx_fold(const FxAcc& s) {
  const fxi m = s.m + s.m2;
  const fxi t = s.hh + (fxi)fx_hi(m);
  if constexpr (SH == 0) {
    return t;
  } else {
    const unsigned w = (unsigned)fx_lo(t);
    return fx_join(fx_funnel_l(w, (unsigned)fx_hi(t), SH),
                   fx_funnel_l((unsigned)fx_lo(m), w, SH));
  }
}
// the same with a run-time shift in [0, 31]; the rounding (1 << 31 - sh) is the
// caller's initial m; top: the high word before the shift
ADER_HD fxi fx_fold_var(const FxAcc& s, int sh, int* top = nullptr) {
  const fxi m = s.m + s.m2;
  const fxi t = s.hh + (fxi)fx_hi(m);
  const unsigned w = (unsigned)fx_lo(t);
  if (top) *top = fx_hi(t);
  return fx_join(fx_funnel_l(w, (unsigned)fx_hi(t), sh),
                 fx_funnel_l((unsigned)fx_lo(m), w, sh));
}

// |x| as a float, within 2^-23 of itself: the low word with its sign, the high one with the
// carry of that (with an unsigned low word a small negative x was up to 128 last places off,
// a change of -5 read as 0).  One conversion of 64 bits in place of the two took 1 to 4 % of
// a step.
ADER_HD float fx_abs_float(fxi x) {
  const int l = fx_lo(x), h = fx_hi(x) + (int)((unsigned)l >> 31);
  return fabsf(fmaf((float)h, 0x1p32f, (float)l));
}

// A convergence test in floats lets an iteration end only where the same test on the
// numbers themselves would: the changes, the iterate's maximum (its high word), the
// tolerance and their product are each within 2^-23
constexpr float kFxTol = 1.0f - 0x1p-20f;

// x 2^-s rounded, s in [0, 62] (|x| below 2^61)
ADER_HD fxi fx_shr(fxi x, int s) { return (x + (((fxi)1 << s) >> 1)) >> s; }

// Formats of the predictor, in the cell's units (|q| < 2): rho and m at frac 61, E
// at frac 57; fluxes and everything that enters a contraction below 2^60 (frac 57).
constexpr int kFxF = 57;
constexpr int kFxM = 61;
// log2 bounds of the row sums of |k~|, |psi| (both ends) and |D~ / w|, by degree:
// a table entry is stored at frac 62 - bound, so the high limbs of a row sum to
// less than 2^30 and no 64-bit sum can overflow.
constexpr int kFxSK[8] = {0, 2, 4, 5, 6, 6, 7, 8};
constexpr int kFxSP[8] = {1, 1, 2, 2, 2, 2, 3, 3};
constexpr int kFxSV[8] = {0, 2, 3, 4, 5, 5, 5, 6};

// The Euler fluxes of D directions in fixed point: q = (rho, m_1 .. m_D, E), rho and m
// at frac 61, E at frac 57, all below 2 in magnitude, to F[d] = (m_d, m_j u_d + p
// (j = d), (E + p) u_d) at frac 57.  g2h, g2l: (gamma - 1) / 2 <= 1/2 at frac 62.  `bad`
// collects nonzero bits when rho is not above 1/8, a |u_d| leaves 2 or a flux leaves 8;
// velocity: the u_d as limbs at frac 60.
//   r   = 1 / rho to 2^-28: float reciprocal of the high limb, one Newton step;
//   u   = u0 + (m - rho u0) r, u0 = m r at frac 28: the remainder is below 2^-26 and
//         exact to 2^-57, so 32-bit arithmetic modulo 2^32 gives it at frac 57;
//   the products' l l terms, left out, stay below 2^-56 (rms 2^-57).
template <int D>
ADER_HD void fx_fluxes(const fxi (&q)[D + 2], int g2h, int g2l, fxi (&F)[D][D + 2],
                       unsigned& bad, Fx2* velocity = nullptr) {
  const Fx2 R = fx_split(q[0]);
  bad |= (unsigned)(R.h - 0x4100000) & 0x80000000u;
  const int r0 = fx_rint(fx_rcpf((float)R.h) * 0x1p57f);  // frac 28
  const int nh = (int)(0u - (unsigned)R.h);
  const fxi e = fx_madw(nh, r0, (fxi)1 << 57);
  const int es = (int)fx_funnel_l((unsigned)fx_lo(e), (unsigned)fx_hi(e), 24);  // e >> 8
  const int r1 = r0 + (fx_hi(fx_madw(r0, es, (fxi)1 << 48)) >> 17);
  Fx2 M[D], U[D];
  unsigned m4[D];
  fxi W = q[D + 1] + q[D + 1], P[D][D];
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int d = 0; d < D; ++d) {
    const fxi m = q[1 + d];
    M[d] = fx_split(m);
    const fxi pu = fx_madw(M[d].h, r1, (fxi)1 << 28);  // frac 57
    bad |= ((unsigned)fx_hi(pu) + (1u << 26)) & 0xf8000000u;
    const int u0 = (int)fx_funnel_l((unsigned)fx_lo(pu), (unsigned)fx_hi(pu), 3);  // pu >> 29
    m4[d] = fx_funnel_l((unsigned)fx_lo(m), (unsigned)fx_hi(m), 28);               // m >> 4
    const int rem = (int)(m4[d] + (unsigned)nh * (unsigned)u0 -
                          (unsigned)fx_hi(fx_madw(R.l, u0, (fxi)1 << 31)));
    const fxi us = fx_madw(rem, r1, (fxi)1 << 24);
    U[d] = fx_split(fx_join((unsigned)(fx_hi(us) >> 25),
                            fx_funnel_l((unsigned)fx_lo(us), (unsigned)fx_hi(us), 7)));
    U[d].h = (int)((unsigned)U[d].h + (unsigned)u0);  // u0 + (us >> 25) at frac 60
    if (velocity) velocity[d] = U[d];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i <= d; ++i) {
      FxAcc a = fx_zero<0>();
      fx_mac(a, M[d].h, M[d].l, U[i]);
      P[d][i] = fx_fold<0>(a);
    }
    W -= P[d][d];
  }
  const Fx2 Ws = fx_split(W);
  FxAcc a = fx_zero<2>();
  fx_mac(a, g2h, g2l, Ws);
  const fxi p = fx_fold<2>(a);
  const Fx2 H = fx_split(q[D + 1] + p);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int d = 0; d < D; ++d) {
    F[d][0] = fx_join((unsigned)(fx_hi(q[1 + d]) >> 4), m4[d]);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < D; ++j) F[d][1 + j] = j == d ? P[d][d] + p : j < d ? P[d][j] : P[j][d];
    a = fx_zero<4>();
    fx_mac(a, H.h, H.l, U[d]);
    F[d][D + 1] = fx_fold<4>(a);
    // 1D: |m u| < 4 and |p| < 4 already
    if (D > 1) bad |= ((unsigned)fx_hi(F[d][1 + d]) + (1u << 28)) & 0xe0000000u;
    bad |= ((unsigned)fx_hi(F[d][D + 1]) + (1u << 28)) & 0xe0000000u;
  }
}

ADER_HD void fx_flux(fxi rho, fxi m, fxi E, int g2h, int g2l, fxi& F0, fxi& F1, fxi& F2,
                     unsigned& bad) {
  const fxi q[3] = {rho, m, E};
  fxi F[1][3];
  fx_fluxes<1>(q, g2h, g2l, F, bad);
  F0 = F[0][0];
  F1 = F[0][1];
  F2 = F[0][2];
}

}  // namespace ader
