// ader_fixs.cuh -- the nested Picard predictors of the reacting system (source terms,
// see ader_source.cuh) and of the tracer system (non-conservative product, see
// ader_tracer.cuh) in the fixed-point arithmetic of ader_fix.h, with the mapping of
// ader_fix.cuh: a warp holds 32 / n cells, lane p owns the xi node p of every tau row
// and, for contractions along xi, the tau row p.
//
// What bounds it.  The FP64 forms iterate the same sweeps on the FP64 pipe, with at
// least two inner iterations per outer one, between block barriers, at 3 blocks per SM
// (N = 5, 10^5 cells: reacting 1.84 ms, tracer 1.34 ms).  Here the source is point-wise
// and kappa~ runs along tau, so the reacting system's inner loop stays in one lane's
// column; the tracer's needs the row derivative of phi each time.  Step times (predictor,
// interface, CFL pass): reacting N = 5, 10^5 cells 1.97 -> 0.56 ms; tracer N = 3, 30011
// cells 363 -> 88 us per step of a solve.
//
// Units.  rho, m, E as in ader_fix.cuh (|u| < 2 velocity units 2^ec); each further
// variable has a power of two of its own above its largest value in the cell and is
// kept at frac 61.  A species that is zero in the whole cell and has a source goes to the
// FP64 code: any unit chosen before it has a size costs it digits (in units of 1, c1 from
// zero by dt c2 came out 1e-14 to 2e-12 off, FP64 4e-16).  The source's coefficients dx and
// dx omega^2 (the source enters as dx S beside k~ F, under (dt/dx) kappa~) are two-limb
// mantissas with an exponent.
#pragma once

#include "ader_fix.cuh"
#include "ader_source.cuh"
#include "ader_tracer.cuh"

namespace ader {

template <int N, int SYS>
struct FixSCfg {
  static constexpr int n = N + 1;
  static constexpr int M = SYS == kSysReacting ? kMR : kMN;
  static constexpr int CPW = 32 / n;
  static constexpr int WPB = 4 * CPW <= kMaxCpb ? 4 : kMaxCpb / CPW;
  static constexpr int THREADS = 32 * WPB;
  static constexpr int CELLS = WPB * CPW;
  static constexpr int CAP = (THREADS + n - 1) / n;
  static constexpr int RS = n <= 2 ? 2 : n <= 6 ? 6 : 10;  // as FixCfg
  static constexpr int PL = CPW * n * RS;
  static constexpr int NK = (n + 1) / 2 * 2;
  // exchange planes, the iterate's planes, the tracer's velocities, the kappa~ table
  static constexpr int WARP_SLOTS = (2 * M + (SYS == kSysTracer ? 1 : 0)) * PL + n * NK + NK;
  static constexpr size_t kFixBytes = (size_t)WPB * WARP_SLOTS * sizeof(int2);
  static constexpr size_t kTileBytes =
      (size_t)CAP * n * M * (3 * n + 1) * sizeof(double) + sizeof(SrcShared<N>);
  static constexpr size_t kSmemBytes = kFixBytes > kTileBytes ? kFixBytes : kTileBytes;
  static constexpr int kBySmem = (int)(228 * 1024 / (kSmemBytes + 2560));
  static constexpr int MIN_BLOCKS = kBySmem < 5 ? kBySmem : 5;
  static constexpr bool kValid = N >= 1 && kSmemBytes <= 225 * 1024;
};

template <int N, int SYS>
static __device__ __noinline__ void fixs_redo(const PredictParams& P, const TileIO& io,
                                              long long tile, double dt, double* smem, int* redo) {
  using C = FixSCfg<N, SYS>;
  constexpr int n = N + 1, M = C::M;
  SrcShared<N>& sh =
      *reinterpret_cast<SrcShared<N>*>(smem + (size_t)C::CAP * n * M * (3 * n + 1));
  const long long cell = tile * C::CELLS + threadIdx.x;
  int mine = 0;
  if (threadIdx.x < C::CELLS && cell < io.ncells) {
    const double* first = P.out_mode == kOutQ ? io.q_out + cell * (long long)(n * n * M)
                                              : io.trace + cell * (long long)(3 * M * n);
    mine = __double_as_longlong(*reinterpret_cast<const volatile double*>(first)) == kFixRedo;
  }
  for (int i = threadIdx.x; i < kMaxCpb + 32; i += C::THREADS) redo[i] = 0;
  if (!__syncthreads_or(mine)) return;
  if (mine) redo[threadIdx.x] = 1;
  __syncthreads();
  if constexpr (SYS == kSysReacting)
    predict_src_tile<N, C::CAP, C::CELLS, C::THREADS>(P, io, tile, dt, smem, sh, redo);
  else
    predict_nc_tile<N, C::CAP, C::CELLS, C::THREADS>(P, io, tile, dt, smem, sh, redo);
}

// k~ along xi of a row of values below 2^60, even/odd form: g at frac (the row's) - 1 - SK
template <int N>
__device__ __forceinline__ void fx_xi_row(const fxi (&f)[N + 1], const OpsI& o, fxi (&g)[N + 1]) {
  constexpr int n = N + 1, h = n / 2, H = (n + 1) / 2;
  Fx2 e[H], d[H];
  fx_even_odd<n>(f, e, d);
#pragma unroll
  for (int j = 0; j < H; ++j) {
    FxAcc S = fx_zero<0>(), T = fx_zero<0>();
#pragma unroll
    for (int k = 0; k < H; ++k)
      if (j < h) fx_mac(S, o.ka[j][k][0], o.ka[j][k][1], e[k]);
#pragma unroll
    for (int k = 0; k < h; ++k) fx_mac(T, o.kb[j][k][0], o.kb[j][k][1], d[k]);
    const fxi t = fx_fold<0>(T), s = j < h ? fx_fold<0>(S) : 0;
    g[j] = t + s;
    if (j < h) g[n - 1 - j] = t - s;
  }
}

// c q: c two limbs times 2^-sh of the product's high word (sh in [1, 62], rounded)
__device__ __forceinline__ fxi fx_mul_shr(int2 c, fxi q, int sh) {
  FxAcc a{(fxi)1 << (sh - 1), 0, 0};
  fx_mac(a, c.x, c.y, fx_split(q));
  return (a.hh + (fxi)fx_hi(a.m + a.m2)) >> sh;
}

// a positive double as a two-limb mantissa in [2^61, 2^62): value = mantissa 2^-frac
__device__ __forceinline__ int2 fx_mantissa(double c, int& frac) {
  const int ex = ((__double2hiint(c) >> 20) & 0x7ff) - 1023;
  frac = 61 - ex;
  const Fx2 v = fx_split(__double2ll_rn(c * fx_pow2(frac)));
  return make_int2(v.h, v.l);
}

template <int N, int SYS>
__device__ __forceinline__ void predict_fixs_warp(const PredictParams& P, const TileIO& io,
                                                  long long tile, double dt, double* smem,
                                                  const FixShared<N>& sh, int& ke, FixStats& st) {
  using C = FixSCfg<N, SYS>;
  constexpr int n = N + 1, h = n / 2, H = (n + 1) / 2, RS = C::RS, PL = C::PL, NK = C::NK;
  constexpr int M = C::M, SK = kFxSK[N], SP = kFxSP[N], SV = kFxSV[N];
  constexpr bool kReact = SYS == kSysReacting;
  const double lam = dt * P.sp.inv_dx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane / n, p = lane - grp * n, base = grp * n;
  const bool act = grp < C::CPW;
  const long long cell = tile * C::CELLS + warp * C::CPW + grp;
  const bool valid = act && cell < io.ncells;
  const OpsI& o = P.opi;
  auto cell_max = [&](auto x) {  // maximum over the cell's lanes (see ader_fix.cuh)
#pragma unroll
    for (int s = 1; s < n; s *= 2) {
      const int r = s < n - s ? s : n - s;
      x = max(x, __shfl_sync(0xffffffffu, x, base + (p + r < n ? p + r : p + r - n)));
    }
    return x;
  };
  int2* wbase = reinterpret_cast<int2*>(smem) + (size_t)warp * C::WARP_SLOTS;
  int2* ex = wbase + (act ? grp : 0) * n * RS;
  int2* row = ex + p * RS;
  int2* col = ex + p;
  fxi* qc = reinterpret_cast<fxi*>(col + M * PL);   // the iterate's column
  int2* qrow = row + M * PL;                         // and its tau row p
  int2* ucol = col + 2 * M * PL;                     // tracer: velocities (limbs, frac 60)
  int2* urow = row + 2 * M * PL;
  int2* K = wbase + C::WARP_SLOTS - (n * NK + NK);

  // the cell's units; es[s]: the further variables'
  unsigned bad = 0u;
  int ea, ec, es[2] = {0, 0};
  fxi u[M];
  const double* src = io.u + ((valid ? cell : 0) * n + p) * (long long)M;
  {
    double ud[M];
    int mx[M];
#pragma unroll
    for (int r = 0; r < M; ++r) {
      ud[r] = src[r];
      mx[r] = cell_max((__double2hiint(ud[r]) >> 20) & 0x7ff);
    }
    ea = mx[0] - 1022;
    ec = max((mx[2] - 1022 - ea + 1) >> 1, mx[1] - 1022 - ea);
    bool out = max(mx[0], max(mx[1], mx[2])) >= 1023 + 60 || abs(ea) > 30 || abs(ec) > 30;
#pragma unroll
    for (int r = 3; r < M; ++r) {
      es[r - 3] = mx[r] ? mx[r] - 1022 : 0;  // all zero: any unit
      out |= abs(es[r - 3]) > 40;
    }
    if constexpr (kReact) out |= mx[3] ? !mx[4] && P.om2 > 0.0 : mx[4] != 0;
    if (out) {
      bad = 1u;
      ea = ec = es[0] = es[1] = 0;
#pragma unroll
      for (int r = 0; r < M; ++r) ud[r] = r == 0 || r == 2 ? 0.5 : 0.0;
    }
#pragma unroll
    for (int r = 0; r < M; ++r)
      u[r] = __double2ll_rn(fx_scale(ud[r], r == 0   ? kFxM - ea
                                            : r == 1 ? kFxM - ea - ec
                                            : r == 2 ? kFxF - ea - 2 * ec
                                                     : kFxM - es[r - 3]));
  }
  // the kappa~ table, as in ader_fix.cuh
  const int lex = (__double2hiint(lam) >> 20) & 0xfff;
  const bool lam_ok = lex > 600 && lex < 1400;
  const int ke_new = lam_ok ? lex - 1022 : 0;
  // (uniform over the warp; the vote lets the compiler know: N = 3, 30011 cells, tracer
  // predictor 62.7 -> 60.5 us)
  if (__any_sync(0xffffffffu, ke_new != ke)) {
    ke = ke_new;
    const double kscale = lam_ok ? -lam * fx_pow2(62 - ke) : 0.0;
    __syncwarp();
    for (int i = lane; i < n * (n + 1); i += 32) {
      const int a = i / (n + 1), b = i - a * (n + 1);
      const Fx2 v = fx_split(__double2ll_rn(kscale * (b < n ? P.ops.kap[a][b] : P.ops.kaprow[a])));
      K[b < n ? a * NK + b : n * NK + a] = make_int2(v.h, v.l);
    }
  }
  int ksh = SK + 3 + ke + ec;
  if (!lam_ok || ksh > 26) {
    bad = 1u;
    ksh = 0;
  }
  const int dsh = min(max(-ksh, 0), 62);
  const bool slow = __any_sync(0xffffffffu, valid && dsh > 0);
  ksh = max(ksh, 0);
  const int gadd = 1 << (27 - ksh);
  const unsigned gmask = ~0u << (28 - ksh);
  // reacting: dx and dx omega^2 against the species' units, and the shifts that bring
  // coefficient x species (frac 61) to the frac 56 - SK - dsh of g
  int2 c3{0, 0}, c4{0, 0};
  int j3 = 62, j4 = 62;
  if constexpr (kReact) {
    const double dx = dt / lam;
    int f3, f4;
    c3 = fx_mantissa(dx, f3);
    j3 = f3 - (es[1] - es[0] - ec) + SK + dsh - 59;
    if (P.om2 > 0.0) {
      c4 = fx_mantissa(dx * P.om2, f4);
      j4 = f4 - (es[0] - es[1] - ec) + SK + dsh - 59;
    }
    if (j3 < 1 || j4 < 1) bad = 1u;
    j3 = min(max(j3, 1), 62);
    j4 = min(max(j4, 1), 62);
  }
  // float scales of the last bits: rho's, a velocity unit, the further variables'
  const float sf1 = fx_pow2f(ec), sfl = fx_pow2f(ea) * 0x1p-61f;
  const int cap = P.fixed_iter > 0 ? P.fixed_iter : P.max_iter;
  const bool fixed = P.fixed_iter > 0;
  const float tol = P.tolf * kFxTol, inf = __int_as_float(0x7f800000);
  auto scale_of = [&](int r) {
    return r == 0   ? sfl
           : r == 1 ? sfl * sf1
           : r == 2 ? sfl * sf1 * sf1 * 16.0f
                    : fx_pow2f(r == 3 ? es[0] : es[1]) * 0x1p-61f;
  };

  bool done = !valid, ok = true;
  int cell_it = 0;
  // q = u in every tau row
  if (act) {
#pragma unroll
    for (int r = 0; r < M; ++r)
#pragma unroll
      for (int p0 = 0; p0 < n; ++p0) qc[r * PL + p0 * RS] = u[r];
  }
  Fx2 gE[3];
  // fluxes at one node: Euler to F, species (reacting) as q u; the velocity's limbs
  auto node_flux = [&](int p0, fxi (&F)[M], Fx2& U) {
    const fxi q[3] = {qc[p0 * RS], qc[PL + p0 * RS], qc[2 * PL + p0 * RS]};
    fxi E[1][3];
    Fx2 Uv[1];
    fx_fluxes<1>(q, o.g2[0], o.g2[1], E, bad, Uv);
    U = Uv[0];
#pragma unroll
    for (int r = 0; r < 3; ++r) F[r] = E[0][r];
#pragma unroll
    for (int r = 3; r < M; ++r) {
      if constexpr (kReact) {
        FxAcc a = fx_zero<0>();
        const Fx2 s = fx_split(qc[r * PL + p0 * RS]);
        fx_mac(a, s.h, s.l, U);
        F[r] = fx_fold<0>(a);
      }
    }
  };
  // tracer: s = u (k~ phi) of tau row p at frac 56 - SK into the phi exchange plane
  auto tracer_rows = [&]() {
    fxi f[n], g[n];
    fx_load_row<n>(qrow + 3 * PL, f);
#pragma unroll
    for (int k = 0; k < n; ++k) f[k] = (f[k] + 2) >> 2;  // frac 59
    fx_xi_row<N>(f, o, g);                               // frac 58 - SK
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const int2 w = urow[k];
      const Fx2 d = fx_split(g[k]);
      FxAcc a = fx_zero<2>();
      fx_mac(a, w.x, w.y, d);
      const Fx2 s = fx_split(fx_fold<2>(a));
      bad |= (unsigned)(s.h + gadd) & gmask;
      row[3 * PL + k] = make_int2(s.h, s.l);
    }
  };
  // kappa~ along tau of a column g (frac 56 - SK) onto variable r; its maxima
  auto kappa_column = [&](int r, const Fx2 (&g)[n], float& dl, float& qs) {
    const int sh_r = r == 2 ? ksh : ksh + 4;
    const fxi rnd = (fxi)1 << (31 - sh_r);
    const fxi ur = r == 0 ? u[0] : r == 1 ? u[1] : r == 2 ? u[2] : r == 3 ? u[3] : u[M - 1];
    float dm = 0.0f;
    int qm = 0;
#pragma unroll
    for (int p0 = 0; p0 < n; ++p0) {
      Fx2 c[n];
      fx_load_row<n>(K + p0 * NK, c);
      FxAcc a{0, rnd, 0};
#pragma unroll
      for (int q0 = 0; q0 < n; ++q0) fx_mac(a, c[q0].h, c[q0].l, g[q0]);
      const fxi v = ur + fx_fold_var(a, sh_r);
      fxi* qp = qc + r * PL + p0 * RS;
      const fxi d = v - *qp;
      *qp = v;
      qm = max(qm, abs(fx_hi(v)));
      dm = fmaxf(dm, fx_abs_float(d));
    }
    const float sc = scale_of(r);
    dl = fmaxf(dl, dm * sc);
    qs = fmaxf(qs, (float)qm * (sc * 0x1p32f));
    if ((unsigned)qm >> (r == 2 ? 26 : 30)) bad = 1u;  // |q| >= 2
  };

  for (int it = 1; it <= cap && __any_sync(0xffffffffu, !done); ++it) {
    if (it == 1) {
      // the same fluxes in every tau row: g at node p once
      fxi F[M];
      Fx2 U;
      node_flux(0, F, U);
      if (act) {
#pragma unroll
        for (int r = 0; r < (kReact ? M : 3); ++r) {
          const Fx2 f = fx_split(F[r]);
          col[r * PL] = make_int2(f.h, f.l);
        }
        if constexpr (!kReact)
#pragma unroll
          for (int p0 = 0; p0 < n; ++p0) ucol[p0 * RS] = make_int2(U.h, U.l);
      }
      __syncwarp();
      Fx2 gs[M];
#pragma unroll
      for (int r = 0; r < (kReact ? M : 3); ++r) {
        FxAcc g = fx_zero<1>();
#pragma unroll
        for (int k = 0; k < n; ++k) {
          const int2 c = sh.kt[p][k], f = ex[r * PL + k];
          fx_mac(g, c.x, c.y, Fx2{f.x, f.y});
        }
        fxi gv = fx_fold<1>(g);
        if (slow) gv = fx_shr(gv, dsh);
        gs[r] = fx_split(gv);
        bad |= (unsigned)(gs[r].h + gadd) & gmask;
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < 3; ++r) gE[r] = gs[r];
      if (act && kReact) {
#pragma unroll
        for (int r = 3; r < M; ++r)
#pragma unroll
          for (int p0 = 0; p0 < n; ++p0) col[r * PL + p0 * RS] = make_int2(gs[r].h, gs[r].l);
      }
    } else {
      if (!done) {
#pragma unroll 1
        for (int p0 = 0; p0 < n; ++p0) {
          fxi F[M];
          Fx2 U;
          node_flux(p0, F, U);
          fxi* fc = reinterpret_cast<fxi*>(col) + p0 * RS;
#pragma unroll
          for (int r = 0; r < (kReact ? M : 3); ++r) fc[r * PL] = F[r];
          if constexpr (!kReact) ucol[p0 * RS] = make_int2(U.h, U.l);
        }
      }
      __syncwarp();
      if (!done) {
#pragma unroll 1
        for (int r = 0; r < (kReact ? M : 3); ++r) {
          fxi f[n], g[n];
          fx_load_row<n>(row + r * PL, f);
          fx_xi_row<N>(f, o, g);
#pragma unroll
          for (int k = 0; k < n; ++k) {
            const Fx2 s = fx_split(g[k]);
            bad |= (unsigned)(s.h + gadd) & gmask;
            row[r * PL + k] = make_int2(s.h, s.l);
          }
        }
        if (slow) fx_shift_rows<n>(row, kReact ? M : 3, PL, dsh);
      }
    }
    __syncwarp();
    if constexpr (!kReact) {
      if (!done) tracer_rows();
      if (slow && !done) fx_shift_rows<n>(row + 3 * PL, 1, PL, dsh);
      __syncwarp();
    }
    // inner iteration 1: every variable; the Euler part does not change after it
    float dlE = 0.0f, qsE = 0.0f;
    if (!done) {
#pragma unroll 1
      for (int r = 0; r < 3; ++r) {
        if (it == 1) {
          // one g for all rows: q' = u - (dt/dx) tau g
          const Fx2 g = r == 0 ? gE[0] : r == 1 ? gE[1] : gE[2];
          const int sh_r = r < 2 ? ksh + 4 : ksh;
          const fxi rnd = (fxi)1 << (31 - sh_r);
          const fxi ur = r == 0 ? u[0] : r == 1 ? u[1] : u[2];
          int qm = 0;
          fxi x = 0;
#pragma unroll
          for (int p0 = 0; p0 < n; ++p0) {
            const int2 c = K[n * NK + p0];
            FxAcc a{0, rnd, 0};
            fx_mac(a, c.x, c.y, g);
            x = fx_fold_var(a, sh_r);
            const fxi v = ur + x;
            qc[r * PL + p0 * RS] = v;
            qm = max(qm, abs(fx_hi(v)));
          }
          const float sc = scale_of(r);
          dlE = fmaxf(dlE, fx_abs_float(x) * sc);
          qsE = fmaxf(qsE, (float)qm * (sc * 0x1p32f));
          if ((unsigned)qm >> (r == 2 ? 26 : 30)) bad = 1u;
        } else {
          Fx2 g[n];
#pragma unroll
          for (int q0 = 0; q0 < n; ++q0) {
            const int2 v = col[r * PL + q0 * RS];
            g[q0] = Fx2{v.x, v.y};
          }
          kappa_column(r, g, dlE, qsE);
        }
      }
      // the Euler exchange columns are free: the further variables at the start of
      // this outer iteration
#pragma unroll
      for (int r = 3; r < M; ++r)
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0)
          reinterpret_cast<fxi*>(col)[(r - 3) * PL + p0 * RS] = qc[r * PL + p0 * RS];
    }
    bool done_i = done;
    float qs_out = 0.0f;
    int m = 0;
    for (m = 1; m <= P.max_iter && __any_sync(0xffffffffu, !done_i); ++m) {
      float dl = m == 1 ? dlE : 0.0f, qs = qsE;
      if constexpr (kReact) {
        if (!done_i) {
          // the source at the latest iterate: - dx S in the units of g
          Fx2 g3[n], g4[n];
#pragma unroll
          for (int q0 = 0; q0 < n; ++q0) {
            const int2 a = col[3 * PL + q0 * RS], b = col[(M - 1) * PL + q0 * RS];
            const fxi q3 = qc[3 * PL + q0 * RS], q4 = qc[(M - 1) * PL + q0 * RS];
            // (h and l joined with their signs)
            g3[q0] = fx_split(((fxi)a.x << 32) + a.y - fx_mul_shr(c3, q4, j3));
            g4[q0] = fx_split(((fxi)b.x << 32) + b.y + fx_mul_shr(c4, q3, j4));
            bad |= (unsigned)(g3[q0].h + gadd) & gmask;
            bad |= (unsigned)(g4[q0].h + gadd) & gmask;
          }
          kappa_column(3, g3, dl, qs);
          kappa_column(M - 1, g4, dl, qs);
        }
      } else {
        if (m > 1) {
          // b with the latest iterate: the velocities change once, with the Euler part
          if (m == 2 && !done_i) {
#pragma unroll 1
            for (int p0 = 0; p0 < n; ++p0) {
              fxi F[M];
              Fx2 U;
              node_flux(p0, F, U);
              ucol[p0 * RS] = make_int2(U.h, U.l);
            }
          }
          __syncwarp();
          if (!done_i) tracer_rows();
          if (slow && !done_i) fx_shift_rows<n>(row + 3 * PL, 1, PL, dsh);
          __syncwarp();
        }
        if (!done_i) {
          Fx2 g[n];
#pragma unroll
          for (int q0 = 0; q0 < n; ++q0) {
            const int2 v = col[3 * PL + q0 * RS];
            g[q0] = Fx2{v.x, v.y};
          }
          kappa_column(3, g, dl, qs);
        }
        __syncwarp();
      }
      dl = cell_max(bad ? inf : dl);
      qs = cell_max(qs);
      if (!done_i) {
        qs_out = qs;
        if (!(dl < inf)) bad = 1u;
        if (bad || dl <= tol * fmaxf(qs, 1.0f)) done_i = true;
      }
    }
    // outer: the change of the whole iterate over this outer iteration
    float dl = dlE;
    if (!done) {
#pragma unroll
      for (int r = 3; r < M; ++r) {
        float dm = 0.0f;
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0)
          dm = fmaxf(dm, fx_abs_float(qc[r * PL + p0 * RS] -
                                  reinterpret_cast<const fxi*>(col)[(r - 3) * PL + p0 * RS]));
        dl = fmaxf(dl, dm * scale_of(r));
      }
    }
    dl = cell_max(dl);
    if (!done) {
      cell_it = it;
      if (!done_i) ok = false;  // the inner loop hit its cap
      if (bad || (fixed ? it == cap : dl <= tol * fmaxf(qs_out, 1.0f))) done = true;
    }
    __syncwarp();
  }
  const bool conv = ok && done;

  // ---- output, rounded to FP64 once ----
  auto unit_of = [&](int r) {
    return r == 0 ? ea : r == 1 ? ea + ec : r == 2 ? ea + 2 * ec : r == 3 ? es[0] : es[1];
  };
  double* dst;
  if (P.out_mode == kOutQ) {
    dst = io.q_out + (valid ? cell : 0) * (long long)(n * n * M);
    if (valid) {
#pragma unroll 1
      for (int p0 = 0; p0 < n; ++p0)
#pragma unroll
        for (int r = 0; r < M; ++r)
          dst[(p0 * n + p) * M + r] =
              fx_to_double(qc[r * PL + p0 * RS], unit_of(r) - (r == 2 ? kFxF : kFxM));
    }
  } else {
    dst = io.trace + (valid ? cell : 0) * (long long)(3 * M * n);
    if (act) {
#pragma unroll 1
      for (int r = 0; r < M; ++r)
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0) {
          const fxi q = qc[r * PL + p0 * RS];  // to frac 59
          reinterpret_cast<fxi*>(col)[r * PL + p0 * RS] = r == 2 ? q * 4 : (q + 2) >> 2;
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int r = 0; r < M; ++r) {
      Fx2 e[H], d[H];
      {
        fxi v[n];
        fx_load_row<n>(row + r * PL, v);
        fx_even_odd<n>(v, e, d);
      }
      FxAcc S = fx_zero<0>(), D = fx_zero<0>();
#pragma unroll
      for (int k = 0; k < H; ++k) fx_mac(S, o.pa[k][0], o.pa[k][1], e[k]);
#pragma unroll
      for (int k = 0; k < h; ++k) fx_mac(D, o.pb[k][0], o.pb[k][1], d[k]);
      if (valid) {
        const fxi s = fx_fold<0>(S), t = fx_fold<0>(D);  // frac 58 - SP
        const int un = unit_of(r) - (58 - SP);
        dst[p * M + r] = fx_to_double(s + t, un);
        dst[n * M + p * M + r] = fx_to_double(s - t, un);
      }
    }
    // time averages at node p: the fluxes, and w . species (reacting) / w . u (k~ phi)
    FxAcc fb[M], sb[2];
#pragma unroll
    for (int r = 0; r < M; ++r) fb[r] = fx_zero<2>();
    sb[0] = sb[1] = fx_zero<2>();
#pragma unroll 1
    for (int p0 = 0; p0 < n; ++p0) {
      const int wh = o.w[p0][0], wl = o.w[p0][1];
      fxi F[M];
      Fx2 U;
      node_flux(p0, F, U);
#pragma unroll
      for (int r = 0; r < (kReact ? M : 3); ++r) fx_mac(fb[r], wh, wl, fx_split(F[r]));
      if constexpr (kReact) {
        fx_mac(sb[0], wh, wl, fx_split((qc[3 * PL + p0 * RS] + 2) >> 2));
        fx_mac(sb[1], wh, wl, fx_split((qc[(M - 1) * PL + p0 * RS] + 2) >> 2));
      } else {
        if (act) ucol[p0 * RS] = make_int2(U.h, U.l);
      }
    }
    __syncwarp();  // the rows have been read
    if constexpr (!kReact) {
      if (act) tracer_rows();
      __syncwarp();
#pragma unroll
      for (int p0 = 0; p0 < n; ++p0) {
        const int2 s = col[3 * PL + p0 * RS];
        fx_mac(sb[0], o.w[p0][0], o.w[p0][1], Fx2{s.x, s.y});
      }
    }
    if (act) {
#pragma unroll
      for (int r = 0; r < (kReact ? M : 3); ++r) {
        const Fx2 v = fx_split(fx_fold<2>(fb[r]));
        col[r * PL] = make_int2(v.h, v.l);
      }
    }
    __syncwarp();
    // u + (dt/dx) (sum_l D~_pl fbar_l) / w_p, the source, the B volume term
#pragma unroll
    for (int r = 0; r < M; ++r) {
      double v = src[r];
      if (r < 3 || kReact) {
        FxAcc a = fx_zero<2>();
#pragma unroll
        for (int l = 0; l < n; ++l) {
          const int2 c = sh.vt[p][l], f = ex[r * PL + l];
          fx_mac(a, c.x, c.y, Fx2{f.x, f.y});
        }
        v = fma(lam, fx_to_double(fx_fold<2>(a), unit_of(r) + ec - (57 - SV)), v);
      }
      if (kReact && r == 3) v = fma(dt, fx_to_double(fx_fold<2>(sb[1]), es[1] - 59), v);
      if (kReact && r == 4) v = fma(-dt * P.om2, fx_to_double(fx_fold<2>(sb[0]), es[0] - 59), v);
      if (!kReact && r == 3)
        v = fma(-lam, fx_to_double(fx_fold<2>(sb[0]), es[0] + ec - (56 - SK)), v);
      if (valid) dst[2 * n * M + p * M + r] = v;
    }
  }
  const unsigned cell_lanes = ((1u << n) - 1u) << base;
  const bool redo = (__ballot_sync(0xffffffffu, bad != 0u) & cell_lanes) != 0u;
  if (valid && p == 0) {
    if (redo) {
      st.redo = true;
      dst[0] = __longlong_as_double(kFixRedo);
    } else {
      st.itmax = max(st.itmax, cell_it);
      st.itsum += cell_it;
      st.ncells += 1;
      if (!conv) st.bad = true;
    }
  }
  __syncwarp();
}

template <int N, int SYS>
__global__ void __launch_bounds__(FixSCfg<N, SYS>::THREADS, FixSCfg<N, SYS>::MIN_BLOCKS)
    predict_fixs_kernel(const __grid_constant__ PredictParams P) {
  using C = FixSCfg<N, SYS>;
  extern __shared__ __align__(16) double smem[];
  __shared__ FixShared<N> sh;
  fix_stage_tables<N>(P, sh);
  double dt;
  if (!fix_step_dt<N>(P, P.sp, &dt, blockIdx.x == 0, sh)) return;  // uniform
  const TileIO io{P.u, P.trace, P.q_out, P.q_in, P.ncells, P.sp.ctl};
  FixStats st;
  int ke = kFixNoTable;
  const long long tiles = (io.ncells + C::CELLS - 1) / C::CELLS;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x)
    predict_fixs_warp<N, SYS>(P, io, t, dt, smem, sh, ke, st);
  if (fix_block_stats<N>(io, sh, st))
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
      fixs_redo<N, SYS>(P, io, t, dt, smem, sh.redo);
      __syncthreads();
    }
}

}  // namespace ader
