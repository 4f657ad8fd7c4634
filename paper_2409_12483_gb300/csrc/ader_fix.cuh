// ader_fix.cuh -- the FP64 form of the 1D LST-DG predictor (Sec. 1.1 eq.
// lst_dg_predictor_picard, initialised by eq. ind_prop, with the epilogue of
// predict_tile) with its inner loop in 60-bit fixed point (ader_fix.h).
//
// What bounds it.  The FP64 form (predict_kernel<N, 0>) keeps GB300's FP64 pipe
// (2 lanes per SM and clock) 88 % busy.  The integer multiplier does 32 lanes of
// 32 x 32 + 64 bits, a two-limb product takes 3 of its multiply-adds, so a product
// costs 12 issue cycles per scheduler against 64 of the FP64 unit; a flux takes ~75
// instructions against ~11 FP64 ones (704 cycles).  Measured, predictor per launch,
// FP64 form -> this one: N = 5, 10^5 cells 0.534 -> 0.146 ms; N = 7, 10^6 cells
// 11.6 -> 2.45 ms; N = 4 FV, 10^6 cells 2.9 -> 0.78 ms; N = 3, 2 10^4 cells
// 64 -> 29 us.  ncu (N = 5): the multiplier pipe 60 % busy, ALU 36 %, FP64 17 %,
// 24 warps per SM resident, the rest fixed-latency waits.
//
// Precision.  Each cell is taken to units of its own (powers of two from its
// largest rho, E and |m|), in which rho and m carry 61 fraction bits, E and the
// fluxes 57: a flux is off by 4e-18 to 1e-17 rms where FP64 is off by 5e-17 to
// 7e-17 (4 10^6 random states against long double), k~ f by 2^-57 of the row sum of
// |k~| max |f|.  Nodes of a cell mix in every contraction, so FP64's own error is
// 2^-53 of the same maxima.  Results are rounded to FP64 once, on output.
//
// Cells whose data do not fit (rho below 1/8 of the cell's power-of-two maximum
// or not positive, |u| or the iterate beyond twice the cell's units, scales outside
// 2^+-30, a time step of 2^15 times the CFL limit, non-finite values) are redone by the
// FP64 tile code.  A cell's result does not depend on the others of its warp or block: the
// split of a mesh over several contexts (halo cells recomputed) relies on that.
//
// Mapping.  A warp holds 32 / n cells, n lanes each; lane p owns the xi node p of
// every tau row for the point-wise work (flux, time average) and the kappa~
// contraction along tau, whose coefficients every lane shares, and the tau row p
// for k~ along xi.  The iterate and the exchanged rows live in shared memory, so
// the loops over tau rows and variables stay rolled: with the iterate in registers
// the unrolled code needed 150-208 registers (12 warps per SM, instruction-fetch
// stalls; N = 5 at 10^5 cells 0.226 ms).  A cell never leaves its warp, so the
// Picard loop has no block barrier and ends per warp.
#pragma once

#include "ader_fix.h"
#include "ader_kernels.cuh"

namespace ader {

// Warps per block WPB: 2, 4 or 8, at most 64 cells per block.
template <int N, int WPB_>
struct FixCfg {
  static constexpr int n = N + 1;
  static constexpr int CPW = 32 / n;  // cells per warp
  static constexpr int WPB = WPB_ * CPW <= kMaxCpb ? WPB_ : kMaxCpb / CPW;
  static constexpr int THREADS = 32 * WPB;
  static constexpr int CELLS = WPB * CPW;
  // cells the FP64 tile code sees: its thread mapping is tid / n
  static constexpr int CAP = (THREADS + n - 1) / n;
  // Exchange planes of a warp, one per variable: [cell][tau row][RS] limb pairs.
  // Rows are 16-byte aligned and 2 x odd long, so that the rows of a warp's lanes
  // (read and written 16 bytes at a time) fall into different banks.
  static constexpr int RS = n <= 2 ? 2 : n <= 6 ? 6 : 10;
  static constexpr int PL = CPW * n * RS;
  static constexpr int NK = (n + 1) / 2 * 2;  // row of the kappa~ table
  // per warp: the exchange planes, the iterate's planes, the kappa~ table, row sums
  static constexpr int WARP_SLOTS = 2 * kM * PL + n * NK + NK;
  static constexpr size_t kFixBytes = (size_t)WPB * WARP_SLOTS * sizeof(int2);
  static constexpr size_t kTileBytes =
      (size_t)CAP * kM * n * (n + 2) * sizeof(double) + sizeof(PredShared<N>);
  static constexpr size_t kSmemBytes = kFixBytes > kTileBytes ? kFixBytes : kTileBytes;
  // resident blocks: shared memory (1 KB reserved and < 1.5 KB static each), and 24
  // warps per SM for the register allocation
  static constexpr int kBySmem = (int)(228 * 1024 / (kSmemBytes + 2560));
  static constexpr int MIN_BLOCKS = kBySmem < 24 / WPB ? kBySmem : 24 / WPB;
  static constexpr bool kValid = N >= 1;
};

template <int N>
struct FixShared {
  int2 kt[N + 1][N + 1];   // k~ and D~ / w rows read per lane
  int2 vt[N + 1][N + 1];
  double dt;
  int go;
  int itmax, ncells, bad;
  unsigned long long itsum;
  int redo[kMaxCpb + 32];  // cells of a tile that take the FP64 tile code
};

// 2^k as a double, |k| < 1000
__device__ __forceinline__ double fx_pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// x 2^k for a normal x (0 below), |k| < 200, on the integer pipe
__device__ __forceinline__ double fx_scale(double x, int k) {
  const int hi = __double2hiint(x);
  return (hi & 0x7ff00000) ? __hiloint2double(hi + (k << 20), __double2loint(x)) : 0.0;
}
// X 2^k rounded once: the limbs enter the significands of 2^52 + .. (two FMAs; the
// first is exact: (2^52 + 2^31 + h) 2^(32+k) - (2^52 + 2^31 + 2^20) 2^(32+k)).
__device__ __forceinline__ double fx_to_double(fxi x, int k) {
  const double hi = __hiloint2double(0x43300000, fx_hi(x) ^ (int)0x80000000);
  const double lo = __hiloint2double(0x43300000, fx_lo(x));
  const double off = __hiloint2double((int)0xc3300000u + ((k + 32) << 20), (int)0x80100000u);
  return fma(lo, fx_pow2(k), fma(hi, fx_pow2(k + 32), off));
}

// n values, or limb pairs, from 16-byte aligned shared memory
template <int n>
__device__ __forceinline__ void fx_load_row(const int2* src, Fx2 (&v)[n]) {
#pragma unroll
  for (int k = 0; k + 1 < n; k += 2) {
    const int4 w = *reinterpret_cast<const int4*>(src + k);
    v[k] = Fx2{w.x, w.y};
    v[k + 1] = Fx2{w.z, w.w};
  }
  if (n & 1) v[n - 1] = Fx2{src[n - 1].x, src[n - 1].y};
}

template <int n>
__device__ __forceinline__ void fx_load_row(const int2* src, fxi (&v)[n]) {
#pragma unroll
  for (int k = 0; k + 1 < n; k += 2) {
    const int4 w = *reinterpret_cast<const int4*>(src + k);
    v[k] = fx_join((unsigned)w.y, (unsigned)w.x);
    v[k + 1] = fx_join((unsigned)w.w, (unsigned)w.z);
  }
  if (n & 1) v[n - 1] = *reinterpret_cast<const fxi*>(src + n - 1);
}
// sums and differences of the mirrored pairs of a row (the middle one of odd n: e[h])
template <int n>
__device__ __forceinline__ void fx_even_odd(const fxi (&f)[n], Fx2 (&e)[(n + 1) / 2],
                                            Fx2 (&o)[(n + 1) / 2]) {
#pragma unroll
  for (int k = 0; k < n / 2; ++k) {
    e[k] = fx_split(f[k] + f[n - 1 - k]);
    o[k] = fx_split(f[k] - f[n - 1 - k]);
  }
  if (n & 1) e[n / 2] = fx_split(f[n / 2]);
}

// the limb pairs of a row of nv variables, planes PL apart, by 2^-s (out of line: for the slow
// cells only)
template <int n>
static __device__ __noinline__ void fx_shift_rows(int2* row, int nv, int PL, int s) {
#pragma unroll 1
  for (int r = 0; r < nv; ++r)
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      const int2 v = row[r * PL + k];
      const Fx2 x = fx_split(fx_shr(((fxi)v.x << 32) + v.y, s));
      row[r * PL + k] = make_int2(x.h, x.l);
    }
}

// A cell the fixed-point form cannot take carries this (not a number the form can
// produce) in the first value of its output until the FP64 tile code has redone it.
constexpr long long kFixRedo = 0x7ff4ade2f1c5ed0dll;

// The marked cells of a block's tile, by the FP64 tile code (out of line: its
// registers and its code stay out of the hot path).  Every thread of the block.
template <int N, int WPB>
static __device__ __noinline__ void fix_redo(const PredictParams& P, const TileIO& io,
                                             long long tile, double lam, double* smem, int* redo) {
  using C = FixCfg<N, WPB>;
  constexpr int n = N + 1;
  PredShared<N>& sh = *reinterpret_cast<PredShared<N>*>(smem + (size_t)C::CAP * kM * n * (n + 2));
  const long long cell = tile * C::CELLS + threadIdx.x;
  int mine = 0;
  if (threadIdx.x < C::CELLS && cell < io.ncells) {
    const double* first = P.out_mode == kOutQ ? io.q_out + cell * (long long)(n * n * kM)
                                              : io.trace + cell * (long long)((P.dg ? 9 : 6) * n);
    mine = __double_as_longlong(*reinterpret_cast<const volatile double*>(first)) == kFixRedo;
  }
  for (int i = threadIdx.x; i < kMaxCpb + 32; i += C::THREADS) redo[i] = 0;
  if (!__syncthreads_or(mine)) return;
  if (mine) redo[threadIdx.x] = 1;
  __syncthreads();
  predict_tile<N, 0, C::CAP, C::CELLS, C::THREADS>(P, io, tile, lam, smem, sh, redo);
}

// What a warp adds to the statistics of the solve.
struct FixStats {
  int itmax = 0, itsum = 0, ncells = 0;
  bool bad = false, redo = false;
};

// The cells of one warp of a block's tile.  ke: the exponent the warp's kappa~ table
// was built with (kFixNoTable at first).
// Q: q is given (io.q_in) and only the epilogue runs; its maxima set the units
// (ader_predict and ader_correct, N = 3, 20011 cells: 62 -> 55 us together).
constexpr int kFixNoTable = 1 << 20;
template <int N, int WPB, bool Q = false>
__device__ __forceinline__ void predict_fix_warp(const PredictParams& P, const TileIO& io,
                                                 long long tile, double lam, double* smem,
                                                 const FixShared<N>& sh, int& ke, FixStats& st) {
  using C = FixCfg<N, WPB>;
  constexpr int n = N + 1, h = n / 2, H = (n + 1) / 2, RS = C::RS, PL = C::PL, NK = C::NK;
  constexpr int SK = kFxSK[N], SP = kFxSP[N], SV = kFxSV[N];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane / n, p = lane - grp * n, base = grp * n;
  const bool act = grp < C::CPW;
  const long long cell = tile * C::CELLS + warp * C::CPW + grp;
  const bool valid = act && cell < io.ncells;
  const OpsI& o = P.opi;
  // maximum over the cell's lanes: cyclic shifts by 1, 2, .. cover all n
  auto cell_max = [&](auto x) {
#pragma unroll
    for (int s = 1; s < n; s *= 2) {
      const int r = s < n - s ? s : n - s;
      x = max(x, __shfl_sync(0xffffffffu, x, base + (p + r < n ? p + r : p + r - n)));
    }
    return x;
  };

  int2* wbase = reinterpret_cast<int2*>(smem) + (size_t)warp * C::WARP_SLOTS;
  int2* ex = wbase + (act ? grp : 0) * n * RS;
  int2* row = ex + p * RS;  // this lane's tau row (xi stage), plane of variable 0
  int2* col = ex + p;       // this lane's xi node of tau row 0 (other stages)
  fxi* qc = reinterpret_cast<fxi*>(col + kM * PL);  // the iterate, as col
  int2* K = wbase + 2 * kM * PL;                     // [n][NK], then the row sums

  // the cell's units: rho < 2^ea, |m| < 2^(ea + ec), E < 2^(ea + 2 ec)
  unsigned bad = 0u;
  int ea, ec;
  fxi u0, u1, u2;
  const double* src = io.u + ((valid ? cell : 0) * n + p) * (long long)kM;
  const double* qsrc = Q ? io.q_in + ((valid ? cell : 0) * n * n + p) * (long long)kM : nullptr;
  {
    double u[kM];
    int mx[kM];
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      int f = 0;
      if constexpr (Q) {
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0)
          f = max(f, (__double2hiint(qsrc[p0 * n * kM + r]) >> 20) & 0x7ff);
        u[r] = 0.0;
      } else {
        u[r] = src[r];
        f = (__double2hiint(u[r]) >> 20) & 0x7ff;
      }
      mx[r] = cell_max(f);
    }
    ea = mx[0] - 1022;
    ec = max((mx[2] - 1022 - ea + 1) >> 1, mx[1] - 1022 - ea);
    if (max(mx[0], max(mx[1], mx[2])) >= 1023 + 60 || abs(ea) > 30 || abs(ec) > 30) {
      bad = 1u;
      ea = ec = 0;
      u[0] = u[2] = 0.5;
      u[1] = 0.0;
    }
    u0 = __double2ll_rn(fx_scale(u[0], kFxM - ea));
    u1 = __double2ll_rn(fx_scale(u[1], kFxM - ea - ec));
    u2 = __double2ll_rn(fx_scale(u[2], kFxF - ea - 2 * ec));
  }
  bool conv = true;
  int cell_it = 0;
  if constexpr (Q) {
    if (act) {
#pragma unroll
      for (int p0 = 0; p0 < n; ++p0)
#pragma unroll
        for (int r = 0; r < kM; ++r)
          qc[r * PL + p0 * RS] =
              bad ? (r == 1 ? 0 : (fxi)1 << (r ? kFxF - 1 : kFxM - 1))
                  : __double2ll_rn(fx_scale(qsrc[p0 * n * kM + r],
                                            (r < 2 ? kFxM : kFxF) - ea - r * ec));
    }
    __syncwarp();
  } else {
  // -(dt/dx) kappa~ at frac 62 - ke (ke: the exponent of dt/dx), so that kappa~ g (g at
  // frac 56 - SK) folds to frac 57 with a left shift ksh = SK + 3 + ke + ec.  A slow cell
  // (ksh < 0: 4 to 64 times below the fastest by degree, or a small time step) has its g
  // shifted right by dsh instead: dt/dx is that much smaller against its units, so g's last bit
  // stays 2^-60 of the result.  Neither depends on the other cells of the warp.
  const int lex = (__double2hiint(lam) >> 20) & 0xfff;  // sign and exponent
  const bool lam_ok = lex > 600 && lex < 1400;
  const int ke_new = lam_ok ? lex - 1022 : 0;
  if (ke_new != ke) {  // uniform over the warp
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
  // rho and m fold 4 bits further, to frac 61; |g| < 2^(59 - ksh) keeps every folded
  // sum below 2^62
  const int gadd = 1 << (27 - ksh);
  const unsigned gmask = ~0u << (28 - ksh);
  // float scales: of a velocity unit, and of the last bit of rho's iterate
  const float sf1 = fx_pow2f(ec), sfl = fx_pow2f(ea) * 0x1p-61f;
  const int cap = P.fixed_iter > 0 ? P.fixed_iter : P.max_iter;
  const bool fixed = P.fixed_iter > 0;
  const float tol = P.tolf * kFxTol;

  bool done = !valid;
  conv = fixed;
  // the cell's maxima of |q' - q| and |q'| (dl, qs, of this lane on entry) end an
  // iteration (rule R3); big: nonzero when |q'| reached 2
  auto close_iteration = [&](int it, float dl, float qs, unsigned big) {
    dl = cell_max((bad | big) ? __int_as_float(0x7f800000) : dl);
    qs = cell_max(qs);
    if (!done) {
      cell_it = it;
      if (!(dl < __int_as_float(0x7f800000))) {
        bad = 1u;
        done = true;
      } else if (!fixed && dl <= tol * fmaxf(qs, 1.0f)) {
        done = true;
        conv = true;
      }
    }
  };

  // iteration 1 from q = u in every tau row: F(u) and k~ F(u) are the same in
  // every row, q' = u - (dt/dx) tau k~ F(u), so lane p needs k~ F(u) at node p only
  {
    fxi F0, F1, F2;
    fx_flux(u0, u1, u2, o.g2[0], o.g2[1], F0, F1, F2, bad);
    const Fx2 f0 = fx_split(F0), f1 = fx_split(F1), f2 = fx_split(F2);
    if (act) {
      col[0] = make_int2(f0.h, f0.l);
      col[PL] = make_int2(f1.h, f1.l);
      col[2 * PL] = make_int2(f2.h, f2.l);
    }
    __syncwarp();
    float dl = 0.0f, qs = 0.0f, sf = sfl;
    unsigned big = 0u;
#pragma unroll 1
    for (int r = 0; r < kM; ++r) {
      FxAcc g = fx_zero<1>();
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const int2 c = sh.kt[p][k], f = ex[r * PL + k];
        fx_mac(g, c.x, c.y, Fx2{f.x, f.y});
      }
      fxi gv = fx_fold<1>(g);
      if (slow) gv = fx_shr(gv, dsh);
      const Fx2 gs = fx_split(gv);
      bad |= (unsigned)(gs.h + gadd) & gmask;
      const fxi u = r == 0 ? u0 : r == 1 ? u1 : u2;
      const int sh_r = r < 2 ? ksh + 4 : ksh;
      const fxi rnd = (fxi)1 << (31 - sh_r);
      int qm = 0;
      fxi x = 0;
#pragma unroll
      for (int p0 = 0; p0 < n; ++p0) {
        const int2 c = K[n * NK + p0];
        FxAcc a{0, rnd, 0};
        fx_mac(a, c.x, c.y, gs);
        x = fx_fold_var(a, sh_r);
        const fxi v = u + x;
        if (act) qc[r * PL + p0 * RS] = v;
        qm = max(qm, abs(fx_hi(v)));
      }
      // the largest change is in the last tau row (tau increases with p0)
      dl = fmaxf(dl, fx_abs_float(x) * sf);
      qs = fmaxf(qs, (float)qm * (sf * 0x1p32f));
      big |= (unsigned)qm >> (r < 2 ? 30 : 26);
      sf *= r == 0 ? sf1 : sf1 * 16.0f;
    }
    __syncwarp();
    close_iteration(1, dl, qs, big);
  }
  for (int it = 2; it <= cap && __any_sync(0xffffffffu, !done); ++it) {
    if (!done) {
#pragma unroll 1
      for (int p0 = 0; p0 < n; ++p0) {
        fxi F0, F1, F2;
        fx_flux(qc[p0 * RS], qc[PL + p0 * RS], qc[2 * PL + p0 * RS], o.g2[0], o.g2[1], F0, F1, F2,
                bad);
        fxi* fc = reinterpret_cast<fxi*>(col) + p0 * RS;
        fc[0] = F0;
        fc[PL] = F1;
        fc[2 * PL] = F2;
      }
    }
    __syncwarp();
    if (!done) {
      // k~ along xi of tau row p, in place (only this lane touches the row here)
#pragma unroll 1
      for (int r = 0; r < kM; ++r) {
        // even/odd form (see kxi_row): g_k = T_k + S_k, g_{n-1-k} = T_k - S_k
        Fx2 e[H], d[H];
        {
          fxi f[n];
          fx_load_row<n>(row + r * PL, f);
          fx_even_odd<n>(f, e, d);
        }
#pragma unroll
        for (int j = 0; j < H; ++j) {
          FxAcc S = fx_zero<0>(), T = fx_zero<0>();
#pragma unroll
          for (int k = 0; k < H; ++k)
            if (j < h) fx_mac(S, o.ka[j][k][0], o.ka[j][k][1], e[k]);
#pragma unroll
          for (int k = 0; k < h; ++k) fx_mac(T, o.kb[j][k][0], o.kb[j][k][1], d[k]);
          const fxi t = fx_fold<0>(T), s = j < h ? fx_fold<0>(S) : 0;
          const Fx2 ga = fx_split(t + s);
          bad |= (unsigned)(ga.h + gadd) & gmask;
          row[r * PL + j] = make_int2(ga.h, ga.l);
          if (j < h) {
            const Fx2 gb = fx_split(t - s);
            bad |= (unsigned)(gb.h + gadd) & gmask;
            row[r * PL + n - 1 - j] = make_int2(gb.h, gb.l);
          }
        }
      }
      if (slow) fx_shift_rows<n>(row, kM, PL, dsh);
    }
    __syncwarp();
    float dl = 0.0f, qs = 0.0f, sf = sfl;
    unsigned big = 0u;
    if (!done) {
      // kappa~ along tau at node p: q' = u - (dt/dx) kappa~ g
#pragma unroll 1
      for (int r = 0; r < kM; ++r) {
        Fx2 g[n];
#pragma unroll
        for (int q0 = 0; q0 < n; ++q0) {
          const int2 v = col[r * PL + q0 * RS];
          g[q0] = Fx2{v.x, v.y};
        }
        const fxi u = r == 0 ? u0 : r == 1 ? u1 : u2;
        const int sh_r = r < 2 ? ksh + 4 : ksh;
        const fxi rnd = (fxi)1 << (31 - sh_r);
        float dm = 0.0f;
        int qm = 0;
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0) {
          Fx2 c[n];
          fx_load_row<n>(K + p0 * NK, c);
          FxAcc a{0, rnd, 0};
#pragma unroll
          for (int q0 = 0; q0 < n; ++q0) fx_mac(a, c[q0].h, c[q0].l, g[q0]);
          const fxi v = u + fx_fold_var(a, sh_r);
          const fxi d = v - qc[r * PL + p0 * RS];
          qc[r * PL + p0 * RS] = v;
          qm = max(qm, abs(fx_hi(v)));
          dm = fmaxf(dm, fx_abs_float(d));
        }
        dl = fmaxf(dl, dm * sf);
        qs = fmaxf(qs, (float)qm * (sf * 0x1p32f));
        big |= (unsigned)qm >> (r < 2 ? 30 : 26);
        sf *= r == 0 ? sf1 : sf1 * 16.0f;
      }
    }
    __syncwarp();
    close_iteration(it, dl, qs, big);
  }
  }

  // ---- output, rounded to FP64 once; variable r's unit is 2^(ea + r ec) ----
  double* dst;
  if (P.out_mode == kOutQ) {
    dst = io.q_out + (valid ? cell : 0) * (long long)(n * n * kM);
    if (valid) {
#pragma unroll 1
      for (int p0 = 0; p0 < n; ++p0) {
#pragma unroll
        for (int r = 0; r < kM; ++r)
          dst[(p0 * n + p) * kM + r] =
              fx_to_double(qc[r * PL + p0 * RS], ea + r * ec - (r < 2 ? kFxM : kFxF));
      }
    }
  } else {
    dst = io.trace + (valid ? cell : 0) * (long long)((P.dg ? 9 : 6) * n);
    if (act) {
#pragma unroll 1
      for (int r = 0; r < kM; ++r)
#pragma unroll
        for (int p0 = 0; p0 < n; ++p0) {
          // at frac 59 (below 2^60)
          const fxi q = qc[r * PL + p0 * RS];
          reinterpret_cast<fxi*>(col)[r * PL + p0 * RS] = r < 2 ? (q + 2) >> 2 : q * 4;
        }
    }
    __syncwarp();
    // traces of tau row p at xi = 1 (qR) and xi = 0 (qL)
#pragma unroll 1
    for (int r = 0; r < kM; ++r) {
      // phi_k(0) = phi_{n-1-k}(1): aR = S + D, aL = S - D over the mirrored pairs
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
        const int st = ea + r * ec - (58 - SP);
        dst[p * kM + r] = fx_to_double(s + t, st);
        dst[n * kM + p * kM + r] = fx_to_double(s - t, st);
      }
    }
    if (P.dg) {
      // time average of the flux at node p, then u + (dt/dx) (sum_l D~_pl fbar_l) / w_p
      FxAcc fb[kM];
#pragma unroll
      for (int r = 0; r < kM; ++r) fb[r] = fx_zero<2>();
#pragma unroll 1
      for (int p0 = 0; p0 < n; ++p0) {
        const int wh = o.w[p0][0], wl = o.w[p0][1];
        fxi F0, F1, F2;
        fx_flux(qc[p0 * RS], qc[PL + p0 * RS], qc[2 * PL + p0 * RS], o.g2[0], o.g2[1], F0, F1, F2,
                bad);
        fx_mac(fb[0], wh, wl, fx_split(F0));
        fx_mac(fb[1], wh, wl, fx_split(F1));
        fx_mac(fb[2], wh, wl, fx_split(F2));
      }
      __syncwarp();  // the rows have been read
      if (act) {
#pragma unroll
        for (int r = 0; r < kM; ++r) {
          const Fx2 v = fx_split(fx_fold<2>(fb[r]));
          col[r * PL] = make_int2(v.h, v.l);
        }
      }
      __syncwarp();
      // D~ fbar / w at frac 57 - SV, in units of the flux (one more velocity unit)
#pragma unroll
      for (int r = 0; r < kM; ++r) {
        FxAcc a = fx_zero<2>();
#pragma unroll
        for (int l = 0; l < n; ++l) {
          const int2 c = sh.vt[p][l], f = ex[r * PL + l];
          fx_mac(a, c.x, c.y, Fx2{f.x, f.y});
        }
        const double vol = fx_to_double(fx_fold<2>(a), ea + (r + 1) * ec - (57 - SV));
        if (valid) dst[2 * n * kM + p * kM + r] = fma(lam, vol, src[r]);
      }
    }
  }
  const unsigned cell_lanes = ((1u << n) - 1u) << base;  // of no use in an idle lane
  const bool redo = (__ballot_sync(0xffffffffu, bad != 0u) & cell_lanes) != 0u;
  if (valid && p == 0) {
    if (redo) {
      st.redo = true;
      dst[0] = __longlong_as_double(kFixRedo);
    } else if (!Q) {
      st.itmax = max(st.itmax, cell_it);
      st.itsum += cell_it;
      st.ncells += 1;
      if (!conv) st.bad = true;
    }
  }
  __syncwarp();  // the planes are free for the next tile
}

template <int N>
__device__ __forceinline__ bool fix_step_dt(const PredictParams& P, const StepParams& sp,
                                            double* dt, bool lead_block, FixShared<N>& sh) {
  if (threadIdx.x == 0) {
    double d = 0.0;
    sh.go = predictor_step_dt(sp, &d, lead_block) ? 1 : 0;
    sh.dt = d;
    sh.itmax = sh.ncells = sh.bad = 0;
    sh.itsum = 0ull;
  }
  __syncthreads();
  *dt = sh.dt;
  return sh.go != 0;
}

template <int N>
__device__ __forceinline__ void fix_stage_tables(const PredictParams& P, FixShared<N>& sh) {
  constexpr int n = N + 1;
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
    const int a = i / n, b = i - a * n;
    sh.kt[a][b] = make_int2(P.opi.kt[a][b][0], P.opi.kt[a][b][1]);
    sh.vt[a][b] = make_int2(P.opi.vt[a][b][0], P.opi.vt[a][b][1]);
  }
}

// A block's share of the statistics; whether a cell of the block has to be redone.
// Every thread of the block.
template <int N>
__device__ __forceinline__ bool fix_block_stats(const TileIO& io, FixShared<N>& sh,
                                                const FixStats& st) {
  const int itmax = __reduce_max_sync(0xffffffffu, st.itmax);
  const int itsum = __reduce_add_sync(0xffffffffu, st.itsum);
  const int ncells = __reduce_add_sync(0xffffffffu, st.ncells);
  const bool bad = __any_sync(0xffffffffu, st.bad);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&sh.itmax, itmax);
    atomicAdd(&sh.itsum, (unsigned long long)itsum);
    atomicAdd(&sh.ncells, ncells);
    if (bad) atomicOr(&sh.bad, 1);
  }
  const bool redo = __syncthreads_or(st.redo);
  if (threadIdx.x == 0 && sh.ncells > 0) {
    DevCtl* c = io.ctl;
    atomicMax(&c->iter_max, sh.itmax);
    atomicAdd(&c->iter_sum, sh.itsum);
    atomicAdd((unsigned long long*)&c->iter_cells, (unsigned long long)sh.ncells);
    if (sh.bad) atomicOr(&c->status, kStNotConverged);
  }
  return redo;
}

// The same, then the cells to redo (tiles tile0, tile0 + stride, ..).
template <int N, int WPB>
__device__ __forceinline__ void fix_finish(const PredictParams& P, const TileIO& io,
                                           long long tile0, long long stride, double lam,
                                           double* smem, FixShared<N>& sh, const FixStats& st) {
  using C = FixCfg<N, WPB>;
  if (fix_block_stats<N>(io, sh, st)) {
    const long long tiles = (io.ncells + C::CELLS - 1) / C::CELLS;
    for (long long t = tile0; t < tiles; t += stride) {
      fix_redo<N, WPB>(P, io, t, lam, smem, sh.redo);
      __syncthreads();
    }
  }
}

// Blocks of a large mesh take several tiles each (the launcher sizes the grid to the
// resident blocks): the tables are built once per block and warp.
template <int N, int WPB, bool Q = false>
__global__ void __launch_bounds__(FixCfg<N, WPB>::THREADS, FixCfg<N, WPB>::MIN_BLOCKS)
    predict_fix_kernel(const __grid_constant__ PredictParams P) {
  using C = FixCfg<N, WPB>;
  extern __shared__ __align__(16) double smem[];
  __shared__ FixShared<N> sh;
  fix_stage_tables<N>(P, sh);
  double dt;
  if (!fix_step_dt<N>(P, P.sp, &dt, blockIdx.x == 0, sh)) return;  // uniform
  const TileIO io{P.u, P.trace, P.q_out, P.q_in, P.ncells, P.sp.ctl};
  const double lam = dt * P.sp.inv_dx;
  FixStats st;
  int ke = kFixNoTable;
  const long long tiles = (io.ncells + C::CELLS - 1) / C::CELLS;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x)
    predict_fix_warp<N, WPB, Q>(P, io, t, lam, smem, sh, ke, st);
  fix_finish<N, WPB>(P, io, blockIdx.x, gridDim.x, lam, smem, sh, st);
}

// Batched form over the tiles of many solves (see predict_multi_kernel).
template <int N, int WPB>
__global__ void __launch_bounds__(FixCfg<N, WPB>::THREADS, FixCfg<N, WPB>::MIN_BLOCKS)
    predict_fix_multi_kernel(const __grid_constant__ PredictParams P, const MultiArgs M) {
  using C = FixCfg<N, WPB>;
  extern __shared__ __align__(16) double smem[];
  __shared__ FixShared<N> sh;
  fix_stage_tables<N>(P, sh);
  for (long long it = blockIdx.x; it < M.nitems; it += gridDim.x) {
    const TileItem item = M.items[it];
    const SlotDesc& d = M.slots[item.slot];
    const int par = M.tick_par ^ d.par0;
    StepParams sp = d.sp;
    sp.par = par;
    double dt;
    const bool go = fix_step_dt<N>(P, sp, &dt, item.tile == 0, sh);
    if (go) {
      const TileIO io{d.u[par], d.trace, nullptr, nullptr, d.ncells, sp.ctl};
      FixStats st;
      int ke = kFixNoTable;  // another solve, another time step
      const double lam = dt * sp.inv_dx;
      predict_fix_warp<N, WPB>(P, io, item.tile, lam, smem, sh, ke, st);
      fix_finish<N, WPB>(P, io, item.tile, 1ll << 60, lam, smem, sh, st);
    }
    __syncthreads();  // shared memory is free for the next tile
  }
}

}  // namespace ader
