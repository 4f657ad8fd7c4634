// ader_fixd.cuh -- the 2D and 3D LST-DG predictors (tensor-product form of Sec. 1.1
// eq. lst_dg_predictor_picard, see ader_kernels2d.cuh and ader_kernels3d.cuh) with
// their sweeps in the fixed-point arithmetic of ader_fix.h: one thread per
// space-time node, several cells per block, the record layout of the FP64 kernels.
//
// What bounds it.  The FP64 kernels keep the FP64 pipe ~90 % busy: a node takes
// D n + n products per variable and sweep, 64 issue cycles of a scheduler each.  In
// two limbs a product is 3 multiply-adds of 4 cycles, and it is fed from shared
// memory: fluxes and the contracted s as limb pairs, one plane per variable, so that
// a warp's 8-byte reads are contiguous.  Predictor per launch, FP64 kernel -> this one:
// 2D N = 5, 160 x 157 cells 3.74 -> 1.17 ms; 2D N = 3, 256^2 2.12 -> 0.70 ms; 2D N = 7,
// 80^2 2.49 -> 0.78 ms; 3D N = 3, 48 x 47 x 45 25.0 -> 7.23 ms; 3D N = 1, 64^3 2.94 ->
// 0.88 ms; 3D N = 4, 16^3 3.21 -> 1.03 ms.  ncu: multiplier pipe 58-64 % busy, the rest
// block barriers (a sweep's phases over the spatial nodes leave most of a block idle)
// and fixed-latency waits; 4 resident blocks of <= 256 threads measured 3-9 % faster
// than 3 (80 registers), 5 the same.
//
// Units and formats are those of ader_fix.cuh, one velocity unit per cell for every
// direction.  (dt/h_d) k~ goes into the first contraction, whose sum s over the
// directions is kept at frac 58 below 2; kappa~ is then a constant table.  Cells that
// do not fit are redone by the FP64 block code.
#pragma once

#include "ader_fix.cuh"
#include "ader_kernels2d.cuh"
#include "ader_kernels3d.cuh"

namespace ader {

template <int D, int N, int T>
struct FixDCfg {
  static constexpr int n = N + 1;
  static constexpr int NS = D == 2 ? n * n : n * n * n;  // spatial nodes
  static constexpr int NST = NS * n;
  static constexpr int M = D + 2;
  static constexpr int CPB = NST >= T / 2 ? 1 : T / NST;  // as Pred2Cfg, Pred3Cfg
  static constexpr int THREADS = CPB * NST;
  static constexpr int REC = (2 * D + 1) * NS * M;
  static constexpr int LD = D == 2 ? 1 : 2;  // log2 bound of the number of directions
  static constexpr int SET = M * CPB * NST;  // one value per node and variable
  // flux planes per direction, s, the iterate; the initial data
  static constexpr size_t kFixBytes = (size_t)((D + 2) * SET + M * CPB * NS) * sizeof(fxi);
  static constexpr bool kValid = N >= 1 && THREADS <= 1024 && kFixBytes <= 200 * 1024;
  static constexpr int MIN_BLOCKS = THREADS <= 256 ? 4 : THREADS <= 512 ? 2 : 1;
};
template <int D, int N, int T>
struct FixDBlock;  // the FP64 block code's shared memory
template <int N, int T>
struct FixDBlock<2, N, T> {
  using Params = Predict2DParams;
  using Shared = Pred2Shared<N, T>;
};
template <int N, int T>
struct FixDBlock<3, N, T> {
  using Params = Predict3DParams;
  using Shared = Pred3Shared<N, T>;
};
template <int D, int N, int T>
constexpr size_t fixd_smem_bytes() {
  constexpr size_t a = FixDCfg<D, N, T>::kFixBytes, b = sizeof(typename FixDBlock<D, N, T>::Shared);
  return a > b ? a : b;
}

template <int D, int N, int CPB>
struct FixDShared {
  int2 kd[D][N + 1][N + 1], vd[D][N + 1][N + 1];  // (dt/h_d) k~ and (dt/h_d) D~ / w
  int2 nk[N + 1][N + 1], nkrow[N + 1];            // -kappa~ and its row sums
  double dt;
  int go;
  int ex[CPB][3];             // largest exponents of rho, the momenta and E
  int ea[CPB], ec[CPB];       // the cell's units
  int bad[CPB];               // the cell goes to the FP64 block code
  unsigned dl[2][CPB], qs[2][CPB];  // max |q' - q|, max |q'| (float bits)
};

template <int D, int N, int T>
static __device__ __noinline__ void fixd_redo(const typename FixDBlock<D, N, T>::Params& P,
                                              void* smem, double dt, const int* only) {
  auto& sh = *reinterpret_cast<typename FixDBlock<D, N, T>::Shared*>(smem);
  if constexpr (D == 2)
    predict2d_block<N, T>(P, sh, dt, only);
  else
    predict3d_block<N, T>(P, sh, dt, only);
}

template <int D, int N, int T>
__global__ void __launch_bounds__(FixDCfg<D, N, T>::THREADS, FixDCfg<D, N, T>::MIN_BLOCKS)
    predict_fixd_kernel(const __grid_constant__ typename FixDBlock<D, N, T>::Params P) {
  using C = FixDCfg<D, N, T>;
  constexpr int n = N + 1, h = n / 2, H = (n + 1) / 2, NS = C::NS, NST = C::NST, CPB = C::CPB;
  constexpr int M = C::M, LD = C::LD, SK = kFxSK[N], SP = kFxSP[N], SET = C::SET;
  extern __shared__ __align__(16) double smem[];
  __shared__ FixDShared<D, N, CPB> sh;
  const int tid = threadIdx.x;
  const OpsI& o = P.opi;
  if (tid == 0) {
    double d = 0.0;
    sh.go = predictor_step_dt(P.sp, &d, blockIdx.x == 0) ? 1 : 0;
    sh.dt = d;
  }
  if (tid < CPB) {
    sh.ex[tid][0] = sh.ex[tid][1] = sh.ex[tid][2] = 0;
    sh.dl[0][tid] = sh.dl[1][tid] = sh.qs[0][tid] = sh.qs[1][tid] = 0u;
  }
  __syncthreads();
  if (!sh.go) return;  // uniform
  const double dt = sh.dt;
  double lam[D];
  lam[0] = dt * P.sp.inv_dx;
  lam[1] = dt * P.inv_dy;
  if constexpr (D == 3) lam[2] = dt * P.inv_dz;

  // node (p0, spatial node sp) of cell lc; packed spatial items (cell sc, node sk)
  const int lc = tid / NST, node = tid - lc * NST;
  const int p0 = node / NS, sp = node - p0 * NS;
  const int sc = tid / NS, sk = tid - sc * NS;
  int stride[D], pd[D], sd[D];
  {
    int s = 1;
#pragma unroll
    for (int d = D - 1; d >= 0; --d) {
      stride[d] = s;
      pd[d] = (sp / s) % n;
      sd[d] = (sk / s) % n;
      s *= n;
    }
  }
  const long long cell = (long long)blockIdx.x * CPB + lc;
  const long long scell = (long long)blockIdx.x * CPB + sc;
  const bool valid = cell < P.ncells;
  const bool sitem = tid < CPB * NS && scell < P.ncells;
  int2* Fp = reinterpret_cast<int2*>(smem);               // [d][r][cell][node]
  int2* Sp = Fp + D * SET;                                // [r][cell][node]
  fxi* Qp = reinterpret_cast<fxi*>(Sp + SET);             // [r][cell][node]
  fxi* Up = Qp + SET;                                     // [r][cell][spatial node]
  constexpr int PL = CPB * NST, UL = CPB * NS;            // plane lengths

  // the cells' units
  double ud[M];
  if (sitem) {
    int em = 0;
#pragma unroll
    for (int r = 0; r < M; ++r) {
      ud[r] = P.u[(scell * NS + sk) * M + r];
      const int e = (__double2hiint(ud[r]) >> 20) & 0x7ff;
      if (r == 0) atomicMax(&sh.ex[sc][0], e);
      if (r > 0 && r <= D) em = max(em, e);
      if (r == M - 1) atomicMax(&sh.ex[sc][2], e);
    }
    atomicMax(&sh.ex[sc][1], em);
  }
  __syncthreads();
  if (tid < CPB) {
    const int er = sh.ex[tid][0], em = sh.ex[tid][1], ee = sh.ex[tid][2];
    const int ea = er - 1022, ec = max((ee - 1022 - ea + 1) >> 1, em - 1022 - ea);
    const bool bad = max(er, max(em, ee)) >= 1023 + 60 || abs(ea) > 30 || abs(ec) > 30;
    sh.ea[tid] = bad ? 0 : ea;
    sh.ec[tid] = bad ? 0 : ec;
    sh.bad[tid] = bad;
  }
  __syncthreads();
  // tables at frac 62 - SK - LD - ke, ke the exponent of the largest dt/h_d; s folds to
  // frac 58 with a left shift, a right one in slow cells (see ader_fix.cuh)
  double lmax = lam[0];
#pragma unroll
  for (int d = 1; d < D; ++d) lmax = lam[d] > lmax ? lam[d] : lmax;
  const int lex = (__double2hiint(lmax) >> 20) & 0xfff;
  const bool lam_ok = lex > 600 && lex < 1400;
  const int ke = lam_ok ? lex - 1022 : 0;
  const double kscale = lam_ok ? fx_pow2(62 - SK - LD - ke) : 0.0;
  for (int i = tid; i < (2 * D + 1) * n * n; i += C::THREADS) {
    const int t = i / (n * n), a = (i / n) % n, b = i % n;
    const double x = t < D       ? lam[t] * P.ops.kt[a][b] * kscale
                     : t < 2 * D ? lam[t - D] * P.ops.vt[a][b] * kscale
                                 : -0x1p62 * P.ops.kap[a][b];
    const Fx2 v = fx_split(__double2ll_rn(x));
    (t < D       ? sh.kd[t][a][b]
     : t < 2 * D ? sh.vd[t - D][a][b]
                 : sh.nk[a][b]) = make_int2(v.h, v.l);
  }
  if (tid < n) {
    const Fx2 v = fx_split(__double2ll_rn(-0x1p62 * P.ops.kaprow[tid]));
    sh.nkrow[tid] = make_int2(v.h, v.l);
  }
  if (tid < CPB) {
    const int ksh = 3 + SK + LD + ke + sh.ec[tid];
    if (!lam_ok || ksh > 26) sh.bad[tid] = 1;
  }
  if (sitem) {
    const int ea = sh.ea[sc], ec = sh.ec[sc];
#pragma unroll
    for (int r = 0; r < M; ++r)
      Up[r * UL + sc * NS + sk] = __double2ll_rn(
          fx_scale(ud[r], r == M - 1 ? kFxF - ea - 2 * ec : kFxM - ea - (r ? ec : 0)));
  }
  __syncthreads();
  // fold of s, its rounding and the check |s| < 2 (frac 58, before the shift)
  auto fold_of = [&](int c) { return sh.bad[c] ? 0 : max(3 + SK + LD + ke + sh.ec[c], -62); };
  const int ksh = fold_of(lc), ksh_s = sitem ? fold_of(sc) : 0;
  const float sf1 = fx_pow2f(sh.ec[lc]), sfl = fx_pow2f(sh.ea[lc]) * 0x1p-61f;
  const int cap = P.fixed_iter > 0 ? P.fixed_iter : P.max_iter;
  const bool fixed = P.fixed_iter > 0;
  bool done = !valid || sh.bad[lc], conv = fixed;

  // fluxes of q (read from src, a plane every len) to the flux planes at slot `at`
  auto store_fluxes = [&](const fxi* src, int len, int at, int* flag) {
    fxi q[M], F[D][M];
    unsigned b = 0u;
#pragma unroll
    for (int r = 0; r < M; ++r) q[r] = src[r * len];
    fx_fluxes<D>(q, o.g2[0], o.g2[1], F, b);
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll
      for (int r = 0; r < M; ++r) {
        const Fx2 v = fx_split(F[d][r]);
        Fp[d * SET + r * PL + at] = make_int2(v.h, v.l);
      }
    if (b) atomicOr(flag, 1);
  };
  // s = sum_d (dt/h_d) k~ F_d at the node with directional indices id, whose lines start
  // at node line0 of the planes
  auto contract = [&](const int (&id)[D], int cell0, int nd, int sh_s, int* flag) {
    int2 c[D][n];
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll
      for (int m = 0; m < n; ++m) c[d][m] = sh.kd[d][id[d]][m];
    const int up = max(sh_s, 0);
    const fxi rnd = (fxi)1 << (31 - up);
    const int add = 1 << (27 - up);
    const unsigned mask = ~0u << (28 - up);
    unsigned b = 0u;
#pragma unroll 1
    for (int r = 0; r < M; ++r) {
      FxAcc a{0, rnd, 0};
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int2* line = Fp + d * SET + r * PL + cell0 + nd - id[d] * stride[d];
#pragma unroll
        for (int m = 0; m < n; ++m) {
          const int2 f = line[m * stride[d]];
          fx_mac(a, c[d][m].x, c[d][m].y, Fx2{f.x, f.y});
        }
      }
      int top;
      const Fx2 s = fx_split(fx_fold_var(a, up, &top));
      b |= (unsigned)(top + add) & mask;
      Sp[r * PL + cell0 + nd] = make_int2(s.h, s.l);
    }
    if (b) atomicOr(flag, 1);
    if (sh_s < 0) fx_shift_rows<1>(Sp + cell0 + nd, M, PL, -sh_s);
  };
  // this thread's part of the maxima of an iteration (rule R3)
  auto report = [&](int it, float dl, float qs, unsigned big) {
    if (big) atomicOr(&sh.bad[lc], 1);
    atomicMax(&sh.dl[it & 1][lc], __float_as_uint(dl));
    atomicMax(&sh.qs[it & 1][lc], __float_as_uint(qs));
  };
  int cell_it = 0;
  auto decide = [&](int it) {
    __syncthreads();
    if (!done) {
      cell_it = it;
      const float dl = __uint_as_float(sh.dl[it & 1][lc]), qs = __uint_as_float(sh.qs[it & 1][lc]);
      if (sh.bad[lc]) {
        done = true;
      } else if (!fixed && dl <= P.tolf * kFxTol * fmaxf(qs, 1.0f)) {
        done = true;
        conv = true;
      }
    }
    if (node == 0) sh.dl[(it + 1) & 1][lc] = sh.qs[(it + 1) & 1][lc] = 0u;
  };

  // iteration 1 from q = u in every tau row: s once per spatial node (tau row 0 of
  // the planes), q' = u - (sum_m kappa~[p0][m]) s
  if (sitem && !sh.bad[sc]) store_fluxes(Up + sc * NS + sk, UL, sc * NST + sk, &sh.bad[sc]);
  __syncthreads();
  if (sitem && !sh.bad[sc]) contract(sd, sc * NST, sk, ksh_s, &sh.bad[sc]);
  __syncthreads();
  if (!done) {
    const int2 c = sh.nkrow[p0];
    float dl = 0.0f, qs = 0.0f, sf = sfl;
    unsigned big = 0u;
#pragma unroll 1
    for (int r = 0; r < M; ++r) {
      const bool last = r == M - 1;
      const int2 s = Sp[r * PL + lc * NST + sp];
      FxAcc a{0, last ? (fxi)1 << 30 : (fxi)1 << 26, 0};
      fx_mac(a, c.x, c.y, Fx2{s.x, s.y});
      const fxi x = fx_fold_var(a, last ? 1 : 5);
      const fxi v = Up[r * UL + lc * NS + sp] + x;
      Qp[r * PL + lc * NST + node] = v;
      const int qm = abs(fx_hi(v));
      if (last) sf *= 16.0f * sf1;
      if (r == 1) sf *= sf1;
      dl = fmaxf(dl, fx_abs_float(x) * sf);
      qs = fmaxf(qs, (float)qm * (sf * 0x1p32f));
      big |= (unsigned)qm >> (last ? 26 : 30);
    }
    report(1, dl, qs, big);
  }
  decide(1);
  int it = 1;
  while (__syncthreads_or(!done && it < cap)) {
    ++it;
    if (!done) store_fluxes(Qp + lc * NST + node, PL, lc * NST + node, &sh.bad[lc]);
    __syncthreads();
    if (!done) contract(pd, lc * NST + p0 * NS, sp, ksh, &sh.bad[lc]);
    __syncthreads();
    if (!done) {
      int2 c[n];
#pragma unroll
      for (int m = 0; m < n; ++m) c[m] = sh.nk[p0][m];
      float dl = 0.0f, qs = 0.0f, sf = sfl;
      unsigned big = 0u;
#pragma unroll 1
      for (int r = 0; r < M; ++r) {
        const bool last = r == M - 1;
        FxAcc a{0, last ? (fxi)1 << 30 : (fxi)1 << 26, 0};
        const int2* col = Sp + r * PL + lc * NST + sp;
#pragma unroll
        for (int m = 0; m < n; ++m) {
          const int2 s = col[m * NS];
          fx_mac(a, c[m].x, c[m].y, Fx2{s.x, s.y});
        }
        const fxi v = Up[r * UL + lc * NS + sp] + fx_fold_var(a, last ? 1 : 5);
        fxi* qp = Qp + r * PL + lc * NST + node;
        const fxi d = v - *qp;
        *qp = v;
        const int qm = abs(fx_hi(v));
        if (last) sf *= 16.0f * sf1;
        if (r == 1) sf *= sf1;
        dl = fmaxf(dl, fx_abs_float(d) * sf);
        qs = fmaxf(qs, (float)qm * (sf * 0x1p32f));
        big |= (unsigned)qm >> (last ? 26 : 30);
      }
      report(it, dl, qs, big);
    }
    decide(it);
  }

  // ---- epilogue: traces at the 2 D sides per tau node, rounded to FP64 once ----
  const int ea = sitem ? sh.ea[sc] : 0, ec = sitem ? sh.ec[sc] : 0;
  double* rec = P.trace + scell * C::REC;
  if (sitem) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      // node m along d of the line of item (l0, transverse nodes) = sd
      int first = sd[0] * NS, t = 1;
#pragma unroll
      for (int e = 0; e < D; ++e)
        if (e != d) first += sd[t++] * stride[e];
#pragma unroll 1
      for (int r = 0; r < M; ++r) {
        Fx2 e[H], f[H];
        {
          fxi v[n];
#pragma unroll
          for (int m = 0; m < n; ++m) {
            const fxi q = Qp[r * PL + sc * NST + first + m * stride[d]];
            v[m] = r < M - 1 ? (q + 2) >> 2 : q * 4;  // frac 59
          }
          fx_even_odd<n>(v, e, f);
        }
        FxAcc S = fx_zero<0>(), A = fx_zero<0>();
#pragma unroll
        for (int k = 0; k < H; ++k) fx_mac(S, o.pa[k][0], o.pa[k][1], e[k]);
#pragma unroll
        for (int k = 0; k < h; ++k) fx_mac(A, o.pb[k][0], o.pb[k][1], f[k]);
        const fxi s = fx_fold<0>(S), a = fx_fold<0>(A);  // frac 58 - SP
        const int st = ea + (r == 0 ? 0 : r < M - 1 ? ec : 2 * ec) - (58 - SP);
        // 2D records hold xi = 1 first, 3D records xi = 0
        rec[((2 * d + (D == 2 ? 0 : 1)) * NS + sk) * M + r] = fx_to_double(s + a, st);
        rec[((2 * d + (D == 2 ? 1 : 0)) * NS + sk) * M + r] = fx_to_double(s - a, st);
      }
    }
  }
  // time averages of the fluxes, then u + sum_d (dt/h_d) (D~ fbar_d) / w
  if (valid && !sh.bad[lc])
    store_fluxes(Qp + lc * NST + node, PL, lc * NST + node, &sh.bad[lc]);
  __syncthreads();
  int2* FB = Sp;  // [d][r][cell][spatial node], over s and the iterate
  if (sitem) {
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll 1
      for (int r = 0; r < M; ++r) {
        FxAcc a = fx_zero<2>();
        const int2* col = Fp + d * SET + r * PL + sc * NST + sk;
#pragma unroll
        for (int m = 0; m < n; ++m) {
          const int2 f = col[m * NS];
          fx_mac(a, o.w[m][0], o.w[m][1], Fx2{f.x, f.y});
        }
        const Fx2 v = fx_split(fx_fold<2>(a));
        FB[(d * M + r) * UL + sc * NS + sk] = make_int2(v.h, v.l);
      }
  }
  __syncthreads();
  if (sitem && !sh.bad[sc]) {
    const int up = max(ksh_s, 0);
    const fxi rnd = (fxi)1 << (31 - up);
    const int add = 1 << (27 - up);
    const unsigned mask = ~0u << (28 - up);
    unsigned b = 0u;
#pragma unroll 1
    for (int r = 0; r < M; ++r) {
      FxAcc a{0, rnd, 0};
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int2* line = FB + (d * M + r) * UL + sc * NS + sk - sd[d] * stride[d];
#pragma unroll
        for (int m = 0; m < n; ++m) {
          const int2 c = sh.vd[d][sd[d]][m], f = line[m * stride[d]];
          fx_mac(a, c.x, c.y, Fx2{f.x, f.y});
        }
      }
      int top;
      fxi x = fx_fold_var(a, up, &top);  // frac 58
      if (ksh_s < 0) x = fx_shr(x, -ksh_s);
      b |= (unsigned)(top + add) & mask;
      const fxi u = Up[r * UL + sc * NS + sk];
      const fxi v = r < M - 1 ? u + x * 8 : u + ((x + 1) >> 1);
      rec[(2 * D * NS + sk) * M + r] =
          fx_to_double(v, ea + (r == 0 ? 0 : r < M - 1 ? ec : 2 * ec) - (r < M - 1 ? kFxM : kFxF));
    }
    if (b) atomicOr(&sh.bad[sc], 1);
  }
  const bool redo = __syncthreads_or(valid && sh.bad[lc]);
  if (valid && node == 0 && !sh.bad[lc]) {
    DevCtl* c = P.sp.ctl;
    if (!conv) atomicOr(&c->status, kStNotConverged);
    atomicAdd(&c->iter_sum, (unsigned long long)cell_it);
    atomicAdd((unsigned long long*)&c->iter_cells, 1ull);
    atomicMax(&c->iter_max, cell_it);
  }
  if (redo) fixd_redo<D, N, T>(P, smem, dt, sh.bad);
}

}  // namespace ader
