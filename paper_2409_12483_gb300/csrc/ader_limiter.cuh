// ader_limiter.cuh -- sm_103a kernels of the a posteriori subcell limiter of the
// 1D Euler ADER-DG scheme (Popov, arXiv 2409.12483: subcell projection
// eq. p_operator and reconstruction eq. r_operator of Sec. 1.4, admissibility
// detectors PAD and NAD eq. nad_ineq of Sec. 1.6, the finite-volume ADER-WENO2
// limiter of Sec. 2).  Run after the interface kernel has written the candidate
// u* in place of u^{n+1}:
//
// lim_detect_kernel  per cell, PAD (rho > 0, e > 0) on the subcell averages P u*
//                    and the relaxed discrete maximum principle against the
//                    extrema of P u^n over the cell and its neighbours, delta =
//                    max(delta0, eps (max - min)), in FP32 with error bounds
//                    (mode 2: every cell is troubled).  Cells that pass with the
//                    bounds to spare are cleared; the others are listed.
// lim_recompute_kernel  one block per listed cell, its lanes sharing the work of
//                    each phase: the FP64 detectors (so every flag is the FP64
//                    detectors' flag), then, where the cell is troubled, the
//                    ADER-WENO2 scheme on its 2N+1 subcells from P u^n (degree-1
//                    WENO and LST-DG predictor of every subcell, the neighbours'
//                    boundary subcells included; the Rusanov flux through each
//                    subcell face averaged over the two tau nodes), the subcell
//                    update, the pseudo-inverse reconstruction R = (P^T P)^-1 P^T
//                    with the mean of the subcell values as fallback when R v has
//                    an inadmissible subcell average; and, for the neighbours, the
//                    difference between the subcell flux and the DG flux (from the
//                    predictor traces) of the cell's own two faces.
// lim_finish_kernel  per cell: a DG cell next to a troubled one has its update
//                    corrected by that difference on the shared face, so the step
//                    stays conservative; then the
//                    screened lambda_max of the limited state for the next
//                    step (the CFL reduction of the unlimited path's interface
//                    kernel, moved here because the limiter changes the state).
//
// What bounds it.  A few listed cells per step: the chains of dependent FP64
// instructions of lone warps (64 cycles each), not bandwidth.  So nothing in FP64 is
// left to one lane that several can share: detectors by (neighbour, subcell,
// variable), predictor by (subcell, space-time node), fluxes by (face, tau node).
// Sod tube, N = 3, 10007 cells, per step, against one lane per cell in the detectors and
// per subcell in the recomputation: detectors 40 -> 10 us, recomputation 67 -> 25, finish
// (which formed the DG fluxes) 31 -> 11; every cell recomputed (mode 2), N = 5, 1e5 cells:
// step 1.82 -> 1.55 ms.
//
// Both cells of a face between two troubled cells form its flux
// from the same four subcell averages (P u^n of the same coefficients by the
// same arithmetic), so they see the same bits.
#pragma once

#include "ader_kernels.cuh"

namespace ader {


__device__ __forceinline__ bool lim_admissible(const double* U) {
  const double rho = U[0];
  const double e = U[2] - 0.5 * U[1] * U[1] / rho;  // internal energy density
  return rho > 0.0 && e > 0.0 && isfinite(rho) && isfinite(e);
}

template <int N>
__device__ __forceinline__ void lim_subcell(const LimParams& P, const double* u, int j, double* v) {
  constexpr int n = N + 1;
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < n; ++k) acc = fma(P.ops.P[j][k], u[k * kM + r], acc);
    v[r] = acc;
  }
}

// FP32 screening of the detectors.  The FP32 image of a coefficient is its
// truncation (integer operations, no FP64 work; relative error below 2^-23),
// P is rounded to FP32 (2^-24) and the n fmaf roundings add n 2^-24, so an FP32
// subcell average differs from the FP64 one by less than
// (n + 4) 2^-24 sum_k |P_jk| max_k |u_k| (the FP64 sum's own rounding and the
// second-order terms included); the bound used is twice that, with
// max_j sum_k |P_jk| in place of the row sum.  A cell whose coefficients leave
// the range where that holds (|u| above 1e30 or all below 1e-30, NaN) gets no
// bound and is decided in FP64.

// FP32 image of a cell's coefficients and the error bound of its subcell
// averages per variable (negative: no bound)
template <int N>
__device__ __forceinline__ void lim_image32(const LimParams& P, const double* u,
                                            float (&uf)[N + 1][kM], float (&bound)[kM]) {
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    float m = 0.f;
#pragma unroll
    for (int k = 0; k <= N; ++k) {
      uf[k][r] = d2f_trunc(u[k * kM + r]);
      m = fmaxf(m, fabsf(uf[k][r]));
    }
    bound[r] = (m < 1e30f && m > 1e-30f) ? (float)(N + 5) * 0x1p-23f * P.pabs * m : -1.f;
  }
}

template <int N>
__device__ __forceinline__ void lim_subcell32(const LimParams& P, const float (&uf)[N + 1][kM],
                                              int j, float* v) {
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k <= N; ++k) acc = fmaf(P.Pf[j][k], uf[k][r], acc);
    v[r] = acc;
  }
}

// neighbour index with the boundary condition (-1: none, outflow boundary)
__device__ __forceinline__ long long lim_neighbour(long long c, long long n, int bc) {
  if (c >= 0 && c < n) return c;
  if (bc == kBcOutflow) return -1;
  return c < 0 ? c + n : c - n;
}

constexpr int kLimDetect = 128;               // threads of a detector block
constexpr int kLimDetectCells = kLimDetect - 2;  // its cells (a halo cell at each end)

// FP32 extrema of the subcell averages of u and their error bound
template <int N>
__device__ __forceinline__ void lim_extrema32(const LimParams& P, const double* u, float* out) {
  float uf[N + 1][kM], bound[kM], lo[kM], hi[kM];
  lim_image32<N>(P, u, uf, bound);
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    lo[r] = INFINITY;
    hi[r] = -INFINITY;
  }
  for (int j = 0; j < P.Ns; ++j) {
    float v[kM];
    lim_subcell32<N>(P, uf, j, v);
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      lo[r] = fminf(lo[r], v[r]);
      hi[r] = fmaxf(hi[r], v[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    out[r] = lo[r];
    out[3 + r] = hi[r];
    out[6 + r] = bound[r];
  }
}

// NAD violated by one value (the FP64 detector)
__device__ __forceinline__ bool lim_outside(double v, double lo, double hi, double delta) {
  return v < lo - delta || v > hi + delta;
}

// the FP64 detectors of one cell by one thread
template <int N>
__device__ __noinline__ bool lim_detect64(const LimParams& P, long long i) {
  double lo[kM], hi[kM];
#pragma unroll
  for (int r = 0; r < kM; ++r) {
    lo[r] = INFINITY;
    hi[r] = -INFINITY;
  }
  for (int d = -1; d <= 1; ++d) {
    const long long c = lim_neighbour(i + d, P.ncells, P.bc);
    if (c < 0) continue;
    for (int j = 0; j < P.Ns; ++j) {
      double v[kM];
      lim_subcell<N>(P, P.u_old + c * ((N + 1) * kM), j, v);
#pragma unroll
      for (int r = 0; r < kM; ++r) {
        lo[r] = fmin(lo[r], v[r]);
        hi[r] = fmax(hi[r], v[r]);
      }
    }
  }
  double delta[kM];
#pragma unroll
  for (int r = 0; r < kM; ++r) delta[r] = fmax(P.delta0, P.eps * (hi[r] - lo[r]));
  bool bad = false;
  for (int j = 0; j < P.Ns; ++j) {
    double v[kM];
    lim_subcell<N>(P, P.u + i * ((N + 1) * kM), j, v);
    if (!lim_admissible(v)) bad = true;
#pragma unroll
    for (int r = 0; r < kM; ++r)
      if (lim_outside(v[r], lo[r], hi[r], delta[r])) bad = true;
  }
  return bad;
}

// A warp with more cells than this left to FP64 decides them itself, one lane each
// (~1000 FP64 instructions for the warp); fewer are listed undecided and decided by
// the blocks of lim_recompute_kernel (~140 warp instructions per cell, all SMs).  Step,
// all in place / this / all listed: Sod tube, N = 5, 1e4 cells 169 / 130 / 130 us; NAD
// with delta = 0 (nearly every cell), N = 3, 1e5 cells 1.49 / 1.49 / 1.57 ms.
constexpr int kLimListed = 8;

template <int N>
__global__ void __launch_bounds__(kLimDetect)
    lim_detect_kernel(const __grid_constant__ LimParams P) {
  __shared__ float s_mm[kLimDetect][9];  // FP32 min, max of P u^n per variable, bound
  double dt;
  int last;
  if (!corrector_step_dt(P.sp, &dt, &last)) return;
  // thread t: the extrema of cell i; threads 1 .. kLimDetectCells also its screen
  const int t = threadIdx.x;
  const long long i = (long long)blockIdx.x * kLimDetectCells + t - 1;
  const bool own = t >= 1 && t <= kLimDetectCells && i < P.ncells;
  if (P.mode == 2) {  // every cell recomputed on its subcells
    if (own) {
      P.troubled[i] = 1;
      P.list[i] = i;
      if (i == 0) {
        P.sp.ctl->lim_n = (unsigned long long)P.ncells;
        atomicAdd(&P.sp.ctl->troubled, (unsigned long long)P.ncells);
      }
    }
    return;
  }
  const long long ci = i <= P.ncells ? lim_neighbour(i, P.ncells, P.bc) : -1;
  if (ci >= 0) lim_extrema32<N>(P, P.u_old + ci * ((N + 1) * kM), s_mm[t]);
  __syncthreads();
  // FP32 screen: the cell is certainly admissible when every FP32 subcell
  // average of u* lies inside the NAD interval and PAD holds with the error
  // bounds to spare; otherwise the FP64 detectors decide
  bool sure = true;
  if (own) {
    float uf[N + 1][kM], bc[kM], lo[kM], hi[kM], bn[kM];
    lim_image32<N>(P, P.u + i * ((N + 1) * kM), uf, bc);
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      lo[r] = INFINITY;
      hi[r] = -INFINITY;
      bn[r] = 0.f;
    }
    for (int d = -1; d <= 1; ++d) {
      if (lim_neighbour(i + d, P.ncells, P.bc) < 0) continue;
      const float* mm = s_mm[t + d];
#pragma unroll
      for (int r = 0; r < kM; ++r) {
        lo[r] = fminf(lo[r], mm[r]);
        hi[r] = fmaxf(hi[r], mm[3 + r]);
        bn[r] = mm[6 + r] < 0.f ? INFINITY : fmaxf(bn[r], mm[6 + r]);
      }
    }
    float slack[kM], dlo[kM];
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      // the FP64 delta is at least max(delta0, eps (hi - lo - 2 bn))
      dlo[r] = fmaxf((float)P.delta0 * (1.f - 1e-6f), (float)P.eps * (hi[r] - lo[r] - 2.f * bn[r]));
      slack[r] = 2.f * (bn[r] + bc[r]);  // doubled for the FP32 roundings below
      if (!(bc[r] >= 0.f) || !(slack[r] < INFINITY)) sure = false;
    }
    for (int j = 0; j < P.Ns && sure; ++j) {
      float v[kM];
      lim_subcell32<N>(P, uf, j, v);
#pragma unroll
      for (int r = 0; r < kM; ++r)
        if (!(v[r] - lo[r] + dlo[r] >= slack[r]) || !(hi[r] - v[r] + dlo[r] >= slack[r]))
          sure = false;
      // PAD: rho > 0 and E - m^2 / (2 rho) > 0 with the first-order error of the
      // FP32 evaluation (four times over)
      const float kin = 0.5f * v[1] * v[1] / v[0];
      const float eb = bc[2] + (fabsf(v[1]) * bc[1] + kin * bc[0]) / v[0];
      if (!(v[0] > 4.f * bc[0]) || !(v[2] - kin > 4.f * eb + 1e-6f * (fabsf(v[2]) + kin)))
        sure = false;
    }
    if (sure) P.troubled[i] = 0;
  }
  const bool here = __popc(__ballot_sync(0xffffffffu, !sure)) > kLimListed;  // uniform
  if (sure) return;
  if (here) {
    const bool bad = lim_detect64<N>(P, i);
    P.troubled[i] = bad ? 1 : 0;
    if (!bad) return;
    atomicAdd(&P.sp.ctl->troubled, 1ull);
  }
  P.list[atomicAdd(&P.sp.ctl->lim_n, 1ull)] = here ? i : ~i;  // ~i: not decided yet
}

// Degree-1 WENO slope of one variable on a subcell with average v0 and neighbours vm,
// vp: slopes of the stencils {j-1, j} and {j, j+1}, smoothness sigma_S = slope_S^2,
// weights (sigma_S + 1e-14)^-8 normalised (written as 1 / (1 + (s_l / s_r)^8)).
__device__ __forceinline__ double lim_slope(double vm, double v0, double vp) {
  const double sl = v0 - vm, sr = vp - v0;
  double t = fma(sl, sl, 1.0e-14) * rcp64(fma(sr, sr, 1.0e-14));
  t *= t;
  t *= t;
  t *= t;
  const double om = rcp64(1.0 + t);  // weight of the left stencil
  return fma(om, sl - sr, sr);
}

// LST-DG predictor of degree 1 on one subcell (eq. lst_dg_predictor_picard with
// the degree-1 operators; lam_s = dt / subcell width) by four lanes, lane p = 2 p0 + p1
// holding the node (tau p0, xi p1) and w its initial value; then the traces at the tau
// node p0: at xi = 1 (p1 = 0) or xi = 0 (p1 = 1).  Convergence as the DG predictor:
// max |q' - q| <= tol max(1, max |q'|), capped by max_iter; fixed_iter > 0 runs exactly
// that many.  Called by whole warps; `idle` lanes take part in the exchanges only.
__device__ __forceinline__ bool lim_predict1(const LimParams& P, double lam_s,
                                             const double (&w)[kM], bool idle, double* trace) {
  const Sub1Ops& s1 = P.s1;
  const int p1 = threadIdx.x & 1, p0 = (threadIdx.x >> 1) & 1;
  constexpr unsigned all = 0xffffffffu;
  // own and exchanged operands: (dt / dx) k~ by xi, then -kappa~ by tau
  const double kto = lam_s * s1.kt[p1][p1], ktx = lam_s * s1.kt[p1][p1 ^ 1];
  const double kao = -s1.kap[p0][p0], kax = -s1.kap[p0][p0 ^ 1];
  auto magnitude = [](double x) {  // the bit pattern of |x|; a NaN does not count (as fmax)
    const unsigned long long b = dbits(x) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b;
  };
  double q[kM] = {w[0], w[1], w[2]};
  const bool fixed = P.fixed_iter > 0;
  const int cap = fixed ? P.fixed_iter : P.max_iter;
  bool done = idle, converged = fixed || idle;
  for (int it = 0; it < cap; ++it) {
    double f[kM], qn[kM];
    euler_flux<double>(q, f, P.gm1);
    unsigned long long delta = 0ull, qmax = 0ull;
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      const double sx = fma(kto, f[r], ktx * __shfl_xor_sync(all, f[r], 1));
      qn[r] = fma(kao, sx, fma(kax, __shfl_xor_sync(all, sx, 2), w[r]));
      delta = umax64(delta, magnitude(qn[r] - q[r]));
      qmax = umax64(qmax, magnitude(qn[r]));
    }
#pragma unroll
    for (int m = 1; m <= 2; m <<= 1) {
      delta = umax64(delta, __shfl_xor_sync(all, delta, m));
      qmax = umax64(qmax, __shfl_xor_sync(all, qmax, m));
    }
    if (!done) {
#pragma unroll
      for (int r = 0; r < kM; ++r) q[r] = qn[r];
      if (!fixed && bitsd(delta) <= P.tol * bitsd(umax64(qmax, dbits(1.0)))) done = converged = true;
    }
    if (__all_sync(all, done)) break;
  }
  const double* psi = p1 ? s1.psi0 : s1.psi1;
  const double pso = psi[p1], psx = psi[p1 ^ 1];
#pragma unroll
  for (int r = 0; r < kM; ++r) trace[r] = fma(pso, q[r], psx * __shfl_xor_sync(all, q[r], 1));
  return converged;
}

template <int N>
struct LimCfg {
  static constexpr int n = N + 1, Ns = 2 * N + 1;
  // four lanes per subcell, the neighbours' boundary subcells included
  static constexpr int THREADS = (4 * (Ns + 2) + 31) / 32 * 32;
  static constexpr int FLUXES = 2 * (Ns + 1) + 2 * n;  // (subcell face, tau) | (side, tau)
};

template <int N>
struct LimSmem {
  static constexpr int n = N + 1, Ns = 2 * N + 1;
  double P[Ns][n], R[n][Ns];
  double v[3][Ns][kM];       // P u^n of the left neighbour, the cell, the right neighbour
  double lo[kM], hi[kM];
  double ve[Ns + 4][kM];     // subcell averages of u^n, subcells -2 .. Ns+1
  double tr[Ns + 2][2][2][kM];  // traces of subcells -1 .. Ns: [tau][at xi = 1, 0]
  double G[LimCfg<N>::FLUXES][kM];
  double F[Ns + 1][kM];      // subcell face fluxes (dt/dx scaling)
  double vnew[Ns][kM];       // (the detectors: P u*)
  double ur[n][kM];
};

template <int N>
__global__ void __launch_bounds__(LimCfg<N>::THREADS)
    lim_recompute_kernel(const __grid_constant__ LimParams P) {
  constexpr int n = N + 1, Ns = 2 * N + 1, T = LimCfg<N>::THREADS, stride = 9 * n;
  __shared__ LimSmem<N> sh;
  double dt;
  int last;
  if (!corrector_step_dt(P.sp, &dt, &last)) return;
  const int tid = threadIdx.x;
  const long long count = (long long)P.sp.ctl->lim_n;
  if (blockIdx.x >= count) return;
  for (int t = tid; t < Ns * n; t += T) {
    (&sh.P[0][0])[t] = P.ops.P[t / n][t % n];
    (&sh.R[0][0])[t] = P.R[t / Ns][t % Ns];
  }
  const double hlam = 0.5 * dt * P.sp.inv_dx;
  const double lam_s = dt * P.sp.inv_dx * (double)Ns;  // dt / subcell width
  for (long long e = blockIdx.x; e < count; e += gridDim.x) {
    const long long entry = P.list[e], i = entry < 0 ? ~entry : entry;
    const long long nb[2] = {lim_neighbour(i - 1, P.ncells, P.bc),
                             lim_neighbour(i + 1, P.ncells, P.bc)};
    __syncthreads();  // the tables; the last cell's shared memory
    // subcell averages of u^n of the three cells: every cell's by the same arithmetic,
    // so both sides of a face between troubled cells see the same bits
    for (int t = tid; t < 3 * Ns * kM; t += T) {
      const int d = t / (Ns * kM), j = t / kM - d * Ns, r = t % kM;
      const long long c = d == 1 ? i : nb[d >> 1];
      double acc = 0.0;
      if (c >= 0) {
#pragma unroll
        for (int k = 0; k < n; ++k) acc = fma(sh.P[j][k], P.u_old[(c * n + k) * kM + r], acc);
      }
      sh.v[d][j][r] = acc;
    }
    __syncthreads();
    if (entry < 0) {
      // FP64 detectors: extrema of the cell and its neighbours from u^n, then PAD
      // and NAD on the subcell averages of u*
      if (tid < 32) {
        const int r = tid >> 3, s = tid & 7;  // eight lanes per variable
        double lo = INFINITY, hi = -INFINITY;
        if (r < kM) {
          for (int t = s; t < 3 * Ns; t += 8) {
            const int d = t / Ns;
            if (d != 1 && nb[d >> 1] < 0) continue;
            const double v = sh.v[d][t - d * Ns][r];
            lo = fmin(lo, v);
            hi = fmax(hi, v);
          }
        }
#pragma unroll
        for (int m = 1; m < 8; m <<= 1) {
          lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, m));
          hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, m));
        }
        if (r < kM && s == 0) {
          const double delta = fmax(P.delta0, P.eps * (hi - lo));
          sh.lo[r] = lo - delta;
          sh.hi[r] = hi + delta;
        }
      }
      for (int t = tid; t < Ns * kM; t += T) {
        const int j = t / kM, r = t % kM;
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < n; ++k) acc = fma(sh.P[j][k], P.u[(i * n + k) * kM + r], acc);
        sh.vnew[j][r] = acc;
      }
      __syncthreads();
      bool bad = false;
      for (int t = tid; t < Ns * (kM + 1); t += T) {  // NAD per value, then PAD per subcell
        if (t < Ns * kM) {
          const double v = sh.vnew[t / kM][t % kM];
          bad = bad || v < sh.lo[t % kM] || v > sh.hi[t % kM];
        } else {
          bad = bad || !lim_admissible(sh.vnew[t - Ns * kM]);
        }
      }
      const bool any = __syncthreads_or(bad);
      if (tid == 0) {
        P.troubled[i] = any ? 1 : 0;
        if (any) atomicAdd(&P.sp.ctl->troubled, 1ull);
      }
      if (!any) continue;  // uniform
    }
    // the cell's subcells and the neighbours' two next to each face (outflow
    // boundary: the boundary subcell itself)
    for (int t = tid; t < (Ns + 4) * kM; t += T) {
      const int j = t / kM - 2, r = t % kM;
      const int side = j < 0 ? 0 : 2;
      double v;
      if (j >= 0 && j < Ns)
        v = sh.v[1][j][r];
      else if (nb[side >> 1] >= 0)
        v = sh.v[side][j < 0 ? Ns + j : j - Ns][r];
      else
        v = sh.v[1][j < 0 ? 0 : Ns - 1][r];
      sh.ve[j + 2][r] = v;
    }
    __syncthreads();
    {
      // subcell s - 1 by lanes 4 s .. 4 s + 3: the slope's variables spread over the
      // lanes, then the predictor
      const int s = tid >> 2, sc = s < Ns + 2 ? s : Ns + 1, l = tid & 3;
      const int rs = l < kM ? l : 0;
      const double slope = lim_slope(sh.ve[sc][rs], sh.ve[sc + 1][rs], sh.ve[sc + 2][rs]);
      double w[kM], tr[kM];
#pragma unroll
      for (int r = 0; r < kM; ++r)
        w[r] = fma(__shfl_sync(0xffffffffu, slope, (tid & 28) | r), P.s1.xi[l & 1] - 0.5,
                   sh.ve[sc + 1][r]);
      const bool ok = lim_predict1(P, lam_s, w, s > Ns + 1, tr);
      if (s <= Ns + 1) {
        if (!ok) atomicOr(&P.sp.ctl->status, kStNotConverged);
#pragma unroll
        for (int r = 0; r < kM; ++r) sh.tr[s][l >> 1][l & 1][r] = tr[r];
      }
    }
    __syncthreads();
    // Rusanov fluxes: item (f, l0) of the subcell faces (f between subcells f - 1 and
    // f), then (side, l0) of the cell's own faces from the DG predictor's traces, bit for
    // bit the interface kernel's flux (mode 2 has no cell that would use the latter).  The two
    // kinds take different code: the second starts at a warp of its own (with both in one
    // warp, one after the other, the Sod tube's step of N = 3, 10007 cells took 3 % longer)
    constexpr int kSub = 2 * (Ns + 1), kOwn = (kSub + 31) / 32 * 32;
    const int fluxes = P.mode == 2 ? kSub : kOwn + 2 * n;
    for (int t = tid; t < fluxes; t += T) {
      if (t >= kSub && t < kOwn) continue;
      double a[kM], b[kM], G2[kM];
      if (t < kSub) {
#pragma unroll
        for (int r = 0; r < kM; ++r) {
          a[r] = sh.tr[t >> 1][t & 1][0][r];
          b[r] = sh.tr[(t >> 1) + 1][t & 1][1][r];
        }
      } else {
        const int side = (t - kOwn) / n, l0 = t - kOwn - side * n;
        const long long cl = side ? i : nb[0], cr = side ? nb[1] : i;
        if (cl < 0 || cr < 0) {
          // outflow boundary: the ghost side holds the boundary cell's mean of u^n
#pragma unroll
          for (int r = 0; r < kM; ++r) {
            double m = 0.0;
#pragma unroll
            for (int k = 0; k < n; ++k) m = fma(P.ops.w[k], P.u_old[(i * n + k) * kM + r], m);
            a[r] = b[r] = m;
          }
        }
#pragma unroll
        for (int r = 0; r < kM; ++r) {
          if (cl >= 0) a[r] = P.trace[cl * stride + l0 * kM + r];
          if (cr >= 0) b[r] = P.trace[cr * stride + (n + l0) * kM + r];
        }
      }
      if (t < kSub)
        rusanov2(a, b, G2, P.gamma, P.gm1);
      else
        face_flux2(a, b, G2, P.gamma, P.gm1, P.gas);
      const int at = t < kSub ? t : t - kOwn + kSub;
#pragma unroll
      for (int r = 0; r < kM; ++r) sh.G[at][r] = G2[r];
    }
    __syncthreads();
    for (int t = tid; t < (Ns + 1) * kM; t += T) {
      const int f = t / kM, r = t - f * kM;
      const double F =
          hlam * fma(P.s1.w[1], sh.G[2 * f + 1][r], P.s1.w[0] * sh.G[2 * f][r]);
      sh.F[f][r] = F;
      if (P.mode != 2 && (f == 0 || f == Ns)) {
        const int side = f ? 1 : 0;
        double g = 0.0;
#pragma unroll
        for (int l0 = 0; l0 < n; ++l0)
          g = fma(P.ops.w[l0], sh.G[2 * (Ns + 1) + side * n + l0][r], g);
        P.gface[i * 6 + side * kM + r] = F - hlam * g;
      }
    }
    __syncthreads();
    for (int t = tid; t < Ns * kM; t += T) {
      const int j = t / kM, r = t - j * kM;
      sh.vnew[j][r] = sh.ve[j + 2][r] - (double)Ns * (sh.F[j + 1][r] - sh.F[j][r]);
    }
    __syncthreads();
    // reconstruction u = R v (item = (k, r))
    for (int t = tid; t < n * kM; t += T) {
      const int k = t / kM, r = t - k * kM;
      double acc = 0.0;
#pragma unroll
      for (int j = 0; j < Ns; ++j) acc = fma(sh.R[k][j], sh.vnew[j][r], acc);
      sh.ur[k][r] = acc;
    }
    __syncthreads();
    for (int t = tid; t < Ns * kM; t += T) {
      const int j = t / kM, r = t - j * kM;
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < n; ++k) acc = fma(sh.P[j][k], sh.ur[k][r], acc);
      sh.v[0][j][r] = acc;
    }
    __syncthreads();
    const bool ok = __syncthreads_and(tid >= Ns || lim_admissible(sh.v[0][tid < Ns ? tid : 0]));
    for (int t = tid; t < n * kM; t += T) {
      const int k = t / kM, r = t - k * kM;
      double val = sh.ur[k][r];
      if (!ok) {  // the mean of the subcell values
        double mean = 0.0;
        for (int j = 0; j < Ns; ++j) mean += sh.vnew[j][r];
        val = mean / (double)Ns;
      }
      P.u[(i * n + k) * kM + r] = val;
    }
  }
}

// Every cell once its state is final: DG neighbours of troubled cells take the
// face term with the subcell flux; then (want_lambda) lambda_max of the limited
// state for the next step's CFL rule, screened like the interface kernel's
// first screen: FP32 bounds on every subcell's speed (speed_bounds_f32), FP64
// wave speeds only for the subcells whose upper bound reaches the block's
// largest lower bound, so the result is the FP64 maximum over all subcells.
template <int N>
__global__ void __launch_bounds__(128) lim_finish_kernel(const __grid_constant__ LimParams P) {
  constexpr int n = N + 1, Ns = 2 * N + 1;
  __shared__ unsigned long long s_wmax[4];
  __shared__ float s_cut;
  __shared__ int s_count;                     // candidate subcells for FP64
  __shared__ unsigned short s_list[128 * Ns];  // their items cell * Ns + j
  __shared__ double s_P[Ns][n];
  double dt;
  int last;
  if (!corrector_step_dt(P.sp, &dt, &last)) return;  // uniform over the grid
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) P.sp.ctl->lim_n = 0;  // for the next step (the control block starts zeroed)
  const bool valid = i < P.ncells;
  double u[n][kM];
  if (valid) {
    double* up = P.u + i * (n * kM);
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int r = 0; r < kM; ++r) u[k][r] = up[k * kM + r];
    if (!P.troubled[i]) {
      const long long il = lim_neighbour(i - 1, P.ncells, P.bc), ir = lim_neighbour(i + 1, P.ncells, P.bc);
      const bool tl = il >= 0 && P.troubled[il], tr = ir >= 0 && P.troubled[ir];
      if (tl || tr) {
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int r = 0; r < kM; ++r) {
            double d = 0.0;
            if (tr) d -= P.ops.psi1[k] * P.gface[ir * 6 + r];
            if (tl) d += P.ops.psi0[k] * P.gface[il * 6 + 3 + r];
            u[k][r] = fma(d, P.ops.rw[k], u[k][r]);
            up[k * kM + r] = u[k][r];
          }
      }
    }
  }
  if (!P.want_lambda) return;  // uniform over the grid
  // A cell whose coefficients equal, bit for bit, those of the previous cell of
  // the block has the same subcell wave speeds, so only the first cell of such
  // a run enters the maximum.  Uniform regions (Riemann data) stay bitwise
  // uniform from cell to cell, and there the screen below would otherwise
  // evaluate nearly every subcell in FP64 (they all tie with the maximum).
  __shared__ double s_u[128][n * kM];
  if (valid) {
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int r = 0; r < kM; ++r) s_u[threadIdx.x][k * kM + r] = u[k][r];
  }
  for (int t = threadIdx.x; t < Ns * n; t += blockDim.x) s_P[t / n][t % n] = P.ops.P[t / n][t % n];
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  bool twin = valid && threadIdx.x > 0;
  if (twin) {
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int r = 0; r < kM; ++r)
        twin = twin && dbits(s_u[threadIdx.x - 1][k * kM + r]) == dbits(u[k][r]);
  }
  const bool own = valid && !twin;  // this cell's subcells enter the maximum
  const float gf = (float)P.gamma, gm1f = (float)P.gm1;
  float uf[n][kM], lt[Ns], lo_loc = 0.f;
#pragma unroll
  for (int k = 0; k < n; ++k)
#pragma unroll
    for (int r = 0; r < kM; ++r) uf[k][r] = d2f_trunc(u[k][r]);
  // FP32 bounds on every subcell's speed (as in the interface kernel: the FP32
  // subcell average is within (n + 4) 2^-24 sum_k |P_jk| |u_k| of P u); FP64
  // below only where the upper bound reaches the block's largest lower bound.
  const float one[1] = {1.f};
  constexpr float eproj = (float)(n + 4) * 0x1p-24f;
#pragma unroll
  for (int j = 0; j < Ns; ++j) {
    float v[kM], e[kM];
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      float acc = 0.f, aab = 0.f;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        acc = fmaf(P.Pf[j][k], uf[k][r], acc);
        aab = fmaf(fabsf(P.Pf[j][k]), fabsf(uf[k][r]), aab);
      }
      v[r] = acc;
      e[r] = fmaf(eproj, aab, 0x1p-100f);
    }
    float lo;
    speed_bounds_f32<1>(v, e, one, gf, gm1f, lo, lt[j]);
    if (own) lo_loc = fmaxf(lo_loc, lo);
  }
  const unsigned long long fm = block_max_bits((unsigned long long)__float_as_uint(lo_loc), s_wmax);
  if (threadIdx.x == 0)
    s_cut = lambda_cut(&P.sp.ctl->lam[P.sp.par ^ 1], __uint_as_float((unsigned)fm));
  __syncthreads();
  const float cut = s_cut;
  // The subcells left to FP64 are few and spread thinly over the cells (on a
  // fine smooth mesh about one per cell): listed first, they are evaluated by
  // whole warps, instead of one pass per subcell index with a few lanes of
  // each warp busy.  The maximum of the same set is the same.
  if (own) {
#pragma unroll
    for (int j = 0; j < Ns; ++j)
      if (lt[j] >= cut) s_list[atomicAdd(&s_count, 1)] = (unsigned short)(threadIdx.x * Ns + j);
  }
  __syncthreads();
  const int ncand = s_count;
  double lmax = 0.0;
  bool bad = false;
  for (int t = threadIdx.x; t < ncand; t += blockDim.x) {
    const int item = s_list[t], c = item / Ns, j = item - c * Ns;
    double v[kM];
#pragma unroll
    for (int r = 0; r < kM; ++r) {
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < n; ++k) acc = fma(s_P[j][k], s_u[c][k * kM + r], acc);
      v[r] = acc;
    }
    lmax = fmax(lmax, wave_speed(v, P.gamma, P.gm1, &bad));
  }
  const unsigned long long bm = block_max_bits(dbits(lmax), s_wmax);
  if (threadIdx.x == 0) atomicMax(&P.sp.ctl->lam[P.sp.par ^ 1], bm);
  if (bad) atomicOr(&P.sp.ctl->status, kStNonPhysical);
}

}  // namespace ader
