// Compiles the fixed-point arithmetic of csrc/ader_fix.h and the Rusanov flux of
// csrc/ader_fixr.cuh for the host and measures them against quadruple precision, beside
// the same flux in FP64.
//
//   flux D gamma mach jump slant   largest errors over random faces, in units of the face's
//                                  rho s, sqrt(rho E) s, E s: fixed point, FP64; the largest
//                                  error of the wave speed handed out over its stated bound,
//                                  and over the speed itself; faces taken
//   predictor_flux gamma mach      fx_flux against quadruple precision and FP64
//   magnitude                      the largest relative error of fx_abs_float
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "ader_fixr.cuh"

#ifdef __SIZEOF_FLOAT128__
typedef __float128 quad;
#else
typedef long double quad;
#endif

static quad qsqrt(quad x) {
  quad y = (quad)sqrtl((long double)x);
  for (int i = 0; i < 2; ++i) y = (y + x / y) / 2;
  return y;
}
static quad qabs(quad x) { return x < 0 ? -x : x; }

static double root(double x) { return std::sqrt(x); }
static quad root(quad x) { return qsqrt(x); }

// twice the Rusanov flux in T's arithmetic; s: the wave speed
template <int D, int DIR, typename T>
static void rusanov2(const double* a, const double* b, double gamma, T* G, T* speed) {
  constexpr int M = D + 2;
  const T g = gamma, gm1 = (T)(gamma - 1.0);
  T F[2][M], s = 0;
  for (int k = 0; k < 2; ++k) {
    const double* v = k ? b : a;
    T K = 0;
    for (int d = 0; d < D; ++d) K += (T)v[1 + d] * ((T)v[1 + d] / (T)v[0]);
    const T p = gm1 * ((T)v[M - 1] - K / 2), u = (T)v[1 + DIR] / (T)v[0];
    F[k][0] = v[1 + DIR];
    for (int d = 0; d < D; ++d) F[k][1 + d] = (T)v[1 + d] * u + (d == DIR ? p : (T)0);
    F[k][M - 1] = ((T)v[M - 1] + p) * u;
    const T sk = (u < 0 ? -u : u) + root(g * p / (T)v[0]);
    if (sk > s) s = sk;
  }
  for (int r = 0; r < M; ++r) G[r] = F[0][r] + F[1][r] - s * ((T)b[r] - (T)a[r]);
  *speed = s;
}

struct Worst {
  double fix = 0, f64 = 0, over = 0, rel = 0;
  long taken = 0;
};

template <int D, int DIR>
static Worst faces(double gamma, double mach, double jump, bool slant, long n) {
  constexpr int M = D + 2;
  std::mt19937_64 gen(12483);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  const ader::FxGas gas = ader::make_fx_gas(gamma);
  Worst w;
  for (long i = 0; i < n; ++i) {
    // primitive states: rho, p log-uniform, |u| = mach c in a random direction (slant: across
    // the face), the two sides apart by up to `jump` in every one
    const double rho = std::exp2(6 * U(gen) - 3), p = std::exp2(6 * U(gen) - 3);
    const double c = std::sqrt(gamma * p / rho);
    double dir[D], norm = 0;
    for (int d = 0; d < D; ++d) {
      dir[d] = slant && d == DIR ? 1e-3 * (U(gen) - 0.5) : 2 * U(gen) - 1;
      norm += dir[d] * dir[d];
    }
    double v[2][M];
    for (int k = 0; k < 2; ++k) {
      auto near1 = [&] { return k ? 1 + jump * (2 * U(gen) - 1) : 1.0; };
      const double r = rho * near1(), q = p * near1();
      double K = 0;
      v[k][0] = r;
      for (int d = 0; d < D; ++d) {
        const double u = mach * c * dir[d] / std::sqrt(norm) * near1();
        v[k][1 + d] = r * u;
        K += r * u * u;
      }
      v[k][M - 1] = q / (gamma - 1.0) + 0.5 * K;
    }
    double G[M], G64[M], S[4], s64;
    quad Gq[M], sq;
    if (!ader::fx_rusanov2<D, DIR>(v[0], v[1], G, gas, S)) continue;
    double plain[M];
    if (!ader::fx_rusanov2<D, DIR>(v[0], v[1], plain, gas)) std::exit(2);
    rusanov2<D, DIR, double>(v[0], v[1], gamma, G64, &s64);
    rusanov2<D, DIR, quad>(v[0], v[1], gamma, Gq, &sq);
    ++w.taken;
    // each variable's size times the largest speed of all directions
    const double sp = (mach + 1) * c, E = v[0][M - 1];
    for (int r = 0; r < M; ++r) {
      const double unit = sp * (r == 0 ? rho : r < M - 1 ? std::sqrt(rho * E) : E);
      w.fix = std::max(w.fix, (double)(qabs((quad)G[r] - Gq[r])) / unit);
      w.fix = std::max(w.fix, (double)(qabs((quad)plain[r] - Gq[r])) / unit);
      w.f64 = std::max(w.f64, (double)(qabs((quad)G64[r] - Gq[r])) / unit);
    }
    const double es = (double)(qabs((quad)S[0] - sq) / sq);
    w.over = std::max(w.over, es / S[3]);
    w.rel = std::max(w.rel, es);
  }
  return w;
}

static int predictor_flux(double gamma, double mach, long n) {
  std::mt19937_64 gen(7);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  const ader::FxGas gas = ader::make_fx_gas(gamma);
  double fix = 0, f64 = 0;
  long taken = 0;
  for (long i = 0; i < n; ++i) {
    // in the cell's units: rho in (1/4, 1), the kinetic energy and the momentum below 1
    const double rho = 0.25 + 0.75 * U(gen);
    const double c2 = 1.0 / (0.5 * mach * mach + 1.0 / (gamma * (gamma - 1.0)));
    const double e = 0.25 + 0.7 * U(gen), c = std::sqrt(c2 * e / rho);
    const double u = mach * c * (U(gen) < 0.5 ? -1 : 1);
    const double v[3] = {rho, rho * u, rho * c * c / (gamma * (gamma - 1.0)) + 0.5 * rho * u * u};
    if (std::fabs(v[1]) >= 1 || v[2] >= 1) continue;
    ader::fxi q[3], F[3];
    for (int r = 0; r < 3; ++r) q[r] = (ader::fxi)llroundl(ldexpl(v[r], r < 2 ? ader::kFxM : ader::kFxF));
    unsigned bad = 0;
    ader::fx_flux(q[0], q[1], q[2], gas.g2h, gas.g2l, F[0], F[1], F[2], bad);
    if (bad) continue;
    ++taken;
    const double inv = 1.0 / v[0], u64 = v[1] * inv, p64 = (gamma - 1.0) * (v[2] - 0.5 * v[1] * u64);
    const double F64[3] = {v[1], v[1] * u64 + p64, (v[2] + p64) * u64};
    const quad uq = (quad)v[1] / (quad)v[0],
               pq = (quad)(gamma - 1.0) * ((quad)v[2] - (quad)v[1] * uq / 2);
    const quad Fq[3] = {(quad)v[1], (quad)v[1] * uq + pq, ((quad)v[2] + pq) * uq};
    for (int r = 0; r < 3; ++r) {
      fix = std::max(fix, (double)qabs((quad)F[r] / ((quad)(1ll << ader::kFxF)) - Fq[r]));
      f64 = std::max(f64, (double)qabs((quad)F64[r] - Fq[r]));
    }
  }
  std::printf("fixed=%.17g fp64=%.17g taken=%ld\n", fix, f64, taken);
  return 0;
}

int main(int argc, char** argv) {
  if (argc == 4 && !std::strcmp(argv[1], "predictor_flux"))
    return predictor_flux(std::atof(argv[2]), std::atof(argv[3]), 10000);
  if (argc == 2 && !std::strcmp(argv[1], "magnitude")) {
    double worst = 0;
    for (int k = 0; k < 62; ++k)
      for (long long m : {1ll << k, (1ll << k) + 1, (1ll << k) / 3 + 1, (1ll << k) / 7 * 5 + 1})
        for (long long x : {m, -m})
          worst = std::max(worst, std::fabs((double)ader::fx_abs_float(x) / (double)m - 1.0));
    std::printf("worst=%.17g\n", worst);
    return 0;
  }
  if (argc != 7 || std::strcmp(argv[1], "flux")) return 1;
  const int D = std::atoi(argv[2]);
  const double gamma = std::atof(argv[3]), mach = std::atof(argv[4]), jump = std::atof(argv[5]);
  const bool slant = std::atoi(argv[6]) != 0;
  const long n = 8000;
  const Worst w = D == 1   ? faces<1, 0>(gamma, mach, jump, false, n)
                  : D == 2 ? faces<2, 1>(gamma, mach, jump, slant, n)
                           : faces<3, 1>(gamma, mach, jump, slant, n);
  std::printf("fixed=%.17g fp64=%.17g over=%.17g rel=%.17g taken=%ld\n", w.fix, w.f64, w.over, w.rel,
              w.taken);
  return 0;
}
