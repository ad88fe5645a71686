// Host check of the fixed-point collision's coefficients (make_coefs, lbm_fixed.cuh): each against the nearest
// integer of the same expression in 113-bit arithmetic, for N random (theta, tau) of the accepted
// range and the ends of it. Prints the number of coefficients that differ and the nanoseconds of a call.
// Usage: fixed_coefs_check N SEED
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "lbm_fixed.cuh"

#if defined(__SIZEOF_FLOAT128__)
typedef __float128 real;
#else
typedef long double real;  // Arm: 113 bits
#endif

using namespace olbm::fx;

static long differ(i64 got, int F, real x) {  // 1 unless got is the integer nearest to x 2^F (ties: either)
  real d = x * (real)std::ldexp(1.0, F) - (real)got;
  return d < 0 ? -d > (real)0.5 : d > (real)0.5;
}
template <int F> static long differ(Fx<F> a, real x) { return differ(a.v, F, x); }
template <int F> static long differ(FxOp<F> a, real x) {
  return differ((i64)((u64)(i64)a.o.h << 32) + (i64)a.o.l, F, x);
}

int main(int argc, char** argv) {
  const long n = atol(argv[1]);
  std::mt19937_64 g(atol(argv[2]));
  (void)argc;
  auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(g); };
  const double thetas[] = {0.21, 0.65, 0.25, 0.5, 1.0 / 3.0, 0.4}, taus[] = {0.5, 0.50000001, 1.0, 2.0, 1e9, 1e6};
  long wrong = 0;
  i64 sink = 0;
  for (long k = 0; k < n; ++k) {
    const double theta = k < 36 ? thetas[k % 6] : U(0.21, 0.65), tau = k < 36 ? taus[k / 6] : 0.5 + std::exp(U(-12.0, 20.0));
    const Coefs c = make_coefs(theta, tau);
    if (!c.on) return 1;
    const real th = theta, one = 1, omp = one - one / (real)tau, q2 = one / (4 * th * th);
    wrong += differ(c.k1, omp * q2) + differ(c.theta_op, th) + differ(c.omp, omp) + differ(c.q2, q2) +
             differ(c.inv_theta, one / th) + differ(c.e2, (one - th) / (2 * th)) + differ(c.theta, th) +
             differ(c.h, th * (one - th)) + differ(c.t, th * (one - 3 * th)) + differ(c.c3, one - 3 * th) +
             differ(c.v0, (one - th) / th) + differ(c.theta2, th * th);
  }
  double ns = 1e9;  // the best of twenty runs: other work on the host does not count
  for (int run = 0; run < 20; ++run) {
    const auto t0 = std::chrono::steady_clock::now();
    for (int k = 0; k < 5000; ++k) sink += make_coefs(0.3 + 1e-9 * k, 0.6).k1.o.l;
    ns = std::min(ns, std::chrono::duration<double, std::nano>(std::chrono::steady_clock::now() - t0).count() / 5e3);
  }
  printf("%ld %.1f %lld\n", wrong, ns, (long long)(sink & 1));
  return 0;
}
