// Host check of the fixed-point adjoint of one collision (lbm_fixed_adjoint.cuh): every model with
// an adjoint on random nodes against the transposed Jacobian of the literal equations, taken in extended
// precision by forward differentiation of every population. The cotangents are whole multiples of 2^-60
// below 2^-4, as the kernel hands them over. Prints one line per model and node family: model, family, nodes,
// nodes taken, and, in units of 2^-60, the largest error and the root mean square errors of the fixed-point
// adjoint and of the same derivative in binary64.
// Usage: fixed_adjoint_check N SEED THETA TAU
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "lbm_fixed_adjoint.cuh"

#if defined(__SIZEOF_FLOAT128__)
typedef __float128 real;
#else
typedef long double real;  // Arm: 113 bits
#endif

static const int CX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, CY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// A value and its derivatives with respect to the nine pulled populations.
template <typename R> struct Dual {
  R v = 0, d[9] = {};
  Dual() {}
  Dual(double x) : v(x) {}
  Dual(real x) : v((R)x) {}
};
template <typename R> static Dual<R> operator+(Dual<R> a, const Dual<R>& b) {
  a.v += b.v;
  for (int i = 0; i < 9; ++i) a.d[i] += b.d[i];
  return a;
}
template <typename R> static Dual<R> operator-(Dual<R> a, const Dual<R>& b) {
  a.v -= b.v;
  for (int i = 0; i < 9; ++i) a.d[i] -= b.d[i];
  return a;
}
template <typename R> static Dual<R> operator*(const Dual<R>& a, const Dual<R>& b) {
  Dual<R> c;
  c.v = a.v * b.v;
  for (int i = 0; i < 9; ++i) c.d[i] = a.d[i] * b.v + a.v * b.d[i];
  return c;
}
template <typename R> static Dual<R> operator/(const Dual<R>& a, const Dual<R>& b) {
  Dual<R> c;
  c.v = a.v / b.v;
  for (int i = 0; i < 9; ++i) c.d[i] = (a.d[i] - c.v * b.d[i]) / b.v;
  return c;
}

// Eq. 1a for one node, every term literally over the populations.
template <typename T> static void collide_literal(const T* f, T theta, T tau, int model, T* out) {
  const T one = 1.0, two = 2.0, zero = 0.0, omp = one - one / tau;
  T rho = zero, jx = zero, jy = zero;
  for (int i = 0; i < 9; ++i) rho = rho + f[i], jx = jx + T((double)CX[i]) * f[i], jy = jy + T((double)CY[i]) * f[i];
  const T u = jx / rho, v = jy / rho;
  auto P = [&](int a, const T& w) { return a == 0 ? one - theta - w * w : (theta + w * w + T((double)a) * w) / two; };
  T eq[9], neq[9], nd = zero, nxy = zero;
  for (int i = 0; i < 9; ++i) {
    eq[i] = rho * P(CX[i], u) * P(CY[i], v);
    neq[i] = f[i] - eq[i];
    nd = nd + T(0.5 * (CX[i] * CX[i] - CY[i] * CY[i])) * neq[i], nxy = nxy + T((double)(CX[i] * CY[i])) * neq[i];
  }
  if (model == 0) {
    for (int i = 0; i < 9; ++i) out[i] = eq[i] + omp * neq[i];
    return;
  }
  const T k1 = nd / (two * theta * theta), k2 = nxy / (theta * theta), t3 = T(3.0) * theta;
  T psi[9];
  const T psx = k1 * u * (one - t3 - u * u), psy = zero - k1 * v * (one - t3 - v * v);
  if (model >= 2)
    for (int i = 1; i < 5; ++i) psi[i] = zero - (T((double)CX[i]) * psx + T((double)CY[i]) * psy) / two;
  if (model >= 3) {
    auto mu = [&](const T& w) { return (theta - w * w) * (one - theta - w * w) / (two * theta * theta); };
    const T pref = model == 4 ? zero - k1 : zero - k1 * (mu(u) + mu(v)) / two, t = theta * (one - t3);
    const T pxx = zero - pref * (u * u * (u * u - one) + t), pyy = pref * (v * v * (v * v - one) + t);
    const T pxy = pref * u * v * (u * u - v * v);
    psi[1] = psi[1] + pyy / two, psi[3] = psi[3] + pyy / two, psi[2] = psi[2] + pxx / two, psi[4] = psi[4] + pxx / two;
    for (int i = 5; i < 9; ++i) psi[i] = zero - (pxx + pyy + T((double)(CX[i] * CY[i])) * pxy) / T(4.0);
  }
  for (int i = 0; i < 9; ++i) {
    const T a = T((double)CX[i]) - u, b = T((double)CY[i]) - v, p = P(CX[i], u) * P(CY[i], v);
    out[i] = eq[i] + omp * (p * (k1 * (a * a - b * b) + k2 * a * b) + psi[i]);
  }
}

// lambda_j = sum_i mu_i d f*_i / d f_j
template <typename R> static void adjoint(const double* f, const double* mu, double theta, double tau, int model, R* lam) {
  Dual<R> x[9], o[9];
  for (int i = 0; i < 9; ++i) x[i] = Dual<R>(f[i]), x[i].d[i] = 1;
  collide_literal<Dual<R>>(x, Dual<R>(theta), Dual<R>(tau), model, o);
  for (int j = 0; j < 9; ++j) {
    lam[j] = 0;
    for (int i = 0; i < 9; ++i) lam[j] += (R)mu[i] * o[i].d[j];
  }
}

int main(int, char** v) {
  using namespace olbm::fx;
  const long n = atol(v[1]);
  std::mt19937_64 g(atol(v[2]));
  const double theta = atof(v[3]), tau = atof(v[4]);
  const Coefs c = make_coefs(theta, tau);
  auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(g); };
  const double unit = std::ldexp(1.0, 60);
  // families: 0 a flow near equilibrium, 1 random populations (spread 0.2), 2 the corners of the
  // range (density 1/2 .. 4, velocities to 1/2, large non-equilibrium)
  for (int model = 0; model < 5; ++model)
    for (int fam = 0; fam < 3; ++fam) {
      long taken = 0;
      double worst = 0, sq = 0, sq64 = 0;
      for (long k = 0; k < n; ++k) {
        double f[9], m[9];
        Fx<60> a[9], mu[9], lam[9];
        const double rho = fam == 2 ? U(0.5, 4.0) : U(0.9, 1.1), s = fam == 2 ? 0.5 : 0.15;
        const double u = U(-s, s), w = U(-s, s), neq = fam == 2 ? U(0, 0.5) : fam == 1 ? 0.2 : 1e-3;
        for (int i = 0; i < 9; ++i) {
          const double px = CX[i] ? (theta + u * u + CX[i] * u) / 2 : 1 - theta - u * u;
          const double py = CY[i] ? (theta + w * w + CY[i] * w) / 2 : 1 - theta - w * w;
          f[i] = rho * (fam == 1 ? (CX[i] ? theta / 2 : 1 - theta) * (CY[i] ? theta / 2 : 1 - theta) : px * py) * (1 + neq * U(-1, 1));
          // a population of the fixed-point format, exact in binary64
          f[i] = std::ldexp((double)(long long)std::ldexp(f[i], 50), -50);
          a[i] = Fx<60>{(i64)std::ldexp(f[i], 60)};
          m[i] = std::ldexp((double)(long long)std::ldexp(U(-1, 1), 48), -52);  // below 2^-4
          mu[i] = Fx<60>{(i64)std::ldexp(m[i], 60)};
        }
        const Moments mo = moments(a);
        if (!moments_in_range(mo.rho, mo.jx, mo.jy)) continue;
        bool ok = false;
        switch (model) {
          case 0: ok = collide_vjp<0>(mo, mu, c, lam); break;
          case 1: ok = collide_vjp<1>(mo, mu, c, lam); break;
          case 2: ok = collide_vjp<2>(mo, mu, c, lam); break;
          case 3: ok = collide_vjp<3>(mo, mu, c, lam); break;
          default: ok = collide_vjp<4>(mo, mu, c, lam); break;
        }
        if (!ok) continue;
        ++taken;
        real r[9];
        double d[9];
        adjoint<real>(f, m, theta, tau, model, r);
        adjoint<double>(f, m, theta, tau, model, d);
        for (int i = 0; i < 9; ++i) {
          const double e = (double)((real)lam[i].v / (real)unit - r[i]), e64 = (double)((real)d[i] - r[i]);
          worst = std::max(worst, std::fabs(e));
          sq += e * e, sq64 += e64 * e64;
        }
      }
      const double q = taken ? 1.0 / std::sqrt(9.0 * taken) : 0.0;
      printf("%d %d %ld %ld %.3f %.3f %.3f\n", model, fam, n, taken, worst * unit, std::sqrt(sq) * q * unit, std::sqrt(sq64) * q * unit);
    }
  return 0;
}
