// Host check of the fixed-point collision (lbm_fixed.cuh): every model on random
// nodes against the literal equations in extended precision, next to the error of
// the same equations in binary64. Prints one line per model and node family: model,
// family, nodes, nodes taken, largest excess of the error over half an ulp of the
// exact population, and the root mean square errors of the fixed-point collision, of
// the binary64 collision and of the exact result rounded to binary64 (all in units
// of 2^-60).
// Usage: fixed_check N SEED THETA TAU
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "lbm_fixed.cuh"

#if defined(__SIZEOF_FLOAT128__)
typedef __float128 real;
#else
typedef long double real;
#endif

static const int CX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, CY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// Eq. 1a for one node, every term literally over the populations.
template <typename T> static void collide_literal(const double* fin, double theta_, double tau_, int model, T* out) {
  const T theta = theta_, om = T(1) / T(tau_), omp = T(1) - om;
  T f[9], rho = 0, jx = 0, jy = 0;
  for (int i = 0; i < 9; ++i) f[i] = fin[i];
  for (int i = 0; i < 9; ++i) rho += f[i], jx += T(CX[i]) * f[i], jy += T(CY[i]) * f[i];
  const T u = jx / rho, v = jy / rho;
  auto P = [&](int a, T w) { return a == 0 ? T(1) - theta - w * w : (theta + w * w + T(a) * w) / T(2); };
  T eq[9], neq[9];
  for (int i = 0; i < 9; ++i) {
    if (model == 5) {
      const T wa = CX[i] ? theta / T(2) : T(1) - theta, wb = CY[i] ? theta / T(2) : T(1) - theta;
      const T cu = T(CX[i]) * u + T(CY[i]) * v;
      eq[i] = rho * wa * wb * (T(1) + cu / theta + cu * cu / (T(2) * theta * theta) - (u * u + v * v) / (T(2) * theta));
    } else {
      eq[i] = rho * P(CX[i], u) * P(CY[i], v);
    }
    neq[i] = f[i] - eq[i];
  }
  if (model == 0 || model == 5) {
    for (int i = 0; i < 9; ++i) out[i] = eq[i] + omp * neq[i];
    return;
  }
  T nd = 0, nxy = 0;
  for (int i = 0; i < 9; ++i) nd += T(CX[i] * CX[i] - CY[i] * CY[i]) * neq[i] / T(2), nxy += T(CX[i] * CY[i]) * neq[i];
  const T k1 = nd / (T(2) * theta * theta), k2 = nxy / (theta * theta);
  T psi[9] = {};
  const T psx = k1 * u * (T(1) - T(3) * theta - u * u), psy = -k1 * v * (T(1) - T(3) * theta - v * v);
  if (model >= 2)
    for (int i = 1; i < 5; ++i) psi[i] = -(T(CX[i]) * psx + T(CY[i]) * psy) / T(2);
  if (model >= 3) {
    auto mu = [&](T w) { return (theta - w * w) * (T(1) - theta - w * w) / (T(2) * theta * theta); };
    const T pref = model == 4 ? -k1 : -k1 * (mu(u) + mu(v)) / T(2), t = theta * (T(1) - T(3) * theta);
    const T pxx = -pref * (u * u * (u * u - T(1)) + t), pyy = pref * (v * v * (v * v - T(1)) + t);
    const T pxy = pref * u * v * (u * u - v * v);
    psi[1] += pyy / T(2), psi[3] += pyy / T(2), psi[2] += pxx / T(2), psi[4] += pxx / T(2);
    for (int i = 5; i < 9; ++i) psi[i] = -(pxx + pyy + T(CX[i] * CY[i]) * pxy) / T(4);
  }
  for (int i = 0; i < 9; ++i) {
    const T a = T(CX[i]) - u, b = T(CY[i]) - v, p = P(CX[i], u) * P(CY[i], v);
    out[i] = eq[i] + omp * (p * (k1 * (a * a - b * b) + k2 * a * b) + psi[i]);
  }
}

static bool collide_fixed(const double* f, const olbm::fx::Coefs& c, int model, double* out) {
  using namespace olbm::fx;
  Fx<60> a[9], o[9];
  bool ok = c.on != 0;
  for (int i = 0; i < 9; ++i) ok = ok && std::fabs(f[i]) < 1.0, a[i] = any_sign(f[i]);
  const Moments m = moments(a);
  Fx<60> ke2;
  ok = ok && moments_in_range(m.rho, m.jx, m.jy);
  if (!ok) return false;
  switch (model) {
    case 0: ok = collide<0>(m, a, c, o, ke2); break;
    case 1: ok = collide<1>(m, a, c, o, ke2); break;
    case 2: ok = collide<2>(m, a, c, o, ke2); break;
    case 3: ok = collide<3>(m, a, c, o, ke2); break;
    case 4: ok = collide<4>(m, a, c, o, ke2); break;
    default: ok = collide<5>(m, a, c, o, ke2); break;
  }
  out[0] = to_double(o[0]);
  for (int i = 1; i < 5; ++i) out[i] = to_double(Fx<61>{o[i].v});
  for (int i = 5; i < 9; ++i) out[i] = to_double(Fx<62>{o[i].v});
  return ok;
}

int main(int argc, char** argv) {
  const long n = argc > 1 ? atol(argv[1]) : 100000;
  std::mt19937_64 g(argc > 2 ? atol(argv[2]) : 1);
  const double theta = argc > 3 ? atof(argv[3]) : 1.0 / 3.0, tau = argc > 4 ? atof(argv[4]) : 0.51;
  const olbm::fx::Coefs c = olbm::fx::make_coefs(theta, tau);
  auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(g); };
  // families: 0 a flow near equilibrium, 1 random populations (spread 0.2), 2 the corners of the
  // range (density 1/2 .. 4, velocities to 1/2, large non-equilibrium), 3 a fluid at rest
  for (int model = 0; model < 6; ++model)
    for (int fam = 0; fam < 4; ++fam) {
      long taken = 0;
      double worst = 0, sq = 0, sq64 = 0, sqr = 0;
      for (long k = 0; k < n; ++k) {
        double f[9];
        const double rho = fam == 2 ? U(0.45, 4.1) : U(0.9, 1.1), m = fam == 2 ? 0.52 : fam == 3 ? 0.0 : 0.15;
        const double u = U(-m, m), v = U(-m, m), neq = fam == 2 ? U(0, 0.5) : fam == 3 ? 0.0 : fam == 1 ? 0.2 : 1e-3;
        for (int i = 0; i < 9; ++i) {
          const double px = CX[i] ? (theta + u * u + CX[i] * u) / 2 : 1 - theta - u * u;
          const double py = CY[i] ? (theta + v * v + CY[i] * v) / 2 : 1 - theta - v * v;
          f[i] = rho * (fam == 1 ? (CX[i] ? theta / 2 : 1 - theta) * (CY[i] ? theta / 2 : 1 - theta) : px * py) * (1 + neq * U(-1, 1));
        }
        double o[9];
        if (!collide_fixed(f, c, model, o)) continue;
        ++taken;
        real r[9];
        double d[9];
        collide_literal<real>(f, theta, tau, model, r);
        collide_literal<double>(f, theta, tau, model, d);
        for (int i = 0; i < 9; ++i) {
          const double e = (double)((real)o[i] - r[i]), e64 = (double)((real)d[i] - r[i]);
          const double v = std::fabs((double)r[i]);
          worst = std::max(worst, std::fabs(e) - 0.5 * std::ldexp(1.0, std::ilogb(v) - 52));
          const double er = (double)((real)(double)r[i] - r[i]);
          sq += e * e, sq64 += e64 * e64, sqr += er * er;
        }
      }
      const double unit = std::ldexp(1.0, 60), w = taken ? 1.0 / std::sqrt(9.0 * taken) : 0.0;
      printf("%d %d %ld %ld %.3f %.3f %.3f %.3f\n", model, fam, n, taken, worst * unit, std::sqrt(sq) * w * unit,
             std::sqrt(sq64) * w * unit, std::sqrt(sqr) * w * unit);
    }
  return 0;
}
