// lbm_fixed_adjoint.cuh -- the transposed Jacobian of one FP64 collision (Eq. 1a) in 64-bit
// fixed point and moment space (see lbm_fixed.cuh for the arithmetic, the moments
// M_pq of the collision and the reason for both; lbm_adjoint.cuh has the same derivative
// over populations).
//
// Given mu = dL/df*, the adjoints of the nine moments are the transposed inverse
// transform of mu (per axis M0~ = mu(0), 2 M1~ = mu(+1) - mu(-1), 2 M2~ = mu(+1) +
// mu(-1) - 2 mu(0)). With n = omega' N_xy and, at fixed M~,
//   a1 = M20~ + u_y M21~ + s_y M22~,  a2 = M02~ + u_x M12~ + s_x M22~,
//   Q = (X + t)(M20~ + M22~) - (Y + t)(M02~ + M22~) + W d M11~,   W = u_x u_y, d = u_y^2 - u_x^2
// the sums over the moments are
//   A1~ = (X + h) a1 - (Y + h) a2 + py s_x u_y M21~ + px s_y u_x M12~ + W d M11~ - Z Q,
//   n~  = M11~ + r_x (M21~ + r_y M22~) + r_y M12~        (r over theta),
//   rho~ (at fixed u) = M00~ + s_x a1 + s_y (M02~ + u_x M12~) + W M11~,
//   u_x~ = rho [2 u_x a1 + u_y M11~ + s_y M12~] + A1 dA1~/du_x + n r_x' (M21~ + r_y M22~)
// (u_y~ likewise), then D~ = k1 A1~, Pi~ = omega' n~ and, through u = j / rho without the
// product with rho and the one that undoes it,
//   j_x~ = M10~ + [2 u_x (a1 - D~) + u_y M11~ + s_y M12~ - u_y Pi~] + (1/rho)(A1 dA1~/du_x + ...).
// About 85 products, against about 210 FP64-pipe operations of the population form.
//
// Scale. mu is aligned to the largest of the node's nine (a power of two, taken
// out again in the results, so the derivative's linearity is exact): its largest magnitude
// lies in [2^-5, 2^-4) with 60 fraction bits, which leaves the sums a range of 2^7 over it.
// Products are rounded, not floored as in the collision: half a unit a product, always downwards,
// adds up over the steps and the lattice (384^2, 100 steps: velocity gradients off by 1.4e-14
// relative, 4.5e-15 rounded, binary64 4.7e-15), for 3 % of the time. (In the forward step the
// floors leave the fields as near to 64-bit arithmetic as binary64 and rounding costs 8 %.)
// A node whose collision or whose sums leave the formats' ranges takes the FP64 arithmetic.
#pragma once

#include "lbm_fixed.cuh"

namespace olbm {
namespace fx {

// Operands whose products are rounded to nearest: the addend of the first partial product.
template <int F> struct FxOpR {
  Op o;
};
template <int F> OLBM_EMU_HD FxOpR<F> rop(Fx<F> a) { return FxOpR<F>{digits(a.v)}; }
OLBM_EMU_HD i64 rounded_product(Op a, Op b) {
  const i64 c = wide(a.l, b.h, wide(a.h, b.l, (i64)1 << 31));
  return wide(a.h, b.h) + (i64)(int32_t)(c >> 32);
}
template <int F, int G> OLBM_EMU_HD Fx<F + G - 64> operator*(FxOpR<F> a, FxOpR<G> b) {
  return Fx<F + G - 64>{rounded_product(a.o, b.o)};
}
template <int F, int G> OLBM_EMU_HD Fx<F + G - 64> operator*(FxOpR<F> a, FxOp<G> b) {
  return Fx<F + G - 64>{rounded_product(a.o, b.o)};
}
template <int F> OLBM_EMU_HD Fx<2 * F - 64> square(FxOpR<F> a) {
  return Fx<2 * F - 64>{wide(a.o.h, a.o.h) + (wide(a.o.h, a.o.l, (i64)1 << 30) >> 31)};
}


template <int F> OLBM_EMU_HD Fx<F> twice(Fx<F> a) { return a + a; }

// m: the node's moments (in range); mu: the nine cotangents, below 2^-4; lam: those of the
// pulled populations. Returns whether every value stayed in its format.
template <int MODEL>
OLBM_EMU_HD bool collide_vjp(const Moments& m, const Fx<60> (&mu)[9], const Coefs& c, Fx<60> (&lam)[9]) {
  const auto ir = rop(reciprocal(m.rho));
  const FxOpR<64> ux = rop(to<64>(rop(to<62>(m.jx)) * ir)), uy = rop(to<64>(rop(to<62>(m.jy)) * ir));
  const Fx<64> ux2 = square(ux), uy2 = square(uy);
  const Fx<62> ux2h = to<62>(ux2), uy2h = to<62>(uy2);
  const auto sx = rop(c.theta + ux2h), sy = rop(c.theta + uy2h);
  // adjoints of the moments: over a, then over b (twice, four times: formats 61 and 62)
  Fx<60> al[3][3];  // [p][b + 1]
  const int I[3][3] = {{7, 3, 6}, {4, 0, 2}, {8, 1, 5}};  // population of velocity (a, b): [a + 1][b + 1]
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const Fx<60> lo = mu[I[0][b]], mid = mu[I[1][b]], hi = mu[I[2][b]];
    al[0][b] = mid, al[1][b] = hi - lo, al[2][b] = hi + lo - twice(mid);
  }
  auto B1 = [&](int p) { return al[p][2] - al[p][0]; };
  auto B2 = [&](int p) { return al[p][2] + al[p][0] - twice(al[p][1]); };
  const Fx<60> m00 = al[0][1];
  const Fx<61> m10{al[1][1].v}, m01{B1(0).v}, m20{al[2][1].v}, m02{B2(0).v};
  const Fx<62> m11{B1(1).v}, m21{B1(2).v}, m12{B2(1).v}, m22{B2(2).v};
  const auto M11 = rop(m11), M21 = rop(m21), M12 = rop(m12), M22 = rop(m22);
  const Fx<62> p12 = ux * M12, p21 = uy * M21, t11 = uy * M11, v11 = ux * M11;
  const Fx<60> r12 = sy * M12, r21 = sx * M21;
  const Fx<60> h20 = to<60>(m20), h02 = to<60>(m02);
  const Fx<60> a1 = h20 + to<60>(p21) + sy * M22;
  const Fx<60> b2 = h02 + to<60>(p12), a2 = b2 + sx * M22;
  const auto a1o = rop(to<62>(a1)), a2o = rop(to<62>(a2));
  Fx<60> rb = m00 + sx * a1o + sy * rop(to<62>(b2)) + to<60>(ux * rop(t11));
  Fx<60> Kx = to<60>(t11) + r12, Ky = to<60>(v11) + r21;  // + 2 u a below
  bool ok = true;
  if constexpr (MODEL == 0) {
    // f* = omega' f + (1 / tau) f^eq: the equilibrium's part times 1 / tau = 1 - omega'
    Kx = Kx + twice(ux * rop(a1)), Ky = Ky + twice(uy * rop(a2));
    rb = rb - (ux * rop(Kx) + uy * rop(Ky));
    const Fx<60> gx = to<60>(m10) + Kx, gy = to<60>(m01) + Ky;
    ok = within(rb.v, 1 << 29) & within(gx.v, 1 << 29) & within(gy.v, 1 << 29);
    auto eq = [&](Fx<60> x) { return x - rop(to<61>(x)) * c.omp; };
    const Fx<60> r = eq(rb), jx = eq(gx), jy = eq(gy);
    lam[0] = r, lam[1] = r + jx, lam[3] = r - jx, lam[2] = r + jy, lam[4] = r - jy;
    lam[5] = lam[1] + jy, lam[8] = lam[1] - jy, lam[6] = lam[3] + jy, lam[7] = lam[3] - jy;
#pragma unroll
    for (int i = 0; i < 9; ++i) lam[i] = lam[i] + rop(to<61>(mu[i])) * c.omp;
    return ok;
  } else {
    // non-equilibrium part of the collision: A1 and n
    const auto jxo = rop(m.jx);
    const Fx<60> E = m.D + (rop(m.jy) * uy - jxo * ux), N = m.Pxy - jxo * uy;
    ok = within(E.v, 1 << 27) & within(N.v, 1 << 27);
    const Fx<60> A1 = rop(to<64>(E)) * c.k1;
    ok = ok & within(A1.v, 1 << 28);
    const auto A1o = rop(to<62>(A1));
    const auto no = rop(rop(to<63>(N)) * c.omp);
    // polynomials of u
    const Fx<62> X = to<62>(square(rop(ux2))) - ux2h, Y = to<62>(square(rop(uy2))) - uy2h;
    const auto Xh = rop(X + c.h), Yh = rop(Y + c.h);
    const auto px = rop(c.c3 - ux2h), py = rop(uy2h - c.c3);
    const Fx<62> one{(i64)1 << 62};
    const auto dX = rop(twice(ux * rop(ux2h + ux2h - one))), dY = rop(twice(uy * rop(uy2h + uy2h - one)));
    const Fx<60> vx = c.v0 - rop(ux2) * c.inv_theta, vy = c.v0 - rop(uy2) * c.inv_theta;
    const auto rx = rop(to<62>(ux * rop(vx))), ry = rop(to<62>(uy * rop(vy)));
    const Fx<60> drx = vx + vx + vx - c.v0 - c.v0, dry = vy + vy + vy - c.v0 - c.v0;
    const Fx<62> d = uy2h - ux2h;
    const auto W = rop(ux * uy);
    // n~ and its velocity parts
    const Fx<60> e1 = to<60>(m21) + ry * M22, e2 = to<60>(m12) + rx * M22;
    const Fx<60> nb = to<60>(m11) + rx * rop(to<62>(e1)) + ry * M12;
    Fx<60> Lx = rop(to<64>(no * rop(to<62>(e1)))) * rop(drx), Ly = rop(to<64>(no * rop(to<62>(e2)))) * rop(dry);
    // A1~ and its derivatives with respect to u
    const Fx<60> f21 = sx * rop(p21), f12 = sy * rop(p12);
    Fx<60> Ab = Xh * a1o - Yh * a2o + py * rop(to<62>(f21)) + px * rop(to<62>(f12));
    Fx<60> Ax = px * rop(to<62>(r12)) + twice(ux * rop(py * rop(p21) - f12)) - Yh * rop(m12 + twice(ux * M22));
    Fx<60> Ay = py * rop(to<62>(r21)) + twice(uy * rop(f21 + px * rop(p12))) + Xh * rop(m21 + twice(uy * M22));
    Fx<60> gx = a1, gy = a2;  // factors of dX and -dY
    const Fx<60> Wd = rop(W * rop(d)) * M11;
    const Fx<60> Wx = rop(uy * rop(uy2h - ux2h - ux2h - ux2h)) * M11, Wy = rop(ux * rop(uy2h + uy2h + uy2h - ux2h)) * M11;
    if constexpr (MODEL <= 2) {
      Ab = Ab + Wd, Ax = Ax + Wx, Ay = Ay + Wy;
    } else {
      const Fx<60> h22 = to<60>(m22), sX = h20 + h22, sY = h02 + h22;
      const auto sXo = rop(to<62>(sX)), sYo = rop(to<62>(sY));
      const Fx<60> Q = rop(X + c.t) * sXo - rop(Y + c.t) * sYo + Wd;
      if constexpr (MODEL == 4) {  // Z = 1
        Ab = Ab + (Wd - Q);
        gx = gx - sX, gy = gy - sY;
      } else {
        ok = ok & within(Q.v, 1 << 28);
        const Fx<62> Zv = to<62>(rop(X + Y + c.h + c.h) * c.q2);
        const auto Z = rop(Zv), omz = rop(one - Zv);
        const Fx<60> qQ = to<60>(rop(to<63>(Q)) * c.q2);
        Ab = Ab + Wd - Z * rop(to<62>(Q));
        Ax = Ax + omz * rop(to<62>(Wx)), Ay = Ay + omz * rop(to<62>(Wy));
        gx = gx - qQ - Z * sXo, gy = gy + qQ - Z * sYo;
      }
    }
    ok = ok & within(gx.v, 1 << 29) & within(gy.v, 1 << 29);
    Ax = Ax + dX * rop(to<62>(gx)), Ay = Ay - dY * rop(to<62>(gy));
    if constexpr (MODEL == 1) {
      // M10 = j_x + A1 u_x (c3 - u_x^2), M01 = j_y + A1 u_y (u_y^2 - c3)
      const auto M10 = rop(to<62>(m10)), M01 = rop(to<62>(m01));
      const Fx<62> gx1 = ux * px, gy1 = uy * py;
      Ab = Ab + rop(gx1) * M10 + rop(gy1) * M01;
      Ax = Ax + rop(c.c3 - ux2h - ux2h - ux2h) * M10;
      Ay = Ay + rop(uy2h + uy2h + uy2h - c.c3) * M01;
    }
    ok = ok & within(Ab.v, 1 << 28) & within(Ax.v, 1 << 29) & within(Ay.v, 1 << 29) & within(nb.v, 1 << 29);
    Lx = Lx + A1o * rop(to<62>(Ax)), Ly = Ly + A1o * rop(to<62>(Ay));
    const Fx<60> Db = to<60>(rop(to<63>(Ab)) * c.k1), Pb = rop(to<61>(nb)) * c.omp;
    ok = ok & within(Lx.v, 1 << 28) & within(Ly.v, 1 << 28) & within(Db.v, 1 << 28) & within(Pb.v, 1 << 28);
    const auto Pbo = rop(Pb);
    const Fx<60> uyP = uy * Pbo, uxP = ux * Pbo;
    Kx = Kx + twice(ux * rop(a1 - Db)) - uyP + rop(to<62>(Lx)) * ir;
    Ky = Ky + twice(uy * rop(a2 + Db)) - uxP + rop(to<62>(Ly)) * ir;
    rb = rb + rop(d) * rop(to<62>(Db)) - ux * rop(uyP) - (ux * rop(Kx) + uy * rop(Ky));
    const Fx<60> jx = to<60>(m10) + Kx, jy = to<60>(m01) + Ky;
    ok = ok & within(rb.v, 1 << 29) & within(jx.v, 1 << 28) & within(jy.v, 1 << 28);
    const Fx<60> sp = rb + Db, sm = rb - Db;
    lam[0] = rb;
    lam[1] = sp + jx, lam[3] = sp - jx, lam[2] = sm + jy, lam[4] = sm - jy;
    const Fx<60> rp = rb + Pb, rm = rb - Pb, ju = jx + jy, jd = jx - jy;
    lam[5] = rp + ju, lam[7] = rp - ju, lam[8] = rm + jd, lam[6] = rm - jd;
    return ok;
  }
}

}  // namespace fx
}  // namespace olbm
