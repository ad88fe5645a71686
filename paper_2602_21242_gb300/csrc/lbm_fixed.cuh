// lbm_fixed.cuh -- the FP64 form's collision (Eq. 1a) in 64-bit fixed point, in
// moment space, on the integer pipes.
//
// What bounds it, and why this form. GB300's FP64 pipe retires two operations a
// clock per SM (an FP64 instruction holds a sub-partition for 64 cycles a warp),
// while a 64-bit integer addition takes 2 cycles a warp and a 32 x 32 -> 64-bit
// product 2 cycles on another pipe (measured: add.s64 1.97, mul.wide.s32 2.07,
// 64-bit shifts 3.8, FP64 add 71 cycles a warp at 1.93 GHz). The populations of a
// lattice Boltzmann node are numbers of order 1/100 to 1, so their binary64 values
// fit 64-bit fixed point with 60 fraction bits, and the whole collision runs there:
// sums are exact, products truncate at 2^-60 where binary64 rounds at 2^-53 of the
// operand, and only the nine stored populations are rounded to binary64 (once, to
// nearest even). Populations are taken exactly down to 2^-8 and truncated at 2^-60
// below that.
//
// Moment space. With m_0 = 1, m_1 = u, m_2 = s = theta + u^2 the moments of Eq. 10's
// per-axis factor P, those of P C are (0, theta, r), r = u (1 - theta - u^2), and
// those of P C^2 are (theta, u (1 - 2 theta - u^2), h + X + theta s), X = u^2 (u^2 - 1),
// h = theta (1 - theta) (exact identities: a^3 = a on the lattice). So the nine
// moments sum a^p b^q f*_(a,b), p, q = 0, 1, 2, of f* = f^eq + omega' (f^OReg + Psi)
// (Eqs. 2, 14, 15 with pref of Eq. 12) are
//   M00 = rho, M10 = j_x, M01 = j_y (with omega' psi for the uncorrected model)
//   M20 = rho theta + j_x u_x + A1 GX,  M02 = rho theta + j_y u_y - A1 GY,
//   M11 = j_x u_y + omega' N_xy + A1 GW,
//   M21 = (rho s_x) u_y + A1 G21 + omega' N_xy r_x / theta,
//   M12 = (rho s_y) u_x + A1 G12 + omega' N_xy r_y / theta,
//   M22 = (rho s_x) s_y + A1 G22 + omega' N_xy r_x r_y / theta^2
// with A1 = omega' K1 and polynomials of u alone
//   GX = X + h - Z (X + t), GY = Y + h - Z (Y + t), GW = (1 - Z) u_x u_y (u_y^2 - u_x^2),
//   G21 = u_y [X + h + s_x (u_y^2 - c3)], G12 = u_x [s_y (c3 - u_x^2) - (Y + h)],
//   G22 = (X + h) s_y - (Y + h) s_x - Z (X - Y),
// t = theta (1 - 3 theta), c3 = 1 - 3 theta, Z = (X + Y + 2 h) / (4 theta^2) for the
// complete model (Eq. 12), 1 with pref from f^neq, 0 for the uncorrected and partial
// models. The populations follow by additions alone: per axis f(0) = M0 - M2,
// 2 f(+-1) = M2 +- M1, the factors 1/2 taken into the final conversion. With A1 and the
// equilibrium parts taken into the common factors that leaves 36 products a node in
// place of the 58 (31 products and 27 of the 43 FMAs) of the population form.
//
// Range. A node takes this path when its populations are below 1 in magnitude, its
// density lies in [1/2, 4), its velocity components are below 1/2, its normal and
// shear non-equilibrium stresses below 1/2 and |A1| < 1, theta lies in
// [0.21, 0.65] and tau is at most 1e9; every other node (a blown-up state, another unit of density) goes to
// the floating-point collision. The choice depends on the node alone, so results do
// not depend on which nodes share a warp. The ranges below are those that the
// formats written as Fx<fraction bits> need; each value stays below 2^63 in its format.
//
// Error. Against 128-bit arithmetic one collision leaves a root mean square error of
// 8 units of 2^-60 in the populations (binary64: 42; the rounding of the stored values
// alone: 7), and 1000 steps of a decaying Taylor-Green vortex drift in mass by 7e-17
// (binary64: 1.1e-13, from the rounding of 1 - theta).
//
// Measured (GB300, 4096^2, complete model, diagnostics every step): 6.33 -> 34.0 GLUPS.
//
// The routines compile for the host as well, where tests compare them with
// extended-precision arithmetic.
#pragma once

#include <stdint.h>
#include <string.h>

#include "lbm_fp64emu.cuh"

namespace olbm {
namespace fx {

using i64 = int64_t;
using u64 = uint64_t;

// A multiplier operand: value = h 2^32 + l with l signed, so that every partial
// product is a signed 32 x 32 -> 64-bit product.
struct Op {
  int32_t h, l;
};

OLBM_EMU_HD Op digits(i64 v) {
  Op o;
  o.l = (int32_t)v;
  o.h = (int32_t)(v >> 32) + (int32_t)((uint32_t)v >> 31);  // one shift-and-add instruction
  return o;
}

// A value v 2^-F.
template <int F> struct Fx {
  i64 v;
  friend OLBM_EMU_HD Fx operator+(Fx a, Fx b) { return Fx{(i64)((u64)a.v + (u64)b.v)}; }
  friend OLBM_EMU_HD Fx operator-(Fx a, Fx b) { return Fx{(i64)((u64)a.v - (u64)b.v)}; }
  friend OLBM_EMU_HD Fx operator-(Fx a) { return Fx{(i64)(0 - (u64)a.v)}; }
};
// Digits of a value with F fraction bits, and of a coefficient (split on the host).
template <int F> struct FxOp {
  Op o;
};
template <int F> OLBM_EMU_HD FxOp<F> op(Fx<F> a) { return FxOp<F>{digits(a.v)}; }
// The same value with G fraction bits (a shift).
template <int G, int F> OLBM_EMU_HD Fx<G> to(Fx<F> a) {
  if constexpr (G >= F)
    return Fx<G>{(i64)((u64)a.v << (G - F))};
  else
    return Fx<G>{a.v >> (F - G)};
}

// 32 x 32 -> 64-bit product (+ c). On the device as the instruction: from C++ the
// compiler builds it out of more (28.7 cycles a warp for the product below against 14.1).
OLBM_EMU_HD i64 wide(int32_t a, int32_t b) {
#if defined(__CUDA_ARCH__)
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (i64)a * b;
#endif
}
OLBM_EMU_HD i64 wide(int32_t a, int32_t b, i64 c) {
#if defined(__CUDA_ARCH__)
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}
OLBM_EMU_HD u64 uwide(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  u64 r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (u64)a * b;
#endif
}

// The high 64 bits of the product: a.h b.h + floor((a.h b.l + a.l b.h) / 2^32). The
// dropped a.l b.l is at most a quarter unit of the result; the floor is one unit.
template <int F, int G> OLBM_EMU_HD Fx<F + G - 64> operator*(FxOp<F> a, FxOp<G> b) {
  const i64 c = wide(a.o.l, b.o.h, wide(a.o.h, b.o.l));
  return Fx<F + G - 64>{wide(a.o.h, b.o.h) + (i64)(int32_t)(c >> 32)};
}
template <int F> OLBM_EMU_HD Fx<2 * F - 64> square(FxOp<F> a) {
  return Fx<2 * F - 64>{wide(a.o.h, a.o.h) + (wide(a.o.h, a.o.l) >> 31)};
}

// Coefficients of one lattice (theta, tau), set on the host.
struct Coefs {
  FxOp<60> k1;         // omega' / (4 theta^2)
  FxOp<63> theta_op;   // theta
  FxOp<63> omp;        // omega'
  FxOp<60> q2;         // 1 / (4 theta^2)
  FxOp<60> inv_theta;  // 1 / theta
  FxOp<61> e2;         // (1 - theta) / (2 theta) (polynomial equilibrium)
  Fx<62> theta, h, t, c3;
  Fx<60> v0;           // (1 - theta) / theta
  Fx<60> theta2;       // theta^2
  int on;              // theta in the range of the formats
};

// A sum h + l of two binary64, |l| at most half an ulp of h: about 104 bits, for the
// coefficients, which no rounding to binary64 shall touch on their way. (Not long double: on Arm
// that is software, 0.67 us for the coefficients of one launch (0.09 so) where the launch of a small
// lattice takes 4.5 us of host time; on x86 it has 64 bits.) Products are written
// as fma(a, b, 0) so that the compiler contracts none of them with an addition.
struct Wide {
  double h, l;
};
inline Wide wide_sum(double a, double b) {  // exact
  const double s = a + b, z = s - a;
  return Wide{s, (a - (s - z)) + (b - z)};
}
inline Wide operator+(Wide a, Wide b) {
  const Wide s = wide_sum(a.h, b.h);
  return wide_sum(s.h, s.l + (a.l + b.l));
}
inline Wide operator-(Wide a, Wide b) { return a + Wide{-b.h, -b.l}; }
inline Wide operator*(Wide a, Wide b) {
  const double p = __builtin_fma(a.h, b.h, 0.0);
  return wide_sum(p, __builtin_fma(a.h, b.h, -p) + __builtin_fma(a.h, b.l, __builtin_fma(a.l, b.h, 0.0)));
}
inline Wide operator/(Wide a, Wide b) {  // two corrections of the quotient of the leading parts
  const double q = a.h / b.h;
  const Wide r = a - b * Wide{q, 0.0};
  const double q1 = r.h / b.h;
  const Wide r1 = r - b * Wide{q1, 0.0};
  return wide_sum(q, q1) + Wide{r1.h / b.h, 0.0};
}

// x to the nearest 2^-F, |x| < 2^(63 - F).
template <int F> inline Fx<F> fx_of(Wide x) {
  const double scale = (double)(1ull << (F - 30)) * (double)(1ull << 30);  // 2^F: exact products
  const double t = __builtin_fma(x.h, scale, 0.0);
  const i64 h = (i64)__builtin_llrint(t);
  return Fx<F>{h + (i64)__builtin_llrint((t - (double)h) + __builtin_fma(x.l, scale, 0.0))};
}

inline Coefs make_coefs(double theta, double tau) {
  Coefs c;
  memset(&c, 0, sizeof c);
  c.on = theta >= 0.21 && theta <= 0.65 && tau <= 1e9 ? 1 : 0;  // omega' < 1 with 63 fraction bits
  if (!c.on) return c;
  const Wide one{1.0, 0.0}, two{2.0, 0.0}, three{3.0, 0.0}, four{4.0, 0.0}, th{theta, 0.0};
  const Wide omp = one - one / Wide{tau, 0.0}, th2 = th * th, rest = one - th, c3 = one - three * th;
  const Wide inv = one / th, q2 = one / (four * th2);
  c.k1 = op(fx_of<60>(omp * q2));
  c.theta_op = op(fx_of<63>(th));
  c.omp = op(fx_of<63>(omp));
  c.q2 = op(fx_of<60>(q2));
  c.inv_theta = op(fx_of<60>(inv));
  c.e2 = op(fx_of<61>(rest * inv / two));
  c.theta = fx_of<62>(th);
  c.h = fx_of<62>(th * rest);
  c.t = fx_of<62>(th * c3);
  c.c3 = fx_of<62>(c3);
  c.v0 = fx_of<60>(rest * inv);
  c.theta2 = fx_of<60>(th2);
  return c;
}

// ---------------------------------------------------------------- binary64 <-> fixed point
OLBM_EMU_HD u64 shr64(u64 v, uint32_t s) {
#if defined(__CUDA_ARCH__)
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));  // clamps: 64 and more give 0
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}

// |x| truncated to F fraction bits, |x| < 2^(63 - F); zeros and subnormals give 0.
template <int F = 60> OLBM_EMU_HD Fx<F> magnitude(double x) {
  const u64 u = emu::bits_of(x);
  const uint32_t e = (uint32_t)(u >> 52) & 0x7FFu;
  return Fx<F>{(i64)shr64((u << 11) | emu::kSign, (uint32_t)(1086 - F) - e)};
}
OLBM_EMU_HD Fx<60> nonnegative(double x) {  // x >= +0
  const u64 u = emu::bits_of(x);
  return Fx<60>{(i64)shr64((u << 11) | emu::kSign, 1026u - (uint32_t)(u >> 52))};
}
template <int F = 60> OLBM_EMU_HD Fx<F> any_sign(double x) {
  const Fx<F> m = magnitude<F>(x);
  return (emu::bits_of(x) & emu::kSign) ? -m : m;
}

// v 2^-F rounded to binary64 (to nearest, ties to even); |v| < 2^62.
// Device: v = a 2^44 + b, b its low 44 bits. b + 2^52 (in units of 2^-F) is a binary64
// with b in its low mantissa bits; a - 2^8 has at most 20 bits, so its FP32
// conversion is exact and widens by moving its exponent field; one FP64 addition
// rounds their sum once.
OLBM_EMU_HD double to_double(i64 v, int F) {
#if defined(__CUDA_ARCH__)
  const int32_t vh = (int32_t)(v >> 32);
  const uint32_t vl = (uint32_t)v;
  const int32_t a = (vh >> 12) - 256;
  const int32_t fb = __float_as_int(__int2float_rn(a));
  const uint32_t hh = ((uint32_t)(fb >> 3) & 0x8FFFFFFFu) + ((uint32_t)(896 + 44 - F) << 20);
  const double hi = __hiloint2double((int)hh, fb << 29);
  const double lo = __hiloint2double((int)(((uint32_t)vh & 0xFFFu) | ((uint32_t)(1075 - F) << 20)), (int)vl);
  return hi + lo;
#else
  return __builtin_ldexp((double)v, -F);
#endif
}
template <int F> OLBM_EMU_HD double to_double(Fx<F> x) { return to_double(x.v, F); }

// v 2^-F rounded to FP32 (to nearest). safe is cleared where v lies within 2^-50 of the
// midpoint of two FP32 numbers (or is so small that this cannot be told): there a
// result computed with an error below 2^-50 may round the other way.
template <int F> OLBM_EMU_HD float to_float(Fx<F> x, bool& safe) {
  const bool neg = x.v < 0;
  const u64 a = neg ? 0 - (u64)x.v : (u64)x.v;
  const uint32_t ah = (uint32_t)(a >> 32);
  const int t = 31 - emu::clz32(ah | 1u);  // top bit of the high word
  const u64 m = a << (31 - t);             // leading bit at 63
  const uint32_t mh = (uint32_t)(m >> 32), rem = ((mh & 0xFFu) << 8) | ((uint32_t)m >> 24);
  const uint32_t off = rem - 0x8000u, dist = rem >= 0x8000u ? off : 0u - off;
  safe = safe & (ah >> 1 != 0) & (dist > ((1u << (F - 43)) >> t) + 1u);
  const uint32_t bits = ((uint32_t)(127 + t + 32 - F - 1) << 23) + (mh >> 8) + (rem >> 15);
  union {
    uint32_t u;
    float f;
  } r;
  r.u = bits | (neg ? 0x80000000u : 0u);
  return r.f;
}

// ---------------------------------------------------------------- 1 / rho
// rho in [1/2, 4) with 60 fraction bits -> 1/rho with 62: a seed of 21 fraction
// bits from the FP32 reciprocal, its residual e = 1 - rho seed exactly (modulo
// 2^64 in units of 2^-81, where |e| < 2^-19 fits), and seed (1 + e + e^2). The seed's
// rounding to 2^-21 leaves |e| below 2^-20 at rho = 4 (2^-21.7 at rho = 1), so the
// dropped e^3 is a relative error of 2^-60 (2^-65).
OLBM_EMU_HD float seed_recip(float x) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
OLBM_EMU_HD Fx<62> reciprocal(Fx<60> rho) {
  const uint32_t rl = (uint32_t)rho.v;
  const int32_t rh = (int32_t)(rho.v >> 32);
  const float s = seed_recip((float)rh);  // 2^-28 / rho
  union {
    float f;
    uint32_t u;
  } m;
  m.f = s * 268435456.0f + 4.0f;                     // in [4.25, 6]: 21 fraction bits left
  const uint32_t R = m.u - 0x40800000u;              // seed 2^21
  const u64 p = uwide(rl, R) + ((u64)((uint32_t)rh * R) << 32);  // rho seed, units of 2^-81, modulo 2^64
  const i64 e = (i64)(0 - p);                        // 2^81 = 0 modulo 2^64
  const int32_t eh = (int32_t)(e >> 32);             // units of 2^-49
  const i64 q = e + (wide(eh, eh) >> 17);            // e + e^2
  const i64 c = wide((int32_t)(q >> 32), (int32_t)R) + (i64)(uwide((uint32_t)q, R) >> 32);  // seed q, units of 2^-70
  return Fx<62>{(i64)((u64)R << 41) + (c >> 8)};
}

// ---------------------------------------------------------------- one node
// Populations from the nine moments sum a^p b^q f_(a,b): out[0] as it is, out[1..4]
// twice, out[5..8] four times the population (Fig. 1a order).
struct MomentSet {
  Fx<60> M00, M10, M01, M20, M02, M11, M21, M12, M22;
};
OLBM_EMU_HD void populations(const MomentSet& M, Fx<60> (&out)[9]) {
  const Fx<60> a0 = M.M00 - M.M20, a1 = M.M01 - M.M21, a2 = M.M02 - M.M22;  // column a = 0: b moments
  const Fx<60> p0 = M.M20 + M.M10, q0 = M.M20 - M.M10;                      // columns a = +1, -1, doubled
  const Fx<60> p1 = M.M21 + M.M11, q1 = M.M21 - M.M11, p2 = M.M22 + M.M12, q2 = M.M22 - M.M12;
  out[0] = a0 - a2;
  out[2] = a2 + a1, out[4] = a2 - a1;
  out[1] = p0 - p2, out[3] = q0 - q2;
  out[5] = p2 + p1, out[8] = p2 - p1, out[6] = q2 + q1, out[7] = q2 - q1;
}

// The guided equilibrium (Eq. 10) of one node, less the rest state of unit density if
// SHIFT: rho in (0, 4), |u| < 1/2; out scaled as by populations().
template <bool SHIFT>
OLBM_EMU_HD void equilibrium(Fx<60> rho, Fx<64> u, Fx<64> v, const Coefs& c, Fx<60> (&out)[9]) {
  const FxOp<60> ro = op(rho);
  const FxOp<64> ux = op(u), uy = op(v);
  const Fx<60> jx = ro * ux, jy = ro * uy;
  const auto jxo = op(jx);
  const Fx<60> rt = op(to<61>(rho)) * c.theta_op;
  const Fx<60> rsx = rt + jxo * ux, rsy = rt + op(jy) * uy;
  MomentSet M;
  M.M00 = rho, M.M10 = jx, M.M01 = jy, M.M20 = rsx, M.M02 = rsy, M.M11 = jxo * uy;
  M.M21 = op(rsx) * uy, M.M12 = op(rsy) * ux;
  M.M22 = to<60>(op(to<61>(rsx)) * op(c.theta + to<62>(square(uy))));
  if constexpr (SHIFT) {  // the rest state's moments: 1, theta, theta, theta^2
    const Fx<60> th = to<60>(c.theta);
    M.M00 = M.M00 - Fx<60>{(i64)1 << 60}, M.M20 = M.M20 - th, M.M02 = M.M02 - th, M.M22 = M.M22 - c.theta2;
  }
  populations(M, out);
}

OLBM_EMU_HD bool within(i64 v, int32_t bound) {  // |v's high word| < bound (slightly inside)
  return (uint32_t)((int32_t)(v >> 32) + (bound - 1)) < (uint32_t)(2 * bound - 2);
}

// rho in (1/2, 4) and |j_a| < rho / 2, by the high words (with |f_i| < 1 every |j_a| < 6, so
// none of these 32-bit sums wraps into the accepted range).
OLBM_EMU_HD bool moments_in_range(Fx<60> rho, Fx<60> jx, Fx<60> jy) {
  const uint32_t rh = (uint32_t)(rho.v >> 32), jxh = (uint32_t)(jx.v >> 32), jyh = (uint32_t)(jy.v >> 32);
  const uint32_t half = (rh >> 1) - 2u, lo = (1u << 27) + 1024u;
  return (rh - lo < (1u << 30) - lo) & (jxh + half < 2u * half) & (jyh + half < 2u * half);
}

// Moments of the pulled populations (60 fraction bits, Fig. 1a order).
struct Moments {
  Fx<60> rho, jx, jy, D, Pxy;  // D = sum (c_x^2 - c_y^2) f, Pxy = sum c_x c_y f
};
OLBM_EMU_HD Moments moments(const Fx<60> (&f)[9]) {
  Moments m;
  const auto s13 = f[1] + f[3], d13 = f[1] - f[3], s24 = f[2] + f[4], d24 = f[2] - f[4];
  const auto s57 = f[5] + f[7], d57 = f[5] - f[7], s68 = f[6] + f[8], d68 = f[6] - f[8];
  m.rho = f[0] + (s13 + s24) + (s57 + s68);
  m.jx = d13 + (d57 - d68), m.jy = d24 + (d57 + d68);
  m.D = s13 - s24, m.Pxy = s57 - s68;
  return m;
}

// m: the node's moments (in range); f: its populations (read by the LBGK models only);
// out, the post-collision populations: out[0] as they are, out[1..4] as twice their value,
// out[5..8] as four times. Returns whether the non-equilibrium part is in range; ke2
// receives j.u, twice the kinetic energy.
template <int MODEL>
OLBM_EMU_HD bool collide(const Moments& m, const Fx<60> (&f)[9], const Coefs& c, Fx<60> (&out)[9], Fx<60>& ke2) {
  const Fx<60> rho = m.rho, jx = m.jx, jy = m.jy;
  bool ok = true;
  const auto ir = op(reciprocal(rho));
  const FxOp<64> ux = op(to<64>(op(to<62>(jx)) * ir)), uy = op(to<64>(op(to<62>(jy)) * ir));
  const Fx<64> ux2 = square(ux), uy2 = square(uy);
  const auto jxo = op(jx), jyo = op(jy);
  const Fx<60> jux = jxo * ux, juy = jyo * uy, jxuy = jxo * uy;
  ke2 = jux + juy;
  const Fx<60> rt = op(to<61>(rho)) * c.theta_op;  // rho theta
  const Fx<60> rsx = rt + jux, rsy = rt + juy;     // rho s_x, rho s_y
  Fx<60> M10 = jx, M01 = jy, M20, M02, M11, M21, M12, M22;
  if constexpr (MODEL == 0) {
    M20 = rsx, M02 = rsy, M11 = jxuy;
    M21 = op(rsx) * uy, M12 = op(rsy) * ux;
    M22 = to<60>(op(to<61>(rsx)) * op(c.theta + to<62>(uy2)));
  } else if constexpr (MODEL == 5) {
    // polynomial equilibrium: rho (theta + u_a^2 (1 - theta)/(2 theta)), rho theta u, and
    // rho (theta^2 + |u|^2 (1 - theta)/2)
    const Fx<60> a = op(to<63>(jux)) * c.e2, b = op(to<63>(juy)) * c.e2;
    M20 = rt + a, M02 = rt + b, M11 = jxuy;
    M21 = op(to<61>(jy)) * c.theta_op, M12 = op(to<61>(jx)) * c.theta_op;
    M22 = op(to<61>(rt + a + b)) * c.theta_op;
  } else {
    const Fx<60> E = m.D + (juy - jux), N = m.Pxy - jxuy;  // 2 N_d, N_xy
    ok = within(E.v, 1 << 27) & within(N.v, 1 << 27);
    const Fx<60> A1 = op(to<64>(E)) * c.k1;  // |k1| <= 5.7, |E| < 1/2
    ok = ok & within(A1.v, 1 << 28);
    const FxOp<62> A1o = op(to<62>(A1));
    const Fx<62> ux2h = to<62>(ux2), uy2h = to<62>(uy2);
    const Fx<62> X = to<62>(square(op(ux2))) - ux2h, Y = to<62>(square(op(uy2))) - uy2h;  // u^2 (u^2 - 1)
    const auto sx = op(c.theta + ux2h), sy = op(c.theta + uy2h);
    const Fx<60> TX = A1o * op(X + c.h), TY = A1o * op(Y + c.h);
    const Fx<60> Ax = A1o * op(c.c3 - ux2h), Ay = A1o * op(uy2h - c.c3);
    // shear part: omega' N_xy and its products with r_x / theta, r_y / theta
    const Fx<62> nw = op(to<63>(N)) * c.omp;
    const auto nwo = op(nw);
    const Fx<60> vx = c.v0 - op(ux2) * c.inv_theta, vy = c.v0 - op(uy2) * c.inv_theta;
    const auto rx = op(to<62>(ux * op(vx))), ry = op(to<62>(uy * op(vy)));
    const Fx<60> nrx = nwo * rx, nry = nwo * ry;
    const Fx<60> T20 = rsx + TX, T02 = rsy - TY;  // T20 < 4
    M21 = uy * op(T20 + sx * op(to<62>(Ay))) + nrx;
    M12 = ux * op(T02 + sy * op(to<62>(Ax))) + nry;
    M22 = to<60>(op(to<61>(T20)) * sy - op(to<61>(TY)) * sx) + op(to<62>(nrx)) * ry;
    M11 = jxuy + to<60>(nw);
    if constexpr (MODEL == 1 || MODEL == 2) {
      M20 = T20, M02 = T02;
      M11 = M11 + A1o * op(op(ux * uy) * op(uy2h - ux2h));
    } else if constexpr (MODEL == 4) {  // Z = 1: A1 (X + t), A1 (Y + t) from A1 (h - t) = 2 theta^2 A1
      const Fx<60> w = A1o * op(c.h - c.t);
      M20 = rsx + w, M02 = rsy - w;
      M22 = M22 - (TX - TY);
    } else {
      const Fx<60> AZ = op(to<64>(TX + TY)) * c.q2;
      const auto AZo = op(to<62>(AZ));
      const Fx<60> ZX = AZo * op(X + c.t), ZY = AZo * op(Y + c.t);
      M20 = T20 - ZX, M02 = T02 + ZY;
      M22 = M22 - (ZX - ZY);
      M11 = M11 + op(to<62>(A1 - AZ)) * op(op(ux * uy) * op(uy2h - ux2h));
    }
    if constexpr (MODEL == 1) {  // omega' psi
      M10 = M10 + ux * op(Ax);
      M01 = M01 + uy * op(Ay);
    }
  }
  populations(MomentSet{rho, M10, M01, M20, M02, M11, M21, M12, M22}, out);
  if constexpr (MODEL == 0 || MODEL == 5) {
    // f* = f^eq + omega' (f - f^eq), in the scaling of out
    out[0] = out[0] + op(to<61>(f[0] - out[0])) * c.omp;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const Fx<60> g{(i64)((u64)f[i].v << (i < 5 ? 1 : 2))};
      out[i] = out[i] + to<60>(op(g - out[i]) * c.omp);
    }
  }
  return ok;
}

}  // namespace fx
}  // namespace olbm
