// fvna_face64.cuh -- the binary64 interface solver, limited flux and cell
// update shared by the 2D and 3D sweeps (arXiv 1311.3004, section 3.2, eqs.
// fv-hr, fluc:m, fluc:p, limiter), for NT = 1 or 2 transverse momenta.
//
// Two forms of each, with the same results bit for bit (a zero's sign aside):
//   *_general  every formula in the order of its definition on the binary64
//              unit (the including units are compiled with -fmad=false; a sum
//              is the fused multiply-add x 1 + y, a product x y + (-0), which
//              round alike and are taken faster, see below).  2048 x 2048 cells
//              wholly in this form (beta 6.3): x1 and x2 sweep 1.92 and 1.84 ms;
//              2.35 and 2.14 with plain operations, a 0/0 a warp and no
//              subsonic form; 1.76 and 2.23 in the kernels before these;
//   *_fast     the same roundings with fewer instructions on that unit:
//              reciprocals, quotients, roots and the products of the solver
//              and of the limiter's sums run in integer arithmetic
//              (fvna_int64f.cuh), comparisons and powers of two as integer
//              operations on the bit patterns.
// What bounds these sweeps is the binary64 unit (16 cycles a warp instruction
// per SM).  A cell of a 2D sweep sent it 214 instructions in general form, 8
// of ten cycles of the sweep; the fast form sends 91, and its 2,200 integer
// instructions run beside them.  Measured, x1 sweep of 2048 x 2048 cells: 2.06
// ms before, 0.78 now; x2 sweep with the source 2.56 and 1.03.  Which products
// go to the integer pipes was found by trying: all of them (67 left on the
// unit) 0.81 ms, none 0.97, those of the solver and the limiter's sums 0.78.
//
// Exact shortcuts of the fast form: halves are moved through products and
// sums, which is exact while nothing is subnormal (S = 2 Z: u = S rcp(S1),
// 2 Z2 = S2, Phi = 1 + (beta2/2)(S1 - 2), flux sums G = 2 F with dt/dx
// halved instead); s1 W2 = W2 s1 is the product the wave already holds; a sum
// is the fused multiply-add x 1 + y and a product x y + (-0), which round
// once like the plain ones and are taken 16 % faster (16.1 against 19.1
// cycles, measured).
//
// The fast form needs q1 within 1/16 of 1, momenta below 2^-4, |beta2| zero or
// in [2^-40, 8] and dt/dx in [2^-40, 2): then c is in (0.69, 1.3) and every
// interface is subsonic.  Integer products and the moved halves are used
// (SOFT) while momenta are zero or at least 2^-400; with smaller ones the
// products and halves are taken on the unit as defined (FAST).  Following the
// smallest nonzero values through from there (a difference of two numbers is
// zero or at least a unit in the last place of the smaller): z 2^-401, sums of
// z and u 2^-455, r13 2^-458, a1 and a2 2^-454, w0 and w1 2^-912.  So every
// factor pair given to mulz is zero or has exponent fields that add up to
// 1034 or more, with two exceptions that do no harm: u u and S2 u, and the
// transverse terms of the acoustic families' dot products, come out as zero
// when they are below 2^-1012, where they are below 2^-54 of the sum they
// join (1, and a1^2 or a1 U.a1, which is 2^-908 or more; the terms of
// that sum have one sign).  The transverse family's own two products stay on
// the unit.  A limiter value below 2^-100 or a transverse flux sum below
// 2^-900 (but not zero) could make the halved sums subnormal: the update then
// takes the general form.
//
// A pulse in a medium at rest sends a precursor of ever smaller momenta ahead
// of itself, a cell a step, down to the subnormals.  One cell in a hundred
// of the 2048^2 pulse is in it, but a marched tile that takes the general form
// there is the slowest of its sweep: with that form below 2^-900 the x2 sweep
// took 1.4 to 1.9 ms instead of 1.0.
#pragma once

#include "fvna_int64f.cuh"

namespace fvna {
namespace f64 {

using int64f::hi_of;
using int64f::mulz;

enum { F64_MC = 0, F64_NONE = 1, F64_LW = 2 };   // the limiter kinds

// 1.0 and -0.0, read from memory so that the compiler cannot see them and
// turn the fused forms back into adds and multiplies
static __device__ double g_unit[2] = {1.0, -0.0};
struct Unit {
  double one, nz;
  __device__ __forceinline__ void load() {
    one = *(volatile double *)&g_unit[0];
    nz = *(volatile double *)&g_unit[1];
  }
  __device__ __forceinline__ double add(double x, double y) const { return __fma_rn(x, one, y); }
  __device__ __forceinline__ double sub(double x, double y) const { return __fma_rn(x, one, -y); }
  __device__ __forceinline__ double mul(double x, double y) const { return __fma_rn(x, y, nz); }
};

// Constants of a sweep.
struct Par {
  Unit U;
  double beta2, bh, lam, hlam;   // 2 (beta - 1), half of it, dt/dx, half of it
  bool ok;                       // the constants allow the fast form
  __device__ __forceinline__ void set(double beta2_, double lam_) {
    U.load();
    beta2 = beta2_;
    bh = 0.5 * beta2_;
    lam = lam_;
    hlam = 0.5 * lam_;
    const double b = fabs(beta2_);
    ok = (b == 0.0 || (b >= 0x1p-40 && b <= 8.0)) && lam_ >= 0x1p-40 && lam_ < 2.0;
  }
};

// The form a cell's values allow: GENERAL any, FAST, SOFT (see above).
enum { GENERAL = 0, FAST = 1, SOFT = 2 };
template <int NT> __device__ __forceinline__ int form_of(const double q[2 + NT]) {
  unsigned lo = 0x3fa00000u, hi = 0;
#pragma unroll
  for (int k = 1; k < 2 + NT; k++) {
    const unsigned h = hi_of(q[k]) & 0x7fffffffu;
    hi = h > hi ? h : hi;
    lo = h < lo && (int64f::bits_of(q[k]) << 1) != 0 ? h : lo;
  }
  if (hi_of(q[0]) - 0x3fee0000u >= 0x3ff10000u - 0x3fee0000u || hi >= 0x3fb00000u) return GENERAL;
  return lo >= 0x26f00000u ? SOFT : FAST;
}
// the form all lanes allow
__device__ __forceinline__ int warp_form(int f) { return (int)__reduce_min_sync(0xffffffffu, (unsigned)f); }
// a product on the integer pipes (SOFT) or on the unit
template <int FORM> __device__ __forceinline__ double prod(const Unit &U, double x, double y) {
  return FORM == SOFT ? mulz(x, y) : U.mul(x, y);
}

// One interface: speeds, and the waves of the two acoustic families
// (a, a s, a r_k) and of the transverse ones (one component each).
template <int NT> struct Face {
  double s0, s1, u;
  double a1, w01, w0[NT];
  double a2, w11, w1[NT];
  double w2[NT];
};
// Flux data of an interface; G is twice the correction flux of eq. limiter.
template <int NT> struct Flux {
  double am[2 + NT], ap[2 + NT], G[2 + NT];
};

// velocities z = (normal, transverse) / q1
template <int NT>
__device__ __forceinline__ void z_general(const Unit &U, const double q[2 + NT], double z[1 + NT]) {
  const double r = 1.0 / q[0];
#pragma unroll
  for (int k = 0; k < 1 + NT; k++) z[k] = U.mul(q[1 + k], r);
}
template <int NT> __device__ __forceinline__ void z_fast(const Par &P, const double q[2 + NT], double z[1 + NT]) {
  const double r = int64f::rcp_mid(q[0]);
#pragma unroll
  for (int k = 0; k < 1 + NT; k++) z[k] = P.U.mul(q[1 + k], r);
}

// Roe solver (section 3.2) of cells L and R; true if the radicand is negative.
template <int NT>
__device__ __forceinline__ bool face_general(const Par &P, const double L[2 + NT],
                                             const double zL[1 + NT], const double R[2 + NT],
                                             const double zR[1 + NT], Face<NT> &F) {
  const Unit &U = P.U;
  const double Z1 = U.mul(0.5, U.add(L[0], R[0]));
  const double Z2 = U.mul(0.5, U.add(zL[0], zR[0]));
  const double Phi = U.add(U.mul(P.beta2, U.add(Z1, -1.0)), 1.0);
  const double rZ1 = 1.0 / Z1;
  const double u = U.mul(Z2, rZ1);
  const double T2 = U.add(Z2, Z2);
  const double D = U.add(U.sub(U.mul(u, u), U.mul(T2, u)), Phi);
  const bool nonreal = D < 0.0;
  const double c = sqrt(D);
  F.s0 = U.add(u, c);
  F.s1 = U.sub(u, c);
  F.u = u;
  const double rc = 1.0 / c;
  const double h = U.mul(0.5, rc);
  const double d1 = U.sub(R[0], L[0]);
  const double d2 = U.sub(R[1], L[1]);
  F.a1 = U.mul(U.sub(d2, U.mul(F.s1, d1)), h);
  F.a2 = U.mul(U.sub(U.mul(F.s0, d1), d2), h);
  F.w01 = U.mul(F.a1, F.s0);
  F.w11 = U.mul(F.a2, F.s1);
#pragma unroll
  for (int k = 0; k < NT; k++) {
    const double v = U.mul(U.mul(0.5, U.add(zL[1 + k], zR[1 + k])), rZ1);
    const double r1 = U.mul(U.mul(v, U.sub(F.s0, T2)), rc);
    const double r2 = U.mul(U.mul(v, U.sub(T2, F.s1)), rc);
    F.w0[k] = U.mul(F.a1, r1);
    F.w1[k] = U.mul(F.a2, r2);
    F.w2[k] = U.sub(U.sub(U.sub(R[2 + k], L[2 + k]), F.w0[k]), F.w1[k]);
  }
  return nonreal;
}

template <int FORM, int NT>
__device__ __forceinline__ void face_fast(const Par &P, const double L[2 + NT],
                                          const double zL[1 + NT], const double R[2 + NT],
                                          const double zR[1 + NT], Face<NT> &F) {
  const Unit &U = P.U;
  const double S1 = U.add(L[0], R[0]);
  const double S2 = U.add(zL[0], zR[0]);
  const double Phi = U.add(prod<FORM>(U, P.bh, U.add(S1, -2.0)), 1.0);
  // 1/S1 with the halves moved out (SOFT), or 1/Z1 and the halves taken as defined
  const double rs = FORM == SOFT ? int64f::rcp_mid(S1) : int64f::twice(int64f::rcp_mid(S1));
  const double Z2 = FORM == SOFT ? S2 : U.mul(0.5, S2);
  const double T2 = FORM == SOFT ? S2 : U.add(Z2, Z2);
  const double u = prod<FORM>(U, Z2, rs);
  const double D = U.add(U.sub(prod<FORM>(U, u, u), prod<FORM>(U, T2, u)), Phi);
  const double c = int64f::sqrt_mid(D);
  F.s0 = U.add(u, c);
  F.s1 = U.sub(u, c);
  F.u = u;
  const double rc = int64f::rcp_mid(c);
  const double h = int64f::half_of(rc);
  const double d1 = U.sub(R[0], L[0]);
  const double d2 = U.sub(R[1], L[1]);
  const double e0 = U.sub(F.s0, T2), e1 = U.sub(T2, F.s1);
  F.a1 = prod<FORM>(U, U.sub(d2, prod<FORM>(U, F.s1, d1)), h);
  F.a2 = prod<FORM>(U, U.sub(prod<FORM>(U, F.s0, d1), d2), h);
  F.w01 = prod<FORM>(U, F.a1, F.s0);
  F.w11 = prod<FORM>(U, F.a2, F.s1);
#pragma unroll
  for (int k = 0; k < NT; k++) {
    const double S = U.add(zL[1 + k], zR[1 + k]);
    const double v = prod<FORM>(U, FORM == SOFT ? S : U.mul(0.5, S), rs);
    const double r1 = prod<FORM>(U, prod<FORM>(U, v, e0), rc);
    const double r2 = prod<FORM>(U, prod<FORM>(U, v, e1), rc);
    F.w0[k] = prod<FORM>(U, F.a1, r1);
    F.w1[k] = prod<FORM>(U, F.a2, r2);
    F.w2[k] = U.sub(U.sub(U.sub(R[2 + k], L[2 + k]), F.w0[k]), F.w1[k]);
  }
}

// Limiter value for the ratio num/den of eq. limiter, 0 for a zero wave (which
// divides 1 by 1: 0/0 would take the division's slow path, for a lane without a
// left neighbour in every warp of the lanes_ forms).
template <int LIM>
__device__ __forceinline__ double phi_general(const Unit &U, double num, double den) {
  if (LIM == F64_NONE) return 0.0;
  if (LIM == F64_LW) return den > 0.0 ? 1.0 : 0.0;
  const bool on = den > 0.0;
  const double theta = (on ? num : 1.0) / (on ? den : 1.0);
  const double a = U.mul(0.5, U.add(theta, 1.0));
  double m = a < 2.0 ? a : 2.0;
  const double b = U.add(theta, theta);
  m = m < b ? m : b;
  m = m > 0.0 ? m : 0.0;
  return on ? m : 0.0;
}
// den >= 0.  theta >= 3 gives 2, theta <= 0 gives 0; between, the smaller of
// (1 + theta)/2 and 2 theta, compared as bit patterns.
template <int LIM>
__device__ __forceinline__ double phi_fast(const Unit &U, double num, double den, bool &tiny) {
  if (LIM == F64_NONE) return 0.0;
  if (LIM == F64_LW) return int64f::bits_of(den) ? 1.0 : 0.0;
  int64f::u64 nb = int64f::bits_of(num), db = int64f::bits_of(den);
  const bool on = (int64f::i64)nb > 0 && db != 0;
  nb = on ? nb : 0x3ff0000000000000ull;
  db = on ? db : 0x3ff0000000000000ull;
  double theta;
  int64f::u64 b;             // 2 theta
  const int64f::u32 nh = (int64f::u32)(nb >> 32), dh = (int64f::u32)(db >> 32);
  if (nh >= 0x00100000u && dh >= 0x00100000u && nh - dh + (900u << 20) < (1800u << 20)) {
    theta = int64f::div_normal(nb, db);
    b = int64f::bits_of(int64f::twice(theta));
  } else {
    theta = int64f::of_bits(nb) / int64f::of_bits(db);
    b = int64f::bits_of(theta + theta);
  }
  const int64f::u64 a = int64f::bits_of(int64f::half_of(U.add(theta, 1.0)));
  int64f::u64 m = a < b ? a : b;
  m = hi_of(theta) >= 0x40080000u ? 0x4000000000000000ull : m;
  m = on ? m : 0;
  tiny |= on && (int64f::u32)(m >> 32) < (923u << 20);
  return int64f::of_bits(m);
}

// Fluctuations and correction flux of face I between the faces Lf and Rf.  In
// 2D a subsonic face's sums over the families are one term each (the others are
// exact zeros), which saves twelve of some 210 instructions a cell; in 3D the
// branch costs the other forms 2 % (145 x 130 x 113 cells, 4 steps: 7.89 ms
// without, 8.04 with).
template <int LIM, int NT>
__device__ __forceinline__ void flux_general(const Par &P, const Face<NT> &I, const Face<NT> &Lf,
                                             const Face<NT> &Rf, Flux<NT> &o) {
  const Unit &U = P.U;
  const double s0 = I.s0, s1 = I.s1, u = I.u;
  const double smu = u < 0.0 ? u : 0.0, spu = u > 0.0 ? u : 0.0;
  const bool l0 = s0 > 0.0, l1 = s1 > 0.0, lu = u > 0.0;
  if (NT == 1 && l0 && s1 < 0.0) {
    o.am[0] = U.mul(s1, I.a2);
    o.ap[0] = U.mul(s0, I.a1);
    o.am[1] = U.mul(s1, I.w11);
    o.ap[1] = U.mul(s0, I.w01);
#pragma unroll
    for (int k = 0; k < NT; k++) {
      o.am[2 + k] = U.add(U.mul(s1, I.w1[k]), U.mul(smu, I.w2[k]));
      o.ap[2 + k] = U.add(U.mul(s0, I.w0[k]), U.mul(spu, I.w2[k]));
    }
  } else {
    const double sm0 = s0 < 0.0 ? s0 : 0.0, sp0 = s0 > 0.0 ? s0 : 0.0;
    const double sm1 = s1 < 0.0 ? s1 : 0.0, sp1 = s1 > 0.0 ? s1 : 0.0;
    o.am[0] = U.add(U.mul(sm0, I.a1), U.mul(sm1, I.a2));
    o.ap[0] = U.add(U.mul(sp0, I.a1), U.mul(sp1, I.a2));
    o.am[1] = U.add(U.mul(sm0, I.w01), U.mul(sm1, I.w11));
    o.ap[1] = U.add(U.mul(sp0, I.w01), U.mul(sp1, I.w11));
#pragma unroll
    for (int k = 0; k < NT; k++) {
      o.am[2 + k] = U.add(U.add(U.mul(sm0, I.w0[k]), U.mul(sm1, I.w1[k])), U.mul(smu, I.w2[k]));
      o.ap[2 + k] = U.add(U.add(U.mul(sp0, I.w0[k]), U.mul(sp1, I.w1[k])), U.mul(spu, I.w2[k]));
    }
  }
  double d0 = U.add(U.mul(I.a1, I.a1), U.mul(I.w01, I.w01));
  double n0 = U.add(U.mul(l0 ? Lf.a1 : Rf.a1, I.a1), U.mul(l0 ? Lf.w01 : Rf.w01, I.w01));
  double d1 = U.add(U.mul(I.a2, I.a2), U.mul(I.w11, I.w11));
  double n1 = U.add(U.mul(l1 ? Lf.a2 : Rf.a2, I.a2), U.mul(l1 ? Lf.w11 : Rf.w11, I.w11));
#pragma unroll
  for (int k = 0; k < NT; k++) {
    d0 = U.add(d0, U.mul(I.w0[k], I.w0[k]));
    n0 = U.add(n0, U.mul(l0 ? Lf.w0[k] : Rf.w0[k], I.w0[k]));
    d1 = U.add(d1, U.mul(I.w1[k], I.w1[k]));
    n1 = U.add(n1, U.mul(l1 ? Lf.w1[k] : Rf.w1[k], I.w1[k]));
  }
  // |s| (1 - dt/dx |s|) phi
  auto coef = [&](double s, double num, double den) {
    const double as = fabs(s);
    return U.mul(U.mul(as, U.sub(1.0, U.mul(P.lam, as))), phi_general<LIM>(U, num, den));
  };
  const double c0 = coef(s0, n0, d0), c1 = coef(s1, n1, d1);
  o.G[0] = U.add(U.mul(c0, I.a1), U.mul(c1, I.a2));
  o.G[1] = U.add(U.mul(c0, I.w01), U.mul(c1, I.w11));
#pragma unroll
  for (int k = 0; k < NT; k++) {
    const double w = lu ? Lf.w2[k] : Rf.w2[k];
    const double c2 = coef(u, U.mul(w, I.w2[k]), U.mul(I.w2[k], I.w2[k]));
    o.G[2 + k] = U.add(U.add(U.mul(c0, I.w0[k]), U.mul(c1, I.w1[k])), U.mul(c2, I.w2[k]));
  }
}

// tiny: halves of G may be subnormal
template <int FORM, int LIM, int NT>
__device__ __forceinline__ void flux_fast(const Par &P, const Face<NT> &I, const Face<NT> &Lf,
                                          const Face<NT> &Rf, Flux<NT> &o, bool &tiny) {
  const Unit &U = P.U;
  const bool neg = (int)hi_of(I.u) < 0;
  o.am[0] = I.w11;
  o.ap[0] = I.w01;
  o.am[1] = U.mul(I.s1, I.w11);
  o.ap[1] = U.mul(I.s0, I.w01);
  double d0 = U.add(prod<FORM>(U, I.a1, I.a1), prod<FORM>(U, I.w01, I.w01));
  double n0 = U.add(prod<FORM>(U, Lf.a1, I.a1), prod<FORM>(U, Lf.w01, I.w01));
  double d1 = U.add(prod<FORM>(U, I.a2, I.a2), prod<FORM>(U, I.w11, I.w11));
  double n1 = U.add(prod<FORM>(U, Rf.a2, I.a2), prod<FORM>(U, Rf.w11, I.w11));
#pragma unroll
  for (int k = 0; k < NT; k++) {
    // the transverse wave joins the fluctuation of the side it moves to
    const double X = U.mul(I.s1, I.w1[k]), Y = U.mul(I.s0, I.w0[k]);
    const double t = U.add(neg ? X : Y, U.mul(I.u, I.w2[k]));
    o.am[2 + k] = neg ? t : X;
    o.ap[2 + k] = neg ? Y : t;
    d0 = U.add(d0, prod<FORM>(U, I.w0[k], I.w0[k]));
    n0 = U.add(n0, prod<FORM>(U, Lf.w0[k], I.w0[k]));
    d1 = U.add(d1, prod<FORM>(U, I.w1[k], I.w1[k]));
    n1 = U.add(n1, prod<FORM>(U, Rf.w1[k], I.w1[k]));
  }
  const double as1 = -I.s1, asu = fabs(I.u);
  const double c0 = U.mul(U.mul(I.s0, U.sub(1.0, U.mul(P.lam, I.s0))), phi_fast<LIM>(U, n0, d0, tiny));
  const double c1 = U.mul(U.mul(as1, U.sub(1.0, U.mul(P.lam, as1))), phi_fast<LIM>(U, n1, d1, tiny));
  const double fu = U.mul(asu, U.sub(1.0, U.mul(P.lam, asu)));
  o.G[0] = U.add(U.mul(c0, I.a1), U.mul(c1, I.a2));
  o.G[1] = U.add(U.mul(c0, I.w01), U.mul(c1, I.w11));
#pragma unroll
  for (int k = 0; k < NT; k++) {
    const double w = neg ? Rf.w2[k] : Lf.w2[k];
    const double c2 =
        U.mul(fu, phi_fast<LIM>(U, U.mul(w, I.w2[k]), U.mul(I.w2[k], I.w2[k]), tiny));
    o.G[2 + k] = U.add(U.add(U.mul(c0, I.w0[k]), U.mul(c1, I.w1[k])), U.mul(c2, I.w2[k]));
    if (FORM == SOFT)
      tiny |= (int64f::bits_of(o.G[2 + k]) & 0x7fffffffffffffffull) - 1 < (123ull << 52);
  }
}

// Cell update of eq. fv-hr.
template <int NT>
__device__ __forceinline__ void update_general(const Par &P, const double q[2 + NT], const double am[],
                                               const double Gr[], const double ap[],
                                               const double Gl[], double o[2 + NT]) {
  const Unit &U = P.U;
#pragma unroll
  for (int k = 0; k < 2 + NT; k++)
    o[k] = U.sub(U.sub(q[k], U.mul(P.lam, U.add(am[k], ap[k]))),
                 U.mul(P.lam, U.sub(U.mul(0.5, Gr[k]), U.mul(0.5, Gl[k]))));
}
template <int NT>
__device__ __forceinline__ void update_fast(const Par &P, const double q[2 + NT], const double am[],
                                            const double Gr[], const double ap[],
                                            const double Gl[], double o[2 + NT]) {
  const Unit &U = P.U;
#pragma unroll
  for (int k = 0; k < 2 + NT; k++)
    o[k] = U.sub(U.sub(q[k], U.mul(P.lam, U.add(am[k], ap[k]))),
                 mulz(P.hlam, U.sub(Gr[k], Gl[k])));
}

// max|s| as a bit pattern (|s3| = |u| never exceeds the other two)
template <int NT>
__device__ __forceinline__ void speed_max(unsigned long long &m, const Face<NT> &F) {
  const unsigned long long b0 = int64f::bits_of(F.s0) & 0x7fffffffffffffffull,
                           b1 = int64f::bits_of(F.s1) & 0x7fffffffffffffffull;
  m = b0 > m ? b0 : m;
  m = b1 > m ? b1 : m;
}

// ---------------------------------------------------------------------------
// A segment of a line across the lanes: lane l holds the CPL consecutive
// cells q[0..CPL-1], lane l + 1 the next ones.  Each lane solves the faces on
// the left of its cells; neighbour cells, faces and fluxes come by shuffles.
// On return o[] is the update of every cell that has two cells of the segment
// on each side.  g = line coordinate of q[0], n = cells of the line: max|s|
// is taken over the faces of the domain cells, the non-real test over the
// extended line's, as the reference evaluation does.  Faces flo..fhi (face f
// lies on the left of cell f) take no correction.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double down1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

template <int FORM, int LIM, int NT, int CPL>
__device__ __forceinline__ void lanes_update(const Par &P, const double q[CPL][2 + NT], int g, int n,
                                             unsigned long long &smax, bool &nonreal,
                                             double o[CPL][2 + NT], int flo, int fhi) {
  const int lane = threadIdx.x & 31;
  double z[CPL][1 + NT], ql[2 + NT], zl[1 + NT];
#pragma unroll
  for (int i = 0; i < CPL; i++) {
    if (FORM) z_fast<NT>(P, q[i], z[i]);
    else z_general<NT>(P.U, q[i], z[i]);
  }
#pragma unroll
  for (int k = 0; k < 2 + NT; k++) ql[k] = up1(q[CPL - 1][k]);
#pragma unroll
  for (int k = 0; k < 1 + NT; k++) zl[k] = up1(z[CPL - 1][k]);
  Face<NT> F[CPL];
#pragma unroll
  for (int i = 0; i < CPL; i++) {
    const double *L = i ? q[i ? i - 1 : 0] : ql, *zL = i ? z[i ? i - 1 : 0] : zl;
    bool nr = false;
    if (FORM) face_fast<FORM, NT>(P, L, zL, q[i], z[i], F[i]);
    else nr = face_general<NT>(P, L, zL, q[i], z[i], F[i]);
    const int gl = g + i - 1;                      // left cell of the face
    if (i > 0 || lane > 0) {
      if (!FORM && gl >= -2 && gl <= n) nonreal |= nr;
      if (gl >= -1 && gl <= n - 1) speed_max(smax, F[i]);
    }
  }
  // the face before this lane's first one, and the one after its last
  Face<NT> A, B;
  A.a1 = up1(F[CPL - 1].a1); A.w01 = up1(F[CPL - 1].w01);
  B.a2 = down1(F[0].a2); B.w11 = down1(F[0].w11);
  if (!FORM) {
    A.a2 = up1(F[CPL - 1].a2); A.w11 = up1(F[CPL - 1].w11);
    B.a1 = down1(F[0].a1); B.w01 = down1(F[0].w01);
  }
#pragma unroll
  for (int k = 0; k < NT; k++) {
    A.w0[k] = up1(F[CPL - 1].w0[k]); A.w2[k] = up1(F[CPL - 1].w2[k]);
    B.w1[k] = down1(F[0].w1[k]); B.w2[k] = down1(F[0].w2[k]);
    if (!FORM) {
      A.w1[k] = up1(F[CPL - 1].w1[k]);
      B.w0[k] = down1(F[0].w0[k]);
    }
  }
  Flux<NT> X[CPL];
  bool tiny = false;
#pragma unroll
  for (int i = 0; i < CPL; i++) {
    const Face<NT> &Lf = i ? F[i ? i - 1 : 0] : A, &Rf = i + 1 < CPL ? F[i + 1 < CPL ? i + 1 : 0] : B;
    if (FORM) flux_fast<FORM, LIM, NT>(P, F[i], Lf, Rf, X[i], tiny);
    else flux_general<LIM, NT>(P, F[i], Lf, Rf, X[i]);
    if (g + i >= flo && g + i <= fhi) {
#pragma unroll
      for (int k = 0; k < 2 + NT; k++) X[i].G[k] = 0.0;
    }
  }
  const bool half = FORM == SOFT && !__any_sync(0xffffffffu, tiny);
  double am[2 + NT], G[2 + NT];                    // the next lane's first face
#pragma unroll
  for (int k = 0; k < 2 + NT; k++) {
    am[k] = down1(X[0].am[k]);
    G[k] = down1(X[0].G[k]);
  }
#pragma unroll
  for (int i = 0; i < CPL; i++) {
    const double *mr = i + 1 < CPL ? X[i + 1 < CPL ? i + 1 : 0].am : am;
    const double *Gr = i + 1 < CPL ? X[i + 1 < CPL ? i + 1 : 0].G : G;
    if (half) update_fast<NT>(P, q[i], mr, Gr, X[i].ap, X[i].G, o[i]);
    else update_general<NT>(P, q[i], mr, Gr, X[i].ap, X[i].G, o[i]);
  }
}

// The segment in the form its data allow.
template <int LIM, int NT, int CPL>
__device__ __forceinline__ void lanes_step(const Par &P, const double q[CPL][2 + NT], int g, int n,
                                           unsigned long long &smax, bool &nonreal,
                                           double o[CPL][2 + NT], int flo = 1, int fhi = 0) {
  int f = P.ok ? SOFT : GENERAL;
#pragma unroll
  for (int i = 0; i < CPL; i++) f = min(f, form_of<NT>(q[i]));
  f = warp_form(f);
  if (f == SOFT) lanes_update<SOFT, LIM, NT, CPL>(P, q, g, n, smax, nonreal, o, flo, fhi);
  else if (f == FAST) lanes_update<FAST, LIM, NT, CPL>(P, q, g, n, smax, nonreal, o, flo, fhi);
  else lanes_update<GENERAL, LIM, NT, CPL>(P, q, g, n, smax, nonreal, o, flo, fhi);
}

// ---------------------------------------------------------------------------
// A line marched by each lane: cells are pushed in order, j = 0, 1, ...; face
// j lies between cells j - 1 and j.  From j = 4 on a push returns the update
// of cell j - 2.  Called by all lanes of the warp together.
// ---------------------------------------------------------------------------
template <int LIM, int NT> struct March {
  double c1[2 + NT], c2[2 + NT], z1[1 + NT];
  Face<NT> f1, f2;            // faces j - 1 and j - 2
  double ap[2 + NT], G[2 + NT];
  int fast, soft;             // cells in a row that allow these forms, the same in all lanes
  bool lhalf;                 // the left face's G may be halved after the fact
  unsigned long long smax;
  bool nonreal;

  __device__ __forceinline__ void init() {
    fast = soft = 0;
    lhalf = true;
    smax = 0;
    nonreal = false;
  }
  // count_speed: face j - 1 counts towards max|s|; count_real: face j towards
  // the non-real test; plain: no correction on face j - 1
  __device__ __forceinline__ bool push(const Par &P, int j, const double q[2 + NT],
                                       double out[2 + NT], bool count_speed, bool count_real,
                                       bool plain) {
    const int f = warp_form(P.ok ? form_of<NT>(q) : GENERAL);
    fast = f >= FAST ? fast + 1 : 0;
    soft = f == SOFT ? soft + 1 : 0;
    const int need = j < 4 ? j : 4;                // this cell and the four before it
    if (soft > need) step<SOFT>(P, j, q, out, count_speed, count_real, plain);
    else if (fast > need) step<FAST>(P, j, q, out, count_speed, count_real, plain);
    else step<GENERAL>(P, j, q, out, count_speed, count_real, plain);
    return j >= 4;
  }
  template <int FORM>
  __device__ __forceinline__ void step(const Par &P, int j, const double q[2 + NT],
                                       double out[2 + NT], bool count_speed, bool count_real,
                                       bool plain) {
    double z[1 + NT];
    if (FORM) z_fast<NT>(P, q, z);
    else z_general<NT>(P.U, q, z);
    if (j > 0) {
      Face<NT> f;
      if (FORM) face_fast<FORM, NT>(P, c1, z1, q, z, f);
      else {
        const bool nr = face_general<NT>(P, c1, z1, q, z, f);
        if (count_real) nonreal |= nr;
      }
      if (j >= 3) {
        Flux<NT> X;
        bool half = FORM == SOFT;
        if (FORM) {
          bool tiny = false;
          flux_fast<FORM, LIM, NT>(P, f1, f2, f, X, tiny);
          half = half && !__any_sync(0xffffffffu, tiny);
        } else {
          flux_general<LIM, NT>(P, f1, f2, f, X);
        }
        if (plain) {
#pragma unroll
          for (int k = 0; k < 2 + NT; k++) X.G[k] = 0.0;
        }
        if (count_speed) speed_max(smax, f1);
        if (j >= 4) {
          if (half && lhalf) update_fast<NT>(P, c2, X.am, X.G, ap, G, out);
          else update_general<NT>(P, c2, X.am, X.G, ap, G, out);
        }
#pragma unroll
        for (int k = 0; k < 2 + NT; k++) {
          ap[k] = X.ap[k];
          G[k] = X.G[k];
        }
        lhalf = half;
      }
      f2 = f1;
      f1 = f;
    }
#pragma unroll
    for (int k = 0; k < 2 + NT; k++) {
      c2[k] = c1[k];
      c1[k] = q[k];
    }
#pragma unroll
    for (int k = 0; k < 1 + NT; k++) z1[k] = z[k];
  }
};

}  // namespace f64
}  // namespace fvna
