// collide.cuh -- cascaded central-moment collision of one node (Sec. 3),
// written in deviation form d_a = f_a - w_a rho0.
//
// Working with deviations keeps the large rest-state constant out of every
// sum: the raw moments of w rho0 are rho0 * (1, 0, 1/3, 0, 1/9) by order, so
// each raw moment k' of f is that constant plus the same moment D of d, and
// the constants cancel analytically in m^(1), in g^_4..g^_9 and in the
// fourth-order attractor terms of g^_16..g^_18 (expanded around rho/3 below).
// The FP32 and FP16-storage forms therefore lose no precision to a rest value
// of order 1, and the FP64 form computes the same expressions.
#pragma once

#include <type_traits>

#include "d3q19.cuh"
#include "log_table.h"
#include "v2.cuh"

namespace clbm {

// Scalar type of the per-lattice constants for a math type R (a pair of FP32
// nodes uses FP32 constants).
template <typename R> struct ScalarOf { using type = R; };
template <> struct ScalarOf<V2> { using type = float; };

// Constants of the FP64 step of the omega solve.
template <typename R> struct SolveConst64 {};
template <> struct SolveConst64<double> {
  double clog;      // log(3 K) + (n-1)/2 log 9
  double eh, nm1;   // (n - 1) / 2, n - 1 (power-law index n)
  double tlo, thi;  // 3 nu_min, 3 nu_max (clamp of 1/w - 1/2)
};

// Per-lattice constants of the collision, in the math precision R.
template <typename R>
struct CollideConst : SolveConst64<R> {
  R rho0;
  R rhoS;        // lam rho0 and lam F: rest density and force of deviations
  R FS[3];       //   carried scaled by lam (FP16 storage: lam = 1024; else 1)
  R r30;         // rhoS / 3
  R K3;          // 3 K lam (K = mu_p, consistency coefficient, Eq. 5)
  R nu_min, nu_max;
  // FP32 solve of every form: n, 1/n, (n-1)/2, log2(3 K lam) + (n-1)/2 log2 9,
  // the clamp of y = log2(1/w - 1/2), lower bound of the invariant g2
  float n, rn, ehalf, clog2, ylo2, yhi2, g2lo;
  int newtonian; // n == 1: omega_nu has a closed form
  int has_force;
  // The rates omega_9..18 enter only as factors of their own relaxation
  // brackets (Eqs. collisionkernelg4..g18; the lower-order g^ terms carry no
  // rate), and omega_9 scales the isotropic part of the strain rate.  They
  // are folded into the brackets' constants: c9 = -omega_9/126,
  // c10..c15 = omega_j/8, c16 = omega_16/12, c17 = omega_17/24,
  // c18 = omega_18/8, cB = omega_9^2 / 6 (unit rates give the constants of
  // the printed forms exactly).
  R c9, c10, c11, c12, c13, c14, c15, c16, c17, c18, cB;
};

// Outputs of one collision besides the populations.
template <typename R>
struct NodeOut {
  R rho, ux, uy, uz, gamma_dot;
};

// Base-2 logarithm and power of two on the special-function unit (PTX
// lg2.approx / ex2.approx, about 22 correct bits): the FP32 solve for
// omega_nu works in base 2, so no conversion factor is spent on either.
__device__ __forceinline__ float lg2f(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2f(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <typename R> __device__ __forceinline__ R rlg2(R x);
template <> __device__ __forceinline__ float rlg2<float>(float x) { return lg2f(x); }
template <typename R> __device__ __forceinline__ R rex2(R x);
template <> __device__ __forceinline__ float rex2<float>(float x) { return ex2f(x); }
// Reciprocal on the special-function unit (1 ulp) in FP32; rcp64 in FP64.
__device__ __forceinline__ float rcpf(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <typename R> __device__ __forceinline__ R rrcp(R x);
template <> __device__ __forceinline__ float rrcp<float>(float x) { return rcpf(x); }
template <> __device__ __forceinline__ V2 rlg2<V2>(V2 x) { return V2(lg2f(x.v.x), lg2f(x.v.y)); }
template <> __device__ __forceinline__ V2 rex2<V2>(V2 x) { return V2(ex2f(x.v.x), ex2f(x.v.y)); }
template <> __device__ __forceinline__ V2 rrcp<V2>(V2 x) { return V2(rcpf(x.v.x), rcpf(x.v.y)); }

// A product that the compiler may not fuse into a later sum.  The unit-rate
// collision and the solve below spell out every fused multiply-add, so that
// one node and a packed pair of nodes, in any kernel, round alike.
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ V2 mulr(V2 a, V2 b) { return a * b; }

// Lower bound of the shear-rate invariant inside the logarithm.
template <typename R> __device__ __forceinline__ R tiny();
template <> __device__ __forceinline__ float tiny<float>() { return 1e-36f; }
template <> __device__ __forceinline__ double tiny<double>() { return 1e-300; }
template <> __device__ __forceinline__ V2 tiny<V2>() { return V2(1e-36f); }

// Starting point of the solve below.  Without the bulk part B, the unknown
// z = 1/omega - 1/2 = 3 nu solves z (z + 1/2)^(n-1) = P, whose two asymptotes
// are z = P^(1/n) (z >> 1/2) and z = 2^(n-1) P (z << 1/2); they meet at
// z = 1/2, where log2 P = -n.  The guess takes the asymptote of its side
// (with A + B for A), which three Newton steps then take to the FP32 rounding
// level over the workloads' range of n, K and shear rate.
__device__ __forceinline__ float regime_guess(float lp, float n, float rn) {
  return lp > -n ? mulr(lp, rn) : lp + (n - 1.0f);
}
__device__ __forceinline__ V2 regime_guess(V2 lp, float n, float rn) {
  return V2(regime_guess(lp.v.x, n, rn), regime_guess(lp.v.y, n, rn));
}

// The solve for omega_nu, on y = log2(1/omega - 1/2):
//   G(y) = y - c - (n-1)/2 log2(g2),  g2 = omega(y)^2 A + B,
// i.e. 1/omega - 1/2 = 3 nu with nu = (K/rho) gamma_dot^(n-1) (Eq. 6,
// Eq. localvarationsrelaxationtimes) and gamma_dot^2 = (9 / rho^2) g2 (see
// strain_AB): the omega part of the strain rate of Eq. strainratetensor is
// traceless, so its invariant (Eq. shearrateexpression) is quadratic in
// omega.  The factor 9 / rho^2 sits in c = log2(3 K) + (n-1)/2 log2 9 - n log2 rho.
// dG/dy = 1 + (n-1) r s with r = omega^2 A / g2 and s = tau omega
// = 1 - omega/2 in (0, 1) (the base of the logarithm cancels), so G is
// increasing with slope between min(n, 1) and max(n, 1) and has one root;
// projecting each iterate onto [ylo, yhi] makes the iteration land on the
// clamp when the root lies beyond it.  The step G / (dG/dy) is taken as
// G g2 / (g2 + (n-1) omega^2 A s): one reciprocal.
template <typename R>
__device__ __forceinline__ R newton_y2(R y, R c, R ehalf, R nm1, R A, R B, R ylo, R yhi, R lo,
                                       int iters) {
#pragma unroll 1
  for (int it = 0; it < iters; ++it) {
    const R w = rrcp<R>(rex2<R>(y) + R(0.5f));
    const R ww = mulr(w, w);
    const R g2 = fmax(fma(ww, A, B), lo);
    const R G = fma(-ehalf, rlg2<R>(g2), y - c);
    const R den = fma(nm1, mulr(mulr(ww, A), fma(R(-0.5f), w, R(1.0f))), g2);
    y = fmin(fmax(fma(-mulr(G, g2), rrcp<R>(den), y), ylo), yhi);
  }
  return y;
}

// omega_nu from rho (scaled by lam), its reciprocal and A, B of strain_AB.
// FP32 (one node or a pair): the regime guess and three Newton steps reach
// the FP32 rounding level.
template <typename R>
__device__ __forceinline__ R solve_y2(const float n, const float rn, const float ehalf,
                                      const float clog2, const float ylo2, const float yhi2,
                                      const float lo, R rho, R A, R B) {
  const R c = fma(R(-n), rlg2<R>(rho), R(clog2));
  const R lp = fma(R(ehalf), rlg2<R>(fmax(A + B, R(lo))), c);
  const R y = fmin(fmax(regime_guess(lp, n, rn), R(ylo2)), R(yhi2));
  return newton_y2<R>(y, c, R(ehalf), R(n - 1.0f), A, B, R(ylo2), R(yhi2), R(lo), 3);
}
template <typename R>
__device__ __forceinline__ R omega_nu(const CollideConst<float>& C, R rho, R rinv, R A, R B) {
  if (C.newtonian) {
    const R nu = fmin(fmax(mulr(R(C.K3 * (1.0f / 3.0f)), rinv), R(C.nu_min)), R(C.nu_max));
    return rrcp<R>(fma(R(3.0f), nu, R(0.5f)));
  }
  const R y = solve_y2<R>(C.n, C.rn, C.ehalf, C.clog2, C.ylo2, C.yhi2, C.g2lo, rho, A, B);
  return rrcp<R>(rex2<R>(y) + R(0.5f));
}

// ---- FP64 helpers -----------------------------------------------------------
// FP64 arithmetic runs at 1/64 of the FP32 rate on this part and bounds the
// FP64 step, so the solve spends as few FP64 instructions as it can: seeds
// come from FP32, and conversions between the types are integer operations
// on the bit patterns (the hardware's conversions share the FP64 rate).

// A normal float as a double, exactly (zero comes out as 2^-127).
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x);
  const unsigned hi = ((b & 0x7fffffffu) >> 3) + 0x38000000u;
  return __hiloint2double(int(hi | (b & 0x80000000u)), int(b << 29));
}

// double(x) for the FP64 sums and outputs of the FP32-math forms: integer
// operations for zero and normal values, the hardware's conversion otherwise.
__device__ __forceinline__ double to64(double x) { return x; }
__device__ __forceinline__ double to64(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u) return widen(x);
  if (m == 0u) return __hiloint2double(int(b), 0);
  return double(x);
}

// A non-negative double below 2^128 truncated to float; zero and values below
// 2^-125 give 2^-125.
__device__ __forceinline__ float narrow(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  return hi < 0x38200000 ? 2.3509887e-38f
                         : __uint_as_float((unsigned(hi - 0x38000000) << 3) | (lo >> 29));
}

// The same for any size: values from 2^110 on, beyond which the FP32 solve's
// products would overflow, give about 2^110.
__device__ __forceinline__ float narrow_any(double x) {
  return narrow(__hiloint2double(min(__double2hiint(x), 0x46d00000), __double2loint(x)));
}

// The same for either sign.
__device__ __forceinline__ float narrow_signed(double x) {
  return copysignf(narrow(fabs(x)), __uint_as_float(unsigned(__double2hiint(x))));
}

// Comparison of two doubles, the second positive, by their bit patterns.
__device__ __forceinline__ bool below(double x, double bound) {
  return __double_as_longlong(x) < __double_as_longlong(bound);
}

// Tests on the upper word's bits: x positive, finite and above 2^-1042; x neither
// infinite nor NaN.
__device__ __forceinline__ bool positive_finite(double x) {
  return unsigned(__double2hiint(x)) - 1u < 0x7fefffffu;
}
__device__ __forceinline__ bool finite_bits(double x) {
  return (unsigned(__double2hiint(x)) & 0x7ff00000u) != 0x7ff00000u;
}

// 1/x for normal x: the FP32 reciprocal of the mantissa as the seed r0, then
// r0 (1 + e + e^2) with e = 1 - x r0 (the cubically convergent iteration):
// the seed's 2^-22 leaves 2^-66, below the rounding of the last operation.
__device__ __forceinline__ double rcp64(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  const float m = __uint_as_float(0x3f800000u | ((unsigned(hi) & 0xfffffu) << 3) | (lo >> 29));
  const unsigned s = __float_as_uint(rcpf(m));
  // exponent of the seed minus that of x, and the sign of x
  const int e = (hi & 0x7ff00000) - 0x3ff00000;
  const double r0 = __hiloint2double(
      (int((s >> 3) + 0x38000000u) - e) | (hi & int(0x80000000u)), int(s << 29));
  const double d = fma(-x, r0, 1.0);
  return fma(r0, fma(d, d, d), r0);
}

template <> __device__ __forceinline__ double rrcp<double>(double x) { return rcp64(x); }

// Natural logarithm of a positive normal x, as (exponent, log of the mantissa)
// with x = 2^ex z: z = 1 + i/1024 to within 1/2048, and with the table's c
// near 1/z, log z = -log c + log1p(r), r = z c - 1, |r| < 2^-10.9 (P. T. P.
// Tang, ACM TOMS 16(4), 1990).  Of log1p(r) = r - r^2/2 + r^3/3 - r^4/4 + r^5/5
// (what is left out is below 2^-68) the terms from r^3 on are below 2^-34, so
// FP32 gives them to 2^-58: five FP64 instructions where a table of 128 and
// an FP64 series took nine.
__device__ __forceinline__ double log_mant(double x, int& ex) {
  const int hi = __double2hiint(x) + 0x200;
  ex = (hi >> 20) - 1023;
  const double z = __hiloint2double(__double2hiint(x) - (ex << 20), __double2loint(x));
  const double2 t = __ldg(&LOG_TAB[(hi >> 10) & 1023]);
  const double r = fma(z, t.x, -1.0);
  const float f = narrow_signed(r), f2 = mulr(f, f);
  const float c = mulr(mulr(f2, f), fma(f, fma(f, 0.2f, -0.25f), 1.0f / 3.0f));
  return t.y + (fma(-0.5, mulr(r, r), r) + widen(c));
}

// FP64: the FP32 solve gives tau0 = 1/omega - 1/2 to about 1e-6, taken as the
// exact value of a float; one Halley step in FP64 on y = log tau then lands
// at the FP64 rounding level (it converges cubically).  With g2, r and s as
// above at tau0, and G = log(tau0 rho) - log(3 K) - (n-1)/2 log(9 g2 / rho^2)
// (two logarithms, each by log_mant),
//   G'  = 1 + (n-1) r s,
//   G'' = (n-1) [s omega r / 2 - 2 r (1 - r) s^2]
// (from ds/dy = tau omega^2 / 2 and dr/dy = -2 r (1 - r) s), and the step is
// dy = d1 (1 - d1 G'' / (2 G')) with d1 = -G/G'.  The correction of the second
// factor is of the order of dy, so it needs FP32 only; tau is carried to the
// new y by exp(dy) = 1 + dy + dy^2/2 + dy^3/6, whose terms beyond d1 likewise.
__device__ __forceinline__ double omega_nu(const CollideConst<double>& C, double rho,
                                           double rinv, double A, double B) {
  if (C.newtonian) {
    const double nu = fmin(fmax(mulr(C.K3 * (1.0 / 3.0), rinv), C.nu_min), C.nu_max);
    return rcp64(fma(3.0, nu, 0.5));
  }
  const float Af = narrow_any(A), Bf = narrow_any(B);
  const float yf = solve_y2<float>(C.n, C.rn, C.ehalf, C.clog2, C.ylo2, C.yhi2, C.g2lo,
                                   narrow(rho), Af, Bf);
  const double tau = widen(ex2f(yf));
  const double w = rcp64(tau + 0.5);
  const double ww = mulr(w, w), wwA = mulr(ww, A);
  double g2 = fma(ww, A, B);
  if (below(g2, 1e-300)) g2 = 1e-300;
  int e1, e2;
  const double l1 = log_mant(mulr(tau, rho), e1);
  const double l2 = log_mant(mulr(mulr(rinv, rinv), g2), e2);
  const double LN2 = 0.69314718055994530942;
  const double L1 = fma(widen(float(e1)), LN2, l1), L2 = fma(widen(float(e2)), LN2, l2);
  const double G = fma(-C.eh, L2, L1 - C.clog);
  const double s = fma(-0.5, w, 1.0);
  const double den = fma(C.nm1, mulr(wwA, s), g2);
  const double d1 = mulr(-mulr(G, g2), rcp64(den));  // -G / G'
  const float wf = narrow(w), sf = narrow(s), nm1 = C.n - 1.0f;
  const float rf = fminf(mulr(narrow(wwA), rcpf(narrow(g2))), 1.0f);
  const float rs = mulr(rf, sf);
  const float G1 = fma(nm1, rs, 1.0f);
  // G'' = (n-1) r s [omega/2 - 2 (1 - r) s]
  const float G2 = mulr(mulr(nm1, rs), fma(-2.0f * sf, 1.0f - rf, 0.5f * wf));
  // tau1 = tau exp(dy), dy = d1 (1 + h): what exp(dy) - 1 has beyond d1 is of
  // the order of d1^2, so FP32 gives it.  |d1| is large only when the root
  // lies beyond a clamp, where the sign of dy decides.
  const float d1f = narrow_signed(d1);
  const float h = fminf(fmaxf(mulr(mulr(-0.5f * G2, rcpf(G1)), d1f), -0.25f), 0.25f);
  const float dyf = fma(d1f, h, d1f);
  const float rest = fma(d1f, h, mulr(mulr(dyf, dyf), fma(dyf, 1.0f / 6.0f, 0.5f)));
  double t1 = fma(tau, d1 + widen(rest), tau);
  if (below(t1, C.tlo)) t1 = C.tlo;
  else if (below(C.thi, t1)) t1 = C.thi;
  const double w1 = rcp64(t1 + 0.5);
  // The logarithms and clamps work on bit patterns and turn anything into a
  // rate.  A density that has none, and moments that are not finite, give NaN:
  // a diverged node then spoils its lattice until the next check step reports it.
  return __hiloint2double(
      positive_finite(rho) && finite_bits(d1) ? __double2hiint(w1) : 0x7ff80000,
      __double2loint(w1));
}

// |gamma_dot| at the solved omega (a diverged node's density may be negative).
template <typename R>
__device__ __forceinline__ R shear_rate(R rinv, R w, R A, R B) {
  return mulr(mulr(R(3), fabs(rinv)), sqrt(fma(mulr(w, w), A, B)));
}

// ---- pair space -------------------------------------------------------------
// The collision works on the nine +/- velocity pairs instead of the 19
// populations.  An axis pair (e, -e) is held as its sum s and difference t;
// in each coordinate plane the two diagonal pairs P (e_i e_j = +1) and
// M (e_i e_j = -1) are held as four moments of the plane, e.g. in the xy
// plane, with sP = d7 + d10, tP = d7 - d10, sM = d9 + d8, tM = d9 - d8,
//   Dxxyy = sP + sM, Dxy = sP - sM, Dxyy = tP + tM, Dxxy = tP - tM.
// These 19 values are the rest population, the axis sums and differences and
// the plane moments: the raw moments of Eq. rawmomentdistributionfunction1
// are sums of them, and the populations are recovered from them exactly.
// The post-collision populations are rebuilt from the pair values and g^
// at the end, so the 19 pre-collision populations need not stay live
// through the collision.
template <typename R>
struct Pairs {
  R d0;
  R sAx, tAx, sAy, tAy, sAz, tAz;
  R Dxxyy, Dxy, Dxyy, Dxxy;  // xy plane: velocities 7, 10 (P) and 9, 8 (M)
  R Dxxzz, Dxz, Dxzz, Dxxz;  // xz plane: 11, 14 (P) and 13, 12 (M)
  R Dyyzz, Dyz, Dyzz, Dyyz;  // yz plane: 15, 18 (P) and 17, 16 (M)
};

// Pair values of 19 populations in the paper's order (Eq. velocityd3qq19).
template <typename R>
__host__ __device__ constexpr Pairs<R> to_pairs(const R (&d)[Q]) {
  Pairs<R> p{};
  p.d0 = d[0];
  p.sAx = d[1] + d[2];
  p.tAx = d[1] - d[2];
  p.sAy = d[3] + d[4];
  p.tAy = d[3] - d[4];
  p.sAz = d[5] + d[6];
  p.tAz = d[5] - d[6];
  {
    const R sP = d[7] + d[10], tP = d[7] - d[10], sM = d[9] + d[8], tM = d[9] - d[8];
    p.Dxxyy = sP + sM;
    p.Dxy = sP - sM;
    p.Dxyy = tP + tM;
    p.Dxxy = tP - tM;
  }
  {
    const R sP = d[11] + d[14], tP = d[11] - d[14], sM = d[13] + d[12], tM = d[13] - d[12];
    p.Dxxzz = sP + sM;
    p.Dxz = sP - sM;
    p.Dxzz = tP + tM;
    p.Dxxz = tP - tM;
  }
  {
    const R sP = d[15] + d[18], tP = d[15] - d[18], sM = d[17] + d[16], tM = d[17] - d[16];
    p.Dyyzz = sP + sM;
    p.Dyz = sP - sM;
    p.Dyzz = tP + tM;
    p.Dyyz = tP - tM;
  }
  return p;
}

// Four populations of a coordinate plane from its four moments plus the
// plane's part of K g^ (Eq. cascadedcollision1): E (shared by the plane),
// Ex (the product moment g4/g5/g6) and the two odd sums Oa, Ob.  With
// q1 = Dii jj/4 + E, q2 = Dij/4 + Ex, q3 = Dijj/4 + Oa, q4 = Diij/4 + Ob the
// populations are P+ = q1+q2+q3+q4, P- = q1+q2-q3-q4, M+ = q1-q2+q3-q4,
// M- = q1-q2-q3+q4 (P+, P-: the pair with e_i e_j = +1, positive and
// negative e_i; M+, M-: the other pair, positive and negative e_i).
template <typename R>
__host__ __device__ constexpr void plane_out(R Diijj, R Dij, R Dijj, R Diij, R E, R Ex, R Oa,
                                             R Ob, R& Pp, R& Pm, R& Mp, R& Mm) {
  const R q1 = R(0.25) * Diijj + E, q2 = R(0.25) * Dij + Ex;
  const R q3 = R(0.25) * Dijj + Oa, q4 = R(0.25) * Diij + Ob;
  const R a = q1 + q2, b = q1 - q2, c = q3 + q4, e = q3 - q4;
  Pp = a + c;
  Pm = a - c;
  Mp = b + e;
  Mm = b - e;
}

// Populations f~ = f + K g^ from the pair values of f and g^_4..g^_18
// (entries 0..3 of g unused): the columns of K grouped by velocity class
// (Sec. 2, the basis vectors).  The rest node; the three axis pairs, which
// share -11 g9 - 4 g16; and the three coordinate planes of diagonal
// velocities, which share 8 g9 + g16.  In a plane the four velocities differ
// only in the sign of the plane's product moment g4/g5/g6 and of two odd
// sums, e.g. in the xy plane g10 + g13 (odd in x) and g11 - g14 (odd in y).
template <typename R>
__host__ __device__ constexpr void from_pairs(const Pairs<R>& p, const R (&g)[Q], R (&d)[Q]) {
  d[0] = p.d0 + (R(-30) * g[9] + R(12) * g[16]);
  const R Ca = R(-11) * g[9] - R(4) * g[16];
  {
    const R hs = R(0.5) * p.sAx + (Ca + (g[7] + g[8]) - R(4) * g[17]);
    const R ht = R(0.5) * p.tAx - R(4) * g[10];
    d[1] = hs + ht;
    d[2] = hs - ht;
  }
  {
    const R hs = R(0.5) * p.sAy + (Ca + (g[8] - g[7]) + R(2) * (g[17] - g[18]));
    const R ht = R(0.5) * p.tAy - R(4) * g[11];
    d[3] = hs + ht;
    d[4] = hs - ht;
  }
  {
    const R hs = R(0.5) * p.sAz + (Ca - R(2) * g[8] + R(2) * (g[17] + g[18]));
    const R ht = R(0.5) * p.tAz - R(4) * g[12];
    d[5] = hs + ht;
    d[6] = hs - ht;
  }
  const R C9 = R(8) * g[9] + g[16];
  plane_out(p.Dxxyy, p.Dxy, p.Dxyy, p.Dxxy, C9 + R(2) * g[8] + (g[17] + g[18]), g[4],
            g[10] + g[13], g[11] - g[14], d[7], d[10], d[9], d[8]);
  plane_out(p.Dxxzz, p.Dxz, p.Dxzz, p.Dxxz, C9 + (g[7] - g[8]) + (g[17] - g[18]), g[5],
            g[10] - g[13], g[12] + g[15], d[11], d[14], d[13], d[12]);
  plane_out(p.Dyyzz, p.Dyz, p.Dyzz, p.Dyyz, C9 - (g[7] + g[8]) - R(2) * g[17], g[6],
            g[11] + g[14], g[12] - g[15], d[15], d[18], d[17], d[16]);
}

// Compile-time checks of the pair space against the basis definitions:
// the populations come back unchanged from their pair values, and a unit
// g^_j adds column j of K to them.
constexpr bool pairs_roundtrip() {
  for (int q = 0; q < Q; ++q) {
    double d[Q] = {}, out[Q] = {}, g[Q] = {};
    d[q] = 1.0;
    from_pairs(to_pairs(d), g, out);
    for (int k = 0; k < Q; ++k)
      if (out[k] != (k == q ? 1.0 : 0.0)) return false;
  }
  return true;
}
constexpr bool pairs_add_K() {
  for (int j = 4; j < Q; ++j) {
    double d[Q] = {}, out[Q] = {}, g[Q] = {};
    g[j] = 1.0;
    from_pairs(to_pairs(d), g, out);
    for (int q = 0; q < Q; ++q)
      if (out[q] != double(kb(j, cx(q), cy(q), cz(q)))) return false;
  }
  return true;
}
static_assert(pairs_roundtrip(), "pair values must give back the populations");
static_assert(pairs_add_K(), "the pair-space back-transform must add the columns of K");

// Half the pair values of the source S_a = w_a [3 e.F + 9 (e.u)(e.F) - 3 u.F]
// of the symmetric force split (reading of the deferred forcing: its moments
// are 0, F and uF + Fu).  Summed over each pair and plane with the D3Q19
// weights (1/3, 1/18, 1/36) they are, with a_i = u_i F_i and t = u.F / 3:
//   rest -u.F; axis i: s = a_i - t, d = F_i / 3;
//   plane ij: Diijj = a_i + a_j - t, Dij = u_i F_j + u_j F_i,
//             Dijj = F_i / 3, Diij = F_j / 3.
template <typename R, typename T>
__device__ __forceinline__ void add_half_source(Pairs<R>& p, R ux, R uy, R uz,
                                                const T (&F)[3]) {
  const R ax = ux * R(F[0]), ay = uy * R(F[1]), az = uz * R(F[2]);
  const R uF = ax + ay + az;
  const R ht = R(1.0 / 6.0) * uF;  // t / 2
  const R f6x = R(T(F[0]) * T(1.0 / 6.0)), f6y = R(T(F[1]) * T(1.0 / 6.0)),
          f6z = R(T(F[2]) * T(1.0 / 6.0));
  p.d0 -= R(0.5) * uF;
  p.sAx += R(0.5) * ax - ht;
  p.sAy += R(0.5) * ay - ht;
  p.sAz += R(0.5) * az - ht;
  p.tAx += f6x;
  p.tAy += f6y;
  p.tAz += f6z;
  p.Dxxyy += R(0.5) * (ax + ay) - ht;
  p.Dxxzz += R(0.5) * (ax + az) - ht;
  p.Dyyzz += R(0.5) * (ay + az) - ht;
  p.Dxy += R(0.5) * (ux * R(F[1]) + uy * R(F[0]));
  p.Dxz += R(0.5) * (ux * R(F[2]) + uz * R(F[0]));
  p.Dyz += R(0.5) * (uy * R(F[2]) + uz * R(F[1]));
  p.Dxyy += f6x;
  p.Dxzz += f6x;
  p.Dxxy += f6y;
  p.Dyzz += f6y;
  p.Dxxz += f6z;
  p.Dyyz += f6z;
}

// Post-collision populations f~ = f + K g^ (+ S, the whole body-force source
// of the symmetric split: half before and half after the collision), added
// to the pre-collision deviations as one correction per population, so that
// each population is rounded once at its own scale.  The correction is
// grouped by velocity class as in from_pairs.  With FP32 populations this
// matters: rebuilding them from pair values rounds sums of populations each
// step, and near a steady state those roundings repeat and accumulate.
// For a +/- pair (e, -e) the source is S_+- = w [9 (e.u)(e.F) - 3 u.F] +- 3 w e.F.
template <typename R, bool FORCE, typename T>
__host__ __device__ constexpr void add_K_g(R (&d)[Q], const R (&g)[Q], R ux, R uy, R uz,
                                           const T (&F)[3]) {
  R se = R(0), so = R(0), uF = R(0);
  if (FORCE) uF = ux * R(F[0]) + uy * R(F[1]) + uz * R(F[2]);
  d[0] += (R(-30) * g[9] + R(12) * g[16]) - (FORCE ? uF : R(0));
  const R Ca = R(-11) * g[9] - R(4) * g[16];
  const R u6 = R(1.0 / 6.0) * uF;  // 3 w u.F for the axis weight 1/18
  {
    const R E = Ca + (g[7] + g[8]) - R(4) * g[17];
    const R O = R(4) * g[10];
    if (FORCE) { se = R(0.5) * ux * R(F[0]) - u6; so = R(T(F[0]) * T(1.0 / 6.0)); }
    d[1] += (E - O) + (se + so);
    d[2] += (E + O) + (se - so);
  }
  {
    const R E = Ca + (g[8] - g[7]) + R(2) * (g[17] - g[18]);
    const R O = R(4) * g[11];
    if (FORCE) { se = R(0.5) * uy * R(F[1]) - u6; so = R(T(F[1]) * T(1.0 / 6.0)); }
    d[3] += (E - O) + (se + so);
    d[4] += (E + O) + (se - so);
  }
  {
    const R E = Ca - R(2) * g[8] + R(2) * (g[17] + g[18]);
    const R O = R(4) * g[12];
    if (FORCE) { se = R(0.5) * uz * R(F[2]) - u6; so = R(T(F[2]) * T(1.0 / 6.0)); }
    d[5] += (E - O) + (se + so);
    d[6] += (E + O) + (se - so);
  }
  const R C9 = R(8) * g[9] + g[16];
  const R u12 = R(1.0 / 12.0) * uF;  // 3 w u.F for the diagonal weight 1/36
  // One plane: pair P = (Pp, Pm) with e_i e_j = +1 and M = (Mp, Mm) with
  // e_i e_j = -1 (first member positive along the plane's first axis); its
  // part of K g^ is E +- Ex (product moment) plus the odd sums (Oa, Ob), and
  // ea/eb, ua/ub are e.F and e.u of the P and M pairs' positive members.
  auto plane = [&](R& Pp, R& Pm, R& Mp, R& Mm, R E, R Ex, R Oa, R Ob, R fP, R fM, R vP,
                   R vM) {
    const R Ep = E + Ex, Em = E - Ex;
    const R Sg = Oa + Ob, Dg = Ob - Oa;
    R sP = R(0), oP = R(0), sM = R(0), oM = R(0);
    if (FORCE) {
      sP = R(0.25) * vP * fP - u12;
      oP = R(1.0 / 12.0) * fP;
      sM = R(0.25) * vM * fM - u12;
      oM = R(1.0 / 12.0) * fM;
    }
    Pp += (Ep + Sg) + (sP + oP);
    Pm += (Ep - Sg) + (sP - oP);
    Mp += (Em - Dg) + (sM + oM);
    Mm += (Em + Dg) + (sM - oM);
  };
  const R Fx = FORCE ? R(F[0]) : R(0), Fy = FORCE ? R(F[1]) : R(0), Fz = FORCE ? R(F[2]) : R(0);
  plane(d[7], d[10], d[9], d[8], C9 + R(2) * g[8] + (g[17] + g[18]), g[4], g[10] + g[13],
        g[11] - g[14], Fx + Fy, Fx - Fy, ux + uy, ux - uy);
  plane(d[11], d[14], d[13], d[12], C9 + (g[7] - g[8]) + (g[17] - g[18]), g[5], g[10] - g[13],
        g[12] + g[15], Fx + Fz, Fx - Fz, ux + uz, ux - uz);
  plane(d[15], d[18], d[17], d[16], C9 - (g[7] + g[8]) - R(2) * g[17], g[6], g[11] + g[14],
        g[12] - g[15], Fy + Fz, Fy - Fz, uy + uz, uy - uz);
}

// Compile-time checks of the additive back-transform: a unit g^_j adds
// column j of K, and the body-force correction equals the source
// w_a [3 e.F + 9 (e.u)(e.F) - 3 u.F] of every direction.
constexpr bool add_K_g_is_K() {
  for (int j = 4; j < Q; ++j) {
    double d[Q] = {}, g[Q] = {};
    const double F[3] = {0.0, 0.0, 0.0};
    g[j] = 1.0;
    add_K_g<double, false>(d, g, 0.0, 0.0, 0.0, F);
    for (int q = 0; q < Q; ++q)
      if (d[q] != double(kb(j, cx(q), cy(q), cz(q)))) return false;
  }
  return true;
}
constexpr bool add_K_g_source() {
  const double F[3] = {0.375, -0.625, 0.8125};
  const double u[3] = {0.25, 0.5, -0.125};
  double d[Q] = {}, g[Q] = {};
  add_K_g<double, true>(d, g, u[0], u[1], u[2], F);
  for (int q = 0; q < Q; ++q) {
    const double eF = cx(q) * F[0] + cy(q) * F[1] + cz(q) * F[2];
    const double eu = cx(q) * u[0] + cy(q) * u[1] + cz(q) * u[2];
    const double uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2];
    const double S = wt<double>(q) * (3.0 * eF + 9.0 * eu * eF - 3.0 * uF);
    const double diff = d[q] - S;
    if (diff > 1e-15 || diff < -1e-15) return false;
  }
  return true;
}
static_assert(add_K_g_is_K(), "the additive back-transform must add the columns of K");
static_assert(add_K_g_source(), "the additive back-transform must add the body-force source");

// gamma_dot^2 = (9 / rho^2) (omega^2 A + B) from Eq. strainratetensor (bulk
// rate omega_9) and Eq. shearrateexpression, for the non-equilibrium moments
// m^(1)_4..9 (Sec. 3.2): the traceless part gives
// A = (m7^2 - m7 m8 + m8^2) / 3 + m4^2 + m5^2 + m6^2 and the isotropic part
// B = omega_9^2 m9^2 / 6.
template <typename R, typename T>
__device__ __forceinline__ void strain_AB(const CollideConst<T>& C, R m4, R m5, R m6, R m7, R m8,
                                          R m9, R& A, R& B) {
  const R d = fma(m7, m7 - m8, mulr(m8, m8));
  A = fma(R(1.0 / 3.0), d, fma(m4, m4, fma(m5, m5, mulr(m6, m6))));
  B = mulr(mulr(R(C.cB), m9), m9);
}

// Collide one node with any relaxation rates omega_9..18 (collide_unit below
// takes the unit rates of Sec. 3.1).  d[19] holds the pre-collision deviations on entry and
// the post-collision deviations f~ - w rho0 on return.
// PAIR_OUT selects how the populations are written back: rebuilt from the
// pair values (fewer registers: the 19 inputs are dead after the pair values
// are formed), which is exact when the inputs are FP16 values decoded to FP32
// (sums of a few of them need no rounding), or as one correction added to
// each input population (add_K_g), which keeps FP32 populations to a single
// rounding per step.
//
// LOG2LAM: the deviations are carried scaled by lam = 2^LOG2LAM (the FP16
// storage scale), and C holds lam rho0, lam F, lam 3K and log(lam 3K).  All
// moments and g^ then scale with lam, rho becomes lam rho and 1/rho
// 1/(lam rho): every term is either linear in the deviations or a product
// whose factors of lam cancel (the attractors a_i a_j / rho, the strain rate
// of m^(1)/rho, the omega solve of 3K/rho), so the scaled populations come
// out exactly as lam times the unscaled ones up to rounding, and only rho
// is unscaled for the output.
template <typename R, bool FORCE, bool PAIR_OUT, int LOG2LAM>
__device__ __forceinline__ void collide_rates(const CollideConst<typename ScalarOf<R>::type>& C,
                                              R (&d)[Q], NodeOut<R>& out) {
  using T = typename ScalarOf<R>::type;
  // ---- mass and momentum (Eqs. hydrodynamicfields1/2) -------------------
  static_assert(cx(1) == 1 && cy(3) == 1 && cz(5) == 1 && cx(7) == 1 && cy(7) == 1 &&
                    cx(9) == 1 && cy(9) == -1 && cx(11) == 1 && cz(11) == 1 && cx(13) == 1 &&
                    cz(13) == -1 && cy(15) == 1 && cz(15) == 1 && cy(17) == 1 && cz(17) == -1,
                "pair members");
  Pairs<R> p = to_pairs(d);
  const R drho = p.d0 + (p.sAx + p.sAy + p.sAz) + (p.Dxxyy + p.Dxxzz + p.Dyyzz);
  const R jx = p.tAx + (p.Dxyy + p.Dxzz), jy = p.tAy + (p.Dxxy + p.Dyzz),
          jz = p.tAz + (p.Dxxz + p.Dyyz);
  const R rho = R(C.rhoS) + drho;
  const R rinv = rrcp<R>(rho);
  R ux, uy, uz;
  if (FORCE) {
    // Symmetric split of the body force: the velocity is (j + F/2)/rho and
    // half of the source is added before the collision, half after.
    ux = (jx + R(T(0.5) * C.FS[0])) * rinv;
    uy = (jy + R(T(0.5) * C.FS[1])) * rinv;
    uz = (jz + R(T(0.5) * C.FS[2])) * rinv;
    add_half_source(p, ux, uy, uz, C.FS);
  } else {
    ux = jx * rinv;
    uy = jy * rinv;
    uz = jz * rinv;
  }

  // ---- raw moments of the deviations (Eq. rawmomentdistributionfunction1)
  // k'_ii = rho0/3 + Dii, k'_ij = Dij, third order k' = D, k'_iijj = rho0/9 + D.
  const R Dxy = p.Dxy, Dxz = p.Dxz, Dyz = p.Dyz;
  const R Dxyy = p.Dxyy, Dxzz = p.Dxzz, Dxxy = p.Dxxy, Dyzz = p.Dyzz, Dxxz = p.Dxxz,
          Dyyz = p.Dyyz;
  const R Dxxyy = p.Dxxyy, Dxxzz = p.Dxxzz, Dyyzz = p.Dyyzz;
  const R Dxx = p.sAx + (Dxxyy + Dxxzz), Dyy = p.sAy + (Dxxyy + Dyyzz),
          Dzz = p.sAz + (Dxxzz + Dyyzz);

  const R ux2 = ux * ux, uy2 = uy * uy, uz2 = uz * uz;
  const R r3 = R(C.rhoS * T(1.0 / 3.0));
  const R kxx = r3 + Dxx, kyy = r3 + Dyy, kzz = r3 + Dzz;

  // ---- non-equilibrium second moments m^(1)_4..9 (Sec. 3.2) -------------
  const R m4 = Dxy - rho * ux * uy;
  const R m5 = Dxz - rho * ux * uz;
  const R m6 = Dyz - rho * uy * uz;
  const R m7 = (Dxx - Dyy) - rho * (ux2 - uy2);
  const R m8 = (Dxx - Dzz) - rho * (ux2 - uz2);
  const R m9 = (Dxx + Dyy + Dzz) - drho - rho * (ux2 + uy2 + uz2);

  R A, B;
  strain_AB(C, m4, m5, m6, m7, m8, m9, A, B);
  const R w = omega_nu(C, rho, rinv, A, B);

  // ---- change of moments, Eqs. collisionkernelg4..g18 --------------------
  // omega_4..8 = w (Sec. 3.1); omega_9..18 from the constants above (1 in Sec. 3.1).
  R g[Q];
  g[4] = R(-0.25) * w * m4;
  g[5] = R(-0.25) * w * m5;
  g[6] = R(-0.25) * w * m6;
  g[7] = R(-1.0 / 12.0) * w * m7;
  g[8] = R(-1.0 / 36.0) * w * (R(2) * m8 - m7);
  g[9] = R(C.c9) * m9;
  const R g4 = g[4], g5 = g[5], g6 = g[6], g7 = g[7], g8 = g[8], g9 = g[9];

  // g^_10..15 in +/- pairs: with the row sums
  //   Xy = ux k'yy - k'xyy + 2 uy k'xy - 2 rho ux uy^2 (and Xz, Yx, Yz, Zx, Zy
  //   alike), the bracket of g^_10 is Xy + Xz and that of g^_13 is Xy - Xz
  //   (k'yy - k'zz = Dyy - Dzz), and so on for 11/14 and 12/15.
  const R tux = R(2) * ux, tuy = R(2) * uy, tuz = R(2) * uz;
  const R rho2 = R(2) * rho;
  const R rx2 = rho2 * ux, ry2 = rho2 * uy, rz2 = rho2 * uz;
  const R Xy = ux * kyy - Dxyy + tuy * Dxy - rx2 * uy2;
  const R Xz = ux * kzz - Dxzz + tuz * Dxz - rx2 * uz2;
  const R Yx = uy * kxx - Dxxy + tux * Dxy - ry2 * ux2;
  const R Yz = uy * kzz - Dyzz + tuz * Dyz - ry2 * uz2;
  const R Zx = uz * kxx - Dxxz + tux * Dxz - rz2 * ux2;
  const R Zy = uz * kyy - Dyyz + tuy * Dyz - rz2 * uy2;
  const R a4y = uy * g4, a5z = uz * g5, a4x = ux * g4, a6z = uz * g6, a5x = ux * g5, a6y = uy * g6;
  const R hx = R(0.75) * ux, hy = R(0.75) * uy, hz = R(1.5) * uz;
  const R w9 = R(14) * g9;
  g[10] = R(C.c10) * (Xy + Xz) + (a4y + a5z) + hx * (w9 - (g7 + g8));
  g[13] = R(C.c13) * (Xy - Xz) + (a4y - a5z) + hx * (R(3) * g8 - g7);
  g[11] = R(C.c11) * (Yx + Yz) + (a4x + a6z) + hy * (w9 + (g7 - g8));
  g[14] = R(C.c14) * (Yz - Yx) + (a6z - a4x) - hy * (g7 + R(3) * g8);
  g[12] = R(C.c12) * (Zx + Zy) + (a5x + a6y) + hz * (g8 + R(7) * g9);
  g[15] = R(C.c15) * (Zx - Zy) + (a5x - a6y) + hz * g7;
  const R g10 = g[10], g11 = g[11], g12 = g[12], g13 = g[13], g14 = g[14], g15 = g[15];

  // Post-collision diagonal central moments k~ii = rho/3 + a_i (the <K g^|e_i^2>
  // rows of Eq. momentscascadedcollisionterm added to k'_ii - rho u_i^2), and
  // the factorised attractors k~ii k~jj / rho expanded around rho/3, so that
  // the rho0/9 of the raw fourth moments cancels analytically.
  const R third = R(1.0 / 3.0);
  const R ax = Dxx - third * drho - rho * ux2 + R(6) * g7 + R(6) * g8 + R(42) * g9;
  const R ay = Dyy - third * drho - rho * uy2 - R(6) * g7 + R(6) * g8 + R(42) * g9;
  const R az = Dzz - third * drho - rho * uz2 - R(12) * g8 + R(42) * g9;

  // The brackets b16..b18 of g^_16..18 are sums over the axis pairs (xy, xz,
  // yz) of one pair term each, e.g.
  //   Wxy = ax ay / rho - k'xxyy + 2 ux k'xyy + 2 uy k'xxy - ux^2 k'yy
  //         - uy^2 k'xx - 4 ux uy k'xy + 3 rho ux^2 uy^2,
  // with b16 = rho/3 - rho0/3 + 2/3 (ax + ay + az) + Wxy + Wxz + Wyz,
  // b17 = (2 ax - ay - az)/3 + Wxy + Wxz - 2 Wyz and b18 = (ay - az)/3 + Wxy - Wxz.
  const R uxy = ux * uy, uxz = ux * uz, uyz = uy * uz;
  const R rho3 = R(3) * rho;
  const R axr = ax * rinv, ayr = ay * rinv;
  const R Wxy = axr * ay - Dxxyy + tux * Dxyy + tuy * Dxxy - ux2 * kyy - uy2 * kxx -
                R(4) * uxy * Dxy + rho3 * (ux2 * uy2);
  const R Wxz = axr * az - Dxxzz + tux * Dxzz + tuz * Dxxz - ux2 * kzz - uz2 * kxx -
                R(4) * uxz * Dxz + rho3 * (ux2 * uz2);
  const R Wyz = ayr * az - Dyyzz + tuy * Dyzz + tuz * Dyyz - uy2 * kzz - uz2 * kyy -
                R(4) * uyz * Dyz + rho3 * (uy2 * uz2);
  const R b16 = third * drho + R(2.0 / 3.0) * (ax + ay + az) + (Wxy + Wxz + Wyz);
  const R b17 = third * (R(2) * ax - ay - az) + (Wxy + Wxz) - R(2) * Wyz;
  const R b18 = third * (ay - az) + (Wxy - Wxz);
  // shared products: ux uy g4, ux uz g5, uy uz g6 and ux g10, uy g11, uz g12
  const R p4 = ux * a4y, p5 = ux * a5z, p6 = uy * a6z;
  const R v10 = ux * g10, v11 = uy * g11, v12 = uz * g12;
  g[16] = R(C.c16) * b16 - R(4.0 / 3.0) * (p4 + p5 + p6) +
          R(0.5) * (ux2 - uy2) * g7 + R(0.5) * (ux2 + uy2 - R(2) * uz2) * g8 +
          (R(-7) * (ux2 + uy2 + uz2) - R(8)) * g9 + R(4.0 / 3.0) * (v10 + v11 + v12);
  g[17] = R(C.c17) * b17 - R(2.0 / 3.0) * (p4 + p5) + R(4.0 / 3.0) * p6 +
          R(0.25) * (ux2 - uy2 - R(3) * uz2 - R(2)) * g7 +
          R(0.25) * (ux2 - R(5) * uy2 + uz2 - R(2)) * g8 +
          R(1.75) * (R(-2) * ux2 + uy2 + uz2) * g9 + R(2.0 / 3.0) * v10 -
          third * (v11 + v12) - uy * g14 + uz * g15;
  g[18] = R(C.c18) * b18 - R(2) * (p4 - p5) +
          R(0.75) * (ux2 - uy2 + uz2 + R(2.0 / 3.0)) * g7 +
          R(0.75) * (R(-3) * ux2 - uy2 + uz2 - R(2)) * g8 + R(5.25) * (uz2 - uy2) * g9 +
          (v11 - v12) + R(2) * ux * g13 - uy * g14 - uz * g15;

  // ---- back-transform f~ = f + K g^ (+ second half of the source) --------
  if constexpr (PAIR_OUT) {
    if (FORCE) add_half_source(p, ux, uy, uz, C.FS);
    from_pairs(p, g, d);
  } else {
    add_K_g<R, FORCE>(d, g, ux, uy, uz, C.FS);
  }
  if constexpr (LOG2LAM != 0) out.rho = rho * R(T(1.0 / double(1 << LOG2LAM)));
  else out.rho = rho;
  out.ux = ux;
  out.uy = uy;
  out.uz = uz;
  out.gamma_dot = shear_rate(rinv, w, A, B);
}

// The reference of the F16R form: lam (rho - rho0) and lam 3 rho u of a node,
// as stored.  Its first-order equilibrium w_q [dr + e_q . v] has the moments
// dr (mass), v/3 (momentum), dr/3 (each D_ii), v_i/9 (D_ijj) and dr/9 (D_iijj).
template <typename R>
struct RefT {
  R dr, vx, vy, vz;
};

// The weights of that equilibrium.  A writer takes it off the moments, a
// reader puts it back population by population, and the two must agree in
// exact arithmetic: with every constant rounded to FP32 by itself they differ
// by (delta_36 - delta_6) v/3 = 3e-8 v/3 of momentum, and that drag in every step
// put 64^3 cavities 28 % further from FP64 after 2000 steps.  So 1/36 is cut to
// 22 bits, which leaves room for the factors 6, 12 and 24 that the moments
// take, and the other weights are multiples of it (the weights' sum stays 1);
// what the reference is exactly does not matter, as it is put back.
constexpr float REF_W = 14913080.0f / 536870912.0f;  // 1/36 (1 - 6e-8)
__host__ __device__ constexpr float ref_wt(int q) {
  return q == 0 ? 1.0f - 24.0f * REF_W : q <= 6 ? 2.0f * REF_W : REF_W;
}
static_assert(double(6.0f * REF_W) == 6.0 * double(REF_W) &&
                  double(12.0f * REF_W) == 12.0 * double(REF_W) &&
                  double(1.0f - 24.0f * REF_W) == 1.0 - 24.0 * double(REF_W),
              "the reference's moments must be exact multiples of its weights");
// collide_unit without a reference to subtract.
struct NoRef {};

// Collide one node with the rates omega_9..18 = 1 of Sec. 3.1, the default.
//
// With unit rates every third- and fourth-order central moment relaxes to its
// attractor in one step (Eqs. centralmomentrelaxation,
// discretecentralmomentattractors), so the post-collision raw moments follow
// from rho, u and the relaxed second-order central moments alone, and the
// brackets of g^_10..g^_18 need not be formed.  With J = rho u, the
// non-equilibrium moments m_ij = k'_ij - J_i u_j (m^(1)_4..6 of Sec. 3.2),
// s_i = D_ii - J_i u_i, their trace part m9 = s_x + s_y + s_z - (rho - rho0)
// (m^(1)_9) and traceless parts e_i = s_i - (s_x + s_y + s_z)/3 (m^(1)_7 and
// m^(1)_8 are differences of them):
//   c_ij  = (1 - omega) m_ij                 relaxed central moments, order 2
//   c_ii  = rho/3 + a_i, a_i = (1 - omega) e_i    (the trace relaxes fully)
//   k_ii  = c_ii + J_i u_i                   raw
//   k_iij = 2 u_i c_ij + u_j k_ii            raw, order 3 (central: 0)
//   k_iijj = c*_iijj + u_i^2 k_jj + u_j^2 c_ii + 4 u_i u_j c_ij
//            with the attractor c*_iijj = (rho/3 + a_i)(rho/3 + a_j)/rho,
// each taken relative to the rest state so that rho0/3 and rho0/9 cancel
// analytically.  The gamma_dot invariant of strain_AB is
// A = (e_x^2 + e_y^2 + e_z^2)/2 + m_xy^2 + m_xz^2 + m_yz^2, B = m9^2 / 6.
// Against collide_rates with the same rates this takes 232 FP operations per
// node instead of 424 (pair output; 240 instead of 475 with one correction
// per population), counted with every possible multiply-add fused.  What it
// gave: the FP64 step is bound by the FP64 pipe and went from 2030 to 978 us
// on 128^3 (with the solve above); on 256^3 FP32 went from 431 to 379 us a
// step (6.7 TB/s), F16S from 395 to 323 and F16R from 792 to 753 us, and the
// register-capped two-buffer FP32 and FP16 kernels of a lone lattice no longer spill
// (of unit rates, the batch's kernels spill 4 to 56 bytes, the capped FP32
// in-place check step 4, F16R's forced check step 8).
//
// PAIR_OUT, LOG2LAM and the body force's symmetric split are as in
// collide_rates.  With PAIR_OUT the populations are rebuilt from the raw
// moments; without it the moments' increments are added to the populations,
// one correction each.
// With a function for `ref` (PAIR_OUT, no force) the post-collision deviations
// come out less the first-order equilibrium of the reference ref(out): taken
// off the moments, that costs a dozen operations instead of one or two and a
// multiply-add per population.
template <typename R, bool FORCE, bool PAIR_OUT, int LOG2LAM, typename Ref = NoRef>
__device__ __forceinline__ void collide_unit(const CollideConst<typename ScalarOf<R>::type>& C,
                                             R (&d)[Q], NodeOut<R>& out, Ref ref = Ref{}) {
  using T = typename ScalarOf<R>::type;
  constexpr bool REF = !std::is_same<Ref, NoRef>::value;
  static_assert(!REF || (PAIR_OUT && !FORCE), "references are taken off rebuilt populations");
  const Pairs<R> p = to_pairs(d);
  // ---- mass, momentum, second moments (Eqs. hydrodynamicfields1/2) --------
  const R Dxx = p.sAx + (p.Dxxyy + p.Dxxzz), Dyy = p.sAy + (p.Dxxyy + p.Dyyzz),
          Dzz = p.sAz + (p.Dxxzz + p.Dyyzz);
  const R drho = (p.d0 + Dxx) + ((p.sAy + p.sAz) + p.Dyyzz);
  const R jx = p.tAx + (p.Dxyy + p.Dxzz), jy = p.tAy + (p.Dxxy + p.Dyzz),
          jz = p.tAz + (p.Dxxz + p.Dyyz);
  const R rho = R(C.rhoS) + drho;
  const R rinv = rrcp<R>(rho);
  R Jx = jx, Jy = jy, Jz = jz;
  if (FORCE) {
    // rho u = j + F/2
    Jx = jx + R(T(0.5) * C.FS[0]);
    Jy = jy + R(T(0.5) * C.FS[1]);
    Jz = jz + R(T(0.5) * C.FS[2]);
  }
  const R ux = mulr(Jx, rinv), uy = mulr(Jy, rinv), uz = mulr(Jz, rinv);
  if constexpr (LOG2LAM != 0) out.rho = mulr(rho, R(T(1.0 / double(1 << LOG2LAM))));
  else out.rho = rho;
  out.ux = ux;
  out.uy = uy;
  out.uz = uz;
  // half of the source S before the collision: S_ii = 2 u_i F_i, S_ij = u_i F_j + u_j F_i
  R Fx(0), Fy(0), Fz(0), hFx(0), hFy(0), hFz(0);
  R hxx = Dxx, hyy = Dyy, hzz = Dzz, hxy = p.Dxy, hxz = p.Dxz, hyz = p.Dyz;
  if (FORCE) {
    Fx = R(C.FS[0]), Fy = R(C.FS[1]), Fz = R(C.FS[2]);
    hFx = R(T(0.5) * C.FS[0]), hFy = R(T(0.5) * C.FS[1]), hFz = R(T(0.5) * C.FS[2]);
    hxx = fma(ux, Fx, hxx);
    hyy = fma(uy, Fy, hyy);
    hzz = fma(uz, Fz, hzz);
    hxy = fma(ux, hFy, fma(uy, hFx, hxy));
    hxz = fma(ux, hFz, fma(uz, hFx, hxz));
    hyz = fma(uy, hFz, fma(uz, hFy, hyz));
  }
  // ---- non-equilibrium second moments -------------------------------------
  const R third = R(T(1.0 / 3.0));
  const R sx = fma(-Jx, ux, hxx), sy = fma(-Jy, uy, hyy), sz = fma(-Jz, uz, hzz);
  const R mxy = fma(-Jx, uy, hxy), mxz = fma(-Jx, uz, hxz), myz = fma(-Jy, uz, hyz);
  const R tr = (sx + sy) + sz;
  const R m9 = tr - drho;
  const R ex = fma(-third, tr, sx), ey = fma(-third, tr, sy), ez = fma(-third, tr, sz);
  const R A = fma(R(T(0.5)), fma(ex, ex, fma(ey, ey, mulr(ez, ez))),
                  fma(mxy, mxy, fma(mxz, mxz, mulr(myz, myz))));
  const R B = mulr(mulr(R(T(1.0 / 6.0)), m9), m9);
  const R w = omega_nu(C, rho, rinv, A, B);

  // ---- relaxed second moments ------------------------------------------------
  const R wm = R(T(1.0)) - w;
  const R cxy = mulr(wm, mxy), cxz = mulr(wm, mxz), cyz = mulr(wm, myz);
  const R ax = mulr(wm, ex), ay = mulr(wm, ey), az = mulr(wm, ez);
  const R dr3 = mulr(third, drho);
  const R zx = fma(wm, ex, dr3), zy = fma(wm, ey, dr3), zz = fma(wm, ez, dr3);  // a_i + dr3
  const R Exx = fma(Jx, ux, zx), Eyy = fma(Jy, uy, zy), Ezz = fma(Jz, uz, zz);
  const R r30 = R(C.r30);
  const R kxx = Exx + r30, kyy = Eyy + r30, kzz = Ezz + r30;
  const R cxx = zx + r30, cyy = zy + r30;

  if constexpr (PAIR_OUT) {
    // a quarter of every plane moment (but for the products k_ij): the
    // populations of a plane are sums and differences of the four quarters
    // (plane_out)
    const R q4 = R(T(0.25)), h2 = R(T(0.5));
    const R qx = mulr(q4, ux), qy = mulr(q4, uy), qz = mulr(q4, uz);
    const R hx = mulr(h2, ux), hy = mulr(h2, uy), hz = mulr(h2, uz);
    R oxyy = mulr(qx, kyy), oxzz = mulr(qx, kzz), oxxy = mulr(qy, kxx), oyzz = mulr(qy, kzz),
      oxxz = mulr(qz, kxx), oyyz = mulr(qz, kyy);
    R ddr = mulr(R(T(1.0 / 36.0)), drho);
    R pxy = fma(Jx, uy, cxy), pxz = fma(Jx, uz, cxz), pyz = fma(Jy, uz, cyz);  // raw k_ij
    R fExx = Exx, fEyy = Eyy, fEzz = Ezz, fdr = drho;
    R gx = mulr(h2, jx), gy = mulr(h2, jy), gz = mulr(h2, jz);
    if constexpr (REF) {
      const RefT<R> r = ref(out);
      const R m6 = R(T(-6.0f * REF_W)), m36 = R(T(-REF_W)), m3 = R(T(-12.0f * REF_W));
      fdr = drho - r.dr;
      ddr = fma(m36, r.dr, ddr);
      fExx = fma(m3, r.dr, Exx);
      fEyy = fma(m3, r.dr, Eyy);
      fEzz = fma(m3, r.dr, Ezz);
      gx = fma(m6, r.vx, gx);
      gy = fma(m6, r.vy, gy);
      gz = fma(m6, r.vz, gz);
      const R vx = mulr(m36, r.vx), vy = mulr(m36, r.vy), vz = mulr(m36, r.vz);
      oxyy = fma(qx, kyy, vx);
      oxzz = fma(qx, kzz, vx);
      oxxy = fma(qy, kxx, vy);
      oyzz = fma(qy, kzz, vy);
      oxxz = fma(qz, kxx, vz);
      oyyz = fma(qz, kyy, vz);
    }
    if (FORCE) {
      // the other half of the source
      const R fx = R(T(C.FS[0]) * T(1.0 / 24.0)), fy = R(T(C.FS[1]) * T(1.0 / 24.0)),
              fz = R(T(C.FS[2]) * T(1.0 / 24.0));
      oxyy = fma(qx, kyy, fx);
      oxzz = fma(qx, kzz, fx);
      oxxy = fma(qy, kxx, fy);
      oyzz = fma(qy, kzz, fy);
      oxxz = fma(qz, kxx, fz);
      oyyz = fma(qz, kyy, fz);
      pxy = fma(ux, hFy, fma(uy, hFx, pxy));
      pxz = fma(ux, hFz, fma(uz, hFx, pxz));
      pyz = fma(uy, hFz, fma(uz, hFy, pyz));
      fExx = fma(ux, Fx, fExx);
      fEyy = fma(uy, Fy, fEyy);
      fEzz = fma(uz, Fz, fEzz);
      gx = fma(h2, jx, hFx);
      gy = fma(h2, jy, hFy);
      gz = fma(h2, jz, hFz);
      ddr = fma(R(T(1.0 / 12.0)), fma(ux, Fx, fma(uy, Fy, mulr(uz, Fz))), ddr);
    }
    oxyy = fma(hy, cxy, oxyy);
    oxzz = fma(hz, cxz, oxzz);
    oxxy = fma(hx, cxy, oxxy);
    oyzz = fma(hz, cyz, oyzz);
    oxxz = fma(hx, cxz, oxxz);
    oyyz = fma(hy, cyz, oyyz);
    // attractors: a quarter of (rho/3 + a_i)(rho/3 + a_j)/rho - rho0/9
    const R qr = mulr(q4, rinv), tw = R(T(1.0 / 12.0));
    const R by = fma(ay, qr, tw), bz = fma(az, qr, tw);
    const R ty = fma(tw, ay, ddr), tz = fma(tw, az, ddr);
    R fxy = fma(ax, by, ty), fxz = fma(ax, bz, tz), fyz = fma(ay, bz, tz);
    const R qxx = mulr(qx, ux), qyy = mulr(qy, uy), qzz = mulr(qz, uz);
    fxy = fma(mulr(ux, uy), cxy, fma(qyy, cxx, fma(qxx, kyy, fxy)));
    fxz = fma(mulr(ux, uz), cxz, fma(qzz, cxx, fma(qxx, kzz, fxz)));
    fyz = fma(mulr(uy, uz), cyz, fma(qzz, cyy, fma(qyy, kzz, fyz)));
    if (FORCE) {
      const R e8 = R(T(-0.125));
      fxy = fma(e8, mulr(uz, Fz), fxy);
      fxz = fma(e8, mulr(uy, Fy), fxz);
      fyz = fma(e8, mulr(ux, Fx), fyz);
    }
    const R m2 = R(T(-2.0));
    const R fs = fxy + fxz;
    d[0] = fma(R(T(4.0)), fs + fyz, fdr - ((fExx + fEyy) + fEzz));
    {
      const R hs = fma(m2, fs, mulr(h2, fExx)), ht = fma(m2, oxyy + oxzz, gx);
      d[1] = hs + ht;
      d[2] = hs - ht;
    }
    {
      const R hs = fma(m2, fxy + fyz, mulr(h2, fEyy)), ht = fma(m2, oxxy + oyzz, gy);
      d[3] = hs + ht;
      d[4] = hs - ht;
    }
    {
      const R hs = fma(m2, fxz + fyz, mulr(h2, fEzz)), ht = fma(m2, oxxz + oyyz, gz);
      d[5] = hs + ht;
      d[6] = hs - ht;
    }
    auto plane = [&](R f, R pr, R oi, R oj, R& Pp, R& Pm, R& Mp, R& Mm) {
      const R a = fma(q4, pr, f), b = fma(-q4, pr, f), c = oi + oj, e = oi - oj;
      Pp = a + c;
      Pm = a - c;
      Mp = b + e;
      Mm = b - e;
    };
    plane(fxy, pxy, oxyy, oxxy, d[7], d[10], d[9], d[8]);
    plane(fxz, pxz, oxzz, oxxz, d[11], d[14], d[13], d[12]);
    plane(fyz, pyz, oyzz, oyyz, d[15], d[18], d[17], d[16]);
  } else {
    // increments of the moments (with the whole source S): n = -omega m + S and r
    // of order 2, t of order 3, q of order 4
    const R nw = -w;
    R nxy(0), nxz(0), nyz(0);  // the source's part of n (see plane)
    const R m93 = mulr(third, m9);
    R rx = fma(nw, ex, -m93), ry = fma(nw, ey, -m93), rz = fma(nw, ez, -m93);
    const R tux = ux + ux, tuy = uy + uy, tuz = uz + uz;
    R bx = -p.Dxyy, cx_ = -p.Dxzz, by_ = -p.Dxxy, cy_ = -p.Dyzz, bz_ = -p.Dxxz, cz_ = -p.Dyyz;
    R dr9 = mulr(R(T(1.0 / 9.0)), drho);
    if (FORCE) {
      const R s6 = R(T(1.0 / 6.0));
      bx = fma(Fx, s6, -p.Dxyy);
      cx_ = fma(Fx, s6, -p.Dxzz);
      by_ = fma(Fy, s6, -p.Dxxy);
      cy_ = fma(Fy, s6, -p.Dyzz);
      bz_ = fma(Fz, s6, -p.Dxxz);
      cz_ = fma(Fz, s6, -p.Dyyz);
      nxy = fma(ux, Fy, fma(uy, Fx, mulr(nw, mxy)));
      nxz = fma(ux, Fz, fma(uz, Fx, mulr(nw, mxz)));
      nyz = fma(uy, Fz, fma(uz, Fy, mulr(nw, myz)));
      rx = fma(tux, Fx, rx);
      ry = fma(tuy, Fy, ry);
      rz = fma(tuz, Fz, rz);
      dr9 = fma(third, fma(ux, Fx, fma(uy, Fy, mulr(uz, Fz))), dr9);
    }
    const R txyy = fma(tuy, cxy, fma(ux, kyy, bx)), txzz = fma(tuz, cxz, fma(ux, kzz, cx_));
    const R txxy = fma(tux, cxy, fma(uy, kxx, by_)), tyzz = fma(tuz, cyz, fma(uy, kzz, cy_));
    const R txxz = fma(tux, cxz, fma(uz, kxx, bz_)), tyyz = fma(tuy, cyz, fma(uz, kyy, cz_));
    const R by = fma(ay, rinv, third), bz = fma(az, rinv, third);
    const R ty = fma(third, ay, dr9), tz = fma(third, az, dr9);
    const R ux2 = mulr(ux, ux), uy2 = mulr(uy, uy), uz2 = mulr(uz, uz);
    R qxy = fma(ax, by, ty - p.Dxxyy), qxz = fma(ax, bz, tz - p.Dxxzz),
      qyz = fma(ay, bz, tz - p.Dyyzz);
    qxy = fma(mulr(tux, tuy), cxy, fma(uy2, cxx, fma(ux2, kyy, qxy)));
    qxz = fma(mulr(tux, tuz), cxz, fma(uz2, cxx, fma(ux2, kzz, qxz)));
    qyz = fma(mulr(tuy, tuz), cyz, fma(uz2, cyy, fma(uy2, kzz, qyz)));
    if (FORCE) {
      const R h2 = R(T(-0.5));
      qxy = fma(h2, mulr(uz, Fz), qxy);
      qxz = fma(h2, mulr(uy, Fy), qxz);
      qyz = fma(h2, mulr(ux, Fx), qyz);
    }
    const R qs = qxy + qxz, half = R(T(0.5));
    d[0] = d[0] + ((qs + qyz) - ((rx + ry) + rz));
    {
      const R e = rx - qs;
      const R o = FORCE ? Fx - (txyy + txzz) : -(txyy + txzz);
      d[1] = fma(half, e + o, d[1]);
      d[2] = fma(half, e - o, d[2]);
    }
    {
      const R e = ry - (qxy + qyz);
      const R o = FORCE ? Fy - (txxy + tyzz) : -(txxy + tyzz);
      d[3] = fma(half, e + o, d[3]);
      d[4] = fma(half, e - o, d[4]);
    }
    {
      const R e = rz - (qxz + qyz);
      const R o = FORCE ? Fz - (txxz + tyyz) : -(txxz + tyyz);
      d[5] = fma(half, e + o, d[5]);
      d[6] = fma(half, e - o, d[6]);
    }
    auto plane = [&](R q, R n, R m, R ti, R tj, R& Pp, R& Pm, R& Mp, R& Mm) {
      const R a = FORCE ? q + n : fma(nw, m, q), b = FORCE ? q - n : fma(w, m, q);
      const R c = ti + tj, e = ti - tj, f = R(T(0.25));
      Pp = fma(f, a + c, Pp);
      Pm = fma(f, a - c, Pm);
      Mp = fma(f, b + e, Mp);
      Mm = fma(f, b - e, Mm);
    };
    plane(qxy, nxy, mxy, txyy, txxy, d[7], d[10], d[9], d[8]);
    plane(qxz, nxz, mxz, txzz, txxz, d[11], d[14], d[13], d[12]);
    plane(qyz, nyz, myz, tyzz, tyyz, d[15], d[18], d[17], d[16]);
  }
  out.gamma_dot = shear_rate(rinv, w, A, B);
}

// rho, u and, when want_gd, |gamma_dot| of a node without colliding it, for
// any rates (only omega_9 enters).  d holds the pre-collision deviations.
template <typename R, bool FORCE, int LOG2LAM>
__device__ __forceinline__ void node_fields(const CollideConst<R>& C, const R (&d)[Q],
                                            bool want_gd, NodeOut<R>& out) {
  const Pairs<R> p = to_pairs(d);
  const R Dxx = p.sAx + (p.Dxxyy + p.Dxxzz), Dyy = p.sAy + (p.Dxxyy + p.Dyyzz),
          Dzz = p.sAz + (p.Dxxzz + p.Dyyzz);
  const R drho = (p.d0 + Dxx) + ((p.sAy + p.sAz) + p.Dyyzz);
  R Jx = p.tAx + (p.Dxyy + p.Dxzz), Jy = p.tAy + (p.Dxxy + p.Dyzz),
    Jz = p.tAz + (p.Dxxz + p.Dyyz);
  const R rho = C.rhoS + drho;
  const R rinv = rrcp<R>(rho);
  if (FORCE) {
    Jx = Jx + R(0.5) * C.FS[0];
    Jy = Jy + R(0.5) * C.FS[1];
    Jz = Jz + R(0.5) * C.FS[2];
  }
  const R ux = mulr(Jx, rinv), uy = mulr(Jy, rinv), uz = mulr(Jz, rinv);
  if (LOG2LAM != 0) out.rho = mulr(rho, R(1.0 / double(1 << LOG2LAM)));
  else out.rho = rho;
  out.ux = ux;
  out.uy = uy;
  out.uz = uz;
  if (!want_gd) return;
  R hxx = Dxx, hyy = Dyy, hzz = Dzz, hxy = p.Dxy, hxz = p.Dxz, hyz = p.Dyz;
  if (FORCE) {  // half of the source, as in collide_unit
    const R hFx = R(0.5) * C.FS[0], hFy = R(0.5) * C.FS[1], hFz = R(0.5) * C.FS[2];
    hxx = fma(ux, C.FS[0], hxx);
    hyy = fma(uy, C.FS[1], hyy);
    hzz = fma(uz, C.FS[2], hzz);
    hxy = fma(ux, hFy, fma(uy, hFx, hxy));
    hxz = fma(ux, hFz, fma(uz, hFx, hxz));
    hyz = fma(uy, hFz, fma(uz, hFy, hyz));
  }
  const R sx = fma(-Jx, ux, hxx), sy = fma(-Jy, uy, hyy), sz = fma(-Jz, uz, hzz);
  const R tr = (sx + sy) + sz;
  R A, B;
  strain_AB(C, fma(-Jx, uy, hxy), fma(-Jx, uz, hxz), fma(-Jy, uz, hyz), sx - sy, sx - sz,
            tr - drho, A, B);
  out.gamma_dot = shear_rate(rinv, omega_nu(C, rho, rinv, A, B), A, B);
}

// UNIT: the rates omega_9..18 are all 1 (PhysParams::unit_rates).
template <typename R, bool FORCE, bool PAIR_OUT, int LOG2LAM, bool UNIT>
__device__ __forceinline__ void collide(const CollideConst<typename ScalarOf<R>::type>& C,
                                        R (&d)[Q], NodeOut<R>& out) {
  if constexpr (UNIT) collide_unit<R, FORCE, PAIR_OUT, LOG2LAM>(C, d, out);
  else collide_rates<R, FORCE, PAIR_OUT, LOG2LAM>(C, d, out);
}

}  // namespace clbm
