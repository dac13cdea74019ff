// fp64_fast.cuh -- double-precision building blocks for a chip whose FP64 pipe
// runs at 1/64 of the FP32 rate (GB300: two FP64 lanes an SM and clock,
// conversions between float and double included).
//
// What the FP64 kernels pay for is therefore the number of instructions on that
// pipe; everything that only has to be approximately right -- a reciprocal's
// seed, a root's start, a Newton step's derivative -- is done in FP32, and the
// conversions on the way by integer operations on the bits.  The final value of
// each helper carries FP64 accuracy (stated with it).
#pragma once
#include <cuda_runtime.h>

#include "float_bits.h"
#include "mg_model.cuh"
#include "sweep32.cuh"

namespace mg {

// double -> float by bits, truncated (relative error below 2^-23), for seeds and
// Newton steps: 0 below 2^-126, NaN from 2^128 on (and for inf and NaN).
__device__ __forceinline__ float d2f_bits(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned a = hi & 0x7fffffffu;
  const unsigned m = __funnelshift_l(lo, a, 3) - (896u << 23);
  const unsigned r = a < (897u << 20) ? 0u : (a >= (1151u << 20) ? 0x7fffffffu : m);
  return __uint_as_float(r | (hi & 0x80000000u));
}

// double -> float as the conversion instruction rounds it: by bits where the result is
// zero or normal, by the instruction elsewhere (a call: as an expression the compiler
// converts every value and selects, 11 us of a CQ residual's 58 at 128^3).
static __device__ __noinline__ float d2f_call(double d) { return (float)d; }
__device__ __forceinline__ float d2f_nearest(double d) {
  bool ok;
  const unsigned r = d2f_nearest_bits((unsigned)__double2hiint(d), (unsigned)__double2loint(d), &ok);
  if (ok) return __uint_as_float(r);
  return d2f_call(d);
}

// float -> double by bits, exact for normal numbers; 0 and subnormals give 0
// (inf and NaN give a number beyond the float range, which callers reject).
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
  if (a < 0x00800000u) return 0.0;
  return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + (896u << 20))), (int)(b << 29));
}

// a / b to about one ulp: FP32 reciprocal seed, one Newton refinement (relative
// error 2^-45), quotient and its exact remainder.  Five FP64 instructions; for b
// outside the range where the seed is a normal float the plain division.
__device__ __forceinline__ double div_fast(double a, double b) {
  const float bf = d2f_bits(b), ab = fabsf(bf);
  if (!(ab > 1e-30f && ab < 1e30f)) return a / b;
  const double y0 = f2d_bits(frcp(bf));
  const double y = fma(y0, fma(-b, y0, 1.0), y0);
  const double q = a * y;
  return fma(fma(-b, q, a), y, q);
}

// Positive root of x^m + p x + q (q < 0; m = n + 2 of f(R) kind K, 3 for the
// symmetron): Newton's method in FP64 from the FP32 root x0.  The polynomial is
// evaluated in FP64 (two or three instructions), the step f / f' in FP32: a step
// of relative size d leaves at most d^2 (the curvature) + 3e-7 d (the FP32
// quotient), so the result is at FP64 rounding once d <= 1e-10.  From the
// closed-form start (1e-6) the second step is ~1e-12.  False (x unspecified) if
// that is not reached or x leaves the branch: the caller takes the FP64 closed
// form.
template <int K>
__device__ __forceinline__ bool newton_root64(double p, double q, float pf, float x0, double* out) {
  if (!(fabsf(x0) > 1e-30f && fabsf(x0) < 1e30f)) return false;
  double x = f2d_bits(x0);
  float xf = x0;
#pragma unroll 1
  for (int it = 0; it < 4; ++it) {
    double f;
    float df;
    if constexpr (K == KFR0) {
      f = fma(x + p, x, q);
      df = 2.f * xf + pf;
    } else if constexpr (K == KFR2) {
      const double x2 = x * x;
      f = fma(x2, x2, fma(p, x, q));
      df = 4.f * xf * xf * xf + pf;
    } else {
      f = fma(fma(x, x, p), x, q);
      df = 3.f * xf * xf + pf;
    }
    const float d = d2f_bits(f) * frcp(df);
    x -= f2d_bits(d);
    xf -= d;
    if (it > 0 && fabsf(d) <= 1e-10f * fabsf(xf)) {
      *out = x;
      return xf * x0 > 0.f;
    }
  }
  return false;
}

// Level constants of the FP64 kernels (the model's, folded with the cell size).
struct Const64 {
  double kap;              // f(R), symmetron: c~^2 / h^2; CQ: 1 / h^2
  double al, al_om, p0;    // f(R): p = al_om rho + p0 - al S - L/6
  double q;                // f(R): -al K
  double om_a, c0, K;      // f(R): N = -kap (L - 6w) + om_a rho + c0 - K/u
  double g12, g2, xi2;     // symmetron: p = rat3 rho + g12, q = -g2 L + xi2 S
  double rat3, msym;
  double ic2, phibar, iphi, pot0, e1, src, pot, beta_ic2;  // CQ
  double pc[6];            // CQ: binomial coefficients of (1 + d)^{-1-alpha} - 1 = d (pc0 + d (pc1 + ...))
  float s, is1;            // f(R): the root's scale (al K)^{1/(n+2)} and 1/s^{n+1}
  int keep_exp;
};

static inline Const64 make_const64(const ModelDev& m, double h) {
  Const64 c = {};
  const double ih2 = 1.0 / (h * h);
  c.kap = m.c2 * ih2;
  if (is_fr(m.kind)) {
    const int np1 = m.kind + 1;
    c.al = h * h / (6.0 * m.c2);
    c.al_om = c.al * m.om_a;
    c.p0 = c.al * (m.K0 - m.om_a);
    c.q = -c.al * m.K;
    c.om_a = m.om_a;
    c.c0 = m.K0 - m.om_a;
    c.K = m.K;
    const double sc = pow(c.al * m.K, 1.0 / (double)(np1 + 1));
    c.s = (float)sc;
    c.is1 = (float)pow(sc, -(double)np1);
  } else if (m.kind == KSYM) {
    const double g = m.c2 * m.xi2_a2 * ih2;
    c.g12 = 12.0 * g - 1.0;
    c.g2 = 2.0 * g;
    c.xi2 = 2.0 * m.xi2_a2;
    c.rat3 = m.rat3;
    c.msym = m.msym;
  } else {
    c.kap = ih2;
    c.ic2 = 1.0 / m.c2;
    c.phibar = m.phibar;
    c.iphi = 1.0 / m.phibar;
    c.pot0 = m.pot0;
    c.e1 = -1.0 - m.alpha;
    c.src = m.cq_src;
    c.pot = m.cq_pot;
    c.beta_ic2 = m.beta / m.c2;
    c.keep_exp = m.keep_exp;
    double b = 1.0;
    for (int k = 0; k < 6; ++k) {
      b *= (c.e1 - k) / (k + 1);
      c.pc[k] = b;
    }
  }
  return c;
}

// CQ: px = (phibar + u/c~^2)^{-1-alpha} and its difference from the background
// value, with d = u / (c~^2 phibar).  For |d| <= 2^-10 (the field is ~1e-6 of
// phibar on every mesh that resolves structure) the binomial series to d^6:
// its first neglected term is below 2^-56 relative for alpha <= 2; above, pow.
__device__ __forceinline__ void cq_power(const Const64& c, double u, double* x, double* dpot) {
  *x = fma(u, c.ic2, c.phibar);
  const double d = u * c.ic2 * c.iphi;
  if (fabs(d) <= 0x1p-10 && c.e1 >= -3.0) {
    double t = c.pc[5];
#pragma unroll
    for (int k = 4; k >= 0; --k) t = fma(t, d, c.pc[k]);
    *dpot = c.pot0 * (t * d);
  } else {
    *dpot = pow(*x, c.e1) - c.pot0;
  }
}

// N_h(u) at one cell from its neighbours' sum (mg_model.cuh has the operators).
template <int K>
__device__ __forceinline__ double local_N64(const Const64& c, double u, double rho, double L) {
  if constexpr (is_fr(K)) {
    const double w = fr_w<K>(u);
    return fma(-c.kap, fma(-6.0, w, L), fma(c.om_a, rho, c.c0)) - div_fast(c.K, u);
  } else if constexpr (K == KSYM) {
    return fma(c.kap, fma(-6.0, u, L), -c.msym * (fma(u, u, fma(rho, c.rat3, -1.0)) * u));
  } else {
    const double E = c.keep_exp ? exp(c.beta_ic2 * u) : 1.0;
    double x, dp;
    cq_power(c, u, &x, &dp);
    return fma(c.kap, fma(-6.0, u, L), fma(c.pot, dp, -c.src * fma(E, rho, -1.0)));
  }
}

// Gauss-Seidel update of one cell: the exact local root for f(R) and the
// symmetron (nonlinear GS, Secs. 3.2.4-3.2.5), one Newton step for CQ
// (Eq. relaxation_iteration, Sec. 3.2.3).  The FAS source S enters p (f(R))
// or q (symmetron) of the local polynomial.
// The root: closed form in FP32, then newton_root64 -- about 15 FP64-pipe
// instructions an update for f(R) n = 1, neighbour sum included, where the FP64
// closed form with its library cube root, square root and cosine takes ~150.
template <int K>
__device__ __forceinline__ double local_update64(const Const64& c, double u, double rho, double S, double L) {
  if constexpr (is_fr(K)) {
    const double p = fma(L, -1.0 / 6.0, fma(-c.al, S, fma(c.al_om, rho, c.p0)));
    const float pf = d2f_bits(p);
    double x;
    if (newton_root64<K>(p, c.q, pf, c.s * fr_root_scaled_fast<K>(pf * c.is1), &x)) return x;
    return fr_root<K>(p, c.q);
  } else if constexpr (K == KSYM) {
    const double p = fma(rho, c.rat3, c.g12);
    const double q = fma(-c.g2, L, c.xi2 * S);
    const float pf = d2f_bits(p), qf = d2f_bits(q);
    double x;
    // the start has the sign opposite to q, which a q below the float range would not show
    if (fabsf(qf) > 1e-30f && newton_root64<K>(p, q, pf, sym_root_fast(pf, qf, 1.f), &x)) return x;
    return sym_root(p, q, u);
  } else {
    double x, dp;
    cq_power(c, u, &x, &dp);
    const double E = c.keep_exp ? exp(c.beta_ic2 * u) : 1.0;
    const double dE = c.keep_exp ? c.beta_ic2 * E : 0.0;
    const double r = fma(c.kap, fma(-6.0, u, L), fma(c.pot, dp, -c.src * fma(E, rho, -1.0))) - S;
    const double dr = -6.0 * c.kap - c.src * dE * rho + c.pot * c.e1 * c.ic2 * div_fast(c.pot0 + dp, x);
    return u - div_fast(r, dr);
  }
}

}  // namespace mg
