// adjoint.cu -- gradients of a loss through the scalar-field solve.
//
// The solve defines u*(delta, theta) by N(u*; delta, theta) = 0 (the discrete
// equations of Eq. fR_eom_codeunit2 / Eq. sym_eom_code_unit, theta =
// ln|f_R0|).  For a loss l(u*) with g = dl/du*, the adjoint field lambda solves
// J^T lambda = g with J = dN/du at u*, and
//   dl/d delta = -(dN/d delta)^T lambda,   dl/d theta = -lambda . dN/d theta.
// With Delta_h the 7-point Laplacian (symmetric) the transposed problem takes
// one screened-Poisson form for both models,
//   -kappa Delta_h lambda + m lambda = sigma g,
//   f(R):      J = -c^2 Delta_h diag((n+1)u^n) + diag(K/u^2), so
//              kappa = c~^2, m = K/((n+1)u^{n+2}), sigma = 1/((n+1)u^n);
//   symmetron: J = c^2 Delta_h - diag(msym (rho a*^3/a^3 - 1 + 3u^2)), so
//              kappa = c~^2, m = msym (rho a*^3/a^3 - 1 + 3u^2), sigma = -1;
// m > 0 in both (the f(R) field is positive; in the symmetron's broken phase
// rho a*^3/a^3 - 1 + 3u^2 = 2u^2 at the local minimum), so the operator is
// symmetric positive definite and red-black Gauss-Seidel multigrid converges.
//
// Solver: FP64 outer residual r = sigma g - A lambda on the fine level, FP32
// correction-scheme V-cycles for A e = r (the same cycle shape, restriction
// and prolongation as the forward solve), lambda += e.  The coarse-level mass
// is the 8-child mean of the fine mass, rebuilt from u* on every call (no state
// of the forward V-cycles is kept).
#include <math.h>
#include <string.h>

#include <chrono>
#include <mutex>

#include "adjoint_levels.h"
#include "ff.cuh"
#include "fp64_fast.cuh"
#include "mg_common.cuh"
#include "mg_internal.h"
#include "sweep32.cuh"

namespace mg {

// ---- per-cell coefficients from the converged field ----

// 1 / x to about half an ulp: FP32 seed y of relative error e <= 2^-22 and the first
// terms of 1 / (1 - e) = 1 + e + e^2 + ..., which leave e^3 (three FP64 instructions,
// where a division takes three times that on a pipe of 1/64 of the FP32 rate); outside
// the range of the seed the division.
__device__ __forceinline__ double rcp_fast(double x) {
  const float xf = d2f_bits(x), ax = fabsf(xf);
  if (!(ax > 1e-30f && ax < 1e30f)) return 1.0 / x;
  const double y = f2d_bits(frcp(xf)), e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// m64, m32 = mass; rhs = sigma * g (FP64); dinv = 1 / (6 kh + m), the inverse
// diagonal; b = float(rhs), the first residual (lambda starts at zero), and
// per-block partial sums of rhs^2, its normaliser.  SPLIT: the FP32 arrays in the
// red-black split layout.  A thread takes the cells k = 2q, 2q + 1 of a row, which
// sit at q of the two colours.  One reciprocal a cell, the powers of 1/u are
// products: ten FP64 instructions for f(R) n = 1, which bound it (512^3: 2.6 ms; 6.5 ms with three divisions).
template <int K, bool SPLIT>
__global__ void __launch_bounds__(kThreads) k_adj_setup(ModelDev m, int n, float kh, const double* __restrict__ u,
                                                        const float* __restrict__ rho32,
                                                        const double* __restrict__ rho_sum,
                                                        const double* __restrict__ g, double* __restrict__ m64,
                                                        float* __restrict__ m32, float* __restrict__ dinv,
                                                        double* __restrict__ rhs, float* __restrict__ b,
                                                        double* __restrict__ partials) {
  const double sl = K == KSYM ? m.msym * m.rat3 * block_ratio((double)n * n * n, rho_sum) : 0.0;
  const double Kn = m.K / (K + 1), inp1 = 1.0 / (K + 1);
  const int h = n >> 1;
  const long long H = (long long)n * n * h;
  double acc = 0.0;
  for (int row = blockIdx.x; row < n * n; row += gridDim.x) {
    const int c0 = (row / n + row % n) & 1;  // colour of the even cells
    for (int q = threadIdx.x; q < h; q += blockDim.x) {
      const long long t = (long long)row * n + 2 * q;
      double mass[2], r[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double uc = u[t + c], gc = g[t + c];
        if constexpr (is_fr(K)) {
          const double ru = rcp_fast(uc), ru2 = ru * ru;
          mass[c] = K == KFR0 ? Kn * ru2 : (K == KFR1 ? Kn * ru2 * ru : Kn * ru2 * ru2);
          r[c] = K == KFR0 ? gc : inp1 * (K == KFR1 ? ru : ru2) * gc;
        } else {
          mass[c] = fma(sl, (double)rho32[t + c], m.msym * fma(3.0 * uc, uc, -1.0));
          r[c] = -gc;
        }
        acc = fma(r[c], r[c], acc);
      }
      *reinterpret_cast<double2*>(m64 + t) = make_double2(mass[0], mass[1]);
      *reinterpret_cast<double2*>(rhs + t) = make_double2(r[0], r[1]);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const long long o = SPLIT ? (long long)(c0 ^ c) * H + (long long)row * h + q : t + c;
        const float mf = d2f_nearest(mass[c]);
        m32[o] = mf;
        dinv[o] = 1.f / (6.f * kh + mf);
        b[o] = d2f_nearest(r[c]);
      }
    }
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// r = rhs - (-kappa Delta_h lambda + m lambda) on the fine level (FP64);
// writes b = float(r) and per-block partial sums of r^2.
__global__ void k_adj_residual64(int n, double kappa, const double* __restrict__ lam, const double* __restrict__ m64,
                                 const double* __restrict__ rhs, float* __restrict__ b,
                                 double* __restrict__ partials) {
  double acc = 0.0;
  for (int r = blockIdx.x; r < n * n; r += gridDim.x) {
    const int i = r / n, j = r - (r / n) * n;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const size_t t = cidx(n, i, j, k);
      const double L = lam[cidx(n, wrapi(i + 1, n), j, k)] + lam[cidx(n, wrapi(i - 1, n), j, k)] +
                       lam[cidx(n, i, wrapi(j + 1, n), k)] + lam[cidx(n, i, wrapi(j - 1, n), k)] +
                       lam[cidx(n, i, j, wrapi(k + 1, n))] + lam[cidx(n, i, j, wrapi(k - 1, n))];
      const double lc = lam[t];
      const double v = rhs[t] - (-kappa * (L - 6.0 * lc) + m64[t] * lc);
      b[t] = (float)v;
      acc += v * v;
    }
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// d 2^ex as float-float.  lambda and the right-hand side enter float-float
// arithmetic times a power of two that brings them near 1 whatever the scale of
// the loss (float-float drops what lies below 2^-74).
__device__ __forceinline__ ff ff_from_double_scaled(double d, int ex) {
  const int hi = __double2hiint(d), e = ((hi >> 20) & 0x7ff) + ex;
  if ((hi & 0x7ff00000) == 0x7ff00000) return ff{__int_as_float(0x7fffffff), 0.f};  // inf, NaN
  if (e < 1 || (hi & 0x7ff00000) == 0) return ff{0.f, 0.f};
  return ff_from_double(__hiloint2double((hi & 0x800fffff) | (min(e, 0x7fe) << 20), __double2loint(d)));
}

// The same fine-level residual in float-float arithmetic (lambda, m and rhs
// split exactly from FP64; ~2^-48 per operation), C adjacent cells per thread
// (C = 2 on 8 x 64 tiles where the side allows, else 1 on 8 x 32): z-marching
// tiles with a four-slot ring of lambda in shared memory, so that one barrier a
// plane suffices, the next plane's lambda in flight while a plane is computed.
// Writes b = float(2^ex r), in the red-black split layout if SPLIT, and per-block
// partial sums of its square.  512^3: 1.00 ms (1.48 ms with one cell a thread, two
// barriers a plane and a normalised sum of the neighbours).
template <int TJ, int C, bool SPLIT, typename IT>
__global__ void __launch_bounds__(TJ * 32) k_adj_residual_ff(int n, int chunk, int ex, ff kappa,
                                                             const double* __restrict__ lam,
                                                             const double* __restrict__ m64,
                                                             const double* __restrict__ rhs, float* __restrict__ b,
                                                             double* __restrict__ partials) {
  constexpr int TK = 32 * C, NT = TJ * 32;
  constexpr int RW = TK + 2, RS = RW + (RW & 1) + 2;  // halo row k0-1 .. k0+TK; its element x at x + 1
  constexpr int PE = (TJ + 2) * RW, PS = (TJ + 2) * RS, NE = (PE + NT - 1) / NT;
  __shared__ __align__(16) float2 s_l[4][PS];
  const int tiles_k = n / TK;
  const int k0 = (blockIdx.x % tiles_k) * TK, j0 = (blockIdx.x / tiles_k) * TJ;
  const int i0 = blockIdx.y * chunk, i1 = min(i0 + chunk, n);
  const int t = threadIdx.x, ty = t >> 5, tx = t & 31;
  const int jg = j0 + ty, kg = k0 + C * tx;
  const int cc = (ty + 1) * RS + C * tx + 2;
  const IT nn = (IT)n * n;
  IT off[NE];
  int pos[NE];
#pragma unroll
  for (int m = 0; m < NE; ++m) {
    const int c = t + m * NT;
    const int y = c / RW, x = c - y * RW;
    off[m] = c < PE ? (IT)wrapi(j0 + y - 1, n) * n + wrapi(k0 + x - 1, n) : 0;
    pos[m] = c < PE ? y * RS + x + 1 : -1;
  }
  double pre[NE];
  auto fetch = [&](int p) {
    const int ig = p < 0 ? p + n : (p >= n ? p - n : p);
    const double* base = lam + (IT)ig * nn;
#pragma unroll
    for (int m = 0; m < NE; ++m) pre[m] = pos[m] >= 0 ? base[off[m]] : 0.0;
  };
  auto commit = [&](int slot) {
#pragma unroll
    for (int m = 0; m < NE; ++m)
      if (pos[m] >= 0) {
        const ff v = ff_from_double_scaled(pre[m], ex);
        s_l[slot][pos[m]] = make_float2(v.hi, v.lo);
      }
  };
  float acc = 0.f;
  fetch(i0 - 1);
  commit((i0 - 1) & 3);
  fetch(i0);
  commit(i0 & 3);
  fetch(i0 + 1);
  for (int i = i0; i < i1; ++i) {
    const IT g = (IT)i * nn + (IT)jg * n + kg;
    double R[C], Mv[C];
    if constexpr (C == 2) {
      const double2 r2 = *reinterpret_cast<const double2*>(rhs + g), m2 = *reinterpret_cast<const double2*>(m64 + g);
      R[0] = r2.x;
      R[1] = r2.y;
      Mv[0] = m2.x;
      Mv[1] = m2.y;
    } else {
      R[0] = rhs[g];
      Mv[0] = m64[g];
    }
    commit((i + 1) & 3);
    __syncthreads();
    if (i + 2 <= i1) fetch(i + 2);
    const int sm = (i - 1) & 3, sl = i & 3, sp = (i + 1) & 3;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int q = cc + c;
      auto add = [&](ffacc& a, float2 v) { acc_add(a, v.x, v.y); };
      const float2 lc = s_l[sl][q], w = s_l[sm][q];
      ffacc La = {w.x, w.y};
      add(La, s_l[sp][q]);
      add(La, s_l[sl][q - RS]);
      add(La, s_l[sl][q + RS]);
      add(La, s_l[sl][q - 1]);
      add(La, s_l[sl][q + 1]);
      const ff l6 = two_prod(lc.x, -6.f);
      acc_add(La, l6.hi, __fmaf_rn(lc.y, -6.f, l6.lo));
      const ff L = acc_ff(La);
      // r = rhs + kappa (L - 6 lambda) - m lambda
      ffacc r = acc_of(ff_from_double_scaled(R[c], ex));
      const ff p = two_prod(kappa.hi, L.hi);
      acc_add(r, p.hi, __fmaf_rn(kappa.hi, L.lo, __fmaf_rn(kappa.lo, L.hi, p.lo)));
      const ff mm = ff_from_double(Mv[c]);
      const ff z = two_prod(mm.hi, lc.x);
      acc_add(r, -z.hi, -__fmaf_rn(mm.hi, lc.y, __fmaf_rn(mm.lo, lc.x, z.lo)));
      const float rv = acc_float(r);
      if constexpr (SPLIT) {
        const int colour = (i + jg + kg + c) & 1;
        b[(IT)colour * ((IT)(n >> 1) * nn) + ((IT)i * n + jg) * (n >> 1) + (kg >> 1)] = rv;
      } else {
        b[g + c] = rv;
      }
      acc += rv * rv;
    }
  }
  const double a = block_sum((double)acc);
  if (t == 0) partials[blockIdx.x + blockIdx.y * gridDim.x] = a;
}

__global__ void k_adj_sum(const double* __restrict__ p, int count, double* __restrict__ out) {
  double a = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) a += p[i];
  a = block_sum(a);
  if (threadIdx.x == 0) *out = a;
}

__global__ void k_adj_finalize(const double* __restrict__ p, const double* __restrict__ p2, int count,
                               double* __restrict__ out) {
  double a = 0.0, a2 = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    a += p[i];
    a2 += p2[i];
  }
  a = block_sum(a);
  if (threadIdx.x == 0) out[0] = a;
  a2 = block_sum(a2);
  if (threadIdx.x == 0) out[1] = a2;
}

// Red-black Gauss-Seidel on one colour: x_i = (b_i + kh sum_nb x) / (6 kh + m_i), kh = kappa/h^2.
__global__ void __launch_bounds__(64) k_adj_smooth32(int n, float kh, float* __restrict__ x, const float* __restrict__ b,
                                                     const float* __restrict__ dinv, int parity) {
  const int i = blockIdx.z, j = blockIdx.y;
  const int kk = blockIdx.x * blockDim.x + threadIdx.x;
  if (kk >= (n >> 1)) return;
  const int k = 2 * kk + ((i + j + parity) & 1);
  const size_t c = cidx(n, i, j, k);
  const float L = x[cidx(n, wrapi(i + 1, n), j, k)] + x[cidx(n, wrapi(i - 1, n), j, k)] +
                  x[cidx(n, i, wrapi(j + 1, n), k)] + x[cidx(n, i, wrapi(j - 1, n), k)] +
                  x[cidx(n, i, j, wrapi(k + 1, n))] + x[cidx(n, i, j, wrapi(k - 1, n))];
  x[c] = (b[c] + kh * L) * dinv[c];
}

// The same colour step, four cells per lane (n % 4 == 0, n >= 8; as smooth_quad):
// block (32, 4), grid (ceil(n/128), n, n/4).  FRESH: the first colour of a level
// whose x is zero and not stored yet: x_i = b_i / (6 kh + m_i), and the quad's
// other cells are set to zero.
template <bool FRESH>
__global__ void __launch_bounds__(128) k_adj_smooth32q(int n, float kh, float* __restrict__ x,
                                                       const float* __restrict__ b, const float* __restrict__ dinv,
                                                       int parity) {
  const int i = blockIdx.z * 4 + threadIdx.y;
  if (i >= n) return;  // whole warps
  const int j = blockIdx.y, lane = threadIdx.x, tq = blockIdx.x * 32 + lane;
  const int nq = n >> 2;
  const bool act = tq < nq;
  const int k0 = 4 * (act ? tq : nq - 1);
  const long long nn = (long long)n * n;
  const long long c0 = (long long)i * nn + (long long)j * n + k0;
  const long long djp = (j + 1 < n) ? (long long)n : -(long long)(n - 1) * n;
  const long long djm = (j > 0) ? -(long long)n : (long long)(n - 1) * n;
  const long long dip = (i + 1 < n) ? nn : -(long long)(n - 1) * nn;
  const long long dim = (i > 0) ? -nn : (long long)(n - 1) * nn;
  float* x0 = x + c0;
  const float4 B = ld4(b + c0), D = ld4(dinv + c0);
  if constexpr (FRESH) {
    const bool even = ((i + j + parity) & 1) == 0;
    if (act)
      *reinterpret_cast<float4*>(x0) =
          even ? make_float4(B.x * D.x, 0.f, B.z * D.z, 0.f) : make_float4(0.f, B.y * D.y, 0.f, B.w * D.w);
    return;
  }
  const float4 X = ld4(x0);
  const float4 P = ld4(x0 + djp), M = ld4(x0 + djm), Q = ld4(x0 + dip), R = ld4(x0 + dim);
  if (((i + j + parity) & 1) == 0) {
    // cells k0 and k0+2
    float km = __shfl_up_sync(0xffffffffu, X.w, 1);
    if (lane == 0) km = x[c0 + (k0 == 0 ? n - 1 : -1)];
    const float LA = (km + X.y) + (P.x + M.x) + (Q.x + R.x);
    const float LB = (X.y + X.w) + (P.z + M.z) + (Q.z + R.z);
    if (act) {
      x0[0] = (B.x + kh * LA) * D.x;
      x0[2] = (B.z + kh * LB) * D.z;
    }
  } else {
    // cells k0+1 and k0+3
    float kp = __shfl_down_sync(0xffffffffu, X.x, 1);
    if (lane == 31 || tq + 1 >= nq) kp = x[c0 + (k0 + 4 == n ? 4 - n : 4)];
    const float LA = (X.x + X.z) + (P.y + M.y) + (Q.y + R.y);
    const float LB = (X.z + kp) + (P.w + M.w) + (Q.w + R.w);
    if (act) {
      x0[1] = (B.y + kh * LA) * D.y;
      x0[3] = (B.w + kh * LB) * D.w;
    }
  }
}

// ---------------------------------------------------------------------------
// The finest level in the red-black split layout (smooth_split, sweep32.cuh)
// ---------------------------------------------------------------------------
//
// A colour pass over interleaved colours moves whole lines of x, b and 1/diagonal
// to use half of each: 16 bytes for each of the level's cells, 0.33 ms at 512^3,
// the measured copy rate.  With the colours apart it moves 8.  And since a cell's
// new value does not read its old one, the correction only has to be prolonged to
// the second colour before post-smoothing, and after pre-smoothing the second
// colour's residual is the rounding of its own update, so the restriction forms
// the first colour's alone.

// One colour pass, four consecutive cells of the colour a lane; block (32, 4), 1D
// grid over the warps of split_lane.  FRESH: x is zero and not stored yet.
// 512^3: 158 us a pass, 6.8 TB/s (interleaved: 330 us).
template <bool FRESH, typename IT>
__global__ void __launch_bounds__(128) k_adj_smooth_split(int n, float kh, float* __restrict__ x,
                                                          const float* __restrict__ b,
                                                          const float* __restrict__ dinv, int colour) {
  const int lane = threadIdx.x;
  long long r;
  int seg;
  bool act;
  split_lane(n, n, (long long)blockIdx.x * 4 + threadIdx.y, lane, &r, &seg, &act);
  const int i = (int)(r / n), j = (int)(r - (long long)i * n);
  const int h = n >> 1, nq = h >> 2, m0 = 4 * seg;
  const IT H = (IT)n * n * h, r0 = ((IT)i * n + j) * h + m0;
  const IT own = (IT)colour * H + r0;
  const float4 B = ld4(b + own), D = ld4(dinv + own);
  float4 out;
  if constexpr (FRESH) {
    out = make_float4(B.x * D.x, B.y * D.y, B.z * D.z, B.w * D.w);
  } else {
    const float* x1 = x + (IT)(colour ^ 1) * H + r0;
    const IT nh = (IT)n * h;
    const IT djp = (j + 1 < n) ? (IT)h : -(IT)(n - 1) * h, djm = (j > 0) ? -(IT)h : (IT)(n - 1) * h;
    const IT dip = (i + 1 < n) ? nh : -(IT)(n - 1) * nh, dim = (i > 0) ? -nh : (IT)(n - 1) * nh;
    const float4 Q = ld4(x1), P = ld4(x1 + djp), M = ld4(x1 + djm), A = ld4(x1 + dip), C = ld4(x1 + dim);
    const int p = (i + j + colour) & 1;  // the cells are k = 2m + p
    float qm = __shfl_up_sync(0xffffffffu, Q.w, 1);
    float qp = __shfl_down_sync(0xffffffffu, Q.x, 1);
    if (p == 0 && (seg == 0 || lane == 0)) qm = x1[m0 == 0 ? h - 1 : -1];
    if (p == 1 && (seg == nq - 1 || lane == 31)) qp = x1[m0 + 4 == h ? 4 - h : 4];
    const float k0s = p ? Q.x + Q.y : qm + Q.x, k1s = p ? Q.y + Q.z : Q.x + Q.y;
    const float k2s = p ? Q.z + Q.w : Q.y + Q.z, k3s = p ? Q.w + qp : Q.z + Q.w;
    out.x = (B.x + kh * (k0s + (P.x + M.x) + (A.x + C.x))) * D.x;
    out.y = (B.y + kh * (k1s + (P.y + M.y) + (A.y + C.y))) * D.y;
    out.z = (B.z + kh * (k2s + (P.z + M.z) + (A.z + C.z))) * D.z;
    out.w = (B.w + kh * (k3s + (P.w + M.w) + (A.w + C.w))) * D.w;
  }
  if (act) *reinterpret_cast<float4*>(x + own) = out;
}

// b^H = R (b - A x) after a sweep, the first colour's residuals only (lane mapping
// of restrict_split_zr): block (32, 4), grid (ceil(nf/128), nc [J], ceil(nc/4) [I]).
template <typename IT>
__global__ void __launch_bounds__(128) k_adj_restrict_split(int nf, float kh, const float* __restrict__ x,
                                                            const float* __restrict__ b,
                                                            const float* __restrict__ m32, float* __restrict__ bH) {
  const int nc = nf >> 1, nq = nf >> 2, h = nf >> 1;
  const int I = blockIdx.z * 4 + threadIdx.y;
  if (I >= nc) return;  // whole warps
  const int J = blockIdx.y, lane = threadIdx.x, tq = blockIdx.x * 32 + lane;
  const bool act = tq < nq;
  const int m0 = 2 * (act ? tq : nq - 1);
  const IT H = (IT)nf * nf * h;
  const int i0 = 2 * I, j0 = 2 * J;
  const int iA = i0 == 0 ? nf - 1 : i0 - 1, iB = i0 + 2 == nf ? 0 : i0 + 2;
  const int jA = j0 == 0 ? nf - 1 : j0 - 1, jB = j0 + 2 == nf ? 0 : j0 + 2;
  auto row = [&](int i, int j) { return ((IT)i * nf + j) * h + m0; };
  auto two = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
  const float* x1 = x + H;
  float2 Q[2][2], qi[2][2], qj[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      Q[a][c] = two(x1 + row(i0 + a, j0 + c));
      qi[a][c] = two(x1 + row(a ? iB : iA, j0 + c));
      qj[a][c] = two(x1 + row(i0 + a, c ? jB : jA));
    }
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const IT r = row(i0 + a, j0 + c);
      const float2 X = two(x + r), B = two(b + r), Mv = two(m32 + r);
      const float2 q = Q[a][c];
      const int p = (a + c) & 1;  // the first colour's cells of the quad are k0 + p and k0 + p + 2
      float qm = __shfl_up_sync(0xffffffffu, q.y, 1);
      float qp = __shfl_down_sync(0xffffffffu, q.x, 1);
      if (p == 0 && lane == 0) qm = x1[r + (m0 == 0 ? h - 1 : -1)];
      if (p == 1 && (lane == 31 || tq + 1 >= nq)) qp = x1[r + (m0 + 2 == h ? 2 - h : 2)];
      const float k0s = p ? q.x + q.y : qm + q.x, k1s = p ? q.y + qp : q.x + q.y;
      const float2 ni = a == 0 ? qi[0][c] : Q[0][c], pi = a == 0 ? Q[1][c] : qi[1][c];
      const float2 nj = c == 0 ? qj[a][0] : Q[a][0], pj = c == 0 ? Q[a][1] : qj[a][1];
      s0 += B.x + kh * (k0s + (ni.x + pi.x) + (nj.x + pj.x) - 6.f * X.x) - Mv.x * X.x;
      s1 += B.y + kh * (k1s + (ni.y + pi.y) + (nj.y + pj.y) - 6.f * X.y) - Mv.y * X.y;
    }
  if (act)
    *reinterpret_cast<float2*>(bH + ((IT)I * nc + J) * nc + m0) = make_float2(0.125f * s0, 0.125f * s1);
}

// x^h += P x^H at the second colour (post-smoothing starts with the first), four
// fine rows a lane from nine coarse rows (prolong_split2x2_second); grid as the
// restriction's.
template <typename IT>
__global__ void __launch_bounds__(128) k_adj_prolong_split(int nc, const float* __restrict__ xH,
                                                           float* __restrict__ xf) {
  const int nf = nc << 1, nq = nf >> 2, h = nf >> 1;
  const int I = blockIdx.z * 4 + threadIdx.y;
  if (I >= nc) return;  // whole warps
  const int J = blockIdx.y, lane = threadIdx.x, tq = blockIdx.x * 32 + lane;
  const bool act = tq < nq;
  const int K0 = 2 * (act ? tq : nq - 1);
  const int Km = K0 == 0 ? nc - 1 : K0 - 1, Kp = K0 + 2 == nc ? 0 : K0 + 2;
  const int Iv[3] = {I == 0 ? nc - 1 : I - 1, I, I + 1 == nc ? 0 : I + 1};
  const int Jv[3] = {J == 0 ? nc - 1 : J - 1, J, J + 1 == nc ? 0 : J + 1};
  const bool edge_m = lane == 0, edge_p = lane == 31 || tq + 1 >= nq;
  float2 d[3][3];
  float dm[3][3], dp[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const IT r = ((IT)Iv[a] * nc + Jv[c]) * nc;
      d[a][c] = *reinterpret_cast<const float2*>(xH + r + K0);
      dm[a][c] = edge_m ? xH[r + Km] : 0.f;
      dp[a][c] = edge_p ? xH[r + Kp] : 0.f;
    }
  constexpr float w = 1.f / 64.f;
  const IT H = (IT)nf * nf * h;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int x2 = a ? 2 : 0, y2 = c ? 2 : 0;
      const float Rx = 9.f * d[1][1].x + 3.f * (d[x2][1].x + d[1][y2].x) + d[x2][y2].x;
      const float Ry = 9.f * d[1][1].y + 3.f * (d[x2][1].y + d[1][y2].y) + d[x2][y2].y;
      float Rm = __shfl_up_sync(0xffffffffu, Ry, 1);
      float Rp = __shfl_down_sync(0xffffffffu, Rx, 1);
      if (edge_m) Rm = 9.f * dm[1][1] + 3.f * (dm[x2][1] + dm[1][y2]) + dm[x2][y2];
      if (edge_p) Rp = 9.f * dp[1][1] + 3.f * (dp[x2][1] + dp[1][y2]) + dp[x2][y2];
      const bool odd = (a + c) & 1;
      const IT o = H + ((IT)(2 * I + a) * nf + 2 * J + c) * h + K0;
      if (act) {
        float2* p = reinterpret_cast<float2*>(xf + o);
        const float2 old = *p;
        *p = make_float2(old.x + (odd ? 3.f * Rx + Rm : 3.f * Rx + Ry) * w,
                         old.y + (odd ? 3.f * Ry + Rx : 3.f * Ry + Rp) * w);
      }
    }
}

// ---------------------------------------------------------------------------
// The coarsest levels in one CTA
// ---------------------------------------------------------------------------
//
// From the first level with at most kAdjTailCells cells the whole rest of the
// V-cycle runs in one CTA, the levels in shared memory: an update is six loads
// and eight operations, so even a 16^3 colour pass is shorter there than a
// kernel's start.  A level's x starts at zero, the finest mesh's (warm) from
// where the cycle before left it.
constexpr int kAdjTailThreads = 1024;
struct AdjTail {
  int T;                     // levels
  int n[kAdjTailLevels];
  float kh[kAdjTailLevels];
  const float* m32[kAdjTailLevels];
  const float* dinv[kAdjTailLevels];
  const float* b;            // first level's right-hand side
  float* x;                  // first level's result
  int nu1, nu2, sweeps;
  int warm;                  // the first level's x is read
};

__device__ __forceinline__ float adj_tail_sum(const float* x, int n, int i, int j, int k) {
  const int nn = n * n, c = (i * n + j) * n + k;
  return x[i + 1 < n ? c + nn : c + nn - n * nn] + x[i > 0 ? c - nn : c - nn + n * nn] +
         x[j + 1 < n ? c + n : c + n - nn] + x[j > 0 ? c - n : c - n + nn] + x[k + 1 < n ? c + 1 : c + 1 - n] +
         x[k > 0 ? c - 1 : c - 1 + n];
}

// Red-black sweeps; a row of odd length (a coarsest level only) gives its last
// cell to the colour of even k.
__device__ __forceinline__ void adj_tail_smooth(int n, float kh, float* x, const float* b, const float* dinv,
                                                int sweeps) {
  const int w = (n + 1) >> 1;
  for (int s = 0; s < 2 * sweeps; ++s) {
    for (int t = threadIdx.x; t < w * n * n; t += blockDim.x) {
      const int kk = t % w, r = t / w, j = r % n, i = r / n;
      const int k = 2 * kk + ((i + j + s) & 1);
      if (k >= n) continue;
      const int c = r * n + k;
      x[c] = (b[c] + kh * adj_tail_sum(x, n, i, j, k)) * dinv[c];
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kAdjTailThreads) k_adj_tail(AdjTail A) {
  extern __shared__ float sm[];
  float *x[kAdjTailLevels], *b[kAdjTailLevels], *mm[kAdjTailLevels], *dd[kAdjTailLevels];
  float* at = sm;
  for (int l = 0; l < A.T; ++l) {
    const int n3 = A.n[l] * A.n[l] * A.n[l];
    x[l] = at;
    b[l] = x[l] + n3;
    mm[l] = b[l] + n3;
    dd[l] = mm[l] + n3;
    at = dd[l] + n3;
    for (int c = threadIdx.x; c < n3; c += blockDim.x) {
      x[l][c] = l == 0 && A.warm ? A.x[c] : 0.f;
      mm[l][c] = A.m32[l][c];
      dd[l][c] = A.dinv[l][c];
      if (l == 0) b[0][c] = A.b[c];
    }
  }
  __syncthreads();
  for (int l = 0; l + 1 < A.T; ++l) {
    const int n = A.n[l], nc = n >> 1;
    const float kh = A.kh[l];
    adj_tail_smooth(n, kh, x[l], b[l], dd[l], A.nu1);
    for (int t = threadIdx.x; t < nc * nc * nc; t += blockDim.x) {
      const int K = t % nc, J = (t / nc) % nc, I = t / (nc * nc);
      float s = 0.f;
      for (int q = 0; q < 8; ++q) {
        const int i = 2 * I + (q >> 2), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q & 1), c = (i * n + j) * n + k;
        s += b[l][c] + kh * (adj_tail_sum(x[l], n, i, j, k) - 6.f * x[l][c]) - mm[l][c] * x[l][c];
      }
      b[l + 1][t] = 0.125f * s;
    }
    __syncthreads();
  }
  adj_tail_smooth(A.n[A.T - 1], A.kh[A.T - 1], x[A.T - 1], b[A.T - 1], dd[A.T - 1], A.sweeps);
  for (int l = A.T - 2; l >= 0; --l) {
    const int n = A.n[l], nc = n >> 1;
    const float* xH = x[l + 1];
    for (int t = threadIdx.x; t < n * n * n; t += blockDim.x) {
      const int k = t % n, j = (t / n) % n, i = t / (n * n);
      const int I = i >> 1, J = j >> 1, K = k >> 1;
      const int I2 = wrapi(I + ((i & 1) ? 1 : -1), nc), J2 = wrapi(J + ((j & 1) ? 1 : -1), nc),
                K2 = wrapi(K + ((k & 1) ? 1 : -1), nc);
#define XH(a, b, c) xH[((a) * nc + (b)) * nc + (c)]
      x[l][t] += (27.f * XH(I, J, K) + 9.f * (XH(I2, J, K) + XH(I, J2, K) + XH(I, J, K2)) +
                  3.f * (XH(I2, J2, K) + XH(I2, J, K2) + XH(I, J2, K2)) + XH(I2, J2, K2)) *
                 (1.f / 64.f);
#undef XH
    }
    __syncthreads();
    adj_tail_smooth(n, A.kh[l], x[l], b[l], dd[l], A.nu2);
  }
  for (int c = threadIdx.x; c < A.n[0] * A.n[0] * A.n[0]; c += blockDim.x) A.x[c] = x[0][c];
}

// Coarse right-hand side: b^H = R (b - A x) over the 8 children (x^H starts at zero).
__global__ void __launch_bounds__(64) k_adj_restrict_resid32(int nf, float kh, const float* __restrict__ x,
                                                             const float* __restrict__ b,
                                                             const float* __restrict__ m32, float* __restrict__ bH) {
  const int nc = nf >> 1;
  const int I = blockIdx.z, J = blockIdx.y;
  const int Kc = blockIdx.x * blockDim.x + threadIdx.x;
  if (Kc >= nc) return;
  float s = 0.f;
  for (int di = 0; di < 2; ++di)
    for (int dj = 0; dj < 2; ++dj)
      for (int dk = 0; dk < 2; ++dk) {
        const int i = 2 * I + di, j = 2 * J + dj, k = 2 * Kc + dk;
        const size_t c = cidx(nf, i, j, k);
        const float L = x[cidx(nf, wrapi(i + 1, nf), j, k)] + x[cidx(nf, wrapi(i - 1, nf), j, k)] +
                        x[cidx(nf, i, wrapi(j + 1, nf), k)] + x[cidx(nf, i, wrapi(j - 1, nf), k)] +
                        x[cidx(nf, i, j, wrapi(k + 1, nf))] + x[cidx(nf, i, j, wrapi(k - 1, nf))];
        s += b[c] - (-kh * (L - 6.f * x[c]) + m32[c] * x[c]);
      }
  const size_t t = cidx(nc, I, J, Kc);
  bH[t] = 0.125f * s;
}

// The same restriction, sixteen fine cells per lane (nf % 4 == 0, as
// restrict_quad): block (32, 4), grid (ceil(nf/128), nc [J], ceil(nc/4) [I]).
__global__ void __launch_bounds__(128) k_adj_restrict_resid32q(int nf, float kh, const float* __restrict__ x,
                                                               const float* __restrict__ b,
                                                               const float* __restrict__ m32, float* __restrict__ bH) {
  const int nc = nf >> 1, nq = nf >> 2;
  const int I = blockIdx.z * 4 + threadIdx.y;
  if (I >= nc) return;  // whole warps
  const int J = blockIdx.y, lane = threadIdx.x, tq = blockIdx.x * 32 + lane;
  const bool act = tq < nq;
  const int k0 = 4 * (act ? tq : nq - 1);
  const int i0 = 2 * I, j0 = 2 * J;
  const int iA = i0 == 0 ? nf - 1 : i0 - 1, iB = i0 + 2 == nf ? 0 : i0 + 2;
  const int jA = j0 == 0 ? nf - 1 : j0 - 1, jB = j0 + 2 == nf ? 0 : j0 + 2;
  auto row = [&](int i, int j) { return ((long long)i * nf + j) * nf + k0; };
  float4 X[2][2];
  long long co[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      co[a][c] = row(i0 + a, j0 + c);
      X[a][c] = ld4(x + co[a][c]);
    }
  float4 xi[2][2], xj[2][2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    xi[0][c] = ld4(x + row(iA, j0 + c));
    xi[1][c] = ld4(x + row(iB, j0 + c));
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    xj[a][0] = ld4(x + row(i0 + a, jA));
    xj[a][1] = ld4(x + row(i0 + a, jB));
  }
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float4 q = X[a][c];
      float qm = __shfl_up_sync(0xffffffffu, q.w, 1);
      float qp = __shfl_down_sync(0xffffffffu, q.x, 1);
      if (lane == 0) qm = x[co[a][c] + (k0 == 0 ? nf - 1 : -1)];
      if (lane == 31 || tq + 1 >= nq) qp = x[co[a][c] + (k0 + 4 == nf ? 4 - nf : 4)];
      const float4 ni = a == 0 ? xi[0][c] : X[0][c], pi = a == 0 ? X[1][c] : xi[1][c];
      const float4 nj = c == 0 ? xj[a][0] : X[a][0], pj = c == 0 ? X[a][1] : xj[a][1];
      const float4 Bv = ld4(b + co[a][c]), Mv = ld4(m32 + co[a][c]);
      auto d = [&](float bb, float mm, float xc, float L) { return bb + kh * (L - 6.f * xc) - mm * xc; };
      s0 += d(Bv.x, Mv.x, q.x, (qm + q.y) + (ni.x + pi.x) + (nj.x + pj.x)) +
            d(Bv.y, Mv.y, q.y, (q.x + q.z) + (ni.y + pi.y) + (nj.y + pj.y));
      s1 += d(Bv.z, Mv.z, q.z, (q.y + q.w) + (ni.z + pi.z) + (nj.z + pj.z)) +
            d(Bv.w, Mv.w, q.w, (q.z + qp) + (ni.w + pi.w) + (nj.w + pj.w));
    }
  if (act) {
    const long long t = ((long long)I * nc + J) * nc + (k0 >> 1);
    *reinterpret_cast<float2*>(bH + t) = make_float2(0.125f * s0, 0.125f * s1);
  }
}

// x^h += P x^H, four fine cells per lane (as prolong_quad, without the
// restricted-solution term): block (32, 4), grid (ceil(nf/128), nf, nf/4).
__global__ void __launch_bounds__(128) k_adj_prolong32q(int nc, const float* __restrict__ xH, float* __restrict__ xf) {
  const int nf = nc << 1, nq = nf >> 2;
  const int i = blockIdx.z * 4 + threadIdx.y, j = blockIdx.y, lane = threadIdx.x, tq = blockIdx.x * 32 + lane;
  const bool act = tq < nq;
  const int t = act ? tq : nq - 1;
  const int k0 = 4 * t, K0 = 2 * t;
  const int I = i >> 1, J = j >> 1;
  int I2 = I + ((i & 1) ? 1 : -1), J2 = J + ((j & 1) ? 1 : -1);
  I2 = I2 < 0 ? nc - 1 : (I2 >= nc ? 0 : I2);
  J2 = J2 < 0 ? nc - 1 : (J2 >= nc ? 0 : J2);
  const long long rA = ((long long)I * nc + J) * nc, rB = ((long long)I2 * nc + J) * nc,
                  rC = ((long long)I * nc + J2) * nc, rD = ((long long)I2 * nc + J2) * nc;
  auto two = [&](long long r) { return *reinterpret_cast<const float2*>(xH + r + K0); };
  const float2 A = two(rA), B = two(rB), C = two(rC), D = two(rD);
  const float Rx = 9.f * A.x + 3.f * (B.x + C.x) + D.x;
  const float Ry = 9.f * A.y + 3.f * (B.y + C.y) + D.y;
  float Rm = __shfl_up_sync(0xffffffffu, Ry, 1);
  float Rp = __shfl_down_sync(0xffffffffu, Rx, 1);
  if (lane == 0) {
    const int Km = K0 == 0 ? nc - 1 : K0 - 1;
    Rm = 9.f * xH[rA + Km] + 3.f * (xH[rB + Km] + xH[rC + Km]) + xH[rD + Km];
  }
  if (lane == 31 || tq + 1 >= nq) {
    const int Kp = K0 + 2 == nc ? 0 : K0 + 2;
    Rp = 9.f * xH[rA + Kp] + 3.f * (xH[rB + Kp] + xH[rC + Kp]) + xH[rD + Kp];
  }
  constexpr float w = 1.f / 64.f;
  float* p = xf + ((long long)i * nf + j) * nf + k0;
  const float4 old = ld4(p);
  if (act)
    *reinterpret_cast<float4*>(p) = make_float4(old.x + (3.f * Rx + Rm) * w, old.y + (3.f * Rx + Ry) * w,
                                                old.z + (3.f * Ry + Rx) * w, old.w + (3.f * Ry + Rp) * w);
}

// x^h += P x^H (27/9/3/1 weights).
__global__ void __launch_bounds__(64) k_adj_prolong32(int nc, const float* __restrict__ xH, float* __restrict__ xf) {
  const int nf = nc << 1;
  const int i = blockIdx.z, j = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nf) return;
  const int I = i >> 1, J = j >> 1, Kc = k >> 1;
  const int I2 = wrapi(I + ((i & 1) ? 1 : -1), nc);
  const int J2 = wrapi(J + ((j & 1) ? 1 : -1), nc);
  const int K2 = wrapi(Kc + ((k & 1) ? 1 : -1), nc);
#define XH(a, b, c) xH[cidx(nc, a, b, c)]
  const float corr = (27.f * XH(I, J, Kc) + 9.f * (XH(I2, J, Kc) + XH(I, J2, Kc) + XH(I, J, K2)) +
                      3.f * (XH(I2, J2, Kc) + XH(I2, J, K2) + XH(I, J2, K2)) + XH(I2, J2, K2)) *
                     (1.f / 64.f);
#undef XH
  xf[cidx(nf, i, j, k)] += corr;
}

// The mass of the next level (8-child mean) and its inverse diagonal; kh: that
// level's.  SPLIT: the fine level in the split layout.
template <bool SPLIT>
__global__ void __launch_bounds__(64) k_adj_restrict_m32(int nf, float kh, const float* __restrict__ fine,
                                                         float* __restrict__ coarse, float* __restrict__ dinv) {
  const int nc = nf >> 1;
  const int I = blockIdx.z, J = blockIdx.y;
  const int Kc = blockIdx.x * blockDim.x + threadIdx.x;
  if (Kc >= nc) return;
  float s = 0.f;
  for (int di = 0; di < 2; ++di)
    for (int dj = 0; dj < 2; ++dj) {
      const int i = 2 * I + di, j = 2 * J + dj;
      if constexpr (SPLIT) {  // the two children of a row sit at Kc of the two colours
        s += fine[split_idx(nf, i, j, 2 * Kc)] + fine[split_idx(nf, i, j, 2 * Kc + 1)];
      } else {
        s += fine[cidx(nf, i, j, 2 * Kc)] + fine[cidx(nf, i, j, 2 * Kc + 1)];
      }
    }
  const size_t t = cidx(nc, I, J, Kc);
  coarse[t] = 0.125f * s;
  dinv[t] = 1.f / (6.f * kh + 0.125f * s);
}

// lambda += s e (ADD) or lambda = s e (the first correction), e in the natural or
// the split layout; a thread takes the cells k = 2q, 2q + 1 of a row.
template <bool SPLIT, bool ADD>
__global__ void __launch_bounds__(kThreads) k_adj_apply(int n, double s, double* __restrict__ lam,
                                                        const float* __restrict__ e) {
  const int h = n >> 1;
  const long long H = (long long)n * n * h;
  for (int row = blockIdx.x; row < n * n; row += gridDim.x) {
    const int c0 = (row / n + row % n) & 1;  // colour of the even cells
    for (int q = threadIdx.x; q < h; q += blockDim.x) {
      const long long t = (long long)row * n + 2 * q, o = (long long)row * h + q;
      const float a = SPLIT ? e[c0 * H + o] : e[t], b = SPLIT ? e[(c0 ^ 1) * H + o] : e[t + 1];
      double2* p = reinterpret_cast<double2*>(lam + t);
      const double2 old = ADD ? *p : make_double2(0.0, 0.0);
      *p = make_double2(fma((double)a, s, old.x), fma((double)b, s, old.y));
    }
  }
}

// dl/d delta = gam lambda with gam = -dN/d delta (f(R): -Om/a; symmetron msym
// (a*/a)^3 u), and partial sums of lambda tq with tq = -dN/d theta (f(R):
// K/((n+1)u)) and of (dl/d delta_i) rho_i, the term the mean-1 normalisation of the
// density adds to the gradient with respect to the caller's rho.  Terms and sums in
// FP64, six instructions of its pipe a cell, which bound it (512^3: 1.4 ms).
template <int K>
__global__ void __launch_bounds__(kThreads) k_adj_outputs(ModelDev m, long long n3, const double* __restrict__ lam,
                                                          const double* __restrict__ u,
                                                          const float* __restrict__ rho32,
                                                          double* __restrict__ grad_rho,
                                                          double* __restrict__ partials,
                                                          double* __restrict__ partials2) {
  double acc = 0.0, acc2 = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x) {
    double g;
    if constexpr (is_fr(K)) {
      g = -m.om_a * lam[t];
      acc = fma(lam[t], rcp_fast(u[t]), acc);
    } else {
      g = m.msym * m.rat3 * u[t] * lam[t];
    }
    grad_rho[t] = g;
    acc2 = fma(g, f2d_exact(rho32[t]), acc2);
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = is_fr(K) ? acc * (m.K / (K + 1)) : 0.0;
  acc2 = block_sum(acc2);
  if (threadIdx.x == 0) partials2[blockIdx.x] = acc2;
}

// Chain rule through delta = rho / mu - 1, mu = sum(rho) / N^3:
//   dl/d rho_j = (dl/d delta_j - sum_i (dl/d delta_i) rho_i / sum(rho)) / mu.
__global__ void k_adj_grad_raw(long long n3, const double* __restrict__ g, const double* __restrict__ dot,
                               const double* __restrict__ rho_sum, double* __restrict__ out) {
  const double S = *rho_sum, shift = *dot / S, inv_mu = (double)n3 / S;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x)
    out[t] = (g[t] - shift) * inv_mu;
}

// ---------------------------------------------------------------------------
// Scratch: one allocation per (device, N): FP64 lambda, m, rhs on the fine level;
// FP32 x, b, m, 1/diagonal on every level; partial sums.
// ---------------------------------------------------------------------------

struct AdjWork {
  int device = -1, N = 0, nlev = 0;
  void* base = nullptr;
  double *lam = nullptr, *m64 = nullptr, *rhs = nullptr;
  double *partials = nullptr, *partials2 = nullptr, *scal = nullptr, *h_scal = nullptr;
  int n[kMaxLevels];
  float *x[kMaxLevels], *b[kMaxLevels], *m32[kMaxLevels], *dinv[kMaxLevels];
};

static std::mutex g_adj_mu;
static AdjWork* g_adj[32];
static int g_nadj = 0;

static int adj_work(int N, int levels, AdjWork** out) {
  int dev = 0;
  MG_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_adj_mu);
  const int nlev = count_levels(N, levels);
  for (int i = 0; i < g_nadj; ++i)
    if (g_adj[i]->device == dev && g_adj[i]->N == N && g_adj[i]->nlev == nlev) {
      *out = g_adj[i];
      return MGGLAM_OK;
    }
  if (g_nadj >= 32) return MGGLAM_ERR_OOM;
  AdjWork* w = new AdjWork();
  w->device = dev;
  w->N = N;
  w->nlev = nlev;
  const size_t n3 = (size_t)N * N * N;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const size_t o_lam = take(n3 * 8), o_m = take(n3 * 8), o_rhs = take(n3 * 8), o_p = take(kMaxReduceBlocks * 8),
               o_p2 = take(kMaxReduceBlocks * 8), o_s = take(64);
  size_t ox[kMaxLevels], ob[kMaxLevels], om[kMaxLevels], od[kMaxLevels];
  for (int l = 0, nn = N; l < nlev; ++l, nn /= 2) {
    const size_t c = (size_t)nn * nn * nn;
    w->n[l] = nn;
    ox[l] = take(c * 4);
    ob[l] = take(c * 4);
    om[l] = take(c * 4);
    od[l] = take(c * 4);
  }
  if (cudaMalloc(&w->base, off) != cudaSuccess) {
    cudaGetLastError();
    delete w;
    return MGGLAM_ERR_OOM;
  }
  if (cudaMallocHost((void**)&w->h_scal, 64) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(w->base);
    delete w;
    return MGGLAM_ERR_OOM;
  }
  char* b = (char*)w->base;
  w->lam = (double*)(b + o_lam);
  w->m64 = (double*)(b + o_m);
  w->rhs = (double*)(b + o_rhs);
  w->partials = (double*)(b + o_p);
  w->partials2 = (double*)(b + o_p2);
  w->scal = (double*)(b + o_s);
  for (int l = 0; l < nlev; ++l) {
    w->x[l] = (float*)(b + ox[l]);
    w->b[l] = (float*)(b + ob[l]);
    w->m32[l] = (float*)(b + om[l]);
    w->dinv[l] = (float*)(b + od[l]);
  }
  g_adj[g_nadj++] = w;
  *out = w;
  return MGGLAM_OK;
}

void release_adjoint_work() {
  std::lock_guard<std::mutex> lk(g_adj_mu);
  int dev = 0;
  cudaGetDevice(&dev);
  int keep = 0;
  for (int i = 0; i < g_nadj; ++i) {
    if (g_adj[i]->device == dev) {
      cudaFree(g_adj[i]->base);
      cudaFreeHost(g_adj[i]->h_scal);
      delete g_adj[i];
    } else {
      g_adj[keep++] = g_adj[i];
    }
  }
  g_nadj = keep;
}

static dim3 grid_k(int n_k, int n_j, int n_i) { return dim3((n_k + 63) / 64, n_j, n_i); }

// How a solve runs its cycles.
struct AdjCtx {
  AdjWork* w;
  const mgglam_params* prm;
  double kappa;
  bool split;  // the finest level in the red-black split layout (32 | N, pre- and post-smoothing)
  int tail;    // first level run by k_adj_tail, or -1
};

static float adj_kh(const AdjCtx& C, int l) { return (float)(C.kappa / ((double)(1 << l) * (double)(1 << l))); }

static bool adj_quad(int n) { return n % 4 == 0 && n >= 8; }

// fresh: the level's x is zero (and, where the first pass takes it so, not stored).
static int adj_smooth(const AdjCtx& C, int l, int sweeps, bool fresh, cudaStream_t st) {
  AdjWork* w = C.w;
  const int n = w->n[l];
  const float kh = adj_kh(C, l);
  const bool split = l == 0 && C.split, quad = adj_quad(n);
  if (fresh && (sweeps <= 0 || !(split || quad)))
    MG_CUDA_TRY(cudaMemsetAsync(w->x[l], 0, (size_t)n * n * n * 4, st));
  for (int s = 0; s < 2 * sweeps; ++s) {
    const int par = s & 1;
    const bool f = fresh && s == 0;
    if (split) {
      const unsigned blocks = (unsigned)((split_warps(n, n) + 3) / 4);
      // 32-bit cell offsets where the level has at most 2^30 cells
      auto kern = n <= 1024 ? (f ? k_adj_smooth_split<true, int> : k_adj_smooth_split<false, int>)
                            : (f ? k_adj_smooth_split<true, long long> : k_adj_smooth_split<false, long long>);
      kern<<<blocks, dim3(32, 4), 0, st>>>(n, kh, w->x[l], w->b[l], w->dinv[l], par);
    } else if (quad) {
      (f ? k_adj_smooth32q<true> : k_adj_smooth32q<false>)<<<dim3((n / 4 + 31) / 32, n, n / 4), dim3(32, 4), 0, st>>>(
          n, kh, w->x[l], w->b[l], w->dinv[l], par);
    } else {
      k_adj_smooth32<<<grid_k(n / 2, n, n), 64, 0, st>>>(n, kh, w->x[l], w->b[l], w->dinv[l], par);
    }
    note_launch(1);
  }
  return MGGLAM_OK;
}

static int adj_vcycle(const AdjCtx& C, int l, bool fresh, cudaStream_t st) {
  AdjWork* w = C.w;
  const mgglam_params* prm = C.prm;
  const int n = w->n[l];
  const float kh = adj_kh(C, l);
  int rc;
  if (l == C.tail) {
    AdjTail A = {};
    A.T = w->nlev - l;
    for (int t = 0; t < A.T; ++t) {
      A.n[t] = w->n[l + t];
      A.kh[t] = adj_kh(C, l + t);
      A.m32[t] = w->m32[l + t];
      A.dinv[t] = w->dinv[l + t];
    }
    A.b = w->b[l];
    A.x = w->x[l];
    A.nu1 = prm->nu1;
    A.nu2 = prm->nu2;
    A.sweeps = prm->coarse_sweeps;
    A.warm = !fresh;
    k_adj_tail<<<1, kAdjTailThreads, adj_tail_smem(A.n, A.T), st>>>(A);
    note_launch(1);
    return MGGLAM_OK;
  }
  if (l == w->nlev - 1) return adj_smooth(C, l, prm->coarse_sweeps, fresh, st);
  if ((rc = adj_smooth(C, l, prm->nu1, fresh, st))) return rc;
  const int nc = w->n[l + 1];
  const bool split = l == 0 && C.split;
  const dim3 b4(32, 4), gr((n / 4 + 31) / 32, nc, (nc + 3) / 4);
  if (split)
    (n <= 1024 ? k_adj_restrict_split<int> : k_adj_restrict_split<long long>)<<<gr, b4, 0, st>>>(
        n, kh, w->x[l], w->b[l], w->m32[l], w->b[l + 1]);
  else if (adj_quad(n))
    k_adj_restrict_resid32q<<<gr, b4, 0, st>>>(n, kh, w->x[l], w->b[l], w->m32[l], w->b[l + 1]);
  else
    k_adj_restrict_resid32<<<grid_k(nc, nc, nc), 64, 0, st>>>(n, kh, w->x[l], w->b[l], w->m32[l], w->b[l + 1]);
  note_launch(1);
  if ((rc = adj_vcycle(C, l + 1, true, st))) return rc;
  if (split)
    (n <= 1024 ? k_adj_prolong_split<int> : k_adj_prolong_split<long long>)<<<gr, b4, 0, st>>>(nc, w->x[l + 1],
                                                                                               w->x[l]);
  else if (adj_quad(n))
    k_adj_prolong32q<<<dim3((n / 4 + 31) / 32, n, n / 4), b4, 0, st>>>(nc, w->x[l + 1], w->x[l]);
  else
    k_adj_prolong32<<<grid_k(n, n, n), 64, 0, st>>>(nc, w->x[l + 1], w->x[l]);
  note_launch(1);
  return adj_smooth(C, l, prm->nu2, false, st);
}

// Dispatch on the model (the adjoint takes f(R) and the symmetron).
#define MG_ADJ_DISPATCH(kind, CALL)                    \
  switch (kind) {                                      \
    case KFR0: { constexpr int KK = KFR0; CALL; } break; \
    case KFR1: { constexpr int KK = KFR1; CALL; } break; \
    case KFR2: { constexpr int KK = KFR2; CALL; } break; \
    default: { constexpr int KK = KSYM; CALL; } break;   \
  }                                                    \
  note_launch(1)

int solve_adjoint(const mgglam_params* prm, double a, const double* field, const float* rho, int N,
                  const double* grad_field, double* grad_rho, double* grad_rho_raw, double* grad_theta, double tol,
                  mgglam_stats* stats, cudaStream_t st) {
  auto t0 = std::chrono::steady_clock::now();
  ModelDev m;
  int rc = make_model(prm, a, N, &m);
  if (rc) return rc;
  if (!(is_fr(m.kind) || m.kind == KSYM)) return MGGLAM_ERR_ARG;
  AdjWork* w = nullptr;
  if ((rc = adj_work(N, prm->levels, &w))) return rc;
  Workspace* ws = nullptr;  // for the density mean scratch
  if ((rc = get_workspace(4, MGGLAM_FP64, 1, &ws))) return rc;
  const long long n3 = (long long)N * N * N;
  if ((rc = launch_density_mean(rho, (size_t)n3, ws->partials, ws->scalars + SC_MEAN, st))) return rc;
  AdjCtx C = {w, prm, m.c2, N % 32 == 0 && prm->nu1 >= 1 && prm->nu2 >= 1, -1};
  C.tail = adj_tail_level(w->n, w->nlev, C.split);
  if (C.tail >= 0)
    MG_CUDA_TRY(cudaFuncSetAttribute(k_adj_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjTailSmem));
  const int rows = N * N < kMaxReduceBlocks ? N * N : kMaxReduceBlocks;  // grid of the row kernels
  const int bh = N >= 512 ? 256 : (N <= 64 ? 32 : ((N / 2 + 31) / 32) * 32);  // their threads, one per pair of cells
  const double* rs = ws->scalars + SC_MEAN;
  if (C.split) {
    MG_ADJ_DISPATCH(m.kind, (k_adj_setup<KK, true><<<rows, bh, 0, st>>>(m, N, adj_kh(C, 0), field, rho, rs, grad_field,
                                                                        w->m64, w->m32[0], w->dinv[0], w->rhs, w->b[0],
                                                                        w->partials)));
  } else {
    MG_ADJ_DISPATCH(m.kind, (k_adj_setup<KK, false><<<rows, bh, 0, st>>>(m, N, adj_kh(C, 0), field, rho, rs, grad_field,
                                                                         w->m64, w->m32[0], w->dinv[0], w->rhs, w->b[0],
                                                                         w->partials)));
  }
  k_adj_sum<<<1, 1024, 0, st>>>(w->partials, rows, w->scal);
  note_launch(1);
  for (int l = 1; l < w->nlev; ++l) {
    auto kern = l == 1 && C.split ? k_adj_restrict_m32<true> : k_adj_restrict_m32<false>;
    kern<<<grid_k(w->n[l], w->n[l], w->n[l]), 64, 0, st>>>(w->n[l - 1], adj_kh(C, l), w->m32[l - 1], w->m32[l],
                                                           w->dinv[l]);
    note_launch(1);
  }
  const int gr = N * N < 2048 ? N * N : 2048;
  const int bt = N >= 256 ? 256 : (N <= 32 ? 32 : ((N + 31) / 32) * 32);
  // the fine residual in float-float on meshes its tiles divide, else FP64
  const bool ffr = N % 32 == 0, pair = N % 64 == 0;
  const ff kappa_ff = {(float)m.c2, (float)(m.c2 - (double)(float)m.c2)};
  auto rk = pair ? (C.split ? (N <= 1024 ? k_adj_residual_ff<8, 2, true, int> : k_adj_residual_ff<8, 2, true, long long>)
                            : (N <= 1024 ? k_adj_residual_ff<8, 2, false, int> : k_adj_residual_ff<8, 2, false, long long>))
                 : (C.split ? k_adj_residual_ff<8, 1, true, long long> : k_adj_residual_ff<8, 1, false, long long>);
  const long long tiles = (long long)(N / (pair ? 64 : 32)) * (N / 8);
  const int chunk = ffr ? march_chunk(N, tiles, (const void*)rk, 256) : N;
  const dim3 gff((unsigned)tiles, (N + chunk - 1) / chunk);
  int ex = 0;  // float-float path: the residuals after the first are in units of 2^-ex
  auto fetch = [&]() -> int {
    MG_CUDA_TRY(cudaMemcpyAsync(w->h_scal, w->scal, sizeof(double), cudaMemcpyDeviceToHost, st));
    MG_CUDA_TRY(cudaStreamSynchronize(st));
    MG_CUDA_TRY(cudaGetLastError());
    return MGGLAM_OK;
  };
  auto residual = [&]() -> int {
    if (ffr) {
      rk<<<gff, 256, 0, st>>>(N, chunk, ex, kappa_ff, w->lam, w->m64, w->rhs, w->b[0], w->partials);
      k_adj_sum<<<1, 1024, 0, st>>>(w->partials, (int)(gff.x * gff.y), w->scal);
    } else {
      k_adj_residual64<<<gr, bt, 0, st>>>(N, m.c2, w->lam, w->m64, w->rhs, w->b[0], w->partials);
      k_adj_sum<<<1, 1024, 0, st>>>(w->partials, gr, w->scal);
    }
    note_launch(2);
    return fetch();
  };
  // lambda starts at zero: the first residual is the right-hand side, which normalises it
  if ((rc = fetch())) return rc;
  const double bnorm = sqrt(w->h_scal[0] / (double)n3);
  const double snorm = bnorm > 0.0 ? bnorm : 1.0;
  double eps = bnorm / snorm;
  if (ffr && bnorm > 0.0 && isfinite(bnorm)) ex = -ilogb(bnorm / m.c2);  // lambda is of the size of rhs / kappa
  mgglam_stats local;
  mgglam_stats* S = stats ? stats : &local;
  memset(S, 0, sizeof(*S));
  S->resid0 = eps;
  S->resid_hist[0] = eps;
  int cyc = 0, outer = 0, nh = 1;
  // inner FP32 cycles per FP64/float-float step: fixed, or (inner_cycles = 0)
  // enough for tol at the observed contraction, capped where one single-
  // precision correction stops gaining (~1e-6), as in the forward solve
  double rho_est = kInitialContraction;
  int status = MGGLAM_OK;
  while (!(eps <= tol) && cyc < prm->max_cycles) {
    if (!isfinite(eps)) { status = MGGLAM_ERR_NONFINITE; break; }
    int inner = prm->inner_cycles;
    if (inner <= 0) {
      const double lr = log(rho_est);
      const int need = (int)ceil(log(fmax(tol, 1e-300) / eps) / lr - 1e-9);
      const int cap = (int)ceil(log(kFp32StepGain) / lr - 1e-9);
      inner = need < 1 ? 1 : (need > cap ? cap : need);
    }
    const double eps_before = eps;
    int done = 0;
    for (int c = 0; c < inner && cyc < prm->max_cycles; ++c, ++cyc, ++done)
      if ((rc = adj_vcycle(C, 0, c == 0, st))) return rc;
    (C.split ? (outer ? k_adj_apply<true, true> : k_adj_apply<true, false>)
             : (outer ? k_adj_apply<false, true> : k_adj_apply<false, false>))<<<rows, bh, 0, st>>>(
        N, outer ? ldexp(1.0, -ex) : 1.0, w->lam, w->x[0]);
    note_launch(1);
    ++outer;
    if ((rc = residual())) return rc;
    eps = ldexp(sqrt(w->h_scal[0] / (double)n3), -ex) / snorm;
    if (nh < 64) S->resid_hist[nh++] = eps;
    if (done > 0 && eps > 0.0 && eps < eps_before && eps / eps_before > kFp32StepGain)
      rho_est = fmin(0.5, fmax(0.01, pow(eps / eps_before, 1.0 / done)));
  }
  if (outer == 0) MG_CUDA_TRY(cudaMemsetAsync(w->lam, 0, (size_t)n3 * 8, st));  // no correction was applied
  const int go = grid_for(n3);
  MG_ADJ_DISPATCH(m.kind, (k_adj_outputs<KK><<<go, kThreads, 0, st>>>(m, n3, w->lam, field, rho, grad_rho, w->partials,
                                                                      w->partials2)));
  k_adj_finalize<<<1, 1024, 0, st>>>(w->partials, w->partials2, go, w->scal);
  note_launch(1);
  if (grad_rho_raw) {
    k_adj_grad_raw<<<stream_grid(n3), kThreads, 0, st>>>(n3, grad_rho, w->scal + 1, ws->scalars + SC_MEAN,
                                                          grad_rho_raw);
    note_launch(1);
  }
  MG_CUDA_TRY(cudaMemcpyAsync(w->h_scal, w->scal, sizeof(double), cudaMemcpyDeviceToHost, st));
  MG_CUDA_TRY(cudaStreamSynchronize(st));
  MG_CUDA_TRY(cudaGetLastError());
  if (grad_theta) *grad_theta = w->h_scal[0];
  if (status == MGGLAM_OK && !isfinite(eps)) status = MGGLAM_ERR_NONFINITE;
  S->cycles = cyc;
  S->outer = outer;
  S->resid = eps;
  S->converged = eps <= tol;
  S->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (status == MGGLAM_OK && !S->converged) status = MGGLAM_ERR_NOT_CONVERGED;
  return status;
}

}  // namespace mg

extern "C" int mgglam_solve_adjoint(const mgglam_params* prm, double a, const double* field, const float* rho,
                                    int N, const double* grad_field, double* grad_rho, double* grad_rho_raw,
                                    double* grad_logfR0, double tol, mgglam_stats* stats, void* stream) {
  if (!prm || !field || !rho || !grad_field || !grad_rho || !(tol >= 0.0)) return MGGLAM_ERR_ARG;
  if (grad_rho_raw == grad_rho) return MGGLAM_ERR_ARG;
  if (N < 4 || N > 2048 || N % 2) return MGGLAM_ERR_SHAPE;
  if (prm->model != MGGLAM_FR && prm->model != MGGLAM_SYMMETRON) return MGGLAM_ERR_ARG;
  return mg::solve_adjoint(prm, a, field, rho, N, grad_field, grad_rho, grad_rho_raw, grad_logfR0, tol, stats,
                           (cudaStream_t)stream);
}
