// fft.cu -- the PM gravity solver: the periodic Poisson equation by FFT
// (Sec. 3.1: FFTs along x, y and z, multiplication by the Green's function of
// the discrete Laplacian, inverse FFTs; Eq. GR_poisson_codeunit).
//
//   grad_h^2 Phi = coef (rho/mean - 1),   Phi_k = -coef delta_k / K_h^2,
//   K_h^2 = sum_d 4 sin^2(pi k_d / N)   (the 7-point Laplacian's eigenvalues),
//   Phi_0 = 0 (the mean of Phi is not fixed by the equation).
//
// Single-precision FFTs of power-of-two length N = R1 R2 (R1, R2 <= 32) by one
// Cooley-Tukey split: with n = R2 n1 + n2 and k = k1 + R1 k2,
//   X[k1 + R1 k2] = sum_n2 W_R2^{n2 k2} [ W_N^{n2 k1} sum_n1 x[R2 n1 + n2] W_R1^{n1 k1} ],
// so a thread computes an R1-point DFT in registers, applies the twiddle
// W_N^{n2 k1} (table formed in double on the host), exchanges through shared
// memory once, and computes an R2-point DFT in registers.  Five passes over the
// mesh, each one read and one write:
//   z forward (real density in) -> y forward -> x forward, times the Green's
//   function, x inverse (one kernel) -> y inverse -> z inverse (real Phi out).
// A sixth launch, behind the first, transforms a density far from unit mean again,
// times a power of two.
// The density is real, so a z row is transformed as M = N/2 complex values
// x[2m] + i x[2m+1] and only its M + 1 independent modes are kept: every pass
// moves half of what complex rows move (40 instead of 72 bytes a cell), and at
// 256^3 the 67 MB of modes stay in the 126 MB L2 between passes while the density
// and the potential stream past them.  Measured with the density's sum: 143 us at
// 256^3 (257 us with complex rows), 1.58 ms at 512^3 (2.65); the row passes take
// about 35 and 42 us of it, bound by shared-memory and instruction issue between
// their barriers, the column passes 24, 34 and 24 us.
// z is the contiguous axis: a CTA transforms whole rows.  For y and x a CTA
// holds an N x TC tile (TC consecutive z modes of one plane or row), so each
// of its global accesses is a contiguous run of TC complex values.
#include <math.h>

#include <mutex>

#include "ff.cuh"
#include "mg_common.cuh"
#include "mg_internal.h"

namespace mg {

constexpr int kFftThreads = 256;

// exp(-2 pi i m / 32), m = 0..15: the twiddles of the register DFTs (R <= 32)
__constant__ float2 c_w32[16] = {
    {1.0f, 0.0f}, {0.980785251f, -0.195090324f}, {0.923879504f, -0.382683426f}, {0.831469595f, -0.555570245f},
    {0.707106769f, -0.707106769f}, {0.555570245f, -0.831469595f}, {0.382683426f, -0.923879504f},
    {0.195090324f, -0.980785251f}, {0.0f, -1.0f}, {-0.195090324f, -0.980785251f}, {-0.382683426f, -0.923879504f},
    {-0.555570245f, -0.831469595f}, {-0.707106769f, -0.707106769f}, {-0.831469595f, -0.555570245f},
    {-0.923879504f, -0.382683426f}, {-0.980785251f, -0.195090324f}};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__host__ __device__ constexpr int bitrev(int k, int R) {
  int r = 0;
  for (int b = 1; b < R; b <<= 1) {
    r = (r << 1) | (k & 1);
    k >>= 1;
  }
  return r;
}

// R-point DFT in registers (R a power of two <= 32): radix-2 decimation in
// frequency, natural input, bit-reversed output (X[k] in v[bitrev(k, R)]).
template <int R, bool INV>
__device__ __forceinline__ void dft_reg(float2 (&v)[R]) {
#pragma unroll
  for (int span = R / 2; span >= 1; span >>= 1) {
#pragma unroll
    for (int s = 0; s < R; s += 2 * span) {
#pragma unroll
      for (int j = 0; j < span; ++j) {
        const float2 a = v[s + j], b = v[s + j + span];
        v[s + j] = make_float2(a.x + b.x, a.y + b.y);
        float2 d = make_float2(a.x - b.x, a.y - b.y);
        if (j != 0) {  // W_{2 span}^j = W_32^{j 32 / (2 span)}
          float2 w = c_w32[j * (32 / (2 * span))];
          if (INV) w.y = -w.y;
          d = cmul(d, w);
        }
        v[s + j + span] = d;
      }
    }
  }
}

template <int R1, int R2>
__host__ __device__ constexpr int fft_threads_per_line() {
  return R1 > R2 ? R1 : R2;
}

// Resident CTAs per SM the register allocation is bounded for: four (64
// registers a thread) while a thread's DFT holds at most 16 complex values,
// two for the 32-point factors, whose 64 values would otherwise spill.
template <int R1, int R2>
__host__ __device__ constexpr int fft_min_ctas() {
  return (R1 > 16 || R2 > 16) ? 2 : 4;
}

// Phase 1 of a transform of length N = R1 R2 for the thread owning n2 (< R2):
// v holds x[R2 n1 + n2], n1 = 0..R1-1 (natural order); writes the twiddled
// R1-point DFT, W_N^{n2 k1} X1[k1], to ex(k1).  TT: the table holds W_N^{n2 k1} at
// k1 R2 + n2, else W_N^m at m: threads of different n2 then read one line.
template <int R1, int R2, bool INV, bool TT = false, class EX>
__device__ __forceinline__ void fft_phase1(float2 (&v)[R1], int n2, const float2* __restrict__ twN, EX ex) {
  dft_reg<R1, INV>(v);
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    float2 w = __ldg(&twN[TT ? k1 * R2 + n2 : n2 * k1]);
    if (INV) w.y = -w.y;
    ex(k1) = cmul(v[bitrev(k1, R1)], w);
  }
}

// Phase 3 for the thread owning k1 (< R1): u holds the twiddled values of all
// n2 (< R2); on return u[k2] = X[k1 + R1 k2] in natural order of k2.
template <int R2, bool INV>
__device__ __forceinline__ void fft_phase3(float2 (&u)[R2]) {
  dft_reg<R2, INV>(u);
  float2 t[R2];
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) t[k2] = u[bitrev(k2, R2)];
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) u[k2] = t[k2];
}

// Row length in the mode array: M + 1 modes, padded to whole 128-byte lines.
__host__ __device__ constexpr int mode_stride(int N) { return N / 2 + (N >= 32 ? 16 : 4); }

// The smaller factor F1 of a row's M = N/2 = F1 F2 complex values.
__host__ __device__ constexpr int row_f1(int N) { return N <= 16 ? 2 : (N <= 64 ? 4 : (N <= 256 ? 8 : 16)); }

// Rows per CTA of the row kernels.
__host__ __device__ constexpr int rows_per_cta(int N) {
  const int F2 = N / 2 / row_f1(N), L = kFftThreads / F2;
  return L < N * N ? L : N * N;
}

// Shared-memory strides of a row's exchange buffer (R1 x R2, padded) and of its M
// values in order; both shift the next row by half the banks at N = 256.
template <int R1, int R2>
__host__ __device__ constexpr int row_ex() { return R1 * (R2 + 1); }
__host__ __device__ constexpr int row_z(int M) { return M + 8; }

// Float-float sum over a warp (error ~1e-14, no FP64 instruction).
__device__ __forceinline__ ff warp_sum_ff(ff v) {
  for (int o = 16; o > 0; o >>= 1)
    v = ff_add(v, ff{__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o)});
  return v;
}

// Every pass but the first is a programmatic dependent launch (launch_pass): its CTAs
// are set up while the previous pass drains, and wait for its end here.
__device__ __forceinline__ void after_previous_pass() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// What the passes after the forward rows take of the density's mean.
struct FftScale {
  float green;   // -coef over the mean of what was transformed
  float factor;  // the rows are to be transformed again, times this power of two; 0: no
};

// The factor of the second transform.  The sums of a density in units of its own
// must stay within float's range -- up to 2 N^3 <= 2^31 times the mean, and the
// small modes above the subnormals -- and so must -coef / mean.  Means within 2^20
// of 1 leave room for all of them; the others are brought near 1, exactly.
__device__ __forceinline__ float fft_factor(double mean, double green) {
  const double m = fabs(mean), g = fabs(green);
  if (!(m < INFINITY)) return 0x1p-100f;  // the sum overflowed (or the density holds an infinity or a NaN)
  if (m == 0.0 || g == 0.0 || (m >= 0x1p-20 && m <= 0x1p20 && g >= 0x1p-100 && g <= 0x1p100)) return 0.f;
  return ldexpf(1.f, max(-126, min(-ilogb(m), 127)));
}

// Contiguous axis (z) forward, L whole rows of N = 2M reals per CTA, M = R1 R2.
// Each phase deals its own work to the CTA's threads, so that whole warps are
// either busy or done: L R2 threads load z[R2 n1 + r], z[m] = x[2m] + i x[2m+1],
// straight into registers (runs of R2 complex values) and exchange through shared
// memory; L R1 threads finish the transform and leave Z in natural order there;
// and M/2 threads a row untangle it:
//   E = Z[k] + conj Z[M-k], O = -i (Z[k] - conj Z[M-k]),
//   2 X[k] = E + W_N^k O,  2 X[M-k] = conj(E - W_N^k O)
// (the factor 2 goes into the inverse's scale).
// The pass also sums the density (float-float per CTA; the last CTA to finish adds
// the partial sums in order) and leaves -coef over its mean, which the Green's
// function takes in: a separate pass over the density took 28 us at 256^3.
// AGAIN: the pass over a density whose mean the first one found far from 1
// (fft_factor), a grid-stride loop whose CTAs otherwise return at once (4 us as an
// ordinary launch; with the dependent launches the whole call takes 143 us at 256^3,
// 150 without either, and 173 for a density of mean 1e35).
// pairs: rho is 8-byte aligned.
template <int R1, int R2, bool AGAIN>
__global__ void __launch_bounds__(kFftThreads, fft_min_ctas<R1, R2>()) k_rfft_rows_fwd(
    const float* __restrict__ rho, float2* __restrict__ modes, bool pairs, double coef,
    const float2* __restrict__ twN, const float2* __restrict__ twM, double* __restrict__ partials,
    unsigned* __restrict__ ticket, FftScale* scale) {
  constexpr int M = R1 * R2, N = 2 * M, S = mode_stride(N), L = rows_per_cta(N), NT = L * R2, H = M / 2;
  static_assert(R2 >= R1, "one thread per load of the first phase");
  extern __shared__ float2 fft_sm[];
  __shared__ ff s_part[kFftThreads / 32];
  __shared__ bool s_last;
  const int t = threadIdx.x;
  if (AGAIN) after_previous_pass();
  const float factor = AGAIN ? scale->factor : 1.f;
  if (AGAIN && factor == 0.f) return;
  float2* Zs = fft_sm + L * row_ex<R1, R2>();
  FloatFloat acc;
  auto rows = [&](unsigned block) {
    const long long row0 = (long long)block * L;
    {
      const int l = t / R2, r = t - l * R2;
      const float* x = rho + 2 * ((row0 + l) * M + r);
      float2 v[R1];
      if (pairs) {
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) v[n1] = __ldcs(reinterpret_cast<const float2*>(x + 2 * R2 * n1));
      } else {
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) v[n1] = make_float2(x[2 * R2 * n1], x[2 * R2 * n1 + 1]);
      }
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) {
        if (AGAIN) v[n1] = make_float2(v[n1].x * factor, v[n1].y * factor);
        acc.add(v[n1].x);
        acc.add(v[n1].y);
      }
      float2* Y = fft_sm + l * row_ex<R1, R2>() + r;
      fft_phase1<R1, R2, false, true>(v, r, twM, [&](int k1) -> float2& { return Y[k1 * (R2 + 1)]; });
    }
    if (!AGAIN) {
      const ff w = warp_sum_ff(ff{acc.hi, acc.lo});
      if ((t & 31) == 0) s_part[t >> 5] = w;
    }
    __syncthreads();
    if (t < L * R1) {
      const int l = t / R1, r = t - l * R1;
      const float2* Y = fft_sm + l * row_ex<R1, R2>() + r * (R2 + 1);
      float2 u[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) u[n2] = Y[n2];
      fft_phase3<R2, false>(u);
      float2* Z = Zs + l * row_z(M) + r;
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) Z[R1 * k2] = u[k2];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (L * H + NT - 1) / NT; ++q) {
      const int m = t + q * NT, l = m / H, k = m - l * H;
      if (l >= L) break;
      const float2* Z = Zs + l * row_z(M);
      float2* out = modes + (row0 + l) * S;
      if (k == 0) {
        // X[0] and X[M] from Z[0], X[M/2] from Z[M/2] (W_N^{M/2} = -i)
        const float2 a = Z[0], c = Z[H];
        out[0] = make_float2(2.f * (a.x + a.y), 0.f);
        out[M] = make_float2(2.f * (a.x - a.y), 0.f);
        out[H] = make_float2(2.f * c.x, -2.f * c.y);
      } else {
        const float2 a = Z[k], b = Z[M - k];
        const float2 e = make_float2(a.x + b.x, a.y - b.y);
        const float2 o = cmul(make_float2(a.y + b.y, b.x - a.x), __ldg(&twN[k]));
        out[k] = make_float2(e.x + o.x, e.y + o.y);
        out[M - k] = make_float2(e.x - o.x, o.y - e.y);
      }
    }
  };
  if constexpr (AGAIN) {
    for (unsigned block = blockIdx.x; block < N * N / L; block += gridDim.x) {
      rows(block);
      __syncthreads();  // the buffers are free for the next rows
    }
    const ff w = warp_sum_ff(ff{acc.hi, acc.lo});
    if ((t & 31) == 0) s_part[t >> 5] = w;
    __syncthreads();
  } else {
    rows(blockIdx.x);
  }
  if (t == 0) {
    ff p = s_part[0];
    for (int i = 1; i < (NT + 31) / 32; ++i) p = ff_add(p, s_part[i]);
    partials[blockIdx.x] = (double)p.hi + (double)p.lo;
    __threadfence();
    s_last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;  // back to 0 with the last CTA
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    double a = 0.0;
    for (unsigned i = t; i < gridDim.x; i += NT) a += __ldcg(&partials[i]);
    a = block_sum(a);
    if (t == 0) {
      const double mean = a / ((double)N * N * N), green = -coef / mean;
      scale->green = (float)green;
      if (!AGAIN) scale->factor = fft_factor(mean, green);
    }
  }
}

// Contiguous axis (z) inverse: the M + 1 modes of a row back to N reals, the
// forward pass in reverse (E and W_N^k O from X[k] and X[M-k], Z = E + i O, the
// inverse transform of length M); the potential is written past L2.
template <int R1, int R2>
__global__ void __launch_bounds__(kFftThreads, fft_min_ctas<R1, R2>()) k_rfft_rows_inv(
    const float2* __restrict__ modes, float* __restrict__ phi, bool pairs, float scale,
    const float2* __restrict__ twN, const float2* __restrict__ twM) {
  constexpr int M = R1 * R2, N = 2 * M, S = mode_stride(N), L = rows_per_cta(N), NT = L * R1;
  static_assert(R1 >= R2, "one thread per store of the last phase");
  extern __shared__ float2 fft_sm[];
  const int t = threadIdx.x;
  const long long row0 = (long long)blockIdx.x * L;
  float2* Zs = fft_sm + L * row_ex<R1, R2>();
  constexpr int H = M / 2;
  after_previous_pass();
#pragma unroll
  for (int q = 0; q < (L * H + NT - 1) / NT; ++q) {
    const int m = t + q * NT, l = m / H, k = m - l * H;
    if (l >= L) break;
    float2* Z = Zs + l * row_z(M);
    const float2* in = modes + (row0 + l) * S;
    if (k == 0) {
      const float2 a = in[0], b = in[M], c = in[H];
      Z[0] = make_float2(a.x + b.x, a.x - b.x);
      Z[H] = make_float2(2.f * c.x, -2.f * c.y);
    } else {
      const float2 a = in[k], b = in[M - k], tw = __ldg(&twN[k]);
      const float2 e = make_float2(a.x + b.x, a.y - b.y);
      const float2 o = cmul(make_float2(a.x - b.x, a.y + b.y), make_float2(tw.x, -tw.y));
      Z[k] = make_float2(e.x - o.y, e.y + o.x);
      Z[M - k] = make_float2(e.x + o.y, o.x - e.y);
    }
  }
  __syncthreads();
  if (t < L * R2) {
    const int l = t / R2, r = t - l * R2;
    const float2* Z = Zs + l * row_z(M) + r;
    float2 v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[n1] = Z[R2 * n1];
    float2* Y = fft_sm + l * row_ex<R1, R2>() + r;
    fft_phase1<R1, R2, true, true>(v, r, twM, [&](int k1) -> float2& { return Y[k1 * (R2 + 1)]; });
  }
  __syncthreads();
  {
    const int l = t / R1, r = t - l * R1;
    const float2* Y = fft_sm + l * row_ex<R1, R2>() + r * (R2 + 1);
    float2 u[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = Y[n2];
    fft_phase3<R2, true>(u);
    float* x = phi + 2 * ((row0 + l) * M + r);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const float2 v = make_float2(u[k2].x * scale, u[k2].y * scale);
      if (pairs) {
        __stcs(reinterpret_cast<float2*>(x + 2 * R1 * k2), v);
      } else {
        x[2 * R1 * k2] = v.x;
        x[2 * R1 * k2 + 1] = v.y;
      }
    }
  }
}

// Strided axis: element m of column c at base + m * stride_axis + c with
// base = blockIdx.y * stride_other + z0, z0 = blockIdx.x * TC; thread (c, r) =
// (t % TC, t / TC), so a warp's global accesses are runs of TC consecutive
// values.  The blocks past the last tile (blockIdx.x = M / TC) take the one
// remaining mode z = M, their columns running over TC values of the other axis.
// Exchange buffer Y[n2][k1] at (k1 R2 + n2) TC + c.
// GREEN (the x pass): the forward result X[k1 + R1 k2] stays in the registers
// of thread k1, is multiplied by -coef / K_h^2 (k_x = k1 + R1 k2, k_y =
// blockIdx.y, k_z = z0 + c) and transformed back with the two factors' roles
// swapped (input index R1 k2 + k1: phase 1 of length R2 over k2 by the thread
// owning k1, phase 3 of length R1), so the inverse starts from the registers;
// its output index is j1 + R2 j2.
template <int R1, int R2, bool INV, bool GREEN>
__global__ void __launch_bounds__(kFftThreads, fft_min_ctas<R1, R2>()) k_fft_cols(float2* __restrict__ data, int TC, long long stride_axis,
                                                             long long stride_other, const float2* __restrict__ twN,
                                                             const float* __restrict__ s2,
                                                             const FftScale* __restrict__ scale) {
  extern __shared__ float2 fft_sm[];
  const int c = threadIdx.x % TC, r = threadIdx.x / TC;
  constexpr int N = R1 * R2, M = N / 2;
  const bool last = (int)blockIdx.x * TC == M;
  after_previous_pass();
  if (last && (int)blockIdx.y * TC >= N) return;
  const int z = last ? M : blockIdx.x * TC + c;
  const int o = last ? blockIdx.y * TC + c : blockIdx.y;
  float2* col = data + (long long)o * stride_other + z;
  if (r < R2) {
    float2 v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[n1] = col[(long long)(R2 * n1 + r) * stride_axis];
    fft_phase1<R1, R2, INV>(v, r, twN, [&](int k1) -> float2& { return fft_sm[(k1 * R2 + r) * TC + c]; });
  }
  __syncthreads();
  float2 u[R2];
  if (r < R1) {
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = fft_sm[(r * R2 + n2) * TC + c];
    fft_phase3<R2, INV>(u);
    if constexpr (!GREEN) {
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) col[(long long)(r + R1 * k2) * stride_axis] = u[k2];
    }
  }
  if constexpr (GREEN) {
    __syncthreads();  // every phase-3 read of the exchange buffer is done
    if (r < R1) {
      const float sc = s2[o] + s2[z];
      const float cf = scale->green;  // delta = rho / mean - 1, whose constant drops out at k = 0
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const float K2 = s2[r + R1 * k2] + sc;
        // fast division (a few ulp): far below the transforms' own rounding
        const float g = K2 > 0.f ? __fdividef(cf, K2) : 0.f;
        u[k2] = make_float2(u[k2].x * g, u[k2].y * g);
      }
      // inverse, roles swapped: length-R2 DFTs over k2, twiddle W_N^{-r j1}
      fft_phase1<R2, R1, true>(u, r, twN, [&](int j1) -> float2& { return fft_sm[(j1 * R1 + r) * TC + c]; });
    }
    __syncthreads();
    if (r < R2) {
      float2 w[R1];
#pragma unroll
      for (int n2 = 0; n2 < R1; ++n2) w[n2] = fft_sm[(r * R1 + n2) * TC + c];
      fft_phase3<R1, true>(w);
#pragma unroll
      for (int j2 = 0; j2 < R1; ++j2) col[(long long)(r + R2 * j2) * stride_axis] = w[j2];
    }
  }
}

// Per-device, per-N plan: the mode array, twiddles and K_h^2 terms.
struct FftPlan {
  int device = -1;
  int N = 0;
  float2* buf = nullptr;
  float2* tw = nullptr;         // W_N^m, m < N; then W_M^{n2 k1} at k1 F2 + n2 and at k1 F1 + n2 (M = N/2 = F1 F2)
  float* s2 = nullptr;
  double* partials = nullptr;   // one per CTA of the forward rows pass
  FftScale* scale = nullptr;    // from the forward rows pass
  unsigned* ticket = nullptr;   // CTAs of the forward rows pass that have finished (0 between calls)
};

static void free_plan(FftPlan* p) {
  cudaFree(p->buf);
  cudaFree(p->tw);
  cudaFree(p->s2);
  cudaFree(p->partials);
  cudaFree(p->scale);
  cudaFree(p->ticket);
  delete p;
}

constexpr int kMaxFftPlans = 8;
static std::mutex g_fft_mu;
static FftPlan* g_fft[kMaxFftPlans];
static int g_nfft = 0;

static int fft_plan(int N, FftPlan** out) {
  int dev = 0;
  MG_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_fft_mu);
  for (int i = 0; i < g_nfft; ++i)
    if (g_fft[i]->device == dev && g_fft[i]->N == N) {
      *out = g_fft[i];
      return MGGLAM_OK;
    }
  if (g_nfft == kMaxFftPlans) return MGGLAM_ERR_OOM;
  FftPlan* p = new FftPlan;
  p->device = dev;
  p->N = N;
  bool ok = cudaMalloc(&p->buf, (size_t)N * N * mode_stride(N) * sizeof(float2)) == cudaSuccess &&
            cudaMalloc(&p->tw, 2 * (size_t)N * sizeof(float2)) == cudaSuccess &&
            cudaMalloc(&p->s2, (size_t)N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&p->partials, (size_t)N * N * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&p->scale, sizeof(FftScale)) == cudaSuccess &&
            cudaMalloc(&p->ticket, sizeof(unsigned)) == cudaSuccess &&
            cudaMemset(p->ticket, 0, sizeof(unsigned)) == cudaSuccess;
  if (ok) {
    float2* tw = new float2[2 * N];
    float* s2 = new float[N];
    for (int m = 0; m < N; ++m) {
      const double ang = -2.0 * M_PI * (double)m / (double)N;
      tw[m] = make_float2((float)cos(ang), (float)sin(ang));
    }
    const int M = N / 2, F1 = row_f1(N), F2 = M / F1;
    for (int m = 0; m < M; ++m) {
      tw[N + m] = tw[2 * ((m / F2) * (m % F2) % M)];
      tw[N + M + m] = tw[2 * ((m / F1) * (m % F1) % M)];
    }
    for (int k = 0; k < N; ++k) {
      const double s = sin(M_PI * (double)k / (double)N);
      s2[k] = (float)(4.0 * s * s);
    }
    ok = cudaMemcpy(p->tw, tw, 2 * (size_t)N * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(p->s2, s2, (size_t)N * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
    delete[] tw;
    delete[] s2;
  }
  if (!ok) {
    cudaGetLastError();
    free_plan(p);
    return MGGLAM_ERR_OOM;
  }
  g_fft[g_nfft++] = p;
  *out = p;
  return MGGLAM_OK;
}

void release_fft_plans() {
  std::lock_guard<std::mutex> lk(g_fft_mu);
  int dev = 0;
  cudaGetDevice(&dev);
  int keep = 0;
  for (int i = 0; i < g_nfft; ++i) {
    FftPlan* p = g_fft[i];
    if (p->device == dev) {
      free_plan(p);
    } else {
      g_fft[keep++] = p;
    }
  }
  g_nfft = keep;
}

static bool pow2_mesh(int N) { return N >= 8 && N <= 1024 && (N & (N - 1)) == 0; }

// Launch of a pass that starts with after_previous_pass.
template <typename... P, typename... A>
static cudaError_t launch_pass(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// CTAs of the second forward rows pass: four an SM.
constexpr unsigned kAgainCtas = 4 * 152;

// The five passes for N = R1 R2 (columns) and N/2 = F1 F2 (forward rows; the
// inverse swaps the two, so that its stores are runs of the larger factor).
// Columns kernel: TC = 256/T z modes per tile (at most N/2).  Dynamic shared
// memory: the exchange buffers (about 33 KB at N = 256, 66 KB at 1024).
template <int R1, int R2>
static int poisson_passes(const float* rho, float* phi, double coef, const FftPlan* p, cudaStream_t st) {
  constexpr int N = R1 * R2, M = N / 2, F1 = row_f1(N), F2 = M / F1, S = mode_stride(N), L = rows_per_cta(N);
  constexpr int T = fft_threads_per_line<R1, R2>();
  const long long NN = (long long)N * N, n3 = NN * N;
  const int TC = kFftThreads / T < M ? kFftThreads / T : M;
  const size_t fwd_smem = (size_t)L * (row_ex<F1, F2>() + row_z(M)) * sizeof(float2);
  const size_t inv_smem = (size_t)L * (row_ex<F2, F1>() + row_z(M)) * sizeof(float2);
  const size_t cols_smem = (size_t)N * TC * sizeof(float2);
  static bool attr_set[64] = {};  // per device: the opt-in above 48 KB, once
  if (p->device < 64 && !attr_set[p->device]) {
    for (auto kern : {k_rfft_rows_fwd<F1, F2, false>, k_rfft_rows_fwd<F1, F2, true>})
      MG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem));
    MG_CUDA_TRY(cudaFuncSetAttribute(k_rfft_rows_inv<F2, F1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)inv_smem));
    MG_CUDA_TRY(cudaFuncSetAttribute(k_fft_cols<R1, R2, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)cols_smem));
    MG_CUDA_TRY(cudaFuncSetAttribute(k_fft_cols<R1, R2, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)cols_smem));
    MG_CUDA_TRY(cudaFuncSetAttribute(k_fft_cols<R1, R2, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)cols_smem));
    attr_set[p->device] = true;
  }
  const unsigned rows_grid = (unsigned)(NN / L);
  const dim3 cols_grid(M / TC + 1, N);
  const long long sy = S, sx = (long long)N * S;
  prof_begin(PC_POISSON_FFT, st, 40.0 * n3);
  const unsigned again_grid = rows_grid < kAgainCtas ? rows_grid : kAgainCtas;
  const bool pairs = (uintptr_t)rho % 8 == 0;
  k_rfft_rows_fwd<F1, F2, false><<<rows_grid, L * F2, fwd_smem, st>>>(rho, p->buf, pairs, coef, p->tw, p->tw + N,
                                                                      p->partials, p->ticket, p->scale);
  MG_CUDA_TRY(launch_pass(k_rfft_rows_fwd<F1, F2, true>, again_grid, L * F2, fwd_smem, st, rho, p->buf, pairs, coef, p->tw,
                          p->tw + N, p->partials, p->ticket, p->scale));
  MG_CUDA_TRY(launch_pass(k_fft_cols<R1, R2, false, false>, cols_grid, TC * T, cols_smem, st, p->buf, TC, sy, sx, p->tw,
                          p->s2, nullptr));
  MG_CUDA_TRY(launch_pass(k_fft_cols<R1, R2, false, true>, cols_grid, TC * T, cols_smem, st, p->buf, TC, sx, sy, p->tw,
                          p->s2, p->scale));
  MG_CUDA_TRY(launch_pass(k_fft_cols<R1, R2, true, false>, cols_grid, TC * T, cols_smem, st, p->buf, TC, sy, sx, p->tw,
                          p->s2, nullptr));
  MG_CUDA_TRY(launch_pass(k_rfft_rows_inv<F2, F1>, rows_grid, L * F2, inv_smem, st, p->buf, phi, (uintptr_t)phi % 8 == 0,
                          (float)(0.5 / (double)n3), p->tw, p->tw + N + M));
  prof_end(st);
  note_launch(6);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int poisson_fft(const float* rho, int N, double coef, float* phi, cudaStream_t st) {
  if (!pow2_mesh(N)) return MGGLAM_ERR_SHAPE;
  FftPlan* p = nullptr;
  int rc = fft_plan(N, &p);
  if (rc) return rc;
  switch (N) {
    case 8: return poisson_passes<4, 2>(rho, phi, coef, p, st);
    case 16: return poisson_passes<4, 4>(rho, phi, coef, p, st);
    case 32: return poisson_passes<8, 4>(rho, phi, coef, p, st);
    case 64: return poisson_passes<8, 8>(rho, phi, coef, p, st);
    case 128: return poisson_passes<16, 8>(rho, phi, coef, p, st);
    case 256: return poisson_passes<16, 16>(rho, phi, coef, p, st);
    case 512: return poisson_passes<32, 16>(rho, phi, coef, p, st);
    default: return poisson_passes<32, 32>(rho, phi, coef, p, st);
  }
}

}  // namespace mg
