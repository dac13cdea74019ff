// solve64.cu -- FP64 multigrid kernels and the plain-FP64 FAS solver.
//
// FAS V-cycle (Sec. 3.2.1): on each level nu1 red-black sweeps, restriction of
// u and of the local residual d (8-child mean), coarse source
// S^H = N^H(R u) - R d (Eq. general_pde_numerical_coarse), coarse initial guess
// R u, recursion, correction u += P(u^H - R u) (Eq. solution_correction, 27/9/3/1
// weights), nu2 sweeps.  The coarsest level is relaxed with a fixed number of
// sweeps by a single CTA.
#include <math.h>
#include <stdio.h>

#include <chrono>

#include "fp64_fast.cuh"
#include "mg_common.cuh"
#include "mg_internal.h"

namespace mg {

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
//
// All of them are bound by the FP64 pipe (fp64_fast.cuh), not by memory: at 96^3
// a colour pass reads 21 MB, 3 us from HBM, and issues 15 FP64 instructions a
// cell, 11 us at 0.58e12 a second.  So the work is laid out to spend few of
// those: products folded into the sums, one reciprocal a cell, transfers that
// share their partial sums, and nothing formed that is known.

// Threads of the 3D kernels: 16 cells along k by 16 rows j of one plane i.  Rows
// of 48 or 80 cells fill them, which 64 threads along k did not.
constexpr int kTx = 16, kTy = 16;
#define MG_CELL3(nk, nj)                              \
  const int k = blockIdx.x * kTx + threadIdx.x;       \
  const int j = blockIdx.y * kTy + threadIdx.y;       \
  const int i = blockIdx.z;                           \
  if (k >= (nk) || j >= (nj)) return

// Sum over the six face neighbours of the field that enters the Laplacian
// (f(R): w = u^{n+1}; symmetron, CQ: u itself), the power folded into the sum.
template <int K>
__device__ __forceinline__ double nb_sum64(const double* u, int n, int i, int j, int k) {
  const int ip = wrapi(i + 1, n), im = wrapi(i - 1, n);
  const int jp = wrapi(j + 1, n), jm = wrapi(j - 1, n);
  const int kp = wrapi(k + 1, n), km = wrapi(k - 1, n);
  const double v[6] = {u[cidx(n, ip, j, k)], u[cidx(n, im, j, k)], u[cidx(n, i, jp, k)],
                       u[cidx(n, i, jm, k)], u[cidx(n, i, j, kp)], u[cidx(n, i, j, km)]};
  double s = fr_or_id<K>(v[0]);
#pragma unroll
  for (int t = 1; t < 6; ++t) {
    if constexpr (K == KFR1) s = fma(v[t], v[t], s);
    else if constexpr (K == KFR2) s = fma(v[t] * v[t], v[t], s);
    else s += v[t];
  }
  return s;
}

// Relax every cell of one colour ((i+j+k) % 2 == parity); one thread per cell.
// Measured (f(R) n = 1): 15.6 us a pass at 96^3, 30.8 us at 128^3 (of that 11 and 26 us is the FP64
// pipe); with cube root, square root and cosine in FP64 a 128^3 pass took 205 us.
template <int K>
__global__ void __launch_bounds__(kTx* kTy) k_smooth64(Const64 c, int n, double* u, const double* __restrict__ rho,
                                                       const double* __restrict__ S, int parity) {
  MG_CELL3(n >> 1, n);
  const int kc = 2 * k + ((i + j + parity) & 1);
  const size_t t = cidx(n, i, j, kc);
  const double Lnb = nb_sum64<K>(u, n, i, j, kc);
  u[t] = local_update64<K>(c, u[t], rho[t], S ? S[t] : 0.0, Lnb);
}

// d = N(u) - S on every cell; optional store of d; per-block partial sums of d^2.
template <int K>
__global__ void __launch_bounds__(kThreads) k_residual64(Const64 c, int n, const double* __restrict__ u,
                                                         const double* __restrict__ rho,
                                                         const double* __restrict__ S, double* __restrict__ d,
                                                         double* __restrict__ partials) {
  double acc = 0.0;
  // grid-stride over rows (i, j), threads along k
  for (int r = blockIdx.x; r < n * n; r += gridDim.x) {
    const int i = r / n, j = r - (r / n) * n;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const size_t t = cidx(n, i, j, k);
      const double N = local_N64<K>(c, u[t], rho[t], nb_sum64<K>(u, n, i, j, k));
      const double v = S ? N - S[t] : N;
      if (d) d[t] = v;
      acc = fma(v, v, acc);
    }
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// Sum 'count' partials in a fixed order into *out (one block).
__global__ void k_finalize_sum(const double* __restrict__ partials, int count, double* __restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += partials[i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) *out = acc;
}

// coarse = mean of the 8 children.
__global__ void __launch_bounds__(kTx* kTy) k_restrict64(int nf, const double* __restrict__ fine,
                                                         double* __restrict__ coarse) {
  const int nc = nf >> 1;
  MG_CELL3(nc, nc);
  double s = 0.0;
  for (int di = 0; di < 2; ++di)
    for (int dj = 0; dj < 2; ++dj)
      for (int dk = 0; dk < 2; ++dk) s += fine[cidx(nf, 2 * i + di, 2 * j + dj, 2 * k + dk)];
  coarse[cidx(nc, i, j, k)] = s * 0.125;
}

// Fused: for each coarse cell, the local residual of its 8 children is formed
// on the fly (the recomputation the paper also does, Sec. 3.2.2) and averaged
// into Rd; the children's solution is averaged into Ru and copied to uH.
// ZR (f(R), symmetron, after pre-smoothing): the second colour ((i+j+k) odd) was
// relaxed last, to the exact root of its own equation, so its residual is that
// root's rounding; it is taken as zero and only the four first-colour children's
// residuals are formed (as the mixed path does).
template <int K, bool ZR>
__global__ void __launch_bounds__(kTx* kTy) k_residual_restrict64(Const64 c, int nf, const double* __restrict__ u,
                                                                  const double* __restrict__ rho,
                                                                  const double* __restrict__ S,
                                                                  double* __restrict__ Ru, double* __restrict__ uH,
                                                                  double* __restrict__ Rd) {
  static_assert(!ZR || K != KCQ, "CQ relaxes by one Newton step: its residual is not zero");
  const int nc = nf >> 1;
  MG_CELL3(nc, nc);
  double su = 0.0, sd = 0.0;
#pragma unroll
  for (int di = 0; di < 2; ++di)
#pragma unroll
    for (int dj = 0; dj < 2; ++dj)
#pragma unroll
      for (int dk = 0; dk < 2; ++dk) {
        const int a = 2 * i + di, b = 2 * j + dj, e = 2 * k + dk;
        const size_t t = cidx(nf, a, b, e);
        const double uc = u[t];
        su += uc;
        if (ZR && ((di + dj + dk) & 1)) continue;
        const double N = local_N64<K>(c, uc, rho[t], nb_sum64<K>(u, nf, a, b, e));
        sd += S ? N - S[t] : N;
      }
  const size_t t = cidx(nc, i, j, k);
  const double ru = su * 0.125;
  Ru[t] = ru;
  uH[t] = ru;
  Rd[t] = sd * 0.125;
}

// In place: S <- N^H(Ru) - S, where S holds R d on entry.
template <int K>
__global__ void __launch_bounds__(kTx* kTy) k_fas_source64(Const64 c, int n, const double* __restrict__ Ru,
                                                           const double* __restrict__ rho, double* __restrict__ S) {
  MG_CELL3(n, n);
  const size_t t = cidx(n, i, j, k);
  S[t] = local_N64<K>(c, Ru[t], rho[t], nb_sum64<K>(Ru, n, i, j, k)) - S[t];
}

// u^h += P(u^H - R u^h), the 27/9/3/1 (/64) weights; f(R): non-positive results
// fall back to half the old value.  One thread per coarse cell, whose eight
// children interpolate from the 27 coarse differences around it: the weights
// factor into (3, 1) per axis, so the children share the sums along k and j (65
// FP64 instructions for eight cells; a child at a time they are 152).
template <bool FR>
__global__ void __launch_bounds__(kTx* kTy) k_prolong_correct64(int nc, const double* __restrict__ uH,
                                                                const double* __restrict__ RuH,
                                                                double* __restrict__ uf,
                                                                unsigned long long* guard) {
  MG_CELL3(nc, nc);
  const int nf = nc << 1;
  const int Iv[3] = {wrapi(i - 1, nc), i, wrapi(i + 1, nc)};
  const int Jv[3] = {wrapi(j - 1, nc), j, wrapi(j + 1, nc)};
  const int Kv[3] = {wrapi(k - 1, nc), k, wrapi(k + 1, nc)};
  double jk[3][2][2];  // [I offset][j child][k child]
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    double r[3][2];  // [J offset][k child]
#pragma unroll
    for (int y = 0; y < 3; ++y) {
      double d[3];
#pragma unroll
      for (int z = 0; z < 3; ++z) {
        const size_t t = cidx(nc, Iv[x], Jv[y], Kv[z]);
        d[z] = uH[t] - RuH[t];
      }
      r[y][0] = fma(3.0, d[1], d[0]);
      r[y][1] = fma(3.0, d[1], d[2]);
    }
#pragma unroll
    for (int ck = 0; ck < 2; ++ck) {
      jk[x][0][ck] = fma(3.0, r[1][ck], r[0][ck]);
      jk[x][1][ck] = fma(3.0, r[1][ck], r[2][ck]);
    }
  }
  unsigned ng = 0;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int ck = 0; ck < 2; ++ck) {
        const double corr = fma(3.0, jk[1][b][ck], jk[a ? 2 : 0][b][ck]);
        const size_t t = cidx(nf, 2 * i + a, 2 * j + b, 2 * k + ck);
        const double old = uf[t];
        double v = fma(corr, 1.0 / 64.0, old);
        if (FR && !(v > 0.0)) {
          v = 0.5 * old;
          ++ng;
        }
        uf[t] = v;
      }
  if (FR) count_guards(guard, ng);
}

// Coarsest level: 'sweeps' red-black sweeps by one CTA (the level is tiny), the
// field in shared memory; a thread's cells are the same in every sweep.
constexpr int kCoarseThreads = 512;
template <int K>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse64(Const64 c, int n, double* __restrict__ u,
                                                             const double* __restrict__ rho,
                                                             const double* __restrict__ S, int sweeps) {
  extern __shared__ double su[];
  const int n3 = n * n * n, h = n >> 1;
  for (int t = threadIdx.x; t < n3; t += blockDim.x) su[t] = u[t];
  __syncthreads();
  for (int s = 0; s < 2 * sweeps; ++s) {
    // the s & 1 colour: cell kk of row (i, j), k = 2 kk + (i + j + s) & 1 (an odd row length
    // leaves its last cell to the colour of even k)
    for (int t = threadIdx.x; t < (h + (n & 1)) * n * n; t += blockDim.x) {
      const int w = h + (n & 1), kk = t % w, r = t / w, j = r % n, i = r / n;
      const int k = 2 * kk + ((i + j + s) & 1);
      if (k >= n) continue;
      const int o = (i * n + j) * n + k;
      const double Lnb = nb_sum64<K>(su, n, i, j, k);
      su[o] = local_update64<K>(c, su[o], rho[o], S ? S[o] : 0.0, Lnb);
    }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < n3; t += blockDim.x) u[t] = su[t];
}

__global__ void k_sum_f32(const float* __restrict__ x, long long n3, double* __restrict__ partials) {
  FloatFloat acc;  // FP32 arithmetic (GB300's FP64 rate is 1/64 of FP32), exact to ~1e-14
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x)
    acc.add(x[t]);
  const double a = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = a;
}

// rho64 = rho32 / mean, mean = sum / n3 read from device memory.
__global__ void k_density_to64(const float* __restrict__ rho32, long long n3, const double* __restrict__ sum,
                               double* __restrict__ rho64) {
  const double inv_mean = block_ratio((double)n3, sum);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x)
    rho64[t] = (double)rho32[t] * inv_mean;
}

// Sum of squares of the model's linear source term (relative-residual scale).
template <int K>
__global__ void k_src_sumsq(ModelDev m, const double* __restrict__ rho, long long n3, double* __restrict__ partials) {
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x) {
    const double delta = rho[t] - 1.0;
    double s;
    if constexpr (is_fr(K)) s = m.om_a * delta;
    else if constexpr (K == KSYM) s = m.msym * m.rat3 * delta * m.ubar;
    else s = m.cq_src * delta;
    acc += s * s;
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// If field[0] is NaN, fill the field with the background value.
__global__ void k_init_background(double* __restrict__ field, long long n3, double ubar) {
  if (!isnan(field[0])) return;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x)
    if (t != 0) field[t] = ubar;
}
__global__ void k_init_background_first(double* __restrict__ field, double ubar) {
  if (isnan(field[0])) field[0] = ubar;
}

// ---------------------------------------------------------------------------
// Launchers (dispatch on the model kind)
// ---------------------------------------------------------------------------

// Grid of the 3D kernels (x: k, y: j, z: i) for blocks of kTx x kTy threads.
static dim3 grid3d(int n_k, int n_j, int n_i) { return dim3((n_k + kTx - 1) / kTx, (n_j + kTy - 1) / kTy, n_i); }
static const dim3 kBlock3(kTx, kTy);

#define MG_DISPATCH(kind, KERNEL_CALL)                       \
  switch (kind) {                                            \
    case KFR0: { constexpr int KK = KFR0; KERNEL_CALL; note_launch(1); } break; \
    case KFR1: { constexpr int KK = KFR1; KERNEL_CALL; note_launch(1); } break; \
    case KFR2: { constexpr int KK = KFR2; KERNEL_CALL; note_launch(1); } break; \
    case KSYM: { constexpr int KK = KSYM; KERNEL_CALL; note_launch(1); } break; \
    case KCQ: { constexpr int KK = KCQ; KERNEL_CALL; note_launch(1); } break;   \
    default: return MGGLAM_ERR_ARG;                          \
  }

int launch_smooth64(const ModelDev& m, int n, double h, double* u, const double* rho, const double* S,
                    int sweeps, cudaStream_t st) {
  const dim3 g = grid3d(n / 2, n, n);
  const Const64 c = make_const64(m, h);
  for (int s = 0; s < sweeps; ++s)
    for (int parity = 0; parity < 2; ++parity) {
      MG_DISPATCH(m.kind, (k_smooth64<KK><<<g, kBlock3, 0, st>>>(c, n, u, rho, S, parity)));
    }
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_residual64(const ModelDev& m, int n, double h, const double* u, const double* rho,
                      const double* S, double* d, double* partials, double* out_sum, cudaStream_t st) {
  const long long n3 = (long long)n * n * n;
  const int g = n * n < 2048 ? n * n : 2048;
  const int bt = n >= 256 ? 256 : (n <= 32 ? 32 : ((n + 31) / 32) * 32);
  MG_DISPATCH(m.kind, (k_residual64<KK><<<g, bt, 0, st>>>(make_const64(m, h), n, u, rho, S, d, partials)));
  k_finalize_sum<<<1, 1024, 0, st>>>(partials, g, out_sum);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_restrict64(int nf, const double* fine, double* coarse, cudaStream_t st) {
  k_restrict64<<<grid3d(nf / 2, nf / 2, nf / 2), kBlock3, 0, st>>>(nf, fine, coarse);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_prolong_correct64(const ModelDev& m, int nc, const double* uH, const double* RuH,
                             unsigned long long* guard, double* uf, cudaStream_t st) {
  const dim3 g = grid3d(nc, nc, nc);
  if (is_fr(m.kind)) k_prolong_correct64<true><<<g, kBlock3, 0, st>>>(nc, uH, RuH, uf, guard);
  else k_prolong_correct64<false><<<g, kBlock3, 0, st>>>(nc, uH, RuH, uf, guard);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_coarse64(const ModelDev& m, int n, double h, double* u, const double* rho, const double* S,
                    int sweeps, cudaStream_t st) {
  if ((long long)n * n * n > 4096) return launch_smooth64(m, n, h, u, rho, S, sweeps, st);
  const size_t smem = (size_t)n * n * n * sizeof(double);  // at most 32 KB
  MG_DISPATCH(m.kind, (k_coarse64<KK><<<1, kCoarseThreads, smem, st>>>(make_const64(m, h), n, u, rho, S, sweeps)));
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_residual_restrict64(const ModelDev& m, int nf, double hf, const double* u, const double* rho,
                               const double* S, double* Ru, double* uH, double* Rd, bool relaxed, cudaStream_t st) {
  const dim3 g = grid3d(nf / 2, nf / 2, nf / 2);
  const Const64 c = make_const64(m, hf);
  if (relaxed && m.kind != KCQ) {
    switch (m.kind) {
      case KFR0: k_residual_restrict64<KFR0, true><<<g, kBlock3, 0, st>>>(c, nf, u, rho, S, Ru, uH, Rd); break;
      case KFR1: k_residual_restrict64<KFR1, true><<<g, kBlock3, 0, st>>>(c, nf, u, rho, S, Ru, uH, Rd); break;
      case KFR2: k_residual_restrict64<KFR2, true><<<g, kBlock3, 0, st>>>(c, nf, u, rho, S, Ru, uH, Rd); break;
      default: k_residual_restrict64<KSYM, true><<<g, kBlock3, 0, st>>>(c, nf, u, rho, S, Ru, uH, Rd); break;
    }
    note_launch(1);
  } else {
    MG_DISPATCH(m.kind, (k_residual_restrict64<KK, false><<<g, kBlock3, 0, st>>>(c, nf, u, rho, S, Ru, uH, Rd)));
  }
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_fas_source64(const ModelDev& m, int nc, double hc, const double* Ru, const double* rho, double* S,
                        cudaStream_t st) {
  MG_DISPATCH(m.kind, (k_fas_source64<KK><<<grid3d(nc, nc, nc), kBlock3, 0, st>>>(make_const64(m, hc), nc, Ru, rho, S)));
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_density_mean(const float* rho32, size_t n3, double* partials, double* out_sum, cudaStream_t st) {
  const int g = stream_grid((long long)n3);
  k_sum_f32<<<g, kThreads, 0, st>>>(rho32, (long long)n3, partials);
  k_finalize_sum<<<1, 1024, 0, st>>>(partials, g, out_sum);
  note_launch(2);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_density_to64(const float* rho32, size_t n3, const double* sum, double* rho64, cudaStream_t st) {
  k_density_to64<<<stream_grid((long long)n3), kThreads, 0, st>>>(rho32, (long long)n3, sum, rho64);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_src_sumsq(const ModelDev& m, const double* rho64, size_t n3, double* partials, double* out,
                     cudaStream_t st) {
  const int g = grid_for((long long)n3);
  MG_DISPATCH(m.kind, (k_src_sumsq<KK><<<g, kThreads, 0, st>>>(m, rho64, (long long)n3, partials)));
  k_finalize_sum<<<1, 1024, 0, st>>>(partials, g, out);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int launch_init_background(const ModelDev& m, double* field, size_t n3, cudaStream_t st) {
  k_init_background<<<stream_grid((long long)n3), kThreads, 0, st>>>(field, (long long)n3, m.ubar);
  k_init_background_first<<<1, 1, 0, st>>>(field, m.ubar);
  note_launch(2);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

// ---------------------------------------------------------------------------
// FP64 solver
// ---------------------------------------------------------------------------

// One multigrid cycle from level l (Sec. 3.2.1): mode 0 V, 1 F, 2 W.
static int vcycle64(const ModelDev& m, Workspace* ws, int l, const mgglam_params* prm, cudaStream_t st,
                    int mode = -1) {
  if (mode < 0) mode = prm->cycle;
  Level& L = ws->lev[l];
  int rc;
  if (l == ws->nlev - 1) return launch_coarse64(m, L.n, L.h, L.u, L.rho, L.S, prm->coarse_sweeps, st);
  if (l == 0) prof_begin(PC_SMOOTH64_FINE, st, 24.0 * L.n3 * prm->nu1);
  if ((rc = launch_smooth64(m, L.n, L.h, L.u, L.rho, L.S, prm->nu1, st))) return rc;
  if (l == 0) prof_end(st);
  Level& C = ws->lev[l + 1];
  // Ru -> C.Ru, u^H = Ru -> C.u, R d -> C.S (then C.S <- N^H(Ru) - R d)
  if (l == 0) prof_begin(PC_RESTRICT64_FINE, st, (16.0 + 3.0) * L.n3);
  if ((rc = launch_residual_restrict64(m, L.n, L.h, L.u, L.rho, L.S, C.Ru, C.u, C.S, prm->nu1 > 0, st))) return rc;
  if (l == 0) { prof_end(st); prof_begin(PC_COARSE_LEVELS, st, 0.0); }
  if ((rc = launch_fas_source64(m, C.n, C.h, C.Ru, C.rho, C.S, st))) return rc;
  if ((rc = vcycle64(m, ws, l + 1, prm, st, mode))) return rc;
  if (mode != 0 && (rc = vcycle64(m, ws, l + 1, prm, st, mode == 2 ? 2 : 0))) return rc;
  if (l == 0) { prof_end(st); prof_begin(PC_PROLONG64_FINE, st, (16.0 + 2.0) * L.n3); }
  if ((rc = launch_prolong_correct64(m, C.n, C.u, C.Ru, guard_of(ws), L.u, st))) return rc;
  if (l == 0) { prof_end(st); prof_begin(PC_SMOOTH64_FINE, st, 24.0 * L.n3 * prm->nu2); }
  rc = launch_smooth64(m, L.n, L.h, L.u, L.rho, L.S, prm->nu2, st);
  if (l == 0) prof_end(st);
  return rc;
}

// Full-multigrid start (prm->fmg): every level poses N^H(u^H) = 0 on its restricted
// density; the coarsest level relaxes from the background value, and each finer
// level starts from the plain prolongation of the coarser result (the correction
// kernel applied to a zero field with a zero coarse reference) and takes one
// cycle.  Level 0 (the caller's field) holds the result.
static int fmg_start64(const ModelDev& m, Workspace* ws, const mgglam_params* prm, cudaStream_t st) {
  const int L = ws->nlev;
  Level& C = ws->lev[L - 1];
  int rc;
  if ((rc = launch_init_background(m, C.u, C.n3, st))) return rc;
  if (L > 1) MG_CUDA_TRY(cudaMemsetAsync(C.S, 0, C.n3 * sizeof(double), st));
  if ((rc = launch_coarse64(m, C.n, C.h, C.u, C.rho, L > 1 ? C.S : nullptr, prm->coarse_sweeps, st))) return rc;
  for (int l = L - 2; l >= 0; --l) {
    Level& F = ws->lev[l];
    Level& H = ws->lev[l + 1];
    MG_CUDA_TRY(cudaMemsetAsync(F.u, 0, F.n3 * sizeof(double), st));
    MG_CUDA_TRY(cudaMemsetAsync(H.Ru, 0, H.n3 * sizeof(double), st));
    if ((rc = launch_prolong_correct64(m, H.n, H.u, H.Ru, nullptr, F.u, st))) return rc;
    if (l > 0) MG_CUDA_TRY(cudaMemsetAsync(F.S, 0, F.n3 * sizeof(double), st));
    if ((rc = vcycle64(m, ws, l, prm, st, 0))) return rc;
  }
  return MGGLAM_OK;
}

int solve_fp64(const mgglam_params* prm, double a, const float* rho, int N, double* field, double tol,
               mgglam_stats* stats, cudaStream_t st) {
  auto t0 = std::chrono::steady_clock::now();
  ModelDev m;
  int rc = make_model(prm, a, N, &m);
  if (rc) return rc;
  Workspace* ws = nullptr;
  if ((rc = get_workspace(N, MGGLAM_FP64, prm->levels, &ws))) return rc;
  Level& F = ws->lev[0];
  F.u = field;
  const size_t n3 = F.n3;
  // density: FP64 mean (a2), normalised FP64 copy, restricted down the levels
  if ((rc = launch_density_mean(rho, n3, ws->partials, ws->scalars + SC_MEAN, st))) return rc;
  if ((rc = launch_density_to64(rho, n3, ws->scalars + SC_MEAN, F.rho, st))) return rc;
  for (int l = 1; l < ws->nlev; ++l)
    if ((rc = launch_restrict64(ws->lev[l - 1].n, ws->lev[l - 1].rho, ws->lev[l].rho, st))) return rc;
  if ((rc = launch_init_background(m, field, n3, st))) return rc;
  MG_CUDA_TRY(cudaMemsetAsync(guard_of(ws), 0, sizeof(unsigned long long), st));
  if ((rc = launch_src_sumsq(m, F.rho, n3, ws->partials, ws->scalars + SC_SRC, st))) return rc;
  if ((rc = launch_residual64(m, F.n, F.h, field, F.rho, nullptr, nullptr, ws->partials,
                              ws->scalars + SC_SUMSQ, st)))
    return rc;
  MG_CUDA_TRY(cudaMemcpyAsync(ws->h_scalars, ws->scalars, SC_COUNT * sizeof(double), cudaMemcpyDeviceToHost, st));
  MG_CUDA_TRY(cudaStreamSynchronize(st));
  const double src = sqrt(ws->h_scalars[SC_SRC] / (double)n3);
  const double snorm = source_norm(m, src);
  double eps = sqrt(ws->h_scalars[SC_SUMSQ] / (double)n3) / snorm;
  mgglam_stats local;
  mgglam_stats* S = stats ? stats : &local;
  memset(S, 0, sizeof(*S));
  S->resid0 = eps;
  S->resid_hist[0] = eps;
  int cyc = 0, nh = 1;
  const int every = prm->check_every > 0 ? prm->check_every : 1;
  int status = MGGLAM_OK;
  while (!(eps <= tol) && cyc < prm->max_cycles) {
    if (!isfinite(eps)) { status = MGGLAM_ERR_NONFINITE; break; }
    if (prm->fmg && m.kind != KCQ && cyc == 0) {
      if ((rc = fmg_start64(m, ws, prm, st))) return rc;
    } else if ((rc = vcycle64(m, ws, 0, prm, st))) {
      return rc;
    }
    ++cyc;
    if (cyc % every == 0 || cyc == prm->max_cycles) {
      if ((rc = launch_residual64(m, F.n, F.h, field, F.rho, nullptr, nullptr, ws->partials,
                                  ws->scalars + SC_SUMSQ, st)))
        return rc;
      MG_CUDA_TRY(cudaMemcpyAsync(ws->h_scalars + SC_SUMSQ, ws->scalars + SC_SUMSQ, sizeof(double),
                                  cudaMemcpyDeviceToHost, st));
      MG_CUDA_TRY(cudaStreamSynchronize(st));
      eps = sqrt(ws->h_scalars[SC_SUMSQ] / (double)n3) / snorm;
      if (nh < 64) S->resid_hist[nh++] = eps;
    }
  }
  if (status == MGGLAM_OK && !isfinite(eps)) status = MGGLAM_ERR_NONFINITE;
  MG_CUDA_TRY(cudaMemcpyAsync(ws->h_scalars + SC_GUARD, guard_of(ws), sizeof(unsigned long long),
                              cudaMemcpyDeviceToHost, st));
  MG_CUDA_TRY(cudaStreamSynchronize(st));
  S->guarded = (long long)*reinterpret_cast<const unsigned long long*>(ws->h_scalars + SC_GUARD);
  S->cycles = cyc;
  S->resid = eps;
  S->converged = eps <= tol;
  S->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (status == MGGLAM_OK && !S->converged) status = MGGLAM_ERR_NOT_CONVERGED;
  return status;
}

}  // namespace mg
