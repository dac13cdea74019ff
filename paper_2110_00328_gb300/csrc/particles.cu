// particles.cu -- CIC density assignment and the fifth-force gather (Sec. 3.1).
//
// Deposit: each particle spreads mass N^3/np over the 8 nearest cell centres
// (centre of cell c at c + 1/2) with weights prod_d (1 - |x_d - c_d - 1/2|),
// periodic.  The weights are accumulated as 64-bit fixed-point integers
// (units of 2^-32 of one particle's weight) with integer atomics, so the sum is
// independent of the order in which particles arrive: the mesh is bitwise
// reproducible.  A second pass scales to float32 density.
//
// Gather: the field transform T (f(R): f_R = -u^{n+1}; symmetron: u^2; CQ:
// beta phi) is formed once per cell in FP64 and stored as the FP32 perturbation
// T - Tbar (Tbar = T of the background field), which keeps the central
// difference (T_{c+1} - T_{c-1})/2 free of cancellation in single precision.
// Each particle then interpolates the three-point differences of the 8 cells
// around it with its CIC weights.
#include <math.h>

#include <mutex>

#include "bricks.cuh"
#include "cic.cuh"
#include "ff.cuh"
#include "mg_common.cuh"
#include "mg_internal.h"

namespace mg {

// round(x * 2^31) for 0 <= x < 2^32 by integer operations on the float's bits
// (exact for x >= 2^-8, whose bits all lie at or above 2^-31).
__device__ __forceinline__ unsigned long long fix31(float x) {
  const unsigned b = __float_as_uint(x);
  const int ex = (int)(b >> 23);
  if (ex == 0) return 0ull;  // zero (or subnormal: far below 2^-31)
  const unsigned long long m = (unsigned long long)((b & 0x7FFFFFu) | 0x800000u);
  const int sh = ex - 127 - 23 + 31;  // x * 2^31 = m * 2^sh
  if (sh >= 0) return m << sh;
  if (sh < -25) return 0ull;
  return (m + (1ull << (-sh - 1))) >> (-sh);
}

// CIC along one axis in fixed point: lower cell c0 = floor(x - 1/2) (periodic, 0 ..
// N-1) and the upper cell's weight F, the fractional part of x - 1/2 in units of
// 2^-31 (the lower one's is 2^31 - F) -- the same numbers the FP64 definition
// gives, without double-precision arithmetic (GB300's FP64 rate is 1/64 of FP32).
// From 1/2 on, x - 1/2, its integer part and its fraction are exact floats; below,
// and for positions to be wrapped, the integer form.
__device__ __noinline__ uint2 cic_axis_edge(float x, int N) {
  const long long xs = (long long)fix31(wrap_pos(x, N)) - (1ll << 30);
  const int c = (int)(xs >> 31);  // -1 .. N-1 (arithmetic shift = floor)
  return make_uint2((unsigned)(c < 0 ? c + N : c), (unsigned)(xs & 0x7FFFFFFFll));
}

__device__ __forceinline__ void cic_axis_fixed(float x, int N, int& c0, unsigned& F) {
  if (x >= 0.5f && x < (float)N) {
    const float xs = x - 0.5f;
    c0 = (int)xs;
    F = (unsigned)((xs - (float)c0) * 2147483648.f);
  } else {
    const uint2 e = cic_axis_edge(x, N);
    c0 = (int)e.x;
    F = e.y;
  }
}

// The upper cell of a pair.
__device__ __forceinline__ int next_cell(int c0, int N) { return c0 + 1 >= N ? 0 : c0 + 1; }

// round(P W / 2^61) 2^29 + (less than 2^29) for P <= 2^62, W <= 2^31: a product of
// three axis weights (units 2^-93), from its bits 32 and up, half a unit of the
// accumulator's 2^-32 added; the bits from 29 up are the rounded weight, exactly.
__device__ __forceinline__ unsigned long long wmul29(unsigned long long P, unsigned W) {
  return (unsigned long long)(unsigned)(P >> 32) * W + (__umulhi((unsigned)P, W) + (1u << 28));
}

// One particle per lane, warps over consecutive particles.  A lane's four
// cells in its upper k plane are the next lane's lower-plane cells whenever
// the two particles share (i0, j0) and sit in adjacent k cells (neighbours in
// a lattice-ordered particle array do): the next lane then adds them to its
// own and this lane skips those atomics.  Integer sums are exact, so the mesh
// does not depend on which lane issues an update.
template <typename IT>
__global__ void __launch_bounds__(kThreads) k_deposit_fixed(const float* __restrict__ pos, long long np, int N,
                                                            unsigned long long* __restrict__ acc,
                                                            const int* by_bricks) {
  if (left_to_bricks(by_bricks)) return;
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < np; base += stride) {
    const long long q = base + lane;
    const bool ok = q < np;
    int i0 = 0, i1 = 0, j0 = 0, j1 = 0, k0 = -1, k1 = -2;
    unsigned X1 = 0, Y1 = 0, Z1 = 0;
    if (ok) {
      cic_axis_fixed(pos[3 * q + 0], N, i0, X1);
      cic_axis_fixed(pos[3 * q + 1], N, j0, Y1);
      cic_axis_fixed(pos[3 * q + 2], N, k0, Z1);
      i1 = next_cell(i0, N);
      j1 = next_cell(j0, N);
      k1 = next_cell(k0, N);
    }
    const unsigned long long X0 = 0x80000000u - X1, Y0 = 0x80000000u - Y1;
    const unsigned Z0 = 0x80000000u - Z1;
    const unsigned long long P[4] = {X0 * Y0, X0 * Y1, X1 * Y0, (unsigned long long)X1 * Y1};  // (a, b) = 00, 01, 10, 11
    unsigned long long lo[4], up[4];                                          // k0 and k1 planes
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      lo[s] = wmul29(P[s], Z0) >> 29;
      up[s] = wmul29(P[s], Z1) >> 29;
    }
    const int pi = __shfl_up_sync(0xffffffffu, i0, 1), pj = __shfl_up_sync(0xffffffffu, j0, 1);
    const int pk = __shfl_up_sync(0xffffffffu, k1, 1);
    const bool take = lane > 0 && ok && pi == i0 && pj == j0 && pk == k0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const unsigned long long w = __shfl_up_sync(0xffffffffu, up[s], 1);
      if (take) lo[s] += w;
    }
    const bool given = __shfl_down_sync(0xffffffffu, (int)take, 1) != 0 && lane < 31;
    if (ok) {
      const IT ri[2] = {(IT)i0 * N, (IT)i1 * N};
      const int jj[2] = {j0, j1};
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const IT row = (ri[s >> 1] + jj[s & 1]) * N;
        if (lo[s]) atomicAdd(&acc[row + k0], lo[s]);
        if (!given && up[s]) atomicAdd(&acc[row + k1], up[s]);
      }
    }
  }
}

// The same deposit for lattice-ordered particles, brick by brick.
//
// k_deposit_fixed is bound by the L2's atomics: at 256^3 particles in a 256^3 mesh
// its 8 updates a particle are 110M requests (149M sectors), 410 us.  Particles
// kept in the order of the lattice they started from -- an M x M x M array, as
// simulations keep them -- stay near their neighbours, so a CTA takes a brick of 8
// x 8 x 32 of the array and adds it up in a window of the mesh in shared memory,
// centred on the brick's mean displacement: three cells of spread or more on every
// side of a brick of unit spacing (8 x 16 x 16 with a 14 x 22 x 22 window: 335 us
// where this one takes 325; its window's rows a warp each: no gain).  Then the
// window is one run of atomics (9M requests in all).  A 64-bit shared atomic is a
// compare-and-swap loop (357 us for as many random ones, against 181 us), so a sum
// is kept as two 32-bit words, of the weights' low 16 bits and of the bits above:
// 2048 weights of at most 2^32 fit.  A particle outside the window (1% of 256^3
// Zel'dovich particles of pixel sigma 1.5) goes to the mesh directly, so any
// positions are taken; the integer sums are the same in any order.
// Measured (those particles, the whole call): 470 us before, 335 with both kernels'
// launches; pixel sigma 5: 654 and 469.  Issue slots (69%) and the 16 shared atomics a
// particle (L1 68%) share the bound; 32-bit sums with a carry (8 atomics and few
// carries a particle) are no faster, nor are two CTAs an SM (348).
constexpr int kWinI = 14, kWinJ = 14, kWinK = 40;               // cells
constexpr int kWinCells = kWinI * kWinJ * kWinK;
constexpr int kBrickThreads = 512, kBrickPer = kBrickI * kBrickJ * kBrickK / kBrickThreads;
constexpr int kBrickOut = 256;                                  // particles outside a window kept for its end
static_assert(kBrickThreads == 2 * kBrickJ * kBrickK && kWinCells % 4 == 0, "two planes of a brick at a time");

// One particle's eight updates of the mesh itself.
template <typename IT>
__device__ __noinline__ void deposit_direct(const float* __restrict__ x, int N, unsigned long long* __restrict__ acc) {
  int c0[3];
  unsigned W1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) cic_axis_fixed(x[d], N, c0[d], W1[d]);
  const int i1 = next_cell(c0[0], N), j1 = next_cell(c0[1], N), k1 = next_cell(c0[2], N);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const unsigned long long P = (unsigned long long)(s & 2 ? W1[0] : 0x80000000u - W1[0]) *
                                 (s & 1 ? W1[1] : 0x80000000u - W1[1]);
    const IT row = ((IT)(s & 2 ? i1 : c0[0]) * N + (s & 1 ? j1 : c0[1])) * N;
    atomicAdd(&acc[row + c0[2]], wmul29(P, 0x80000000u - W1[2]) >> 29);
    atomicAdd(&acc[row + k1], wmul29(P, W1[2]) >> 29);
  }
}

template <typename IT>
__device__ __forceinline__ void deposit_brick(unsigned b, const float* __restrict__ pos, int M, int ni, int nbj, int nbk,
                                              int N, unsigned long long* __restrict__ acc) {
  extern __shared__ __align__(16) unsigned win[];  // low words, then high words; cleared 16 bytes at a time
  __shared__ int s_sum[4], s_nout;
  __shared__ unsigned short s_out[kBrickOut];  // particles outside the window
  const int t = threadIdx.x;
  const unsigned bij = b / (unsigned)nbk, bk = b - bij * nbk, bi = bij / (unsigned)nbj, bj = bij - bi * nbj;
  const int i0 = bi * kBrickI + t / (kBrickJ * kBrickK), j0 = bj * kBrickJ + (t / kBrickK) % kBrickJ,
            k0 = bk * kBrickK + t % kBrickK;
  const float* brick = pos + 3 * (((long long)bi * kBrickI * M + bj * kBrickJ) * M + bk * kBrickK);  // its first particle
  const float* mine = pos + 3 * (((long long)i0 * M + j0) * M + k0);  // this thread's, two planes apart
  const long long two = 6ll * M * M;
  const int mp = j0 < M && k0 < M ? min(kBrickPer, (ni - i0 + 1) >> 1) : 0;  // this thread's particles
  float x[kBrickPer][3];
#pragma unroll
  for (int r = 0; r < kBrickPer; ++r)
#pragma unroll
    for (int d = 0; d < 3; ++d) x[r][d] = r < mp ? mine[r * two + d] : 0.f;
  if (t < 4) s_sum[t] = 0;
  if (t == 4) s_nout = 0;
  uint4* z = reinterpret_cast<uint4*>(win);
  for (int i = t; i < 2 * kWinCells / 4; i += kBrickThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  // window origin: the particles' mean place, measured from the brick's first one, less half a
  // window
  const float ref[3] = {wrap_pos(brick[0], N), wrap_pos(brick[1], N), wrap_pos(brick[2], N)};
  {
    const float fN = (float)N, iN = 1.f / (float)N;
    int sum[4] = {0, 0, 0, mp};
#pragma unroll
    for (int r = 0; r < kBrickPer; ++r)
      if (r < mp) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float o = x[r][d] - ref[d];
          sum[d] += (int)rintf(o - fN * rintf(o * iN));  // nearest image: at most N/2, unless the position is far outside
        }
      }
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const int w = __reduce_add_sync(0xffffffffu, sum[d]);
      if ((t & 31) == 0) atomicAdd(&s_sum[d], w);
    }
  }
  __syncthreads();
  int org[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int half = (d == 0 ? kWinI : (d == 1 ? kWinJ : kWinK)) / 2;
    org[d] = ((int)(ref[d] + __fdividef((float)s_sum[d], (float)s_sum[3])) - half) % N;
    org[d] += org[d] < 0 ? N : 0;
  }
#pragma unroll
  for (int r = 0; r < kBrickPer; ++r) {
    if (r >= mp) break;
    int c[3];
    unsigned F[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cic_axis_fixed(x[r][d], N, c[d], F[d]);
      c[d] -= org[d];
      c[d] += c[d] < 0 ? N : 0;
    }
    if (c[0] + 1 < kWinI && c[1] + 1 < kWinJ && c[2] + 1 < kWinK) {
      const unsigned X0 = 0x80000000u - F[0], Y0 = 0x80000000u - F[1], Z0 = 0x80000000u - F[2];
      unsigned* w = win + (c[0] * kWinJ + c[1]) * kWinK + c[2];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const unsigned long long P = (unsigned long long)(s & 2 ? F[0] : X0) * (s & 1 ? F[1] : Y0);
        const unsigned long long w0 = wmul29(P, Z0), w1 = wmul29(P, F[2]);
        unsigned* a = w + ((s >> 1) * kWinJ + (s & 1)) * kWinK;
        atomicAdd(a, (unsigned)(w0 >> 29) & 0xffffu);
        atomicAdd(a + kWinCells, (unsigned)(w0 >> 45));
        atomicAdd(a + 1, (unsigned)(w1 >> 29) & 0xffffu);
        atomicAdd(a + kWinCells + 1, (unsigned)(w1 >> 45));
      }
    } else {
      const int q = atomicAdd(&s_nout, 1);
      if (q < kBrickOut) s_out[q] = (unsigned short)(t + r * kBrickThreads);
      else deposit_direct<IT>(mine + r * two, N, acc);
    }
  }
  __syncthreads();
  for (int a = t; a < kWinCells; a += kBrickThreads) {
    const unsigned long long v = ((unsigned long long)win[kWinCells + a] << 16) + win[a];
    if (v) {
      const int ij = a / kWinK, wi = ij / kWinJ;
      int i = org[0] + wi, j = org[1] + ij - wi * kWinJ, k = org[2] + a - ij * kWinK;
      i -= i >= N ? N : 0;  // N >= the window's sides: one wrap
      j -= j >= N ? N : 0;
      k -= k >= N ? N : 0;
      atomicAdd(&acc[((IT)i * N + j) * N + k], v);
    }
  }
  for (int q = t; q < min(s_nout, kBrickOut); q += kBrickThreads) {
    const int p = s_out[q];
    const int i = p / (kBrickJ * kBrickK), j = (p / kBrickK) % kBrickJ, k = p % kBrickK;
    deposit_direct<IT>(brick + 3 * (((long long)i * M + j) * M + k), N, acc);
  }
}

// Three CTAs an SM for the whole kernel, which take the bricks in turns: where the
// particles are in no order 456 CTAs come and go in a microsecond, one a brick in five
// (256^3, 192^3: 1270 and 278 us a call, 1259 and 276 so, 1259 and 274 by singles alone).
constexpr unsigned kBrickCtas = 3 * 152;
template <typename IT>
__global__ void __launch_bounds__(kBrickThreads, 3) k_deposit_bricks(const float* __restrict__ pos, int M, int ni,
                                                                     int nbj, int nbk, unsigned bricks, int N,
                                                                     unsigned long long* __restrict__ acc,
                                                                     const int* by_bricks) {
  next_may_start();
  if (!*by_bricks) return;
#pragma unroll 1
  for (unsigned b = blockIdx.x; b < bricks; b += gridDim.x) {
    deposit_brick<IT>(b, pos, M, ni, nbj, nbk, N, acc);
    __syncthreads();  // the window is free for the next brick
  }
}

// acc <- 0, and brick_probe beside it.
__global__ void __launch_bounds__(kThreads) k_deposit_clear(unsigned long long* __restrict__ acc, long long n3,
                                                            const float* __restrict__ pos, int N, BrickGrid b,
                                                            int* __restrict__ by_bricks) {
  if (blockIdx.x == 0) brick_probe(pos, N, b, by_bricks);
  ulonglong2* a = reinterpret_cast<ulonglong2*>(acc);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3 >> 1;
       t += (long long)gridDim.x * blockDim.x)
    a[t] = make_ulonglong2(0ull, 0ull);
  if ((n3 & 1) && blockIdx.x == 0 && threadIdx.x == 0) acc[n3 - 1] = 0ull;
}

// Where the deposit's kernels learn whether the particles go by bricks: the word behind
// acc's N^3.
static int* deposit_flag(unsigned long long* acc, int N) { return reinterpret_cast<int*>(acc + (long long)N * N * N); }

// Clears acc for np particles, and asks for the deposit's order where it will be in question.
static int clear_deposit(const float* pos, long long np, long long lattice, int N, unsigned long long* acc,
                         cudaStream_t st) {
  const long long n3 = (long long)N * N * N;
  const BrickGrid b = brick_grid(np, lattice, N, kWinK);
  if (!b.blocks) {
    MG_CUDA_TRY(cudaMemsetAsync(acc, 0, (size_t)n3 * sizeof(unsigned long long), st));
    return MGGLAM_OK;
  }
  k_deposit_clear<<<stream_grid(n3), kThreads, 0, st>>>(acc, n3, pos, N, b, deposit_flag(acc, N));
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

// The deposit of np particles on acc, brick by brick (brick_grid; at fewer particles the
// window's zeroing and flush, four cells a particle, cost more than the atomics they
// save) or in the order of the array.  lattice: M, or 0.  probed: clear_deposit has asked
// which, of these particles.
static int launch_deposit(const float* pos, long long np, long long lattice, int N, unsigned long long* acc,
                          bool probed, cudaStream_t st) {
  const BrickGrid b = brick_grid(np, lattice, N, kWinK);
  // 32-bit cell offsets where the mesh has at most 2^30 cells
  auto singles = N <= 1024 ? k_deposit_fixed<int> : k_deposit_fixed<long long>;
  if (b.blocks) {
    constexpr int smem = 2 * kWinCells * (int)sizeof(unsigned);
    auto kern = N <= 1024 ? k_deposit_bricks<int> : k_deposit_bricks<long long>;
    MG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int* by_bricks = deposit_flag(acc, N);
    if (!probed) k_brick_probe<<<1, 256, 0, st>>>(pos, N, b, by_bricks);
    kern<<<b.blocks < kBrickCtas ? b.blocks : kBrickCtas, kBrickThreads, smem, st>>>(pos, b.M, b.ni, b.nbj, b.nbk, b.blocks, N,
                                                                                      acc, by_bricks);
    MG_CUDA_TRY(launch_beside_bricks(singles, grid_for(np, kThreads, 1 << 20), kThreads, st, pos, np, N, acc, by_bricks));
    note_launch(probed ? 1 : 2);
  } else {
    singles<<<grid_for(np, kThreads, 1 << 20), kThreads, 0, st>>>(pos, np, N, acc, nullptr);
  }
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

__global__ void k_deposit_finish(const unsigned long long* __restrict__ acc, long long n3, double mass,
                                 float* __restrict__ rho) {
  // single-precision scaling of the correctly rounded float of the sum (the
  // output is FP32): within one ulp of the exact product
  const float s = (float)(mass / 4294967296.0);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x)
    rho[t] = __ull2float_rn(acc[t]) * s;
}

// Scratch for the fixed-point accumulator, cached per (device, N).
static int deposit_scratch(int N, unsigned long long** acc) {
  Workspace* ws = nullptr;
  int rc = get_workspace(N < 4 ? 4 : (N % 2 ? N + 1 : N), MGGLAM_FP64, 1, &ws);
  if (rc) return rc;
  const size_t need = ((size_t)N * N * N + 1) * sizeof(unsigned long long);  // and by_bricks
  if (ws->cic_bytes < need) {
    if (ws->cic_acc) cudaFree(ws->cic_acc);
    ws->cic_acc = nullptr;
    ws->cic_bytes = 0;
    if (cudaMalloc((void**)&ws->cic_acc, need) != cudaSuccess) {
      cudaGetLastError();
      return MGGLAM_ERR_OOM;
    }
    ws->cic_bytes = need;
  }
  *acc = (unsigned long long*)ws->cic_acc;
  return MGGLAM_OK;
}

int deposit_cic(const float* pos, long long np, int N, float* rho, cudaStream_t st) {
  unsigned long long* acc = nullptr;
  int rc = deposit_scratch(N, &acc);
  if (rc) return rc;
  const long long n3 = (long long)N * N * N;
  if ((rc = clear_deposit(pos, np, lattice_side(np), N, acc, st))) return rc;
  prof_begin(PC_DEPOSIT, st, 12.0 * np);
  if ((rc = launch_deposit(pos, np, lattice_side(np), N, acc, true, st))) return rc;
  prof_end(st);
  prof_begin(PC_DEPOSIT_FINISH, st, 12.0 * n3);
  k_deposit_finish<<<stream_grid(n3), kThreads, 0, st>>>(acc, n3, (double)n3 / (double)np, rho);
  prof_end(st);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

// ---------------------------------------------------------------------------
// Gather
// ---------------------------------------------------------------------------

// T - Tbar per cell, stored in FP32.  f(R) and the symmetron form it in
// float-float (FP32 instructions; the exact split of the FP64 field, v - ubar
// exact to first order, ~48-bit products), which rounds to the same float as
// FP64 would at 1/64 of FP32's rate; CQ (one product) stays in FP64.
// Also brick_probe, where b is a grid of bricks.
template <int K>
__global__ void __launch_bounds__(kThreads) k_transform(const double* __restrict__ u, long long n3, double ubar,
                                                        double beta, float* __restrict__ T,
                                                        const float* __restrict__ pos, int N, BrickGrid b,
                                                        int* __restrict__ by_bricks) {
  if (b.blocks && blockIdx.x == 0) brick_probe(pos, N, b, by_bricks);
  const ff ub = ff_from_double(ubar);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n3;
       t += (long long)gridDim.x * blockDim.x) {
    if constexpr (K == KCQ) {
      T[t] = (float)(beta * u[t]);
    } else {
      const ff v = ff_from_double(u[t]);
      const ff dv = ff_sub(v, ub);  // v - ubar
      ff d;
      if constexpr (K == KFR0) d = ff_neg(dv);
      else if constexpr (K == KFR1) d = ff_neg(ff_mul(dv, ff_add(v, ub)));
      else if constexpr (K == KFR2) d = ff_neg(ff_mul(dv, ff_add(ff_add(ff_sqr(v), ff_mul(v, ub)), ff_sqr(ub))));
      else d = ff_mul(dv, ff_add(v, ub));  // symmetron: u^2 - ubar^2
      T[t] = ff_to_float(d);
    }
  }
}

// One particle per thread (cic_grad: the 32 distinct cells its three central
// differences at the 8 CIC cells touch).
template <typename IT, int THREADS>
__global__ void __launch_bounds__(THREADS) k_gather(const float* __restrict__ T, int N, const float* __restrict__ pos,
                                                    long long np, float scale, float* __restrict__ force,
                                                    const int* by_bricks) {
  if (left_to_bricks(by_bricks)) return;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < np;
       q += (long long)gridDim.x * blockDim.x) {
    const float3 g = cic_grad<IT>(T, N, pos[3 * q + 0], pos[3 * q + 1], pos[3 * q + 2]);
    force[3 * q + 0] = scale * g.x;
    force[3 * q + 1] = scale * g.y;
    force[3 * q + 2] = scale * g.z;
  }
}

// The same gather brick by brick (brick_gradients).  Measured (256^3 Zel'dovich
// particles of pixel sigma 1.5, with the transform's 39 us): 361 us before, 285 with both
// kernels' launches; sigma 3: 605 and 378.
template <typename IT, bool QUADS>
__global__ void __launch_bounds__(kTileThreads, 4) k_gather_bricks(const float* __restrict__ T, int N,
                                                                   const float* __restrict__ pos, BrickGrid b,
                                                                   float scale, float* __restrict__ force,
                                                                   const int* by_bricks) {
  next_may_start();
  if (!*by_bricks) return;
  brick_gradients<IT, QUADS>(T, N, pos, b, [&](long long p, float3 g) {
    force[p] = scale * g.x;
    force[p + 1] = scale * g.y;
    force[p + 2] = scale * g.z;
  });
}

// Beside the bricks the particles go by blocks of 768 threads (two an SM): fewer that
// come and go, and they keep more of a warp's lines in L1.  Shuffled 256^3 particles 1598
// us, 1649 by blocks of 256 alone; ordered ones 283 by bricks with 16384 such blocks
// beside, 289 with one for every 768 particles.
constexpr int kWideThreads = 768, kWideBlocks = 16384;

// The gather's bricks: the deposit's, in a mesh of at least the window's longest side,
// where N np >= 8.4e8.  In a mesh much coarser than the lattice the particles of a warp
// share their cells, the single-particle kernel finds them in L1, and few bricks are no
// gain.  Measured (singles / bricks, us; cells, particles): 96^3, 177^3 85 / 88; 128^3,
// 185^3 98 / 100; 64^3, 216^3 133 / 135; on the other side 160^3, 177^3 115 / 100; 128^3,
// 192^3 112 / 104; 96^3, 216^3 139 / 137; 64^3, 256^3 213 / 203.
static BrickGrid gather_bricks(long long np, long long lattice, int N) {
  return brick_grid(np, (double)N * (double)np >= 8.4e8 ? lattice : 0, N, kTileK);
}

// The gather of np particles.  lattice, probed: as launch_deposit's (the transform asks).
static int launch_gather(const float* T, int N, const float* pos, long long np, long long lattice, float scale,
                         float* force, int* by_bricks, bool probed, cudaStream_t st) {
  const BrickGrid b = gather_bricks(np, lattice, N);
  if (b.blocks) {
    constexpr int smem = kTileCells * (int)sizeof(float);
    const bool quads = N % 4 == 0;  // T's rows on 16-byte boundaries (the workspace's mesh is)
    auto kern = N <= 1024 ? (quads ? k_gather_bricks<int, true> : k_gather_bricks<int, false>)
                          : (quads ? k_gather_bricks<long long, true> : k_gather_bricks<long long, false>);
    MG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (!probed) k_brick_probe<<<1, 256, 0, st>>>(pos, N, b, by_bricks);
    kern<<<b.blocks, kTileThreads, smem, st>>>(T, N, pos, b, scale, force, by_bricks);
    auto singles = N <= 1024 ? k_gather<int, kWideThreads> : k_gather<long long, kWideThreads>;
    MG_CUDA_TRY(launch_beside_bricks(singles, grid_for(np, kWideThreads, kWideBlocks), kWideThreads, st, T, N, pos, np,
                                     scale, force, by_bricks));
    note_launch(probed ? 1 : 2);
  } else {
    // 32-bit cell offsets where the mesh has at most 2^30 cells
    (N <= 1024 ? k_gather<int, kThreads> : k_gather<long long, kThreads>)<<<grid_for(np, kThreads, 1 << 20), kThreads, 0,
                                                                            st>>>(T, N, pos, np, scale, force, nullptr);
  }
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

// Force prefactor of the gather (the spatial factor of the model's fifth force, times the caller's).
static double force_scale(const ModelDev& m, int kind, const mgglam_params* prm) {
  if (is_fr(kind)) return 0.5 * m.c2;  // F = (c~^2/2) grad f_R
  if (kind == KSYM)
    return -3.0 * prm->xi * prm->xi * prm->omega_m * prm->beta_star * prm->beta_star * m.c2 /
           (prm->a_star * prm->a_star * prm->a_star);
  return -1.0;  // F = -grad(beta phi)
}

// The gather of a range of particles on the mesh T the last gather_force call
// on this stream formed (the workspace's scratch mesh).
int gather_chunk(const ModelDev& m, int kind, const mgglam_params* prm, int N, const float* pos, long long np,
                 float* force, double prefactor, cudaStream_t st, long long lattice) {
  Workspace* ws = nullptr;
  int rc = get_workspace(N, MGGLAM_MIXED, 0, &ws);
  if (rc) return rc;
  const float* T = ws->lev[0].ub;
  prof_begin(PC_GATHER, st, 24.0 * np);
  rc = launch_gather(T, N, pos, np, lattice, (float)(force_scale(m, kind, prm) * prefactor), force,
                     by_bricks_of(ws), false, st);
  prof_end(st);
  return rc;
}

int gather_force(const ModelDev& m, int kind, int n_fr, const mgglam_params* prm, const double* field, int N,
                 const float* pos, long long np, float* force, double prefactor, cudaStream_t st, long long lattice) {
  (void)n_fr;
  Workspace* ws = nullptr;
  int rc = get_workspace(N, MGGLAM_MIXED, 0, &ws);
  if (rc) return rc;
  float* T = ws->lev[0].ub;  // scratch mesh of N^3 floats
  const long long n3 = (long long)N * N * N;
  const int g = stream_grid(n3);
  if (lattice < 0) lattice = lattice_side(np);
  const BrickGrid b = gather_bricks(np, lattice, N);
  int* by_bricks = by_bricks_of(ws);
  double scale;
  prof_begin(PC_TRANSFORM, st, 12.0 * n3);
  switch (kind) {
    case KFR0: k_transform<KFR0><<<g, kThreads, 0, st>>>(field, n3, m.ubar, 0.0, T, pos, N, b, by_bricks); break;
    case KFR1: k_transform<KFR1><<<g, kThreads, 0, st>>>(field, n3, m.ubar, 0.0, T, pos, N, b, by_bricks); break;
    case KFR2: k_transform<KFR2><<<g, kThreads, 0, st>>>(field, n3, m.ubar, 0.0, T, pos, N, b, by_bricks); break;
    case KSYM: k_transform<KSYM><<<g, kThreads, 0, st>>>(field, n3, m.ubar, 0.0, T, pos, N, b, by_bricks); break;
    default: k_transform<KCQ><<<g, kThreads, 0, st>>>(field, n3, 0.0, prm->beta, T, pos, N, b, by_bricks); break;
  }
  prof_end(st);
  scale = force_scale(m, kind, prm);
  prof_begin(PC_GATHER, st, 24.0 * np + 4.0 * n3);
  note_launch(1);
  rc = launch_gather(T, N, pos, np, lattice, (float)(scale * prefactor), force, by_bricks, true, st);
  prof_end(st);
  return rc;
}

// ---------------------------------------------------------------------------
// Host input / output overlapped with the kernels
// ---------------------------------------------------------------------------
//
// The particles live in page-locked host memory.  The deposit copies them to a
// device buffer in chunks on a second stream, and deposits chunk c as soon as
// its copy has landed (stream-ordered by an event), so the host-link copy and
// the atomics overlap; the gather computes chunk c and copies its forces back
// while chunk c+1 is computed.  One copy stream and an event pool per device.

constexpr int kMaxIoChunks = 32;

struct HostIo {
  int device = -1;
  cudaStream_t cs = nullptr;
  cudaEvent_t ev[kMaxIoChunks + 2] = {};
};

static int host_io(HostIo** out) {
  static std::mutex mu;
  static HostIo io[16];
  int dev = 0;
  MG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 16) return MGGLAM_ERR_CUDA;
  std::lock_guard<std::mutex> lk(mu);
  HostIo& h = io[dev];
  if (h.device != dev) {
    MG_CUDA_TRY(cudaStreamCreateWithFlags(&h.cs, cudaStreamNonBlocking));
    for (int i = 0; i < kMaxIoChunks + 2; ++i)
      MG_CUDA_TRY(cudaEventCreateWithFlags(&h.ev[i], cudaEventDisableTiming));
    h.device = dev;
  }
  *out = &h;
  return MGGLAM_OK;
}

int deposit_cic_host(const float* pos_host, float* pos_dev, long long np, int N, float* rho, int chunks,
                     cudaStream_t st) {
  unsigned long long* acc = nullptr;
  int rc = deposit_scratch(N, &acc);
  if (rc) return rc;
  HostIo* io = nullptr;
  if ((rc = host_io(&io))) return rc;
  const long long n3 = (long long)N * N * N;
  const long long per = (np + chunks - 1) / chunks;
  MG_CUDA_TRY(cudaMemsetAsync(acc, 0, (size_t)n3 * sizeof(unsigned long long), st));
  // the copies must not overwrite pos_dev before earlier work on st is done with it
  MG_CUDA_TRY(cudaEventRecord(io->ev[kMaxIoChunks], st));
  MG_CUDA_TRY(cudaStreamWaitEvent(io->cs, io->ev[kMaxIoChunks], 0));
  prof_begin(PC_DEPOSIT, st, 12.0 * np);
  for (int c = 0; c < chunks; ++c) {
    const long long q0 = c * per, cnt = q0 >= np ? 0 : (np - q0 < per ? np - q0 : per);
    if (cnt <= 0) break;
    MG_CUDA_TRY(cudaMemcpyAsync(pos_dev + 3 * q0, pos_host + 3 * q0, (size_t)cnt * 12, cudaMemcpyHostToDevice,
                                io->cs));
    MG_CUDA_TRY(cudaEventRecord(io->ev[c], io->cs));
    MG_CUDA_TRY(cudaStreamWaitEvent(st, io->ev[c], 0));
    // a chunk that ends between lattice planes is no lattice
    const long long M = lattice_side(np);
    if ((rc = launch_deposit(pos_dev + 3 * q0, cnt, M > 0 && q0 % (M * M) == 0 ? M : 0, N, acc, false, st)))
      return rc;
  }
  prof_end(st);
  prof_begin(PC_DEPOSIT_FINISH, st, 12.0 * n3);
  k_deposit_finish<<<stream_grid(n3), kThreads, 0, st>>>(acc, n3, (double)n3 / (double)np, rho);
  prof_end(st);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}

int gather_force_host(const ModelDev& m, int kind, const mgglam_params* prm, const double* field, int N,
                      const float* pos_dev, long long np, float* force_dev, float* force_host, double prefactor,
                      int chunks, cudaStream_t st) {
  HostIo* io = nullptr;
  int rc = host_io(&io);
  if (rc) return rc;
  // the transform and the first chunk's gather, then per chunk: gather, hand the chunk to the copy stream
  const long long per = (np + chunks - 1) / chunks;
  const long long M = lattice_side(np);
  for (int c = 0; c < chunks; ++c) {
    const long long q0 = c * per, cnt = q0 >= np ? 0 : (np - q0 < per ? np - q0 : per);
    if (cnt <= 0) break;
    const long long lattice = M > 0 && q0 % (M * M) == 0 ? M : 0;  // a chunk that ends between planes is no lattice
    if (c == 0) {
      // transform + gather of the first chunk through the common path
      if ((rc = gather_force(m, kind, prm->n, prm, field, N, pos_dev, cnt, force_dev, prefactor, st, lattice)))
        return rc;
    } else {
      if ((rc = gather_chunk(m, kind, prm, N, pos_dev + 3 * q0, cnt, force_dev + 3 * q0, prefactor, st,
                             lattice)))
        return rc;
    }
    MG_CUDA_TRY(cudaEventRecord(io->ev[c], st));
    MG_CUDA_TRY(cudaStreamWaitEvent(io->cs, io->ev[c], 0));
    MG_CUDA_TRY(cudaMemcpyAsync(force_host + 3 * q0, force_dev + 3 * q0, (size_t)cnt * 12, cudaMemcpyDeviceToHost,
                                io->cs));
  }
  // the caller's stream completes after the last copy
  MG_CUDA_TRY(cudaEventRecord(io->ev[kMaxIoChunks + 1], io->cs));
  MG_CUDA_TRY(cudaStreamWaitEvent(st, io->ev[kMaxIoChunks + 1], 0));
  return MGGLAM_OK;
}

}  // namespace mg

// ---------------------------------------------------------------------------
// Deposit without allocation (mgglam_deposit_cic_static)
// ---------------------------------------------------------------------------
//
// The accumulator lives in a fixed file-scope device array instead of the
// scratch cache, so this entry point never calls cudaMalloc.  The array's name
// is only a host-side stand-in in host code; the device address comes from
// cudaGetSymbolAddress, looked up once per device (with that device current)
// on the first call and cached until mgglam_release runs on that device (a
// reset device reloads the module, which may move the array).

namespace mg {

constexpr int kStaticDepositMaxN = 128;
constexpr size_t kStaticDepositCells = (size_t)kStaticDepositMaxN * kStaticDepositMaxN * kStaticDepositMaxN;
constexpr int kStaticMaxDevices = 64;

static __device__ __align__(256) unsigned long long g_static_deposit_acc[kStaticDepositCells + 1];  // and by_bricks

static std::mutex g_static_mu;
static unsigned long long* g_static_acc_ptr[kStaticMaxDevices];

static int static_deposit_scratch(unsigned long long** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return MGGLAM_ERR_CUDA;
  }
  if (dev < 0 || dev >= kStaticMaxDevices) return MGGLAM_ERR_ARG;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_acc_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_deposit_acc);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return MGGLAM_ERR_CUDA;
    }
    g_static_acc_ptr[dev] = (unsigned long long*)p;
  }
  *out = g_static_acc_ptr[dev];
  return MGGLAM_OK;
}

void forget_static_deposit_address() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  if (dev < 0 || dev >= kStaticMaxDevices) return;
  std::lock_guard<std::mutex> lk(g_static_mu);
  g_static_acc_ptr[dev] = nullptr;
}

}  // namespace mg

extern "C" int mgglam_deposit_cic_static(const float* pos, long long np, int N, float* rho, void* stream) {
  using namespace mg;
  if (!pos || !rho || np < 1) return MGGLAM_ERR_ARG;
  if (N < 2 || N > kStaticDepositMaxN) return MGGLAM_ERR_SHAPE;
  unsigned long long* acc = nullptr;
  int rc = static_deposit_scratch(&acc);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const long long n3 = (long long)N * N * N;
  // the array keeps the previous call's sums: clear the part this call uses
  if ((rc = clear_deposit(pos, np, lattice_side(np), N, acc, st))) return rc;
  if ((rc = launch_deposit(pos, np, lattice_side(np), N, acc, true, st))) return rc;
  k_deposit_finish<<<stream_grid(n3), kThreads, 0, st>>>(acc, n3, (double)n3 / (double)np, rho);
  note_launch(1);
  MG_CUDA_TRY(cudaGetLastError());
  return MGGLAM_OK;
}
