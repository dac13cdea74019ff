// bricks.cuh -- particles in the order of a lattice, taken a brick of the lattice at a
// time: the deposit's sums and the gradients' mesh values then sit in shared memory.
#pragma once
#include <cuda_pipeline.h>
#include <math.h>
#include "cic.cuh"

namespace mg {

constexpr int kBrickI = 8, kBrickJ = 8, kBrickK = 32;  // particles

constexpr long long kBrickBlocks = 3000;

// The bricks of an M x M x ni array; blocks = 0: not taken.
struct BrickGrid {
  int M, ni, nbj, nbk;
  unsigned blocks;
};

// np particles (a multiple of M^2; M = lattice, or 0: in no such order) go by bricks from
// 3000 bricks (177^3 particles) and half a particle a cell on -- the window of a sparser
// lattice's brick covers fewer of its particles -- in a mesh of at least the window's
// longest side.  Fewer bricks are a few waves of CTAs with a last one that is nearly
// empty.  Measured (singles / bricks, us, whole calls; cells, particles): deposit 128^3,
// 177^3 121 / 112; 176^3, 177^3 161 / 134; 192^3, 185^3 190 / 153; 192^3, 192^3 204 / 154;
// 240^3, 192^3 248 / 199; 320^3, 256^3 573 / 446; gather, in the same order but for the
// first (gather_bricks), 132 / 112; 153 / 128; 160 / 131; 205 / 168; 505 / 375.  Below, the
// kernels alone: deposit 128^3, 104^3 45.4 / 49.2; 128^3, 128^3 63.5 / 55.1; gather 34.9 /
// 39.6; 45.1 / 43.1.
static inline BrickGrid brick_grid(long long np, long long lattice, int N, int window) {
  const long long M = lattice, ni = M > 0 ? np / (M * M) : 0;
  const long long nbj = (M + kBrickJ - 1) / kBrickJ, nbk = (M + kBrickK - 1) / kBrickK,
                  blocks = (ni + kBrickI - 1) / kBrickI * nbj * nbk;
  if (!(M > 0 && M <= 65536 && N >= window && ni * M * M == np && 2 * M * M * M >= (long long)N * N * N &&
        blocks >= kBrickBlocks && blocks <= 0x7fffffffLL))
    return BrickGrid{0, 0, 0, 0, 0};
  return BrickGrid{(int)M, (int)ni, (int)nbj, (int)nbk, (unsigned)blocks};
}

// The side M of an array of M^3 particles, or 0.
static inline long long lattice_side(long long np) {
  const long long M = llround(cbrt((double)np));
  return M * M * M == np ? M : 0;
}

// Whether M^3 particles are indeed in the order of a lattice: of 256 bricks, how many
// have a particle from their middle within 12 cells of where the lattice puts it from
// the first.  By bricks particles in no order take longer than by singles (shuffled 256^3:
// the deposit 1398 against 1256 us, the gather, whose staging kernel keeps fewer warps,
// 2598 against 1645), so both kernels are launched and the one not meant returns at once.
// One block of 256 threads of a kernel that runs before them asks, beside its own work.
static __device__ __forceinline__ void brick_probe(const float* __restrict__ pos, int N, const BrickGrid& G,
                                                   int* __restrict__ by_bricks) {
  const unsigned b = (unsigned)((unsigned long long)threadIdx.x * G.blocks / 256);
  const int bk = b % G.nbk, bj = b / G.nbk % G.nbj, bi = b / G.nbk / G.nbj;
  const int i = bi * kBrickI, j = bj * kBrickJ, k = bk * kBrickK;
  const int di = min(kBrickI / 2, G.ni - 1 - i), dj = min(kBrickJ / 2, G.M - 1 - j), dk = min(kBrickK / 4, G.M - 1 - k);
  const float* x = pos + 3 * (((long long)i * G.M + j) * G.M + k);
  const float* y = x + 3 * (((long long)di * G.M + dj) * G.M + dk);
  const float h = (float)N / (float)G.M, fN = (float)N, iN = 1.f / fN;
  const int d[3] = {di, dj, dk};
  bool in = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float o = y[c] - x[c] - h * (float)d[c];
    in = in && fabsf(o - fN * rintf(o * iN)) < 12.f;
  }
  const int n = __syncthreads_count(in);
  if (threadIdx.x == 0) *by_bricks = n >= 128;
}

static __global__ void __launch_bounds__(256) k_brick_probe(const float* __restrict__ pos, int N, BrickGrid G,
                                                            int* __restrict__ by_bricks) {
  brick_probe(pos, N, G, by_bricks);
}

// The single-particle kernel is a programmatic dependent launch of the brick kernel,
// whose blocks call next_may_start as they begin: its own blocks, which need nothing of
// the brick kernel's, then come and go beside the last bricks.  Whether they are meant
// was written before the brick kernel began.  Block 0 stays for the brick kernel's end,
// so that what follows in the stream follows both.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ bool left_to_bricks(const int* by_bricks) {
  if (!by_bricks) return false;
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  return *by_bricks;
}

template <typename... P, typename... A>
static cudaError_t launch_beside_bricks(void (*kern)(P...), unsigned blocks, int threads, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// The gradients of a mesh scalar at lattice-ordered particles (cic_grad), brick by brick.
//
// k_gather is bound by L1: its 32 loads a particle hit about seven lines a warp
// (320 us at 256^3).  As in k_deposit_bricks a CTA takes a brick of 8 x 8 x 32 of the
// array and stages the window of the mesh about the brick's mean displacement in
// shared memory, whose banks serve the scattered lanes side by side.  The window's
// rows start at multiples of four cells, so that they arrive as 16-byte copies (four
// times fewer instructions) where N is one too.  A particle outside the window reads
// the mesh itself, after the others.  The sums are cic_grad's, in its order.
// More warps matter more than a wider window (the gather's 270 us at 256^3 without other launches): 16 x
// 16 x 48 cells 274 us, three CTAs an SM 302, 512 threads a CTA 310.
constexpr int kTileI = 15, kTileJ = 15, kTileK = 48;  // cells
constexpr int kTileCells = kTileI * kTileJ * kTileK;
constexpr int kTileThreads = kBrickJ * kBrickK;       // one plane of a brick at a time
constexpr int kTileOut = 512;

template <typename IT>
__device__ __noinline__ float3 gradient_direct(const float* T, int N, const float* x) {
  return cic_grad<IT>(T, N, x[0], x[1], x[2]);
}

// emit(3 q, gradient of particle q), once a particle.  QUADS: N % 4 == 0 and T on a 16-byte boundary.
template <typename IT, bool QUADS, class Emit>
__device__ __forceinline__ void brick_gradients(const float* __restrict__ T, int N, const float* pos,
                                                const BrickGrid& G, const Emit& emit) {
  extern __shared__ __align__(16) float tile[];
  __shared__ int s_sum[4], s_nout;
  __shared__ unsigned short s_out[kTileOut];  // particles outside the window
  const int t = threadIdx.x;
  const int M = G.M, ni = G.ni;
  const unsigned b = blockIdx.x, bij = b / (unsigned)G.nbk, bk = b - bij * G.nbk, bi = bij / (unsigned)G.nbj,
                 bj = bij - bi * G.nbj;
  const int i0 = bi * kBrickI, j0 = bj * kBrickJ + t / kBrickK, k0 = bk * kBrickK + t % kBrickK;
  const long long brick = ((long long)i0 * M + bj * kBrickJ) * M + bk * kBrickK;  // its first particle
  const long long mine = ((long long)i0 * M + j0) * M + k0;                       // this thread's first
  const long long plane = (long long)M * M;                                       // and the next ones' distance
  const int mp = j0 < M && k0 < M ? min(kBrickI, ni - i0) : 0;                    // this thread's particles
  if (t < 4) s_sum[t] = 0;
  if (t == 4) s_nout = 0;
  __syncthreads();
  // window origin: the mean place of a middle plane's particles, measured from the brick's first one, less half a window
  const float ref[3] = {wrap_pos(pos[3 * brick], N), wrap_pos(pos[3 * brick + 1], N), wrap_pos(pos[3 * brick + 2], N)};
  {
    const float fN = (float)N, iN = 1.f / (float)N;
    int sum[4] = {0, 0, 0, mp > 0};
    if (mp > 0) {
      const float* x = pos + 3 * (mine + (mp >> 1) * plane);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float o = x[d] - ref[d];
        sum[d] = (int)rintf(o - fN * rintf(o * iN));  // nearest image
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
    const int half = (d == 0 ? kTileI : (d == 1 ? kTileJ : kTileK)) / 2;
    org[d] = ((int)(ref[d] + __fdividef((float)s_sum[d], (float)s_sum[3])) - half) % N;
    org[d] += org[d] < 0 ? N : 0;
  }
  if (QUADS) {
    org[2] &= ~3;
#pragma unroll 4
    for (int a = t; a < kTileCells / 4; a += kTileThreads) {
      const int ij = a / (kTileK / 4), wi = ij / kTileJ;
      int i = org[0] + wi, j = org[1] + ij - wi * kTileJ, k = org[2] + 4 * (a - ij * (kTileK / 4));
      i -= i >= N ? N : 0;  // N >= the window's sides: one wrap
      j -= j >= N ? N : 0;
      k -= k >= N ? N : 0;
      __pipeline_memcpy_async(tile + 4 * a, T + ((IT)i * N + j) * N + k, 16);
    }
    __pipeline_commit();
    __pipeline_wait_prior(0);
  } else {
#pragma unroll 4
    for (int a = t; a < kTileCells; a += kTileThreads) {
      const int ij = a / kTileK, wi = ij / kTileJ;
      int i = org[0] + wi, j = org[1] + ij - wi * kTileJ, k = org[2] + a - ij * kTileK;
      i -= i >= N ? N : 0;
      j -= j >= N ? N : 0;
      k -= k >= N ? N : 0;
      tile[a] = T[((IT)i * N + j) * N + k];
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int r = 0; r < mp; ++r) {
    const long long p = 3 * (mine + r * plane);
    int c[3], c1;
    float w[3][2];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cic_axis_f(pos[p + d], N, c[d], c1, w[d][0], w[d][1]);
      c[d] -= org[d];
      c[d] += c[d] < 0 ? N : 0;
    }
    if (c[0] >= 1 && c[0] + 2 < kTileI && c[1] >= 1 && c[1] + 2 < kTileJ && c[2] >= 1 && c[2] + 2 < kTileK) {
      const float* at = tile + ((c[0] - 1) * kTileJ + c[1] - 1) * kTileK + c[2] - 1;
      const float3 g =
          cic_grad_core([&](int a, int bb, int cc) { return at[(a * kTileJ + bb) * kTileK + cc]; }, w[0], w[1], w[2]);
      emit(p, g);
    } else {
      const int q = atomicAdd(&s_nout, 1);
      if (q < kTileOut) s_out[q] = (unsigned short)(t + r * kTileThreads);
      else emit(p, gradient_direct<IT>(T, N, pos + p));
    }
  }
  __syncthreads();
  for (int q = t; q < min(s_nout, kTileOut); q += kTileThreads) {
    const int x = s_out[q];
    const int i = x / (kBrickJ * kBrickK), j = (x / kBrickK) % kBrickJ, k = x % kBrickK;
    const long long p = 3 * (brick + ((long long)i * M + j) * M + k);
    emit(p, gradient_direct<IT>(T, N, pos + p));
  }
}

}  // namespace mg
