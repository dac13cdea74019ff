// mg_common.cuh -- shared device helpers: indexing, deterministic block
// reductions, launch geometry.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "mg_model.cuh"

namespace mg {

constexpr int kThreads = 256;
constexpr int kMaxReduceBlocks = 8192;  // size of the partial-sum array
// Grid cap of the grid-stride elementwise kernels: about two waves of
// 256-thread blocks on 152 SMs, so that per-thread setup (a division, a
// scalar read) is paid once per ~30 cells, not once per cell.
constexpr int kStreamBlocks = 2432;

__host__ __device__ __forceinline__ size_t cidx(int n, int i, int j, int k) {
  return ((size_t)i * n + j) * n + k;
}

// Block-wide sum of one double per thread; result valid in thread 0.  Fixed
// shuffle/tree order, so the result is deterministic for a fixed launch shape.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  v = 0.0;
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    v = lane < nw ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

// a / *b, formed by one thread of the block: a FP64 division is some thirty
// instructions of the 1/64-rate pipe, which 2432 blocks of 256 threads would spend 20
// us on (the source norm of a 128^3 mesh: 28 us, 20 so).  Every thread calls this.
__device__ __forceinline__ double block_ratio(double a, const double* b) {
  __shared__ double r;
  if (threadIdx.x == 0) r = a / *b;
  __syncthreads();
  return r;
}

// Positivity-guard replacements (reading C11): each thread adds its own count to
// the solve's counter (a 64-bit integer in the workspace scalars); the guard is
// rare, so the atomic is almost never issued.  guard may be null (not counted).
__device__ __forceinline__ void count_guards(unsigned long long* guard, unsigned c) {
  if (c && guard) atomicAdd(guard, (unsigned long long)c);
}

// Grid for a grid-stride loop over 'work' items, capped so that partial sums fit.
inline int grid_for(long long work, int threads = kThreads, int cap = kMaxReduceBlocks) {
  long long g = (work + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

// Grid for a grid-stride elementwise kernel.
inline int stream_grid(long long work) { return grid_for(work, kThreads, kStreamBlocks); }

// Error-free accumulation of single-precision values (Knuth's two-sum): after
// any number of steps hi + lo equals the exact sum up to the rounding of lo,
// i.e. to ~2^-46 relative, without double-precision arithmetic.
struct FloatFloat {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x);
    const float bp = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
    lo = __fadd_rn(lo, err);
  }
};

// float -> double, exact; normal numbers and zeros by bits, without the conversion, which
// is an instruction of the 1/64-rate FP64 pipe.
__device__ __forceinline__ bool f2d_by_bits(float f) {
  const unsigned a = __float_as_uint(f) & 0x7fffffffu;
  return a - 0x00800000u < 0x7f000000u || a == 0u;
}
__device__ __forceinline__ double f2d_of_bits(float f) {
  const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
  return __hiloint2double((int)((b & 0x80000000u) | (a ? (a >> 3) + (896u << 20) : 0u)), (int)(b << 29));
}
// (a call for the other numbers: as an expression the compiler converts every value and selects)
static __device__ __noinline__ double f2d_call(float f) { return (double)f; }
__device__ __forceinline__ double f2d_exact(float f) {
  if (f2d_by_bits(f)) return f2d_of_bits(f);
  return f2d_call(f);
}

// The sum of a block of kThreads threads in thread 0, in FP64, whose range and 53 bits
// the sum needs: one warp adds the threads' values, two FP64 additions a value of its
// lanes' eight, instead of the five of every warp's shuffles (k_sum_f32 of a 128^3 mesh
// 9.2 us; 14.6 by shuffles in FP64).
__device__ __forceinline__ double block_sum(FloatFloat v) {
  constexpr int P = kThreads / 32;
  __shared__ float2 sh[kThreads];
  const int t = threadIdx.x;
  __syncthreads();
  sh[t] = make_float2(v.hi, v.lo);
  __syncthreads();
  double s = 0.0;
  if (t < 32) {
    float2 x[P];
    bool bits = true;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      x[i] = sh[t + 32 * i];
      bits = bits && f2d_by_bits(x[i].x) && f2d_by_bits(x[i].y);
    }
    double l = 0.0;
    if (bits) {
#pragma unroll
      for (int i = 0; i < P; ++i) s += f2d_of_bits(x[i].x), l += f2d_of_bits(x[i].y);
    } else {
#pragma unroll 1
      for (int i = 0; i < P; ++i) s += (double)sh[t + 32 * i].x, l += (double)sh[t + 32 * i].y;
    }
    s += l;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;
}

}  // namespace mg
