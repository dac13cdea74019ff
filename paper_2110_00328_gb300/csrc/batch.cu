// batch.cu -- many independent solves (uneven meshes, models, parameters) at once.
//
// All solves of a batch follow the mixed-precision scheme of solve_mixed.cu
// (FP64 outer residual and update, FP32 correction-form FAS V-cycles) in lock
// step.  Each phase of a V-cycle (one colour of smoothing on level l,
// restriction l -> l+1, coarse source on l+1, the one-block tails or coarsest-level
// relaxations, prolongation l+1 -> l) is one kernel launch covering the blocks of
// every solve of one model that takes part in it: a block finds its solve by binary search in a
// prefix table of per-solve block counts and then works exactly as the single-
// solve kernel does.  One V-cycle of the whole batch is captured once as a CUDA
// graph and replayed.  Solves that have converged are masked by a device flag
// (their blocks exit at once), so the graph never needs re-capturing.  The
// smoother's block width is chosen by timing the candidates on the batch's
// finest levels on first use (a small autotuner), and cached with the batch.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <mutex>
#include <vector>

#include "mg_common.cuh"
#include "mg_internal.h"
#include "mixed_common.cuh"
#include "sweep32.cuh"
#include "tail32.cuh"

namespace mg {

// One level of one solve.
struct BDesc {
  int n;      // level side
  int solve;  // index of the solve in the batch
  int split;  // this level (the finest) in the red-black split layout
  LevelF lf;  // constants of this level
  float *e, *ub, *S, *rho, *Re;      // this level
  float* q;                          // split f(R) n = 1, 2: the stored neighbour quantity, else nullptr
  float *eH, *ubH, *SH, *ReH;        // next coarser level (if any)
};

// Finest-level descriptor for the FP64 outer kernels.
struct BFine {
  int n, solve;
  ModelDev m;
  double* u;
  const double* src;   // CQ: FP64 source term
  const FFC* ffc;      // f(R), symmetron: float-float residual constants
  const float* rho;    // f(R), symmetron: the caller's density
  float *ub, *tau, *e;
  float* q;            // the finest level's stored neighbour quantity (zeroed with e), or nullptr
};

// Planes a CTA of the outer residual marches: short, so that a batch of small meshes
// fills the GPU (two prologue planes each).
constexpr int kBatchPlanes = 16;

// Level layouts of the batched kernels: the quad kernels take levels whose side
// is a multiple of 4 (>= 8); others fall back to one cell per thread.
__host__ __device__ __forceinline__ bool quad_level(int n) { return (n & 3) == 0 && n >= 8; }

__device__ __forceinline__ int find_slot(const int* __restrict__ prefix, int cnt, int b) {
  int lo = 0, hi = cnt - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// ---- batched phase kernels (bodies as in solve_mixed.cu) ----

// Block (32, ROWS).  Quad levels: ceil(n/128) x n x ceil(n/ROWS) blocks per
// solve (lanes along k, ROWS planes i per block); others: one cell of the
// colour per thread, flat.
template <int K, int ROWS>
__global__ void __launch_bounds__(32 * ROWS) kb_smooth(const BDesc* __restrict__ D, const int* __restrict__ prefix,
                                                       int cnt, const int* __restrict__ active, int parity) {
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BDesc& d = D[s];
  if (!active[d.solve]) return;
  const int n = d.n;
  const int b = blockIdx.x - prefix[s];
  if (d.split) {
    long long r;
    int seg;
    bool act;
    split_lane(n, n, (long long)b * ROWS + threadIdx.y, threadIdx.x, &r, &seg, &act);
    const int i = (int)r / n, j = (int)r - i * n;  // rows: n^2 < 2^31
    constexpr bool QS = K == KFR1 || K == KFR2;    // these levels store q
    if (n <= 1024)  // 32-bit cell offsets
      smooth_split<K, QS, 0, int>(d.lf, n, d.e, d.ub, d.rho, d.S, i, j, seg, act, parity, threadIdx.x, d.q);
    else
      smooth_split<K, QS>(d.lf, n, d.e, d.ub, d.rho, d.S, i, j, seg, act, parity, threadIdx.x, d.q);
    return;
  }
  if (quad_level(n)) {
    const int nbx = ((n >> 2) + 31) / 32;
    const int xb = b % nbx, r = b / nbx, nr = n / quad_rows(n), i = (r / nr) * ROWS + threadIdx.y;
    if (i >= n) return;  // whole warps
    const QuadLane<true> ql(n, r % nr, xb, threadIdx.x);
    if (n <= 1024)
      smooth_quad<K, false, int>(d.lf, n, d.e, d.ub, d.rho, d.S, i, ql.j, ql.tq, threadIdx.x, parity);
    else
      smooth_quad<K>(d.lf, n, d.e, d.ub, d.rho, d.S, i, ql.j, ql.tq, threadIdx.x, parity);
    return;
  }
  const long long t = (long long)b * (32 * ROWS) + threadIdx.y * 32 + threadIdx.x;
  const int h = n >> 1;
  if (t >= (long long)h * n * n) return;
  const int kk = (int)(t % h), j = (int)((t / h) % n), i = (int)(t / ((long long)h * n));
  const int k = 2 * kk + ((i + j + parity) & 1);
  const size_t c = cidx(n, i, j, k);
  const float Lnb = nb_sum_g<K>(d.e, d.ub, n, i, j, k);
  d.e[c] = update_e_fast<K>(d.lf, d.ub[c], d.e[c], d.rho ? d.rho[c] : 1.f, d.S[c], Lnb);
}

static int smooth_blocks(int n, int rows, bool split) {
  if (split) return (int)((split_warps(n, n) + rows - 1) / rows);
  if (quad_level(n)) return (((n >> 2) + 31) / 32) * (n / quad_rows(n)) * ((n + rows - 1) / rows);
  return (int)(((long long)(n >> 1) * n * n + 32 * rows - 1) / (32 * rows));
}

// Restriction of level l into l+1, d = M(e) - S at 8 children; block (32, 4).
// Quad levels: ceil(nf/128) x nc x ceil(nc/4) blocks per solve; others: one
// coarse cell per thread, flat.  ZR: after pre-smoothing the second colour's defect
// is zero (restrict_quad, restrict_split_zr).
template <int K, bool ZR>
__global__ void __launch_bounds__(128) kb_restrict(const BDesc* __restrict__ D, const int* __restrict__ prefix, int cnt,
                                                   const int* __restrict__ active) {
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BDesc& d = D[s];
  if (!active[d.solve]) return;
  const int nf = d.n, nc = nf >> 1;
  const int b = blockIdx.x - prefix[s];
  if (quad_level(nf)) {
    const int nbx = ((nf >> 2) + 31) / 32;
    const int xb = b % nbx, r = b / nbx, nr = nc / quad_rows(nf), I = (r / nr) * 4 + threadIdx.y;
    if (I >= nc) return;  // whole warps
    const QuadLane<> ql(nf, r % nr, xb, threadIdx.x);
    const int J = ql.j, tq = ql.tq, lane = threadIdx.x;
    constexpr bool QS = K == KFR1 || K == KFR2;  // split levels of these store q
    if (d.split) {
      if constexpr (QS && ZR) {
        if (nf <= 1024) restrict_split_zr<K, int>(d.lf, nf, d.e, d.ub, d.S, d.q, d.ReH, d.eH, d.ubH, d.SH, I, J, tq, lane);
        else restrict_split_zr<K>(d.lf, nf, d.e, d.ub, d.S, d.q, d.ReH, d.eH, d.ubH, d.SH, I, J, tq, lane);
      } else {
        restrict_quad<K, SplitLayout, QS, ZR>(d.lf, nf, d.e, d.ub, d.rho, d.S, d.ReH, d.eH, d.ubH, d.SH, I, J, tq, lane,
                                              d.q);
      }
    } else if (nf <= 1024) {
      restrict_quad<K, NatLayout32, false, ZR>(d.lf, nf, d.e, d.ub, d.rho, d.S, d.ReH, d.eH, d.ubH, d.SH, I, J, tq, lane);
    } else {
      restrict_quad<K, NatLayout, false, ZR>(d.lf, nf, d.e, d.ub, d.rho, d.S, d.ReH, d.eH, d.ubH, d.SH, I, J, tq, lane);
    }
    return;
  }
  const long long t = (long long)b * 128 + threadIdx.y * 32 + threadIdx.x;
  if (t >= (long long)nc * nc * nc) return;
  const int Kc = (int)(t % nc), J = (int)((t / nc) % nc), I = (int)(t / ((long long)nc * nc));
  float se = 0.f, su = 0.f, sd = 0.f;
  for (int di = 0; di < 2; ++di)
    for (int dj = 0; dj < 2; ++dj)
      for (int dk = 0; dk < 2; ++dk) {
        const int i = 2 * I + di, j = 2 * J + dj, k = 2 * Kc + dk;
        const size_t c = cidx(nf, i, j, k);
        const float ec = d.e[c], uc = d.ub[c];
        se += ec;
        su += uc;
        sd += local_M<K>(d.lf, uc, ec, d.rho ? d.rho[c] : 1.f, nb_sum_g<K>(d.e, d.ub, nf, i, j, k)) - d.S[c];
      }
  const size_t o = cidx(nc, I, J, Kc);
  d.ReH[o] = 0.125f * se;
  d.eH[o] = 0.125f * se;
  d.ubH[o] = 0.125f * su;
  d.SH[o] = 0.125f * sd;
}

static int restrict_blocks(int nf) {
  const int nc = nf >> 1;
  if (quad_level(nf)) return (((nf >> 2) + 31) / 32) * (nc / quad_rows(nf)) * ((nc + 3) / 4);
  return (int)(((long long)nc * nc * nc + 127) / 128);
}

// Coarse source on level l (descriptors of level l): S <- M(Re) - S; block (32, 4).
// Quad levels: ceil(n/128) x n x n/4 blocks per solve; others: one cell per thread, flat.
template <int K>
__global__ void __launch_bounds__(128) kb_fas(const BDesc* __restrict__ D, const int* __restrict__ prefix, int cnt,
                                              const int* __restrict__ active) {
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BDesc& d = D[s];
  if (!active[d.solve]) return;
  const int n = d.n;
  const int b = blockIdx.x - prefix[s];
  if (quad_level(n)) {
    const int nbx = ((n >> 2) + 31) / 32;
    const int xb = b % nbx, r = b / nbx, nr = n / quad_rows(n), i = (r / nr) * 4 + threadIdx.y;
    const QuadLane<> ql(n, r % nr, xb, threadIdx.x);
    if (n <= 1024) fas_quad<K, int>(d.lf, n, d.Re, d.ub, d.rho, d.S, i, ql.j, ql.tq, threadIdx.x);
    else fas_quad<K>(d.lf, n, d.Re, d.ub, d.rho, d.S, i, ql.j, ql.tq, threadIdx.x);
    return;
  }
  const long long t = (long long)b * 128 + threadIdx.y * 32 + threadIdx.x;
  if (t >= (long long)n * n * n) return;
  const int k = (int)(t % n), j = (int)((t / n) % n), i = (int)(t / ((long long)n * n));
  d.S[t] = local_M<K>(d.lf, d.ub[t], d.Re[t], d.rho ? d.rho[t] : 1.f, nb_sum_g<K>(d.Re, d.ub, n, i, j, k)) - d.S[t];
}

static int fas_blocks(int n) {
  if (quad_level(n)) return (((n >> 2) + 31) / 32) * (n / quad_rows(n)) * (n / 4);
  return (int)(((long long)n * n * n + 127) / 128);
}

// Prolongation-correction of level l from l+1; block (32, 4).  Quad levels:
// ceil(nf/128) x nf x ceil(nf/4) blocks per solve; others: one fine cell per
// thread, flat.
// SO (post-smoothing follows): a split finest level has its second colour corrected
// only (prolong_split2x2_second; CQ's batched levels are not split), for which
// the blocks are those of the restriction.
template <int K, bool SO>
__global__ void __launch_bounds__(128) kb_prolong(const BDesc* __restrict__ D, const int* __restrict__ prefix, int cnt,
                                                  const int* __restrict__ active, unsigned long long* guards) {
  constexpr bool FR = is_fr(K);
  constexpr int QK = K == KFR1 || K == KFR2 ? K : -1;  // split levels of these store q
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BDesc& d = D[s];
  if (!active[d.solve]) return;
  unsigned long long* guard = guards + d.solve;
  const int nf = d.n, nc = nf >> 1;
  const int b = blockIdx.x - prefix[s];
  if (quad_level(nf)) {
    const int nbx = ((nf >> 2) + 31) / 32, xb = b % nbx, r = b / nbx, lane = threadIdx.x, per = quad_rows(nf);
    if constexpr (SO && K != KFR0) {
      if (d.split) {
        const int nr = nc / per, I = (r / nr) * 4 + threadIdx.y;
        if (I >= nc) return;  // whole warps
        const QuadLane<> ql(nf, r % nr, xb, lane);
        const int J = ql.j, tq = ql.tq;
        if (nf <= 1024)
          prolong_split2x2_second<QK, false, int>(nc, d.eH, d.ReH, d.ub, d.e, I, J, tq, lane, guard, d.q);
        else
          prolong_split2x2_second<QK>(nc, d.eH, d.ReH, d.ub, d.e, I, J, tq, lane, guard, d.q);
        return;
      }
    }
    const int nr = nf / per, i = (r / nr) * 4 + threadIdx.y;
    if (i >= nf) return;  // whole warps
    const QuadLane<> ql(nf, r % nr, xb, lane);
    const int j = ql.j, tq = ql.tq;
    if (d.split) prolong_quad<FR, SplitLayout, QK>(nc, d.eH, d.ReH, d.ub, d.e, i, j, tq, lane, guard, d.q);
    else if (nf <= 1024) prolong_quad<FR, NatLayout32>(nc, d.eH, d.ReH, d.ub, d.e, i, j, tq, lane, guard);
    else prolong_quad<FR>(nc, d.eH, d.ReH, d.ub, d.e, i, j, tq, lane, guard);
    return;
  }
  const long long t = (long long)b * 128 + threadIdx.y * 32 + threadIdx.x;
  if (t >= (long long)nf * nf * nf) return;
  const int k = (int)(t % nf), j = (int)((t / nf) % nf), i = (int)(t / ((long long)nf * nf));
  const int I = i >> 1, J = j >> 1, Kc = k >> 1;
  const int I2 = wrapi(I + ((i & 1) ? 1 : -1), nc);
  const int J2 = wrapi(J + ((j & 1) ? 1 : -1), nc);
  const int K2 = wrapi(Kc + ((k & 1) ? 1 : -1), nc);
#define EH(a, b, c) (d.eH[cidx(nc, a, b, c)] - d.ReH[cidx(nc, a, b, c)])
  const float corr = (27.f * EH(I, J, Kc) + 9.f * (EH(I2, J, Kc) + EH(I, J2, Kc) + EH(I, J, K2)) +
                      3.f * (EH(I2, J2, Kc) + EH(I2, J, K2) + EH(I, J2, K2)) + EH(I2, J2, K2)) *
                     (1.f / 64.f);
#undef EH
  const size_t o = cidx(nf, i, j, k);
  const float old = d.e[o];
  float v = old + corr;
  if (FR && !(d.ub[o] + v > 0.f)) {
    v = 0.5f * (old - d.ub[o]);
    count_guards(guard, 1u);
  }
  d.e[o] = v;
}

// second: the split level's second-colour form.
static int prolong_blocks(int nf, bool second) {
  if (second) return restrict_blocks(nf);
  if (quad_level(nf)) return (((nf >> 2) + 31) / 32) * (nf / quad_rows(nf)) * ((nf + 3) / 4);
  return (int)(((long long)nf * nf * nf + 127) / 128);
}

// Coarsest levels: one CTA per solve.
template <int K>
__global__ void __launch_bounds__(512) kb_coarse(const BDesc* __restrict__ D, const int* __restrict__ active,
                                                 int sweeps) {
  const BDesc& d = D[blockIdx.x];
  if (!active[d.solve]) return;
  const int n = d.n, n3 = n * n * n;
  for (int s = 0; s < sweeps; ++s)
    for (int parity = 0; parity < 2; ++parity) {
      for (int t = threadIdx.x; t < n3; t += blockDim.x) {
        const int k = t % n, j = (t / n) % n, i = t / (n * n);
        if (((i + j + k) & 1) != parity) continue;
        const float Lnb = nb_sum_g<K>(d.e, d.ub, n, i, j, k);
        d.e[t] = update_e_fast<K>(d.lf, d.ub[t], d.e[t], d.rho ? d.rho[t] : 1.f, d.S[t], Lnb);
      }
      __syncthreads();
    }
}

// The coarsest levels of every solve, one CTA each (tail32.cuh).
template <int K>
__global__ void __launch_bounds__(kTailThreads) kb_tail(const TailArgs* __restrict__ args,
                                                        const int* __restrict__ solve,
                                                        const int* __restrict__ active) {
  if (!active[solve[blockIdx.x]]) return;
  extern __shared__ float tail_sm[];
  __shared__ TailArgs A;
  static_assert(sizeof(TailArgs) % 4 == 0, "copied by words");
  for (int i = threadIdx.x; i < (int)(sizeof(TailArgs) / 4); i += kTailThreads)
    reinterpret_cast<int*>(&A)[i] = reinterpret_cast<const int*>(args + blockIdx.x)[i];
  __syncthreads();
  tail_cycle<K, 2>(A, tail_sm);
}

// FP64 fine residual of every active solve (tiles of 8 x 32, chunks of kBatchPlanes planes).
template <int K>
__global__ void __launch_bounds__(256) kb_outer_residual(const BFine* __restrict__ F, const int* __restrict__ prefix,
                                                         int cnt, const int* __restrict__ active,
                                                         double* __restrict__ partials) {
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BFine& f = F[s];
  const int b = blockIdx.x - prefix[s];
  double a = 0.0;
  if (active[f.solve]) {
    const int tiles = (f.n / 32) * (f.n / 8);
    if constexpr (K == KCQ) {
      a = cq_residual_tile<false, 8, 32, false>(f.m, CqSeries{}, 0.0, f.n, kBatchPlanes, f.u, f.src, nullptr, f.ub, f.tau,
                                                b % tiles, b / tiles);
    } else {
      const FFC c = *f.ffc;
      a = outer_residual_tile_ff<K, 8, 32, true>(c, f.n, kBatchPlanes, f.u, f.rho, f.ub, f.tau, b % tiles, b / tiles);
    }
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = a;
}

// Per-solve sums of the partials: out[solve] = sum over its blocks.
__global__ void kb_finalize(const BFine* __restrict__ F, const int* __restrict__ prefix, int cnt,
                            const double* __restrict__ partials, double* __restrict__ out) {
  const int s = blockIdx.x;
  double a = 0.0;
  for (int i = prefix[s] + threadIdx.x; i < prefix[s + 1]; i += blockDim.x) a += partials[i];
  a = block_sum(a);
  if (threadIdx.x == 0) out[F[s].solve] = a;
}

// u64 += e, e <- 0 and the stored q <- 0 for every active solve; a thread takes the
// cells k = 4w .. 4w + 3 of a row (sides are multiples of 32), which sit at 2w, 2w + 1
// of the two colours of a split level.
__global__ void __launch_bounds__(256) kb_apply(const BFine* __restrict__ F, const int* __restrict__ prefix, int cnt,
                                                const int* __restrict__ active) {
  const int s = find_slot(prefix, cnt, blockIdx.x);
  const BFine& f = F[s];
  if (!active[f.solve]) return;
  const int n = f.n, w4 = n >> 2, h = n >> 1;
  const long long t = (long long)(blockIdx.x - prefix[s]) * 256 + threadIdx.x;  // < 2^31: n <= 2048
  if (t >= (long long)n * n * w4) return;
  const int row = (int)((unsigned)t / (unsigned)w4), w = (int)t - row * w4;
  const int i = row / n, j = row - i * n;
  double* u = f.u + (long long)row * n + 4 * w;
  float4 e;
  if (f.m.kind == KCQ) {
    float4* p = reinterpret_cast<float4*>(f.e + (long long)row * n + 4 * w);
    e = *p;
    *p = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    const long long H = (long long)n * n * h, o = (long long)row * h + 2 * w;
    const long long a = (i + j) & 1 ? H + o : o, b = (i + j) & 1 ? o : H + o;
    const float2 x = *reinterpret_cast<const float2*>(f.e + a), y = *reinterpret_cast<const float2*>(f.e + b);
    e = make_float4(x.x, y.x, x.y, y.y);
    const float2 z = make_float2(0.f, 0.f);
    *reinterpret_cast<float2*>(f.e + a) = z;
    *reinterpret_cast<float2*>(f.e + b) = z;
    if (f.q) {  // Delta w(u, 0)
      *reinterpret_cast<float2*>(f.q + a) = z;
      *reinterpret_cast<float2*>(f.q + b) = z;
    }
  }
  if ((uintptr_t)f.u % 16 == 0) {
    double2* p = reinterpret_cast<double2*>(u);
    const double2 a = p[0], b = p[1];
    p[0] = make_double2(a.x + (double)e.x, a.y + (double)e.y);
    p[1] = make_double2(b.x + (double)e.z, b.y + (double)e.w);
  } else {
    u[0] += (double)e.x;
    u[1] += (double)e.y;
    u[2] += (double)e.z;
    u[3] += (double)e.w;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

struct Phase {                    // one batched launch of one kind
  int cnt = 0, blocks = 0;
  size_t d_off = 0, p_off = 0;    // descriptor table and block prefix (cnt + 1) in the batch's tables
};

constexpr int kBatchKinds = 5;  // model kinds

struct Batch {
  int device = -1;
  std::vector<int> Ns, levels_req;   // signature
  int count = 0;
  void* base = nullptr;
  size_t bytes = 0;
  // per solve
  struct S {
    int N, nlev, kind;
    double* src64;
    float *e[kMaxLevels], *ub[kMaxLevels], *S32[kMaxLevels], *Re[kMaxLevels], *rho32[kMaxLevels];
    float* q0;  // the finest level's stored neighbour quantity (used for f(R) n = 1, 2)
  };
  std::vector<S> sv;
  double* partials = nullptr;  // outer-residual partials
  double* sums = nullptr;      // per solve: sum r^2
  double* ssum = nullptr;      // per solve: source sum of squares
  double* rmean = nullptr;     // per solve: density sum
  int* active = nullptr;       // per solve flag (device)
  unsigned long long* guards = nullptr;    // per solve: positivity-guard replacements (device)
  unsigned long long* h_guards = nullptr;  // pinned host mirror
  int* h_active = nullptr;     // pinned host mirror
  double* h_sums = nullptr;    // pinned host mirror of sums (count) and ssum (count)
  char* tables = nullptr;      // descriptor tables and prefixes
  size_t tables_bytes = 0;     // their capacity
  cudaGraphExec_t vexec = nullptr;
  cudaStream_t cap[kBatchKinds] = {};  // capture streams, one per kind of the batch
  cudaEvent_t ev[kBatchKinds] = {};
  unsigned long long vsig = 0;
  long long vlaunches = 0;
  int rows = 0;                // autotuned smoother block height (planes per block)
  FFC* ffc = nullptr;          // per solve: float-float residual constants
};

static std::mutex g_bmu;
static std::vector<Batch*> g_batches;

static void free_batch(Batch* b) {
  if (b->vexec) cudaGraphExecDestroy(b->vexec);
  for (int k = 0; k < kBatchKinds; ++k) {
    if (b->cap[k]) cudaStreamDestroy(b->cap[k]);
    if (b->ev[k]) cudaEventDestroy(b->ev[k]);
  }
  if (b->tables) cudaFree(b->tables);
  if (b->base) cudaFree(b->base);
  if (b->h_active) cudaFreeHost(b->h_active);
  if (b->h_sums) cudaFreeHost(b->h_sums);
  if (b->h_guards) cudaFreeHost(b->h_guards);
  delete b;
}

void release_batches() {
  std::lock_guard<std::mutex> lk(g_bmu);
  int dev = 0;
  cudaGetDevice(&dev);
  std::vector<Batch*> keep;
  for (Batch* b : g_batches) {
    if (b->device == dev) free_batch(b);
    else keep.push_back(b);
  }
  g_batches = keep;
}

static int get_batch(int count, const int* N, const mgglam_params* prm, Batch** out) {
  int dev = 0;
  MG_CUDA_TRY(cudaGetDevice(&dev));
  std::vector<int> ns(N, N + count), lv(count);
  for (int s = 0; s < count; ++s) lv[s] = prm[s].levels;
  std::lock_guard<std::mutex> lk(g_bmu);
  for (Batch* b : g_batches)
    if (b->device == dev && b->Ns == ns && b->levels_req == lv) {
      *out = b;
      return MGGLAM_OK;
    }
  Batch* b = new Batch();
  b->device = dev;
  b->Ns = ns;
  b->levels_req = lv;
  b->count = count;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  struct O { size_t src, q0, e[kMaxLevels], ub[kMaxLevels], S[kMaxLevels], Re[kMaxLevels], rho[kMaxLevels]; };
  std::vector<O> o(count);
  size_t total_blocks = 0;
  b->sv.resize(count);
  for (int s = 0; s < count; ++s) {
    Batch::S& v = b->sv[s];
    v.N = N[s];
    v.nlev = count_levels(N[s], prm[s].levels);
    o[s].src = take((size_t)N[s] * N[s] * N[s] * 8);
    o[s].q0 = take((size_t)N[s] * N[s] * N[s] * 4);  // the plan is cached per mesh set, the models may change
    for (int l = 0, n = N[s]; l < v.nlev; ++l, n /= 2) {
      const size_t c = (size_t)n * n * n * 4;
      o[s].e[l] = take(c);
      o[s].ub[l] = take(c);
      o[s].S[l] = take(c);
      o[s].Re[l] = take(c);
      o[s].rho[l] = take(c);
    }
    total_blocks += (size_t)(N[s] / 32) * (N[s] / 8) * ((N[s] + kBatchPlanes - 1) / kBatchPlanes);
  }
  const size_t o_part = take(std::max<size_t>(total_blocks, kMaxReduceBlocks) * 8);
  const size_t o_sums = take(count * 8), o_ssum = take(count * 8), o_rmean = take(count * 8), o_act = take(count * 4);
  const size_t o_ffc = take(count * sizeof(FFC));
  const size_t o_guard = take(count * sizeof(unsigned long long));
  if (cudaMalloc(&b->base, off) != cudaSuccess) {
    cudaGetLastError();
    delete b;
    return MGGLAM_ERR_OOM;
  }
  if (cudaMallocHost((void**)&b->h_active, count * 4) != cudaSuccess ||
      cudaMallocHost((void**)&b->h_sums, count * 16) != cudaSuccess ||
      cudaMallocHost((void**)&b->h_guards, count * sizeof(unsigned long long)) != cudaSuccess) {
    cudaGetLastError();
    free_batch(b);
    return MGGLAM_ERR_OOM;
  }
  b->bytes = off;
  char* base = (char*)b->base;
  for (int s = 0; s < count; ++s) {
    Batch::S& v = b->sv[s];
    v.src64 = (double*)(base + o[s].src);
    v.q0 = (float*)(base + o[s].q0);
    for (int l = 0; l < v.nlev; ++l) {
      v.e[l] = (float*)(base + o[s].e[l]);
      v.ub[l] = (float*)(base + o[s].ub[l]);
      v.S32[l] = (float*)(base + o[s].S[l]);
      v.Re[l] = (float*)(base + o[s].Re[l]);
      v.rho32[l] = (float*)(base + o[s].rho[l]);
    }
  }
  b->partials = (double*)(base + o_part);
  b->sums = (double*)(base + o_sums);
  b->ssum = (double*)(base + o_ssum);
  b->rmean = (double*)(base + o_rmean);
  b->active = (int*)(base + o_act);
  b->ffc = (FFC*)(base + o_ffc);
  b->guards = (unsigned long long*)(base + o_guard);
  g_batches.push_back(b);
  *out = b;
  return MGGLAM_OK;
}

// Kernel-group dispatch for batched launches.
#define MG_BDISPATCH(kind, CALL)                                        \
  switch (kind) {                                                       \
    case KFR0: { constexpr int KK = KFR0; CALL; } break;                \
    case KFR1: { constexpr int KK = KFR1; CALL; } break;                \
    case KFR2: { constexpr int KK = KFR2; CALL; } break;                \
    case KSYM: { constexpr int KK = KSYM; CALL; } break;                \
    default: { constexpr int KK = KCQ; CALL; } break;                   \
  }

// The launches of one kind's solves: per level l the phases of the solves that go
// below l (smoothing, restriction, prolongation, and the source on l + 1, which a
// tail forms itself), the solves whose V-cycle ends on l with a coarsest
// relaxation, and those whose rest runs as a tail.
struct KindPlan {
  int kind = 0;
  struct L {
    Phase smooth, restrict_, fas, prolong, coarse;
  };
  std::vector<L> lv;
  int tails = 0;
  size_t tail_off = 0, tail_solve_off = 0, tail_smem = 0;
  Phase outer, apply;
  size_t fine_off = 0;
};

struct Plan {
  std::vector<KindPlan> kinds;
};

// First level of solve s's one-block tail (tail32.cuh), or -1.
static int batch_tail(const Batch::S& v) {
  int n[kMaxLevels];
  for (int l = 0; l < v.nlev; ++l) n[l] = v.N >> l;
  for (int l = 1; l < v.nlev; ++l)
    if (tail_fits(n, v.nlev, l)) return l;
  return -1;
}

// Build all descriptor tables and bring them to the device (one copy, into memory
// the batch keeps).
static int build_plan(Batch* B, const std::vector<ModelDev>& models, const std::vector<std::vector<LevelF>>& lfs,
                      const std::vector<const float*>& rho_in, double* const* field, const mgglam_params* prm,
                      int rows, Plan* P, cudaStream_t st) {
  const int count = B->count;
  std::vector<char> host;
  auto put = [&](const void* data, size_t bytes) {
    const size_t off = (host.size() + 255) & ~(size_t)255;
    host.resize(off + bytes);
    memcpy(host.data() + off, data, bytes);
    return off;
  };
  auto phase = [&](size_t d_off, const std::vector<int>& blocks) {
    Phase ph;
    ph.cnt = (int)blocks.size();
    ph.d_off = d_off;
    std::vector<int> pf(blocks.size() + 1);
    for (size_t i = 0; i < blocks.size(); ++i) pf[i + 1] = pf[i] + blocks[i];
    ph.blocks = pf.back();
    ph.p_off = put(pf.data(), pf.size() * sizeof(int));
    return ph;
  };
  auto rho_needed = [&](int s) {
    return models[s].kind == KSYM || (models[s].kind == KCQ && models[s].keep_exp);
  };
  auto desc = [&](int s, int l) {
    const Batch::S& v = B->sv[s];
    BDesc d;
    memset(&d, 0, sizeof(d));
    d.n = v.N >> l;
    d.solve = s;
    d.split = (l == 0 && models[s].kind != KCQ) ? 1 : 0;  // split finest level (float-float residual)
    d.q = (l == 0 && (models[s].kind == KFR1 || models[s].kind == KFR2)) ? v.q0 : nullptr;
    d.lf = lfs[s][l];
    d.e = v.e[l];
    d.ub = v.ub[l];
    d.S = v.S32[l];
    d.rho = rho_needed(s) ? v.rho32[l] : nullptr;
    d.Re = v.Re[l];
    if (l + 1 < v.nlev) {
      d.eH = v.e[l + 1];
      d.ubH = v.ub[l + 1];
      d.SH = v.S32[l + 1];
      d.ReH = v.Re[l + 1];
    }
    return d;
  };
  std::vector<int> kinds;
  for (auto& m : models)
    if (std::find(kinds.begin(), kinds.end(), m.kind) == kinds.end()) kinds.push_back(m.kind);
  P->kinds.assign(kinds.size(), {});
  for (size_t g = 0; g < kinds.size(); ++g) {
    KindPlan& G = P->kinds[g];
    G.kind = kinds[g];
    std::vector<int> own, tail(count), last(count);
    int Lmax = 0;
    for (int s = 0; s < count; ++s) {
      if (models[s].kind != G.kind) continue;
      own.push_back(s);
      tail[s] = batch_tail(B->sv[s]);
      last[s] = tail[s] > 0 ? tail[s] : B->sv[s].nlev - 1;  // the level whose V-cycle is one launch
      Lmax = std::max(Lmax, last[s] + 1);
    }
    G.lv.assign(Lmax, {});
    for (int l = 0; l < Lmax; ++l) {
      std::vector<BDesc> go, src, end;
      std::vector<int> bsm, bre, bfa, bpr;
      for (int s : own) {
        const int n = B->sv[s].N >> l;
        const bool split = l == 0 && G.kind != KCQ;
        if (l < last[s]) {
          go.push_back(desc(s, l));
          bsm.push_back(smooth_blocks(n, rows, split));
          bre.push_back(restrict_blocks(n));
          bpr.push_back(prolong_blocks(n, split && G.kind != KFR0 && prm[0].nu2 >= 1));
          if (l + 1 != tail[s]) {
            src.push_back(desc(s, l + 1));
            bfa.push_back(fas_blocks(n / 2));
          }
        } else if (l == last[s] && tail[s] < 0) {
          end.push_back(desc(s, l));
        }
      }
      KindPlan::L& L = G.lv[l];
      if (!go.empty()) {
        const size_t d = put(go.data(), go.size() * sizeof(BDesc));
        L.smooth = phase(d, bsm);
        L.restrict_ = phase(d, bre);
        L.prolong = phase(d, bpr);
      }
      if (!src.empty()) L.fas = phase(put(src.data(), src.size() * sizeof(BDesc)), bfa);
      if (!end.empty()) L.coarse = phase(put(end.data(), end.size() * sizeof(BDesc)), std::vector<int>(end.size(), 1));
    }
    std::vector<TailArgs> ta;
    std::vector<int> ts;
    std::vector<BFine> fine;
    std::vector<int> bo, ba;
    for (int s : own) {
      const Batch::S& v = B->sv[s];
      if (tail[s] > 0) {
        TailArgs A;
        memset(&A, 0, sizeof(A));
        const int t = tail[s];
        A.T = v.nlev - t;
        for (int m = 0; m < A.T; ++m) {
          A.n[m] = v.N >> (t + m);
          A.lf[m] = lfs[s][t + m];
          A.rho[m] = rho_needed(s) ? v.rho32[t + m] : nullptr;
          A.zr[m] = G.kind != KCQ || cq_linear(lfs[s][t + m]);
        }
        A.e = v.e[t];
        A.ub = v.ub[t];
        A.S = v.S32[t];
        A.nu1 = prm[0].nu1;
        A.nu2 = prm[0].nu2;
        A.coarse_sweeps = prm[0].coarse_sweeps;
        A.guard = B->guards + s;
        G.tail_smem = std::max(G.tail_smem, tail_layout(A));
        ta.push_back(A);
        ts.push_back(s);
      }
      BFine f;
      memset(&f, 0, sizeof(f));
      f.n = v.N;
      f.solve = s;
      f.m = models[s];
      f.u = field[s];
      f.src = v.src64;
      f.ffc = B->ffc + s;
      f.rho = rho_in[s];
      f.ub = v.ub[0];
      f.tau = v.S32[0];
      f.e = v.e[0];
      f.q = (G.kind == KFR1 || G.kind == KFR2) ? v.q0 : nullptr;
      fine.push_back(f);
      bo.push_back((v.N / 32) * (v.N / 8) * ((v.N + kBatchPlanes - 1) / kBatchPlanes));
      ba.push_back((int)(((size_t)v.N * v.N * (v.N / 4) + 255) / 256));
    }
    G.tails = (int)ta.size();
    if (G.tails) {
      G.tail_off = put(ta.data(), ta.size() * sizeof(TailArgs));
      G.tail_solve_off = put(ts.data(), ts.size() * sizeof(int));
    }
    G.fine_off = put(fine.data(), fine.size() * sizeof(BFine));
    G.outer = phase(G.fine_off, bo);
    G.apply = phase(G.fine_off, ba);
  }
  if (B->tables_bytes < host.size()) {
    if (B->tables) cudaFree(B->tables);
    B->tables = nullptr;
    B->tables_bytes = 0;
    const size_t cap = host.size() + host.size() / 2;  // other models of the same meshes fit too
    if (cudaMalloc((void**)&B->tables, cap) != cudaSuccess) {
      cudaGetLastError();
      return MGGLAM_ERR_OOM;
    }
    B->tables_bytes = cap;
  }
  MG_CUDA_TRY(cudaMemcpyAsync(B->tables, host.data(), host.size(), cudaMemcpyHostToDevice, st));
  MG_CUDA_TRY(cudaStreamSynchronize(st));
  return MGGLAM_OK;
}

static const BDesc* descs(const Batch* B, const Phase& ph) { return (const BDesc*)(B->tables + ph.d_off); }
static const int* prefix_of(const Batch* B, const Phase& ph) { return (const int*)(B->tables + ph.p_off); }

static void launch_smooth_phase(const Batch* B, int kind, const Phase& ph, int rows, int parity, cudaStream_t st) {
  if (ph.blocks == 0) return;
  const BDesc* d = descs(B, ph);
  const int* pf = prefix_of(B, ph);
  switch (rows) {
    case 2: MG_BDISPATCH(kind, (kb_smooth<KK, 2><<<ph.blocks, dim3(32, 2), 0, st>>>(d, pf, ph.cnt, B->active, parity))); break;
    case 8: MG_BDISPATCH(kind, (kb_smooth<KK, 8><<<ph.blocks, dim3(32, 8), 0, st>>>(d, pf, ph.cnt, B->active, parity))); break;
    default: MG_BDISPATCH(kind, (kb_smooth<KK, 4><<<ph.blocks, dim3(32, 4), 0, st>>>(d, pf, ph.cnt, B->active, parity))); break;
  }
  note_launch(1);
}

template <int K>
static void launch_batch_restrict(const Batch* B, const Phase& p, bool relaxed, cudaStream_t st) {
  // CQ's one Newton step leaves a defect in general
  if (K != KCQ && relaxed)
    kb_restrict<K, K != KCQ><<<p.blocks, dim3(32, 4), 0, st>>>(descs(B, p), prefix_of(B, p), p.cnt, B->active);
  else
    kb_restrict<K, false><<<p.blocks, dim3(32, 4), 0, st>>>(descs(B, p), prefix_of(B, p), p.cnt, B->active);
}

template <int K>
static void launch_batch_tail(const Batch* B, const KindPlan& G, cudaStream_t st) {
  kb_tail<K><<<G.tails, kTailThreads, G.tail_smem, st>>>((const TailArgs*)(B->tables + G.tail_off),
                                                         (const int*)(B->tables + G.tail_solve_off), B->active);
}

template <int K>
static int allow_batch_tail() {
  MG_CUDA_TRY(cudaFuncSetAttribute(kb_tail<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024));
  return MGGLAM_OK;
}

// One V-cycle of every active solve of one kind.
static void batch_vcycle(const Batch* B, const KindPlan& G, const mgglam_params& prm, cudaStream_t st) {
  const int Lmax = (int)G.lv.size();
  const dim3 b4(32, 4);
  for (int l = 0; l < Lmax; ++l) {
    const KindPlan::L& L = G.lv[l];
    for (int s = 0; s < 2 * prm.nu1; ++s) launch_smooth_phase(B, G.kind, L.smooth, B->rows, s & 1, st);
    if (L.restrict_.blocks) {
      MG_BDISPATCH(G.kind, (launch_batch_restrict<KK>(B, L.restrict_, prm.nu1 > 0, st)));
      note_launch(1);
    }
    const Phase& f = L.fas;
    if (f.blocks) {
      MG_BDISPATCH(G.kind, (kb_fas<KK><<<f.blocks, b4, 0, st>>>(descs(B, f), prefix_of(B, f), f.cnt, B->active)));
      note_launch(1);
    }
    if (L.coarse.cnt) {
      MG_BDISPATCH(G.kind, (kb_coarse<KK><<<L.coarse.cnt, 512, 0, st>>>(descs(B, L.coarse), B->active, prm.coarse_sweeps)));
      note_launch(1);
    }
  }
  if (G.tails) {
    MG_BDISPATCH(G.kind, (launch_batch_tail<KK>(B, G, st)));
    note_launch(1);
  }
  for (int l = Lmax - 1; l >= 0; --l) {
    const KindPlan::L& L = G.lv[l];
    const Phase& p = L.prolong;
    if (!p.blocks) continue;
    if (prm.nu2 >= 1) {
      MG_BDISPATCH(G.kind, (kb_prolong<KK, true><<<p.blocks, b4, 0, st>>>(descs(B, p), prefix_of(B, p), p.cnt, B->active,
                                                                          B->guards)));
    } else {
      MG_BDISPATCH(G.kind, (kb_prolong<KK, false><<<p.blocks, b4, 0, st>>>(descs(B, p), prefix_of(B, p), p.cnt, B->active,
                                                                           B->guards)));
    }
    note_launch(1);
    for (int s = 0; s < 2 * prm.nu2; ++s) launch_smooth_phase(B, G.kind, L.smooth, B->rows, s & 1, st);
  }
}

int solve_batch(int count, const mgglam_params* prm, const double* a, const float* const* rho, const int* N,
                double* const* field, double tol, mgglam_stats* stats, cudaStream_t st) {
  auto t0 = std::chrono::steady_clock::now();
  // models and constants
  std::vector<ModelDev> models(count);
  std::vector<std::vector<LevelF>> lfs(count);
  int rc;
  for (int s = 0; s < count; ++s) {
    if ((rc = make_model(&prm[s], a[s], N[s], &models[s]))) return rc;
    const int nl = count_levels(N[s], prm[s].levels);
    for (int l = 0; l < nl; ++l) lfs[s].push_back(make_levelf(models[s], (double)(1 << l)));
  }
  Batch* B = nullptr;
  if ((rc = get_batch(count, N, prm, &B))) return rc;
  // per-solve setup (density mean, FP64 source, density pyramid, background, source norm)
  for (int s = 0; s < count; ++s) {
    const Batch::S& v = B->sv[s];
    const long long n3 = (long long)v.N * v.N * v.N;
    if ((rc = launch_density_mean(rho[s], (size_t)n3, B->partials, B->rmean + s, st))) return rc;
    if (models[s].kind == KCQ) {
      k_src64<<<stream_grid(n3), kThreads, 0, st>>>(rho[s], n3, B->rmean + s, v.src64);
    } else {
      k_ff_consts<<<1, 32, 0, st>>>(models[s], n3, B->rmean + s, B->ffc + s);
    }
    const bool split = models[s].kind != KCQ;
    // the density pyramid, where the operator takes it
    const bool rho_needed = models[s].kind == KSYM || (models[s].kind == KCQ && models[s].keep_exp);
    if (!rho_needed) {
    } else if (split) {
      k_density_norm32_split<<<stream_grid(n3), kThreads, 0, st>>>(rho[s], v.N, B->rmean + s, v.rho32[0]);
    } else {
      k_density_norm32<<<stream_grid(n3), kThreads, 0, st>>>(rho[s], n3, B->rmean + s, v.rho32[0]);
    }
    for (int l = 1; l < v.nlev && rho_needed; ++l) {
      const int nc = v.N >> l;
      if (l == 1 && split)
        k_restrict32_from_split<<<dim3((nc + 63) / 64, nc, nc), 64, 0, st>>>(v.N, v.rho32[0], v.rho32[1]);
      else
        k_restrict32<<<dim3((nc + 63) / 64, nc, nc), 64, 0, st>>>(v.N >> (l - 1), v.rho32[l - 1], v.rho32[l]);
    }
    if ((rc = launch_init_background(models[s], field[s], (size_t)n3, st))) return rc;
    MG_BDISPATCH(models[s].kind, (k_src_sumsq32<KK><<<stream_grid(n3), kThreads, 0, st>>>(
                                     models[s], rho[s], n3, B->rmean + s, B->partials)));
    k_finalize_sum32<<<1, 1024, 0, st>>>(B->partials, stream_grid(n3), B->ssum + s);
    MG_CUDA_TRY(cudaMemsetAsync(v.e[0], 0, (size_t)n3 * 4, st));
    MG_CUDA_TRY(cudaMemsetAsync(v.q0, 0, (size_t)n3 * 4, st));  // Delta w(u, 0) = 0
    note_launch(4 + (rho_needed ? v.nlev : 0));
  }
  Plan P;
  const std::vector<const float*> rho_in(rho, rho + count);
  if ((rc = build_plan(B, models, lfs, rho_in, field, prm, B->rows ? B->rows : 4, &P, st))) return rc;
  auto fine_of = [&](const KindPlan& G) { return (const BFine*)(B->tables + G.fine_off); };
  auto outer_residual = [&]() -> int {
    int base = 0;  // partial slots: each kind's blocks after the previous ones'
    for (const KindPlan& G : P.kinds) {
      const Phase& o = G.outer;
      MG_BDISPATCH(G.kind, (kb_outer_residual<KK><<<o.blocks, 256, 0, st>>>(fine_of(G), prefix_of(B, o), o.cnt,
                                                                             B->active, B->partials + base)));
      kb_finalize<<<o.cnt, 256, 0, st>>>(fine_of(G), prefix_of(B, o), o.cnt, B->partials + base, B->sums);
      note_launch(2);
      base += o.blocks;
    }
    MG_CUDA_TRY(cudaMemcpyAsync(B->h_sums, B->sums, count * 8, cudaMemcpyDeviceToHost, st));
    MG_CUDA_TRY(cudaMemcpyAsync(B->h_sums + count, B->ssum, count * 8, cudaMemcpyDeviceToHost, st));
    MG_CUDA_TRY(cudaStreamSynchronize(st));
    MG_CUDA_TRY(cudaGetLastError());
    return MGGLAM_OK;
  };
  for (int s = 0; s < count; ++s) B->h_active[s] = 1;
  MG_CUDA_TRY(cudaMemcpyAsync(B->active, B->h_active, count * 4, cudaMemcpyHostToDevice, st));
  MG_CUDA_TRY(cudaMemsetAsync(B->guards, 0, count * sizeof(unsigned long long), st));
  if ((rc = outer_residual())) return rc;
  // autotune the smoother's block height once per batch (timed on the fine
  // levels' sweeps, after the first residual has set the base field and source)
  if (B->rows == 0) {
    int best = 4;
    float best_ms = 1e30f;
    for (int cand : {2, 4, 8}) {
      Plan Pt;
      if ((rc = build_plan(B, models, lfs, rho_in, field, prm, cand, &Pt, st))) return rc;
      for (int s = 0; s < count; ++s) B->h_active[s] = 1;
      MG_CUDA_TRY(cudaMemcpyAsync(B->active, B->h_active, count * 4, cudaMemcpyHostToDevice, st));
      cudaEvent_t e0, e1;
      cudaEventCreate(&e0);
      cudaEventCreate(&e1);
      auto pass = [&](int parity) {
        for (const KindPlan& G : Pt.kinds) launch_smooth_phase(B, G.kind, G.lv[0].smooth, cand, parity, st);
      };
      pass(0);  // warm
      cudaEventRecord(e0, st);
      for (int rep = 0; rep < 3; ++rep) pass(rep & 1);
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      if (ms < best_ms) { best_ms = ms; best = cand; }
    }
    B->rows = best;
    // the timing sweeps changed e on the fine levels: start again from zero
    for (int s = 0; s < count; ++s) {
      const size_t bytes = (size_t)B->sv[s].N * B->sv[s].N * B->sv[s].N * 4;
      MG_CUDA_TRY(cudaMemsetAsync(B->sv[s].e[0], 0, bytes, st));
      MG_CUDA_TRY(cudaMemsetAsync(B->sv[s].q0, 0, bytes, st));
    }
    if ((rc = build_plan(B, models, lfs, rho_in, field, prm, B->rows, &P, st))) return rc;
  }
  std::vector<double> snorm(count), eps(count);
  std::vector<mgglam_stats> lst(count);
  for (int s = 0; s < count; ++s) {
    const double n3 = (double)B->sv[s].N * B->sv[s].N * B->sv[s].N;
    const double src = sqrt(B->h_sums[count + s] / n3);
    snorm[s] = source_norm(models[s], src);
    eps[s] = sqrt(B->h_sums[s] / n3) / snorm[s];
    memset(&lst[s], 0, sizeof(mgglam_stats));
    lst[s].resid0 = eps[s];
    lst[s].resid_hist[0] = eps[s];
  }
  // Graph of one batched V-cycle: the kinds' chains of launches are branches of it,
  // so that one kind's small levels, bound by latency, run beside another's.  All a
  // launch bakes in is its table's place and block count; the constants and buffers
  // are in the tables, so other parameters or fields of the same meshes replay the
  // same graph.
  for (size_t k = 0; k < P.kinds.size(); ++k) {
    if (!B->cap[k] && cudaStreamCreateWithFlags(&B->cap[k], cudaStreamNonBlocking) != cudaSuccess) return MGGLAM_ERR_CUDA;
    if (!B->ev[k] && cudaEventCreateWithFlags(&B->ev[k], cudaEventDisableTiming) != cudaSuccess) return MGGLAM_ERR_CUDA;
    if (P.kinds[k].tails) {
      MG_BDISPATCH(P.kinds[k].kind, rc = allow_batch_tail<KK>());
      if (rc) return rc;
    }
  }
  unsigned long long sig = 1469598103934665603ull;
  auto mix = [&](unsigned long long v) { sig = (sig ^ v) * 1099511628211ull; };
  auto mix_phase = [&](const Phase& p) {
    mix(p.cnt);
    mix(p.blocks);
    mix(p.d_off);
    mix(p.p_off);
  };
  for (const KindPlan& G : P.kinds) {
    mix(G.kind);
    mix(G.tails);
    mix(G.tail_off);
    mix(G.tail_solve_off);
    mix(G.tail_smem);
    mix(G.lv.size());
    for (const KindPlan::L& L : G.lv)
      for (const Phase* p : {&L.smooth, &L.restrict_, &L.fas, &L.prolong, &L.coarse}) mix_phase(*p);
  }
  for (int v : {prm[0].nu1, prm[0].nu2, prm[0].coarse_sweeps, B->rows}) mix((unsigned long long)v);
  mix((unsigned long long)(uintptr_t)B->tables);
  if (!(B->vexec && B->vsig == sig)) {
    if (B->vexec) { cudaGraphExecDestroy(B->vexec); B->vexec = nullptr; }
    const long long n0 = launch_count();
    cudaGraph_t g = nullptr;
    bool ok = cudaStreamBeginCapture(B->cap[0], cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      ok = cudaEventRecord(B->ev[0], B->cap[0]) == cudaSuccess;
      for (size_t k = 1; k < P.kinds.size() && ok; ++k) ok = cudaStreamWaitEvent(B->cap[k], B->ev[0], 0) == cudaSuccess;
      for (size_t k = 0; k < P.kinds.size() && ok; ++k) batch_vcycle(B, P.kinds[k], prm[0], B->cap[k]);
      for (size_t k = 1; k < P.kinds.size() && ok; ++k)
        ok = cudaEventRecord(B->ev[k], B->cap[k]) == cudaSuccess &&
             cudaStreamWaitEvent(B->cap[0], B->ev[k], 0) == cudaSuccess;
      ok = cudaStreamEndCapture(B->cap[0], &g) == cudaSuccess && g && ok;
    }
    B->vlaunches = launch_count() - n0;
    note_launch((int)-B->vlaunches);
    if (ok) ok = cudaGraphInstantiate(&B->vexec, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    if (!ok) { cudaGetLastError(); B->vexec = nullptr; return MGGLAM_ERR_CUDA; }
    B->vsig = sig;
  }
  int cyc = 0, outer = 0, status = MGGLAM_OK;
  double rho_est = kInitialContraction;
  const int maxc = prm[0].max_cycles;
  auto worst = [&]() {
    double w = 0.0;
    for (int s = 0; s < count; ++s)
      if (B->h_active[s]) w = fmax(w, eps[s] / fmax(tol, 1e-300));
    return w;
  };
  while (cyc < maxc) {
    bool any = false;
    for (int s = 0; s < count; ++s) {
      const bool act = !(eps[s] <= tol) && isfinite(eps[s]);
      B->h_active[s] = act ? 1 : 0;
      any = any || act;
    }
    if (!any) break;
    MG_CUDA_TRY(cudaMemcpyAsync(B->active, B->h_active, count * 4, cudaMemcpyHostToDevice, st));
    int inner = prm[0].inner_cycles;
    if (inner <= 0) {
      const double lr = log(rho_est);
      const int need = (int)ceil(log(1.0 / worst()) / lr - 1e-9);
      const int cap = (int)ceil(log(kFp32StepGain) / lr - 1e-9);
      inner = need < 1 ? 1 : (need > cap ? cap : need);
    }
    double worst_before = worst();
    int done = 0;
    for (int c = 0; c < inner && cyc < maxc; ++c, ++cyc, ++done) {
      MG_CUDA_TRY(cudaGraphLaunch(B->vexec, st));
      note_launch((int)B->vlaunches);
      for (int s = 0; s < count; ++s)
        if (B->h_active[s]) ++lst[s].cycles;
    }
    for (const KindPlan& G : P.kinds) {  // which leaves e at zero for the next step
      kb_apply<<<G.apply.blocks, 256, 0, st>>>(fine_of(G), prefix_of(B, G.apply), G.apply.cnt, B->active);
      note_launch(1);
    }
    ++outer;
    if ((rc = outer_residual())) return rc;
    for (int s = 0; s < count; ++s) {
      if (!B->h_active[s]) continue;
      const double n3 = (double)B->sv[s].N * B->sv[s].N * B->sv[s].N;
      eps[s] = sqrt(B->h_sums[s] / n3) / snorm[s];
      ++lst[s].outer;
      if (lst[s].outer < 64) lst[s].resid_hist[lst[s].outer] = eps[s];
    }
    const double worst_after = worst();
    if (done > 0 && worst_after > 0.0 && worst_after < worst_before && worst_after / worst_before > kFp32StepGain)
      rho_est = fmin(0.5, fmax(0.01, pow(worst_after / worst_before, 1.0 / done)));
  }
  MG_CUDA_TRY(cudaMemcpyAsync(B->h_guards, B->guards, count * sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                              st));
  MG_CUDA_TRY(cudaStreamSynchronize(st));
  const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  for (int s = 0; s < count; ++s) {
    lst[s].guarded = (long long)B->h_guards[s];
    lst[s].resid = eps[s];
    lst[s].converged = eps[s] <= tol;
    lst[s].seconds = secs;
    if (!isfinite(eps[s])) status = MGGLAM_ERR_NONFINITE;
    else if (status == MGGLAM_OK && !lst[s].converged) status = MGGLAM_ERR_NOT_CONVERGED;
    if (stats) stats[s] = lst[s];
  }
  return status;
}

}  // namespace mg

extern "C" int mgglam_solve_batch(int count, const mgglam_params* prm, const double* a, const float* const* rho,
                                  const int* N, double* const* field, double tol, mgglam_stats* stats, void* stream) {
  if (count < 1 || !prm || !a || !rho || !N || !field || !(tol >= 0.0)) return MGGLAM_ERR_ARG;
  for (int s = 0; s < count; ++s) {
    if (!rho[s] || !field[s]) return MGGLAM_ERR_ARG;
    if (N[s] < 32 || N[s] > 2048 || N[s] % 32) return MGGLAM_ERR_SHAPE;
    if (prm[s].nu1 != prm[0].nu1 || prm[s].nu2 != prm[0].nu2 || prm[s].coarse_sweeps != prm[0].coarse_sweeps)
      return MGGLAM_ERR_ARG;
    if (prm[s].nu1 < 0 || prm[s].nu2 < 0 || prm[s].coarse_sweeps < 0) return MGGLAM_ERR_ARG;
    if (prm[s].cycle != 0) return MGGLAM_ERR_ARG;  // batched solves run V-cycles
  }
  return mg::solve_batch(count, prm, a, rho, N, field, tol, stats, (cudaStream_t)stream);
}
