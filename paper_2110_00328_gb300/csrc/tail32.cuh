// tail32.cuh -- the coarsest levels of an FP32 correction-form V-cycle in one
// thread block.
//
// At 16^3 cells and below a level's kernels are bound by launch latency, not by
// work (a 16^3 colour pass is 2048 updates; its kernel takes 2 us in a graph).
// From the first level with at most kTailMaxCells cells down to the coarsest, the
// whole V-cycle -- FAS source, pre-smoothing, restriction of the defect, the
// coarsest relaxation, prolongation-correction and post-smoothing (Sec. 3.2.1) --
// runs inside one CTA with the levels held in shared memory.
//
// What bounds it is the latency of one step -- shared-memory loads, a local solve
// and a barrier, a hundred times over -- and instruction fetch, since most of the
// code runs once or twice.  So a thread owns the same pairs of cells (i, j, 2kk),
// (i, j, 2kk + 1), one of each colour, in every step of a level: base field,
// source, correction and neighbour offsets stay in its registers through a
// smoothing call; a cell reads its six neighbours' quantity q = Delta w(u, e) (e
// itself for the symmetron and CQ) from shared memory, not e and u; the levels
// are stored colour by colour, pair t at t, so that a warp's reads are free of
// bank conflicts; the way down and the way up share one smoothing loop; and a
// level of at most 32 pairs is one warp's, without block barriers.  Every step
// applies the per-cell arithmetic of the one-kernel-per-step path in the same
// red-black order, so the result is the same iterate.
// Measured: a V(2,2) tail from 16^3 with 16 coarsest sweeps takes 24.6 us (f(R) n = 1);
// its 16^3 level as ten kernels and the levels below as one block took about 40.  A
// 16^3 colour pass is 0.9 us of it, an 8^3 one 0.35 us, a 4^3 one 0.23 us.
#pragma once
#include "mixed_common.cuh"

namespace mg {

constexpr int kTailMaxCells = 4096;  // the first tail level has at most this many cells
constexpr int kTailMaxLevels = 6;
constexpr int kTailThreads = 1024;

// A level's numbers, formed on the host (each CTA would spend a microsecond on them):
// side, half side, pairs n^2 h, place in shared memory (floats), TailDiv's factors,
// and whether the density and R e are held.
struct __align__(16) TailDims {
  int n, h, np, at, mn, mh, rho, re;
};

struct TailArgs {
  TailDims dim[kTailMaxLevels];
  int T;                              // tail levels (first, ..., coarsest), of even side
  int n[kTailMaxLevels];              // their sides
  LevelF lf[kTailMaxLevels];
  int zr[kTailMaxLevels];             // restriction: the second colour's defect is zero (relaxed last, exactly)
  float* e;                           // first tail level, global: R e on entry, the correction on return
  const float* ub;                    // base field
  const float* S;                     // R d, the restricted defect (the FAS source is formed here)
  const float* rho[kTailMaxLevels];   // density pyramid (nullptr when the operator takes none)
  int nu1, nu2, coarse_sweeps;
  unsigned long long* guard;          // positivity-guard replacements (counted), or nullptr
};

// Whether levels l .. nlev-1 can run as a tail.
static inline bool tail_fits(const int* n, int nlev, int l) {
  if (nlev - l > kTailMaxLevels || (long long)n[l] * n[l] * n[l] > kTailMaxCells) return false;
  for (int m = l; m < nlev; ++m)
    if (n[m] % 2) return false;
  return true;
}

// Places the levels in shared memory -- three sums a pair of the first level, then
// per level e, u, S, q, R e (on the first only when inner) and the density where
// used -- and returns the bytes (at most 120 KB, 137 KB when inner).
static inline size_t tail_layout(TailArgs& A, bool inner = false) {
  int at = 3 * (A.n[0] * A.n[0] * A.n[0] / 2);
  for (int m = 0; m < A.T; ++m) {
    const int n = A.n[m], h = n / 2;
    const int re = m > 0 || inner, rho = A.rho[m] ? 1 : 0;
    A.dim[m] = {n, h, n * n * h, at, (65536 + n - 1) / n, (65536 + h - 1) / h, rho, re};
    at += n * n * n * (4 + re + rho);
  }
  return (size_t)at * sizeof(float);
}

// Pairs of the first level a thread owns.
static inline int tail_cpt(int n0) { return n0 * n0 * n0 / 2 > kTailThreads ? 2 : 1; }

// One level in shared memory: np pairs; colour k of e, ub, S, q, rho at k np, R e in
// natural order.
struct TailLevel {
  int n, h, np;
  float *e, *ub, *S, *q, *Re, *rho;
  __device__ __forceinline__ TailLevel(const TailDims& d, float* sm) {
    n = d.n;
    h = d.h;
    np = d.np;
    e = sm + d.at;
    ub = e + 2 * np;
    S = ub + 2 * np;
    q = S + 2 * np;
    Re = q + 2 * np;
    rho = d.rho ? Re + (d.re ? 2 * np : 0) : nullptr;
  }
};

// x / d for x < 4096, 1 <= d <= 16, or x < 2048, d <= 32: m = ceil(2^16 / d) overestimates 1/d by less than
// d / 2^16, which x (d - 1) < 2^16 keeps from reaching the next integer.
struct TailDiv {
  int m;
  __device__ __forceinline__ int div(int x) const { return (x * m) >> 16; }
};

// Pair t of a level: the offsets of the i and j neighbours' pairs (the same for
// both cells), the pairs of the k neighbours outside the pair, and the colour p of
// its even-k cell.
struct TailPair {
  int t, dip, dim, djp, djm, kl, kr, p, row, kk;
  __device__ __forceinline__ void set(int n, int h, int x, TailDiv dn, TailDiv dh) {
    t = x;
    row = dh.div(x);
    kk = x - row * h;
    const int i = dn.div(row), j = row - i * n, nh = n * h;
    dip = i + 1 < n ? nh : nh - n * nh;
    dim = i > 0 ? -nh : n * nh - nh;
    djp = j + 1 < n ? h : h - nh;
    djm = j > 0 ? -h : nh - h;
    kl = kk > 0 ? t - 1 : t + h - 1;
    kr = kk + 1 < h ? t + 1 : t + 1 - h;
    p = (i + j) & 1;
  }
  // the neighbour sum of the colour-k cell; q1: the other colour's q
  __device__ __forceinline__ float sum(const float* q1, int k) const {
    return (q1[t + dip] + q1[t + dim]) + (q1[t + djp] + q1[t + djm]) + (q1[t] + q1[(p ^ k) ? kr : kl]);
  }
};

// The V-cycle on the tail's levels; CPT pairs of the first level a thread.  INNER:
// the first level is in shared memory already, and its e^H - R e is left there.
template <int K, int CPT, bool INNER = false>
__device__ __forceinline__ void tail_cycle(const TailArgs& A, float* sm) {
  const int t0 = threadIdx.x, w0 = t0 & ~31;  // the warp's first pair: a warp works or skips as a whole
  for (int m = 0; m < A.T; ++m) {
    const TailDims D = A.dim[m];
    const TailLevel L(D, sm);
    const TailDiv dn{D.mn}, dh{D.mh};
    if ((m == 0 && !INNER) || L.rho) {
      for (int t = t0; t < L.np; t += kTailThreads) {
        const int row = dh.div(t), i = dn.div(row), g = 2 * t, p = (i + row - i * L.n) & 1;
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          const int x = (p ^ o) * L.np + t;
          if (L.rho) L.rho[x] = A.rho[m][g + o];
          if (m == 0 && !INNER) {
            const float e = A.e[g + o], u = A.ub[g + o];
            L.e[x] = e;
            L.ub[x] = u;
            L.S[x] = A.S[g + o];
            L.q[x] = nbq<K>(u, e);
          }
        }
      }
    }
  }
  __syncthreads();
  unsigned ng = 0;
#pragma unroll 1
  for (int step = 0; step < 2 * A.T - 1; ++step) {
    const bool down = step < A.T;
    const int m = down ? step : 2 * A.T - 2 - step;
    const LevelF& f = A.lf[m];
    const TailDims D = A.dim[m];
    const TailLevel L(D, sm);
    const int np = L.np;
    const TailDiv dn{D.mn}, dh{D.mh};
    TailPair P[CPT];
    float u[CPT][2], s[CPT][2], e[CPT][2], r[CPT][2];  // [cell by colour]
#pragma unroll
    for (int a = 0; a < CPT; ++a)
      if (w0 + a * kTailThreads < np) {
        P[a].set(L.n, L.h, min(t0 + a * kTailThreads, np - 1), dn, dh);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int x = k * np + P[a].t;
          u[a][k] = L.ub[x];
          s[a][k] = L.S[x];
          e[a][k] = L.e[x];
          r[a][k] = L.rho ? L.rho[x] : 1.f;
        }
      }
    if (down) {
      // FAS source: S <- M(R e) - R d (S holds R d, e and q those of R e)
#pragma unroll
      for (int a = 0; a < CPT; ++a)
        if (w0 + a * kTailThreads < np) {
#pragma unroll
          for (int k = 0; k < 2; ++k)
            s[a][k] = local_M<K>(f, u[a][k], e[a][k], r[a][k], P[a].sum(L.q + (k ^ 1) * np, k)) - s[a][k];
          if (t0 + a * kTailThreads < np) {
#pragma unroll
            for (int k = 0; k < 2; ++k) L.S[k * np + P[a].t] = s[a][k];
          }
        }
    } else {
      // e += P(e^H - R e), which the coarser level left in its R e; f(R): where u + e would
      // not be positive the total field halves
      const int nc = L.h;
      const float* Dc = TailLevel(A.dim[m + 1], sm).Re;
#pragma unroll
      for (int a = 0; a < CPT; ++a)
        if (t0 + a * kTailThreads < np) {
          const int kk = P[a].kk, i = dn.div(P[a].row), j = P[a].row - i * L.n;
          const int I = i >> 1, J = j >> 1;
          const int I2 = wrapi(I + ((i & 1) ? 1 : -1), nc), J2 = wrapi(J + ((j & 1) ? 1 : -1), nc);
          const float *a0 = Dc + (I * nc + J) * nc, *a1 = Dc + (I2 * nc + J) * nc, *a2 = Dc + (I * nc + J2) * nc,
                      *a3 = Dc + (I2 * nc + J2) * nc;
          auto row = [&](int k) { return 9.f * a0[k] + 3.f * (a1[k] + a2[k]) + a3[k]; };
          const float R = 3.f * row(kk);
          const float c[2] = {(R + row(kk > 0 ? kk - 1 : nc - 1)) * (1.f / 64.f),
                              (R + row(kk + 1 < nc ? kk + 1 : 0)) * (1.f / 64.f)};
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float old = e[a][k];
            float v = old + ((P[a].p ^ k) ? c[1] : c[0]);
            if (is_fr(K) && !(u[a][k] + v > 0.f)) {
              v = 0.5f * (old - u[a][k]);
              ++ng;
            }
            e[a][k] = v;
            L.q[k * np + P[a].t] = nbq<K>(u[a][k], v);
          }
        }
    }
    __syncthreads();
    // red-black sweeps
    const int sweeps = down ? (m + 1 < A.T ? A.nu1 : A.coarse_sweeps) : A.nu2;
    const bool solo = np <= 32;
    if (!solo || w0 == 0) {
#pragma unroll 1
      for (int sw = 0; sw < sweeps; ++sw)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
          for (int a = 0; a < CPT; ++a)
            if (w0 + a * kTailThreads < np) {
              const float v = update_quad<K>(f, u[a][k], e[a][k], r[a][k], s[a][k],
                                             P[a].sum(L.q + (k ^ 1) * np, k));
              e[a][k] = v;
              if (t0 + a * kTailThreads < np) L.q[k * np + P[a].t] = nbq<K>(u[a][k], v);
            }
          if (solo) __syncwarp();
          else __syncthreads();
        }
    }
    if (down && m + 1 < A.T) {
      // d = M(e) - S at the 8 children of each coarse cell, averaged: three sums a pair,
      // then a coarse cell's four pairs; coarse e starts at R e
      const bool zr = A.zr[m] && A.nu1 > 0;
#pragma unroll
      for (int a = 0; a < CPT; ++a)
        if (t0 + a * kTailThreads < np) {
          const int t = P[a].t;
          float d = local_M<K>(f, u[a][0], e[a][0], r[a][0], P[a].sum(L.q + np, 0)) - s[a][0];
          if (!zr) d += local_M<K>(f, u[a][1], e[a][1], r[a][1], P[a].sum(L.q, 1)) - s[a][1];
          sm[t] = e[a][0] + e[a][1];
          sm[np + t] = u[a][0] + u[a][1];
          sm[2 * np + t] = d;
          L.e[t] = e[a][0];
          L.e[np + t] = e[a][1];
        }
      __syncthreads();
      const TailLevel H(A.dim[m + 1], sm);
      const int nc = H.n;
      const TailDiv dc{D.mh};
      for (int t = t0; t < nc * nc * nc; t += kTailThreads) {
        const int IJ = dc.div(t), Kc = t - IJ * nc, I = dc.div(IJ), J = IJ - I * nc;
        const int b = (2 * I * L.n + 2 * J) * nc + Kc;
        auto mean = [&](const float* v) {
          return 0.125f * ((v[b] + v[b + nc]) + (v[b + L.n * nc] + v[b + L.n * nc + nc]));
        };
        const int x = ((I + J + Kc) & 1) * H.np + (t >> 1);
        const float em = mean(sm), um = mean(sm + np);
        H.e[x] = em;
        H.Re[t] = em;
        H.ub[x] = um;
        H.S[x] = mean(sm + 2 * np);
        H.q[x] = nbq<K>(um, em);
      }
    } else {
      // what the finer level takes: e^H - R e in place of R e; the first level's e
#pragma unroll
      for (int a = 0; a < CPT; ++a)
        if (t0 + a * kTailThreads < np) {
          const int g = 2 * P[a].t;
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            const float v = (P[a].p ^ o) ? e[a][1] : e[a][0];
            if (m > 0 || INNER) L.Re[g + o] = v - L.Re[g + o];
            else A.e[g + o] = v;
          }
        }
    }
    __syncthreads();
  }
  if (is_fr(K)) count_guards(A.guard, ng);
}

template <int K, int CPT>
__global__ void __launch_bounds__(kTailThreads) k_tail32(TailArgs A) {
  extern __shared__ float sm[];
  tail_cycle<K, CPT>(A, sm);
}

// ---------------------------------------------------------------------------
// k_tail32_cluster: the tail from a level of side 20 .. 32 on (the finest: 8 .. 32)
// ---------------------------------------------------------------------------
//
// At 32^3 a level's kernels are still bound by their launches: eight colour passes,
// restriction, FAS source and prolongation took 33 us in a graph ahead of the one-
// block tail's 18, with 16384 updates a pass.  One block is too narrow for them (at
// 16^3 it spends more than half its time issuing instructions), so the first two
// levels are spread over a cluster, two planes of a level a CTA and a pair of cells a
// thread, kept in registers as in the one-block tail; shared memory holds the quantity
// q of the CTA's planes and of one more on either side, which the neighbouring CTAs
// write.  A step then costs a cluster barrier instead of a launch.  A coarse plane is
// restricted into the memory of the CTA that relaxes it, and the coarse difference
// left there for its neighbours to read; from the third level on (8^3) the first CTA
// runs the one-block tail while the others wait.  The finest level of a solve of such
// a side takes the same form, all inner cycles of an outer step in one launch.
// Measured (V(2,2), f(R) n = 1): a 32^3 cycle 28 us -- a 32^3 colour pass 0.76 us of it,
// a 16^3 one 0.53 (one block: 0.9), an 8^3 one 0.20, a 4^3 one 0.16, the transfers 11 --
// against 67 as kernels and a one-block tail; a 32^3 solve 676 us before, 490 now.  With
// eight CTAs of four planes, a thread's two pairs spilled: 50 us a cycle.
constexpr int kTailMaxSide = 16;      // beyond, a tail is a cluster's
constexpr int kClusterCells = 32768;  // its first level has at most this many cells
constexpr int kClusterCtas = 16;      // CTAs beyond a level's planes / 2 only take part in the barriers

struct ClusterArgs {
  TailArgs in;              // the levels below the second (T = 0: none)
  LevelF lf[2];             // the first two levels: sides n, n / 2
  const float* rho[2];
  int n, mn, mh, mq;        // TailDiv's factors of n, n / 2 and n / 4
  int zr[2];                // as TailArgs'
  int split;                // the first level's arrays in the red-black split layout
  int finest, fresh;        // the finest level: S is the equation's own; e = 0 on entry, not read
  int second;               // prolong to the second colour only (the first is relaxed next, from nothing of its own)
  int cycles;               // V-cycles to run (1 unless finest)
  float* e;
  const float *ub, *S;
};

// Whether level l can be a cluster's first level: beyond the one-block tail's sides,
// or the finest, which that tail does not take.
static inline bool cluster_fits(const int* n, int nlev, int l) {
  return n[l] % 4 == 0 && n[l] >= (l > 0 ? kTailMaxSide + 4 : 8) && n[l] <= 2 * kClusterCtas && l + 1 < nlev &&
         tail_fits(n, nlev, l + 1);
}

// Floats of a level of side n before the next one's: q of four planes, three sums a
// pair, three planes of the coarse difference; the second level also e, u, S as they
// arrive and its own difference.
__host__ __device__ __forceinline__ constexpr int cluster_floats(int n, bool second) {
  return 4 * n * n + 3 * n * n + 3 * (n / 2) * (n / 2) + (second ? 6 * n * n + 2 * n * n : 0);
}

static inline size_t cluster_layout(ClusterArgs& A) {
  const int n = A.n, h = n / 2, d = n / 4;
  A.mn = (65536 + n - 1) / n;
  A.mh = (65536 + h - 1) / h;
  A.mq = (65536 + d - 1) / d;
  return (size_t)(cluster_floats(n, false) + cluster_floats(h, true)) * sizeof(float) +
         (A.in.T ? tail_layout(A.in, true) : 0);
}

__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();  // the aligned form wants whole warps (2% of a cycle faster than the other)
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of p's counterpart in CTA rank's shared memory, and accesses to it
__device__ __forceinline__ unsigned cluster_addr(const float* p, unsigned rank) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_st(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float cluster_ld(unsigned a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// A thread's pair of a level of side n, two planes a CTA: TailPair with whole planes on
// either side.  warp: the thread's warp has pairs; own: the thread has.
template <int K>
struct ClusterPair {
  float *q, *sums, *Dc;  // the level's arrays: colour k of q at 2 n^2 k
  int nh, t, djp, djm, kl, kr, p, g;
  unsigned halo;         // the pair's colour-0 q in the neighbouring CTA's halo
  bool warp, own;
  float u[2], s[2], e[2], r[2];

  __device__ __forceinline__ void set(int n, TailDiv dn, TailDiv dh, int rank, float* sm) {
    const int h = n >> 1, nact = h, np = rank < nact ? n * n : 0, t0 = threadIdx.x;
    nh = n * h;
    q = sm;
    sums = q + 8 * nh;
    Dc = sums + 6 * nh;
    warp = (t0 & ~31) < np;
    own = t0 < np;
    const int x = min(t0, n * n - 1), row = dh.div(x), kk = x - row * h, pl = dn.div(row), j = row - pl * n;
    t = x + nh;
    djp = j + 1 < n ? h : h - nh;
    djm = j > 0 ? -h : nh - h;
    kl = t + (kk > 0 ? -1 : h - 1);
    kr = t + (kk + 1 < h ? 1 : 1 - h);
    p = (pl + j) & 1;  // a CTA's first plane is even
    g = 2 * rank * nh + x;
    const int to = pl ? rank + 1 : rank - 1;
    halo = cluster_addr(pl ? q + x - nh : q + 3 * nh + x, to < 0 ? nact - 1 : (to < nact ? to : 0));
  }
  __device__ __forceinline__ float sum(int k) const {  // of the colour-k cell's neighbours
    const float* q1 = q + (k ^ 1) * 4 * nh;
    return (q1[t + nh] + q1[t - nh]) + (q1[t + djp] + q1[t + djm]) + (q1[t] + q1[(p ^ k) ? kr : kl]);
  }
  __device__ __forceinline__ void put(int k) const {  // the cell's q, here and as a neighbour's halo
    const float v = nbq<K>(u[k], e[k]);
    if (own) {
      q[4 * nh * k + t] = v;
      cluster_st(halo + 16 * nh * k, v);
    }
  }
  // FAS source: S <- M(R e) - R d
  __device__ __forceinline__ void fas(const LevelF& f) {
    if (warp) {
#pragma unroll
      for (int k = 0; k < 2; ++k) s[k] = local_M<K>(f, u[k], e[k], r[k], sum(k)) - s[k];
    }
    cluster_barrier();
  }
  __device__ __forceinline__ void smooth(const LevelF& f, int sweeps) {
#pragma unroll 1
    for (int sw = 0; sw < sweeps; ++sw)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (warp) {
          e[k] = update_quad<K>(f, u[k], e[k], r[k], s[k], sum(k));
          put(k);
        }
        cluster_barrier();
      }
  }
  // The three sums of each pair for the restriction, and a coarse cell's mean of its four pairs' (J, Kc of plane rank)
  __device__ __forceinline__ void restrict_sums(const LevelF& f, bool zr) {
    if (own) {
      float d = local_M<K>(f, u[0], e[0], r[0], sum(0)) - s[0];
      if (!zr) d += local_M<K>(f, u[1], e[1], r[1], sum(1)) - s[1];
      float* o = sums + t - nh;
      o[0] = e[0] + e[1];
      o[2 * nh] = u[0] + u[1];
      o[4 * nh] = d;
    }
    __syncthreads();
  }
  static __device__ __forceinline__ float mean(const float* v, int nh, int h) {
    return 0.125f * ((v[0] + v[h]) + (v[nh] + v[nh + h]));
  }
  // e += P(D) from the three planes of the coarse difference about the CTA's
  __device__ __forceinline__ void prolong(int h, TailDiv dn, TailDiv dh, bool second, unsigned& ng) {
    if (warp) {
      int x = t - nh;
      asm("" : "+r"(x));  // formed anew rather than kept in registers
      const int row = dh.div(x), kk = x - row * h, pl = dn.div(row), j = row - pl * 2 * h;
      const int I2 = pl ? 2 : 0, J = j >> 1, J2 = wrapi(J + ((j & 1) ? 1 : -1), h);
      const float *a0 = Dc + (h + J) * h, *a1 = Dc + (I2 * h + J) * h, *a2 = Dc + (h + J2) * h,
                  *a3 = Dc + (I2 * h + J2) * h;
      auto wrow = [&](int k) { return 9.f * a0[k] + 3.f * (a1[k] + a2[k]) + a3[k]; };
      const float R = 3.f * wrow(kk);
      const float c[2] = {(R + wrow(kk > 0 ? kk - 1 : h - 1)) * (1.f / 64.f),
                          (R + wrow(kk + 1 < h ? kk + 1 : 0)) * (1.f / 64.f)};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (k == 0 && second) continue;
        const float old = e[k];
        float v = old + ((p ^ k) ? c[1] : c[0]);
        if (is_fr(K) && !(u[k] + v > 0.f)) {
          v = 0.5f * (old - u[k]);
          ng += own;
        }
        e[k] = v;
        put(k);
      }
    }
    cluster_barrier();
  }
};

// The levels below the second, apart from the cluster kernel's registers.
template <int K>
__device__ __noinline__ void cluster_inner(const TailArgs& A, float* sm) {
  tail_cycle<K, 1, true>(A, sm);
}

template <int K>
__global__ void __launch_bounds__(kTailThreads) k_tail32_cluster(const __grid_constant__ ClusterArgs A) {
  extern __shared__ float sm[];
  int rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int n = A.n, h = n >> 1, d = n >> 2, t0 = threadIdx.x;
  const TailDiv dn{A.mn}, dh{A.mh}, dd{A.mq};
  float* const sm1 = sm + cluster_floats(n, false);
  float* const in1 = sm1 + 7 * h * h + 3 * d * d;  // the second level's e, u, S: colour k of array a at (2 a + k) h^2
  float* const D1 = in1 + 6 * h * h;               // its e^H - R e, natural order
  float* const inner = D1 + 2 * h * h;
  ClusterPair<K> c;
  c.set(n, dn, dh, rank, sm);
  if (c.warp) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int x = A.split ? k * n * c.nh + c.g : 2 * c.g + (c.p ^ k);
      c.u[k] = A.ub[x];
      c.s[k] = A.S[x];
      c.e[k] = A.fresh ? 0.f : A.e[x];
      c.r[k] = A.rho[0] ? A.rho[0][x] : 1.f;
    }
  }
  cluster_barrier();  // every CTA runs: its memory can be written
  if (c.warp) {
    c.put(0);
    c.put(1);
  }
  cluster_barrier();
  if (!A.finest) c.fas(A.lf[0]);
  unsigned ng = 0;
#pragma unroll 1
  for (int cyc = 0; cyc < A.cycles; ++cyc) {
    c.smooth(A.lf[0], A.in.nu1);
    // plane 'rank' of the second level, into the CTA that relaxes it
    c.restrict_sums(A.lf[0], A.zr[0] && A.in.nu1 > 0);
    if (rank < h && t0 < h * h) {
      const int J = dh.div(t0), Kc = t0 - J * h;
      const float* v = c.sums + 2 * J * h + Kc;
      const int col = (rank + J + Kc) & 1;
      const float* o = in1 + col * h * h + ((rank & 1) * h + J) * d + (Kc >> 1);
#pragma unroll
      for (int a = 0; a < 3; ++a)
        cluster_st(cluster_addr(o + 2 * a * h * h, rank >> 1), ClusterPair<K>::mean(v + 2 * a * c.nh, c.nh, h));
    }
    cluster_barrier();
    {
      ClusterPair<K> b;
      b.set(h, dh, dd, rank, sm1);
      float Re[2];
      if (b.warp) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float* o = in1 + k * h * h + b.t - b.nh;
          Re[k] = b.e[k] = o[0];
          b.u[k] = o[2 * h * h];
          b.s[k] = o[4 * h * h];
          b.r[k] = A.rho[1] ? A.rho[1][2 * b.g + (b.p ^ k)] : 1.f;
          b.put(k);
        }
      }
      cluster_barrier();
      b.fas(A.lf[1]);
      b.smooth(A.lf[1], A.in.T ? A.in.nu1 : A.in.coarse_sweeps);
      if (A.in.T) {
        const TailLevel H(A.in.dim[0], inner);
        b.restrict_sums(A.lf[1], A.zr[1] && A.in.nu1 > 0);
        if (rank < d && t0 < d * d) {
          const int J = dd.div(t0), Kc = t0 - J * d;
          const float* v = b.sums + 2 * J * d + Kc;
          const int g = (rank * d + J) * d + Kc, x = ((rank + J + Kc) & 1) * H.np + (g >> 1);
          const float em = ClusterPair<K>::mean(v, b.nh, d), um = ClusterPair<K>::mean(v + 2 * b.nh, b.nh, d);
          cluster_st(cluster_addr(H.e + x, 0), em);
          cluster_st(cluster_addr(H.Re + g, 0), em);
          cluster_st(cluster_addr(H.ub + x, 0), um);
          cluster_st(cluster_addr(H.S + x, 0), ClusterPair<K>::mean(v + 4 * b.nh, b.nh, d));
          cluster_st(cluster_addr(H.q + x, 0), nbq<K>(um, em));
        }
        cluster_barrier();
        if (rank == 0) cluster_inner<K>(A.in, inner);
        cluster_barrier();
        if (rank < d && t0 < 3 * d * d) {
          const int Il = dd.div(dd.div(t0)), src = t0 + (wrapi(rank - 1 + Il, d) - Il) * d * d;
          b.Dc[t0] = cluster_ld(cluster_addr(H.Re + src, 0));
        }
        __syncthreads();
        b.prolong(d, dh, dd, false, ng);
        b.smooth(A.lf[1], A.in.nu2);
      }
      if (b.own) {
        const int g = 2 * (b.t - b.nh);
#pragma unroll
        for (int k = 0; k < 2; ++k) D1[g + (b.p ^ k)] = b.e[k] - Re[k];
      }
    }
    cluster_barrier();
    if (rank < h && t0 < 3 * h * h) {
      const int Il = dh.div(dh.div(t0)), I = wrapi(rank - 1 + Il, h);
      c.Dc[t0] = cluster_ld(cluster_addr(D1 + t0 + ((I & 1) - Il) * h * h, I >> 1));
    }
    __syncthreads();
    c.prolong(h, dn, dh, A.second, ng);
    c.smooth(A.lf[0], A.in.nu2);
  }
  if (c.own) {
#pragma unroll
    for (int k = 0; k < 2; ++k) A.e[A.split ? k * n * c.nh + c.g : 2 * c.g + (c.p ^ k)] = c.e[k];
  }
  if (is_fr(K)) count_guards(A.in.guard, ng);
}

}  // namespace mg
