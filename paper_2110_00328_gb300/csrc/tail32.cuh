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
// side, half side, pairs n^2 h, place in shared memory (floats), TailDiv's factors.
struct __align__(16) TailDims {
  int n, h, np, at, mn, mh, rho, pad;
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
// per level e, u, S, q, R e (except on the first) and the density where used -- and
// returns the bytes (at most 120 KB).
static inline size_t tail_layout(TailArgs& A) {
  int at = 3 * (A.n[0] * A.n[0] * A.n[0] / 2);
  for (int m = 0; m < A.T; ++m) {
    const int n = A.n[m], h = n / 2;
    A.dim[m] = {n, h, n * n * h, at, (65536 + n - 1) / n, (65536 + h - 1) / h, A.rho[m] ? 1 : 0, 0};
    at += A.n[m] * A.n[m] * A.n[m] * (4 + (m > 0 ? 1 : 0) + (A.rho[m] ? 1 : 0));
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
  __device__ __forceinline__ TailLevel(const TailDims& d, int m, float* sm) {
    n = d.n;
    h = d.h;
    np = d.np;
    e = sm + d.at;
    ub = e + 2 * np;
    S = ub + 2 * np;
    q = S + 2 * np;
    Re = q + 2 * np;
    rho = d.rho ? Re + (m > 0 ? 2 * np : 0) : nullptr;
  }
};

// x / d for x < 4096, 1 <= d <= 16: m = ceil(2^16 / d) overestimates 1/d by less than
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

// The V-cycle on the tail's levels; CPT pairs of the first level a thread.
template <int K, int CPT>
__device__ __forceinline__ void tail_cycle(const TailArgs& A, float* sm) {
  const int t0 = threadIdx.x, w0 = t0 & ~31;  // the warp's first pair: a warp works or skips as a whole
  for (int m = 0; m < A.T; ++m) {
    const TailDims D = A.dim[m];
    const TailLevel L(D, m, sm);
    const TailDiv dn{D.mn}, dh{D.mh};
    if (m == 0 || L.rho) {
      for (int t = t0; t < L.np; t += kTailThreads) {
        const int row = dh.div(t), i = dn.div(row), g = 2 * t, p = (i + row - i * L.n) & 1;
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          const int x = (p ^ o) * L.np + t;
          if (L.rho) L.rho[x] = A.rho[m][g + o];
          if (m == 0) {
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
    const TailLevel L(D, m, sm);
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
      const float* Dc = TailLevel(A.dim[m + 1], m + 1, sm).Re;
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
      const TailLevel H(A.dim[m + 1], m + 1, sm);
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
            if (m > 0) L.Re[g + o] = v - L.Re[g + o];
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

}  // namespace mg
