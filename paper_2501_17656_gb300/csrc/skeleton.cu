// skeleton.cu -- nested cluster bases by recursive skeletonization (interpolative
// decompositions), the tolerance-driven alternative to Chebyshev interpolation.
//
// The paper's H2 matrices come from an algebraic construction to a relative accuracy
// eps with adaptive ranks (Sec. 4.1, "relative accuracy 1e-9"). Here every cluster
// tau gets a skeleton, a subset of its points whose matrix rows interpolate the
// cluster's far-field rows:
//     A(X_tau, F_tau) ~= T_tau A(skel_tau, F_tau),   T_tau[skel_tau, :] = I.
// Skeletons are nested: a leaf chooses among its points, a parent among the union of
// its children's skeletons (the candidates, first child first). The factors play the
// roles of the Chebyshev ones -- leaf basis U = T_leaf, transfer E_c = the rows of
// T_parent belonging to child c's skeleton, coupling S^0 = A(skel_tau, skel_sigma) --
// and the QR chain of fill.cu orthonormalises them unchanged.
//
// Per cluster tau at tree level ell (levels L down to t*, one launch per level):
//  1. the far-field sample F_tau: the candidates of every far partner of tau at
//     level ell, then, for every far partner sigma' of tau's parent, the candidates
//     of sigma''s two children concatenated and thinned to every s-th entry from the
//     first, s = ceil(count / 128);
//  2. R0 = the R factor of W = A(F_tau, candidates): the sampled rows are generated
//     in chunks of 32 and folded into an upper-triangular R in shared memory by
//     Householder reflections that touch only row j of R and the chunk (a
//     tall-skinny QR; W itself is never stored);
//  3. greedy column-pivoted Householder QR of R0 (the column of largest remaining
//     norm; columns within a relative 1e-10 of the largest squared norm are tied and
//     the lowest index wins), stopped at rank_max, at min(rows, candidates), or once
//     the best remaining norm is <= tol * the first pivot's norm;
//  4. T[pivot a] = e_a for the r pivots and T[pivot r + b] = (R11^{-1} R12)[:, b].
// A cluster with an empty sample keeps its first min(candidates, rank_max)
// candidates with T = [I; 0].
#include <algorithm>
#include <cmath>
#include <cstddef>

#include "internal.h"

namespace h2mg {

constexpr int SK_CAND = 128;        // candidates of a cluster at most (two skeletons of <= 64)
constexpr int SK_CHUNK = 32;        // sampled rows folded into R at a time
constexpr int SK_SAMPLE_CAP = 128;  // points kept per far partner of the parent
constexpr double SK_TIE = 1e-10;    // relative tie band of the pivot choice

// Block-wide max / min helpers; red has one entry per warp.
__device__ double block_max(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double m = red[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = fmax(m, red[i]);
  __syncthreads();
  return m;
}
__device__ int block_min_int(int v, int* red) {
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int m = red[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = min(m, red[i]);
  __syncthreads();
  return m;
}

// How a CTA folds the rows of a cluster with at most NC candidates: NG groups of warps, each
// with a chunk of its own in hand, LPC lanes per column, and two warps per group for the
// reflectors.
template <int NC>
struct Skel {
  static constexpr int NG = NC == 64 ? 3 : 2, LPC = NC == 64 ? 4 : 2;
  static constexpr int OWN = SK_CHUNK / LPC;               // rows of a column per lane, in registers
  static constexpr int CPW = 32 / LPC;                     // columns per warp
  static constexpr int GROUP = NC * LPC + 64, THREADS = NG * GROUP;
  static constexpr int FILL = 8;                           // kernel values staged at a time
};

// What the warps of a group share.
template <int NC>
struct SkelGroup {
  double stage[Skel<NC>::FILL * NC * Skel<NC>::LPC];   // kernel values on their way into the owning thread's registers
  alignas(16) double v[2][SK_CHUNK]; // reflectors j and j + 1; row i at (i % LPC) * OWN + i / LPC (read in pairs)
  double col[SK_CHUNK];              // column j + 1 of the chunk, on its way to the first warps
  double alpha;                      // R's diagonal there
  double tau[2];
  int go[2];
  int done;                          // reflectors applied so far, over all its chunks
};

// Shared memory of k_skeletonize<NC>. R is column-major with ld NC + 1: rows and columns are
// both read without bank conflicts.
template <int NC>
struct SkelSmem {
  double R[NC * (NC + 1)];
  SkelGroup<NC> g[Skel<NC>::NG];
  double nrm[NC], sig[NC];
  double red[32];
  double bcast[3];
  int piv[NC];
  int ired[32];
  int late;                          // a wait for another group ran out
};

static_assert(offsetof(SkelSmem<64>, g) % 16 == 0 && sizeof(SkelGroup<64>) % 16 == 0 &&
                  offsetof(SkelGroup<64>, v) % 16 == 0 && offsetof(SkelSmem<128>, g) % 16 == 0 &&
                  sizeof(SkelGroup<128>) % 16 == 0 && offsetof(SkelGroup<128>, v) % 16 == 0,
              "reflectors are read 16 bytes at a time");

// Reflector j of a chunk, by the group's first two warps: v = column j (one row per lane) /
// (alpha - beta), alpha = R_jj, and tau, each with a division of its own behind the square
// root. A column of zeros leaves everything as it is.
template <int NC>
__device__ __forceinline__ void make_reflector(SkelGroup<NC>& sg, double* R, int j, int warp, int lane) {
  using K = Skel<NC>;
  const double c = sg.col[lane];
  double s = __dmul_rn(c, c);
  for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
  const double alpha = sg.alpha;
  const bool go = s > 0.0;
  if (go) {
    const double beta = -copysign(sqrt(__fma_rn(alpha, alpha, s)), alpha);
    const double quot = __ddiv_rn(warp ? __dsub_rn(beta, alpha) : c, warp ? beta : __dsub_rn(alpha, beta));
    if (warp == 0) sg.v[j & 1][(lane % K::LPC) * K::OWN + lane / K::LPC] = quot;
    if (warp == 1 && lane == 0) {
      sg.tau[j & 1] = quot;
      R[j + j * (NC + 1)] = beta;
    }
  }
  if (warp == 0 && lane == 0) sg.go[j & 1] = go;
}

// Waits until a group has applied `want` reflectors, two seconds at most; after a wait that
// ran out, no wait of the CTA waits any more.
__device__ __forceinline__ void wait_group(const int* done, int want, int* late) {
  const volatile int* d = done;
  if (*d >= want) return;
  const long long t0 = clock64();
  while (*d < want && !*(volatile int*)late)
    if (clock64() - t0 > (1ll << 32)) *(volatile int*)late = 1;
}

// Folds chunk number `ch` (32 rows) into R: lane q of the LPC that own column k holds c[OWN],
// the rows q, q + LPC, .. The group's first two warps own no column: while the others apply
// reflector j they make reflector j + 1, as soon as the warp that owns column j + 1 has handed
// it over. Chunks go to the groups in turn, and each follows the one before it through the
// columns: step j waits until that one has finished with row j of R. Every sum over the rows is
// one tree of pairs (16, 8, 4, 2, 1 rows apart), rounded step by step, and the chunks meet R
// one after the other: R, and with it every skeleton and basis, has the same bits as with a
// warp per column and a row per lane, so that FP32 and split-TF32 products of the bases round
// alike. (Chunks of 128 rows, and parts of a cluster's rows on CTAs of their own, built 8192
// points in 99 ms, but turned last bits of FP32 results.)
//
// A step is the columns' work, 98 float64 operations per column of 32 rows (3700 clocks on
// average for 128 columns on a pipe of 2 per clock and SM), and the next reflector's chain: a
// sum, a square root and a division. Together they keep the float64 pipe 72 to 83% busy. A
// warp per column spent 8 operations for every 2 of the columns' own, mostly on warp-wide sums
// and on the reflector in every warp: 8192 points in 296 ms. One group of four lanes per
// column 171 ms; with the groups, one's chain runs beside another's columns: 138 ms.
template <int NC>
__device__ __forceinline__ void fold_chunk(SkelSmem<NC>& sm, int nc, int64_t ch, int group, int k, int q,
                                           double (&c)[Skel<NC>::OWN]) {
  using K = Skel<NC>;
  const int w = (int)(threadIdx.x % K::GROUP >> 5) - 2, lane = threadIdx.x & 31;
  SkelGroup<NC>& sg = sm.g[group];
  const int before = (int)((ch / K::NG) * nc);                          // of this group's earlier chunks
  const int* ahead = ch > 0 ? &sm.g[(group + K::NG - 1) % K::NG].done : nullptr;
  const int ahead0 = ch > 0 ? (int)(((ch - 1) / K::NG) * nc) : 0;
  auto publish = [&](int j) {
    if (k == j) {
#pragma unroll
      for (int t = 0; t < K::OWN; ++t) sg.col[q + K::LPC * t] = c[t];
      if (q == 0) sg.alpha = sm.R[j + j * (NC + 1)];
    }
  };
  auto group_sync = [&]() {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(K::GROUP) : "memory");
  };
  // rows 0 .. j of R are the chunk's own from here on
  auto follow = [&](int j) {
    if (ahead && threadIdx.x % K::GROUP == 0) {
      wait_group(ahead, ahead0 + min(j + 1, nc), &sm.late);
      __threadfence_block();
    }
  };
  follow(1);
  group_sync();
  if (w >= 0) publish(0);
  group_sync();
  if (w < 0) make_reflector<NC>(sg, sm.R, 0, w + 2, lane);
  group_sync();
  for (int j = 0; j < nc; ++j) {
    if (w < 0) {
      if (j + 1 < nc) {
        __syncwarp();
        asm volatile("bar.sync %0, 96;" ::"r"(1 + K::NG + group) : "memory");
        make_reflector<NC>(sg, sm.R, j + 1, w + 2, lane);
      }
      follow(j + 2);
    } else if (K::CPW * (w + 1) - 1 > j && K::CPW * w < nc) {
      if (sg.go[j & 1]) {
        const bool active = k > j && k < nc;
        const double tau = sg.tau[j & 1];
        double* r = sm.R + j + (active ? k : j) * (NC + 1);
        const double rv = *r;               // before the shuffles: the column's first lane changes it after them
        const double2* v = reinterpret_cast<const double2*>(sg.v[j & 1] + q * K::OWN);
        double p[K::OWN];
#pragma unroll
        for (int t = 0; t < K::OWN / 2; ++t) {
          const double2 x = v[t];
          p[2 * t] = __dmul_rn(x.x, c[2 * t]);
          p[2 * t + 1] = __dmul_rn(x.y, c[2 * t + 1]);
        }
#pragma unroll
        for (int h = K::OWN / 2; h > 0; h >>= 1)
#pragma unroll
          for (int t = 0; t < h; ++t) p[t] = __dadd_rn(p[t], p[t + h]);
        double s = p[0];
#pragma unroll
        for (int o = K::LPC / 2; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
        if (active) {
          const double wk = __dmul_rn(tau, __dadd_rn(rv, s));
          if (q == 0) *r = __dsub_rn(rv, wk);
#pragma unroll
          for (int t = 0; t < K::OWN / 2; ++t) {
            const double2 x = v[t];
            c[2 * t] = __fma_rn(-wk, x.x, c[2 * t]);
            c[2 * t + 1] = __fma_rn(-wk, x.y, c[2 * t + 1]);
          }
        }
      }
      if (j + 1 < nc && (j + 1) / K::CPW == w) {
        __syncwarp();
        publish(j + 1);
        __syncwarp();
        asm volatile("bar.arrive %0, 96;" ::"r"(1 + K::NG + group) : "memory");
      }
    }
    group_sync();
    if (threadIdx.x % K::GROUP == 0) {
      __threadfence_block();
      *(volatile int*)&sg.done = before + j + 1;
    }
  }
}

// One CTA per cluster of the level.
//   cand   [ncl][SK_CAND]: candidate tree positions, ncand[ncl] of them
//   samp   sampled tree positions of all clusters, cluster c at samp[soff[c] .. soff[c+1])
//   out:   skel[ncl][64] (tree positions, pivot order), rank[ncl], T[ncl][SK_CAND x 64]
//          (rows = candidates in their original order, column-major, ld SK_CAND)
template <int NC>
__global__ void __launch_bounds__(Skel<NC>::THREADS)
    k_skeletonize(const int* __restrict__ cand, const int* __restrict__ ncand, const int* __restrict__ samp,
                  const int64_t* __restrict__ soff, const double* __restrict__ X, const double* __restrict__ sw,
                  int dim, KernelParams kp, double tol, int rank_max, int* __restrict__ skel,
                  int* __restrict__ rank_out, double* __restrict__ Tout, int* __restrict__ late) {
  extern __shared__ __align__(16) unsigned char dsm[];
  SkelSmem<NC>& sm = *reinterpret_cast<SkelSmem<NC>*>(dsm);
  constexpr int LD = NC + 1;
  double* R = sm.R;
  double* nrm = sm.nrm;
  double* red = sm.red;
  double* bcast = sm.bcast;
  int* piv = sm.piv;
  int* ired = sm.ired;
  const int c = blockIdx.x;
  const int nc = ncand[c];
  const int* cd = cand + (int64_t)c * SK_CAND;
  using K = Skel<NC>;
  const int group = threadIdx.x / K::GROUP;
  const int own = (int)(threadIdx.x % K::GROUP) - 64;      // the group's first two warps own no column
  const int k = own >= 0 ? own / K::LPC : NC, q = own & (K::LPC - 1);
  const int64_t s0 = soff[c], s1 = soff[c + 1];
  const int64_t m = s1 - s0;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) piv[i] = i;
  for (int i = threadIdx.x; i < NC * LD; i += blockDim.x) R[i] = 0.0;
  if (threadIdx.x < K::NG) sm.g[threadIdx.x].done = 0;
  if (threadIdx.x == 0) sm.late = 0;
  __syncthreads();
  int r = 0;
  if (m > 0 && nc > 0) {
    // ---- 2. tall-skinny QR of the sampled rows
    double cc[K::OWN];
    double x[3] = {0.0, 0.0, 0.0}, wk = 0.0;
    if (k < nc) {
      const int p = cd[k];
      for (int d = 0; d < dim; ++d) x[d] = X[(int64_t)p * dim + d];
      wk = sw[p];
    }
    double* stage = sm.g[group].stage + max(own, 0);
    for (int64_t ch = group; ch * SK_CHUNK < m; ch += K::NG) {
      const int64_t row0 = ch * SK_CHUNK + q;
#pragma unroll
      for (int f0 = 0; f0 < K::OWN; f0 += K::FILL) {
#pragma unroll 1
        for (int t = 0; t < K::FILL; ++t) {
          const int64_t row = row0 + K::LPC * (f0 + t);
          double v = 0.0;
          if (k < nc && row < m) {
            const int f = samp[s0 + row];
            v = sw[f] * kernel_eval(kp, X + (int64_t)f * dim, x, dim) * wk;
          }
          if (own >= 0) stage[t * NC * K::LPC] = v;        // read back by this thread alone
        }
#pragma unroll
        for (int t = 0; t < K::FILL; ++t) cc[f0 + t] = own >= 0 ? stage[t * NC * K::LPC] : 0.0;
      }
      fold_chunk<NC>(sm, nc, ch, group, k, q, cc);
    }
    __syncthreads();
    if (sm.late && threadIdx.x == 0) atomicExch(late, 1);
    // ---- 3. greedy column-pivoted Householder QR of R0 (rows: min(m, nc))
    const int rows = (int)(m < nc ? m : nc);
    const int kmax = min(rank_max, min(rows, nc));
    double first = 0.0;
    for (int j = 0; j < kmax; ++j) {
      for (int k = j + threadIdx.x; k < nc; k += blockDim.x) {
        double s = R[j + k * LD] * R[j + k * LD], below = 0.0;
        for (int i = j + 1; i < nc; ++i) {
          s = fma(R[i + k * LD], R[i + k * LD], s);
          below = fma(R[i + k * LD], R[i + k * LD], below);
        }
        nrm[k] = s;
        sm.sig[k] = below;
      }
      __syncthreads();
      double mv = -1.0;
      for (int k = j + threadIdx.x; k < nc; k += blockDim.x) mv = fmax(mv, nrm[k]);
      const double big = block_max(mv, red);
      if (j == 0) {
        first = sqrt(big);
        if (first == 0.0) break;
      } else if (sqrt(big) <= tol * first) {
        break;
      }
      int cand_k = 1 << 30;
      for (int k = j + threadIdx.x; k < nc; k += blockDim.x)
        if (nrm[k] >= big * (1.0 - SK_TIE)) cand_k = min(cand_k, k);
      const int p = block_min_int(cand_k, ired);
      if (p != j) {
        for (int i = threadIdx.x; i < nc; i += blockDim.x) {
          const double t = R[i + j * LD];
          R[i + j * LD] = R[i + p * LD];
          R[i + p * LD] = t;
        }
        if (threadIdx.x == 0) {
          const int t = piv[j];
          piv[j] = piv[p];
          piv[p] = t;
        }
        __syncthreads();
      }
      // reflector of R[j:, j]
      if (threadIdx.x == 0) {
        const double alpha = R[j + j * LD], sigma = sm.sig[p];
        double beta = alpha, tau = 0.0, scale = 0.0;
        if (sigma > 0.0) {
          beta = -copysign(sqrt(alpha * alpha + sigma), alpha);
          tau = (beta - alpha) / beta;
          scale = 1.0 / (alpha - beta);
        }
        bcast[0] = beta;
        bcast[1] = tau;
        bcast[2] = scale;
      }
      __syncthreads();
      const double beta = bcast[0], tau = bcast[1], scale = bcast[2];
      if (tau != 0.0) {
        for (int i = j + 1 + threadIdx.x; i < nc; i += blockDim.x) R[i + j * LD] *= scale;
        __syncthreads();
        for (int k = j + 1 + threadIdx.x; k < nc; k += blockDim.x) {
          double wk = R[j + k * LD];
          for (int i = j + 1; i < nc; ++i) wk = fma(R[i + j * LD], R[i + k * LD], wk);
          wk *= tau;
          R[j + k * LD] -= wk;
          for (int i = j + 1; i < nc; ++i) R[i + k * LD] = fma(-wk, R[i + j * LD], R[i + k * LD]);
        }
        __syncthreads();
        if (threadIdx.x == 0) R[j + j * LD] = beta;
        for (int i = j + 1 + threadIdx.x; i < nc; i += blockDim.x) R[i + j * LD] = 0.0;
      }
      __syncthreads();
      r = j + 1;
    }
    r = max(r, 1);
    // ---- 4. R11^{-1} R12 by back substitution, one thread per column of R12
    if (R[0] != 0.0) {
      for (int b = r + threadIdx.x; b < nc; b += blockDim.x) {
        for (int a = r - 1; a >= 0; --a) {
          double v = R[a + b * LD];
          for (int a2 = a + 1; a2 < r; ++a2) v = fma(-R[a + a2 * LD], R[a2 + b * LD], v);
          R[a + b * LD] = v / R[a + a * LD];
        }
      }
    } else {
      for (int b = r + threadIdx.x; b < nc; b += blockDim.x)
        for (int a = 0; a < r; ++a) R[a + b * LD] = 0.0;
    }
    __syncthreads();
  } else {
    r = min(nc, rank_max);   // empty sample: the first candidates, T = [I; 0]
  }
  // ---- outputs
  double* Tc = Tout + (int64_t)c * SK_CAND * 64;
  for (int e = threadIdx.x; e < SK_CAND * 64; e += blockDim.x) Tc[e] = 0.0;
  __syncthreads();
  const bool id = (m > 0 && nc > 0);
  for (int e = threadIdx.x; e < nc * r; e += blockDim.x) {
    const int k = e % nc, a = e / nc;   // pivot position k, column a
    double v;
    if (k < r) v = (k == a) ? 1.0 : 0.0;
    else v = id ? R[a + k * LD] : 0.0;
    Tc[piv[k] + a * SK_CAND] = v;
  }
  for (int a = threadIdx.x; a < 64; a += blockDim.x) skel[(int64_t)c * 64 + a] = a < r ? cd[piv[a]] : -1;
  if (threadIdx.x == 0) rank_out[c] = r;
}

// Candidates of the clusters of level ell (< L): the skeleton of child 2j, then that
// of child 2j + 1 (ranks rk of level ell + 1).
__global__ void k_skel_cand(const int* __restrict__ skel_child, const int* __restrict__ rk_child, int ncl,
                            int* __restrict__ cand, int* __restrict__ ncand) {
  const int j = blockIdx.x;
  if (j >= ncl) return;
  const int r1 = rk_child[2 * j], r2 = rk_child[2 * j + 1];
  for (int i = threadIdx.x; i < r1 + r2; i += blockDim.x)
    cand[(int64_t)j * SK_CAND + i] =
        i < r1 ? skel_child[(int64_t)(2 * j) * 64 + i] : skel_child[(int64_t)(2 * j + 1) * 64 + i - r1];
  if (threadIdx.x == 0) ncand[j] = r1 + r2;
}

// Candidates of the leaves: their points in tree order.
__global__ void k_skel_cand_leaf(const int* __restrict__ leafoff, int* __restrict__ cand, int* __restrict__ ncand) {
  const int j = blockIdx.x;
  const int p0 = leafoff[j], nl = leafoff[j + 1] - p0;
  for (int i = threadIdx.x; i < nl; i += blockDim.x) cand[(int64_t)j * SK_CAND + i] = p0 + i;
  if (threadIdx.x == 0) ncand[j] = nl;
}

// Sample positions of every cluster, from a list of (destination offset, source
// cluster, kind) segments: kind 0 = all candidates of cluster src; kind s >= 1 = the
// candidates of clusters 2 src and 2 src + 1 concatenated, every s-th from the first.
struct SampleSeg {
  int64_t dst;
  int src;
  int kind;
};
__global__ void k_skel_samples(const SampleSeg* __restrict__ seg, int nseg, const int* __restrict__ cand,
                               const int* __restrict__ ncand, int* __restrict__ samp) {
  const int g = blockIdx.x;
  if (g >= nseg) return;
  const SampleSeg S = seg[g];
  if (S.kind == 0) {
    const int nn = ncand[S.src];
    for (int i = threadIdx.x; i < nn; i += blockDim.x) samp[S.dst + i] = cand[(int64_t)S.src * SK_CAND + i];
  } else {
    const int a = 2 * S.src, b = 2 * S.src + 1;
    const int na = ncand[a], nb = ncand[b];
    const int cnt = (na + nb + S.kind - 1) / S.kind;
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
      const int k = i * S.kind;
      samp[S.dst + i] = k < na ? cand[(int64_t)a * SK_CAND + k] : cand[(int64_t)b * SK_CAND + k - na];
    }
  }
}

// Skeleton coordinates and sqrt(w) of every slot (the coupling points of k_fill_S).
__global__ void k_skel_nodes(const int* __restrict__ skel, const int* __restrict__ rank, int nsl, int KC, int dim,
                             const double* __restrict__ X, const double* __restrict__ sw, double* __restrict__ nodes,
                             double* __restrict__ nsw) {
  const int t = blockIdx.x;
  if (t >= nsl) return;
  const int r = rank[t];
  for (int a = threadIdx.x; a < KC; a += blockDim.x) {
    const int p = a < r ? skel[(int64_t)t * 64 + a] : -1;
    for (int d = 0; d < dim; ++d) nodes[((int64_t)t * KC + a) * dim + d] = p >= 0 ? X[(int64_t)p * dim + d] : 0.0;
    nsw[(int64_t)t * KC + a] = p >= 0 ? sw[p] : 0.0;
  }
}

template <int NC>
static void skeletonize_level(Matrix& M, int ncl, const int* cand, const int* ncand, const int* samp,
                              const int64_t* soff, int* skel, int* rank, double* T) {
  const int smem = (int)sizeof(SkelSmem<NC>);
  H2_CUDA(cudaFuncSetAttribute(k_skeletonize<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  { k_skeletonize<NC><<<ncl, Skel<NC>::THREADS, smem, M.stream>>>(cand, ncand, samp, soff, M.d_X, M.d_sw, M.dim, M.kp,
                                                                  M.basis_tol, M.k, skel, rank, T, M.d_flag + 2);
    ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
}

// Skeletons of every cluster at levels t*..L, bottom-up, into M.d_skel (slot-indexed,
// 64 per slot), M.d_Tid (slot-indexed, SK_CAND x 64) and M.h_rank / M.d_rank.
void build_skeletons(Matrix& M) {
  cudaStream_t s = M.stream;
  const int L = M.L, ts = M.tstar;
  const int nsl = M.nslots();
  M.d_skel = (int*)M.alloc(sizeof(int) * (size_t)nsl * 64);
  M.tid.bytes = sizeof(double) * (size_t)nsl * SK_CAND * 64;
  M.tid.p = M.alloc(M.tid.bytes);
  M.h_rank.assign(nsl, 0);
  M.d_rank = (int*)M.alloc(sizeof(int) * nsl);
  // candidates of two consecutive levels (this one and the one below)
  std::vector<int> ncand_h;                      // of level ell
  int* d_cand = (int*)M.alloc(sizeof(int) * ((size_t)1 << L) * SK_CAND);
  int* d_ncand = (int*)M.alloc(sizeof(int) * ((size_t)1 << L));
  H2_CUDA(cudaMemsetAsync(M.d_flag + 2, 0, sizeof(int), s));
  for (int ell = L; ell >= ts; --ell) {
    const int ncl = 1 << ell;
    if (ell == L) {
      { k_skel_cand_leaf<<<ncl, 64, 0, s>>>(M.d_leafoff, d_cand, d_ncand); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      ncand_h.assign(ncl, 0);
      for (int j = 0; j < ncl; ++j) ncand_h[j] = M.offsets[L][j + 1] - M.offsets[L][j];
    } else {
      { k_skel_cand<<<ncl, 128, 0, s>>>(M.d_skel + (size_t)M.slot0(ell + 1) * 64, M.d_rank + M.slot0(ell + 1), ncl,
                                        d_cand, d_ncand); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      ncand_h.assign(ncl, 0);
      for (int j = 0; j < ncl; ++j)
        ncand_h[j] = M.h_rank[M.slot0(ell + 1) + 2 * j] + M.h_rank[M.slot0(ell + 1) + 2 * j + 1];
    }
    // sample segments: own far partners, then the parent's far partners (thinned)
    std::vector<SampleSeg> segs;
    std::vector<int64_t> soff(ncl + 1, 0);
    const HostCSR& F = M.far[ell];
    const HostCSR* Fp = (ell - 1 >= ts) ? &M.far[ell - 1] : nullptr;
    int64_t tot = 0;
    for (int j = 0; j < ncl; ++j) {
      soff[j] = tot;
      for (int e = F.rowptr[j]; e < F.rowptr[j + 1]; ++e) {
        const int sg = F.col[e];
        segs.push_back({tot, sg, 0});
        tot += ncand_h[sg];
      }
      if (Fp) {
        const int pj = j >> 1;
        for (int e = Fp->rowptr[pj]; e < Fp->rowptr[pj + 1]; ++e) {
          const int sg = Fp->col[e];
          const int cnt = ncand_h[2 * sg] + ncand_h[2 * sg + 1];
          const int step = std::max(1, (cnt + SK_SAMPLE_CAP - 1) / SK_SAMPLE_CAP);
          segs.push_back({tot, sg, step});
          tot += (cnt + step - 1) / step;
        }
      }
    }
    soff[ncl] = tot;
    int* d_samp = (int*)M.alloc(sizeof(int) * std::max<int64_t>(tot, 1));
    int64_t* d_soff = (int64_t*)M.alloc(sizeof(int64_t) * (ncl + 1));
    SampleSeg* d_seg = (SampleSeg*)M.alloc(sizeof(SampleSeg) * std::max<size_t>(segs.size(), 1));
    H2_CUDA(cudaMemcpyAsync(d_soff, soff.data(), sizeof(int64_t) * (ncl + 1), cudaMemcpyHostToDevice, s));
    if (!segs.empty()) {
      H2_CUDA(cudaMemcpyAsync(d_seg, segs.data(), sizeof(SampleSeg) * segs.size(), cudaMemcpyHostToDevice, s));
      const int64_t CH = 1 << 20;
      for (int64_t g0 = 0; g0 < (int64_t)segs.size(); g0 += CH) {
        const int ng = (int)std::min<int64_t>(CH, (int64_t)segs.size() - g0);
        { k_skel_samples<<<ng, 128, 0, s>>>(d_seg + g0, ng, d_cand, d_ncand, d_samp); ::h2mg::count_launch(); }
        H2_LAUNCH_CHECK();
      }
    }
    const int most = *std::max_element(ncand_h.begin(), ncand_h.end());
    (most <= 64 ? skeletonize_level<64> : skeletonize_level<SK_CAND>)(
        M, ncl, d_cand, d_ncand, d_samp, d_soff, M.d_skel + (size_t)M.slot0(ell) * 64, M.d_rank + M.slot0(ell),
        (double*)M.tid.p + (size_t)M.slot0(ell) * SK_CAND * 64);
    H2_CUDA(cudaMemcpyAsync(M.h_rank.data() + M.slot0(ell), M.d_rank + M.slot0(ell), sizeof(int) * ncl,
                            cudaMemcpyDeviceToHost, s));
    int late = 0;
    H2_CUDA(cudaMemcpyAsync(&late, M.d_flag + 2, sizeof(int), cudaMemcpyDeviceToHost, s));
    H2_CUDA(cudaStreamSynchronize(s));
    H2_REQUIRE(late == 0, H2MG_ERR_TIMEOUT, "a skeletonization timed out waiting for its warps");
    M.free_owned(d_samp);
    M.free_owned(d_soff);
    M.free_owned(d_seg);
  }
  M.free_owned(d_cand);
  M.free_owned(d_ncand);
  // coupling points: skeleton coordinates and sqrt(w), KC per slot
  M.d_nodes = (double*)M.alloc(sizeof(double) * (size_t)nsl * M.KC * M.dim);
  M.d_nsw = (double*)M.alloc(sizeof(double) * (size_t)nsl * M.KC);
  { k_skel_nodes<<<nsl, 64, 0, s>>>(M.d_skel, M.d_rank, nsl, M.KC, M.dim, M.d_X, M.d_sw, M.d_nodes, M.d_nsw);
    ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  H2_CUDA(cudaStreamSynchronize(s));
}

}  // namespace h2mg
