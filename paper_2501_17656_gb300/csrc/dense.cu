// dense.cu -- the coarsest operator A_l as a dense matrix, its Cholesky factor and
// the coarse solve e_l = dir_sol(A_l, r_l) (Sec. 3.3, Algorithm 1).
//
// A_l acts on the coefficients of tree level m = m(l). Its coupling part is the H2
// chain of levels t*..m expanded densely: G_{t*} holds the far blocks of level t*,
// G_{ell+1} = T_ell G_ell T_ell^T + (far blocks of level ell+1) with T_ell the
// block-diagonal orthonormal transfers, and A_l = G_m + P_l. For l = 1 (no far
// field, or a forced single level) A_1 = D + U_1 G_L U_1^T on the point slots.
// Padded slots (beyond a cluster's rank or a leaf's size) get a unit diagonal so
// the factor exists; they are zero in every right-hand side.
#include <algorithm>
#include <cmath>

#include "fx_tile.cuh"
#include "internal.h"

namespace h2mg {

__device__ void unswz_d(int pos, int K, int V, int& i, int& j) {
  int LPC = K / 8, CPP = 32 / LPC, P = 8 / V;
  int sub = pos % V;
  int lane = (pos / V) % 32;
  int tk = pos / (V * 32);
  int t = tk / P, k = tk % P;
  i = 8 * (lane % LPC) + k * V + sub;
  j = t * CPP + lane / LPC;
}

__device__ __forceinline__ double load_elem_d(const void* pool, int fmt, int64_t idx) {
  if (fmt == FMT_F64) return ((const double*)pool)[idx];
  if (fmt == FMT_DF) {
    float2 v = ((const float2*)pool)[idx];
    return (double)v.x + (double)v.y;
  }
  return (double)((const float*)pool)[idx];
}

// dense[t*K + i, s*K + j] += B_ts[i, j] (and the transpose for t != s)
__global__ void k_scatter(const int* __restrict__ pt, const int* __restrict__ ps,
                          const void* __restrict__ pool, int fmt, int K, double* __restrict__ G,
                          int64_t n) {
  int64_t b = blockIdx.x;
  int t = pt[b], s = ps[b];
  int V = fmt == FMT_F32 ? 4 : 2;
  for (int pos = threadIdx.x; pos < K * K; pos += blockDim.x) {
    int i, j;
    unswz_d(pos, K, V, i, j);
    double v = load_elem_d(pool, fmt, b * K * K + pos);
    int64_t r = (int64_t)t * K + i, c = (int64_t)s * K + j;
    G[r + c * n] += v;
    if (t != s) G[c + r * n] += v;
  }
}

// out block (a, a') = B_a G(p(a), p(a')) B_a'^T, B_a of size Ra x C (column-major),
// G of order nc = 2^ell * C, out of order no = 2^(ell+1) * Ra.
__global__ void k_expand(const double* __restrict__ G, int64_t nc, const double* __restrict__ B,
                         int Ra, int C, int ncl_out, int shift, double* __restrict__ out, int64_t no) {
  extern __shared__ double sm[];
  double* Gb = sm;            // C x C
  double* T = Gb + C * C;     // C x Ra
  int a = blockIdx.x % ncl_out, ap = blockIdx.x / ncl_out;
  int pa = a >> shift, pap = ap >> shift;   // shift 1: parent cluster; 0: same cluster
  for (int e = threadIdx.x; e < C * C; e += blockDim.x) {
    int i = e % C, j = e / C;
    Gb[e] = G[((int64_t)pa * C + i) + ((int64_t)pap * C + j) * nc];
  }
  __syncthreads();
  const double* Ba = B + (int64_t)a * Ra * C;
  const double* Bap = B + (int64_t)ap * Ra * C;
  // T[b][j] = sum_c Gb[b][c] Bap[j][c]
  for (int e = threadIdx.x; e < C * Ra; e += blockDim.x) {
    int bb = e % C, j = e / C;
    double v = 0.0;
    for (int c = 0; c < C; ++c) v += Gb[bb + c * C] * Bap[j + c * Ra];
    T[e] = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < Ra * Ra; e += blockDim.x) {
    int i = e % Ra, j = e / Ra;
    double v = 0.0;
    for (int bb = 0; bb < C; ++bb) v += Ba[i + bb * Ra] * T[bb + j * C];
    out[((int64_t)a * Ra + i) + ((int64_t)ap * Ra + j) * no] = v;
  }
}

// k_expand for 64 x 64 blocks, tile (a, ap <= a) per CTA: the other half of the symmetric
// result is its mirror image. Two products of 64 x 64 matrices per tile on the integer pipe
// (fx_tile.cuh), 35 k clocks of an SM each with loads and encoding; on the float64 pipe, and
// for both halves, it was bound by 131 k clocks each: order 4096 took 3.62 ms, now 0.48 ms.
__global__ void __launch_bounds__(256, 2) k_expand64(const double* __restrict__ G, int64_t nc,
                                                     const double* __restrict__ B, int shift,
                                                     double* __restrict__ out, int64_t no) {
  extern __shared__ __align__(16) unsigned char dsm[];
  int a = 0, ap = blockIdx.x;
  while (ap > a) {
    ap -= a + 1;
    ++a;
  }
  const double* Gb = G + (int64_t)(a >> shift) * FXT + (int64_t)(ap >> shift) * FXT * nc;
  const double* Ba = B + (int64_t)a * FXT * FXT;
  const double* Bap = B + (int64_t)ap * FXT * FXT;
  FxPair t(dsm);
  FxAcc c;
  double v[4][4];
  // T = G B_ap^T
  fx_tile_load(t.P, t.ep, [&](int b, int k) { return Gb[b + k * nc]; });
  fx_tile_load(t.Q, t.eq, [&](int j, int k) { return Bap[j + k * FXT]; });
  __syncthreads();
  c.clear();
  fx_tile_mma(t, c);
  fx_values(t, c, v);
  __syncthreads();
  // B_a T
  fx_tile_store_q(t.Q, t.eq, v);
  fx_tile_load(t.P, t.ep, [&](int i, int b) { return Ba[i + b * FXT]; });
  __syncthreads();
  c.clear();
  fx_tile_mma(t, c);
  fx_values(t, c, v);
  __syncthreads();
  double* S = (double*)dsm;
  const int64_t a0 = (int64_t)a * FXT, ap0 = (int64_t)ap * FXT;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = fx_a() + r, j = fx_b() + 16 * q;
      if (a != ap) out[ap0 + j + (a0 + i) * no] = v[r][q];
      S[i + j * FXLD] = v[r][q];
    }
  __syncthreads();
  for (int e = threadIdx.x; e < FXT * FXT; e += blockDim.x) {
    const int i = e & 63, j = e >> 6;
    out[a0 + i + (ap0 + j) * no] = a == ap && i < j ? S[j + i * FXLD] : S[i + j * FXLD];
  }
}

__global__ void k_pad_diag(double* __restrict__ A, int64_t n, const unsigned char* __restrict__ valid) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && !valid[i]) A[i + i * n] = 1.0;
}

// ----------------------------------------------------------------------------- scaling
// Powers of two s_i that bring the diagonal of s A_l s into [1, 4). A float64 Cholesky does
// not depend on such a scaling; the blocked one does: a tile row has one exponent, and with
// rows of widely different size (weights over many decades) the entries of L_kk^-1 go with
// 1 / d_m and those of A_bk with d_m along the sum index m, so that each loses the digits
// that the other needs. Scaled exactly, 2 n^2 multiplications beside n^3 / 2.
__global__ void k_diag_scale(const double* __restrict__ A, int64_t n, double* __restrict__ sc) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double d = A[i + i * n];
  sc[i] = d > 0.0 && isfinite(d) ? ldexp(1.0, -(ilogb(d) >> 1)) : 1.0;
}

__global__ void k_scale_sym(const double* __restrict__ A, int64_t n, const double* __restrict__ sc,
                            double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int64_t j = blockIdx.y; j < n; j += gridDim.y) out[i + j * n] = A[i + j * n] * sc[i] * sc[j];
}

// ----------------------------------------------------------------------------- factor and inverse
// A_l = L L^T, X = L^-1 and A_l^-1 = X^T X by 64 x 64 blocks, all three with n^3 / 6 FMAs.
// Step k of one sweep over the block columns finishes L's column k and X's row k, then
// updates every block below: A_ij -= L_ik L_jk^T for k < j <= i and, on the rows of the
// forward substitution L X = I (zero at the start), B_ij -= L_ik X_kj for j <= k. The
// products run on the integer pipe (fx_tile.cuh); the 64 x 64 diagonal block is factored and
// inverted in float64 by the CTA that updates it first, beside the rest of its step.
// X and B are stored transposed, so that every tile is read along consecutive addresses.
//
// n^3 / 2 FMAs are 5 ms of integer multiply-adds for n = 4096 at the instruction's own 63 per
// clock and SM, and 55 ms on the float64 pipe. Measured for n = 4096: 21.7 ms (updates 14.7,
// inverse 5.3, panels 1.5), before 180 ms (32-column panels with unblocked substitution, and
// an inverse from two dense triangular solves). A tile takes 40 k clocks of an SM, 12 k of
// them multiply-adds at that rate: issue slots and the ALU pipe are 45 % busy, the FMA pipe
// 21 %, with 16 warps that wait for one another's operands (dispatch and fixed latencies).
constexpr int DB = FXT;                                     // block edge
constexpr size_t DENSE_SMEM = FX_PAIR_BYTES;

// Cholesky factor of the lower triangle of S (64 x 64, column-major, ld FXLD; rows from nb
// on are a unit diagonal) and the inverse X of the factor. 256 threads.
__device__ void factor_diag(double* S, double* X, double* dg, int nb, int* flag) {
  const int tid = threadIdx.x;
  for (int j = 0; j < DB; ++j) {
    if (tid < DB) {
      double d = S[j + j * FXLD];
      if (!(d > 0.0)) {
        if (tid == 0 && j < nb) atomicOr(flag, 1);
        d = 1.0;
      }
      const double l = sqrt(d);
      if (tid == j) dg[j] = l;
      if (tid > j) S[tid + j * FXLD] /= l;
    }
    __syncthreads();
    const int i = tid & 63;
    const double lij = S[i + j * FXLD];
    for (int c = j + 1 + (tid >> 6); c <= i; c += 4) S[i + c * FXLD] = fma(-lij, S[c + j * FXLD], S[i + c * FXLD]);
    __syncthreads();
  }
  // rows of X = L^-1 in turn: four lanes per column
  const int c = tid >> 2, part = tid & 3;
  for (int i = 0; i < DB; ++i) {
    double s = 0.0;
    for (int m = part; m < i; m += 4) s = fma(S[i + m * FXLD], X[m + c * FXLD], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (part == 0) X[i + c * FXLD] = c > i ? 0.0 : ((c == i ? 1.0 : 0.0) - s) / dg[i];
    __syncthreads();
  }
}

// The diagonal block at k0, read from shared memory S: its factor's inverse goes to Li
// (column-major, 64 x 64).
__device__ void finish_diag(double* S, double* X, double* dg, int nb, int* flag, double* __restrict__ Li) {
  __syncthreads();
  factor_diag(S, X, dg, nb, flag);
  for (int e = threadIdx.x; e < DB * DB; e += blockDim.x) Li[e] = X[(e & 63) + (e >> 6) * FXLD];
}

__global__ void __launch_bounds__(256) k_chol_first(const double* __restrict__ A, int64_t n, int* __restrict__ flag,
                                                    double* __restrict__ Li) {
  extern __shared__ __align__(16) unsigned char dsm[];
  double* S = (double*)dsm;
  double* X = S + DB * FXLD;
  double* dg = X + DB * FXLD;
  const int nb = (int)min((int64_t)DB, n);
  for (int e = threadIdx.x; e < DB * DB; e += blockDim.x) {
    const int i = e & 63, j = e >> 6;
    S[i + j * FXLD] = i < n && j < n ? A[i + (int64_t)j * n] : (i == j ? 1.0 : 0.0);
  }
  finish_diag(S, X, dg, nb, flag, Li);
}

// Step k, first half: block b > k: L_bk = A_bk L_kk^-T; b < k: X_kb = L_kk^-1 B_kb; b = k:
// X_kk = L_kk^-1. XT holds X (and B) transposed.
__global__ void __launch_bounds__(256, 2) k_chol_panel(double* __restrict__ A, double* __restrict__ XT, int64_t n,
                                                       int k, const double* __restrict__ Li) {
  extern __shared__ __align__(16) unsigned char dsm[];
  const int b = blockIdx.x;
  const int64_t k0 = (int64_t)k * DB, b0 = (int64_t)b * DB;
  if (b == k) {
    for (int e = threadIdx.x; e < DB * DB; e += blockDim.x) {
      const int j = e & 63, m = e >> 6;
      if (k0 + j < n && k0 + m < n) XT[k0 + j + (k0 + m) * n] = Li[m + j * DB];
    }
    return;
  }
  FxPair t(dsm);
  double* M = b > k ? A : XT;
  fx_tile_load(t.P, t.ep, [&](int a, int m) { return Li[a + m * DB]; });
  fx_tile_load(t.Q, t.eq, [&](int i, int m) { return b0 + i < n && k0 + m < n ? M[b0 + i + (k0 + m) * n] : 0.0; });
  __syncthreads();
  FxAcc c;
  c.clear();
  fx_tile_mma(t, c);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t col = k0 + fx_a() + r, row = b0 + fx_b() + 16 * q;
      if (row < n && col < n) M[row + col * n] = fx_value(t, c, r, q);
    }
}

// Step k, second half: the updates of block row i > k, one tile (i, j <= i) per CTA; the
// first CTA takes tile (k + 1, k + 1) and factors it.
__global__ void __launch_bounds__(256, 2) k_chol_update(double* __restrict__ A, double* __restrict__ XT, int64_t n,
                                                        int k, int* __restrict__ flag, double* __restrict__ Li) {
  extern __shared__ __align__(16) unsigned char dsm[];
  const int first = k + 1;                                   // the first row has tiles 0 .. k + 1
  int idx = blockIdx.x == 0 ? first : (blockIdx.x == first ? 0 : blockIdx.x);
  int i = first, j = idx;
  while (j > i) {
    j -= i + 1;
    ++i;
  }
  const int64_t k0 = (int64_t)k * DB, i0 = (int64_t)i * DB, j0 = (int64_t)j * DB;
  const bool inv = j <= k;
  // tile (a, b): A^T's (column c of block j, row r of block i), or B^T's (row r, column c)
  const double* pm = A + (inv ? i0 : j0);
  const double* qm = inv ? XT + j0 : A + i0;
  const int64_t pn = n - (inv ? i0 : j0), qn = n - (inv ? j0 : i0);
  FxPair t(dsm);
  fx_tile_load(t.P, t.ep, [&](int a, int m) { return a < pn && k0 + m < n ? pm[a + (k0 + m) * n] : 0.0; });
  fx_tile_load(t.Q, t.eq, [&](int b, int m) { return b < qn && k0 + m < n ? qm[b + (k0 + m) * n] : 0.0; });
  __syncthreads();
  FxAcc c;
  c.clear();
  fx_tile_mma(t, c);
  double* out = inv ? XT + j0 + i0 * n : A + i0 + j0 * n;
  double v[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int a = fx_a() + r, b = fx_b() + 16 * q;
      v[r][q] = a == b ? 1.0 : 0.0;                          // rows past n: a unit diagonal
      if (a < pn && b < qn) {
        v[r][q] = out[b + a * n] - fx_value(t, c, r, q);
        out[b + a * n] = v[r][q];
      }
    }
  if (i == first && j == first) {
    double* S = (double*)dsm;
    double* X = S + DB * FXLD;
    double* dg = X + DB * FXLD;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) S[fx_b() + 16 * q + (fx_a() + r) * FXLD] = v[r][q];
    finish_diag(S, X, dg, (int)min((int64_t)DB, n - i0), flag, Li);
  }
}

// A_l^-1 = s X^T X s, tile (i, j <= i) per CTA: the sum over block rows m >= i of X_mi^T X_mj.
__global__ void __launch_bounds__(256, 2) k_chol_inverse(const double* __restrict__ XT, int64_t n, int blocks,
                                                         const double* __restrict__ sc, double* __restrict__ Ainv) {
  extern __shared__ __align__(16) unsigned char dsm[];
  int i = 0, j = blockIdx.x;
  while (j > i) {
    j -= i + 1;
    ++i;
  }
  const int64_t i0 = (int64_t)i * DB, j0 = (int64_t)j * DB;
  FxPair t(dsm);
  double s[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) s[r][q] = 0.0;
  for (int m = i; m < blocks; ++m) {
    const int64_t m0 = (int64_t)m * DB;
    fx_tile_load(t.P, t.ep, [&](int a, int k) { return j0 + a < n && m0 + k < n ? XT[j0 + a + (m0 + k) * n] : 0.0; });
    fx_tile_load(t.Q, t.eq, [&](int b, int k) { return i0 + b < n && m0 + k < n ? XT[i0 + b + (m0 + k) * n] : 0.0; });
    __syncthreads();
    FxAcc c;
    c.clear();
    fx_tile_mma(t, c);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) s[r][q] += fx_value(t, c, r, q);
    __syncthreads();
  }
  double* S = (double*)dsm;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int a = fx_a() + r, b = fx_b() + 16 * q;
      if (j0 + a < n && i0 + b < n) {
        s[r][q] = s[r][q] * sc[j0 + a] * sc[i0 + b];
        Ainv[i0 + b + (j0 + a) * n] = s[r][q];
      }
      S[a + b * FXLD] = s[r][q];
    }
  if (i == j) return;
  __syncthreads();
  for (int e = threadIdx.x; e < DB * DB; e += blockDim.x) {
    const int a = e & 63, b = e >> 6;
    if (j0 + a < n && i0 + b < n) Ainv[j0 + a + (i0 + b) * n] = S[a + b * FXLD];
  }
}

// out[:, c] = base[:, c] + sign A[:, :] v[:, c] (base null: 0) for NR columns (leading
// dimension n) and a symmetric A: one warp per output row reads that column of A once for
// all NR columns. base may be out.
template <int NR>
__global__ void k_symv_multi(const double* __restrict__ A, int64_t n, const double* v, const double* base,
                             double sign, double* out) {
  chain_wait();
  int64_t i = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (i >= n) return;
  const double* col = A + i * n;
  double s[NR];
#pragma unroll
  for (int c = 0; c < NR; ++c) s[c] = 0.0;
  for (int64_t j = lane; j < n; j += 32) {
    const double a = col[j];
#pragma unroll
    for (int c = 0; c < NR; ++c) s[c] = fma(a, v[c * n + j], s[c]);
  }
#pragma unroll
  for (int c = 0; c < NR; ++c) {
    for (int o = 16; o > 0; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
    if (lane == 0) out[c * n + i] = fma(sign, s[c], base ? base[c * n + i] : 0.0);
  }
}

// Factors a scaled copy of A_l (d_Al) and, if it is positive definite, leaves the inverse there.
static void factor_and_invert(Matrix& M) {
  cudaStream_t s = M.stream;
  const int64_t n = M.nl;
  const int blocks = ceil_div(n, DB);
  H2_CUDA(cudaFuncSetAttribute(k_chol_first, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM));
  H2_CUDA(cudaFuncSetAttribute(k_chol_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM));
  H2_CUDA(cudaFuncSetAttribute(k_chol_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM));
  H2_CUDA(cudaFuncSetAttribute(k_chol_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM));
  double* F = (double*)M.alloc(sizeof(double) * n * n);
  double* XT = (double*)M.alloc(sizeof(double) * n * n);
  double* Li = (double*)M.alloc(sizeof(double) * DB * DB);
  double* sc = (double*)M.alloc(sizeof(double) * n);
  { k_diag_scale<<<ceil_div(n, 256), 256, 0, s>>>(M.d_Al, n, sc); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  { k_scale_sym<<<dim3(ceil_div(n, 256), (unsigned)std::min<int64_t>(n, 4096)), 256, 0, s>>>(M.d_Al, n, sc, F); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  H2_CUDA(cudaMemsetAsync(M.d_flag, 0, sizeof(int), s));
  { k_chol_first<<<1, 256, DENSE_SMEM, s>>>(F, n, M.d_flag, Li); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  for (int k = 0; k < blocks; ++k) {
    { k_chol_panel<<<blocks, 256, DENSE_SMEM, s>>>(F, XT, n, k, Li); ::h2mg::count_launch(); }
    H2_LAUNCH_CHECK();
    const int64_t tiles = (int64_t)blocks * (blocks + 1) / 2 - (int64_t)(k + 1) * (k + 2) / 2;
    if (tiles > 0) {
      { k_chol_update<<<(int)tiles, 256, DENSE_SMEM, s>>>(F, XT, n, k, M.d_flag, Li); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
    }
  }
  int flag = 0;
  H2_CUDA(cudaMemcpyAsync(&flag, M.d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  H2_CUDA(cudaStreamSynchronize(s));
  M.coarse_ok = (flag == 0);
  if (M.coarse_ok) {
    { k_chol_inverse<<<blocks * (blocks + 1) / 2, 256, DENSE_SMEM, s>>>(XT, n, blocks, sc, F); ::h2mg::count_launch(); }
    H2_LAUNCH_CHECK();
    M.d_Ainv = F;
  } else {
    M.free_owned(F);
  }
  M.free_owned(XT);
  M.free_owned(Li);
  M.free_owned(sc);
}

static void upload_i32(Matrix& M, const std::vector<int>& v, int** d) {
  *d = (int*)M.alloc(sizeof(int) * std::max<size_t>(v.size(), 1));
  if (!v.empty()) H2_CUDA(cudaMemcpyAsync(*d, v.data(), sizeof(int) * v.size(), cudaMemcpyHostToDevice, M.stream));
}

// Scatter the upper entries of a full level list (strict: far lists) from a pool.
static void scatter_level(Matrix& M, const HostCSR& C, int ncl, bool strict, const void* pool,
                          int64_t blk0, int K, double* G, int64_t n) {
  std::vector<int> pt, ps;
  for (int t = 0; t < ncl; ++t)
    for (int e = C.rowptr[t]; e < C.rowptr[t + 1]; ++e)
      if (strict ? C.col[e] > t : C.col[e] >= t) {
        pt.push_back(t);
        ps.push_back(C.col[e]);
      }
  if (pt.empty()) return;
  int *dt, *ds;
  upload_i32(M, pt, &dt);
  upload_i32(M, ps, &ds);
  const char* base = (const char*)pool + (size_t)blk0 * K * K * fmt_bytes(M.fmt);
  { k_scatter<<<(int)pt.size(), 256, 0, M.stream>>>(dt, ds, base, M.fmt, K, G, n); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
}

// One step of the chain: every block of `out` from its block of G. `spread`: clusters whose
// rows have widely different scales are among them (mark_spread).
static void expand(const double* G, int64_t ng, const double* B, int Ra, int C, int ncl, int shift, bool spread,
                   double* out, int64_t no, cudaStream_t s) {
  if (Ra == FXT && C == FXT && !spread) {
    H2_CUDA(cudaFuncSetAttribute(k_expand64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM));
    { k_expand64<<<ncl * (ncl + 1) / 2, 256, DENSE_SMEM, s>>>(G, ng, B, shift, out, no); ::h2mg::count_launch(); }
  } else {
    const size_t sm = sizeof(double) * ((size_t)C * C + C * Ra);
    H2_CUDA(cudaFuncSetAttribute(k_expand, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    { k_expand<<<ncl * ncl, 256, sm, s>>>(G, ng, B, Ra, C, ncl, shift, out, no); ::h2mg::count_launch(); }
  }
  H2_LAUNCH_CHECK();
}

void build_dense_coarse(Matrix& M) {
  cudaStream_t s = M.stream;
  const int L = M.L, KC = M.KC, KD = M.KD;
  const int l = M.lev;
  double* G = nullptr;
  int64_t ng = 0;
  int mtop = (l == 1) ? L : L - l + 2;   // tree level whose coefficients the chain reaches
  if (M.tstar >= 0) {
    int ts = M.tstar;
    ng = (int64_t)(1 << ts) * KC;
    G = (double*)M.alloc(sizeof(double) * ng * ng);
    scatter_level(M, M.far[ts], 1 << ts, true, M.poolS.p, M.s_level_base[ts], KC, G, ng);
    for (int ell = ts; ell < mtop; ++ell) {
      int64_t nn = (int64_t)(1 << (ell + 1)) * KC;
      double* G2 = (double*)M.alloc(sizeof(double) * nn * nn);
      int ncl = 1 << (ell + 1);
      expand(G, ng, M.d_E + (size_t)M.slot0(ell + 1) * KC * KC, KC, KC, ncl, 1,
             level_spread(M, ell) || level_spread(M, ell + 1), G2, nn, s);
      scatter_level(M, M.far[ell + 1], ncl, true, M.poolS.p, M.s_level_base[ell + 1], KC, G2, nn);
      H2_CUDA(cudaStreamSynchronize(s));
      cudaFree(G);   // intermediate levels are released right away
      M.owned.erase(std::remove_if(M.owned.begin(), M.owned.end(), [&](const DevBuf& d) { return d.p == G; }),
                    M.owned.end());
      G = G2;
      ng = nn;
    }
  }
  std::vector<unsigned char> valid;
  if (l >= 2) {
    // A_l = G_m + P_l
    int m = mtop;
    M.nl = (int)ng;
    scatter_level(M, M.inadm[m], 1 << m, false, M.poolP[l].p, 0, KC, G, ng);
    valid.assign(ng, 0);
    for (int j = 0; j < (1 << m); ++j)
      for (int a = 0; a < M.h_rank[M.slot0(m) + j]; ++a) valid[(size_t)j * KC + a] = 1;
    M.d_Al = G;
  } else {
    // A_1 = D + U G_L U^T on the padded point slots
    int64_t np = (int64_t)(1 << L) * KD;
    H2_REQUIRE(np <= 16384, H2MG_ERR_UNSUPPORTED, "a single-level (dense) hierarchy needs n <= 16384");
    double* A1 = (double*)M.alloc(sizeof(double) * np * np);
    if (M.tstar >= 0) {
      int ncl = 1 << L;
      expand(G, ng, M.d_U, KD, KC, ncl, 0, level_spread(M, L), A1, np, s);
    }
    M.nl = (int)np;
    valid.assign(np, 0);
    for (int j = 0; j < (1 << L); ++j)
      for (int i = 0; i < M.offsets[L][j + 1] - M.offsets[L][j]; ++i) valid[(size_t)j * KD + i] = 1;
    M.d_Al = A1;
    scatter_level(M, M.inadm[L], 1 << L, false, M.poolD.p, 0, KD, A1, np);
  }
  unsigned char* dv = (unsigned char*)M.alloc(valid.size());
  H2_CUDA(cudaMemcpyAsync(dv, valid.data(), valid.size(), cudaMemcpyHostToDevice, s));
  { k_pad_diag<<<ceil_div(M.nl, 256), 256, 0, s>>>(M.d_Al, M.nl, dv); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  factor_and_invert(M);
  M.wcoarse.bytes = sizeof(double) * (2 + NRMAX) * (size_t)M.nl;
  M.wcoarse.p = M.alloc(M.wcoarse.bytes);
}

__global__ void k_to_slots(const double* __restrict__ v, const int* __restrict__ slot_of, int64_t n,
                           double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[slot_of[i]] = v[i];
}
__global__ void k_from_slots(const double* __restrict__ v, const int* __restrict__ slot_of, int64_t n,
                             double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = v[slot_of[i]];
}

// E = A_l^-1 R for NR columns of the padded operator: the product with the stored inverse and
// one step of refinement, E += A_l^-1 (R - A_l E). The inverse X^T X is off by the square of
// X's condition, and not column by column like substitution's: without the step the
// residual of a solve of 430 Gaussian points with nugget 1e-8 was 2e7 roundings of |A| |E|
// and its error 55 times that of two substitutions; with it the residual is below one. It
// costs two more products of order nl per cycle; the inverse by substitution on all columns
// would cost n^3 / 3 more FMAs per build.
template <int NR>
static void dense_solve(const Matrix& M, const double* r, double* e, cudaStream_t s) {
  const int64_t n = M.nl;
  double* t = (double*)M.wcoarse.p + 2 * n;
  const int g = ceil_div(n, 8);
  launch_chain(k_symv_multi<NR>, g, 256, 0, s, M.d_Ainv, n, r, nullptr, 1.0, e);
  H2_LAUNCH_CHECK();
  launch_chain(k_symv_multi<NR>, g, 256, 0, s, M.d_Al, n, e, r, -1.0, t);
  H2_LAUNCH_CHECK();
  launch_chain(k_symv_multi<NR>, g, 256, 0, s, M.d_Ainv, n, t, e, 1.0, e);
  H2_LAUNCH_CHECK();
}

// e = A_l^{-1} r. For l = 1 the vectors are in user point order and are mapped to and from
// the padded point slots.
void coarse_solve(Matrix& M, const double* r, double* e, cudaStream_t s) {
  int64_t n = M.nl;
  double* w = (double*)M.wcoarse.p;
  double* x = w + n;
  const double* rin = r;
  double* eout = e;
  if (M.lev == 1) {
    H2_CUDA(cudaMemsetAsync(w, 0, sizeof(double) * n, s));
    { k_to_slots<<<ceil_div(M.n, 256), 256, 0, s>>>(r, M.d_slot_of, M.n, w); ::h2mg::count_launch(); }
    H2_LAUNCH_CHECK();
    rin = w;
    eout = x;
  } else if (r == e) {
    H2_CUDA(cudaMemcpyAsync(w, r, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    rin = w;
  }
  dense_solve<1>(M, rin, eout, s);
  if (M.lev == 1) {
    { k_from_slots<<<ceil_div(M.n, 256), 256, 0, s>>>(x, M.d_slot_of, M.n, e); ::h2mg::count_launch(); }
    H2_LAUNCH_CHECK();
  }
}

// The coarse solve for nr columns of the coarsest level (leading dimension nl); r and
// e must not overlap. Level l = 1 (the whole matrix is dense) goes column by column.
void coarse_solve_multi(Matrix& M, const double* r, double* e, int nr, cudaStream_t s) {
  if (M.lev == 1) {
    for (int c = 0; c < nr; ++c) coarse_solve(M, r + c * M.n, e + c * M.n, s);
    return;
  }
  switch (nr) {
    case 1: dense_solve<1>(M, r, e, s); break;
    case 2: dense_solve<2>(M, r, e, s); break;
    case 3: dense_solve<3>(M, r, e, s); break;
    case 4: dense_solve<4>(M, r, e, s); break;
    default: throw Error{H2MG_ERR_INVALID_ARG, "too many columns for one coarse solve"};
  }
}

}  // namespace h2mg
