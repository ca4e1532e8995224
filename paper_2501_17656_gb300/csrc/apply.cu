// apply.cu -- the level-synchronous H2 matrix-vector product of every multigrid level.
//
// Sec. 3.1: y = D x + U_1 (S_1 x_1 + U_2 (... (S_{l-1} x_l + U_l S_l x_l) ...)) with
// x_i = V_i x_{i-1} (upward pass) and y_{i-1} = D_i x_{i-1} + U_i y_i (downward pass).
// For multigrid level i >= 2 the operator A_i (eq. a2_str) has the same shape on the
// coefficients of tree level m(i), with P_i in place of D and the identity as the
// basis of level m(i).
//
// GPU layout: one symmetric block-sparse product (k_bsgemv) covers the close blocks
// or every coupling level at once: one CTA per block row, each warp streams whole
// K x K blocks (swizzled so that every warp load is one contiguous 512 B segment),
// and each block is used twice -- y_t += B x_s for its row and, for s != t, the
// transposed product B^T x_t for its column, both added atomically into a zeroed row
// buffer. Float64 blocks of 32 and 64 go through k_bsgemv_fx (fixed point on the integer
// pipe), smaller blocks through k_bsgemv_small; these deal entries to warps. The upward pass
// (k_leaf_in, k_up_tree) forms the cluster coefficients of every level; the downward pass
// (k_down_tree) adds the transfer from the parent to each level's row results and writes the
// finest level out (k_leaf_final at i = 1).
//
// Arithmetic per block format: F64 (fixed point, DFMA where it does not serve), DF
// (double-float on the FP32 pipes: the error-free products/sums of Dekker and Knuth), F32
// (FP32 FMA). Vectors inside the product are in the same format; the multigrid vectors
// outside are float64.
#include <algorithm>

#include "fixed.cuh"
#include "internal.h"

namespace h2mg {

// ----------------------------------------------------------------------------- arithmetic
template <int FMT>
struct Ar;

template <>
struct Ar<FMT_F64> {
  static constexpr int V = 2;
  using yo_t = double;       // type of the atomically accumulated row outputs
  __device__ static yo_t to_yo(double a) { return a; }
  __device__ static void atomic_add(yo_t* p, double a) { atomicAdd(p, a); }
  __device__ static double from_yo(yo_t v) { return v; }
  using vec_t = double;
  using mel_t = double;
  using acc_t = double;
  using ld_t = double2;
  __device__ static acc_t zero() { return 0.0; }
  __device__ static void decode(const ld_t& v, mel_t* m) {
    m[0] = v.x;
    m[1] = v.y;
  }
  __device__ static void fma(acc_t& a, mel_t m, vec_t x) { a = ::fma(m, x, a); }
  __device__ static void add(acc_t& a, acc_t b) { a += b; }
  __device__ static void norm(acc_t&) {}
  __device__ static acc_t shfl(acc_t a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }
  __device__ static vec_t out(acc_t a) { return a; }
  __device__ static double to_d(vec_t v) { return v; }
  __device__ static vec_t from_d(double v) { return v; }
};

template <>
struct Ar<FMT_DF> {
  static constexpr int V = 2;
  using yo_t = double;
  __device__ static yo_t to_yo(float2 a) { return (double)a.x + (double)a.y; }
  __device__ static void atomic_add(yo_t* p, float2 a) { atomicAdd(p, to_yo(a)); }
  __device__ static float2 from_yo(yo_t v) { return from_d(v); }
  using vec_t = float2;
  using mel_t = float2;
  using acc_t = float2;
  using ld_t = float4;
  __device__ static acc_t zero() { return make_float2(0.f, 0.f); }
  __device__ static void decode(const ld_t& v, mel_t* m) {
    m[0] = make_float2(v.x, v.y);
    m[1] = make_float2(v.z, v.w);
  }
  __device__ static void fma(acc_t& a, mel_t m, vec_t x) { df_fma(a.x, a.y, m.x, m.y, x.x, x.y); }
  __device__ static void add(acc_t& a, acc_t b) { df_add(a.x, a.y, b.x, b.y); }
  __device__ static void norm(acc_t& a) { df_norm(a.x, a.y); }
  __device__ static acc_t shfl(acc_t a, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, m), __shfl_xor_sync(0xffffffffu, a.y, m));
  }
  __device__ static vec_t out(acc_t a) {
    df_norm(a.x, a.y);
    return a;
  }
  __device__ static double to_d(vec_t v) { return (double)v.x + (double)v.y; }
  __device__ static vec_t from_d(double v) {
    df2 d = df_from_double(v);
    return make_float2(d.hi, d.lo);
  }
};

template <>
struct Ar<FMT_F32> {
  static constexpr int V = 4;
  using yo_t = float;
  __device__ static yo_t to_yo(float a) { return a; }
  __device__ static void atomic_add(yo_t* p, float a) { atomicAdd(p, a); }
  __device__ static float from_yo(yo_t v) { return v; }
  using vec_t = float;
  using mel_t = float;
  using acc_t = float;
  using ld_t = float4;
  __device__ static acc_t zero() { return 0.f; }
  __device__ static void decode(const ld_t& v, mel_t* m) {
    m[0] = v.x;
    m[1] = v.y;
    m[2] = v.z;
    m[3] = v.w;
  }
  __device__ static void fma(acc_t& a, mel_t m, vec_t x) { a = fmaf(m, x, a); }
  __device__ static void add(acc_t& a, acc_t b) { a += b; }
  __device__ static void norm(acc_t&) {}
  __device__ static acc_t shfl(acc_t a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }
  __device__ static vec_t out(acc_t a) { return a; }
  __device__ static double to_d(vec_t v) { return (double)v; }
  __device__ static vec_t from_d(double v) { return __double2float_rn(v); }
};

// Float64 blocks, double-double vectors and sums (the extended-precision residual).
template <>
struct Ar<FMT_DD> {
  static constexpr int V = 2;
  using yo_t = double2;
  __device__ static yo_t to_yo(double2 a) { return a; }
  __device__ static void atomic_add(yo_t* p, double2 a) { dd_atomic_add(p, a); }
  __device__ static double2 from_yo(yo_t v) { return v; }
  using vec_t = double2;
  using mel_t = double;
  using acc_t = double2;
  using ld_t = double2;
  __device__ static acc_t zero() { return make_double2(0.0, 0.0); }
  __device__ static void decode(const ld_t& v, mel_t* m) {
    m[0] = v.x;
    m[1] = v.y;
  }
  __device__ static void fma(acc_t& a, mel_t m, vec_t x) { dd_fma(a.x, a.y, m, x.x, x.y); }
  __device__ static void add(acc_t& a, acc_t b) { dd_add(a.x, a.y, b.x, b.y); }
  __device__ static void norm(acc_t& a) { dd_norm(a.x, a.y); }
  __device__ static acc_t shfl(acc_t a, int m) {
    return make_double2(__shfl_xor_sync(0xffffffffu, a.x, m), __shfl_xor_sync(0xffffffffu, a.y, m));
  }
  __device__ static vec_t out(acc_t a) {
    dd_norm(a.x, a.y);
    return a;
  }
  __device__ static double to_d(vec_t v) { return v.x + v.y; }
  __device__ static vec_t from_d(double v) { return make_double2(v, 0.0); }
};

// NR consecutive elements from shared memory, as one vector load where the row is 8
// or 16 bytes (rows are aligned to their size).
template <class T, int NR>
__device__ __forceinline__ void load_row(const T* p, T* out) {
  if constexpr (sizeof(T) * NR == 16) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    memcpy(out, &v, 16);
  } else if constexpr (sizeof(T) * NR == 8) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    memcpy(out, &v, 8);
  } else {
#pragma unroll
    for (int j = 0; j < NR; ++j) out[j] = p[j];
  }
}

// yrow[0..NR-1] += v: one vector reduction for two or four FP32 columns (interleaved, so
// aligned to their size), else one atomic per column. Four columns on the second level of a
// sphere of 18000 panels: 89 -> 80 us.
template <int FMT, int NR>
__device__ __forceinline__ void add_columns(typename Ar<FMT>::yo_t* p, const typename Ar<FMT>::acc_t (&v)[NR]) {
  using A = Ar<FMT>;
  if constexpr (FMT == FMT_F32 && NR == 4) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
  } else if constexpr (FMT == FMT_F32 && NR == 2) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v[0]), "f"(v[1]) : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < NR; ++j) A::atomic_add(p + j, A::out(v[j]));
  }
}

// ----------------------------------------------------------------------------- block GEMV
// One CTA (8 warps) per block row t of a symmetric upper-stored block operator:
// yrow[t] += sum_e B_e x_col(e) and, for every off-diagonal entry e = (t, s),
// yrow[s] += B_e^T x_t. All contributions are atomic adds (FP64 for the F64 and DF
// copies, FP32 for the F32 copy) into a row buffer zeroed before the launch, so the
// summation order, and the last bits of a sum, may differ from run to run. When the
// operator has few rows, each row is split over `split` CTAs (strided entries).
// NR right-hand sides share every block read: vectors are interleaved, element
// (slot, coefficient, column j) at ((slot * K + coefficient) * NR + j).
// CTAs per SM the register allocation must allow: the FP32 products are HBM-bound and
// need the occupancy; the float64 / double-float ones are ALU-bound.
template <int FMT, int NR>
constexpr int bsgemv_min_ctas() {
  return FMT == FMT_F32 ? (NR >= 4 ? 2 : (NR == 2 ? 3 : 4)) : 2;
}

template <int K, int FMT, int NR>
__global__ void __launch_bounds__(256, bsgemv_min_ctas<FMT, NR>()) k_bsgemv(const int* __restrict__ rowptr,
                                                const int* __restrict__ col,
                                                const void* const* __restrict__ blk,
                                                const typename Ar<FMT>::vec_t* x,
                                                typename Ar<FMT>::yo_t* yrow, int split, bool first) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using mel_t = typename A::mel_t;
  using acc_t = typename A::acc_t;
  using ld_t = typename A::ld_t;
  constexpr int LPC = K / 8, CPP = 32 / LPC, T = K * K / 256;
  constexpr int CH = T < LPC ? T : LPC;
  constexpr int V = A::V, P = 8 / V;
  __shared__ acc_t red[8][K * NR];
  // x of the block row (input of the transposed products), one padding row after
  // every 8 rows so that the 8 row groups of a warp read distinct banks
  __shared__ __align__(16) vec_t sxt[(K + K / 8) * NR];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row = blockIdx.x / split, part = blockIdx.x % split;
  const int rb = 8 * (lane % LPC), cl = lane / LPC;
  const int e0 = rowptr[row], e1 = rowptr[row + 1];
  constexpr unsigned kBlockBytes = K * K / V * (unsigned)sizeof(ld_t);   // one stored block
  // the warp's first block, while the kernel before this one runs
  if (first && lane == 0 && e0 + part * 8 + w < e1) prefetch_l2_bulk(blk[e0 + part * 8 + w], kBlockBytes);
  chain_wait();
  for (int i = threadIdx.x; i < K * NR; i += blockDim.x) {
    const int r = i / NR;
    sxt[(r + r / 8) * NR + i % NR] = x[(int64_t)row * K * NR + i];
  }
  __syncthreads();
  const vec_t* xt = sxt + (rb + rb / 8) * NR;   // rows rb..rb+7 of this lane
  acc_t ya[8][NR];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < NR; ++j) ya[r][j] = A::zero();
  for (int e = e0 + part * 8 + w; e < e1; e += 8 * split) {
    const int s = col[e];
    const ld_t* B = (const ld_t*)blk[e];
    // with one column the loads of 32 warps per SM already cover the DRAM latency, and
    // prefetched blocks would be evicted from L2 before use; with several columns
    // (fewer resident warps) the prefetch keeps the stream going
    if constexpr (NR >= 2)
      if (lane == 0 && e + 8 * split < e1) prefetch_l2_bulk(blk[e + 8 * split], kBlockBytes);
    const vec_t* xs = x + (int64_t)s * K * NR;
    const bool off = (s != row);
#pragma unroll 1
    for (int ch = 0; ch < T / CH; ++ch) {
      acc_t zc[CH][NR];
#pragma unroll
      for (int tt = 0; tt < CH; ++tt) {
        const int t = ch * CH + tt;
        mel_t m[8];
#pragma unroll
        for (int k = 0; k < P; ++k) {
          ld_t v = __ldcs(B + (t * P + k) * 32 + lane);
          A::decode(v, m + k * V);
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          const vec_t xv = xs[(cl + CPP * t) * NR + j];
#pragma unroll
          for (int r = 0; r < 8; ++r) A::fma(ya[r][j], m[r], xv);
          acc_t zz = A::zero();
#pragma unroll
          for (int r = 0; r < 8; ++r) A::fma(zz, m[r], xt[r * NR + j]);
          zc[tt][j] = zz;
        }
        if ((t & 3) == 3) {
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int j = 0; j < NR; ++j) A::norm(ya[r][j]);
        }
      }
      if (off) {
        // reduce the CH partial columns over the LPC lanes that share them
        acc_t zs[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          if (CH == LPC) {
#pragma unroll
            for (int h = CH / 2; h >= 1; h >>= 1) {
              const bool up = (lane & h) != 0;
#pragma unroll
              for (int q = 0; q < h; ++q) {
                acc_t send = up ? zc[q][j] : zc[q + h][j];
                acc_t keep = up ? zc[q + h][j] : zc[q][j];
                A::add(keep, A::shfl(send, h));
                zc[q][j] = keep;
              }
            }
          } else {
#pragma unroll
            for (int h = LPC / 2; h >= 1; h >>= 1) A::add(zc[0][j], A::shfl(zc[0][j], h));
          }
          zs[j] = zc[0][j];
        }
        if (CH == LPC || (lane % LPC) == 0)
          add_columns<FMT, NR>(yrow + ((int64_t)s * K + cl + CPP * (ch * CH + (lane & (CH - 1)))) * NR, zs);
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) A::norm(ya[r][j]);
  }
  // rows: sum over the lanes that share them, then over the warps
#pragma unroll
  for (int h = LPC; h < 32; h <<= 1)
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) A::add(ya[r][j], A::shfl(ya[r][j], h));
  if (lane < LPC)
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) red[w][(rb + r) * NR + j] = ya[r][j];
  __syncthreads();
  for (int i = threadIdx.x; i < K * NR; i += blockDim.x) {
    acc_t s = red[0][i];
#pragma unroll
    for (int ww = 1; ww < 8; ++ww) A::add(s, red[ww][i]);
    A::atomic_add(yrow + (int64_t)row * K * NR + i, A::out(s));
  }
}

// ----------------------------------------------------------------------------- small blocks
// The product of k_bsgemv for blocks of 16 and 32: every warp owns `per` consecutive entries
// and adds its row sums when the row changes. A block is one pass (16) or four (32) of a
// warp, so a CTA per row with eight warps and a CTA-wide sum leaves most warps without an
// entry. Bound by latency at the sizes where it matters: the 112 block rows of 16 of the
// second level of 4096 points (F64, 1.3 MB of blocks) took 35 us and now take 6.
template <int K, int FMT, int NR>
__global__ void __launch_bounds__(256) k_bsgemv_small(const int* __restrict__ erow, const int* __restrict__ col,
                                                      const void* const* __restrict__ blk,
                                                      const typename Ar<FMT>::vec_t* x,
                                                      typename Ar<FMT>::yo_t* yrow, int nnz, int per) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using mel_t = typename A::mel_t;
  using acc_t = typename A::acc_t;
  using ld_t = typename A::ld_t;
  constexpr int LPC = K / 8, CPP = 32 / LPC, T = K * K / 256;
  constexpr int V = A::V, P = 8 / V;
  const int lane = threadIdx.x & 31;
  const int rb = 8 * (lane % LPC), cl = lane / LPC;
  const int64_t e0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * per;
  const int e1 = (int)min(e0 + per, (int64_t)nnz);
  if (lane == 0 && e0 < e1) prefetch_l2_bulk(blk[e0], K * K / V * (unsigned)sizeof(ld_t));
  chain_wait();
  acc_t ya[8][NR];
  vec_t xt[8][NR];
  int row = -1;
  auto flush = [&]() {
    // sum over the lanes that share rows; lane group cl keeps rows cl, cl + CPP, ..
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      acc_t v[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        A::norm(ya[r][j]);
#pragma unroll
        for (int h = LPC; h < 32; h <<= 1) A::add(ya[r][j], A::shfl(ya[r][j], h));
        v[j] = ya[r][j];
      }
      if (r == cl) add_columns<FMT, NR>(yrow + ((int64_t)row * K + rb + r) * NR, v);
    }
  };
  for (int e = (int)e0; e < e1; ++e) {
    const int t = erow[e], s = col[e];
    const ld_t* B = (const ld_t*)blk[e];
    ld_t q[T][P];
#pragma unroll
    for (int p = 0; p < T; ++p)
#pragma unroll
      for (int k = 0; k < P; ++k) q[p][k] = __ldcs(B + (p * P + k) * 32 + lane);
    const vec_t* xs = x + (int64_t)s * K * NR;
    if (t != row) {
      if (row >= 0) flush();
      row = t;
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          xt[r][j] = x[((int64_t)t * K + rb + r) * NR + j];
          ya[r][j] = A::zero();
        }
    }
#pragma unroll
    for (int p = 0; p < T; ++p) {
      mel_t m[8];
#pragma unroll
      for (int k = 0; k < P; ++k) A::decode(q[p][k], m + k * V);
      acc_t z[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        const vec_t xv = xs[(cl + CPP * p) * NR + j];
        z[j] = A::zero();
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          A::fma(ya[r][j], m[r], xv);
          A::fma(z[j], m[r], xt[r][j]);
        }
#pragma unroll
        for (int h = 1; h < LPC; h <<= 1) A::add(z[j], A::shfl(z[j], h));
      }
      if (s != t && (lane % LPC) == 0) add_columns<FMT, NR>(yrow + ((int64_t)s * K + cl + CPP * p) * NR, z);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) A::norm(ya[r][j]);
  }
  if (row >= 0) flush();
}

// ----------------------------------------------------------------------------- float64 block GEMV
// Exponent of every stored float64 block (one warp per block): the biased exponent of its
// largest magnitude, FX_EZERO for an all-zero block, FX_NONE where fixed point does not
// serve: exponents outside FX_EMIN..FX_VMAX (Inf and NaN among them), or, with `skip`
// given, a row or column cluster it marks.
__global__ void k_block_exponents(const void* const* __restrict__ blk, const int* __restrict__ row,
                                  const int* __restrict__ col, const unsigned char* __restrict__ skip, int nnz,
                                  int elems, short* __restrict__ bexp) {
  const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (e >= nnz) return;
  const double2* B = (const double2*)blk[e];
  int m = 0;
  bool any = false;
  for (int i = lane; i < elems / 2; i += 32) {
    const double2 v = B[i];
    any = any || v.x != 0.0 || v.y != 0.0;
    m = max(m, max(fx_exponent(v.x), fx_exponent(v.y)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  any = __any_sync(0xffffffffu, any);
  if (lane == 0) {
    int E = any ? ((m < FX_EMIN || m > FX_VMAX) ? FX_NONE : m) : FX_EZERO;
    if (skip && (skip[row[e]] || skip[col[e]])) E = FX_NONE;
    bexp[e] = (short)E;
  }
}

// Smallest and largest exponents of the diagonal entries |A_ii| and of sqrt(w_i) of every leaf:
// (dg, dg, sw, sw).
__global__ void k_leaf_spread(const int* __restrict__ leafoff, const double* __restrict__ dg,
                              const double* __restrict__ sw, int nleaf, short4* __restrict__ out) {
  const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (l >= nleaf) return;
  int lo = 4095, hi = 0, slo = 4095, shi = 0;
  for (int p = leafoff[l] + lane; p < leafoff[l + 1]; p += 32) {
    const int x = fx_exponent(dg[p]), s = fx_exponent(sw[p]);
    lo = min(lo, x);
    hi = max(hi, x);
    slo = min(slo, s);
    shi = max(shi, s);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  slo = __reduce_min_sync(0xffffffffu, slo);
  shi = __reduce_max_sync(0xffffffffu, shi);
  if (lane == 0) out[l] = make_short4((short)lo, (short)hi, (short)slo, (short)shi);
}

// The product of k_bsgemv for float64 blocks in fixed point (fixed.cuh). Every warp owns
// `per` consecutive units of work, a unit being CH of the T column passes of one entry, and
// flushes its row sums when the row changes: no CTA-wide step, and operators with few
// entries spread over the whole GPU. A block's values are encoded as they arrive (16 integer
// operations each) and used for both products (6 multiply-adds); the sums of a unit are
// exact and are scaled into float64 once. The blocks stream through a ring of FX_RING
// passes (2 KB each) per warp in shared memory, filled by cp.async: a lane reads back what
// it asked for itself, so the ring needs no synchronisation. What bounds it: see
// launch_bsgemv_fx.
constexpr int FX_RING = 4;
constexpr int FXB = 29;          // bits per part: at most 16 terms per accumulator
// Point values that span more than 2^20 inside a leaf go through float64 with the leaf's
// blocks: below that the smallest keep 38 bits. Normally distributed values exceed it in one
// leaf of 10000. (At 2^16, one of 700, the few warps that meet such leaves end last: two
// columns of 65536 points took 1.85 ms instead of 1.76.) Coefficients, of orthonormal bases,
// have no such limit: what counts there is their norm, and smooth vectors span many decades.
constexpr int FX_SPREAD = 20;
template <int K, int NR>
constexpr size_t fx_smem() {
  return 8 * (FX_RING * 2048 + sizeof(double) * 8 * NR * 32 + sizeof(Fx) * K * NR);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

template <int K, int NR>
__global__ void __launch_bounds__(256, NR == 1 ? 2 : 1)
    k_bsgemv_fx(const int* __restrict__ erow, const int* __restrict__ col, const void* const* __restrict__ blk,
                const short* __restrict__ bexp, const double* x, double* yrow,
                int64_t units, int per, int spread) {
  constexpr int LPC = K / 8, CPP = 32 / LPC, T = K * K / 256, CH = T < LPC ? T : LPC, NCH = T / CH;
  constexpr int XL = K * NR / 32;                // elements of x_s per lane
  extern __shared__ __align__(16) unsigned char dsm[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int rb = 8 * (lane % LPC), cl = lane / LPC;
  const int64_t u0 = ((int64_t)blockIdx.x * 8 + w) * per;
  const int64_t u1 = u0 + per < units ? u0 + per : units;
  if (u0 >= u1) return;
  double2* ring = (double2*)dsm + w * FX_RING * 128 + lane;          // [FX_RING][4][32], this lane's column
  double(*yad)[32] = (double(*)[32])(dsm + 8 * FX_RING * 2048) + w * 8 * NR;   // float64 row sums, between entries
  Fx* xs = (Fx*)(dsm + 8 * (FX_RING * 2048 + sizeof(double) * 8 * NR * 32)) + w * K * NR;   // encoded x of the column
  Fx xt[8][NR];
  int Et[NR];
  bool tfast = false;
  int row = -1;
  const double* xrow = x;

  // first pass of a unit, as this lane reads it (nullptr past the end)
  auto unit_ptr = [&](int64_t u) -> const double2* {
    return u < u1 ? (const double2*)blk[u / NCH] + (u % NCH) * (CH * 128) + lane : nullptr;
  };
  const double2* cur = unit_ptr(u0);
  const double2* nxt = unit_ptr(u0 + 1);
  // starts the copy of pass tt of the unit at p; one group per call, an empty one past the end
  auto issue = [&](const double2* p, int tt) {
    if (p)
#pragma unroll
      for (int k = 0; k < 4; ++k) cp_async16(ring + (tt % FX_RING) * 128 + k * 32, p + tt * 128 + k * 32);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // reads pass tt of the current unit; the slot read before it is refilled
  auto take = [&](int tt, double2* d) {
    asm volatile("cp.async.wait_group %0;" ::"n"(FX_RING - 2) : "memory");
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = ring[(tt % FX_RING) * 128 + k * 32];
    constexpr int A = FX_RING - 1;
    if (tt + A < CH)
      issue(cur, tt + A);
    else
      issue(nxt, tt + A - CH);
  };
  auto next_unit = [&](int64_t u) {              // u: the unit that has just been finished
    cur = nxt;
    nxt = unit_ptr(u + 2);
  };
  static_assert(CH % FX_RING == 0, "a unit starts at slot 0");
#pragma unroll
  for (int tt = 0; tt < FX_RING - 1; ++tt) issue(cur, tt);
  chain_wait();                                  // the first blocks are under way before it

  // adds the row sums of the lanes that share rows (32 / LPC of them) and stores them
  auto flush = [&]() {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        double v = yad[r * NR + j][lane];
#pragma unroll
        for (int h = 16; h >= LPC; h >>= 1) v += __shfl_xor_sync(0xffffffffu, v, h);
        // every lane of a group holds the sum; lane group cl stores rows cl, cl + CPP, ..
        if (r % CPP == cl) atomicAdd(yrow + ((int64_t)row * K + rb + r) * NR + j, v);
      }
  };

  // z[.][j]: this lane's part of the CH column sums of chunk ch, block column s. Sums them over
  // the LPC lanes that share a column; lane keeps column lane % CH
  auto add_column = [&](auto& z, int j, int ch, int s, double scale) {
#pragma unroll
    for (int h = CH / 2; h >= 1; h >>= 1) {
      const bool up = (lane & h) != 0;
#pragma unroll
      for (int q = 0; q < h; ++q) {
        const auto send = up ? z[q][j] : z[q + h][j], keep = up ? z[q + h][j] : z[q][j];
        z[q][j] = keep + __shfl_xor_sync(0xffffffffu, send, h);
      }
    }
#pragma unroll
    for (int h = CH; h < LPC; h <<= 1) z[0][j] += __shfl_xor_sync(0xffffffffu, z[0][j], h);
    if ((lane % LPC) < CH)
      atomicAdd(yrow + ((int64_t)s * K + cl + CPP * (ch * CH + (lane & (CH - 1)))) * NR + j, (double)z[0][j] * scale);
  };

  // largest exponent, and smallest of a value that is not zero (a subnormal one: 0)
  auto widest = [](double v, int& hi, int& lo) {
    const int x = fx_exponent(v);
    hi = max(hi, x);
    lo = min(lo, fx_is_zero(v) ? 4095 : x);
  };
  // exponents of a piece of the vector, from all lanes' hi and lo; false: float64
  auto vector_exponents = [&](int (&hi)[NR], const int (&lo)[NR]) {
    bool out = false;
#pragma unroll
    for (int j = 0; j < NR; ++j) hi[j] = __reduce_max_sync(0xffffffffu, hi[j]);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      out = out || lo[j] < hi[j] - spread || (hi[j] < FX_EMIN && lo[j] < 4095) || hi[j] > FX_VMAX;
      hi[j] = hi[j] == 0 ? FX_EZERO : hi[j];
    }
    return !__any_sync(0xffffffffu, out);
  };

  for (int64_t u = u0; u < u1;) {
    const int e = (int)(u / NCH);
    const int c0 = (int)(u % NCH), c1 = (int)min((int64_t)NCH, c0 + (u1 - u));
    int64_t uc = u;                              // the unit in hand
    u += c1 - c0;
    const int t = erow[e], s = col[e], Eb = bexp[e];
    if (t != row) {
      if (row >= 0) flush();
      row = t;
      xrow = x + (int64_t)t * K * NR;
      double v[8][NR];
      int lo[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        Et[j] = 0;
        lo[j] = 4095;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          v[r][j] = xrow[(rb + r) * NR + j];
          widest(v[r][j], Et[j], lo[j]);
          yad[r * NR + j][lane] = 0.0;
        }
      }
      tfast = vector_exponents(Et, lo);
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) xt[r][j] = fx_encode<FXB>(v[r][j], Et[j] + 1);   // a bit less: 64 terms below 2^63
    }
    const bool off = (s != t);
    // x of the entry's column: its exponents, then encoded into this warp's shared row
    const double* xcol = x + (int64_t)s * K * NR;
    int Es[NR];
    bool fast = tfast && Eb != FX_NONE;
    {
      double v[XL];
      int lo[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        Es[j] = 0;
        lo[j] = 4095;
      }
#pragma unroll
      for (int q = 0; q < XL; ++q) {
        v[q] = xcol[lane * XL + q];          // XL is a multiple of NR: element q is column q % NR
        widest(v[q], Es[q % NR], lo[q % NR]);
      }
      fast = vector_exponents(Es, lo) && fast;
#pragma unroll
      for (int j = 0; j < NR; ++j) fast = fast && Eb + min(Es[j], Et[j]) >= FX_VSUM;
      __syncwarp();                          // the previous entry's reads are done
      if (fast)
#pragma unroll
        for (int q = 0; q < XL; ++q) xs[lane * XL + q] = fx_encode<FXB>(v[q], Es[q % NR]);
      __syncwarp();
    }
    if (__builtin_expect(fast, 1)) {
      int64_t yh[8][NR], ym[8][NR];
      double sr[NR], sc[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        sr[j] = fx_scale_a(Eb) * fx_scale_b(Es[j]);
        sc[j] = fx_scale_a(Eb) * fx_scale_b(Et[j] + 1);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          yh[r][j] = 0;
          ym[r][j] = fx_half<FXB>();
        }
#pragma unroll 1
      for (int ch = c0; ch < c1; ++ch) {
        int64_t z[CH][NR];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
          const int p = ch * CH + tt;
          double2 d[4];
          take(tt, d);
          Fx xv[NR];
#pragma unroll
          for (int j = 0; j < NR; ++j) xv[j] = xs[(cl + CPP * p) * NR + j];
          int64_t zh[NR], zm[NR];
#pragma unroll
          for (int j = 0; j < NR; ++j) {
            zh[j] = 0;
            zm[j] = fx_half<FXB>();
          }
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const Fx b = fx_encode<FXB>((r & 1) ? d[r / 2].y : d[r / 2].x, Eb);
#pragma unroll
            for (int j = 0; j < NR; ++j) {
              fx_mad(yh[r][j], b.h, xv[j].h);
              fx_mad(ym[r][j], b.h, xv[j].l);
              fx_mad(ym[r][j], b.l, xv[j].h);
              fx_mad(zh[j], b.h, xt[r][j].h);
              fx_mad(zm[j], b.h, xt[r][j].l);
              fx_mad(zm[j], b.l, xt[r][j].h);
            }
          }
#pragma unroll
          for (int j = 0; j < NR; ++j) z[tt][j] = fx_join<FXB>(zh[j], zm[j]);
        }
        if (off)
#pragma unroll
          for (int j = 0; j < NR; ++j) add_column(z, j, ch, s, sc[j]);
        next_unit(uc++);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          double& y = yad[r * NR + j][lane];
          y = fma((double)fx_join<FXB>(yh[r][j], ym[r][j]), sr[j], y);
        }
    } else {
      // Float64 arithmetic: blocks or vectors outside the range of fixed point. Bound by the
      // float64 pipe like k_bsgemv, with sums in registers and column sums exchanged as above:
      // all blocks of 65536 Gaussian points that way 1.90 ms (one column) and 3.80 ms (two),
      // k_bsgemv 1.92 and 3.73; with row sums in shared memory and a sum over the lanes per
      // column it was 2.12 and 4.21.
      double y[8][NR], xr[8][NR];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          y[r][j] = 0.0;
          xr[r][j] = xrow[(rb + r) * NR + j];
        }
#pragma unroll 1
      for (int ch = c0; ch < c1; ++ch) {
        double z[CH][NR];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
          double2 d[4];
          take(tt, d);
          const double m[8] = {d[0].x, d[0].y, d[1].x, d[1].y, d[2].x, d[2].y, d[3].x, d[3].y};
#pragma unroll
          for (int j = 0; j < NR; ++j) {
            const double xv = xcol[(cl + CPP * (ch * CH + tt)) * NR + j];
            z[tt][j] = 0.0;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              y[r][j] = fma(m[r], xv, y[r][j]);
              z[tt][j] = fma(m[r], xr[r][j], z[tt][j]);
            }
          }
        }
        if (off)
#pragma unroll
          for (int j = 0; j < NR; ++j) add_column(z, j, ch, s, 1.0);
        next_unit(uc++);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) yad[r * NR + j][lane] += y[r][j];
    }
  }
  flush();
}

// ----------------------------------------------------------------------------- passes
// A value another CTA of this launch has written: read from L2.
__device__ __forceinline__ float load_cg(const float* p) { return __ldcg(p); }
__device__ __forceinline__ double load_cg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ float2 load_cg(const float2* p) { return __ldcg(p); }
__device__ __forceinline__ double2 load_cg(const double2* p) { return __ldcg(p); }

// What a product's first kernel does besides its own work. Its input vector is x (float64,
// column j at x + j * ldx) or, inside a CG step (r given), the new direction: per column,
// rho' = r^T r from its partials; stop if rho' <= thresh, else p = r + (rho' / rho) p, which
// is written back to p = x. Every CTA takes the same decision from the same partials, and
// the state it writes is not what the others read. It also clears the row sums that the
// block products add into.
struct VecIn {
  const double* x;
  int64_t ldx;
  const double* r;          // CG: residual (leading dimension ldx), or null
  const double* prr;        // CG: partials of r^T r, CG_PARTS per column
  int np, par;
  CGState* st;
  uint4* zero[3];           // regions cleared by the grid
  int64_t nzero[3];         // their sizes in 16-byte units
};

// Per column: whether the direction changes, and by which factor. Warp j sums column j's
// partials (every CTA in the same order), so that the columns take one barrier together.
template <int NR>
__device__ __forceinline__ void cg_beta(const VecIn& in, bool* go, double* be) {
  __shared__ double sbe[NR];
  __shared__ int sgo[NR];
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    go[j] = false;
    be[j] = 0.0;
  }
  if (!in.r) return;
  const int j = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (j < NR) {
    const double* part = in.prr + j * CG_PARTS;
    CGState* st = in.st + j;
    const int stopped = st->stopped;
    const double rho = st->rho[in.par], thresh = st->thresh;
    double rn = 0.0;
    for (int i = lane; i < in.np; i += 32) rn += part[i];
    for (int o = 16; o > 0; o >>= 1) rn += __shfl_xor_sync(0xffffffffu, rn, o);
    if (lane == 0) {
      const bool stop = stopped || rn <= thresh;
      sgo[j] = !stop;
      sbe[j] = stop ? 0.0 : rn / rho;
      if (blockIdx.x == 0) {
        if (stop)
          st->stopped = 1;
        else
          st->rho[in.par ^ 1] = rn;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    go[q] = sgo[q] != 0;
    be[q] = sbe[q];
  }
}
__device__ __forceinline__ double cg_value(const VecIn& in, int64_t i, bool go, double be) {
  double v = in.x[i];
  if (go) {
    v = fma(be, v, in.r[i]);
    const_cast<double*>(in.x)[i] = v;
  }
  return v;
}
__device__ __forceinline__ void clear_regions(const VecIn& in) {
#pragma unroll
  for (int z = 0; z < 3; ++z)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < in.nzero[z];
         i += (int64_t)gridDim.x * blockDim.x)
      in.zero[z][i] = make_uint4(0, 0, 0, 0);
}

// coefficient vectors (KC per cluster) -> interleaved, for operators without transfers
template <int FMT, int NR>
__global__ void __launch_bounds__(256) k_coef_in(VecIn in, int64_t n, typename Ar<FMT>::vec_t* xc) {
  bool go[NR];
  double be[NR];
  chain_wait();
  cg_beta<NR>(in, go, be);
  clear_regions(in);
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
#pragma unroll
    for (int j = 0; j < NR; ++j) xc[i * NR + j] = Ar<FMT>::from_d(cg_value(in, i + j * in.ldx, go[j], be[j]));
}

// Float -> double by moving the bits: the conversion instruction runs at the float64 rate (2
// per clock and SM), as many as the products it feeds. For finite values; subnormals become
// zero, which the bases do not hold: QR leaves roundings of 1e-17 in the rows of least weight.
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
  return m < 0x00800000u ? 0.0 : __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double d) { return d; }

// Values of the leaf kernels: float64, or double-double.
template <int FMT>
struct LeafVal {
  using t = double;
  __device__ static t zero() { return 0.0; }
  __device__ static void fma(t& a, double u, t x) { a = ::fma(u, x, a); }
  __device__ static void add(t& a, t b) { a += b; }
  __device__ static t in(typename Ar<FMT>::vec_t v) { return Ar<FMT>::to_d(v); }
  __device__ static typename Ar<FMT>::vec_t out(t a) { return Ar<FMT>::from_d(a); }
  __device__ static t row(typename Ar<FMT>::yo_t v) { return (double)v; }
  __device__ static double val(t a) { return a; }
};
template <>
struct LeafVal<FMT_DD> {
  using t = double2;
  __device__ static t zero() { return make_double2(0.0, 0.0); }
  __device__ static void fma(t& a, double u, t x) { dd_fma(a.x, a.y, u, x.x, x.y); }
  __device__ static void add(t& a, t b) { dd_add(a.x, a.y, b.x, b.y); }
  __device__ static t in(double2 v) { return v; }
  __device__ static double2 out(t a) {
    dd_norm(a.x, a.y);
    return a;
  }
  __device__ static t row(double2 v) { return v; }
  __device__ static double val(t a) { return a.x + a.y; }
};

constexpr int LEAF_CTAS = CG_PARTS;   // the leaf kernels' grids: one partial per CTA at most

// Point vectors (user order) -> padded tree slots, zero in the padding, and, with a far
// field, x_hat(leaf l)[b] = sum_i U_l[i, b] x_l[i] (UT = U^T, KC x KD column-major): 256 / KC
// threads share each sum.
template <int FMT, class BT, int NR>
__global__ void __launch_bounds__(256) k_leaf_in(VecIn in, const BT* __restrict__ UT, int KD, int KC, int nleaf,
                                                 const int* __restrict__ leafoff, const int* __restrict__ perm,
                                                 typename Ar<FMT>::vec_t* xp,
                                                 typename Ar<FMT>::vec_t* xc) {
  using V = LeafVal<FMT>;
  using v_t = typename V::t;
  __shared__ v_t xs[64 * NR];
  __shared__ v_t red[256 * NR];
  bool go[NR];
  double be[NR];
  if (UT && threadIdx.x == 0) prefetch_l2_bulk(UT + (int64_t)blockIdx.x * KD * KC, KD * KC * (unsigned)sizeof(BT));
  chain_wait();
  cg_beta<NR>(in, go, be);
  clear_regions(in);
  const int b = threadIdx.x % KC, part = threadIdx.x / KC, parts = 256 / KC;
  for (int l = blockIdx.x; l < nleaf; l += gridDim.x) {
    const int p0 = leafoff[l], nl = leafoff[l + 1] - p0;
    for (int e = threadIdx.x; e < KD * NR; e += 256) {
      const int i = e % KD, j = e / KD;
      typename Ar<FMT>::vec_t v = Ar<FMT>::from_d(0.0);
      if (i < nl) {
        const int64_t o = perm[p0 + i] + j * in.ldx;
        bool g = go[0];
        double f = be[0];
#pragma unroll
        for (int q = 1; q < NR; ++q)
          if (j == q) {
            g = go[q];
            f = be[q];
          }
        v = Ar<FMT>::from_d(cg_value(in, o, g, f));
      }
      xp[((int64_t)l * KD + i) * NR + j] = v;
      xs[i * NR + j] = V::in(v);
    }
    if (!UT) continue;
    __syncthreads();
    const BT* Ul = UT + (int64_t)l * KD * KC + b;
    v_t acc[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) acc[j] = V::zero();
#pragma unroll 4
    for (int i = part; i < KD; i += parts) {
      const double u = widen(Ul[i * KC]);
#pragma unroll
      for (int j = 0; j < NR; ++j) V::fma(acc[j], u, xs[i * NR + j]);
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) red[(part * KC + b) * NR + j] = acc[j];
    __syncthreads();
    for (int e = threadIdx.x; e < KC * NR; e += 256) {
      v_t t = red[e];
      for (int q = 1; q < parts; ++q) V::add(t, red[q * KC * NR + e]);
      xc[(int64_t)l * KC * NR + e] = V::out(t);
    }
    __syncthreads();
  }
}

// Transfer passes as block products. Every orthonormal transfer E'_c (K x K, rows =
// child coefficients, columns = parent coefficients) is stored swizzled like the
// blocks of k_bsgemv, and one warp streams one transfer with the same lane layout:
// the upward pass uses the transposed product E'_c^T x_c (reduce-scatter over the
// lanes that share a column), the downward pass the row product E'_c y_parent.
//
// The upward pass is one launch: a CTA owns two siblings of the bottom level, and of the two
// CTAs below a cluster the one that comes second goes on with it (k_up_tree). The downward
// pass covers up to five levels per launch: a CTA owns 4 (or 2) clusters of the bottom level
// and recomputes the path of their ancestors, one transfer per level (k_down_tree).

// v = E'^T x over the TPW tiles starting at tile t0 of one K x K transfer at B
// (warp-wide; x: K*NR values, any address space). A tile covers CPP whole columns of
// E', so the tiles of one transfer can be split over several warps, each writing the
// outputs of its own columns.
template <int K, int FMT, int NR, int TPW>
__device__ __forceinline__ void warp_transfer_t(const void* __restrict__ Bv, const typename Ar<FMT>::vec_t* x,
                                                typename Ar<FMT>::acc_t* v, int t0) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using mel_t = typename A::mel_t;
  using acc_t = typename A::acc_t;
  using ld_t = typename A::ld_t;
  constexpr int LPC = K / 8, CPP = 32 / LPC;
  constexpr int CH = TPW < LPC ? TPW : LPC;
  constexpr int V = A::V, P = 8 / V;
  const int lane = threadIdx.x & 31;
  const int rb = 8 * (lane % LPC), cl = lane / LPC;
  vec_t xt[8][NR];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < NR; ++j) xt[r][j] = x[(rb + r) * NR + j];
  const ld_t* B = (const ld_t*)Bv;
#pragma unroll 1
  for (int ch = 0; ch < TPW / CH; ++ch) {
    acc_t zc[CH][NR];
#pragma unroll
    for (int tt = 0; tt < CH; ++tt) {
      const int t = t0 + ch * CH + tt;
      mel_t m[8];
#pragma unroll
      for (int k = 0; k < P; ++k) {
        ld_t q = __ldg(B + (t * P + k) * 32 + lane);
        A::decode(q, m + k * V);
      }
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        acc_t zz = A::zero();
#pragma unroll
        for (int r = 0; r < 8; ++r) A::fma(zz, m[r], xt[r][j]);
        zc[tt][j] = zz;
      }
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      // butterfly over the CH tiles (lane keeps tile lane & (CH-1)), then the rest of
      // the LPC lanes that share a column
#pragma unroll
      for (int h = CH / 2; h >= 1; h >>= 1) {
        const bool up = (lane & h) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
          acc_t send = up ? zc[q][j] : zc[q + h][j];
          acc_t keep = up ? zc[q + h][j] : zc[q][j];
          A::add(keep, A::shfl(send, h));
          zc[q][j] = keep;
        }
      }
#pragma unroll
      for (int h = CH; h < LPC; h <<= 1) A::add(zc[0][j], A::shfl(zc[0][j], h));
      if ((lane % LPC) < CH) v[(cl + CPP * (t0 + ch * CH + (lane & (CH - 1)))) * NR + j] = zc[0][j];
    }
  }
}

// Splits one transfer's T tiles over `wpb` warps (a power of two): warp `sub` takes
// T / wpb consecutive tiles (warps beyond T do nothing).
template <int K, int FMT, int NR>
__device__ __forceinline__ void warp_transfer_t_part(const void* B, const typename Ar<FMT>::vec_t* x,
                                                     typename Ar<FMT>::acc_t* v, int wpb, int sub) {
  constexpr int T = K * K / 256;
  const int w = wpb < T ? wpb : T;
  if (sub >= w) return;
  const int tpw = T / w;
  if constexpr (T >= 16) if (tpw == 16) { warp_transfer_t<K, FMT, NR, 16>(B, x, v, 0); return; }
  if constexpr (T >= 8) if (tpw == 8) { warp_transfer_t<K, FMT, NR, 8>(B, x, v, sub * 8); return; }
  if constexpr (T >= 4) if (tpw == 4) { warp_transfer_t<K, FMT, NR, 4>(B, x, v, sub * 4); return; }
  if constexpr (T >= 2) if (tpw == 2) { warp_transfer_t<K, FMT, NR, 2>(B, x, v, sub * 2); return; }
  warp_transfer_t<K, FMT, NR, 1>(B, x, v, sub);
}

// s = rows of E' y over the tiles [t0, t1) of one K x K transfer at B (warp-wide;
// y: K*NR values, any address space); partial sums over those tiles' columns.
template <int K, int FMT, int NR>
__device__ __forceinline__ void warp_transfer(const void* __restrict__ Bv, const typename Ar<FMT>::vec_t* y,
                                              typename Ar<FMT>::acc_t* s, int t0, int t1) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using mel_t = typename A::mel_t;
  using acc_t = typename A::acc_t;
  using ld_t = typename A::ld_t;
  constexpr int LPC = K / 8, CPP = 32 / LPC;
  constexpr int V = A::V, P = 8 / V;
  const int lane = threadIdx.x & 31;
  const int rb = 8 * (lane % LPC), cl = lane / LPC;
  acc_t ya[8][NR];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < NR; ++j) ya[r][j] = A::zero();
  const ld_t* B = (const ld_t*)Bv;
#pragma unroll 4
  for (int t = t0; t < t1; ++t) {
    mel_t m[8];
#pragma unroll
    for (int k = 0; k < P; ++k) {
      ld_t q = __ldg(B + (t * P + k) * 32 + lane);
      A::decode(q, m + k * V);
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      const vec_t xv = y[(cl + CPP * t) * NR + j];
#pragma unroll
      for (int r = 0; r < 8; ++r) A::fma(ya[r][j], m[r], xv);
    }
  }
#pragma unroll
  for (int h = LPC; h < 32; h <<= 1)
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) A::add(ya[r][j], A::shfl(ya[r][j], h));
  if (lane < LPC)
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j) s[(rb + r) * NR + j] = ya[r][j];
}

// Upward pass from level `lb` (2^lb clusters, coefficients xc + slot0(lb) ..) to level `lt`,
// in one launch: CTA b maps clusters 2b and 2b + 1 of level lb to their parent; then one
// ticket per parent pair decides which CTA goes on: the first to arrive leaves its result in
// xc and ends, the second reads it and maps both to the next level. No CTA waits for another.
// A level takes two transfers on 8 warps (4 per transfer); eight clusters per CTA with a warp
// each, as before, kept 64 of the 152 SMs busy for 512 clusters and took a second launch.
// Bound by latency, about 2 us per level: 512 clusters of 64 over four levels (FP32, one
// column) 16 -> 10 us.
// With in.x the bottom coefficients come from the float64 input vector: the CTA writes them
// to xc for the block product and does the rest of VecIn's work. The tickets are zero
// between launches: the second arrival resets its own.
template <int K, int FMT, int NR>
__global__ void __launch_bounds__(256) k_up_tree(const char* __restrict__ epool, VecIn in,
                                                 typename Ar<FMT>::vec_t* xc, int lb, int lt, int ts,
                                                 unsigned* ticket) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using acc_t = typename A::acc_t;
  constexpr size_t kBlk = (size_t)K * K * (FMT == FMT_F32 ? 4 : 8);
  __shared__ acc_t v[2][K * NR];
  __shared__ vec_t xin[2][K * NR];
  __shared__ unsigned second;
  const int w = threadIdx.x >> 5;
  auto slot0 = [&](int l) { return (int64_t)((1 << l) - (1 << ts)); };
  int idx = blockIdx.x;                       // parent at level l - 1
  if (threadIdx.x == 0)
    for (int l = lb, i = idx; l > lt; --l, i >>= 1) {
      prefetch_l2_bulk(epool + (size_t)(slot0(l) + 2 * (int64_t)i) * kBlk, 2 * (unsigned)kBlk);
      if (i & 1) break;
    }
  chain_wait();
  vec_t* xb = xc + (slot0(lb) + 2 * (int64_t)idx) * K * NR;
  if (in.x) {
    bool go[NR];
    double be[NR];
    cg_beta<NR>(in, go, be);
    clear_regions(in);
#pragma unroll
    for (int j = 0; j < NR; ++j)
      for (int e = threadIdx.x; e < 2 * K; e += 256) {
        const int64_t i = 2 * (int64_t)idx * K + e;
        const vec_t o = A::from_d(cg_value(in, i + j * in.ldx, go[j], be[j]));
        xin[e / K][(e % K) * NR + j] = o;
        xb[e * NR + j] = o;
      }
  } else {
    for (int e = threadIdx.x; e < 2 * K * NR; e += 256) xin[e / (K * NR)][e % (K * NR)] = xb[e];
  }
  __syncthreads();
  for (int l = lb;; --l) {
    const int b = w >> 2;
    warp_transfer_t_part<K, FMT, NR>(epool + (size_t)(slot0(l) + 2 * (int64_t)idx + b) * kBlk, xin[b], v[b], 4, w & 3);
    __syncthreads();
    vec_t* out = xc + slot0(l - 1) * K * NR;
    for (int i = threadIdx.x; i < K * NR; i += 256) {
      acc_t t = v[0][i];
      A::add(t, v[1][i]);
      const vec_t o = A::out(t);
      out[(int64_t)idx * K * NR + i] = o;
      xin[idx & 1][i] = o;
    }
    if (l - 1 == lt) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned* t = ticket + slot0(l - 1) + (idx & ~1);
      second = atomicAdd(t, 1);
      if (second) *t = 0;
    }
    __syncthreads();
    if (!second) return;
    __threadfence();
    const int sib = idx ^ 1;
    for (int i = threadIdx.x; i < K * NR; i += 256) xin[sib & 1][i] = load_cg(out + (int64_t)sib * K * NR + i);
    idx >>= 1;
    __syncthreads();
  }
}

// part[j * CG_PARTS + CTA] = sum of v over the threads with threadIdx.x % NR == j (256 threads).
template <int NR>
__device__ __forceinline__ void column_partials(double v, double* __restrict__ part) {
  __shared__ double sh[8][NR];
  for (int o = 16; o >= NR; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) < NR) sh[threadIdx.x >> 5][threadIdx.x & 31] = v;
  __syncthreads();
  if (threadIdx.x < NR) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += sh[w][threadIdx.x];
    part[threadIdx.x * CG_PARTS + blockIdx.x] = s;
  }
}

// Downward pass from level lt to level lb (at most 5 levels): y_c = yrow_c + E'_c y_parent(c)
// (no transfer term at the coupling top level ts). A CTA owns S clusters of level lb; above
// the levels where they are S and S/2 clusters it follows one cluster per level, which the
// CTAs below that cluster all compute: one transfer on 8 warps is a step of about a
// microsecond, while a CTA per top cluster left most SMs idle (512 clusters, five levels:
// 17 -> 9 us; S = 4 only where S = 2 gives every SM several CTAs). ypar: coefficients of level
// lt - 1. The last level goes to yout (float64, column j at yout + j * ldo), when given, with
// the CTA's partial of pdot_j^T yout_j (leading dimension ldo) in part[j * CG_PARTS + CTA],
// else to yc.
template <int K, int FMT, int NR, int S>
__global__ void __launch_bounds__(256) k_down_tree(const char* __restrict__ epool,
                                                   const typename Ar<FMT>::yo_t* yrow,
                                                   const typename Ar<FMT>::vec_t* ypar,
                                                   typename Ar<FMT>::vec_t* yc, int lt, int lb, int ts,
                                                   double* yout, int64_t ldo,
                                                   const double* pdot, double* part) {
  using A = Ar<FMT>;
  using vec_t = typename A::vec_t;
  using acc_t = typename A::acc_t;
  constexpr size_t kBlk = (size_t)K * K * (FMT == FMT_F32 ? 4 : 8);
  constexpr int T = K * K / 256;
  __shared__ acc_t sv[8][K * NR];
  __shared__ vec_t ys[2][S][K * NR];            // this level's and the parents' coefficients
  const int w = threadIdx.x >> 5;
  auto slot0 = [&](int l) { return (int64_t)((1 << l) - (1 << ts)); };
  double dot = 0.0;
  const int nb = 1 << lb;
  if (threadIdx.x == 0)
    for (int l = lb, c = blockIdx.x * S, n = min(S, nb); l >= max(lt, ts + 1); --l, c >>= 1, n = max(1, n >> 1)) {
      prefetch_l2_bulk(epool + (size_t)(slot0(l) + c) * kBlk, n * (unsigned)kBlk);
      if (n == 1 && (c & 1)) break;
    }
  chain_wait();
  for (int c0 = blockIdx.x * S; c0 < nb; c0 += gridDim.x * S)
    for (int l = lt; l <= lb; ++l) {
      const int first = c0 >> (lb - l);                            // clusters first .. first + per - 1
      const int per = max(1, min(S >> (lb - l), (1 << l) - first));
      const int share = per <= 1 ? 8 : (per == 2 ? 4 : 2);         // warps per transfer,
      const int hold = share < T ? share : T;                      // of which hold tiles
      vec_t(*cur)[K * NR] = ys[l & 1];
      vec_t(*par)[K * NR] = ys[(l & 1) ^ 1];
      const int b = w / share, sub = w % share;
      if (l > ts && b < per && sub < hold) {
        const int c = first + b, tpw = T / hold;
        const vec_t* yp = l == lt ? ypar + (int64_t)(c >> 1) * K * NR : par[(c >> 1) - (first >> 1)];
        warp_transfer<K, FMT, NR>(epool + (size_t)(slot0(l) + c) * kBlk, yp, sv[w], sub * tpw, (sub + 1) * tpw);
      }
      __syncthreads();   // every parent value and partial of this level is in place
      const bool last = l == lb;
      for (int e = threadIdx.x; e < per * K * NR; e += 256) {
        const int bb = e / (K * NR), i = e % (K * NR);
        const int c = first + bb;
        acc_t acc = A::from_yo(yrow[(slot0(l) + c) * K * NR + i]);
        if (l > ts)
          for (int q = 0; q < hold; ++q) A::add(acc, sv[bb * share + q][i]);
        const vec_t o = A::out(acc);
        if (!last) {
          cur[bb][i] = o;
        } else if (yout) {
          const int a = i / NR, j = i % NR;      // j is the same for all of a thread's e: NR divides 256
          const int64_t at = (int64_t)c * K + a + j * ldo;
          const double q = A::to_d(o);
          yout[at] = q;
          if (pdot) dot = fma(pdot[at], q, dot);
        } else {
          yc[(slot0(l) + c) * K * NR + i] = o;
        }
      }
      __syncthreads();
    }
  if (pdot) column_partials<NR>(dot, part);
}

// natural column-major K x K blocks (float64) -> swizzled blocks in a format
__global__ void k_swizzle_blocks(const double* __restrict__ in, int K, void* __restrict__ out, int fmt) {
  int64_t b = blockIdx.x;
  int V = fmt == FMT_F32 ? 4 : 2, LPC = K / 8, CPP = 32 / LPC, P = 8 / V;
  for (int pos = threadIdx.x; pos < K * K; pos += blockDim.x) {
    int sub = pos % V, ln = (pos / V) % 32, tk = pos / (V * 32);
    int t = tk / P, k = tk % P;
    int i = 8 * (ln % LPC) + k * V + sub, j = t * CPP + ln / LPC;
    double v = in[b * K * K + i + (int64_t)j * K];
    int64_t idx = b * K * K + pos;
    if (fmt == FMT_F64) {
      ((double*)out)[idx] = v;
    } else if (fmt == FMT_DF) {
      float h = __double2float_rn(v);
      ((float2*)out)[idx] = make_float2(h, __double2float_rn(v - (double)h));
    } else {
      ((float*)out)[idx] = __double2float_rn(v);
    }
  }
}

// y(point) = yrowD + U y_hat(leaf), scattered to user order (column j at y + j*ldy), and, with
// pdot given, the CTA's partial of pdot_j^T y_j (as in k_down_tree). 256 / KD threads share
// each sum.
template <int FMT, class BT, int NR>
__global__ void __launch_bounds__(256) k_leaf_final(int KD, int KC, int nleaf,
                                                    const typename Ar<FMT>::yo_t* yrow,
                                                    const BT* __restrict__ U,
                                                    const typename Ar<FMT>::vec_t* yleaf,
                                                    const int* __restrict__ leafoff, const int* __restrict__ perm,
                                                    double* y, int64_t ldy,
                                                    const double* pdot, double* part) {
  using V = LeafVal<FMT>;
  using v_t = typename V::t;
  __shared__ v_t ps[64 * NR];
  __shared__ v_t red[256 * NR];
  const int i = threadIdx.x % KD, pt = threadIdx.x / KD, parts = 256 / KD;
  double dot = 0.0;
  if (U && threadIdx.x == 0) prefetch_l2_bulk(U + (int64_t)blockIdx.x * KD * KC, KD * KC * (unsigned)sizeof(BT));
  chain_wait();
  for (int l = blockIdx.x; l < nleaf; l += gridDim.x) {
    const int p0 = leafoff[l], nl = leafoff[l + 1] - p0;
    if (U) {
      for (int e = threadIdx.x; e < KC * NR; e += 256) ps[e] = V::in(yleaf[(int64_t)l * KC * NR + e]);
      __syncthreads();
      const BT* Ul = U + (int64_t)l * KD * KC + i;
      v_t acc[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) acc[j] = V::zero();
#pragma unroll 4
      for (int b = pt; b < KC; b += parts) {
        const double u = widen(Ul[b * KD]);
#pragma unroll
        for (int j = 0; j < NR; ++j) V::fma(acc[j], u, ps[b * NR + j]);
      }
#pragma unroll
      for (int j = 0; j < NR; ++j) red[(pt * KD + i) * NR + j] = acc[j];
      __syncthreads();
    }
    for (int e = threadIdx.x; e < nl * NR; e += 256) {
      v_t v = V::row(yrow[(int64_t)l * KD * NR + e]);
      if (U)
        for (int q = 0; q < parts; ++q) V::add(v, red[q * KD * NR + e]);
      const int64_t o = perm[p0 + e / NR] + (e % NR) * ldy;
      const double r = V::val(v);
      y[o] = r;
      if (pdot) dot = fma(pdot[o], r, dot);
    }
    __syncthreads();
  }
  if (pdot) column_partials<NR>(dot, part);
}

__global__ void k_transpose_blocks(const double* __restrict__ in, int R, int C, double* __restrict__ out) {
  // per block: in R x C column-major -> out C x R column-major
  int64_t b = blockIdx.x;
  for (int e = threadIdx.x; e < R * C; e += blockDim.x) {
    int i = e % R, j = e / R;
    out[b * R * C + j + (int64_t)i * C] = in[b * R * C + e];
  }
}
__global__ void k_transpose_blocks32(const float* __restrict__ in, int R, int C, float* __restrict__ out) {
  int64_t b = blockIdx.x;
  for (int e = threadIdx.x; e < R * C; e += blockDim.x) {
    int i = e % R, j = e / R;
    out[b * R * C + j + (int64_t)i * C] = in[b * R * C + e];
  }
}

// ----------------------------------------------------------------------------- host
struct OpHost {
  std::vector<int> rowptr, col;
  std::vector<int64_t> blk;     // block index in the pool of the entry
  std::vector<int> pool;        // 0: D/S pool, 1: P pool
  std::vector<int> rowof;
};

static int64_t upper_pos(const HostCSR& C, int t, int s, bool strict) {
  auto b = C.col.begin() + C.rowptr[t], e = C.col.begin() + C.rowptr[t + 1];
  auto it = std::lower_bound(b, e, s);
  if (it == e || *it != s) return -1;
  auto first = std::lower_bound(b, e, strict ? t + 1 : t);
  return it - first;
}

static std::vector<int64_t> ubase(const HostCSR& C, int nrows, bool strict) {
  std::vector<int64_t> ub(nrows + 1, 0);
  for (int t = 0; t < nrows; ++t) {
    int cnt = 0;
    for (int e = C.rowptr[t]; e < C.rowptr[t + 1]; ++e) cnt += strict ? (C.col[e] > t) : (C.col[e] >= t);
    ub[t + 1] = ub[t] + cnt;
  }
  return ub;
}

// Float64 blocks multiplied in fixed point: 16 x 16 blocks hold too few terms per scaled
// sum (8 per lane) to pay for their scaling.
static bool fx_product(int fmt, int K) { return fmt == FMT_F64 && K >= 32; }

static SymOp upload_op(Matrix& M, const OpHost& H, int K, const void* pool0, const void* pool1,
                       const void* pool0_32, const void* pool1_32, const std::vector<unsigned char>& skip) {
  SymOp op;
  op.K = K;
  op.nrows = (int)H.rowptr.size() - 1;
  op.nnz = (int)H.col.size();
  cudaStream_t s = M.stream;
  auto up = [&](const void* src, size_t bytes) {
    void* d = M.alloc(std::max<size_t>(bytes, 8));
    if (bytes) H2_CUDA(cudaMemcpyAsync(d, src, bytes, cudaMemcpyHostToDevice, s));
    return d;
  };
  op.rowptr = (int*)up(H.rowptr.data(), sizeof(int) * H.rowptr.size());
  op.col = (int*)up(H.col.data(), sizeof(int) * H.col.size());
  std::vector<const void*> p(op.nnz), p32(op.nnz);
  size_t b64 = (size_t)K * K * fmt_bytes(M.fmt), b32 = (size_t)K * K * 4;
  for (int e = 0; e < op.nnz; ++e) {
    p[e] = (const char*)(H.pool[e] ? pool1 : pool0) + H.blk[e] * b64;
    const void* q = H.pool[e] ? pool1_32 : pool0_32;
    p32[e] = q ? (const char*)q + H.blk[e] * b32 : nullptr;
  }
  op.blk = (const void**)up(p.data(), sizeof(void*) * p.size());
  op.blk32 = (const void**)up(p32.data(), sizeof(void*) * p32.size());
  int64_t noff = 0;
  std::vector<int> rowof(op.nnz);
  for (int t = 0; t < op.nrows; ++t)
    for (int e = H.rowptr[t]; e < H.rowptr[t + 1]; ++e) {
      noff += (H.col[e] != t);
      rowof[e] = t;
    }
  op.noff = noff;
  op.erow = (int*)up(rowof.data(), sizeof(int) * rowof.size());
  if (fx_product(M.fmt, K) && op.nnz > 0) {
    op.bexp = (short*)M.alloc(sizeof(short) * op.nnz);
    unsigned char* d_skip = nullptr;
    if (std::find(skip.begin(), skip.end(), 1) != skip.end()) d_skip = (unsigned char*)up(skip.data(), skip.size());
    { k_block_exponents<<<ceil_div(op.nnz, 8), 256, 0, s>>>(op.blk, op.erow, op.col, d_skip, op.nnz, K * K, op.bexp);
      ::h2mg::count_launch(); }
    H2_LAUNCH_CHECK();
    M.free_owned(d_skip);
  }
  H2_CUDA(cudaStreamSynchronize(s));   // the host lists go out of scope
  return op;
}

// Coupling rows of levels t*..top (+ the P_i blocks of level top when i >= 2).
static OpHost coupling_rows(const Matrix& M, int top, int i) {
  OpHost H;
  H.rowptr.push_back(0);
  for (int ell = M.tstar; ell <= top; ++ell) {
    const HostCSR& F = M.far[ell];
    auto ubF = ubase(F, 1 << ell, true);
    const HostCSR* Ip = (i >= 2 && ell == top) ? &M.inadm[ell] : nullptr;
    std::vector<int64_t> ubI;
    if (Ip) ubI = ubase(*Ip, 1 << ell, false);
    for (int t = 0; t < (1 << ell); ++t) {
      // merge far (strict upper) and close (upper incl. diagonal) columns
      std::vector<std::pair<int, std::pair<int, int64_t>>> ent;
      for (int e = F.rowptr[t]; e < F.rowptr[t + 1]; ++e)
        if (F.col[e] > t)
          ent.push_back({F.col[e], {0, M.s_level_base[ell] + ubF[t] + upper_pos(F, t, F.col[e], true)}});
      if (Ip)
        for (int e = Ip->rowptr[t]; e < Ip->rowptr[t + 1]; ++e)
          if (Ip->col[e] >= t) ent.push_back({Ip->col[e], {1, ubI[t] + upper_pos(*Ip, t, Ip->col[e], false)}});
      std::sort(ent.begin(), ent.end());
      for (auto& en : ent) {
        H.col.push_back(M.slot0(ell) + en.first);
        H.pool.push_back(en.second.first);
        H.blk.push_back(en.second.second);
      }
      H.rowptr.push_back((int)H.col.size());
    }
  }
  return H;
}

// Rows have natural scales: sqrt(w_i) off the diagonal, sqrt(A_ii) on it. Where they differ by
// more than 2^6 inside a cluster, one exponent per block or tile row would not carry the
// digits of the small ones, so everything that touches the cluster stays in float64: the
// close blocks of a leaf (either scale), and for the clusters of all levels (weights) the
// couplings, the coarse near fields and the dense expansion, whose orthonormal bases are
// then graded. Without the guard above the leaves, the middle row of a product with 3000
// points, a far field and weights over 24 decades was off by 1.6e-12 of itself (float64:
// 5.4e-16). So do clusters whose entries are all far too large or too small for the exponents
// of fixed point. The skeletons and bases themselves are made in float64. A sibling on its base's
// bases (Chebyshev) takes over the base's marks.
void mark_spread(Matrix& M, const Matrix* base) {
  const int L = M.L, nleaf = 1 << L;
  short4* d = (short4*)M.alloc(sizeof(short4) * nleaf);
  { k_leaf_spread<<<ceil_div(nleaf, 8), 256, 0, M.stream>>>(M.d_leafoff, M.d_dg, M.d_sw, nleaf, d); ::h2mg::count_launch(); }
  H2_LAUNCH_CHECK();
  std::vector<short4> h(nleaf);
  H2_CUDA(cudaMemcpyAsync(h.data(), d, sizeof(short4) * nleaf, cudaMemcpyDeviceToHost, M.stream));
  H2_CUDA(cudaStreamSynchronize(M.stream));
  M.free_owned(d);
  constexpr int BITS = 6;
  // scales of the entries that the tiles' exponents (FX_EMIN..FX_EMAX) carry with room to spare
  constexpr int LEAST = 400, MOST = 1700;
  std::vector<unsigned char> out(nleaf);                    // clusters with a leaf outside
  M.spread_leaf.assign(nleaf, 0);
  for (int j = 0; j < nleaf; ++j) {
    const int m = std::max<int>(h[j].y, 2 * h[j].w - 1023);
    out[j] = m < LEAST || m > MOST;
    M.spread_leaf[j] = out[j] || h[j].y - h[j].x > 2 * BITS || h[j].w - h[j].z > BITS;
  }
  if (base) {
    M.spread_slot = base->spread_slot;
    return;
  }
  M.spread_slot.assign(std::max(M.nslots(), 0), 0);
  if (M.tstar < 0) return;
  for (int ell = L; ell >= M.tstar; --ell) {
    for (int j = 0; j < (1 << ell); ++j) M.spread_slot[M.slot0(ell) + j] = out[j] || h[j].w - h[j].z > BITS;
    for (int j = 0; j < (1 << ell) / 2; ++j) {
      h[j].z = std::min(h[2 * j].z, h[2 * j + 1].z);
      h[j].w = std::max(h[2 * j].w, h[2 * j + 1].w);
      out[j] = out[2 * j] || out[2 * j + 1];
    }
  }
}

bool level_spread(const Matrix& M, int ell) {
  const auto b = M.spread_slot.begin() + M.slot0(ell);
  return std::find(b, b + (1 << ell), 1) != b + (1 << ell);
}

static void allow_fx_smem();

void setup_operators(Matrix& M) {
  cudaStream_t s = M.stream;
  if (M.fmt == FMT_F64) allow_fx_smem();
  const int L = M.L;
  // close part of level 1
  {
    OpHost H;
    const HostCSR& N = M.inadm[L];
    H.rowptr.push_back(0);
    int64_t b = 0;
    for (int t = 0; t < (1 << L); ++t) {
      for (int e = N.rowptr[t]; e < N.rowptr[t + 1]; ++e)
        if (N.col[e] >= t) {
          H.col.push_back(N.col[e]);
          H.blk.push_back(b++);
          H.pool.push_back(0);
        }
      H.rowptr.push_back((int)H.col.size());
    }
    M.opD = upload_op(M, H, M.KD, M.poolD.p, nullptr, M.poolD32.p, nullptr, M.spread_leaf);
    M.opD.spread = FX_SPREAD;
  }
  M.opC.assign(M.lev + 1, SymOp{});
  if (M.tstar >= 0) {
    for (int i = 1; i <= M.lev; ++i) {
      if (M.apply_only && i > 1) break;
      int top = (i == 1) ? L : L - i + 2;
      OpHost H = coupling_rows(M, top, i);
      const void* pP = (i >= 2) ? M.poolP[i].p : nullptr;
      const void* pP32 = (i >= 2 && M.with_f32) ? M.poolP32[i].p : nullptr;
      M.opC[i] = upload_op(M, H, M.KC, M.poolS.p, pP, M.with_f32 ? M.poolS32.p : nullptr, pP32,
                            M.spread_slot);
    }
    // transposed copies of the transfers and leaf bases (coalesced upward pass) and the
    // swizzled transfer pools; a sibling matrix already has its base's
    size_t nu = (size_t)(1 << L), ne = (size_t)M.nslots();
    if (!M.d_UT) {
      double* UT = (double*)M.alloc(sizeof(double) * nu * M.KD * M.KC);
      double* ET = (double*)M.alloc(sizeof(double) * ne * M.KC * M.KC);
      { k_transpose_blocks<<<(int)nu, 256, 0, s>>>(M.d_U, M.KD, M.KC, UT); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      { k_transpose_blocks<<<(int)ne, 256, 0, s>>>(M.d_E, M.KC, M.KC, ET); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      M.d_UT = UT;
      M.d_ET = ET;
      M.poolE.bytes = ne * M.KC * M.KC * fmt_bytes(M.fmt);
      M.poolE.p = M.alloc(M.poolE.bytes);
      { k_swizzle_blocks<<<(int)ne, 256, 0, s>>>(M.d_E, M.KC, M.poolE.p, M.fmt); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
    }
    if (M.with_f32) {
      M.poolE32.bytes = ne * M.KC * M.KC * 4;
      M.poolE32.p = M.alloc(M.poolE32.bytes);
      { k_swizzle_blocks<<<(int)ne, 256, 0, s>>>(M.d_E, M.KC, M.poolE32.p, FMT_F32); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      float* UT32 = (float*)M.alloc(sizeof(float) * nu * M.KD * M.KC);
      float* ET32 = (float*)M.alloc(sizeof(float) * ne * M.KC * M.KC);
      { k_transpose_blocks32<<<(int)nu, 256, 0, s>>>(M.d_U32, M.KD, M.KC, UT32); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      { k_transpose_blocks32<<<(int)ne, 256, 0, s>>>(M.d_E32, M.KC, M.KC, ET32); ::h2mg::count_launch(); }
      H2_LAUNCH_CHECK();
      M.d_UT32 = UT32;
      M.d_ET32 = ET32;
    }
  }
  // product workspaces hold up to NRMAX interleaved columns
  size_t ncoef = (size_t)std::max(M.nslots(), 1) * M.KC * NRMAX;
  size_t npts = (size_t)(1 << L) * M.KD * NRMAX;
  M.d_ticket = (unsigned*)M.alloc(sizeof(unsigned) * std::max(M.nslots(), 1));
  M.wx.p = M.alloc(8 * ncoef);
  M.wyrow.p = M.alloc(8 * ncoef);
  M.wyc.p = M.alloc(8 * ncoef);
  M.wxp.p = M.alloc(8 * npts);
  M.wyp.p = M.alloc(8 * npts);
  H2_CUDA(cudaStreamSynchronize(s));
}

// Fixed-point product: work in units of one chunk of an entry, dealt to CTAs of 8 warps;
// `waves` CTAs per SM in all (0: the default), fewer when there is less than one unit per
// warp. Float64 FMAs (k_bsgemv) take 2 x 4096 / 2 clocks of an SM per 64 x 64 block, where
// its 32 KB take 1500 at the copy bandwidth; in fixed point the encoding (22 operations a
// value) and the multiply-adds (6) keep the ALU pipe at 60% and the DRAM at 57% of its peak
// (30011 points, one column: 4.6 TB/s), with 16 resident warps (128 registers) as the limit;
// two columns (252 registers, 8 warps) 43% and 30%. Whole products of 65536 Gaussian points in
// the cube: one column 1.92 -> 0.91 ms, two 3.73 -> 1.73 ms; of 100003 points, one column,
// 4.38 -> 2.05 ms. CTAs per SM 4 / 8 / 16, one column: 16384 points 215 / 204 / 216 us, 30011
// 493 / 495 / 499, 65536 on the square 182 / 194 / 193.
//
// Relative error against the double-double product (mean of 8 normal vectors), float64 FMAs
// / here: Gaussian cube of 20000 points 3.7e-16 / 2.3e-16, of 65536 5.0e-16 / 2.3e-16, Matern
// 4.4e-16 / 2.6e-16, square 3.3e-16 / 2.8e-16, sphere 3.8e-16 / 2.7e-16, skeleton Gaussian
// 2.4e-16 / 2.8e-16 (rows of few blocks, which more warps now add into by atomics). With parts
// of 28 bits a column A e_j of 2000 Gaussian points was off by 4.0e-17 of its largest entry;
// now it is within 2^-55.7.
constexpr int FX_WAVES = 8;
template <int NR>
static void launch_bsgemv_fx(const SymOp& op, const double* x, double* yrow, int waves, cudaStream_t s) {
  const int nch = op.K == 64 ? 2 : 1;
  const int64_t units = (int64_t)op.nnz * nch;
  if (units == 0) return;
  const int64_t warps = (int64_t)(waves > 0 ? waves : FX_WAVES) * SMS * 8;
  const int per = (int)((units + warps - 1) / warps);
  const int grid = (int)((units + 8 * (int64_t)per - 1) / (8 * (int64_t)per));
  if (op.K == 64) {
    launch_chain(k_bsgemv_fx<64, NR>, grid, 256, fx_smem<64, NR>(), s, op.erow, op.col, op.blk, op.bexp, x, yrow, units,
                 per, op.spread);
  } else {
    launch_chain(k_bsgemv_fx<32, NR>, grid, 256, fx_smem<32, NR>(), s, op.erow, op.col, op.blk, op.bexp, x, yrow, units,
                 per, op.spread);
  }
}

// Once per matrix (setup_operators): the kernels' dynamic shared memory.
static void allow_fx_smem() {
  auto allow = [](const void* f, size_t bytes) {
    H2_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  };
  allow((const void*)k_bsgemv_fx<64, 1>, fx_smem<64, 1>());
  allow((const void*)k_bsgemv_fx<64, 2>, fx_smem<64, 2>());
  allow((const void*)k_bsgemv_fx<32, 1>, fx_smem<32, 1>());
  allow((const void*)k_bsgemv_fx<32, 2>, fx_smem<32, 2>());
}

template <int FMT, int NR>
static void launch_bsgemv(Matrix& M, const SymOp& op, bool f32, const void* x, void* yrow, cudaStream_t s,
                          int force_split = 0) {   // yrow: cleared by the caller
  using vt = typename Ar<FMT>::vec_t;
  using yt = typename Ar<FMT>::yo_t;
  if (op.nrows == 0) return;
  // CTAs per block row: the autotuner's choice, else enough CTAs to fill the GPU when
  // the operator has few block rows
  // the double-double product has no tuned value: the float64 one counts CTAs per SM
  int tuned = 0;
  if constexpr (FMT != FMT_DD) tuned = op.split[FMT][nr_index(NR)];
  const int waves = force_split > 0 ? force_split : tuned;   // CTAs per SM of the kernels that take warps by entry
  const int split = waves > 0 ? waves : split_heuristic(op.nrows);
  const int grid = op.nrows * split;
  const void* const* blk = f32 ? op.blk32 : op.blk;
  Profile& P = M.prof;
  const bool rec = P.on && (!P.f32_only || FMT == FMT_F32);
  if (rec && P.cap_ev) {
    // inside a graph capture: the records become event nodes of the graph
    H2_REQUIRE(2 * P.cap_next + 2 <= P.cap_ev->size(), H2MG_ERR_UNSUPPORTED, "graph profiling events exhausted");
    H2_CUDA(cudaEventRecordWithFlags((*P.cap_ev)[2 * P.cap_next], s, cudaEventRecordExternal));
  } else if (rec) {
    if (P.used * 2 + 2 > P.ev.size()) {
      for (int i = 0; i < 64; ++i) {
        cudaEvent_t e;
        H2_CUDA(cudaEventCreate(&e));
        P.ev.push_back(e);
      }
    }
    H2_CUDA(cudaEventRecord(P.ev[2 * P.used], s));
  }
  if constexpr (FMT == FMT_F64) {
    if (op.bexp) launch_bsgemv_fx<NR>(op, (const double*)x, (double*)yrow, waves, s);
  }
  if (op.bexp && FMT == FMT_F64) {
  } else if (op.K == 64) {
    if constexpr (FMT != FMT_F64) {
      // The warps' first blocks are asked for ahead (about 80 MB over the first wave of CTAs). One
      // column: only where the previous kernel runs beside it, and not for operators of several
      // times the L2, whose other blocks then miss it. Per FP32 CG step, without / with: level 2
      // of 8000 points (0.10 GB) 39.5 / 35.1 us, of 16384 (0.31 GB) 76.2 / 73.3, of 20000 (0.85
      // GB) 162.7 / 166.7, of 40000 (1.8 GB) 313.7 / 320.3; level 1, two operators in turn, of
      // 8000 (36 MB) 58.4 / 52.5, of 16384 (0.13 and 0.18 GB) 96.1 / 99.6, of 20000 (0.54 GB) 195 /
      // 203. The line lies between the level-2 operators of 0.31 and 0.85 GB.
      const double bytes = (double)op.nnz * 4096 * (FMT == FMT_F32 ? 4 : 8);
      const bool first = NR >= 2 || (bytes <= 512e6 && chained(s));
      launch_chain(k_bsgemv<64, FMT, NR>, grid, 256, 0, s, op.rowptr, op.col, blk, (const vt*)x, (yt*)yrow, split, first);
    }
  } else if (op.nnz > 0) {
    const int64_t warps = (int64_t)(waves > 0 ? waves : FX_WAVES) * SMS * 8;
    const int per = (int)((op.nnz + warps - 1) / warps);
    const int g = ceil_div(op.nnz, 8 * (int64_t)per);
    if (op.K == 16) {
      launch_chain(k_bsgemv_small<16, FMT, NR>, g, 256, 0, s, op.erow, op.col, blk, (const vt*)x, (yt*)yrow, op.nnz, per);
    } else if constexpr (FMT != FMT_F64) {
      launch_chain(k_bsgemv_small<32, FMT, NR>, g, 256, 0, s, op.erow, op.col, blk, (const vt*)x, (yt*)yrow, op.nnz, per);
    }
  }
  H2_LAUNCH_CHECK();
  if (rec && P.cap_ev) {
    H2_CUDA(cudaEventRecordWithFlags((*P.cap_ev)[2 * P.cap_next + 1], s, cudaEventRecordExternal));
    P.cap_next++;
    P.cap_bytes->push_back((double)op.bytes(FMT == FMT_F32 ? 4 : 8, sizeof(vt) * NR));
  } else if (rec) {
    H2_CUDA(cudaEventRecord(P.ev[2 * P.used + 1], s));
    P.used++;
    P.bytes.push_back((double)op.bytes(FMT == FMT_F32 ? 4 : 8, sizeof(vt) * NR));
  }
}

// Upward pass from tree level `lb` to level `ts`. `in` (optional): the work of the product's
// first kernel, which this launch takes over.
template <int FMT, int NR>
static void pass_up(const Matrix& M, const char* epool, void* xc, int lb, int ts, unsigned* ticket, cudaStream_t s,
                    const VecIn* in = nullptr) {
  using vt = typename Ar<FMT>::vec_t;
  const int KC = M.KC;
  vt* x = (vt*)xc;
  if (lb == ts) {
    if (!in) return;
    const int64_t n = (int64_t)(1 << lb) * KC;
    launch_chain(k_coef_in<FMT, NR>, std::min(ceil_div(n, 256), 1024), 256, 0, s, *in, n, x);
    H2_LAUNCH_CHECK();
    return;
  }
  const VecIn vi = in ? *in : VecIn{};
  const int grid = 1 << (lb - 1);
  switch (KC) {
    case 16: launch_chain(k_up_tree<16, FMT, NR>, grid, 256, 0, s, epool, vi, x, lb, ts, ts, ticket); break;
    case 32: launch_chain(k_up_tree<32, FMT, NR>, grid, 256, 0, s, epool, vi, x, lb, ts, ts, ticket); break;
    default: launch_chain(k_up_tree<64, FMT, NR>, grid, 256, 0, s, epool, vi, x, lb, ts, ts, ticket); break;
  }
  H2_LAUNCH_CHECK();
}

// Downward pass from the coupling top level ts to level `lbot`, up to 5 levels per
// launch (the first launch takes the odd ones); the last level goes to yout (when given)
// instead of the coefficient buffer, with partials of pdot^T yout. Returns the last launch's
// CTAs. Two clusters per CTA where four would leave SMs without one: per FP32 CG step on level
// 2, S = 2 / 4: 256 clusters 72.9 / 73.7 us, 512 162.8 / 161.3, 1024 316.9 / 313.4.
constexpr int DOWN_LEVELS = 5;
template <int FMT, int NR>
static int pass_down(const Matrix& M, const char* epool, const void* yrow, void* yc, int ts, int lbot, double* yout,
                     int64_t ldo, const double* pdot, double* part, cudaStream_t s) {
  using vt = typename Ar<FMT>::vec_t;
  using yt = typename Ar<FMT>::yo_t;
  const int KC = M.KC;
  int grid = 0;
  for (int lt = ts; lt <= lbot;) {
    const int lb = lt + (lbot - lt) % DOWN_LEVELS;
    const vt* ypar = lt > ts ? (const vt*)yc + (size_t)M.slot0(lt - 1) * KC * NR : nullptr;
    const bool last = lb == lbot;
    double* yo = last ? yout : nullptr;
    const double* pd = last ? pdot : nullptr;
    const int S = (1 << lb) >= 4 * SMS ? 4 : 2;
    grid = std::min(std::max(1, (1 << lb) / S), CG_PARTS);
    auto go = [&](auto kernel) {
      launch_chain(kernel, grid, 256, 0, s, epool, (const yt*)yrow, ypar, (vt*)yc, lt, lb, ts, yo, ldo, pd, part);
    };
    switch (KC) {
      case 16: S == 4 ? go(k_down_tree<16, FMT, NR, 4>) : go(k_down_tree<16, FMT, NR, 2>); break;
      case 32: S == 4 ? go(k_down_tree<32, FMT, NR, 4>) : go(k_down_tree<32, FMT, NR, 2>); break;
      default: S == 4 ? go(k_down_tree<64, FMT, NR, 4>) : go(k_down_tree<64, FMT, NR, 2>); break;
    }
    H2_LAUNCH_CHECK();
    lt = lb + 1;
  }
  return grid;
}

// y = A_i x for NR columns (x, y column-major with leading dimensions ldx, ldy). With `cg`,
// x is the CG direction, formed by the first kernel, and the last one leaves partials of
// x^T y: returns their number.
template <int FMT, class BT, int NR>
static int apply_impl(Matrix& M, int i, const double* x, int64_t ldx, double* y, int64_t ldy, cudaStream_t s,
                      const BT* U, const BT* UT, const ApplyWork* ws = nullptr, const CgStep* cg = nullptr) {
  using vt = typename Ar<FMT>::vec_t;
  using yt = typename Ar<FMT>::yo_t;
  const int L = M.L, KC = M.KC, KD = M.KD, ts = M.tstar;
  const bool f32 = (FMT == FMT_F32);
  vt* xc = (vt*)(ws ? ws->xc : M.wx.p);
  yt* yr = (yt*)(ws ? ws->yr : M.wyrow.p);
  vt* yc = (vt*)(ws ? ws->yc : M.wyc.p);
  const char* epool = (const char*)(FMT == FMT_F32 ? M.poolE32.p : M.poolE.p);
  auto cslot = [&](int ell) { return (size_t)M.slot0(ell) * KC * NR; };   // first element of a level
  VecIn in{};
  in.x = x;
  in.ldx = ldx;
  const double* pdot = nullptr;
  double* part = nullptr;
  if (cg) {
    in.r = cg->r;             // null: x is the direction already
    in.prr = cg->prr;
    in.np = cg->nprr;
    in.par = cg->par;
    in.st = cg->st;
    pdot = x;
    part = cg->ppq;
  }
  // the row sums of the levels in use: K * NR elements of 4, 8 or 16 bytes per slot
  if (ts >= 0) {
    in.zero[0] = (uint4*)yr;
    in.nzero[0] = (int64_t)((1 << ((i == 1 ? L : L - i + 2) + 1)) - (1 << ts)) * KC * NR * sizeof(yt) / 16;
  }
  if (i == 1) {
    vt* xp = (vt*)(ws ? ws->xp : M.wxp.p);
    yt* yp = (yt*)(ws ? ws->yp : M.wyp.p);
    in.zero[1] = (uint4*)yp;
    in.nzero[1] = (int64_t)(1 << L) * KD * NR * sizeof(yt) / 16;
    // level 1 keeps the upward pass's tickets in the downward pass's buffer, which is idle
    // until then, so that a product in a caller's workspace uses nothing of the handle
    unsigned* ticket = (unsigned*)yc;
    in.zero[2] = (uint4*)ticket;
    in.nzero[2] = ts >= 0 ? ((int64_t)M.nslots() * sizeof(unsigned) + 15) / 16 : 0;
    const int grid = std::min(1 << L, LEAF_CTAS);
    launch_chain(k_leaf_in<FMT, BT, NR>, grid, 256, 0, s, in, ts >= 0 ? UT : nullptr, KD, KC, 1 << L, M.d_leafoff, M.d_perm, xp,
                                                  ts >= 0 ? xc + cslot(L) : nullptr);
    H2_LAUNCH_CHECK();
    if (ts >= 0) pass_up<FMT, NR>(M, epool, xc, L, ts, ticket, s);
    launch_bsgemv<FMT, NR>(M, M.opD, f32, xp, yp, s);
    if (ts >= 0) {
      launch_bsgemv<FMT, NR>(M, M.opC[1], f32, xc, yr, s);
      pass_down<FMT, NR>(M, epool, yr, yc, ts, L, nullptr, 0, nullptr, nullptr, s);
    }
    launch_chain(k_leaf_final<FMT, BT, NR>, grid, 256, 0, s, KD, KC, 1 << L, yp, ts >= 0 ? U : nullptr,
                                                     ts >= 0 ? yc + cslot(L) : nullptr, M.d_leafoff, M.d_perm, y, ldy,
                                                     pdot, part);
    H2_LAUNCH_CHECK();
    return grid;
  }
  const int m = L - i + 2;
  pass_up<FMT, NR>(M, epool, xc, m, ts, M.d_ticket, s, &in);
  launch_bsgemv<FMT, NR>(M, M.opC[i], f32, xc, yr, s);
  return pass_down<FMT, NR>(M, epool, yr, yc, ts, m, y, ldy, pdot, part, s);
}

template <int FMT, class BT>
static int apply_cols(Matrix& M, int i, const double* x, int64_t ldx, double* y, int64_t ldy, int nr,
                      cudaStream_t s, const BT* U, const BT* UT, const CgStep* cg) {
  int c = 0, np = 0;
  while (c < nr) {
    int left = nr - c;
    CgStep g{};
    if (cg) g = cg->columns_from(c, ldx);
    const CgStep* gp = cg ? &g : nullptr;
    if constexpr (FMT == FMT_F32) {
      if (left >= 4) {
        np = apply_impl<FMT, BT, 4>(M, i, x + c * ldx, ldx, y + c * ldy, ldy, s, U, UT, nullptr, gp);
        c += 4;
        continue;
      }
    }
    if (left >= 2) {
      np = apply_impl<FMT, BT, 2>(M, i, x + c * ldx, ldx, y + c * ldy, ldy, s, U, UT, nullptr, gp);
      c += 2;
    } else {
      np = apply_impl<FMT, BT, 1>(M, i, x + c * ldx, ldx, y + c * ldy, ldy, s, U, UT, nullptr, gp);
      c += 1;
    }
  }
  return np;
}

static int apply_any(Matrix& M, int i, bool f32, const double* x, int64_t ldx, double* y, int64_t ldy, int nr,
                     cudaStream_t s, const CgStep* cg) {
  if (f32) {
    H2_REQUIRE(M.with_f32, H2MG_ERR_INVALID_ARG, "matrix was built without an FP32 copy");
    return apply_cols<FMT_F32, float>(M, i, x, ldx, y, ldy, nr, s, M.d_U32, M.d_UT32, cg);
  }
  if (M.fmt == FMT_DF) return apply_cols<FMT_DF, double>(M, i, x, ldx, y, ldy, nr, s, M.d_U, M.d_UT, cg);
  return apply_cols<FMT_F64, double>(M, i, x, ldx, y, ldy, nr, s, M.d_U, M.d_UT, cg);
}

// Y = A_i X for nr columns; columns go through the block products NR at a time
// (4 for the FP32 copy, 2 for float64 / double-float), each block read once per group.
void apply_level_multi(Matrix& M, int i, bool f32, const double* x, int64_t ldx, double* y, int64_t ldy, int nr,
                       cudaStream_t s) {
  apply_any(M, i, f32, x, ldx, y, ldy, nr, s, nullptr);
}

int apply_cg_step(Matrix& M, int i, bool f32, double* p, double* q, int64_t ld, int nr, const CgStep& cg,
                  cudaStream_t s) {
  return apply_any(M, i, f32, p, ld, q, ld, nr, s, &cg);
}

void apply_level(Matrix& M, int i, bool f32, const double* x, double* y, cudaStream_t s) {
  int64_t n = level_size(M, i);
  apply_level_multi(M, i, f32, x, n, y, n, 1, s);
}

// y = A x at level 1 from the float64 blocks with double-double vectors and sums (one
// column): the outer residual b - A x of a solve whose x is much larger than b, where
// the float64 sum would round at the level of the residual itself.
void apply_level1_dd(Matrix& M, const double* x, double* y, cudaStream_t s) {
  H2_REQUIRE(M.fmt == FMT_F64, H2MG_ERR_INVALID_ARG, "the double-double product needs float64 storage");
  apply_impl<FMT_DD, double, 1>(M, 1, x, M.n, y, M.n, s, M.d_U, M.d_UT);
}

// Level-1 product in the primary format with caller-supplied workspace (the
// handle's own buffers are not touched).
void apply_level1_ws(Matrix& M, const double* x, double* y, cudaStream_t s, const ApplyWork& ws) {
  if (M.fmt == FMT_DF)
    apply_impl<FMT_DF, double, 1>(M, 1, x, M.n, y, M.n, s, M.d_U, M.d_UT, &ws);
  else
    apply_impl<FMT_F64, double, 1>(M, 1, x, M.n, y, M.n, s, M.d_U, M.d_UT, &ws);
}

// Bytes of each workspace region of the level-1 product.
void apply_level1_ws_sizes(const Matrix& M, size_t* coef, size_t* pts) {
  *coef = 8 * (size_t)std::max(M.nslots(), 1) * M.KC;
  *pts = 8 * (size_t)(1 << M.L) * M.KD;
}

// ----------------------------------------------------------------------------- autotuner
// Times `reps` launches of one block product with launch shape `split` on the handle's
// workspaces. The vector is cleared: the float64 product takes its arithmetic from the data,
// and zeros take the usual one (earlier contents can be NaN or the halves of other formats).
template <int FMT, int NR>
static float time_product(Matrix& M, SymOp& op, bool pts, int split, int reps, cudaStream_t s, cudaEvent_t e0,
                          cudaEvent_t e1) {
  const bool f32 = FMT == FMT_F32;
  void* x = pts ? M.wxp.p : M.wx.p;
  void* y = pts ? M.wyp.p : M.wyrow.p;
  H2_CUDA(cudaMemsetAsync(x, 0, sizeof(typename Ar<FMT>::vec_t) * (size_t)op.nrows * op.K * NR, s));
  H2_CUDA(cudaMemsetAsync(y, 0, sizeof(typename Ar<FMT>::yo_t) * (size_t)op.nrows * op.K * NR, s));
  launch_bsgemv<FMT, NR>(M, op, f32, x, y, s, split);   // warm-up
  H2_CUDA(cudaEventRecord(e0, s));
  for (int r = 0; r < reps; ++r) launch_bsgemv<FMT, NR>(M, op, f32, x, y, s, split);
  H2_CUDA(cudaEventRecord(e1, s));
  H2_CUDA(cudaEventSynchronize(e1));
  float ms = 0.f;
  H2_CUDA(cudaEventElapsedTime(&ms, e0, e1));
  return ms / reps;
}

template <int FMT, int NR>
static void tune_one(Matrix& M, SymOp& op, bool pts, int opi, cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1,
                     std::vector<double>& rep) {
  if (op.nrows == 0 || op.nnz == 0) return;
  const bool fx = op.K < 64 || (FMT == FMT_F64 && op.bexp);   // a candidate is the CTAs per SM of the launch
  const int heur = fx ? FX_WAVES : split_heuristic(op.nrows);
  const int cands[] = {1, 2, 4, 8, 16, 32, 64};
  const float base = time_product<FMT, NR>(M, op, pts, heur, 3, s, e0, e1);
  float best = base;
  int bs = heur;
  for (int c : cands) {
    if (c == heur || (!fx && (int64_t)op.nrows * c > (1 << 22))) continue;
    if (!fx && c > 1 && op.nnz < op.nrows * c) continue;       // more CTAs than blocks: idle CTAs
    const float t = time_product<FMT, NR>(M, op, pts, c, 3, s, e0, e1);
    if (t < best) {
      best = t;
      bs = c;
    }
  }
  op.split[FMT][nr_index(NR)] = bs;
  rep.insert(rep.end(), {(double)opi, (double)NR, (double)base, (double)best});
}

// Every operator of the hierarchy (index 0 = the close part of level 1, i = the
// coupling operator of level i), in the primary format for 1 and 2 columns and, with
// an FP32 copy, in FP32 for 1, 2 and 4 columns.
int autotune_products(Matrix& M, cudaStream_t s, double* out, int cap) {
  H2_REQUIRE(!M.prof.on, H2MG_ERR_INVALID_ARG, "stop h2mg_profile before tuning");
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  H2_CUDA(cudaEventCreate(&e0));
  H2_CUDA(cudaEventCreate(&e1));
  std::vector<double> rep;
  try {
    for (int oi = 0; oi < (int)M.opC.size(); ++oi) {
      SymOp& op = oi == 0 ? M.opD : M.opC[oi];
      const bool pts = oi == 0;
      if (M.fmt == FMT_DF) {
        tune_one<FMT_DF, 1>(M, op, pts, oi, s, e0, e1, rep);
        tune_one<FMT_DF, 2>(M, op, pts, oi, s, e0, e1, rep);
      } else {
        tune_one<FMT_F64, 1>(M, op, pts, oi, s, e0, e1, rep);
        tune_one<FMT_F64, 2>(M, op, pts, oi, s, e0, e1, rep);
      }
      if (M.with_f32 && op.blk32) {
        tune_one<FMT_F32, 1>(M, op, pts, oi, s, e0, e1, rep);
        tune_one<FMT_F32, 2>(M, op, pts, oi, s, e0, e1, rep);
        tune_one<FMT_F32, 4>(M, op, pts, oi, s, e0, e1, rep);
      }
    }
  } catch (...) {
    best_effort(cudaEventDestroy(e0), "cudaEventDestroy (tune)");
    best_effort(cudaEventDestroy(e1), "cudaEventDestroy (tune)");
    throw;
  }
  best_effort(cudaEventDestroy(e0), "cudaEventDestroy (tune)");
  best_effort(cudaEventDestroy(e1), "cudaEventDestroy (tune)");
  const int n = (int)rep.size() / 4;
  if (out)
    for (int k = 0; k < std::min(n, cap); ++k)
      for (int j = 0; j < 4; ++j) out[4 * k + j] = rep[4 * k + j];
  return n;
}

// Algorithmic bytes of one A_i apply in the primary format: every stored block once,
// the transfers (and leaf bases at i = 1) twice, the input and output vectors once.
int64_t apply_bytes(const Matrix& M, int i) {
  int64_t eb = fmt_bytes(M.fmt);
  int64_t bytes = 0;
  if (i == 1) {
    bytes += (int64_t)M.opD.nnz * M.KD * M.KD * eb + 2 * 8 * M.n;
    if (M.tstar >= 0) {
      bytes += (int64_t)M.opC[1].nnz * M.KC * M.KC * eb;
      bytes += 2 * 8 * ((int64_t)(1 << M.L) * M.KD * M.KC);
      for (int ell = M.tstar + 1; ell <= M.L; ++ell) bytes += 2 * 8 * ((int64_t)(1 << ell) * M.KC * M.KC);
    }
    return bytes;
  }
  int m = M.L - i + 2;
  bytes += (int64_t)M.opC[i].nnz * M.KC * M.KC * eb + 2 * 8 * ((int64_t)(1 << m) * M.KC);
  for (int ell = M.tstar + 1; ell <= m; ++ell) bytes += 2 * 8 * ((int64_t)(1 << ell) * M.KC * M.KC);
  return bytes;
}

}  // namespace h2mg
