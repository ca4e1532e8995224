// fx_tile.cuh -- 64 x 64 x 64 float64 products on the integer pipe (see fixed.cuh), by CTAs
// of 256 threads.
//
// Operands P (a, k) and Q (b, k) are 64 x 64 tiles in shared memory, encoded with one
// exponent per row, so that element (a, b) of P Q^T has the exact integer sum of its 64
// terms and the scale of row a and row b; inputs are rounded at 2^-57 of the scale of their
// row (up to twice its largest magnitude). 3 integer multiply-adds stand in for one float64
// FMA, at up to 57 against 2 per clock and SM (this pattern from registers, 8 warps; with the
// reads and the encoding a product takes 35 to 43 k clocks of an SM, 131 k on the float64
// pipe). Thread (ti, tj) = (tid / 16, tid % 16) owns rows 4 ti .. + 3 of P and rows tj + 16 q
// of Q: per k it reads 8 values for 48 multiply-adds.
#pragma once

#include "fixed.cuh"

namespace h2mg {

constexpr int FXT = 64;                                  // tile edge
constexpr int FXLD = FXT + 1;                            // row stride of a tile, in values
constexpr size_t FX_TILE_BYTES = sizeof(Fx) * FXT * FXLD;
constexpr size_t FX_PAIR_BYTES = 2 * FX_TILE_BYTES + 2 * FXT * sizeof(int);

struct FxPair {                                          // the operands in dynamic shared memory
  Fx *P, *Q;
  int *ep, *eq;                                          // exponents of their rows
  __device__ explicit FxPair(void* sm)
      : P((Fx*)sm), Q(P + FXT * FXLD), ep((int*)(Q + FXT * FXLD)), eq(ep + FXT) {}
};

struct FxAcc {
  int64_t hh[4][4], mid[4][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        hh[r][q] = 0;
        mid[r][q] = fx_half();
      }
  }
};

__device__ __forceinline__ int fx_a() { return (threadIdx.x >> 4) * 4; }      // first row of P of this thread
__device__ __forceinline__ int fx_b() { return threadIdx.x & 15; }            // first row of Q

// Encodes a tile whose element (row, k) is load(row, k); thread t asks for row t % 64 and
// k = t / 64 + 4 q, so consecutive threads read consecutive rows. Exponents above
// FX_EMAX (Inf, NaN) make the row's products NaN. Callers synchronise before and after.
template <class F>
__device__ __forceinline__ void fx_tile_load(Fx* T, int* ex, F load) {
  const int r = threadIdx.x & 63, k0 = threadIdx.x >> 6;
  if (threadIdx.x < FXT) ex[threadIdx.x] = FX_EMIN;
  double v[16];
  int m = 0;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    v[q] = load(r, k0 + 4 * q);
    m = max(m, fx_exponent(v[q]));
  }
  __syncthreads();
  atomicMax(ex + r, m);
  __syncthreads();
  const int E = ex[r];
#pragma unroll
  for (int q = 0; q < 16; ++q) T[(k0 + 4 * q) * FXLD + r] = fx_encode_even(v[q], E);
}

// The same with k along consecutive threads: thread t asks for k = t % 64 and rows t / 64 +
// 4 q. `margin` extra bits of headroom (1 for sums of 128 terms); `other(row, k)`, if the
// exponents are to cover a second tile too, is that tile's element.
struct FxNoOther {
  __device__ double operator()(int, int) const { return 0.0; }
};
template <class F, class G = FxNoOther>
__device__ __forceinline__ void fx_tile_load_k(Fx* T, int* ex, F load, int margin = 0, G other = G()) {
  const int k = threadIdx.x & 63, r0 = threadIdx.x >> 6;
  if (threadIdx.x < FXT) ex[threadIdx.x] = FX_EMIN;
  __syncthreads();
  double v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    v[q] = load(r0 + 4 * q, k);
    const int m = __reduce_max_sync(0xffffffffu, max(fx_exponent(v[q]), fx_exponent(other(r0 + 4 * q, k))));
    if ((threadIdx.x & 31) == 0) atomicMax(ex + r0 + 4 * q, m + margin);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 16; ++q) T[k * FXLD + r0 + 4 * q] = fx_encode_even(v[q], ex[r0 + 4 * q]);
}

// c += P Q^T.
__device__ __forceinline__ void fx_tile_mma(const FxPair& t, FxAcc& c) {
  const Fx* P = t.P + fx_a();
  const Fx* Q = t.Q + fx_b();
#pragma unroll 2
  for (int k = 0; k < FXT; ++k) {
    Fx p[4], q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      p[i] = P[k * FXLD + i];
      q[i] = Q[k * FXLD + 16 * i];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        fx_mad(c.hh[r][j], p[r].h, q[j].h);
        fx_mad(c.mid[r][j], p[r].h, q[j].l);
        fx_mad(c.mid[r][j], p[r].l, q[j].h);
      }
  }
}

// 2^(E - 1050): the two rows' scales multiply a joined sum one after the other.
__device__ __forceinline__ double fx_row_scale(int E) {
  return E > FX_EMAX ? __hiloint2double(0x7FF80000, 0) : __hiloint2double((E - 27) << 20, 0);
}

// Encodes a product as the next one's operand Q (b, k): element (a, b) of this thread's
// values becomes k = a of row b. Callers synchronise before (P and Q are idle) and after.
__device__ __forceinline__ void fx_tile_store_q(Fx* T, int* ex, const double (&v)[4][4]) {
  if (threadIdx.x < FXT) ex[threadIdx.x] = FX_EMIN;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int m = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) m = max(m, fx_exponent(v[r][q]));
    atomicMax(ex + fx_b() + 16 * q, m);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int b = fx_b() + 16 * q, E = ex[b];
#pragma unroll
    for (int r = 0; r < 4; ++r) T[(fx_a() + r) * FXLD + b] = fx_encode_even(v[r][q], E);
  }
}

// Element (fx_a() + r, fx_b() + 16 q) of P Q^T.
__device__ __forceinline__ double fx_value(const FxPair& t, const FxAcc& c, int r, int q) {
  return (double)fx_join(c.hh[r][q], c.mid[r][q]) * fx_row_scale(t.ep[fx_a() + r]) *
         fx_row_scale(t.eq[fx_b() + 16 * q]);
}

// All elements of this thread.
__device__ __forceinline__ void fx_values(const FxPair& t, const FxAcc& c, double (&v)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) v[r][q] = fx_value(t, c, r, q);
}

}  // namespace h2mg
