// Device helpers shared by the kernels of the library: complex arithmetic on
// double-float and float2, and deterministic block / grid reductions.
#pragma once

#include <cuda_runtime.h>

#include "gps_internal.h"

namespace gps {

// Double-float number: the unevaluated sum hi + lo of two floats, about 48
// significant bits.  Arithmetic by error-free transformations (Knuth's
// TwoSum, FMA-based TwoProd) runs on the FP32 pipe, which on this GPU issues
// 64x the FP64 rate.  Neither addition nor multiplication
// renormalizes its result: hi is the rounded result of the hi parts and lo
// collects the exact error terms, so each operation's error stays bounded by
// a small multiple of u^2 (|a| + |b|) or u^2 |a||b| (u = 2^-24), the
// norm-wise bound an FFT's error analysis needs, while |lo| may reach a few
// ulps of hi along a chain of butterflies.
using ::fma;

struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ explicit constexpr df(double d)
      : hi((float)d), lo((float)(d - (double)(float)d)) {}
  __host__ __device__ explicit constexpr df(int i) : df((double)i) {}
  __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
};

// Addition without the final renormalization: the TwoSum of the hi parts is
// exact for any operands, so hi + lo stays the sum to within the rounding of
// the lo parts.  In the FFT passes an element goes through a few additions
// and at most one product per stage, so lo grows by a few ulps of hi and the
// norm-wise error bound keeps its u^2 order (tested: df64 spectra match the
// FP64 oracle to 1e-12).
// The operations are the rounding intrinsics, which the compiler does not
// contract: an FMA in place of a product and a sum of an error-free
// transformation counts the product's rounding error twice, which leaves FP32
// accuracy (seen once in the radix-2 last stage of a 128-point transform).
__device__ __forceinline__ float df_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ df operator+(df a, df b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = df_sub(s, a.hi);
  const float e = __fadd_rn(df_sub(a.hi, df_sub(s, bb)), df_sub(b.hi, bb));   // TwoSum error of hi parts
  return df(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
// Product without the final renormalization, like operator+: hi is the
// rounded product of the hi parts, lo its exact TwoProd error plus the cross
// terms, so hi + lo is the product to within u^2 |a||b| while lo may exceed
// half an ulp of hi (by the few ulps that a chain of butterflies adds).
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);                     // TwoProd error
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return df(p, e);
}
// a b + s c d (s = +1 or -1) as one double-float: the TwoSum of the two hi
// products, their TwoProd errors and the four cross terms accumulated in the
// low part (16 FP32 operations against 22 for two products and a sum).
template <int S>
__device__ __forceinline__ df df_dot2(df a, df b, df c, df d) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float q = S > 0 ? __fmul_rn(c.hi, d.hi) : -__fmul_rn(c.hi, d.hi);
  const float e1 = fmaf(a.hi, b.hi, -p);
  const float e2 = S > 0 ? fmaf(c.hi, d.hi, -q) : fmaf(-c.hi, d.hi, -q);
  const float s = __fadd_rn(p, q);
  const float bb = df_sub(s, p);
  float lo = __fadd_rn(df_sub(p, df_sub(s, bb)), df_sub(q, bb));   // TwoSum error of p + q
  lo = __fadd_rn(lo, __fadd_rn(e1, e2));
  lo = fmaf(a.hi, b.lo, lo);
  lo = fmaf(a.lo, b.hi, lo);
  lo = S > 0 ? fmaf(c.hi, d.lo, lo) : fmaf(-c.hi, d.lo, lo);
  lo = S > 0 ? fmaf(c.lo, d.hi, lo) : fmaf(-c.lo, d.hi, lo);
  return df(s, lo);
}
__device__ __forceinline__ df fma(df a, df b, df c) { return a * b + c; }

// IEEE 754 conversions on the integer pipe.  On this GPU the FP64 pipe,
// which also carries the double <-> float conversion instructions, issues at
// 1/64 of the FP32 rate, so a pass that converts every point is FP64-bound
// unless the conversion is done with integer operations.  Written from the
// binary64 / binary32 formats: d2f_rn rounds to nearest, ties to even;
// results below the smallest normal float flush to signed zero (f2d flushes
// float subnormals the same way); overflow gives a signed infinity; a NaN
// stays a (quiet) NaN.
__device__ __forceinline__ float d2f_rn(double d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned int hi = (unsigned int)(u >> 32), lo = (unsigned int)u;
  const unsigned int sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7FFu);
  const unsigned int m = ((hi & 0xFFFFFu) << 3) | (lo >> 29);   // top 23 mantissa bits
  const unsigned int rest = lo & 0x1FFFFFFFu;                   // the 29 bits rounded off
  const int ef = e - 1023 + 127;
  unsigned int bits;
  if (e == 0x7FF) {
    bits = 0x7F800000u | ((m | rest) ? 0x400000u | m : 0u);
  } else if (ef >= 0xFF) {
    bits = 0x7F800000u;
  } else if (ef <= 0) {
    bits = 0u;
  } else {
    bits = ((unsigned int)ef << 23) | m;
    if (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) bits += 1u;   // may carry to inf
  }
  return __uint_as_float(bits | sign);
}

__device__ __forceinline__ double f2d(float f) {
  const unsigned int b = __float_as_uint(f);
  const unsigned int sign = b & 0x80000000u;
  const unsigned int e = (b >> 23) & 0xFFu;
  const unsigned int m = b & 0x7FFFFFu;
  unsigned int hi;
  if (e == 0) return __longlong_as_double((long long)((unsigned long long)sign << 32));
  if (e == 0xFF) hi = 0x7FF00000u | (m ? 0x80000u : 0u) | (m >> 3);
  else hi = ((e + 896u) << 20) | (m >> 3);
  return __longlong_as_double((long long)(((unsigned long long)(hi | sign) << 32) | (unsigned long long)(m << 29)));
}

// double -> double-float and back with one FP64 operation each.
__device__ __forceinline__ df df_of(double d) {
  const float h = d2f_rn(d);
  return df(h, d2f_rn(d - f2d(h)));
}
__device__ __forceinline__ double dbl_of(df a) { return f2d(a.hi) + f2d(a.lo); }

// Complex double-float (16 bytes, the size of a double2).
struct __align__(16) dfc {
  df x, y;
};

template <typename V> struct Real;
template <> struct Real<float2> { using T = float; };
template <> struct Real<dfc> { using T = df; };

template <typename V>
__device__ __forceinline__ V mk(typename Real<V>::T x, typename Real<V>::T y) {
  V v; v.x = x; v.y = y; return v;
}
template <typename V> __device__ __forceinline__ V czero() {
  using T = typename Real<V>::T;
  return mk<V>(T(0), T(0));
}
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cconj(V a) { return mk<V>(a.x, -a.y); }
template <typename V> __device__ __forceinline__ V cscale(V a, typename Real<V>::T s) { return mk<V>(a.x * s, a.y * s); }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  return mk<V>(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// a * conj(b)
template <typename V> __device__ __forceinline__ V cmulc(V a, V b) {
  return mk<V>(fma(a.x, b.x, a.y * b.y), fma(a.y, b.x, -a.x * b.y));
}
// double-float complex products: each component one two-product sum
template <> __device__ __forceinline__ dfc cmul<dfc>(dfc a, dfc b) {
  return mk<dfc>(df_dot2<-1>(a.x, b.x, a.y, b.y), df_dot2<+1>(a.x, b.y, a.y, b.x));
}
template <> __device__ __forceinline__ dfc cmulc<dfc>(dfc a, dfc b) {
  return mk<dfc>(df_dot2<+1>(a.x, b.x, a.y, b.y), df_dot2<-1>(a.y, b.x, a.x, b.y));
}

// Sums of K values over the block (blockDim.x a multiple of 32, at most 256):
// sum k ends up in the first lane of warp k.  The FP64 pipe takes 16 cycles
// for a warp's addition, so the lanes are folded once by a shuffle and the
// rest goes through shared memory to one warp per sum: 16 warp additions a
// sum and 256-thread block against 45 of a shuffle tree in every warp.
// Needs a __syncthreads() before it is called again.
template <int K>
__device__ __forceinline__ double block_sums(const double (&v)[K]) {
  __shared__ double sh[K][128];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double x = v[k] + __shfl_down_sync(0xffffffffu, v[k], 16);
    if (lane < 16) sh[k][wid * 16 + lane] = x;
  }
  __syncthreads();
  double x = 0.0;
  if (wid < K) {
    const double* a = sh[0] + wid * 128 + lane;      // 16 nw values of sum wid
    if (nw == 8) x = (a[0] + a[32]) + (a[64] + a[96]);
    else
      for (int i = lane; i < 16 * nw; i += 32) x += sh[wid][i];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  }
  return x;
}

// Sum of v over the block; result valid in every thread.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double total;
  const double a[1] = {v};
  const double x = block_sums(a);
  if (threadIdx.x == 0) total = x;
  __syncthreads();
  return total;
}

// Blocks of one slot: the x-y plane of the grid (blockIdx.z is the slot).
__device__ __forceinline__ unsigned int linear_block() { return blockIdx.x + gridDim.x * blockIdx.y; }
__device__ __forceinline__ unsigned int num_blocks() { return gridDim.x * gridDim.y; }

// Deterministic grid reduction of K sums over the blocks of one slot: every
// block stores its partials; the last block to arrive (one atomic ticket)
// sums all partials in a fixed order and returns true in all of its threads
// with *res[k] set.  The sum order does not depend on which block arrives
// last, so results are bitwise reproducible.  The last block keeps eight
// loads of each sum in flight per thread: up to 8192 partials, in a tail
// that nothing overlaps.
template <int K>
__device__ __forceinline__ bool grid_reduce_k(const double (&v)[K], double* const (&part)[K], unsigned int* counter,
                                              double* const (&res)[K]) {
  static_assert(K <= 4, "one warp per sum");
  __shared__ bool am_last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  const double bs = block_sums(v);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (wid == k && lane == 0) part[k][linear_block()] = bs;
  // The ticket is thread 0's, so the fences around it are too: before it, after
  // the barrier that makes the other warps' partials known to thread 0, and
  // after it, before the barrier that passes on what the last ticket saw.
  if (K > 1) __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    am_last = atomicAdd(counter, 1u) == num_blocks() - 1;
    if (am_last) __threadfence();
  }
  __syncthreads();
  if (!am_last) return false;
  const unsigned int nb = num_blocks(), bd = blockDim.x;
  double s[K];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k] = 0.0;
  for (unsigned int i = threadIdx.x; i < nb; i += 8 * bd) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = i + u * bd < nb ? __ldcg(part[k] + i + u * bd) : 0.0;
      if (i + 4 * bd < nb) s[k] += (t[4] + t[5]) + (t[6] + t[7]);
      s[k] += (t[0] + t[1]) + (t[2] + t[3]);
    }
  }
  const double total = block_sums(s);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (wid == k && lane == 0) *res[k] = total;
  if (threadIdx.x == 0) *counter = 0u;
  __threadfence_block();
  __syncthreads();
  return true;
}

__device__ __forceinline__ bool grid_reduce(double v, double* partials, unsigned int* counter,
                                            double* result) {
  const double a[1] = {v};
  double* const p[1] = {partials};
  double* const r[1] = {result};
  return grid_reduce_k(a, p, counter, r);
}

__device__ __forceinline__ bool grid_reduce3(double a, double b, double c, double* pa, double* pb,
                                             double* pc, unsigned int* counter, double* ra,
                                             double* rb, double* rc) {
  const double v[3] = {a, b, c};
  double* const p[3] = {pa, pb, pc};
  double* const r[3] = {ra, rb, rc};
  return grid_reduce_k(v, p, counter, r);
}

}  // namespace gps
