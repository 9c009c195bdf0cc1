// Order-16 central first derivatives on the grid (the paper's finite-
// difference filters, Sec. "Numerical results"): d/dx u ~ (1/h) sum_j d_j
// (u(x + jh) - u(x - jh)), j = 1..8.  Periodic axes wrap (they must have at
// least 8 points); free axes continue the field by its face value.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "fix64.cuh"

namespace gps {

struct Stencil16 {
  int nx, ny, nz;
  int perx, pery, perz;   // axes that wrap
  double ihx, ihy, ihz;   // 1 / h
  double d[9];            // d_1..d_8 (d[0] unused)
};

__device__ __forceinline__ void point_of16(size_t idx, const Stencil16& s, int* i, int* j, int* k) {
  *i = (int)(idx % s.nx);
  *j = (int)((idx / s.nx) % s.ny);
  *k = (int)(idx / ((size_t)s.nx * s.ny));
}

__device__ __forceinline__ int shift16(int i, int m, int n, int per) {
  if (per) return i + m >= n ? i + m - n : (i + m < 0 ? i + m + n : i + m);
  const int t = i + m;
  return t >= n ? n - 1 : (t < 0 ? 0 : t);
}

// grad u at point idx = (i, j, k).
__device__ __forceinline__ double3 grad16(const double* __restrict__ u, size_t idx, int i, int j, int k,
                                          const Stencil16& s) {
  const double* row = u + (idx - i);
  const size_t sy = s.nx, sz = (size_t)s.nx * s.ny;
  const size_t bxz = (size_t)k * sz + i, bxy = (size_t)j * s.nx + i;
  double dx = 0.0, dy = 0.0, dz = 0.0;
#pragma unroll
  for (int m = 1; m <= 8; ++m) {
    const double c = s.d[m];
    dx = fma(c, row[shift16(i, m, s.nx, s.perx)] - row[shift16(i, -m, s.nx, s.perx)], dx);
    dy = fma(c, u[bxz + (size_t)shift16(j, m, s.ny, s.pery) * sy] - u[bxz + (size_t)shift16(j, -m, s.ny, s.pery) * sy],
             dy);
    dz = fma(c, u[bxy + (size_t)shift16(k, m, s.nz, s.perz) * sz] - u[bxy + (size_t)shift16(k, -m, s.nz, s.perz) * sz],
             dz);
  }
  return make_double3(dx * s.ihx, dy * s.ihy, dz * s.ihz);
}

// ---- tiles ------------------------------------------------------------------
//
// Derivatives of a field on a tile of 32 x 8 x 8 points (8 along z per thread
// of a 256-thread block) as 64-bit fixed point.  FP64 issues at 1/64 of the
// integer rate, so the 48 FP64 operations of grad16 bound every pass that uses
// it; here a difference is two integer additions and its product with a
// coefficient three integer multiply-adds, accumulated over the eight
// distances.  One axis at a time, the values of the tile and of the axis' halo
// are loaded, brought to the largest magnitude among their lines (60 bits) and
// staged in shared memory.
//
// The lines that share a scale are those that a reduction finds for nothing: a
// warp's rows (x), the columns of a lane (y), a thread's column (z).  The unit
// is 2^-60 of the scale, twice the power of two below the largest value, so
// values down to 2^-7 of that power are staged exactly and others to the
// nearest unit.  A derivative is off by a unit or two, at most six: 2^-50
// of the largest value of its stencil where one of four of its values
// reaches that 2^-7 (kNear), as FP64 differences are.  Every other point takes
// FP64 differences, and so do lines with values that are not finite.  One scale
// a tile would send warps of a smooth potential there too (energy at periodic 128^3:
// 126 against 150 us); one a row instead of a warp's rows along x
// costs more than it saves (k_pol 275 against 286 us).  The points that remain
// (in a potential of cavities in a solvent 3 % along x, in 9 % of the warps) are
// dealt to all lanes of their warp, 32 at a time: each lane on its own, a warp
// took as many turns as its worst lane has points (k_pol 310 -> 275 us, k_veps 149 -> 135).
struct Tile16 {
  static constexpr int X = 32, Y = 8, Z = 8, H = 8, T = X * Y;   // points, halo, threads
  static constexpr int N = X * Y * (Z + 2 * H);                  // most values of an axis (y and z)
  long long v[N];
  int top[2][X];                                                 // largest exponents of a lane's columns, in turn
  unsigned char list[Y][X * Z];                                  // points of a warp: lane + 32 tz
};

// Q62 digits of a coefficient.
struct Q62 { int h, l; };

// sum_j d_j (p[j stride] - p[-j stride]), d_j = (-1)^(j+1) (8!)^2 / (j (8-j)!
// (8+j)!); |values| <= 2^60.  The cross products of all eight distances sum to
// less than 2^63.  near: whether a value at distance 1 or 8 reaches kNear.
constexpr int kNear = 1 << 21;           // 2^53: high word
__device__ __forceinline__ long long diff16(const long long* p, int stride, bool& near) {
  constexpr Q62 c[8] = {{954437177, -477218588}, {-334053012, 381774871}, {121473823, -2091085088}, {-37960570, 1995641370}, {9344140, 830293600}, {-1668596, -1988966984}, {190697, -1122536352}, {-10429, 1168684963}};
  unsigned long long hi = 0ull - (1ull << 31), mid = (1ull << 63) + (1ull << 29);
  const long long *a = p, *b = p;
  int top = 0, bottom = 0;
#pragma unroll
  for (int j = 1; j <= 8; ++j) {
    int h, l;
    a += stride;
    b -= stride;
    if (j == 1 || j == 8) {
      top = max(top, max(hi32(*a), hi32(*b)));
      bottom = min(bottom, min(hi32(*a), hi32(*b)));
    }
    digits(*a - *b, h, l);
    hi += (unsigned long long)mul32(h, c[j - 1].h);
    mid += (unsigned long long)(mul32(h, c[j - 1].l) + mul32(l, c[j - 1].h));
  }
  near = top >= kNear || bottom < -kNear;
  return (long long)((hi << 2) + (mid >> 30));
}

// Index of position p of an axis of n points, -8 <= p: wrapped, or clamped to
// the faces; positions past the halo of the last point are not used and read
// as its end.
__device__ __forceinline__ int axis16(int p, int n, int per) {
  p = min(p, n + 7);
  if (per) return p < 0 ? p + n : p >= n ? p - n : p;
  return min(max(p, 0), n - 1);
}

// Derivatives along `axis` (0 x, 1 y, 2 z) of u, without the 1/h, at the
// thread's points (i0 + tx, j0 + ty, k0 + tz).  turn: 0, 1, 0, .. from call to
// call; t.top zero before the first (and a barrier).  The axis is a
// run-time argument and the callers loop over it, so that the unrolled
// conversion and differences exist once (six copies overran the instruction
// cache: k_pol 270 us).
__device__ __forceinline__ void derivative16(Tile16& t, int axis, int turn, const double* __restrict__ u, int i0, int j0,
                                             int k0, const Stencil16& s, double (&d)[Tile16::Z]) {
  constexpr int X = Tile16::X, Y = Tile16::Y, Z = Tile16::Z, H = Tile16::H, XW = X + 2 * H, YW = Y + 2 * H;
  constexpr int NV = Z + 2 * H;          // values of a thread (x: 2 Z)
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const size_t sy = s.nx, sz = (size_t)s.nx * s.ny;
  const int ic = min(i0 + tx, s.nx - 1), jc = min(j0 + ty, s.ny - 1);
  double v[NV];
  if (axis == 2) {
    const double* col = u + (size_t)jc * sy + ic;
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = col[(size_t)axis16(k0 + q - H, s.nz, s.perz) * sz];
  } else {
    // positions of the thread in a plane: three rows (y), or two halves of a row (x)
    size_t at[3];
    if (axis == 1) {
#pragma unroll
      for (int r = 0; r < 3; ++r) at[r] = (size_t)axis16(j0 + ty + 8 * r - H, s.ny, s.pery) * sy + ic;
    } else {
      at[0] = (size_t)jc * sy + axis16(i0 + tx - H, s.nx, s.perx);
      at[1] = tx < 2 * H ? (size_t)jc * sy + axis16(i0 + tx + X - H, s.nx, s.perx) : at[0];
      at[2] = at[0];
    }
#pragma unroll
    for (int z = 0; z < Z; ++z) {
      const double* plane = u + (size_t)min(k0 + z, s.nz - 1) * sz;
#pragma unroll
      for (int r = 0; r < 3; ++r) v[3 * z + r] = plane[at[r]];
    }
  }
  int top = 1;
#pragma unroll
  for (int q = 0; q < NV; ++q) top = max(top, (__double2hiint(v[q]) >> 20) & 0x7ff);
  if (axis == 0) top = __reduce_max_sync(0xffffffffu, top);
  if (axis == 1) atomicMax(&t.top[turn][tx], top);
  __syncthreads();                       // also: the previous set has been read
  if (axis == 1) top = t.top[turn][tx];
  // The other words, last read before the barrier above, are cleared here: the
  // barrier below orders it before the next call's atomicMax.
  if (ty == 0) t.top[turn ^ 1][tx] = 0;
  const int e0 = top + 1024 + 2;         // exponent of the staged values
  // value 3 z + r goes to first + z step + r part
  const int first = axis == 0 ? ty * XW + tx : ty * X + tx;
  const int step = axis == 0 ? Y * XW : axis == 1 ? YW * X : 3 * Y * X;
  const int part = axis == 0 ? X : Y * X;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    long long m;
    int e;
    fx_of_finite(v[q], m, e);            // of a line with other values: not used
    m = ((m >> min(e0 - e - 1, 60)) + 1) >> 1;   // nearest unit; nonzero normal values stay so
    const bool put = axis > 0 || q % 3 == 0 || (q % 3 == 1 && tx < 2 * H);
    if (put) t.v[first + (q / 3) * step + (q % 3) * part] = m;
  }
  __syncthreads();
  const int stride = axis == 0 ? 1 : axis == 1 ? X : Y * X;
  const int next = axis == 0 ? Y * XW : axis == 1 ? YW * X : Y * X;
  const long long* p = &t.v[first + H * stride];
  unsigned int far = 0;                  // points that take FP64 differences ...
#pragma unroll
  for (int tz = 0; tz < Z; ++tz) {
    bool near;
    d[tz] = fx_to_double(diff16(p + tz * next, stride, near), e0);
    far |= near ? 0u : 1u << tz;
  }
  if (top == 0x7ff) far = (1u << Z) - 1;
  else if (top == 1) far = 0;            // zeros, or values next to the smallest normal number, which are exact
  else {
    // ... unless their values are all zero, as in the cavity of a dielectric
#pragma unroll 1
    for (unsigned int left = far; left; left &= left - 1) {
      const long long* c = p + (__ffs((int)left) - 1) * next;
      long long any = 0;
#pragma unroll
      for (int m = 1; m <= 8; ++m) any |= c[m * stride] | c[-m * stride];
      if (any == 0) far ^= left & (0u - left);
    }
  }
  if (!__any_sync(0xffffffffu, far != 0)) return;
  // a warp's points 32 at a time, whichever lanes they belong to
  int at[Z], total = 0;
#pragma unroll
  for (int tz = 0; tz < Z; ++tz) {
    const unsigned int b = __ballot_sync(0xffffffffu, far >> tz & 1);
    at[tz] = far >> tz & 1 ? total + __popc(b & ((1u << tx) - 1)) : -32;
    if (far >> tz & 1) t.list[ty][at[tz]] = (unsigned char)(tx + 32 * tz);
    total += __popc(b);
  }
  __syncwarp();
#pragma unroll 1
  for (int base = 0; base < total; base += 32) {
    const int w = t.list[ty][min(base + tx, total - 1)];
    const int x = min(i0 + (w & 31), s.nx - 1), z = min(k0 + (w >> 5), s.nz - 1);
    const int i = axis == 0 ? x : axis == 1 ? jc : z;
    const int n = axis == 0 ? s.nx : axis == 1 ? s.ny : s.nz;
    const int per = axis == 0 ? s.perx : axis == 1 ? s.pery : s.perz;
    const size_t st = axis == 0 ? 1 : axis == 1 ? sy : sz;
    const double* line = u + ((size_t)z * sz + (size_t)jc * sy + x) - i * st;
    double a = 0.0;
#pragma unroll
    for (int m = 1; m <= 8; ++m)
      a = fma(s.d[m], line[shift16(i, m, n, per) * st] - line[shift16(i, -m, n, per) * st], a);
#pragma unroll
    for (int tz = 0; tz < Z; ++tz) {
      const double v = __shfl_sync(0xffffffffu, a, (at[tz] - base) & 31);
      if (at[tz] >= base && at[tz] < base + 32) d[tz] = v;
    }
  }
  __syncwarp();                          // the list has been read
}

}  // namespace gps
