// Register-resident transforms of power-of-two lengths L = 64 .. 1024: radix
// plan, per-stage twiddle layout, butterflies on a thread's elements, and the
// exchange between stages through a padded shared-memory line.  Used by the
// FP32 and double-float passes (fft_col.cu) and the FP64 passes (fft_fix.cu).
#pragma once

#include "fft_common.cuh"

namespace gps {

enum ColMode { COL_Y_FWD = 0, COL_Y_INV = 1, COL_Z = 2 };

// Columns of the column passes -- (kx, ky) in the z pass, (kx, z) in the y
// passes -- numbered through with kx fastest: every CTA but the last is full,
// where tiles of each row would leave 15 of 80 columns idle at Hx = 65 and 31
// of 64 at Hx = 33.  A row counts Hp columns (Hx rounded up to even), so that
// tiles start on a 32-byte sector in every row.  Measured, FP64 spectrum: z
// pass of free 64^3 39 -> 33 us, y pass of periodic 128^3 22.5 -> 18.7 us.
template <int MODE>
__device__ __forceinline__ bool column_of(const PassGeom& g, int id, int* kx, int* outer) {
  *outer = id / g.Hp;
  *kx = id - *outer * g.Hp;
  return *kx < g.Hx && *outer < (MODE == COL_Z ? g.Py : g.nz);
}
inline int column_ctas(const PassGeom& g, int mode, int tc) {
  return (g.Hp * (mode == COL_Z ? g.Py : g.nz) + tc - 1) / tc;
}

// Radix plan: radix-8 stages, then one stage of radix L / 8^k when L is not a
// power of 8.  rev = true gives the stages in reverse order.
template <int L> struct ColPlan {
  static_assert(L == 64 || L == 128 || L == 256 || L == 512 || L == 1024, "unsupported length");
  static constexpr int nst = L == 64 ? 2 : L == 1024 ? 4 : 3;
  static constexpr int last = L == 128 ? 2 : L == 256 ? 4 : L == 1024 ? 2 : 8;
  __host__ __device__ static constexpr int radix(int s, bool rev) {
    return (rev ? nst - 1 - s : s) == nst - 1 ? last : 8;
  }
  __host__ __device__ static constexpr int ns(int s, bool rev) {
    int p = 1;
    for (int i = 0; i < s; ++i) p *= radix(i, rev);
    return p;
  }
};

// Twiddles of the stages, laid out per stage as W[s][r - 1][k] (k < Ns, the
// factor W_(Ns R)^(r k)), so that the threads of a warp, which hold
// consecutive k, read consecutive addresses (the index r k L/(Ns R) into the
// plain table scatters them).  The twiddle array of a length L served here
// holds three tables of L entries: the plain e^{-2 pi i m/L}, this layout for
// the forward radix order, and for the reversed order (built once per shape
// by the engine, col_stage_twiddle_index).  Offset of stage s in the layout:
template <int L, bool REV>
__host__ __device__ constexpr int stage_tw_offset(int s) {
  int o = 0;
  for (int i = 0; i < s; ++i) o += (ColPlan<L>::radix(i, REV) - 1) * ColPlan<L>::ns(i, REV);
  return o;
}
template <int L, bool REV>
__host__ __device__ constexpr int stage_tw_size() { return stage_tw_offset<L, REV>(ColPlan<L>::nst); }

// Butterflies of one stage (radix R, Ns = NS) on the thread's E elements:
// butterfly q is b = t + q L/E with inputs x[q R + r] = in[b + r L/R].
// tws: this stage's twiddles W[r - 1][k].  HALF (first stage only): the
// inputs r >= R/2 are the zero padding of the line (rows >= L/2), so each
// butterfly runs as two R/2-point ones (Dft::run_half).
template <typename V, int L, int E, int DIR, int R, int NS, bool HALF = false>
__device__ __forceinline__ void col_butterflies(V (&x)[E], int t, const V* tws) {
  constexpr int TPC = L / E, Q = E / R;
  static_assert(!HALF || NS == 1, "zero-half pruning applies to the first stage");
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if constexpr (NS > 1) {
      const int k = (t + q * TPC) & (NS - 1);
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const V w = tws[(r - 1) * NS + k];
        x[q * R + r] = DIR < 0 ? cmul(x[q * R + r], w) : cmulc(x[q * R + r], w);
      }
    }
    if constexpr (HALF) Dft<V, DIR, R>::run_half(x + q * R);
    else Dft<V, DIR, R>::run(x + q * R);
  }
}

// Scatter of a stage's outputs to out[(b - k) R + k + r Ns] in the column's
// shared line, then gather of the next stage's inputs in[b + r L/R2].
template <typename V, int L, int E, int R, int NS, int R2>
__device__ __forceinline__ void col_exchange(V (&x)[E], int t, V* line) {
  constexpr int TPC = L / E;
#pragma unroll
  for (int q = 0; q < E / R; ++q) {
    const int b = t + q * TPC;
    const int k = b & (NS - 1);
    const int base = (b - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) line[pidx<V>(base + r * NS)] = x[q * R + r];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < E / R2; ++q) {
    const int b = t + q * TPC;
#pragma unroll
    for (int r = 0; r < R2; ++r) x[q * R2 + r] = line[pidx<V>(b + r * (L / R2))];
  }
  __syncthreads();
}

// Stages S .. nst-1 of one transform.  On return x[q RL + r] = out[b + r L/RL]
// with RL the radix of the last stage.  HALF: the transform's input is zero
// beyond L/2 (pruned first stage).  rem (FP64 spectrum, L > 512): bits that
// the line is still to be shifted down before the last stage (fix64.cuh).
template <typename V, int L, int E, int DIR, bool REV, int S, bool HALF = false>
__device__ __forceinline__ void col_stages(V (&x)[E], int t, const V* tw, V* line, int rem = 0) {
  if constexpr (std::is_same<V, i64c>::value && (L > 512) && S + 1 == ColPlan<L>::nst) {
    if (rem > 0) {
#pragma unroll
      for (int i = 0; i < E; ++i) {
        x[i].x.v = shift_round(x[i].x.v - (i & 1), rem);
        x[i].y.v = shift_round(x[i].y.v - (i & 1), rem);
      }
    }
  }
  constexpr int R = ColPlan<L>::radix(S, REV), NS = ColPlan<L>::ns(S, REV);
  col_butterflies<V, L, E, DIR, R, NS, HALF && S == 0>(x, t, tw + stage_tw_offset<L, REV>(S));
  if constexpr (S + 1 < ColPlan<L>::nst) {
    col_exchange<V, L, E, R, NS, ColPlan<L>::radix(S + 1, REV)>(x, t, line);
    col_stages<V, L, E, DIR, REV, S + 1>(x, t, tw, line, rem);
  }
}

}  // namespace gps
