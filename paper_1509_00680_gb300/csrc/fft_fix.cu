// Register-resident passes of the FP64 spectrum (64-bit fixed point, see
// fix64.cuh) for power-of-two lengths 64 .. 1024; other lengths use the
// shared-memory kernels of fft.cu.
//
// The structure is that of the double-float passes in fft_col.cu: a CTA of 256
// threads holds 256 / (L/8) columns (y and z passes) or row pairs (x passes),
// a thread 8 elements of one line, the stages exchange through one padded
// shared line.  Before a transform the elements of a line are brought to the
// line's scale: the largest exponent and the sum of magnitudes are reduced
// over its threads (shuffles, then one shared-memory atomic per warp).
//
// Bound: issue (integer multiply-adds).  Measured against the same passes in
// FP64 (shared-memory kernels on the FP64 pipe): surface 160 x 160 x 256, z
// pass of 512 points 705 -> 168 us; free 64^3, one application 217 -> 100 us;
// free 256^3 12.2 -> 2.9 ms.
#include "fft_reg.cuh"

namespace gps {
namespace {

template <int L> struct Fix {
  static constexpr int E = 8, TPC = L / E, TC = kThreads / TPC, LS = line_stride<i64c>(L);
  // Resident CTAs per SM asked of the register allocator (80 registers a
  // thread; k_fix_x_inv<L, false> spills 48 to 76 bytes at that): the passes
  // are bound by issue and shared-memory exchanges.
  static constexpr int B = 3;
};

// Reduction scratch of a CTA's lines.
template <int N> struct ScaleSmem {
  int e[N];
  unsigned int sum[N];
};

// Brings the first EN elements x[i] (mantissas at exponents e[i]) of a line to
// one scale; the line's threads are the TPC threads of group g: threads g, g +
// TC, .. (COLS) or TPC consecutive ones.  parity: of the elements' positions
// in the line (see shift_round).  extra: bits kept free below 2^62.
// Returns the exponent of the transformed line; rem: see col_stages.
// ok(i): whether element i of the thread may be nonzero (the others are zero).
template <int L, bool COLS, typename F>
__device__ __forceinline__ int scale_line(i64c (&x)[8], const int (&e)[8], F ok, int g, int parity, int extra,
                                          ScaleSmem<Fix<L>::TC>& sm, int& rem) {
  constexpr int TPC = Fix<L>::TPC, TC = Fix<L>::TC;
  // lanes of the line in this warp: xor offsets [LO, HI); ONE: no other warp holds any
  constexpr int LO = COLS ? (TC < 32 ? TC : 32) : 1, HI = COLS ? 32 : (TPC < 32 ? TPC : 32);
  constexpr bool ONE = !COLS && TPC <= 32;
  const int lane = threadIdx.x & 31;
  const bool lead = COLS ? lane < TC : (lane & (HI - 1)) == 0;
  int top = -(1 << 28);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (ok(i)) top = max(top, e[i]);
#pragma unroll
  for (int o = LO; o < HI; o <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if constexpr (!ONE) {
    if (lead) atomicMax(&sm.e[g], top);
    __syncthreads();
    top = sm.e[g];
  }
  unsigned int sum = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (ok(i)) sum += mag_part(x[i].x.v, x[i].y.v, top - e[i]);
#pragma unroll
  for (int o = LO; o < HI; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if constexpr (!ONE) {
    if (lead) atomicAdd(&sm.sum[g], sum);
    __syncthreads();
    sum = sm.sum[g];
  }
  const int shift = max(sum_shift(sum) + extra, 1), first = min(shift, kHeadroom + extra);
  rem = shift - first;
  const int base = top + first;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (ok(i)) {
      x[i].x.v = shift_round(x[i].x.v - parity, base - e[i]);
      x[i].y.v = shift_round(x[i].y.v - parity, base - e[i]);
    }
  return top + shift;
}

template <int N>
__device__ __forceinline__ void clear(ScaleSmem<N>& sm) {
  if (threadIdx.x < N) {
    sm.e[threadIdx.x] = -(1 << 28);
    sm.sum[threadIdx.x] = 0u;
  }
}

// HALF: rows >= L/2 of every column are the zero padding (forward y and z of
// padded axes); they are neither read nor transformed.
template <int L, int MODE, bool HALF>
__global__ void __launch_bounds__(kThreads, Fix<L>::B) k_fix_col(PassGeom g, const i64c* __restrict__ twg, Batch b,
                                                                PipeArgs a) {
  constexpr int E = 8, TPC = Fix<L>::TPC, TC = Fix<L>::TC;
  const int slot = pass_slot<i64c>(b);
  if (slot < 0) return;
  i64c* __restrict__ W = reinterpret_cast<i64c*>(a.W) + slot * a.wstride;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ScaleSmem<TC> sm[MODE == COL_Z ? 2 : 1];
  const i64c* tw = twg + L;                        // forward-order stage twiddles
  const i64c* twr = twg + 2 * L;                   // reversed-order stage twiddles (z inverse)
  const int c = threadIdx.x % TC, t = threadIdx.x / TC;
  int kx, outer;
  const bool act = column_of<MODE>(g, blockIdx.x * TC + c, &kx, &outer);
  i64c* line = reinterpret_cast<i64c*>(smem_raw) + c * Fix<L>::LS;
  size_t stride;
  i64c* col;
  int nload, nstore;
  if constexpr (MODE == COL_Z) {
    stride = (size_t)g.Py * g.Hp;
    col = W + (size_t)outer * g.Hp + kx;
    nload = g.nz;
    nstore = g.nz;
  } else {
    stride = g.Hp;
    col = W + (size_t)outer * g.Py * g.Hp + kx;
    nload = MODE == COL_Y_FWD ? g.ny : L;
    nstore = MODE == COL_Y_FWD ? L : g.ny;
  }
  constexpr int R0 = ColPlan<L>::radix(0, false), RL = ColPlan<L>::radix(ColPlan<L>::nst - 1, false);
  clear(sm[0]);
  if constexpr (MODE == COL_Z) clear(sm[1]);
  i64c x[E];
  int e[E];
  auto nonzero = [](int i) { return !HALF || (i % R0) < R0 / 2; };
#pragma unroll
  for (int q = 0; q < E / R0; ++q)
#pragma unroll
    for (int r = 0; r < R0; ++r) {
      const int row = t + q * TPC + r * (L / R0);
      x[q * R0 + r] = (nonzero(r) && act && row < nload) ? col[(size_t)row * stride] : czero<i64c>();
    }
  __syncthreads();                                 // scratch cleared
#pragma unroll
  for (int i = 0; i < E; ++i)
    if (nonzero(i)) {
      e[i] = packed_exp(x[i]);
      x[i].x.v = packed_man(x[i].x.v);
      x[i].y.v = packed_man(x[i].y.v);
    }
  int rem;
  int el = scale_line<L, true>(x, e, nonzero, c, t & 1, 0, sm[0], rem);
  col_stages<i64c, L, E, MODE == COL_Y_INV ? +1 : -1, false, 0, HALF>(x, t, tw, line, rem);
  if constexpr (MODE != COL_Z) pdl_trigger();
  if constexpr (MODE == COL_Z) {
    const int ky = act ? outer : 0;
    const int kyp = min(ky, g.Py - ky);
    const int hy = g.Py / 2 + 1;
    const size_t t0 = (size_t)kyp * g.Hx + (act ? kx : 0);
    const size_t tz = (size_t)hy * g.Hx;
    const bool use_k0 = a.slot_k0 && b.st && b.st[slot].use_k0;
    const bool at0 = use_k0 && act && kx == 0 && ky == 0;
#pragma unroll
    for (int q = 0; q < E / RL; ++q)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int kz = t + q * TPC + r * (L / RL);
        const int kzp = min(kz, L - kz);
        double tv = a.table[t0 + (size_t)kzp * tz];
        if (at0 && kz == 0) tv = b.st[slot].k0;
        e[q * RL + r] = el;
        fx_apply(x[q * RL + r], e[q * RL + r], tv);
      }
    el = scale_line<L, true>(x, e, [](int) { return true; }, c, t & 1, 0, sm[1], rem);
    col_stages<i64c, L, E, +1, true, 0>(x, t, twr, line, rem);
    pdl_trigger();
    // the reversed transform ends with radix R0
#pragma unroll
    for (int q = 0; q < E / R0; ++q)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        const int row = t + q * TPC + r * (L / R0);
        if (act && row < nstore) col[(size_t)row * stride] = fx_pack(x[q * R0 + r], el);
      }
  } else {
#pragma unroll
    for (int q = 0; q < E / RL; ++q)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int row = t + q * TPC + r * (L / RL);
        if (act && row < nstore) col[(size_t)row * stride] = fx_pack(x[q * RL + r], el);
      }
  }
}

// Row pairs as one complex transform; HALF: rows padded to twice their length.
template <int L, bool HALF>
__global__ void __launch_bounds__(kThreads, Fix<L>::B) k_fix_x_fwd(PassGeom g, const i64c* __restrict__ twg, Batch b,
                                                                  PipeArgs a) {
  constexpr int E = 8, TPC = Fix<L>::TPC, NL = Fix<L>::TC;
  const int slot = pass_slot<i64c>(b);
  if (slot < 0) return;
  const double* __restrict__ in = a.in + slot * b.vstride;
  const double* __restrict__ scale = a.in_scale ? a.in_scale + slot * b.vstride : nullptr;
  i64c* __restrict__ W = reinterpret_cast<i64c*>(a.W) + slot * a.wstride;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ScaleSmem<NL> sm;
  const int l = threadIdx.x / TPC, t = threadIdx.x % TPC;
  i64c* line = reinterpret_cast<i64c*>(smem_raw) + l * Fix<L>::LS;
  const int npairs = (g.nrows + 1) >> 1;
  const int pr = blockIdx.x * NL + l;
  const bool act = pr < npairs;
  const int ra = 2 * pr;
  const bool hasb = act && ra + 1 < g.nrows;
  const bool red = a.red_mu && b.st;
  double sum = 0.0;
  constexpr int R0 = ColPlan<L>::radix(0, false), RL = ColPlan<L>::radix(ColPlan<L>::nst - 1, false);
  clear(sm);
  i64c x[E];
  int e[E];
  auto nonzero = [](int i) { return !HALF || (i % R0) < R0 / 2; };
  auto column = [&](int i) { return t + (i / R0) * TPC + (i % R0) * (L / R0); };
  double va[E], vb[E];
  load_pairs(in, g.nx, (size_t)ra * g.nx, act, hasb, nonzero, column, va, vb);
  if (scale) {
    double sa[E], sb[E];
    load_pairs(scale, g.nx, (size_t)ra * g.nx, act, hasb, nonzero, column, sa, sb);
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (nonzero(i)) {
        va[i] *= sa[i];
        vb[i] *= sb[i];
      }
  }
  if (red) {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (nonzero(i)) sum += va[i] + vb[i];
  }
#pragma unroll
  for (int i = 0; i < E; ++i) {
    if (nonzero(i)) fx_of_doubles(va[i], vb[i], x[i].x.v, x[i].y.v, e[i]);
    else x[i] = czero<i64c>();
  }
  __syncthreads();
  int rem;
  // one bit free: the unpacking below adds two values
  const int el = scale_line<L, false>(x, e, nonzero, l, t & 1, 1, sm, rem);
  col_stages<i64c, L, E, -1, false, 0, HALF>(x, t, twg + L, line, rem);
  pdl_trigger();
  // Z in natural order; Z_k and Z_(L-k) meet through the line
#pragma unroll
  for (int q = 0; q < E / RL; ++q)
#pragma unroll
    for (int r = 0; r < RL; ++r) line[pidx<i64c>(t + q * TPC + r * (L / RL))] = x[q * RL + r];
  __syncthreads();
  if (act) {
    i64c* wa = W + row_offset(g, ra);
    i64c* wb = hasb ? W + row_offset(g, ra + 1) : nullptr;
    for (int k = t; k < g.Hx; k += TPC) {
      const i64c zk = line[pidx<i64c>(k)];
      const i64c zm = line[pidx<i64c>(k == 0 ? 0 : L - k)];
      // A_k = (Z_k + conj Z_(L-k))/2 ; B_k = -i (Z_k - conj Z_(L-k))/2
      wa[k] = fx_pack(mk<i64c>(zk.x + zm.x, zk.y - zm.y), el - 1);
      if (hasb) wb[k] = fx_pack(mk<i64c>(zk.y + zm.y, zm.x - zk.x), el - 1);
    }
  }
  if (red)
    grid_reduce(sum, b.partials + (size_t)slot * b.pstride, &b.st[slot].counter[CNT_MU], &b.st[slot].mu_sum);
}

// HALF: only the lower half of a padded row is computed and stored (free 256^3:
// 293 -> 270 us; the column passes measured no faster, or up to 3 % slower,
// with their unused half left out).
template <int L, bool HALF>
__global__ void __launch_bounds__(kThreads, Fix<L>::B) k_fix_x_inv(PassGeom g, const i64c* __restrict__ twg, Batch b,
                                                                  PipeArgs a) {
  constexpr int E = 8, TPC = Fix<L>::TPC, NL = Fix<L>::TC;
  const int slot = pass_slot<i64c>(b);
  if (slot < 0) return;
  const i64c* __restrict__ W = reinterpret_cast<const i64c*>(a.W) + slot * a.wstride;
  double* __restrict__ out = a.out + slot * b.vstride;
  const double* __restrict__ out_scale = a.out_scale ? a.out_scale + slot * b.vstride : nullptr;
  const double* __restrict__ dot_with = a.dot_with ? a.dot_with + slot * b.vstride : nullptr;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ScaleSmem<NL> sm;
  const int l = threadIdx.x / TPC, t = threadIdx.x % TPC;
  i64c* line = reinterpret_cast<i64c*>(smem_raw) + l * Fix<L>::LS;
  const int npairs = (g.nrows + 1) >> 1;
  const int pr = blockIdx.x * NL + l;
  const bool act = pr < npairs;
  const int ra = 2 * pr;
  const bool hasb = act && ra + 1 < g.nrows;
  const i64c* wa = act ? W + row_offset(g, ra) : W;
  const i64c* wb = hasb ? W + row_offset(g, ra + 1) : W;
  constexpr int R0 = ColPlan<L>::radix(0, false), RL = ColPlan<L>::radix(ColPlan<L>::nst - 1, false);
  clear(sm);
  i64c x[E];
  int e[E];
#pragma unroll
  for (int q = 0; q < E / R0; ++q)
#pragma unroll
    for (int r = 0; r < R0; ++r) {
      const int i = q * R0 + r;
      const int k = t + q * TPC + r * (L / R0);
      const bool mirror = k >= g.Hx;               // Hermitian half: conjugates of L - k
      const int ks = mirror ? L - k : k;
      i64c A = czero<i64c>(), B = czero<i64c>();
      if (act) {
        A = wa[ks];
        if (hasb) B = wb[ks];
        if (ks == 0 || 2 * ks == L) {              // DC and Nyquist are real
          A.y.v &= 63;
          B.y.v &= 63;
        }
      }
      fx_align(A, B, e[i], t & 1);           // k has the parity of t
      if (mirror) {
        A.y = -A.y;
        B.y = -B.y;
      }
      x[i] = mk<i64c>(A.x - B.y, A.y + B.x);       // Z = A + i B
    }
  __syncthreads();
  int rem;
  const int el = scale_line<L, false>(x, e, [](int) { return true; }, l, t & 1, 0, sm, rem);
  col_stages<i64c, L, E, +1, false, 0>(x, t, twg + L, line, rem);
  pdl_trigger();
  const bool want_wsum = a.red_wsum && b.st && b.st[slot].gauge;
  double dot = 0.0, wsum = 0.0;
  constexpr int RS = HALF ? RL / 2 : RL;         // stored outputs of a butterfly
#pragma unroll
  for (int i0 = 0; i0 < E / RL * RS; i0 += 4) {
    auto element = [&](int i) { return (i0 + i) / RS * RL + (i0 + i) % RS; };
    auto column = [&](int i) { return t + element(i) / RL * TPC + element(i) % RL * (L / RL); };
    const i64c z[4] = {x[element(0)], x[element(1)], x[element(2)], x[element(3)]};
    store_pairs(z, el, out, out_scale, (const float*)nullptr, dot_with, g.nx, (size_t)ra * g.nx, act, hasb, column,
                dot, want_wsum, wsum);
  }
  if (b.st) reduce_inverse(b, slot, dot_with != nullptr, dot, want_wsum, wsum);
}

template <typename K>
void launch(K kernel, dim3 grid, size_t sm, const PassGeom& g, const i64c* tw, const Batch& b, const PipeArgs& a,
            cudaStream_t st) {
  if (sm + kStaticSmemAllowance > 48 * 1024)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  count_launch();
  launch_pdl(kernel, grid, kThreads, sm, st, g, tw, b, a);
}

template <int L>
void launch_x(bool inverse, const PassGeom& g, const i64c* tw, const Batch& b, const PipeArgs& a, int nslots,
              cudaStream_t st) {
  constexpr int NL = Fix<L>::TC;
  const size_t sm = (size_t)NL * Fix<L>::LS * sizeof(i64c);
  const dim3 grid(((g.nrows + 1) / 2 + NL - 1) / NL, 1, nslots);
  if (inverse && 2 * g.nx == L) launch(k_fix_x_inv<L, true>, grid, sm, g, tw, b, a, st);
  else if (inverse) launch(k_fix_x_inv<L, false>, grid, sm, g, tw, b, a, st);
  else if (2 * g.nx == L) launch(k_fix_x_fwd<L, true>, grid, sm, g, tw, b, a, st);
  else launch(k_fix_x_fwd<L, false>, grid, sm, g, tw, b, a, st);
}

template <int L>
void launch_col(int mode, const PassGeom& g, const i64c* tw, const Batch& b, const PipeArgs& a, int nslots,
                cudaStream_t st) {
  constexpr int TC = Fix<L>::TC;
  const size_t sm = (size_t)TC * Fix<L>::LS * sizeof(i64c);
  const dim3 grid(column_ctas(g, mode, TC), 1, nslots);
  if (mode == COL_Y_FWD) {
    if (2 * g.ny == L) launch(k_fix_col<L, COL_Y_FWD, true>, grid, sm, g, tw, b, a, st);
    else launch(k_fix_col<L, COL_Y_FWD, false>, grid, sm, g, tw, b, a, st);
  } else if (mode == COL_Y_INV) {
    launch(k_fix_col<L, COL_Y_INV, false>, grid, sm, g, tw, b, a, st);
  } else {
    if (2 * g.nz == L) launch(k_fix_col<L, COL_Z, true>, grid, sm, g, tw, b, a, st);
    else launch(k_fix_col<L, COL_Z, false>, grid, sm, g, tw, b, a, st);
  }
}

}  // namespace

bool launch_fix_x(bool inverse, int L, const PassGeom& g, const i64c* tw, const Batch& b, const PipeArgs& a,
                  int nslots, cudaStream_t st) {
  if (g.plain_tw) return false;
  switch (L) {
    case 64: launch_x<64>(inverse, g, tw, b, a, nslots, st); return true;
    case 128: launch_x<128>(inverse, g, tw, b, a, nslots, st); return true;
    case 256: launch_x<256>(inverse, g, tw, b, a, nslots, st); return true;
    case 512: launch_x<512>(inverse, g, tw, b, a, nslots, st); return true;
    case 1024: launch_x<1024>(inverse, g, tw, b, a, nslots, st); return true;
    default: return false;
  }
}

bool launch_fix_col(int mode, int L, const PassGeom& g, const i64c* tw, const Batch& b, const PipeArgs& a,
                    int nslots, cudaStream_t st) {
  if (g.plain_tw) return false;
  switch (L) {
    case 64: launch_col<64>(mode, g, tw, b, a, nslots, st); return true;
    case 128: launch_col<128>(mode, g, tw, b, a, nslots, st); return true;
    case 256: launch_col<256>(mode, g, tw, b, a, nslots, st); return true;
    case 512: launch_col<512>(mode, g, tw, b, a, nslots, st); return true;
    case 1024: launch_col<1024>(mode, g, tw, b, a, nslots, st); return true;
    default: return false;
  }
}

}  // namespace gps
