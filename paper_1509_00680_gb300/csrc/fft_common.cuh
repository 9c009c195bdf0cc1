// Pieces shared by the spectrum-pass kernels: radix-R butterflies, the padded
// shared-memory line layout, and the slot test of a pass.
#pragma once

#include <type_traits>

#include "device_util.cuh"
#include "fix64.cuh"
#include "gps_internal.h"

namespace gps {

template <> struct Real<i64c> { using T = fx; };
// Complex products of the FP64 spectrum; the factor b is in Q62 digits.
template <> __device__ __forceinline__ i64c cmul<i64c>(i64c a, i64c b) {
  const int dh = hi32(b.y.v), dl = lo32(b.y.v);
  return fx_cmul(a, hi32(b.x.v), lo32(b.x.v), dh, dl, -dh, -dl);
}
template <> __device__ __forceinline__ i64c cmulc<i64c>(i64c a, i64c b) {
  const int dh = hi32(b.y.v), dl = lo32(b.y.v);
  return fx_cmul(a, hi32(b.x.v), lo32(b.x.v), -dh, -dl, dh, dl);
}

// Radix-R butterflies, DIR = -1 forward (e^{-2 pi i/R}), +1 inverse.
template <typename V, int DIR>
__device__ __forceinline__ V rot_i(V a) {  // a * (DIR * i)
  return DIR < 0 ? mk<V>(a.y, -a.x) : mk<V>(-a.y, a.x);
}

// k x for a constant k; x / 2; a (c + i DIR s) for constants c, s.
template <class K, typename T>
__device__ __forceinline__ T mulk(T x) {
  if constexpr (std::is_same<T, fx>::value) return fx_mul(x, K::h, K::l);
  else return T(K::d) * x;
}
template <typename T>
__device__ __forceinline__ T halve(T x) {
  // ties to even: rounded one way, the odd sums of a stage's radix-3 butterflies
  // would add up
  if constexpr (std::is_same<T, fx>::value) return fx((x.v + ((x.v >> 1) & 1)) >> 1);
  else return T(0.5) * x;
}
template <typename V, int DIR, class C, class S>
__device__ __forceinline__ V rotk(V a) {
  if constexpr (std::is_same<V, i64c>::value) {
    return DIR < 0 ? fx_cmul(a, C::h, C::l, -S::h, -S::l, S::h, S::l)
                   : fx_cmul(a, C::h, C::l, S::h, S::l, -S::h, -S::l);
  } else {
    using T = typename Real<V>::T;
    const T cr = T(C::d), si = T(DIR < 0 ? -S::d : S::d);
    return mk<V>(a.x * cr - a.y * si, a.x * si + a.y * cr);
  }
}

template <typename V, int DIR, int R> struct Dft;

// run_half(x): the same transform when x[R/2..R-1] are zero (the zero-padded
// half of a line in the first stage of a forward pass): X_(2m) is the R/2-point
// transform of x[0..R/2-1], X_(2m+1) that of x_r w^r, w = e^{DIR 2 pi i / R}.
template <typename V, int DIR> struct Dft<V, DIR, 2> {
  __device__ __forceinline__ static void run(V* x) {
    V a = x[0], b = x[1];
    x[0] = cadd(a, b);
    x[1] = csub(a, b);
  }
  __device__ __forceinline__ static void run_half(V* x) { x[1] = x[0]; }
};

template <typename V, int DIR> struct Dft<V, DIR, 4> {
  __device__ __forceinline__ static void run(V* x) {
    V a0 = cadd(x[0], x[2]), a1 = csub(x[0], x[2]);
    V a2 = cadd(x[1], x[3]), a3 = rot_i<V, DIR>(csub(x[1], x[3]));
    x[0] = cadd(a0, a2);
    x[2] = csub(a0, a2);
    x[1] = cadd(a1, a3);
    x[3] = csub(a1, a3);
  }
  __device__ __forceinline__ static void run_half(V* x) {
    const V o = rot_i<V, DIR>(x[1]);
    const V e0 = x[0], e1 = x[1];
    x[0] = cadd(e0, e1);
    x[2] = csub(e0, e1);
    x[1] = cadd(e0, o);
    x[3] = csub(e0, o);
  }
};

template <typename V, int DIR> struct Dft<V, DIR, 8> {
  __device__ __forceinline__ static void run(V* x) {
    V e[4] = {x[0], x[2], x[4], x[6]};
    V o[4] = {x[1], x[3], x[5], x[7]};
    Dft<V, DIR, 4>::run(e);
    Dft<V, DIR, 4>::run(o);
    // o_k *= e^{DIR 2 pi i k / 8}
    if (DIR < 0) {
      o[1] = mk<V>(mulk<KSqrtHalf>(o[1].x + o[1].y), mulk<KSqrtHalf>(o[1].y - o[1].x));
      o[2] = mk<V>(o[2].y, -o[2].x);
      o[3] = mk<V>(mulk<KSqrtHalf>(o[3].y - o[3].x), mulk<KNeg<KSqrtHalf>>(o[3].x + o[3].y));
    } else {
      o[1] = mk<V>(mulk<KSqrtHalf>(o[1].x - o[1].y), mulk<KSqrtHalf>(o[1].x + o[1].y));
      o[2] = mk<V>(-o[2].y, o[2].x);
      o[3] = mk<V>(mulk<KNeg<KSqrtHalf>>(o[3].x + o[3].y), mulk<KSqrtHalf>(o[3].x - o[3].y));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = cadd(e[k], o[k]);
      x[k + 4] = csub(e[k], o[k]);
    }
  }
  __device__ __forceinline__ static void run_half(V* x) {
    V e[4] = {x[0], x[1], x[2], x[3]};
    V o[4] = {x[0], x[1], x[2], x[3]};
    // o_r *= e^{DIR 2 pi i r / 8}
    if (DIR < 0) {
      o[1] = mk<V>(mulk<KSqrtHalf>(o[1].x + o[1].y), mulk<KSqrtHalf>(o[1].y - o[1].x));
      o[2] = mk<V>(o[2].y, -o[2].x);
      o[3] = mk<V>(mulk<KSqrtHalf>(o[3].y - o[3].x), mulk<KNeg<KSqrtHalf>>(o[3].x + o[3].y));
    } else {
      o[1] = mk<V>(mulk<KSqrtHalf>(o[1].x - o[1].y), mulk<KSqrtHalf>(o[1].x + o[1].y));
      o[2] = mk<V>(-o[2].y, o[2].x);
      o[3] = mk<V>(mulk<KNeg<KSqrtHalf>>(o[3].x + o[3].y), mulk<KSqrtHalf>(o[3].x - o[3].y));
    }
    Dft<V, DIR, 4>::run(e);
    Dft<V, DIR, 4>::run(o);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      x[2 * m] = e[m];
      x[2 * m + 1] = o[m];
    }
  }
};

// 16 points as two 8-point transforms of the even and odd elements joined by
// the twiddles e^{DIR 2 pi i k / 16}, k = 0..7.
template <typename V, int DIR> struct Dft<V, DIR, 16> {
  __device__ __forceinline__ static void run(V* x) {
    V e[8], o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      e[k] = x[2 * k];
      o[k] = x[2 * k + 1];
    }
    Dft<V, DIR, 8>::run(e);
    Dft<V, DIR, 8>::run(o);
    o[1] = rotk<V, DIR, KCosPi8, KSinPi8>(o[1]);
    o[2] = rotk<V, DIR, KSqrtHalf, KSqrtHalf>(o[2]);
    o[3] = rotk<V, DIR, KSinPi8, KCosPi8>(o[3]);
    o[4] = DIR < 0 ? mk<V>(o[4].y, -o[4].x) : mk<V>(-o[4].y, o[4].x);
    o[5] = rotk<V, DIR, KNeg<KSinPi8>, KCosPi8>(o[5]);
    o[6] = rotk<V, DIR, KNeg<KSqrtHalf>, KSqrtHalf>(o[6]);
    o[7] = rotk<V, DIR, KNeg<KCosPi8>, KSinPi8>(o[7]);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      x[k] = cadd(e[k], o[k]);
      x[k + 8] = csub(e[k], o[k]);
    }
  }
  __device__ __forceinline__ static void run_half(V* x) {
    V e[8], o[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) e[r] = x[r];
    o[0] = x[0];
    o[1] = rotk<V, DIR, KCosPi8, KSinPi8>(x[1]);
    o[2] = rotk<V, DIR, KSqrtHalf, KSqrtHalf>(x[2]);
    o[3] = rotk<V, DIR, KSinPi8, KCosPi8>(x[3]);
    o[4] = DIR < 0 ? mk<V>(x[4].y, -x[4].x) : mk<V>(-x[4].y, x[4].x);
    o[5] = rotk<V, DIR, KNeg<KSinPi8>, KCosPi8>(x[5]);
    o[6] = rotk<V, DIR, KNeg<KSqrtHalf>, KSqrtHalf>(x[6]);
    o[7] = rotk<V, DIR, KNeg<KCosPi8>, KSinPi8>(x[7]);
    Dft<V, DIR, 8>::run(e);
    Dft<V, DIR, 8>::run(o);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      x[2 * m] = e[m];
      x[2 * m + 1] = o[m];
    }
  }
};

template <typename V, int DIR> struct Dft<V, DIR, 3> {
  __device__ __forceinline__ static void run(V* x) {
    using s3 = typename std::conditional<(DIR > 0), KSqrt3Half, KNeg<KSqrt3Half>>::type;
    V t1 = cadd(x[1], x[2]);
    V t2 = mk<V>(x[0].x - halve(t1.x), x[0].y - halve(t1.y));
    V d = csub(x[1], x[2]);
    V u = mk<V>(mulk<s3>(d.x), mulk<s3>(d.y));   // u = DIR sqrt(3)/2 (x1 - x2)
    V iu = mk<V>(-u.y, u.x);
    x[0] = cadd(x[0], t1);
    x[1] = cadd(t2, iu);
    x[2] = csub(t2, iu);
  }
};

template <typename V, int DIR> struct Dft<V, DIR, 5> {
  __device__ __forceinline__ static void run(V* x) {
    using c1 = KCos2Pi5;
    using c2 = KCos4Pi5;
    using s1 = typename std::conditional<(DIR > 0), KSin2Pi5, KNeg<KSin2Pi5>>::type;
    using s2 = typename std::conditional<(DIR > 0), KSin4Pi5, KNeg<KSin4Pi5>>::type;
    V a1 = cadd(x[1], x[4]), b1 = csub(x[1], x[4]);
    V a2 = cadd(x[2], x[3]), b2 = csub(x[2], x[3]);
    V p1 = mk<V>(x[0].x + mulk<c1>(a1.x) + mulk<c2>(a2.x), x[0].y + mulk<c1>(a1.y) + mulk<c2>(a2.y));
    V p2 = mk<V>(x[0].x + mulk<c2>(a1.x) + mulk<c1>(a2.x), x[0].y + mulk<c2>(a1.y) + mulk<c1>(a2.y));
    V q1 = mk<V>(mulk<s1>(b1.x) + mulk<s2>(b2.x), mulk<s1>(b1.y) + mulk<s2>(b2.y));
    V q2 = mk<V>(mulk<s2>(b1.x) - mulk<s1>(b2.x), mulk<s2>(b1.y) - mulk<s1>(b2.y));
    V iq1 = mk<V>(-q1.y, q1.x), iq2 = mk<V>(-q2.y, q2.x);
    x[0] = cadd(x[0], cadd(a1, a2));
    x[1] = cadd(p1, iq1);
    x[4] = csub(p1, iq1);
    x[2] = cadd(p2, iq2);
    x[3] = csub(p2, iq2);
  }
};

// Shared-memory layout of a line: one pad element after every 128 bytes
// (8 complex values of 16 bytes, 16 complex floats), so that the stride-R scatters of
// the early Stockham stages spread over all banks.
template <typename V> struct PadShift;
template <> struct PadShift<float2> { static constexpr int v = 4; };
template <> struct PadShift<dfc> { static constexpr int v = 3; };
template <> struct PadShift<i64c> { static constexpr int v = 3; };

template <typename V> struct SpecOf;
template <> struct SpecOf<i64c> { static constexpr int v = SPEC_FP64; };
template <> struct SpecOf<float2> { static constexpr int v = SPEC_FP32; };
template <> struct SpecOf<dfc> { static constexpr int v = SPEC_DF64; };

template <typename V>
__device__ __forceinline__ int pidx(int i) { return i + (i >> PadShift<V>::v); }

template <typename V>
__host__ __device__ constexpr int line_stride(int L) { return L + (L >> PadShift<V>::v) + 1; }

__device__ __forceinline__ size_t row_offset(const PassGeom& g, int row) {
  const int y = row % g.ny, z = row / g.ny;
  return ((size_t)z * g.Py + y) * g.Hp;
}

constexpr int kThreads = 256;

// Upper bound on the static shared memory of a spectrum-pass kernel; a
// launcher opts a kernel in to more dynamic shared memory once dynamic plus
// this allowance may exceed the default 48 KB per block.
constexpr size_t kStaticSmemAllowance = 6144;


// Slot served by this block for a spectrum pass of precision V, or -1.
template <typename V>
__device__ __forceinline__ int pass_slot(const Batch& b) {
  int s = batch_slot(b);
  if (s >= 0 && b.st && b.prec >= 0 && b.st[s].spec != SpecOf<V>::v) s = -1;
  if (s >= 0) mark_acted(b);
  return s;
}

// Rows of an x pass: a[i], b[i] = the values at column(i) of a row (offset row) and of the next
// one, zero outside the data: all loads of a thread are issued before any is
// used.
template <typename S, int N, typename F, typename C>
__device__ __forceinline__ void load_pairs(const S* __restrict__ src, int nx, size_t row, bool act, bool hasb,
                                           F ok, C column, S (&a)[N], S (&b)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    a[i] = S(0);
    b[i] = S(0);
    if (ok(i)) {
      const int j = column(i);
      const bool in = act && j < nx;
      if (in) a[i] = src[row + j];
      if (in && hasb) b[i] = src[row + nx + j];
    }
  }
}

// Input values of an x pass: a, b (loaded from `in`) times the scale factors
// at the same places, as doubles, and their sum if it is wanted (red) ...
template <typename V, int N, typename F, typename C>
__device__ __forceinline__ void scale_pairs(const double* scale, const float* scale32, int nx, size_t row, bool act,
                                            bool hasb, F ok, C column, bool red, double& sum, const double (&a)[N],
                                            const double (&b)[N], typename Real<V>::T (&xa)[N],
                                            typename Real<V>::T (&xb)[N]) {
  // ... the FP32 spectrum multiplies in FP32 unless the FP64 sum is wanted
  if constexpr (std::is_same<V, float2>::value) {
    if (!red) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        xa[i] = d2f_rn(a[i]);
        xb[i] = d2f_rn(b[i]);
      }
      if (scale32) {
        float sa[N], sb[N];
        load_pairs(scale32, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          xa[i] *= sa[i];
          xb[i] *= sb[i];
        }
      } else if (scale) {
        double sa[N], sb[N];
        load_pairs(scale, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          xa[i] *= d2f_rn(sa[i]);
          xb[i] *= d2f_rn(sb[i]);
        }
      }
      return;
    }
  }
  double va[N], vb[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    va[i] = a[i];
    vb[i] = b[i];
  }
  if (scale) {
    double sa[N], sb[N];
    load_pairs(scale, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (ok(i)) {
        va[i] *= sa[i];
        vb[i] *= sb[i];
      }
  }
  if (red) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (ok(i)) sum += va[i] + vb[i];
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if constexpr (std::is_same<V, float2>::value) {
      xa[i] = d2f_rn(va[i]);
      xb[i] = d2f_rn(vb[i]);
    } else {
      xa[i] = ok(i) ? df_of(va[i]) : df(0.f, 0.f);
      xb[i] = ok(i) ? df_of(vb[i]) : df(0.f, 0.f);
    }
  }
}

// Real value of a spectrum line as a double (integer-pipe conversions).  e:
// exponent of the line (FP64 spectrum only).
template <typename V>
__device__ __forceinline__ double unscaled(typename Real<V>::T z, int e = 0) {
  if constexpr (std::is_same<V, float2>::value) return f2d(z);
  else if constexpr (std::is_same<V, dfc>::value) return dbl_of(z);
  else return fx_to_double(z.v, e);
}

// Results of an x inverse pass: v = z scale (the FP32 spectrum scales in
// FP32) to out, (v, r) into dot and the sum of z into wsum where they are
// wanted, for the N elements x at column(i) of a row pair.  The scale factors
// and r are loaded before anything is stored: with a load, a product and a
// store per element the pass waited for HBM once per element (periodic
// 128^3, FP64 spectrum, with the same change in the forward pass: x passes 98
// -> 74 us).
template <typename V, int N, typename C>
__device__ __forceinline__ void store_pairs(const V (&x)[N], int e, double* __restrict__ out,
                                            const double* __restrict__ scale, const float* __restrict__ scale32,
                                            const double* __restrict__ dot_with, int nx, size_t row, bool act,
                                            bool hasb, C column, double& dot, bool want_wsum, double& wsum) {
  auto ok = [&](int) { return true; };
  double va[N], vb[N], ra[N], rb[N];
  if (dot_with) load_pairs(dot_with, nx, row, act, hasb, ok, column, ra, rb);
  if constexpr (std::is_same<V, float2>::value) {
    float fa[N], fb[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      fa[i] = x[i].x;
      fb[i] = x[i].y;
    }
    if (scale32) {
      float sa[N], sb[N];
      load_pairs(scale32, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        fa[i] *= sa[i];
        fb[i] *= sb[i];
      }
    } else if (scale) {
      double sa[N], sb[N];
      load_pairs(scale, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        fa[i] *= d2f_rn(sa[i]);
        fb[i] *= d2f_rn(sb[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      va[i] = f2d(fa[i]);
      vb[i] = f2d(fb[i]);
    }
    if (want_wsum) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const bool in = act && column(i) < nx;
        if (in) wsum += f2d(x[i].x);
        if (in && hasb) wsum += f2d(x[i].y);
      }
    }
  } else {
    double sa[N], sb[N];
    if (scale) load_pairs(scale, nx, row, act, hasb, ok, column, sa, sb);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool in = act && column(i) < nx;
      va[i] = in ? unscaled<V>(x[i].x, e) : 0.0;
      vb[i] = in && hasb ? unscaled<V>(x[i].y, e) : 0.0;
    }
    if (want_wsum) {
#pragma unroll
      for (int i = 0; i < N; ++i) wsum += va[i] + vb[i];
    }
    if (scale) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        va[i] *= sa[i];
        vb[i] *= sb[i];
      }
    }
  }
  if (dot_with) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool in = act && column(i) < nx;
      if (in) dot += va[i] * ra[i];
      if (in && hasb) dot += vb[i] * rb[i];
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (act && column(i) < nx) {
      out[row + column(i)] = va[i];
      if (hasb) out[row + nx + column(i)] = vb[i];
    }
}

// (v, r) and, for the gauge, the sum of w of an x inverse pass (want: the
// slot projects); the last block flags that v exists.
__device__ __forceinline__ void reduce_inverse(const Batch& b, int slot, bool want_dot, double dot, bool want_wsum,
                                               double wsum) {
  SlotState& S = b.st[slot];
  double* pd = b.partials + (size_t)slot * b.pstride;
  if (want_dot && want_wsum) {
    const double v[2] = {dot, wsum};
    double* const p[2] = {pd, b.partials2 + (size_t)slot * b.pstride};
    double* const r[2] = {&S.vr, &S.wsum};
    if (grid_reduce_k(v, p, &S.counter[CNT_VR], r) && threadIdx.x == 0) S.vdone = 1;
  } else if (want_dot) {
    if (grid_reduce(dot, pd, &S.counter[CNT_VR], &S.vr) && threadIdx.x == 0) S.vdone = 1;
  } else if (want_wsum) {
    grid_reduce(wsum, pd, &S.counter[CNT_VR], &S.wsum);
  }
}

}  // namespace gps
