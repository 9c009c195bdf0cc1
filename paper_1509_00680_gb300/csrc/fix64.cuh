// 64-bit fixed-point arithmetic of the FP64 spectrum.
//
// On this GPU the FP64 pipe issues at 1/64 of the rate of the integer and
// FP32 pipes (measured: 1.8 FP64 additions per clock and SM against 64 64-bit
// integer additions and 26 32 x 32 + 64-bit multiply-adds), so the butterflies
// of the FP64 spectrum run on 64-bit integers and the FP64 pipe only touches
// the real input and output of a solve.  Measured issue slots (of 128 per
// clock and SM): complex addition and subtraction 8 against 284, complex
// product 70 against 287.
//
// Two forms of a complex value, 16 bytes each:
//
//   packed  (HBM and, before a transform, shared memory): two mantissas in
//           the upper 58 bits of two 64-bit words, the larger one normalized
//           (its magnitude in [2^61, 2^62)), and a 12-bit exponent shared by
//           both in the low 6 bits of each word: (re + i im) 2^(e - kBias).
//           Rounded to nearest, to 2^-56 of the larger component (FP64:
//           2^-53): a truncation would be a common bias of all elements,
//           which the Green's function amplifies at k = 0.  e = kNaN marks a value that came from
//           an infinity or a NaN.
//   scaled  (inside a transform): plain 64-bit integers that share one
//           exponent per line (block floating point).
//
// A line is scaled so that the sum of its magnitudes stays below 2^62, which
// bounds every partial sum of its transform: no butterfly can overflow, no
// addition rounds, and only the input (half a unit), the products (about
// half a unit) and the halves of the radix-3 butterflies (ties, to even) do.  With L elements of similar size the unit is about L 2^-62
// of an element, below the rounding unit of FP64 up to L = 512; longer
// transforms keep up to kHeadroom bits below the final scale until their last
// stages.
#pragma once

#include <cuda_runtime.h>

namespace gps {

constexpr int kBias = 2108;       // packed exponent: m 2^(e - kBias); a double of biased exponent E has e = E + 1024
constexpr int kNaN = 4095;
constexpr int kHeadroom = 11;     // bits a line is scaled down before its first stage: covers 512-point products

// A real number of a scaled line; products take the other factor as Q62 in
// the digit form below.
struct fx {
  long long v;
  fx() = default;
  __host__ __device__ explicit constexpr fx(long long v_) : v(v_) {}
};

struct __align__(16) i64c {
  fx x, y;
};

// Q62 number w as two signed digits, w = h 2^32 + l, in one 64-bit word
// (high word h, low word l): the cross products of two such numbers are plain
// signed 32 x 32 products.  l = -2^31 is avoided so that -l exists, and so are
// factors of exactly 1/2 (sixth roots of unity): their products with odd
// numbers are ties, which round up, and in the columns that hold real values
// nothing is added to them; a unit more, and the sign of the number decides
// (white noise on a periodic 6 x 1458 x 18 grid: 2.2e-15 -> 5.8e-16).
__host__ __device__ inline long long q62_digits(long long w) {
  if (w == 1ll << 61 || w == -(1ll << 61)) w += 1;
  int l = (int)(unsigned int)(w & 0xffffffffll);
  const long long h = (w - l) / 4294967296ll;          // exact
  if (l == (int)0x80000000) l += 1;                    // off by one unit
  return (long long)(((unsigned long long)h << 32) | (unsigned int)l);
}

// Constant factors of the butterflies, as doubles and as Q62 digits.
struct KSqrtHalf { static constexpr double d = 0.70710678118654752440; static constexpr int h = 759250125, l = -25716447; };
struct KCosPi8 { static constexpr double d = 0.92387953251128675613; static constexpr int h = 992008094, l = 1696238673; };
struct KSinPi8 { static constexpr double d = 0.38268343236508977173; static constexpr int h = 410903207, l = -1364630830; };
struct KSqrt3Half { static constexpr double d = 0.86602540378443864676; static constexpr int h = 929887697, l = -1332128537; };
struct KCos2Pi5 { static constexpr double d = 0.30901699437494742410; static constexpr int h = 331804471, l = 803819395; };
struct KCos4Pi5 { static constexpr double d = -0.80901699437494742410; static constexpr int h = -868675383, l = -803819395; };
struct KSin2Pi5 { static constexpr double d = 0.95105651629515357212; static constexpr int h = 1021189159, l = -2002125123; };
struct KSin4Pi5 { static constexpr double d = 0.58778525229247312917; static constexpr int h = 631129609, l = -357254181; };
template <class K> struct KNeg { static constexpr double d = -K::d; static constexpr int h = -K::h, l = -K::l; };

#ifdef __CUDACC__

__device__ __forceinline__ fx operator+(fx a, fx b) { return fx(a.v + b.v); }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx(a.v - b.v); }
__device__ __forceinline__ fx operator-(fx a) { return fx(-a.v); }

__device__ __forceinline__ int lo32(long long v) { return (int)v; }
__device__ __forceinline__ int hi32(long long v) { return (int)(v >> 32); }
// signed digits of a scaled value
__device__ __forceinline__ void digits(long long v, int& h, int& l) {
  l = lo32(v);
  h = hi32(v) + (int)((unsigned int)l >> 31);
}
__device__ __forceinline__ long long mul32(int a, int b) { return (long long)a * b; }

// x w, w = h 2^32 + l in Q62: the high digits' product and the two cross
// products (the product of the low digits is below one unit); |x| <= 2^62.5.
__device__ __forceinline__ fx fx_mul(fx x, int h, int l) {
  int xh, xl;
  digits(x.v, xh, xl);
  const long long mid = (1ll << 29) + mul32(xh, l) + mul32(xl, h);
  return fx((mul32(xh, h) << 2) + (mid >> 30));
}

// (a + i b)(c + i d): four products per component accumulated before one
// shift.  (eh, el) = -(dh, dl).
__device__ __forceinline__ i64c fx_cmul(i64c a, int ch, int cl, int dh, int dl, int eh, int el) {
  int ah, al, bh, bl;
  digits(a.x.v, ah, al);
  digits(a.y.v, bh, bl);
  const long long hr = mul32(ah, ch) + mul32(bh, eh);
  const long long hi = mul32(ah, dh) + mul32(bh, ch);
  const long long mr = (1ll << 29) + mul32(ah, cl) + mul32(al, ch) + mul32(bh, el) + mul32(bl, eh);
  const long long mi = (1ll << 29) + mul32(ah, dl) + mul32(al, dh) + mul32(bh, cl) + mul32(bl, ch);
  i64c r;
  r.x.v = (hr << 2) + (mr >> 30);
  r.y.v = (hi << 2) + (mi >> 30);
  return r;
}

// v 2^-s rounded to nearest, s >= 1; ties upwards.  Values that come from
// doubles or from packed words end in zeros, so ties are common where a line
// is scaled: the callers pass v - p with p alternating over the elements that
// are summed, which turns every other tie downwards.  (A common direction would add up at
// k = 0, where the Green's function is largest: 10 times the error of FP64
// butterflies for white noise at 96^3.)
__device__ __forceinline__ long long shift_round(long long v, int s) {
  const long long t = v >> min(s - 1, 63);
  return (t + 1) >> 1;
}

// ---- packed values ---------------------------------------------------------

__device__ __forceinline__ int packed_exp(i64c w) {
  return (lo32(w.x.v) & 63) | ((lo32(w.y.v) & 63) << 6);
}
__device__ __forceinline__ long long packed_man(long long w) { return w & ~63ll; }

// 32 bits of |v| from the top: bitwise complement for negative values (off by
// one unit, far below what the callers use).
__device__ __forceinline__ unsigned int mag_hi(long long v) {
  const int h = hi32(v);
  return (unsigned int)(h ^ (h >> 31));
}

// Normalizes (re, im) 2^(e - kBias), |re|, |im| < 2^62: the larger magnitude
// goes to [2^61, 2^62) (values below 2^31 stay below that: they are exact).
__device__ __forceinline__ void fx_normalize(long long& re, long long& im, int& e) {
  const int s = __clz((int)(mag_hi(re) | mag_hi(im))) - 2;
  re <<= s;
  im <<= s;
  e -= s;
}

// Packs a normalized pair.
__device__ __forceinline__ i64c fx_pack_normalized(long long re, long long im, int e) {
  if (e < 0) {        // below 2^-2000: zero
    re = im = 0;
    e = 0;
  }
  if (e > kNaN) e = kNaN;
  i64c w;
  w.x.v = ((re + 32) & ~63ll) | (long long)(e & 63);
  w.y.v = ((im + 32) & ~63ll) | (long long)(e >> 6);
  return w;
}

// Packs a scaled value of a line with exponent e (a line marked kNaN stays so).
__device__ __forceinline__ i64c fx_pack(i64c z, int e) {
  if (e >= kNaN) return i64c{fx(kNaN & 63), fx(kNaN >> 6)};
  long long re = z.x.v, im = z.y.v;
  fx_normalize(re, im, e);
  return fx_pack_normalized(re, im, e);
}

// Mantissa and exponent of a finite double: v = m 2^(e - kBias), m normalized
// unless v is zero or subnormal (exponent of the smallest normal numbers).
// Returns the biased exponent.
__device__ __forceinline__ int fx_of_finite(double v, long long& m, int& e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int be = (int)((u >> 52) & 0x7ffu);
  m = (long long)(((u & 0xfffffffffffffull) | (be == 0 ? 0ull : 0x10000000000000ull)) << 9);
  if ((long long)u < 0) m = -m;
  e = max(be, 1) + 1024;
  return be;
}
// The same of any double; infinities and NaN as e = kNaN.
__device__ __forceinline__ void fx_of_double(double v, long long& m, int& e) {
  if (fx_of_finite(v, m, e) == 0x7ff) e = kNaN;
}

// Packed pair of two doubles.
__device__ __forceinline__ void fx_of_doubles(double a, double b, long long& re, long long& im, int& e) {
  int ea, eb;
  fx_of_double(a, re, ea);
  fx_of_double(b, im, eb);
  e = max(ea, eb);
  if (e > ea) re = shift_round(re, e - ea);
  if (e > eb) im = shift_round(im, e - eb);
}

// m 2^(e - kBias) with the sign bit `sign` as the nearest double (ties away
// from zero; gradual underflow).
__device__ __forceinline__ double fx_compose(unsigned long long sign, unsigned long long m, int e) {
  const unsigned int mh = (unsigned int)(m >> 32);
  const int lz = mh ? __clz((int)mh) : 32 + __clz((int)(unsigned int)m);
  if (lz >= 64) return __longlong_as_double((long long)sign);
  m <<= lz;                                              // top bit at 63: v = m 2^(e - kBias - lz)
  const int be = e - kBias - lz + 63 + 1023;             // biased exponent of the leading bit
  if (be <= 0) {                                         // subnormal
    if (be < -52) return __longlong_as_double((long long)sign);
    return __longlong_as_double((long long)(sign | (((m >> (11 - be)) + 1ull) >> 1)));
  }
  if (be >= 0x7ff) return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull));
  const unsigned long long q = (m >> 11) + ((m >> 10) & 1ull);
  return __longlong_as_double((long long)(sign | (((unsigned long long)(be - 1) << 52) + q)));
}
// v 2^(e - kBias) likewise.
__device__ __forceinline__ double fx_to_double(long long v, int e) {
  if (e >= kNaN) return __longlong_as_double(0x7ff8000000000000ll);
  return fx_compose((unsigned long long)v & 0x8000000000000000ull,
                    v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v, e);
}

// Digits and exponent of a table factor: t = (w / 2^62) 2^(e - 1022) with
// |w| in [2^61, 2^62); subnormals count as zero.
__device__ __forceinline__ void fx_factor(double t, int& h, int& l, int& e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(t);
  e = (int)((u >> 52) & 0x7ffu);
  long long w = (long long)(((u & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
  if (e == 0) w = 0;
  if ((long long)u < 0) w = -w;
  digits(w, h, l);
}

// Table product (re + i im) t of a scaled value with line exponent e,
// normalized; a line marked kNaN stays so.
__device__ __forceinline__ void fx_apply(i64c& z, int& e, double t) {
  int h, l, et;
  fx_factor(t, h, l, et);
  z.x = fx_mul(z.x, h, l);
  z.y = fx_mul(z.y, h, l);
  const int ez = e >= kNaN ? kNaN : min(e + et - 1022, kNaN - 1);
  e = ez;
  fx_normalize(z.x.v, z.y.v, e);
  if (ez >= kNaN || et == 0x7ff) e = kNaN;
}

// Two packed values as mantissas at one exponent e, a bit below the top so
// that sums of two stay below 2^62 in magnitude; parity: of their position in
// the line (see shift_round).
__device__ __forceinline__ void fx_align(i64c& a, i64c& b, int& e, int parity) {
  const int ea = packed_exp(a), eb = packed_exp(b);
  const int top = max(ea, eb);
  const int sa = min(top - ea + 1, 63), sb = min(top - eb + 1, 63);
  const long long ha = (1ll << (sa - 1)) - parity, hb = (1ll << (sb - 1)) - parity;
  a.x.v = (packed_man(a.x.v) + ha) >> sa;
  a.y.v = (packed_man(a.y.v) + ha) >> sa;
  b.x.v = (packed_man(b.x.v) + hb) >> sb;
  b.y.v = (packed_man(b.y.v) + hb) >> sb;
  e = top >= kNaN ? kNaN : top + 1;
}

// ---- scale of a line -------------------------------------------------------

// Contribution of one normalized element, whose exponent is s below the
// reference, to the sum of magnitudes (in units of 2^45; rounded up).
__device__ __forceinline__ unsigned int mag_part(long long re, long long im, int s) {
  return ((mag_hi(re) + mag_hi(im)) >> min(13 + s, 31)) + 1u;
}
// Bits by which the elements of a line (relative to the reference exponent)
// are shifted down so that the sum of magnitudes stays below 2^62 (with 2^-10
// to spare for the low words that the sum leaves out and for rounding).
__device__ __forceinline__ int sum_shift(unsigned int sum) {
  return max(15 - __clz((int)(sum + (sum >> 10) + 1u)), 0);
}

#endif  // __CUDACC__

}  // namespace gps
