// Elementary functions of doubles on the integer pipe (FP64 issues at 1/64 of
// its rate), with the arithmetic of fix64.cuh.
#pragma once

#include "fix64.cuh"

namespace gps {

// ln x (the FP64 log costs about fifty FP64 operations a point).  Argument
// reduction by a table of reciprocals (Tang, ACM TOMS 16, 1990): x = 2^k m, c
// ~ 1/m in steps of 2^-10 from the top seven bits of m, r = m c - 1 exactly (|r|
// <= 2^-7), ln x = k ln 2 - ln c + r S(r) with S(r) = 1 - r/2 + r^2/3 - .. +
// r^8/9 in 62-bit fixed point.  Within 2^-7 of 1 the sum is r S(r) alone and
// keeps its relative accuracy.  For k = 0 the sum has 64 fractional bits (with
// 59 the smallest results of this branch were off by up to 1.26 units in the
// last place), otherwise 61: its magnitude, below 5.55, then takes all 64 bits.
// Below one unit in the last place for 2^-7 <= x < 2^8 (0.53 seen over 10^7
// arguments); other arguments take log().
struct LogEntry {
  int c;            // 2^10 / m
  long long t;      // -ln(c 2^-10), less ln 2 where k counts the next power; Q64
};
__device__ const LogEntry kLog[128] = {
    {1024, 0ll}, {1012, 217449402910135620ll}, {1004, 363852902130987047ll}, {997, 492916105791551876ll},
    {989, 641531161979034824ll}, {982, 772558814357976946ll}, {975, 904523821220465167ll},
    {967, 1056506094520383395ll}, {960, 1190525582320469641ll}, {953, 1325525880113686902ll},
    {946, 1461521449748507975ll}, {940, 1578892433671965565ll}, {933, 1716775839671240844ll},
    {926, 1855697645811877951ll}, {920, 1975611897379757024ll}, {913, 2116504244618060346ll},
    {907, 2238131569247314719ll}, {901, 2360566160788172870ll}, {895, 2483818806891349249ll},
    {889, 2607900512898827746ll}, {883, 2732822507740801840ll}, {877, 2858596250033651404ll},
    {871, 2985233434387237051ll}, {865, 3112745997930193658ll}, {859, 3241146127062327672ll},
    {854, 3348833205060016471ll}, {848, 3478893044001375095ll}, {843, 3587981144728763741ll},
    {838, 3697718196926968058ll}, {832, 3830270221691897566ll}, {827, 3941462505760077071ll},
    {822, 4053329095246964985ll}, {817, 4165878218482716586ll}, {812, 4279118255333998699ll},
    {807, 4393057740948001826ll}, {802, 4507705369612800438ll}, {797, 4623069998738427277ll},
    {792, 4739160652963219918ll}, {787, 4855986528390199858ll}, {783, 4949982879917862053ll},
    {778, 5068155891833629052ll}, {773, 5187090823981735259ll}, {769, 5282793991037459835ll},
    {764, 5403125429299924605ll}, {760, 5499958953883438787ll}, {755, 5621720082921211662ll},
    {751, 5719710985719572930ll}, {747, 5818225206901671492ll}, {743, 5917268366034059704ll},
    {738, 6041824842466999975ll}, {734, 6142079133112771157ll}, {730, 6242881264131408774ll},
    {726, 6344237255791980452ll}, {722, -6340155417054629666ll}, {718, -6237673241947637361ll},
    {714, -6134618537752890175ll}, {710, -6030984871508813501ll}, {707, -5952875746730335691ll},
    {703, -5848213088235548201ll}, {699, -5742953207345004463ll}, {695, -5637089249226162881ll},
    {692, -5557290664480559961ll}, {688, -5450352718192624241ll}, {684, -5342791223505227131ll},
    {681, -5261706503614631935ll}, {677, -5153036121157597427ll}, {674, -5071111142354304413ll},
    {670, -4961308770096562555ll}, {667, -4878525935247593925ll}, {664, -4795369923323071870ll},
    {660, -4683908894941053804ll}, {657, -4599868913257257143ll}, {654, -4515444307892006414ll},
    {650, -4402273743891906514ll}, {647, -4316937844256562819ll}, {644, -4231205339480400567ll},
    {641, -4145072525837730946ll}, {638, -4058535647478120774ll}, {635, -3971590895443670323ll},
    {632, -3884234406663022002ll}, {629, -3796462262921435593ll}, {626, -3708270489806243500ll},
    {623, -3619655055626976363ll}, {620, -3530611870309425440ll}, {617, -3441136784262883231ll},
    {614, -3351225587219777939ll}, {611, -3260874007046890488ll}, {608, -3170077708527314833ll},
    {605, -3078832292112293269ll}, {603, -3017750302282572813ll}, {600, -2925746400471432400ll},
    {597, -2833281324293745646ll}, {594, -2740350427127064061ll}, {592, -2678135379708233368ll},
    {589, -2584417596044838233ll}, {586, -2490221251411663057ll}, {584, -2427155398279344845ll},
    {581, -2332150497772475841ll}, {579, -2268540972419636943ll}, {576, -2172713514977912298ll},
    {574, -2108550862207147358ll}, {571, -2011886479926060167ll}, {569, -1947160995717971526ll},
    {566, -1849644940921122012ll}, {564, -1784346663626416374ll}, {561, -1685963795362353988ll},
    {559, -1620082496500726674ll}, {557, -1553965063446734927ll}, {554, -1454342441078812732ll},
    {552, -1387627199918624915ll}, {550, -1320669797642671865ll}, {547, -1219775777259060748ll},
    {545, -1152205210593624476ll}, {543, -1084386222168607453ll}, {541, -1016316978606872166ll},
    {538, -913739824164369855ll}, {536, -845036787304660515ll}, {534, -776076916065200710ll},
    {532, -706858282976718805ll}, {530, -637378938790526945ll}, {527, -532666770730725625ll},
    {525, -462526974920836371ll}, {523, -392119469317874213ll}, {521, -321442202498300337ll},
    {519, -250493099368188280ll}, {517, -179270060797655839ll}, {512, 0ll}, {512, 0ll}};

__device__ __forceinline__ double fx_log(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int be = (int)(u >> 52);                       // sign included: negative arguments fall through
  if (be < 1023 - 7 || be >= 1023 + 8) return log(x);
  const int j = (int)(u >> 45) & 127;
  const int k = be - 1023 + (j >= 53 ? 1 : 0);
  const int c = __ldg(&kLog[j].c);
  const long long t = __ldg(&kLog[j].t);
  const long long r = (long long)(((u & 0xfffffffffffffull) | 0x10000000000000ull) * (unsigned long long)c) -
                      (1ll << 62);                     // Q62
  int h, l;
  digits(r << 7, h, l);
  constexpr long long a[9] = {4611686018427387904ll, -2305843009213693952ll, 1537228672809129301ll, -1152921504606846976ll, 922337203685477581ll, -768614336404564651ll, 658812288346769701ll, -576460752303423488ll, 512409557603043100ll};
  long long s = a[8];
#pragma unroll
  for (int i = 7; i >= 0; --i) s = a[i] + ((fx_mul(fx(s), h, l).v + 64) >> 7);
  if (k == 0 && t == 0) {
    if (r == 0) return 0.0;
    const int sh = __clzll((unsigned long long)(r < 0 ? -r : r)) - 2;
    digits(r << sh, h, l);
    return fx_to_double(fx_mul(fx(s), h, l).v, kBias - 62 - sh);
  }
  const int q = k == 0 ? 0 : 3;
  const long long rs = fx_mul(fx(s), h, l).v;          // r S(r), Q69
  // modulo 2^64: the magnitude of the sum takes all of its bits
  const unsigned long long v = (unsigned long long)((t + (1 << q >> 1)) >> q) + (unsigned long long)k * 1598288580650331957ull +
                               (unsigned long long)((rs + (16ll << q)) >> (5 + q));
  const bool neg = be < 1023;
  return fx_compose(neg ? 1ull << 63 : 0ull, neg ? 0ull - v : v, kBias - 64 + q);
}

// a / b, correctly rounded, on the integer pipe (an FP64 division costs about
// ten FP64 operations): the reciprocal of b's mantissa by two Newton steps in
// 62-bit fixed point from a float, the quotient's 53 bits from a product with it,
// off by at most one, and the exact remainder, which decides.  (With the product
// alone, or with a product by a rounded reciprocal, a quotient may round the
// other way.)  Zeros apart, operands and quotients that are not normal numbers
// take FP64 division.
struct FxDivisor {
  double b;
  unsigned long long m;   // mantissa, 53 bits
  int h, l;               // digits of 2^52 / m, Q62
  int e;                  // biased exponent, 0 where FP64 division serves
};

__device__ __forceinline__ FxDivisor fx_divisor(double b) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(b);
  FxDivisor d;
  d.b = b;
  d.e = (int)(u >> 52) & 0x7ff;
  d.m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  if (d.e == 0x7ff) d.e = 0;
  const float f = __uint_as_float(0x3f800000u | (unsigned int)((u >> 29) & 0x7fffffu));
  long long r = (long long)__float2uint_rn(__frcp_rn(f) * 2147483648.0f) << 31;               // [1/2, 1]
  digits(r, d.h, d.l);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const long long t = (1ll << 61) - fx_mul(fx((long long)(d.m << 9)), d.h, d.l).v;          // 1 - m r, Q61
    r += fx_mul(fx(t), d.h, d.l).v << 1;
    digits(r, d.h, d.l);
  }
  return d;
}

// 2^k pi, ready made.
__device__ __forceinline__ FxDivisor fx_pi(int k) {
  return FxDivisor{3.14159265358979323846 * (1 << k), 7074237752028440ull, 683565276, -1819212355, 1024 + k};
}

__device__ __forceinline__ double fx_div(double a, const FxDivisor& d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const unsigned long long sign = (u ^ (unsigned long long)__double_as_longlong(d.b)) & 0x8000000000000000ull;
  const int ea = (int)(u >> 52) & 0x7ff;
  const unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  const int s = m >= d.m ? 52 : 53;                      // quotient m 2^s / d.m in [2^52, 2^53)
  const int e = ea - d.e + 1023 + 52 - s;
  if (d.e == 0 || ea == 0 || ea == 0x7ff || e < 1 || e > 2046) {
    if (d.e != 0 && (u << 1) == 0) return __longlong_as_double((long long)sign);
    return a / d.b;
  }
  unsigned long long q = (unsigned long long)((fx_mul(fx((long long)(m << (s - 44))), d.h, d.l).v + 128) >> 8);
  const long long rem = (long long)((m << s) - q * d.m);   // modulo 2^64; |rem| < 2^54
  if (2 * rem > (long long)d.m) ++q;
  if (2 * rem < -(long long)d.m) --q;
  return __longlong_as_double((long long)(sign | (((unsigned long long)(e - 1) << 52) + q)));
}

}  // namespace gps
