// Device headers run on the host (host_cuda.h) for test_host_device_code.py.
#include <chrono>

#include "host_cuda.h"

#include "device_util.cuh"
#include "fft_common.cuh"
#include "fixmath.cuh"
#include "stencil16.cuh"

using namespace gps;

static void nap() { std::this_thread::sleep_for(std::chrono::milliseconds(20)); }

// Two derivatives in a row along `axis`, of u0 and of u1, on the tile at the
// origin, as the passes call them; thread 0 leaves every barrier late.
extern "C" void derivative_pair(const Stencil16* s, int axis, const double* u0, const double* u1, double* d0,
                                double* d1) {
  static Tile16 tile;
  for (int i = 0; i < 2 * Tile16::X; ++i) tile.top[0][i] = 0;
  host_cuda::after_barrier = [](int t) {
    if (t == 0) nap();
  };
  host_cuda::run_block(Tile16::T, [&] {
    double a[Tile16::Z], b[Tile16::Z];
    derivative16(tile, axis, 0, u0, 0, 0, 0, *s, a);
    derivative16(tile, axis, 1, u1, 0, 0, 0, *s, b);
    for (int z = 0; z < Tile16::Z; ++z) {
      d0[z * Tile16::T + threadIdx.x] = a[z];
      d1[z * Tile16::T + threadIdx.x] = b[z];
    }
  });
  host_cuda::after_barrier = nullptr;
}

// d -> fixed point -> double, with the mantissa shifted down by `drop` bits
// and the exponent moved by the same and by k.
extern "C" void fixed_round_trip(const double* d, double* out, int n, int drop, int k) {
  for (int i = 0; i < n; ++i) {
    long long m;
    int e;
    fx_of_double(d[i], m, e);
    out[i] = fx_to_double(m >> drop, e + drop + k);
  }
}

extern "C" void fixed_log(const double* x, double* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_log(x[i]);
}

extern "C" void fixed_divide(const double* a, const double* b, double* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_div(a[i], fx_divisor(b[i]));
}
extern "C" void fixed_divide_by_pi(const double* a, double* out, int n, int k) {
  for (int i = 0; i < n; ++i) out[i] = fx_div(a[i], fx_pi(k));
}

extern "C" void fixed_digits(const long long* w, long long* out, int n) {
  for (int i = 0; i < n; ++i) {
    const long long d = q62_digits(w[i]);
    out[i] = (long long)hi32(d) * 4294967296ll + lo32(d);
    if (lo32(d) == (int)0x80000000) out[i] = 1ll << 63;   // has no negative
  }
}

// out[i] = X_1 + X_2 - (2 x_0 - x_1 - x_2) of three-point transforms, real part.
extern "C" void fixed_radix3(const long long* x, long long* out, int n, int forward) {
  for (int i = 0; i < n; ++i) {
    i64c v[3] = {{fx(x[3 * i]), fx(0)}, {fx(x[3 * i + 1]), fx(0)}, {fx(x[3 * i + 2]), fx(0)}};
    if (forward) Dft<i64c, -1, 3>::run(v);
    else Dft<i64c, +1, 3>::run(v);
    out[i] = v[1].x.v + v[2].x.v - (2 * x[3 * i] - x[3 * i + 1] - x[3 * i + 2]);
  }
}

// Error, in units, of the second of two packed values where the first's
// exponent is `shift` higher; i counts positions in a line.
extern "C" void fixed_align(const long long* m, double* out, int n, int shift) {
  for (int i = 0; i < n; ++i) {
    i64c a = fx_pack_normalized(1ll << 61, 0, 2000 + shift), b = fx_pack_normalized(m[i], m[i], 2000);
    const long long w = packed_man(b.x.v);
    int e;
    fx_align(a, b, e, i & 1);
    out[i] = std::ldexp((double)((b.x.v << (shift + 1)) - w), -(shift + 1));
  }
}

// Real part, in units, of x times a factor whose real part is +-1/2, less its
// exact value.
extern "C" void fixed_half_product(const long long* x, double* out, int n, int negative) {
  const long long c = negative ? -(1ll << 61) : 1ll << 61;
  const i64c w{fx(q62_digits(c)), fx(q62_digits(3993765219463853012ll))};   // sqrt(3)/2
  for (int i = 0; i < n; ++i) {
    const i64c p = cmul(i64c{fx(x[i]), fx(0)}, w);
    out[i] = (double)(2 * p.x.v - (negative ? -x[i] : x[i])) / 2;
  }
}

// One block's K = 3 grid reduction: out[k] = partial k as a thread that takes
// the ticket has published it, i.e. at that thread's last fence; later warps
// leave every barrier late.
extern "C" void published_partials(double* out) {
  static double part[3];
  static unsigned int counter;
  double seen[3] = {-1.0, -1.0, -1.0}, res[3];
  for (double& x : part) x = -1.0;
  counter = 0;
  gridDim = {2, 1, 1};                   // not the last block
  host_cuda::after_barrier = [](int t) {
    if (t >= 32) nap();
  };
  host_cuda::on_fence = [&](int t) {
    if (t == 0) std::memcpy(seen, part, sizeof seen);
  };
  host_cuda::on_ticket = [&] { std::memcpy(out, seen, sizeof seen); };
  host_cuda::run_block(128, [&] {
    const double v[3] = {1.0, 2.0, 3.0};
    double* const p[3] = {&part[0], &part[1], &part[2]};
    double* const r[3] = {&res[0], &res[1], &res[2]};
    grid_reduce_k(v, p, &counter, r);
  });
  host_cuda::after_barrier = nullptr;
  host_cuda::on_fence = nullptr;
  host_cuda::on_ticket = nullptr;
  gridDim = {1, 1, 1};
}
