// Quantities a DFT code takes from the generalized Poisson solve:
//
//   sccs dielectric (Eq. sccs): eps = 1 (rho_elec >= rho_max), eps0
//       (rho_elec <= rho_min), eps0^w in between, w = (z - sin z)/(2 pi),
//       z = 2 pi ln(rho_max / rho_elec) / ln(rho_max / rho_min) (the printed
//       middle branch eps0 exp(w) is discontinuous at both thresholds; eps0^w
//       is continuous), and d eps / d rho_elec;
//   polarization charge (Eqs. remap, rhopol): rho_pol = grad ln eps . grad phi
//       / 4 pi - ((eps - 1)/eps) rho (the sign Eq. remap requires);
//   v_eps (Eq. veps) = -(1/8 pi) (d eps / d rho_elec) |grad phi|^2;
//   electrostatic energy: (1/2) sum rho phi and (1/8 pi) sum eps |grad phi|^2
//       (times h^3, by the host).
//
// Gradients by the order-16 central differences of stencil16.cuh.  One-off
// post-processing passes: pointwise or one stencil per point, no iteration.
#include <algorithm>
#include <cmath>

#include "device_util.cuh"
#include "fixmath.cuh"
#include "gps_internal.h"
#include "kernels.h"

namespace gps {

constexpr int kTd = 256;

#define DFT_STRIDE(i, n) \
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (n); i += (size_t)gridDim.x * blockDim.x)

// Bound by the FP64 sincos and exp of the transition region; the logarithm and
// the divisions run on the integer pipe (periodic 128^3: 137 -> 81 us).
__global__ void k_sccs(const double* __restrict__ rho, double* __restrict__ eps, double* __restrict__ deps,
                       size_t n, double rmax, double rmin, double inv_lnr, double lne, double eps0) {
  DFT_STRIDE(i, n) {
    const double x = rho[i];
    double e, d = 0.0;
    if (x >= rmax) {
      e = 1.0;
    } else if (x <= rmin) {
      e = eps0;
    } else {
      const FxDivisor by_x = fx_divisor(x);
      const double z = 2.0 * kPi * fx_log(fx_div(rmax, by_x)) * inv_lnr;
      double sz, cz;
      sincos(z, &sz, &cz);
      e = exp(fx_div(z - sz, fx_pi(1)) * lne);
      d = fx_div(-e * lne * (1.0 - cz) * inv_lnr, by_x);
    }
    eps[i] = e;
    if (deps) deps[i] = d;
  }
}

__global__ void k_log(const double* __restrict__ eps, double* __restrict__ out, size_t n) {
  DFT_STRIDE(i, n) out[i] = fx_log(eps[i]);
}

// The stencil passes walk over tiles of the grid (stencil16.cuh): point (tx,
// ty, tz) of a tile belongs to thread tx + 32 ty, tz = 0 .. 7.
struct TileGrid {
  int tx, ty, tz;   // tiles per axis
};

__host__ __device__ inline TileGrid tile_grid(const Stencil16& s) {
  return TileGrid{(s.nx + Tile16::X - 1) / Tile16::X, (s.ny + Tile16::Y - 1) / Tile16::Y,
                  (s.nz + Tile16::Z - 1) / Tile16::Z};
}

#define TILE_LOOP(s)                                                                          \
  extern __shared__ __align__(16) unsigned char smem_raw[];                                   \
  Tile16& tile = *reinterpret_cast<Tile16*>(smem_raw);                                        \
  if (threadIdx.x < 2 * Tile16::X) tile.top[0][threadIdx.x] = 0;                                      \
  __syncthreads();                                                                            \
  const TileGrid tg = tile_grid(s);                                                           \
  const int ntiles = tg.tx * tg.ty * tg.tz;                                                   \
  for (int id = blockIdx.x; id < ntiles; id += gridDim.x)

#define TILE_POINTS(s)                                                                        \
  const int i0 = (id % tg.tx) * Tile16::X, j0 = (id / tg.tx % tg.ty) * Tile16::Y;             \
  const int k0 = id / (tg.tx * tg.ty) * Tile16::Z;                                            \
  const int i = i0 + (threadIdx.x & 31), j = j0 + (threadIdx.x >> 5);                         \
  auto inside = [&](int tz) { return i < s.nx && j < s.ny && k0 + tz < s.nz; };               \
  auto index = [&](int tz) { return ((size_t)(k0 + tz) * s.ny + j) * s.nx + i; };

// Measured at periodic 128^3 against FP64 differences, log() and divisions:
// k_log and k_pol together 910 -> 275 us, both energies 270 -> 126 us.  What is
// left is issue (about 62 instructions a value and axis, 2.0 of 4 issued a
// clock at two resident blocks) and some 30 us, in k_pol for the bulk solvent's
// potential, in each for one of cavities in a solvent, of telling zeros from values far
// below their lines' largest and of FP64 differences there.
__global__ void __launch_bounds__(Tile16::T, 2) k_pol(Stencil16 s, const double* __restrict__ lne,
                                                      const double* __restrict__ phi, const double* __restrict__ rho,
                                                      const double* __restrict__ eps, double* __restrict__ out) {
  TILE_LOOP(s) {
    TILE_POINTS(s)
    double acc[Tile16::Z];
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz) acc[tz] = 0.0;
    double a[Tile16::Z];
#pragma unroll 1
    for (int q = 0; q < 6; ++q) {        // each axis: grad ln eps, then grad phi
      double g[Tile16::Z];
      derivative16(tile, q >> 1, q & 1, q & 1 ? phi : lne, i0, j0, k0, s, g);
      const double ih = q < 2 ? s.ihx : q < 4 ? s.ihy : s.ihz;
#pragma unroll
      for (int tz = 0; tz < Tile16::Z; ++tz) {
        if (q & 1) acc[tz] = fma(a[tz] * g[tz], ih * ih, acc[tz]);
        else a[tz] = g[tz];
      }
    }
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz)
      if (inside(tz)) {
        const double e = eps[index(tz)];
        out[index(tz)] = fx_div(acc[tz], fx_pi(2)) - fx_div(e - 1.0, fx_divisor(e)) * rho[index(tz)];
      }
  }
}

// |grad phi|^2 at the thread's points.
__device__ __forceinline__ void grad_square(Tile16& t, const double* __restrict__ phi, int i0, int j0, int k0, int& turn,
                                            const Stencil16& s, double (&g2)[Tile16::Z]) {
#pragma unroll
  for (int tz = 0; tz < Tile16::Z; ++tz) g2[tz] = 0.0;
#pragma unroll 1
  for (int axis = 0; axis < 3; ++axis) {
    double g[Tile16::Z];
    derivative16(t, axis, turn, phi, i0, j0, k0, s, g);
    const double ih = axis == 0 ? s.ihx : axis == 1 ? s.ihy : s.ihz;
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz) g2[tz] = fma(g[tz] * g[tz], ih * ih, g2[tz]);
    turn ^= 1;
  }
}

__global__ void __launch_bounds__(Tile16::T, 2) k_veps(Stencil16 s, const double* __restrict__ deps,
                                                       const double* __restrict__ phi, double* __restrict__ out) {
  int turn = 0;
  TILE_LOOP(s) {
    TILE_POINTS(s)
    double d[Tile16::Z];
    bool any = false;
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz) {
      d[tz] = inside(tz) ? deps[index(tz)] : 0.0;
      any |= d[tz] != 0.0;   // outside the sccs transition d eps / d rho = 0
    }
    double g2[Tile16::Z];
    if (__syncthreads_or(any)) grad_square(tile, phi, i0, j0, k0, turn, s, g2);
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz)
      if (inside(tz)) out[index(tz)] = d[tz] != 0.0 ? fx_div(-d[tz] * g2[tz], fx_pi(3)) : 0.0;
  }
}

// Per-block partial sums of rho phi and eps |grad phi|^2 into part[2 b], part[2 b + 1].
__global__ void __launch_bounds__(Tile16::T, 2) k_energy(Stencil16 s, const double* __restrict__ rho,
                                                         const double* __restrict__ eps,
                                                         const double* __restrict__ phi, double* __restrict__ part) {
  double a = 0.0, b = 0.0;
  int turn = 0;
  TILE_LOOP(s) {
    TILE_POINTS(s)
    double g2[Tile16::Z];
    grad_square(tile, phi, i0, j0, k0, turn, s, g2);
#pragma unroll
    for (int tz = 0; tz < Tile16::Z; ++tz)
      if (inside(tz)) {
        a = fma(rho[index(tz)], phi[index(tz)], a);
        b = fma(eps[index(tz)], g2[tz], b);
      }
  }
  const double sa = block_sum(a);
  const double sb = block_sum(b);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = sa;
    part[2 * blockIdx.x + 1] = sb;
  }
}

int dft_blocks(size_t n) {
  size_t b = (n + kTd - 1) / kTd;
  if (b > 152 * 4) b = 152 * 4;
  return b < 1 ? 1 : (int)b;
}

void launch_sccs(const double* rho, double* eps, double* deps, size_t n, double rho_max, double rho_min,
                 double eps0, cudaStream_t st) {
  count_launch();
  k_sccs<<<dft_blocks(n), kTd, 0, st>>>(rho, eps, deps, n, rho_max, rho_min, 1.0 / std::log(rho_max / rho_min),
                                        std::log(eps0), eps0);
}

int tile_blocks(const Stencil16& s) {
  const TileGrid t = tile_grid(s);
  // two resident blocks an SM
  return std::min({t.tx * t.ty * t.tz, 152 * 2, dft_blocks((size_t)s.nx * s.ny * s.nz)});
}

template <typename K, typename... A>
static void launch_tiles(K kernel, const Stencil16& s, cudaStream_t st, A... args) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Tile16));
  count_launch();
  kernel<<<tile_blocks(s), Tile16::T, sizeof(Tile16), st>>>(s, args...);
}

void launch_polarization(const Stencil16& s, const double* rho, const double* eps, const double* phi,
                         double* tmp, double* out, size_t n, cudaStream_t st) {
  count_launch();
  k_log<<<dft_blocks(n), kTd, 0, st>>>(eps, tmp, n);
  launch_tiles(k_pol, s, st, (const double*)tmp, phi, rho, eps, out);
}

void launch_veps(const Stencil16& s, const double* deps, const double* phi, double* out, cudaStream_t st) {
  launch_tiles(k_veps, s, st, deps, phi, out);
}

void launch_energy(const Stencil16& s, const double* rho, const double* eps, const double* phi, double* part,
                   cudaStream_t st) {
  launch_tiles(k_energy, s, st, rho, eps, phi, part);
}

}  // namespace gps
