// Runs the library's device headers on the host: one block at a time, a
// std::thread per CUDA thread, barriers and warp collectives in lock step, so
// that their arithmetic and the order of their shared accesses can be tested
// without a GPU.  `after_barrier` delays threads of the tester's choice when
// they leave a block barrier: a schedule that the hardware may take.
#pragma once

#include <atomic>
#include <barrier>
#include <bit>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#undef __shared__
#define __shared__ static
#ifndef __CUDACC__
#define __CUDACC__
#endif

namespace host_cuda {
struct Idx { unsigned int x = 0, y = 0, z = 0; };
struct Warp {
  std::barrier<> bar{32};
  uint64_t v[32];
};
struct Block {
  std::barrier<> bar;
  std::vector<std::unique_ptr<Warp>> warps;
  explicit Block(int threads) : bar(threads) {
    for (int w = 0; w < threads / 32; ++w) warps.push_back(std::make_unique<Warp>());
  }
};
inline Block* block = nullptr;
inline std::mutex atomics;
inline std::function<void(int)> after_barrier, on_fence;   // argument: the thread
inline std::function<void()> on_ticket;                     // an atomicAdd, before it is made

// Runs f in every thread of one block (a multiple of 32 threads).
template <typename F> void run_block(int threads, F f);
}  // namespace host_cuda

inline thread_local host_cuda::Idx threadIdx;
inline host_cuda::Idx blockIdx, gridDim{1, 1, 1}, blockDim;

template <typename F> void host_cuda::run_block(int threads, F f) {
  Block b(threads);
  block = &b;
  blockDim = {(unsigned)threads, 1, 1};
  std::vector<std::thread> t;
  for (int i = 0; i < threads; ++i)
    t.emplace_back([&, i] {
      threadIdx = {(unsigned)i, 0, 0};
      f();
    });
  for (auto& x : t) x.join();
  block = nullptr;
}

inline void __syncthreads() {
  host_cuda::block->bar.arrive_and_wait();
  if (host_cuda::after_barrier) host_cuda::after_barrier((int)threadIdx.x);
}
inline int __syncthreads_or(int v) {
  static std::atomic<int> any{0};
  if (v) any = 1;
  __syncthreads();
  const int r = any;
  host_cuda::block->bar.arrive_and_wait();
  if (threadIdx.x == 0) any = 0;
  __syncthreads();
  return r;
}
inline void __threadfence_block() {}
inline void __threadfence() {
  if (host_cuda::on_fence) host_cuda::on_fence((int)threadIdx.x);
}

// g(values of the warp's lanes, own lane) after all lanes have posted theirs
template <typename T, typename G> T host_warp(T v, G g) {
  host_cuda::Warp& w = *host_cuda::block->warps[threadIdx.x / 32];
  const int lane = threadIdx.x % 32;
  w.v[lane] = 0;
  std::memcpy(&w.v[lane], &v, sizeof v);
  w.bar.arrive_and_wait();
  const T r = g([&](int l) {
    T x;
    std::memcpy(&x, &w.v[l], sizeof x);
    return x;
  }, lane);
  w.bar.arrive_and_wait();
  return r;
}
template <typename T> T __shfl_down_sync(unsigned, T v, int o) {
  return host_warp(v, [&](auto at, int l) { return at(l + o < 32 ? l + o : l); });
}
inline int __reduce_max_sync(unsigned, int v) {
  return host_warp(v, [](auto at, int) {
    int m = at(0);
    for (int l = 1; l < 32; ++l) m = at(l) > m ? at(l) : m;
    return m;
  });
}
inline unsigned int __ballot_sync(unsigned, int v) {
  return host_warp(v, [](auto at, int) {
    unsigned int b = 0;
    for (int l = 0; l < 32; ++l) b |= (at(l) != 0 ? 1u : 0u) << l;
    return (int)b;
  });
}
inline int __any_sync(unsigned m, int v) { return __ballot_sync(m, v) != 0; }
template <typename T> T __shfl_sync(unsigned, T v, int from) {
  return host_warp(v, [&](auto at, int) { return at(from & 31); });
}
inline void __syncwarp() { host_cuda::block->warps[threadIdx.x / 32]->bar.arrive_and_wait(); }
inline int atomicMax(int* p, int v) {
  std::lock_guard<std::mutex> lock(host_cuda::atomics);
  const int old = *p;
  if (v > old) *p = v;
  return old;
}
inline unsigned int atomicAdd(unsigned int* p, unsigned int v) {
  std::lock_guard<std::mutex> lock(host_cuda::atomics);
  if (host_cuda::on_ticket) host_cuda::on_ticket();
  const unsigned int old = *p;
  *p += v;
  return old;
}

inline int min(int a, int b) { return a < b ? a : b; }
inline int max(int a, int b) { return a > b ? a : b; }
template <typename T> T __ldg(const T* p) { return *p; }
template <typename T> T __ldcg(const T* p) { return *p; }
inline int __clz(int v) { return std::countl_zero((unsigned int)v); }
inline int __popc(unsigned int v) { return std::popcount(v); }
inline int __ffs(int v) { return v ? std::countr_zero((unsigned int)v) + 1 : 0; }
inline int __clzll(long long v) { return std::countl_zero((unsigned long long)v); }
inline long long __double_as_longlong(double d) { return std::bit_cast<long long>(d); }
inline double __longlong_as_double(long long v) { return std::bit_cast<double>(v); }
inline int __double2hiint(double d) { return (int)(std::bit_cast<long long>(d) >> 32); }
inline unsigned int __float_as_uint(float f) { return std::bit_cast<unsigned int>(f); }
inline float __uint_as_float(unsigned int u) { return std::bit_cast<float>(u); }
inline float __frcp_rn(float f) { return 1.0f / f; }
inline unsigned int __float2uint_rn(float f) { return (unsigned int)std::nearbyint(f); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
