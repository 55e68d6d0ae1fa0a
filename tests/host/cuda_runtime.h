// Stand-in for the CUDA runtime header that lets a kernel's source be compiled by a
// plain C++20 compiler and run as one CTA on host threads, one per CUDA thread: for
// checks of barriers, shared memory and index arithmetic that a GPU run cannot make
// or must not make.  Barriers and warp collectives are real (std::barrier); hold()
// delays one warp after one of its CTA barriers, which every schedule of the GPU's
// warps may do.  Included in place of <cuda_runtime.h> by the tests' include path.
#pragma once

#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <barrier>
#include <chrono>
#include <cmath>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#define __host__
#define __device__
#define __global__
#define __forceinline__ inline
#define __shared__ static
#define __launch_bounds__(...)
#define __align__(n) alignas(n)

using std::max;
using std::min;
using std::fma;
using std::isfinite;

struct uint3 { unsigned x, y, z; };
struct int2 { int x, y; };
inline thread_local uint3 threadIdx{}, blockIdx{};
inline uint3 blockDim{1, 1, 1}, gridDim{1, 1, 1};

namespace host_cta {

struct Warp {
  std::barrier<> sync{32};
  unsigned long long word[32];
};

struct Cta {
  std::unique_ptr<std::barrier<>> all;
  std::vector<std::unique_ptr<Warp>> warps;
  int held_warp = -1, held_at = -1;
};

inline Cta cta;
inline thread_local int passed = 0;   // CTA barriers this thread has passed
inline std::mutex atomics;

// The warp that waits 20 ms after its n-th CTA barrier (counted from 0).
inline void hold(int warp, int n) {
  cta.held_warp = warp;
  cta.held_at = n;
}

inline Warp& warp() { return *cta.warps[threadIdx.x >> 5]; }

// Runs `kernel` on `threads` host threads (a multiple of 32).
inline void run(int threads, const std::function<void()>& kernel) {
  cta.all = std::make_unique<std::barrier<>>(threads);
  cta.warps.clear();
  for (int w = 0; w < threads / 32; ++w) cta.warps.push_back(std::make_unique<Warp>());
  blockDim = {(unsigned)threads, 1, 1};
  std::vector<std::thread> pool;
  for (int t = 0; t < threads; ++t)
    pool.emplace_back([&, t] {
      threadIdx = {(unsigned)t, 0, 0};
      blockIdx = {0, 0, 0};
      passed = 0;
      kernel();
      cta.all->arrive_and_drop();   // an exited thread counts as arrived
    });
  for (auto& th : pool) th.join();
}

template <typename T>
unsigned long long to_word(T v) {
  static_assert(sizeof(T) <= 8);
  unsigned long long w = 0;
  memcpy(&w, &v, sizeof(T));
  return w;
}
template <typename T>
T of_word(unsigned long long w) {
  T v;
  memcpy(&v, &w, sizeof(T));
  return v;
}

}  // namespace host_cta

inline void __syncthreads() {
  using namespace host_cta;
  cta.all->arrive_and_wait();
  if ((int)(threadIdx.x >> 5) == cta.held_warp && passed == cta.held_at)
    std::this_thread::sleep_for(std::chrono::milliseconds(20));
  ++passed;
}
inline void __syncwarp(unsigned = 0xffffffffu) { host_cta::warp().sync.arrive_and_wait(); }

template <typename T>
T __shfl_sync(unsigned, T v, int src) {
  host_cta::Warp& w = host_cta::warp();
  w.word[threadIdx.x & 31] = host_cta::to_word(v);
  w.sync.arrive_and_wait();
  const T r = host_cta::of_word<T>(w.word[src & 31]);
  w.sync.arrive_and_wait();
  return r;
}
template <typename T>
T __shfl_xor_sync(unsigned m, T v, int off) { return __shfl_sync(m, v, (int)(threadIdx.x & 31) ^ off); }
inline unsigned __ballot_sync(unsigned, bool p) {
  host_cta::Warp& w = host_cta::warp();
  w.word[threadIdx.x & 31] = p;
  w.sync.arrive_and_wait();
  unsigned r = 0;
  for (int l = 0; l < 32; ++l) r |= (unsigned)(w.word[l] & 1u) << l;
  w.sync.arrive_and_wait();
  return r;
}
inline int __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
inline int __reduce_max_sync(unsigned m, int v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(m, v, o));
  return v;
}

inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __popcll(unsigned long long v) { return __builtin_popcountll(v); }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __ffsll(long long v) { return __builtin_ffsll(v); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (hi << s) | (lo >> (32 - s)); }
inline long long __double_as_longlong(double v) { return host_cta::of_word<long long>(host_cta::to_word(v)); }
inline double __longlong_as_double(long long v) { return host_cta::of_word<double>(host_cta::to_word(v)); }
inline int __double2hiint(double v) { return (int)(__double_as_longlong(v) >> 32); }
inline int __double2loint(double v) { return (int)(__double_as_longlong(v) & 0xffffffffll); }
inline int __float_as_int(float v) { return host_cta::of_word<int>(host_cta::to_word(v)); }
inline float __int_as_float(int v) { return host_cta::of_word<float>(host_cta::to_word(v)); }
inline float __uint_as_float(unsigned v) { return host_cta::of_word<float>(host_cta::to_word(v)); }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fmul_rn(float a, float b) { return a * b; }

template <typename T>
T __ldcg(const T* p) { return *p; }
inline void __threadfence() {}

template <typename T, class Op>
T host_atomic(T* p, Op op) {
  std::lock_guard<std::mutex> lock(host_cta::atomics);
  const T old = *p;
  *p = op(old);
  return old;
}
template <typename T, typename V>
T atomicMax(T* p, V v) { return host_atomic(p, [&](T o) { return max(o, (T)v); }); }
template <typename T, typename V>
T atomicMin(T* p, V v) { return host_atomic(p, [&](T o) { return min(o, (T)v); }); }
template <typename T, typename V>
T atomicOr(T* p, V v) { return host_atomic(p, [&](T o) { return o | (T)v; }); }
template <typename T, typename V>
T atomicAdd(T* p, V v) { return host_atomic(p, [&](T o) { return o + (T)v; }); }

// The runtime calls of the host code under test; a test may let the n-th allocation fail.
typedef int cudaError_t;
typedef struct host_stream* cudaStream_t;
typedef struct host_graph* cudaGraphExec_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
namespace host_cta {
inline std::vector<void*> blocks;   // allocated and not freed
inline int allocations = 0, fail_at = -1;
}  // namespace host_cta
inline cudaError_t cudaMalloc(void** p, size_t bytes) {
  using namespace host_cta;
  if (allocations++ == fail_at) return cudaErrorMemoryAllocation;   // *p is left as it was
  *p = malloc(bytes);
  blocks.push_back(*p);
  return cudaSuccess;
}
inline cudaError_t cudaFree(void* p) {
  auto& b = host_cta::blocks;
  const auto at = std::find(b.begin(), b.end(), p);
  if (at == b.end()) abort();   // freed twice, or never allocated
  b.erase(at);
  free(p);
  return cudaSuccess;
}
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
