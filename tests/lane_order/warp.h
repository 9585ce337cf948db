// Runs warp-level device code on the host, one thread per lane, so that a data race
// detector (-fsanitize=thread) sees the memory ordering the CUDA programming model
// gives: __syncwarp and __syncthreads order the lanes' accesses; votes, shuffles, matches
// and reductions exchange values but order nothing.
#pragma once
#include <sched.h>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <atomic>
#include <thread>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __shared__
#define __align__(n) __attribute__((aligned(n)))

struct Dim { int x = 0; };
extern thread_local Dim threadIdx, blockIdx;
extern Dim blockDim, gridDim;
thread_local Dim threadIdx, blockIdx;
Dim blockDim, gridDim;

using std::max;
using std::min;
constexpr int kLanes = 32;
static unsigned long long g_slot[kLanes];
static int g_arrived;
static unsigned g_gen;

// The rendezvous of a collective, which the race detector does not see.
__attribute__((no_sanitize("thread"), noinline)) static void meet() {
  const unsigned g = __atomic_load_n(&g_gen, __ATOMIC_SEQ_CST);
  if (__atomic_add_fetch(&g_arrived, 1, __ATOMIC_SEQ_CST) == kLanes) {
    __atomic_store_n(&g_arrived, 0, __ATOMIC_SEQ_CST);
    __atomic_store_n(&g_gen, g + 1, __ATOMIC_SEQ_CST);
  } else {
    while (__atomic_load_n(&g_gen, __ATOMIC_SEQ_CST) == g) sched_yield();
  }
}
__attribute__((no_sanitize("thread"), noinline)) static void exchange(unsigned long long v,
                                                                      unsigned long long* all) {
  __atomic_store_n(&g_slot[threadIdx.x & 31], v, __ATOMIC_SEQ_CST);
  meet();
  for (int l = 0; l < kLanes; ++l) all[l] = __atomic_load_n(&g_slot[l], __ATOMIC_SEQ_CST);
  meet();
}

template <class T>
static unsigned long long bits_of(T v) {
  unsigned long long u = 0;
  std::memcpy(&u, &v, sizeof(T));
  return u;
}
template <class T>
static T of_bits(unsigned long long u) {
  T v;
  std::memcpy(&v, &u, sizeof(T));
  return v;
}

// Orders the lanes' accesses, and the race detector sees it.
static std::atomic<int> g_sync_n{0};
static std::atomic<unsigned> g_sync_gen{0};
inline void __syncwarp(unsigned = 0xffffffffu) {
  const unsigned g = g_sync_gen.load();
  if (g_sync_n.fetch_add(1) + 1 == kLanes) {
    g_sync_n.store(0);
    g_sync_gen.store(g + 1);
  } else {
    while (g_sync_gen.load() == g) sched_yield();
  }
}
inline void __syncthreads() { __syncwarp(); }  // (one warp at a time runs here)

template <class T>
T __shfl_sync(unsigned, T v, int src, int width = 32) {
  unsigned long long a[kLanes];
  exchange(bits_of(v), a);
  return of_bits<T>(a[((threadIdx.x & 31) & ~(width - 1)) + (src & (width - 1))]);
}
template <class T>
T __shfl_up_sync(unsigned, T v, int d) {
  unsigned long long a[kLanes];
  exchange(bits_of(v), a);
  const int l = threadIdx.x & 31;
  return of_bits<T>(a[l >= d ? l - d : l]);
}
template <class T>
T __shfl_xor_sync(unsigned, T v, int d, int = 32) {
  unsigned long long a[kLanes];
  exchange(bits_of(v), a);
  return of_bits<T>(a[(threadIdx.x & 31) ^ d]);
}
inline unsigned __ballot_sync(unsigned, bool p) {
  unsigned long long a[kLanes];
  exchange(p, a);
  unsigned m = 0;
  for (int l = 0; l < kLanes; ++l) m |= (unsigned)(a[l] != 0) << l;
  return m;
}
inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
inline bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == 0xffffffffu; }
inline unsigned __match_any_sync(unsigned, int v) {
  unsigned long long a[kLanes];
  exchange(bits_of(v), a);
  unsigned m = 0;
  for (int l = 0; l < kLanes; ++l) m |= (unsigned)(of_bits<int>(a[l]) == v) << l;
  return m;
}
inline int __reduce_max_sync(unsigned, int v) {
  unsigned long long a[kLanes];
  exchange(bits_of(v), a);
  int r = of_bits<int>(a[0]);
  for (int l = 1; l < kLanes; ++l) r = max(r, of_bits<int>(a[l]));
  return r;
}

inline int __popc(unsigned m) { return __builtin_popcount(m); }
inline int __ffs(unsigned m) { return __builtin_ffs((int)m); }
inline double __fma_rn(double a, double b, double c) { return __builtin_fma(a, b, c); }
inline void __nanosleep(unsigned) {}
template <class T>
T __ldcg(const T* p) { return *p; }
inline int atomicCAS(int* p, int expect, int v) {
  __atomic_compare_exchange_n(p, &expect, v, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED);
  return expect;
}
inline int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
inline unsigned atomicAdd(unsigned* p, unsigned v) {
  return __atomic_fetch_add(p, v, __ATOMIC_RELAXED);
}
inline int ld_volatile_i32(const int* p) { return __atomic_load_n(p, __ATOMIC_RELAXED); }
inline int ld_acquire_i32(const int* p) { return __atomic_load_n(p, __ATOMIC_ACQUIRE); }
inline void st_release_i32(int* p, int v) { __atomic_store_n(p, v, __ATOMIC_RELEASE); }

inline unsigned long long dmag(double x) { return bits_of(x) & 0x7fffffffffffffffull; }
inline bool d_isnan(double x) { return x != x; }
inline bool d_eq0(double x) { return x == 0.0; }
inline bool d_gt0(double x) { return x > 0.0; }
inline bool d_lt0(double x) { return x < 0.0; }

// f on the 32 lanes of warp `warp` of block 0.
template <class F>
void run_warp(int warp, F f) {
  std::vector<std::thread> t;
  for (int l = 0; l < kLanes; ++l)
    t.emplace_back([=] {
      threadIdx.x = 32 * warp + l;
      blockIdx.x = 0;
      f();
    });
  for (auto& x : t) x.join();
}
