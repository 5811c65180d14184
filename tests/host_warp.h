// A warp on the host: 32 lanes as coroutines that take turns at every warp
// operation, and the CUDA intrinsics that fixed_moments.cuh uses, so that the
// header's own arithmetic can be run and checked on the CPU.
#pragma once

#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
using std::max;
using std::min;

static struct { unsigned x; } threadIdx;
static ucontext_t warp_lane[32], warp_caller;
static bool warp_done[32];
static const std::function<void(int)>* warp_main;
static long long warp_slot[32];

// The next lane's turn: a lane runs on when every other has come as far.
static void next_lane() {
  const int me = threadIdx.x;
  for (int k = 1; k <= 32; ++k) {
    const int i = (me + k) & 31;
    if (!warp_done[i]) {
      threadIdx.x = i;
      if (i != me) swapcontext(&warp_lane[me], &warp_lane[i]);
      return;
    }
  }
  setcontext(&warp_caller);  // all done
}
static void lane_entry() {
  const int me = threadIdx.x;
  (*warp_main)(me);
  warp_done[me] = true;
  next_lane();
}

template <typename T> static T lane_value(int lane) {
  T v;
  memcpy(&v, &warp_slot[lane], sizeof(T));
  return v;
}
// every lane's value, combined by f after all have written theirs
template <typename T, typename F> static auto warp_exchange(T v, F f) {
  memcpy(&warp_slot[threadIdx.x], &v, sizeof(T));
  next_lane();
  auto r = f();
  next_lane();
  return r;
}
static inline unsigned __ballot_sync(unsigned, bool p) {
  return warp_exchange<int>(p, [] {
    unsigned m = 0;
    for (int i = 0; i < 32; ++i) m |= (unsigned)(lane_value<int>(i) != 0) << i;
    return m;
  });
}
static inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
static inline void __syncwarp() { next_lane(); }
template <typename T> static T __shfl_sync(unsigned, T v, int src) {
  return warp_exchange<T>(v, [=] { return lane_value<T>(src & 31); });
}
template <typename T> static T __shfl_xor_sync(unsigned, T v, int o) {
  const int src = threadIdx.x ^ o;
  return warp_exchange<T>(v, [=] { return lane_value<T>(src); });
}
static inline int __reduce_max_sync(unsigned, int v) {
  return warp_exchange<int>(v, [] {
    int r = lane_value<int>(0);
    for (int i = 1; i < 32; ++i) r = max(r, lane_value<int>(i));
    return r;
  });
}
static inline uint64_t double_bits(double v) { uint64_t b; memcpy(&b, &v, 8); return b; }
static inline int __double2hiint(double v) { return (int)(double_bits(v) >> 32); }
static inline int __double2loint(double v) { return (int)(uint32_t)double_bits(v); }
static inline double __hiloint2double(int hi, int lo) {
  const uint64_t b = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double v;
  memcpy(&v, &b, 8);
  return v;
}
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) {
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> (s & 31));
}
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) {
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32);
}
static inline int __ffs(unsigned m) { return __builtin_ffs((int)m); }
static inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }

static inline void run_warp(const std::function<void(int)>& lane_main) {
  constexpr size_t kStack = 1 << 18;
  std::vector<char> stacks(32 * kStack);
  warp_main = &lane_main;
  for (int i = 0; i < 32; ++i) {
    warp_done[i] = false;
    getcontext(&warp_lane[i]);
    warp_lane[i].uc_stack.ss_sp = stacks.data() + i * kStack;
    warp_lane[i].uc_stack.ss_size = kStack;
    warp_lane[i].uc_link = nullptr;
    makecontext(&warp_lane[i], lane_entry, 0);
  }
  threadIdx.x = 0;
  swapcontext(&warp_caller, &warp_lane[0]);
}
