// cuda_on_host.h -- what device functions need to run on the host, so that a
// test can compile them from the kernels' own source: the lanes of a warp are
// threads, warp operations are barriers over the lanes of their mask, and a
// variable that a warp shares is one copy per lane, brought up to date from
// lane 0 only by __syncwarp (the memory model promises no more).  A barrier
// that some lane of its mask does not reach ends the program with status 3.
#pragma once

#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __shared__
#define __restrict__
#define __noinline__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))
#define __CUDACC_ON_HOST__ 1
#define CUDART_INF_F INFINITY
#define CUDART_INF ((double)INFINITY)

struct Dim3 {
  unsigned x = 0, y = 0, z = 0;
};
static Dim3 gridDim, blockDim;
static thread_local Dim3 blockIdx, threadIdx;

// ---------------------------------------------------------------- lanes
struct Meeting {
  std::atomic<unsigned> waiting{0}, round{0};
};
struct WarpState {
  std::mutex mu;
  std::map<unsigned, Meeting> meetings;  // by mask
  uint64_t slot[32] = {};
  int* view[32] = {};                    // each lane's copy of the warp's shared int
  Meeting& meeting(unsigned m) {
    std::lock_guard<std::mutex> lk(mu);
    return meetings[m];
  }
};
static thread_local WarpState* warp_state = nullptr;
static inline int lane_id() { return (int)(threadIdx.x & 31u); }

static inline void meet(unsigned mask) {
  Meeting& M = warp_state->meeting(mask);
  const unsigned n = (unsigned)__builtin_popcount(mask), r = M.round.load();
  if (M.waiting.fetch_add(1) + 1 == n) {
    M.waiting.store(0);
    M.round.fetch_add(1);
    return;
  }
  const auto t0 = std::chrono::steady_clock::now();
  while (M.round.load() == r) {
    std::this_thread::yield();
    if (std::chrono::steady_clock::now() - t0 > std::chrono::seconds(20)) {
      fprintf(stderr, "a lane of mask %08x never came\n", mask);
      _Exit(3);
    }
  }
}

static inline void __syncwarp(unsigned mask = 0xFFFFFFFFu) {
  meet(mask);
  int* v = warp_state->view[lane_id()];
  if (v && warp_state->view[0] && lane_id() != 0) *v = *warp_state->view[0];
  meet(mask);
}
template <typename T>
static inline T __shfl_sync(unsigned mask, T v, int src) {
  uint64_t u = 0;
  memcpy(&u, &v, sizeof v);
  warp_state->slot[lane_id()] = u;
  meet(mask);
  u = warp_state->slot[src & 31];
  meet(mask);
  T r;
  memcpy(&r, &u, sizeof r);
  return r;
}
template <typename T>
static inline T __shfl_xor_sync(unsigned mask, T v, int x) {
  return __shfl_sync(mask, v, lane_id() ^ x);
}
static inline unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) {
  return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST);
}

// run f(lane) on n lanes of one warp
template <typename F>
static void on_lanes(int n, F f) {
  WarpState W;
  std::vector<std::thread> th;
  for (int l = 0; l < n; ++l)
    th.emplace_back([&W, l, &f] {
      warp_state = &W;
      threadIdx.x = (unsigned)l;
      f(l);
    });
  for (auto& t : th) t.join();
}

// ------------------------------------------------------------ arithmetic
static inline int __popc(unsigned v) { return __builtin_popcount(v); }
static inline int __ffs(unsigned v) { return v ? __builtin_ctz(v) + 1 : 0; }
static inline long long __double_as_longlong(double v) {
  long long u;
  memcpy(&u, &v, 8);
  return u;
}
static inline double __longlong_as_double(long long u) {
  double v;
  memcpy(&v, &u, 8);
  return v;
}
static inline int __double2hiint(double v) { return (int)(__double_as_longlong(v) >> 32); }
static inline int __double2loint(double v) { return (int)__double_as_longlong(v); }
static inline double __hiloint2double(int hi, int lo) {
  return __longlong_as_double((long long)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo));
}
static inline float __int_as_float(int u) {
  float v;
  memcpy(&v, &u, 4);
  return v;
}
static inline float __uint_as_float(unsigned u) { return __int_as_float((int)u); }
static inline float __saturatef(float v) { return v > 0.0f ? (v < 1.0f ? v : 1.0f) : 0.0f; }
static inline void sincospif(float x, float* s, float* c) {
  *s = (float)sin(M_PI * (double)x);
  *c = (float)cos(M_PI * (double)x);
}
static inline void sincospi(double x, double* s, double* c) {
  *s = sin(M_PI * x);
  *c = cos(M_PI * x);
}
template <typename T>
static inline T __ldg(const T* p) {
  return *p;
}
