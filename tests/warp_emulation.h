// Runs a kernel of gts.cu on the host, one fiber per lane of one warp, under the thread sanitizer.  Each lane runs
// up to its next warp-wide call, then the next lane; only __syncwarp orders memory between lanes (a vote, shuffle or
// reduction does not), so the sanitizer reports accesses that no __syncwarp keeps apart.  Relaxed atomics stay atomic.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <ucontext.h>
#include <vector>

extern "C" {
void *__tsan_create_fiber(unsigned);
void __tsan_switch_to_fiber(void *, unsigned);
void *__tsan_get_current_fiber();
void __tsan_acquire(void *);
void __tsan_release(void *);
}

#define __device__
#define __host__
#define __global__
#define __grid_constant__
#define __forceinline__ inline
#define __noinline__
#define __restrict__
#define __launch_bounds__(...)
#define __align__(x)
#define UNSEEN __attribute__((no_sanitize("thread"), noinline))

struct alignas(8) uint2 { uint32_t x, y; };
struct alignas(16) uint4 { uint32_t x, y, z, w; };
inline uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
inline uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }
template <class A, class B> inline std::common_type_t<A, B> min(A a, B b) {
  using T = std::common_type_t<A, B>;
  return T(a) < T(b) ? T(a) : T(b);
}
template <class A, class B> inline std::common_type_t<A, B> max(A a, B b) {
  using T = std::common_type_t<A, B>;
  return T(a) > T(b) ? T(a) : T(b);
}

constexpr unsigned NO_SYNC = 1;  // a switch of fibers orders nothing
static ucontext_t main_ctx, lane_ctx[32];
static void *main_fiber, *lane_fiber[32];
static int cur_lane, line_of[32], start_object, sync_object;
static uint64_t vals[2][32];
static uint32_t phase[32];
static bool ended[32];
static void (*warp_body)();

UNSEEN static void to_main() {
  const int me = cur_lane;
  __tsan_switch_to_fiber(main_fiber, NO_SYNC);
  swapcontext(&lane_ctx[me], &main_ctx);
}
// Leaves v for the other lanes and returns what all of them left.
UNSEEN static const uint64_t *meet(uint64_t v, int line) {
  const int me = cur_lane, ph = phase[me] & 1;
  vals[ph][me] = v;
  line_of[me] = line;
  to_main();
  phase[me]++;
  return vals[ph];
}
UNSEEN static uint32_t reduce(uint32_t v, int line, int op) {
  const uint64_t *all = meet(v, line);
  uint32_t r = op == 0 ? ~0u : 0u;
  for (int i = 0; i < 32; i++) {
    const uint32_t x = (uint32_t)all[i];
    r = op == 0 ? (x < r ? x : r) : op == 1 ? (x > r ? x : r) : op == 2 ? r + x : r | (x ? 1u << i : 0u);
  }
  return r;
}
UNSEEN static uint64_t pick(uint64_t v, int src, int line) { return meet(v, line)[src & 31]; }
UNSEEN static int lane_now() { return cur_lane; }

#define __syncwarp() (__tsan_release(&sync_object), (void)meet(0, __LINE__), __tsan_acquire(&sync_object))
#define __reduce_min_sync(m, x) reduce(x, __LINE__, 0)
#define __reduce_max_sync(m, x) reduce(x, __LINE__, 1)
#define __reduce_add_sync(m, x) reduce(x, __LINE__, 2)
#define __ballot_sync(m, p) reduce((p) ? 1u : 0u, __LINE__, 3)
#define __any_sync(m, p) (reduce((p) ? 1u : 0u, __LINE__, 3) != 0u)
#define __shfl_sync(m, x, s) static_cast<decltype(+(x))>(pick((uint64_t)(x), (int)(s), __LINE__))
#define __shfl_xor_sync(m, x, o) static_cast<decltype(+(x))>(pick((uint64_t)(x), lane_now() ^ (o), __LINE__))
inline int __popc(uint32_t x) { return __builtin_popcount(x); }
inline int __ffs(uint32_t x) { return __builtin_ffs((int)x); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
template <class T> inline void __stcs(T *p, T v) { *p = v; }
inline void __threadfence() {}
inline uint32_t atomicAdd(uint32_t *p, uint32_t v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
inline uint32_t atomicSub(uint32_t *p, uint32_t v) { return __atomic_fetch_sub(p, v, __ATOMIC_RELAXED); }
inline uint32_t atomicOr(uint32_t *p, uint32_t v) { return __atomic_fetch_or(p, v, __ATOMIC_RELAXED); }
inline uint32_t atomicMax(uint32_t *p, uint32_t v) {
  uint32_t o = __atomic_load_n(p, __ATOMIC_RELAXED);
  while (o < v && !__atomic_compare_exchange_n(p, &o, v, true, __ATOMIC_RELAXED, __ATOMIC_RELAXED)) {}
  return o;
}
inline uint2 load_pair(const uint2 *p) {
  return {__atomic_load_n(&p->x, __ATOMIC_RELAXED), __atomic_load_n(&p->y, __ATOMIC_RELAXED)};
}
inline void store_pair(uint2 *p, uint32_t v) {
  __atomic_store_n(&p->x, v, __ATOMIC_RELAXED);
  __atomic_store_n(&p->y, v, __ATOMIC_RELAXED);
}

struct LaneIndex { struct X { operator unsigned() const { return (unsigned)lane_now(); } } x; } static threadIdx;
struct Dim { unsigned x; } static const blockIdx{0}, blockDim{32}, gridDim{1};
static uint32_t *shared_words;

UNSEEN static void lane_main() {
  __tsan_acquire(&start_object);
  warp_body();
  __tsan_release(&start_object);
  ended[cur_lane] = true;
  to_main();
}
UNSEEN static void run_warp(void (*body)(), bool backwards) {
  warp_body = body;
  __tsan_release(&start_object);
  main_fiber = __tsan_get_current_fiber();
  for (int i = 0; i < 32; i++) {
    lane_fiber[i] = __tsan_create_fiber(0);
    getcontext(&lane_ctx[i]);
    lane_ctx[i].uc_stack.ss_sp = malloc(1 << 18);
    lane_ctx[i].uc_stack.ss_size = 1 << 18;
    lane_ctx[i].uc_link = nullptr;
    makecontext(&lane_ctx[i], lane_main, 0);
  }
  for (int left = 32; left;) {
    left = 0;
    for (int k = 0; k < 32; k++) {
      const int i = backwards ? 31 - k : k;
      if (ended[i]) continue;
      cur_lane = i;
      __tsan_switch_to_fiber(lane_fiber[i], NO_SYNC);
      swapcontext(&main_ctx, &lane_ctx[i]);
      left += !ended[i];
    }
    for (int i = 0; i < 32; i++)
      if (ended[i] != ended[0] || line_of[i] != line_of[0]) {
        fprintf(stderr, "lane %d at line %d, lane 0 at line %d\n", i, line_of[i], line_of[0]);
        abort();
      }
  }
  __tsan_acquire(&start_object);
}
