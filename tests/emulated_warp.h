// A warp of 32 host threads for device functions whose lanes meet in warp-wide
// operations: each `_sync` operation waits for the lanes of its mask that have
// not returned, at the same place in the source, as the language asks. When no
// lane can go on (some wait at one place, the others at another), or a shuffle
// reads a lane that has returned, the run is a fault: `run_warp` gives false.
#pragma once

#include <algorithm>
#include <cfenv>
#include <climits>
#include <cmath>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <thread>
#include <utility>
#include <vector>

namespace emu {

struct Dim {
  unsigned x = 0, y = 0, z = 0;
};

struct Fault {};

struct Meeting {
  unsigned arrived = 0;   // lanes here
  unsigned members = 0;   // lanes that left together (set on completion)
  int to_leave = 0;
  unsigned long long value[32];
};

struct Warp {
  std::mutex m;
  std::condition_variable cv;
  unsigned live = 0xffffffffu, waiting = 0;
  bool fault = false;
  std::map<std::pair<int, unsigned>, Meeting> at;

  void complete_all() {
    bool some = false;
    for (auto& kv : at) {
      Meeting& q = kv.second;
      if (!q.members && q.arrived && q.arrived == (kv.first.second & live)) {
        q.members = q.arrived;
        q.to_leave = __builtin_popcount(q.arrived);
        waiting &= ~q.arrived;
        some = true;
      }
    }
    if (!some && live && waiting == live) fault = true;  // (none waits at the CTA's barrier)
    cv.notify_all();
  }
};

// A CTA's barrier: every thread that has not returned.
struct Cta {
  std::mutex m;
  std::condition_variable cv;
  unsigned live = 0, arrived = 0;
  unsigned long long turn = 0;

  void release() {
    if (arrived && arrived == live) {
      arrived = 0;
      ++turn;
      cv.notify_all();
    }
  }
};

inline thread_local Warp* g_warp = nullptr;
inline thread_local Cta* g_cta = nullptr;
inline thread_local unsigned t_thread = 0, t_lane = 0;

inline void cta_barrier() {
  Cta& c = *g_cta;
  std::unique_lock<std::mutex> lock(c.m);
  const unsigned long long turn = c.turn;
  ++c.arrived;
  c.release();
  c.cv.wait(lock, [&] { return c.turn != turn; });
}

// Meets the lanes of `mask` at source line `line`; every lane's value, and the
// lanes that took part.
inline unsigned meet(int line, unsigned mask, unsigned long long v, unsigned long long* all) {
  Warp& w = *g_warp;
  std::unique_lock<std::mutex> lock(w.m);
  Meeting& q = w.at[{line, mask}];
  w.cv.wait(lock, [&] { return w.fault || !q.members; });  // the last meeting here has left
  if (w.fault) throw Fault();
  q.value[t_lane] = v;
  q.arrived |= 1u << t_lane;
  w.waiting |= 1u << t_lane;
  w.complete_all();
  w.cv.wait(lock, [&] { return w.fault || (q.members >> t_lane & 1u); });
  if (w.fault) throw Fault();
  const unsigned members = q.members;
  std::memcpy(all, q.value, sizeof(q.value));
  if (--q.to_leave == 0) {
    q.arrived = q.members = 0;
    w.cv.notify_all();
  }
  return members;
}

inline unsigned ballot(int line, unsigned mask, bool p) {
  unsigned long long all[32];
  const unsigned members = meet(line, mask, p, all);
  unsigned out = 0;
  for (unsigned i = 0; i < 32; ++i)
    if ((members >> i & 1u) && all[i]) out |= 1u << i;
  return out;
}

template <class T>
T from_lane(int line, unsigned mask, T v, unsigned src) {
  static_assert(sizeof(T) <= 8, "one word a lane");
  unsigned long long all[32], mine = 0;
  std::memcpy(&mine, &v, sizeof(T));
  const unsigned members = meet(line, mask, mine, all);
  if (!(members >> src & 1u)) {
    std::lock_guard<std::mutex> lock(g_warp->m);
    g_warp->fault = true;
    g_warp->cv.notify_all();
    throw Fault();
  }
  std::memcpy(&v, &all[src], sizeof(T));
  return v;
}

template <class T>
T shfl(int line, unsigned mask, T v, int src, int width = 32) {
  const unsigned base = t_lane & ~static_cast<unsigned>(width - 1);
  return from_lane(line, mask, v, base + (static_cast<unsigned>(src) & static_cast<unsigned>(width - 1)));
}

template <class T>
unsigned match_any(int line, unsigned mask, T v) {
  unsigned long long all[32], mine = 0;
  std::memcpy(&mine, &v, sizeof(T));
  const unsigned members = meet(line, mask, mine, all);
  unsigned out = 0;
  for (unsigned i = 0; i < 32; ++i)
    if ((members >> i & 1u) && all[i] == mine) out |= 1u << i;
  return out;
}

// The threads of a CTA (whole warps) run f(thread); false when the lanes of a
// warp could not all go on.
inline bool run_cta(unsigned threads, const std::function<void(unsigned)>& f) {
  std::vector<Warp> warps(threads / 32);
  Cta cta;
  cta.live = threads;
  std::vector<std::thread> run;
  for (unsigned t = 0; t < threads; ++t)
    run.emplace_back([&, t] {
      Warp& w = warps[t / 32];
      g_warp = &w;
      g_cta = &cta;
      t_thread = t;
      t_lane = t & 31u;
      try {
        f(t);
      } catch (const Fault&) {
      }
      {
        std::lock_guard<std::mutex> lock(w.m);
        w.live &= ~(1u << t_lane);
        w.complete_all();
      }
      std::lock_guard<std::mutex> lock(cta.m);
      --cta.live;
      cta.release();
    });
  for (auto& t : run) t.join();
  return std::none_of(warps.begin(), warps.end(), [](const Warp& w) { return w.fault; });
}

inline bool run_warp(const std::function<void(unsigned)>& f) { return run_cta(32, f); }

// memory operations that the device code writes in PTX
template <class K, class P>
void ld_relaxed_gpu_global_u64(K& k, P p) { k = *reinterpret_cast<const volatile unsigned long long*>(p); }
template <class K, class P>
void ld_relaxed_gpu_global_u32(K& k, P p) { k = *reinterpret_cast<const volatile unsigned*>(p); }
inline unsigned g_entry_loads = 0;  // table entries read
template <class K, class P>
void ld_global_ca_v2_u64(K& a, K& b, P p) {
  __atomic_fetch_add(&g_entry_loads, 1u, __ATOMIC_SEQ_CST);
  a = reinterpret_cast<const volatile unsigned long long*>(p)[0];
  b = reinterpret_cast<const volatile unsigned long long*>(p)[1];
}
template <class K, class P>
void ld_global_cg_v2_u64(K& a, K& b, P p) { ld_global_ca_v2_u64(a, b, p); }
inline std::mutex g_red;
inline void red_relaxed_gpu_global_add_f32(float* p, float v) {
  std::lock_guard<std::mutex> lock(g_red);
  *p += v;
}
template <class Q>
void red_relaxed_gpu_global_add_v4_f32(Q* p, float a, float b, float c, float d) {
  std::lock_guard<std::mutex> lock(g_red);
  p->x += a; p->y += b; p->z += c; p->w += d;
}
template <class Q>
void red_relaxed_gpu_global_add_v2_f32(Q* p, float a, float b) {
  std::lock_guard<std::mutex> lock(g_red);
  p->x += a; p->y += b;
}
inline void red_relaxed_gpu_global_add_u32(unsigned* p, unsigned v) { __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
template <class T>
void mov_u64(T& t) { t = 0; }

}  // namespace emu

// the names that device code uses
#define __host__
#define __device__
#define __global__
#define __shared__ static
#define __forceinline__ inline
#define __noinline__
#define __grid_constant__
#define __launch_bounds__(...)
#define __align__(n) alignas(n)
#define __ballot_sync(m, p) emu::ballot(__LINE__, m, p)
#define __any_sync(m, p) (emu::ballot(__LINE__, m, p) != 0)
#define __syncwarp() emu::ballot(__LINE__, 0xffffffffu, true)
#define __shfl_sync(m, ...) emu::shfl(__LINE__, m, __VA_ARGS__)
#define __match_any_sync(m, v) emu::match_any(__LINE__, m, v)
#define __syncthreads() emu::cta_barrier()
#define threadIdx (emu::Dim{emu::t_thread, 0, 0})
#define blockIdx (emu::Dim{0, 0, 0})
#define blockDim (emu::Dim{256, 1, 1})

struct float2 { float x, y; };
struct alignas(16) float4 { float x, y, z, w; };
struct alignas(16) int4 { int x, y, z, w; };
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
struct alignas(16) ulonglong2 { unsigned long long x, y; };
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(unsigned x) { return __builtin_ffs(static_cast<int>(x)); }
inline unsigned __fns(unsigned m, unsigned from, int n) {
  for (unsigned i = from; i < 32; ++i)
    if ((m >> i & 1u) && --n == 0) return i;
  return 0xffffffffu;
}
template <class T> T __ldg(const T* p) { return *p; }
template <class T> T atomicCAS(T* p, T expect, T v) {
  __atomic_compare_exchange_n(p, &expect, v, false, __ATOMIC_SEQ_CST, __ATOMIC_SEQ_CST);
  return expect;
}
// additions to one watched word are counted
inline unsigned* g_watched = nullptr;
inline unsigned g_watched_adds = 0;
inline int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
inline unsigned atomicAdd(unsigned* p, unsigned v) {
  if (p == g_watched) __atomic_fetch_add(&g_watched_adds, 1u, __ATOMIC_SEQ_CST);
  return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST);
}
inline unsigned atomicOr(unsigned* p, unsigned v) { return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }
inline int atomicExch(int* p, int v) { return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST); }
inline void __threadfence() { __atomic_thread_fence(__ATOMIC_SEQ_CST); }
inline void __nanosleep(unsigned) { std::this_thread::yield(); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdiv_rn(float a, float b) { return a / b; }
inline unsigned g_reciprocals = 0;  // one a projection
inline float __frcp_rn(float a) {
  __atomic_fetch_add(&g_reciprocals, 1u, __ATOMIC_SEQ_CST);
  return 1.0f / a;
}
inline float __fsqrt_rn(float a) { return std::sqrt(a); }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
inline float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
inline int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
inline unsigned __float_as_uint(float f) { return static_cast<unsigned>(__float_as_int(f)); }
inline float __fadd_rd(float a, float b) {
  std::fesetround(FE_DOWNWARD);
  volatile float x = a, y = b;
  volatile float s = x + y;
  std::fesetround(FE_TONEAREST);
  return s;
}
using std::isfinite;
