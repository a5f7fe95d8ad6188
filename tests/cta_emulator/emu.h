// One CTA of a kernel on the host, a thread per CUDA thread: what the kernels use of ptx.cuh and of CUDA's builtins, with
// barriers that really wait, copies and MMAs that complete after a delay, and a record of what the exit path must not do.
// For the order of events only: loads, products and tensor memory carry no data (zeros).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#include <algorithm>
#include <atomic>
#include <barrier>
#include <chrono>
#include <condition_variable>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <set>
#include <string>
#include <thread>
#include <vector>
#undef __shared__
#define __shared__ static
#define __launch_bounds__(...)
#undef __grid_constant__
#define __grid_constant__

namespace emu {
using Clock = std::chrono::steady_clock;
using Ms = std::chrono::milliseconds;

// ---- what a test sets: when copies land (by call number; the others after 1 ms), how long an MMA takes, how long a
// suspended mbarrier.try_wait of a warp lasts, when the preceding kernel is done, when the cluster's copies arrive
inline std::map<int, int> load_ms;
inline int mma_us = 20, pdl_ms = 0, copy_ms = 1, load_parts = 1;
inline std::map<int, int> suspend_ms;

struct Dim { unsigned x = 1, y = 1, z = 1; };
inline Dim block_idx{0, 0, 0}, grid_dim, block_dim;
inline thread_local Dim thread_idx{0, 0, 0};

inline std::mutex mu;
inline std::condition_variable cv;
inline std::set<std::string> faults;
struct Bar { int count = 0, left = 0, phase = 0; long long tx = 0, armed = 0; };
inline std::map<const void*, Bar> bars;
struct Named { int arrived = 0, generation = 0; };
inline Named named[16];
struct Mma { const void* commit; };                       // an MMA, or (commit != null) a commit behind those before it
inline std::deque<Mma> pipe;
inline int loads_issued = 0, loads_flying = 0, copies_flying = 0, copies_due = 0, cluster_arrived = 0, cluster_generation = 0;
inline bool tmem_held = false, done = false;
inline std::multimap<Clock::time_point, std::pair<const void*, long long>> landing;   // (barrier, bytes)
inline const void* copies_bar = nullptr;

inline void advance(Bar& b) {                             // (with mu held)
  if (b.left == 0 && b.tx == 0) { b.phase ^= 1; b.left = b.count; }
}
inline void arrive(const void* bar) { Bar& b = bars[bar]; --b.left; advance(b); cv.notify_all(); }
inline void fault(const char* what) { faults.insert(what); }

// lands copies and retires MMAs, in order
inline void engine() {
  std::unique_lock<std::mutex> lk(mu);
  auto mma_at = Clock::now();
  while (!done) {
    const auto now = Clock::now();
    while (!landing.empty() && landing.begin()->first <= now) {
      const auto [bar, bytes] = landing.begin()->second;
      landing.erase(landing.begin());
      Bar& b = bars[bar];
      b.tx -= bytes;
      advance(b);
      if (bar == copies_bar) --copies_flying; else --loads_flying;
      if (bar != copies_bar && !tmem_held) fault("a load lands when TMEM has been given back");   // (what the block does by then)
      cv.notify_all();
    }
    while (!pipe.empty() && (pipe.front().commit || mma_at + std::chrono::microseconds(mma_us) <= now)) {
      if (pipe.front().commit) arrive(pipe.front().commit); else mma_at = now;
      pipe.pop_front();
    }
    if (pipe.empty()) mma_at = now;
    lk.unlock();
    std::this_thread::sleep_for(std::chrono::microseconds(10));
    lk.lock();
  }
}

struct Warp {
  std::barrier<> sync{32};
  unsigned long long slot[32];
};
inline std::vector<std::unique_ptr<Warp>> warps;
inline std::unique_ptr<std::barrier<>> block;
inline Warp& warp() { return *warps[thread_idx.x / 32]; }
inline int lane() { return thread_idx.x % 32; }
// every lane's value to every lane
template <class T, class F> auto exchange(T v, F f) {
  Warp& w = warp();
  unsigned long long raw = 0;
  memcpy(&raw, &v, sizeof(T));
  w.slot[lane()] = raw;
  w.sync.arrive_and_wait();
  T all[32];
  for (int i = 0; i < 32; ++i) memcpy(&all[i], &w.slot[i], sizeof(T));
  w.sync.arrive_and_wait();
  return f(all);
}

// runs `kernel` as one CTA of `threads`; what went wrong, one line each
template <class F> int run(int threads, F kernel) {
  block_dim.x = threads;
  block = std::make_unique<std::barrier<>>(threads);
  for (int i = 0; i < threads / 32; ++i) warps.push_back(std::make_unique<Warp>());
  std::thread eng(engine);
  std::vector<std::thread> all;
  for (int t = 0; t < threads; ++t) all.emplace_back([t, kernel] { thread_idx.x = t; kernel(); });
  for (auto& t : all) t.join();
  {
    std::lock_guard<std::mutex> lk(mu);
    if (loads_flying) fault("a load is in flight at the exit");
    if (copies_flying + copies_due) fault("a copy of the cluster is in flight at the exit");
    for (auto& m : pipe) fault(m.commit ? "a commit is in flight at the exit" : "an MMA is in flight at the exit");
    if (tmem_held) fault("TMEM is not given back");
    done = true;
  }
  eng.join();
  for (auto& f : faults) printf("FAULT %s\n", f.c_str());
  return faults.empty() ? 0 : 1;
}
inline void touch_tmem(const char* what) {
  std::lock_guard<std::mutex> lk(mu);
  if (!tmem_held) fault(what);
}
}  // namespace emu

#define threadIdx emu::thread_idx
#define blockIdx emu::block_idx
#define blockDim emu::block_dim
#define gridDim emu::grid_dim
#define clock64() static_cast<long long>(emu::Clock::now().time_since_epoch().count())

template <class A, class B> auto min(A a, B b) { return a < b ? a : b; }
template <class A, class B> auto max(A a, B b) { return a < b ? b : a; }
inline unsigned __float_as_uint(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
inline float __uint_as_float(unsigned u) { float f; memcpy(&f, &u, 4); return f; }
inline void __syncthreads() { emu::block->arrive_and_wait(); }
inline int __syncthreads_and(int v) {
  static std::atomic<int> bad{0};
  if (!v) bad = 1;
  __syncthreads();
  const int r = !bad;
  __syncthreads();
  bad = 0;
  __syncthreads();
  return r;
}
inline void __syncwarp() { emu::warp().sync.arrive_and_wait(); }
inline int __all_sync(unsigned, int v) { return emu::exchange(v, [](int* a) { int r = 1; for (int i = 0; i < 32; ++i) r &= a[i] != 0; return r; }); }
inline int __any_sync(unsigned, int v) { return emu::exchange(v, [](int* a) { int r = 0; for (int i = 0; i < 32; ++i) r |= a[i] != 0; return r; }); }
inline unsigned __ballot_sync(unsigned, int v) { return emu::exchange(v, [](int* a) { unsigned r = 0; for (int i = 0; i < 32; ++i) r |= (a[i] != 0 ? 1u : 0u) << i; return r; }); }
template <class T> T __shfl_xor_sync(unsigned, T v, int o) { return emu::exchange(v, [o](T* a) { return a[emu::lane() ^ o]; }); }
template <class T> T __shfl_up_sync(unsigned, T v, int o) { return emu::exchange(v, [o](T* a) { const int l = emu::lane(); return l >= o ? a[l - o] : a[l]; }); }
template <class T> T __reduce_add_sync(unsigned, T v) { return emu::exchange(v, [](T* a) { T r = 0; for (int i = 0; i < 32; ++i) r += a[i]; return r; }); }
template <class T> T __reduce_min_sync(unsigned, T v) { return emu::exchange(v, [](T* a) { T r = a[0]; for (int i = 0; i < 32; ++i) r = min(r, a[i]); return r; }); }
inline unsigned __reduce_and_sync(unsigned, unsigned v) { return emu::exchange(v, [](unsigned* a) { unsigned r = ~0u; for (int i = 0; i < 32; ++i) r &= a[i]; return r; }); }
inline unsigned __reduce_or_sync(unsigned, unsigned v) { return emu::exchange(v, [](unsigned* a) { unsigned r = 0; for (int i = 0; i < 32; ++i) r |= a[i]; return r; }); }
template <class T> T atomicExch(T* p, T v) { return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST); }
inline int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
inline unsigned long long atomicMax(unsigned long long* p, unsigned long long v) {
  std::lock_guard<std::mutex> lk(emu::mu);
  const auto old = *p;
  if (v > old) *p = v;
  return old;
}
inline unsigned long long atomicMin(unsigned long long* p, unsigned long long v) {
  std::lock_guard<std::mutex> lk(emu::mu);
  const auto old = *p;
  if (v < old) *p = v;
  return old;
}
template <class T> T __ldcg(const T* p) { return *p; }
inline int __clzll(long long v) { return v ? __builtin_clzll(v) : 64; }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __popc(unsigned v) { return __builtin_popcount(v); }

// ---- ptx.cuh
namespace kvc {
inline uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p)); }
inline void mbar_init(uint64_t* bar, uint32_t n) {
  std::lock_guard<std::mutex> lk(emu::mu);
  emu::bars[bar] = emu::Bar{static_cast<int>(n), static_cast<int>(n), 0, 0, 0};
}
inline void mbar_fence_init() {}
inline void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  std::lock_guard<std::mutex> lk(emu::mu);
  emu::bars[bar].tx += bytes;
  emu::bars[bar].armed = bytes;
  if (emu::copies_due && !emu::copies_bar) emu::copies_bar = bar;      // (a key split arms it first, for its peers' copies)
  emu::arrive(bar);
}
inline void mbar_arrive(uint64_t* bar) { std::lock_guard<std::mutex> lk(emu::mu); emu::arrive(bar); }
inline bool emu_wait(uint64_t* bar, uint32_t parity, int ms) {
  std::unique_lock<std::mutex> lk(emu::mu);
  return emu::cv.wait_for(lk, emu::Ms(ms), [&] { return emu::bars[bar].phase != static_cast<int>(parity); });
}
inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {          // suspends the thread for a while
  const auto it = emu::suspend_ms.find(threadIdx.x / 32);
  return emu_wait(bar, parity, it == emu::suspend_ms.end() ? 2 : it->second);
}
inline bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  std::this_thread::yield();
  return emu_wait(bar, parity, 0);
}
inline void fence_proxy_async_smem() {}
inline void tc_fence_before_sync() {}
inline void tc_fence_after_sync() {}
inline void tma_prefetch_desc(const void*) {}
inline void tma_load_4d(void*, const void*, uint64_t* bar, int, int, int, int) {
  std::lock_guard<std::mutex> lk(emu::mu);
  const auto it = emu::load_ms.find(emu::loads_issued++);
  ++emu::loads_flying;
  emu::landing.insert({emu::Clock::now() + emu::Ms(it == emu::load_ms.end() ? 1 : it->second), {bar, emu::bars[bar].armed / emu::load_parts}});
}
inline void tma_prefetch_l2_4d(const void*, int, int, int, int) {}
inline void tma_store_4d(const void*, const void*, int, int, int, int) {}
inline void tma_store_commit() {}
inline void tma_store_wait_read() {}
inline void tma_store_wait_all() {}
inline void tmem_alloc(uint32_t* result, uint32_t) {
  std::lock_guard<std::mutex> lk(emu::mu);
  *result = 0;
  emu::tmem_held = true;
}
inline void tmem_relinquish() {}
inline void tmem_dealloc(uint32_t, uint32_t) {
  __syncwarp();
  if (emu::lane() == 0) {
    std::lock_guard<std::mutex> lk(emu::mu);
    for (auto& m : emu::pipe)
      if (!m.commit) emu::fault("TMEM is given back under an MMA");
    emu::tmem_held = false;
  }
  __syncwarp();
}
inline uint64_t smem_desc_sw128(uint32_t, uint32_t, uint32_t) { return 0; }
inline uint32_t smem_desc_lo(uint32_t, uint32_t) { return 0; }
constexpr uint32_t smem_desc_hi_sw128(uint32_t) { return 0; }
constexpr uint32_t idesc_bf16_f32(int, int, int, int) { return 0; }
inline void emu_mma() {
  std::lock_guard<std::mutex> lk(emu::mu);
  if (!emu::tmem_held) emu::fault("an MMA is issued after TMEM was given back");
  emu::pipe.push_back({nullptr});
}
inline void mma_ss(uint32_t, uint64_t, uint64_t, uint32_t, uint32_t) { emu_mma(); }
inline void mma_ss_lh(uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t) { emu_mma(); }
inline void mma_ts_lh(uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t) { emu_mma(); }
inline void mma_commit(uint64_t* bar) { std::lock_guard<std::mutex> lk(emu::mu); emu::pipe.push_back({bar}); }
template <int N> void emu_ld(uint32_t* r) { emu::touch_tmem("TMEM is read after it was given back"); memset(r, 0, N * 4); }
inline void tmem_ld16(uint32_t, uint32_t* r) { emu_ld<16>(r); }
inline void tmem_ld32(uint32_t, uint32_t* r) { emu_ld<32>(r); }
inline void tmem_ld2(uint32_t, uint32_t& a, uint32_t& b) { a = b = 0; emu::touch_tmem("TMEM is read after it was given back"); }
inline void tmem_st16(uint32_t, const uint32_t*) { emu::touch_tmem("TMEM is written after it was given back"); }
inline void tmem_st32(uint32_t, const uint32_t*) { emu::touch_tmem("TMEM is written after it was given back"); }
inline void tmem_st2(uint32_t, uint32_t, uint32_t) { emu::touch_tmem("TMEM is written after it was given back"); }
inline void tmem_wait_ld() {}
inline void tmem_wait_st() {}
// the CTA is rank 0 of its cluster; its peers are on time, and their copies arrive copy_ms after the first cluster barrier
inline uint32_t cluster_ctarank() { return 0; }
inline void cluster_arrive() {
  std::lock_guard<std::mutex> lk(emu::mu);
  if (++emu::cluster_arrived < static_cast<int>(blockDim.x)) return;
  emu::cluster_arrived = 0;
  if (emu::cluster_generation++ == 0 && emu::copies_bar) {
    emu::landing.insert({emu::Clock::now() + emu::Ms(emu::copy_ms), {emu::copies_bar, emu::bars[emu::copies_bar].armed}});
    ++emu::copies_flying;
    emu::copies_due = 0;
  }
  emu::cv.notify_all();
}
inline void cluster_arrive_relaxed() { cluster_arrive(); }
inline thread_local int emu_cluster_waits = 0;
inline void cluster_wait() {
  std::unique_lock<std::mutex> lk(emu::mu);
  const int want = ++emu_cluster_waits;
  emu::cv.wait(lk, [&] { return emu::cluster_generation >= want; });
}
inline uint32_t dsmem_addr(uint32_t a, uint32_t) { return a; }
inline void bulk_copy_to_cluster(uint32_t, uint32_t, uint32_t, uint32_t) {}
inline float dsmem_ld_f32(uint32_t) { return 0.f; }
template <int N> void reg_inc() {}
template <int N> void reg_dec() {}
inline void emu_named(int id, int count, bool wait) {
  std::unique_lock<std::mutex> lk(emu::mu);
  emu::Named& n = emu::named[id];
  const int generation = n.generation;
  if (++n.arrived == count) { n.arrived = 0; ++n.generation; emu::cv.notify_all(); }
  else if (wait) emu::cv.wait(lk, [&] { return n.generation != generation; });
}
inline void named_barrier(int id, int count) { emu_named(id, count, true); }
inline void named_barrier_arrive(int id, int count) { emu_named(id, count, false); }
inline void pdl_wait() { std::this_thread::sleep_for(emu::Ms(emu::pdl_ms)); }
inline void pdl_launch_dependents() {}
inline float fast_exp2(float x) { return exp2f(x); }
inline float fmax3(float a, float b, float c) { return fmaxf(a, fmaxf(b, c)); }
inline uint64_t f32x2(float a, float b) { return static_cast<uint64_t>(__float_as_uint(b)) << 32 | __float_as_uint(a); }
inline void f32x2_split(uint64_t v, float& a, float& b) { a = __uint_as_float(static_cast<uint32_t>(v)); b = __uint_as_float(v >> 32); }
inline uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  float x[3], y[3];
  f32x2_split(a, x[0], y[0]); f32x2_split(b, x[1], y[1]); f32x2_split(c, x[2], y[2]);
  return f32x2(fmaf(x[0], x[1], x[2]), fmaf(y[0], y[1], y[2]));
}
inline uint64_t add_f32x2(uint64_t a, uint64_t b) {
  float x[2], y[2];
  f32x2_split(a, x[0], y[0]); f32x2_split(b, x[1], y[1]);
  return f32x2(x[0] + x[1], y[0] + y[1]);
}
inline void st_global_v8(void* p, const uint32_t* r) { memcpy(p, r, 32); }
inline uint32_t pack_bf16x2(float a, float b) { return __float_as_uint(a) >> 16 | (__float_as_uint(b) & 0xffff0000u); }
}  // namespace kvc
