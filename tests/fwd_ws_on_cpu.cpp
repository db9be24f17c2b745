// The roles of the tensor-core forward kernel on CPU threads, one per warp: barriers, copies and products stand for themselves only
// (no numbers are computed).  A copy arrives late, past the limit of the waits; the CTA must then come to its end on every
// warp, with no copy and no product in flight.  // Built by tests/test_forward_roles_cpu.py, which puts the kernel's own
// text into fwd_ws_kernel.inc.
#include <bit>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#include "litevar_internal.h"

using std::max;
using std::min;
using Clock = std::chrono::steady_clock;
using CUtensorMap = int;

constexpr std::chrono::milliseconds kWait{60}, kLate{180}, kHang{10000};

struct Hang {};
struct Cta {
  std::mutex mutex;
  std::condition_variable changed;
  struct Bar {
    int expected, pending, phase = 0;
    long tx = 0;
  };
  std::map<void*, Bar> bars;           // mbarriers
  std::map<int, std::pair<int, int>> named;  // threads arrived, phases
  std::vector<std::pair<void*, Clock::time_point>> products;  // commits
  struct Copy {
    void* bar;
    long bytes;
    Clock::time_point due;
  };
  std::vector<Copy> copies;  // in flight
  int copies_seen = 0, late = -1, status = 0;
  bool second_pass = false, hung = false, done = false;
  uint8_t* smem = nullptr;

  void settle(Bar& b) {
    if (b.pending == 0 && b.tx == 0) {
      ++b.phase;
      b.pending = b.expected;
      changed.notify_all();
    }
  }
  void engine() {  // completes copies and products
    std::unique_lock<std::mutex> lock(mutex);
    while (!done) {
      const auto now = Clock::now();
      for (size_t i = 0; i < copies.size();)
        if (copies[i].due <= now) {
          Bar& b = bars[copies[i].bar];
          b.tx -= copies[i].bytes;
          settle(b);
          copies.erase(copies.begin() + i);
        } else {
          ++i;
        }
      while (!products.empty() && products.front().second <= now) {
        Bar& b = bars[products.front().first];
        --b.pending;
        settle(b);
        products.erase(products.begin());
      }
      changed.wait_for(lock, std::chrono::microseconds(100));
    }
  }
};
thread_local Cta* cta;
thread_local struct { unsigned x; } threadIdx;
const struct { unsigned x; } blockIdx{0}, gridDim{1};

namespace litevar {
constexpr uint32_t kTileBytes = kBlockN * kHeadDim * 2;
constexpr unsigned long long kWaitLimitNs = 500000000ull;
struct TensorMaps {
  CUtensorMap o, q, kr, vr, k2[kMaxPatchScales], v2[kMaxPatchScales];
};
struct ChunkAt {
  int row, col, map, h, b;
};
inline uint32_t smem_u32(const void* p) { return (uint32_t)(uintptr_t)p; }
inline uint64_t make_desc(uint32_t a) { return a; }
inline unsigned long long global_ns() { return Clock::now().time_since_epoch() / std::chrono::nanoseconds(1); }
inline void mbar_init(uint64_t* bar, int n) {
  std::lock_guard<std::mutex> lock(cta->mutex);
  cta->bars[bar] = Cta::Bar{n, n};
}
inline void mbar_arrive(uint64_t* bar, int n = 1, long bytes = 0) {
  std::lock_guard<std::mutex> lock(cta->mutex);
  Cta::Bar& b = cta->bars[bar];
  b.tx += bytes;
  b.pending -= n;
  cta->settle(b);
}
inline void mbar_expect_tx(uint64_t* bar, long bytes) { mbar_arrive(bar, 1, bytes); }
inline bool mbar_try(uint64_t* bar, uint32_t parity) {
  std::lock_guard<std::mutex> lock(cta->mutex);
  return ((cta->bars[bar].phase ^ 1) & 1) == (int)parity;
}
inline bool mbar_wait_long(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  const auto t0 = Clock::now();
  while (!mbar_try(bar, parity)) {
    if (*abort_flag) return false;
    if (cta->late >= 0 && Clock::now() - t0 > kWait) {
      *abort_flag = 1;
      *status = 1;
      return false;
    }
    std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
  return true;
}
inline bool mbar_wait_idle(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  return mbar_wait_long(bar, parity, abort_flag, status);
}
inline void copy(uint64_t* bar, long bytes) {
  std::lock_guard<std::mutex> lock(cta->mutex);
  const bool late = cta->copies_seen++ == cta->late;
  cta->copies.push_back({bar, bytes, Clock::now() + (late ? kLate : std::chrono::milliseconds(0))});
}
inline void tma_load_4d(void*, const CUtensorMap*, int, int, int, int, uint64_t* bar) { copy(bar, kHeadDim * 64); }
inline void load_chunk(void*, const CUtensorMap*, const CUtensorMap*, const ChunkAt&, uint64_t* bar) {
  mbar_expect_tx(bar, 1);
  copy(bar, 1);
}
inline void load_q_tile(void*, const TensorMaps&, const FwdParams&, int, int, int, uint64_t* bar) { copy(bar, kTileBytes); }
template <class T>
void load_scales(T&, const float*, const float*, int, int, int, uint64_t* bar) { mbar_arrive(bar, 32); }
inline void wait_met(const int* at, int n) {
  while (*(volatile const int*)at < n) std::this_thread::yield();
}
inline void mma_commit_one(uint64_t* bar) {
  std::lock_guard<std::mutex> lock(cta->mutex);
  cta->products.push_back({bar, Clock::now() + std::chrono::milliseconds(cta->late < 0 ? 0 : 2)});
}
inline void bar_meet(int id, int n, bool wait) {
  std::unique_lock<std::mutex> lock(cta->mutex);
  auto& b = cta->named[id];
  const int phase = b.second;
  if ((b.first += 32) == n) {
    b = {0, phase + 1};
    cta->changed.notify_all();
  } else if (wait && !cta->changed.wait_for(lock, kHang, [&] { return b.second != phase; })) {
    cta->hung = true;
    throw Hang();
  }
}
inline void bar_sync(int id, int n) { bar_meet(id, n, true); }
inline void bar_arrive(int id, int n) { bar_meet(id, n, false); }
inline void __syncthreads() { bar_sync(0, 320); }
inline void __syncwarp() {}
inline void __nanosleep(unsigned ns) { std::this_thread::sleep_for(std::chrono::nanoseconds(ns)); }
template <class T>
T __shfl_sync(unsigned, T v, int) { return v; }
inline bool __any_sync(unsigned, bool v) { return v; }
template <class T>
T __ldg(const T* p) { return *p; }
inline float __uint_as_float(uint32_t v) { return std::bit_cast<float>(v); }
inline float __saturatef(float x) { return x; }
inline float2 __ffma2_rn(float2 a, float2, float2) { return a; }
inline float2 __fmul2_rn(float2 a, float2) { return a; }
inline float largest_score(const uint32_t*) { return 0.f; }
inline float2 exp2_fma2(float2 x) { return x; }
inline float fast_exp2(float x) { return x; }
inline uint32_t pack_bf16(float, float) { return 0; }
template <bool, bool>
constexpr bool on_fma_pipe(int) { return false; }
inline bool elect_one() { return true; }
inline KeyChunk chunk_at(const KeyChunk* c) { return *c; }
inline void tc_fence_before() {}
inline void tc_fence_after() {}
inline void tmem_wait_ld() {}
inline void tmem_wait_st() {}
inline void tmem_ld32(uint32_t, uint32_t* r) { memset(r, 0, 128); }
inline void tmem_ld8(uint32_t, uint32_t* r) { memset(r, 0, 32); }
inline void tmem_ld4(uint32_t, uint32_t* r) {  // the row sums: 4 or, for the second pass, 0
  for (int i = 0; i < 4; ++i) r[i] = cta->second_pass ? 0u : 0x3f800000u;
}
inline void tmem_ld1(uint32_t, uint32_t& r) { r = cta->second_pass ? 0u : 0x3f800000u; }
inline void tmem_st16(uint32_t, const uint32_t*) {}
inline void q_to_tmem(uint32_t, uint64_t) {}
template <int, int>
void mma_ts_x4_one(uint32_t, uint32_t, uint64_t, uint32_t, uint32_t) {}
template <class T>
void widen_chunk(const uint8_t*, T&, uint8_t*, int) {}
inline void tma_store_4d(const CUtensorMap*, const void*, int, int, int, int) {}
inline void tma_store_5d(const CUtensorMap*, const void*, int, int, int, int, int) {}
inline void work_item(const FwdParams&, int, int item, int& rank, int& unit) { rank = item, unit = 0; }
constexpr uint32_t kIdescS = 0, kIdescO = 0;
constexpr float kClampHigh = 100.f, kClampSpan = 225.f;
#include "fwd_ws_kernel.inc"
}  // namespace litevar

// One CTA over lists of `chunks` chunks each; copy number `late` arrives late (-1: none).  Returns the copies it saw, or -1.
template <bool KV8, bool MANY>
int run(const std::vector<int>& chunks, bool second_pass, int late) {
  using namespace litevar;
  Cta c;
  c.late = late;
  c.second_pass = second_pass;
  c.smem = static_cast<uint8_t*>(aligned_alloc(1024, 1 << 18));
  memset(c.smem, 0, 1 << 18);
  std::vector<int32_t> ptr(1, 0);
  for (int n : chunks) ptr.push_back(ptr.back() + n);
  std::vector<KeyChunk> list(ptr.back() + 1, KeyChunk{0, 0, 0xaaaa, -1});
  FwdParams p;
  memset(&p, 0, sizeof p);
  p.set0.chunk_ptr = ptr.data();
  p.set0.chunks = list.data();
  p.n_heads = 1;
  p.n_k = 128 * (int)chunks.size();
  p.sm_scale = 0.125f;
  p.status = &c.status;
  const TensorMaps tm{};
  std::thread engine([&] { c.engine(); });
  std::vector<std::thread> warps;
  for (int w = 0; w < 10; ++w)
    warps.emplace_back([&, w] {
      cta = &c;
      threadIdx.x = 32 * w;
      try {
        fwd_ws_kernel<KV8, MANY>(tm, p, (int)chunks.size(), (int)chunks.size());
      } catch (const Hang&) {
      }
    });
  for (auto& w : warps) w.join();
  int in_flight;
  {
    std::lock_guard<std::mutex> lock(c.mutex);
    in_flight = (int)(c.copies.size() + c.products.size());
    c.done = true;
  }
  engine.join();
  free(c.smem);
  const bool bad = c.hung || in_flight || c.status != (late >= 0);
  if (bad) {
    printf("KV8 %d MANY %d second pass %d copy %d late, lists", KV8, MANY, second_pass, late);
    for (int n : chunks) printf(" %d", n);
    printf(": %s%d copies or products in flight, status %d\n", c.hung ? "hangs, " : "", in_flight, c.status);
  }
  return bad ? -1 : c.copies_seen;
}

template <bool KV8, bool MANY>
int all(const std::vector<std::vector<int>>& cases, bool second_pass) {
  int failed = 0;
  for (const auto& lists : cases) {
    const int n = run<KV8, MANY>(lists, second_pass, -1);
    if (n < 0) return 1;
    std::vector<std::thread> runs;
    std::vector<int> result(n);
    for (int late = 0; late < n; ++late) {
      runs.emplace_back([&, late] { result[late] = run<KV8, MANY>(lists, second_pass, late); });
      if (runs.size() == 8 || late + 1 == n) {
        for (auto& r : runs) r.join();
        runs.clear();
      }
    }
    for (int r : result) failed += r < 0;
  }
  return failed;
}

int main(int argc, char** argv) {
  const std::string build = argc > 1 ? argv[1] : "";
  const bool second_pass = argc > 2;
  int failed = 1;
  if (build == "one-tile") failed = all<false, false>({{1}, {2}, {5}, {12}}, second_pass);
  if (build == "8-bit") failed = all<true, false>({{1}, {2}, {5}, {12}}, second_pass);
  if (build == "many-tiles") failed = all<false, true>({{4, 4, 4}, {1, 2, 3, 7}}, second_pass);
  return failed != 0;
}
