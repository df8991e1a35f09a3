// Harness of the one-launch step's warps when a launch gives up (test
// infrastructure, built by tests/test_stash_warps.py).  The device code of the
// workers, the drawer and the closer, cut from lamb_stash.cu as it stands, runs
// on the host with a thread for each lane: votes, shuffles and __syncwarp are
// meetings of 32 threads.  Each scenario lets one half of a warp see that the
// launch gives up at a moment when the other half does not; a lane that leaves
// while others wait in a warp-wide operation is the fault that is looked for (on
// the GPU the others would wait for ever).  Argument: the scenario.  Exit status
// 0: the lanes left together.
#include <cuda_runtime_api.h>
#include <vector_functions.h>

#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "lamb_stash.h"

#undef __device__
#undef __forceinline__
#define __device__
#define __forceinline__ inline

// ---- a warp of threads ------------------------------------------------------
struct Left {};   // thrown in a lane whose meeting can no longer happen

struct Warp {
  std::mutex m;
  std::condition_variable cv;
  int count = 0, kind = 0;
  uint64_t turn = 0, value[2][32];
  uint32_t gone = 0;
  bool fault = false;

  const uint64_t* meet(int what, int lane, uint64_t v) {
    std::unique_lock<std::mutex> lock(m);
    const uint64_t now = turn;
    if (count == 0) kind = what;
    if (gone || what != kind) fault = true;
    value[now & 1][lane] = v;
    if (!fault && ++count == 32) {
      count = 0;
      ++turn;
      cv.notify_all();
      return value[now & 1];
    }
    while (turn == now && !fault && !gone) cv.wait(lock);
    if (turn == now) {
      fault = true;
      cv.notify_all();
      throw Left{};
    }
    return value[now & 1];
  }
  void leave(int lane) {
    std::lock_guard<std::mutex> lock(m);
    gone |= 1u << lane;
    cv.notify_all();
  }
  bool upper_gone() {
    std::lock_guard<std::mutex> lock(m);
    return gone >> 16 == 0xffffu;
  }
};

static Warp g_warp;
static thread_local struct { unsigned x; } threadIdx;
static struct { unsigned x; } gridDim = {1}, blockIdx = {0};
static int lane_id() { return (int)(threadIdx.x & 31u); }
static bool upper() { return lane_id() >= 16; }

// what a scenario replaces
static std::function<bool(uint64_t*)> g_passed = [](uint64_t*) { return true; };
static std::function<void()> g_sleep = [] {};
static std::function<void()> g_voted = [] {};
static std::function<uint32_t()> g_counter = [] { return 0u; };
static thread_local bool t_stores = false;   // tensor memory stores not waited for

template <typename T> static uint64_t bits_of(T x) {
  uint64_t v = 0;
  std::memcpy(&v, &x, sizeof x);
  return v;
}
template <typename T> static T of_bits(uint64_t v) {
  T x;
  std::memcpy(&x, &v, sizeof x);
  return x;
}
static void __syncwarp(unsigned = 0xffffffffu) {
  g_warp.meet(1, lane_id(), 0);
}
static bool __all_sync(unsigned, bool p) {
  const uint64_t* v = g_warp.meet(2, lane_id(), p);
  bool r = true;
  for (int i = 0; i < 32; ++i) r = r && v[i];
  if (!r) g_voted();
  return r;
}
static bool __any_sync(unsigned, bool p) {
  const uint64_t* v = g_warp.meet(3, lane_id(), p);
  bool r = false;
  for (int i = 0; i < 32; ++i) r = r || v[i];
  return r;
}
template <typename T> static T __shfl_sync(unsigned, T x, int from) {
  return of_bits<T>(g_warp.meet(4, lane_id(), bits_of(x))[from & 31]);
}
template <typename T> static T __shfl_xor_sync(unsigned m, T x, int o) {
  (void)m;
  return of_bits<T>(g_warp.meet(5, lane_id(), bits_of(x))[lane_id() ^ o]);
}
template <typename T> static T __shfl_down_sync(unsigned, T x, int o) {
  const int from = lane_id() + o;
  return of_bits<T>(
      g_warp.meet(6, lane_id(), bits_of(x))[from < 32 ? from : lane_id()]);
}

// ---- what the cut code calls ------------------------------------------------
struct __nv_bfloat16 { unsigned short x; };
using std::isfinite;
using std::isnan;
template <typename T> static T min(T a, T b) { return a < b ? a : b; }
template <typename T> static T max(T a, T b) { return a > b ? a : b; }
static void __nanosleep(unsigned) {
  std::this_thread::sleep_for(std::chrono::microseconds(50));
  g_sleep();
}
template <typename T> static T __ldcg(const T* p) { return *p; }
template <typename T> static T __ldcs(const T* p) { return *p; }
static uint32_t atomicAdd(uint32_t* p, uint32_t v) {
  return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST);
}
static uint32_t atomicOr(uint32_t* p, uint32_t v) {
  return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST);
}
static uint32_t atomicExch(uint32_t* p, uint32_t v) {
  return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST);
}
static void __threadfence() {}
static float __uint_as_float(uint32_t x) { return of_bits<float>(x); }
static uint32_t __float_as_uint(float x) { return (uint32_t)bits_of(x); }
static float __double2float_rn(double x) { return (float)x; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }

namespace lamb {
namespace {

struct LambConsts {
  float b1, omb1, b2, omb2, c1, c2, eps, am, ag, bv, bg;
};
void lamb_moments(float, float&, float&, const LambConsts&) {}
float lars_momentum(float, float m, float, float, float, float) { return m; }
float lamb_direction(float m, float, float, float, const LambConsts&) {
  return m;
}
template <int kNest>
float nlamb_direction(float m, float, float, float, float, const LambConsts&) {
  return m;
}
void st4(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
void st4_last(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
void st_copy4(void*, int64_t, float4) {}
void st_copy1(void*, int64_t, float) {}
float warp_sum(float x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}
double phi_of(double z, const StepParams&) { return z; }

uint32_t ld_relaxed_u32(const uint32_t*) { return g_counter(); }
uint32_t ld_acquire_u32(const uint32_t* p) { return *p; }
uint64_t ld_relaxed_u64(const uint64_t* p) { return *p; }
void st_relaxed_u64(uint64_t* p, uint64_t v) { *p = v; }
uint32_t atom_add_acq_rel(uint32_t* p, uint32_t v) { return atomicAdd(p, v); }
uint64_t global_ns() { return 0; }
bool mbar_test(uint64_t* b, uint32_t) { return g_passed(b); }
bool mbar_try(uint64_t* b, uint32_t) { return g_passed(b); }
void mbar_arrive(uint64_t*) {}
void mbar_expect(uint64_t*, uint32_t) {}
void bulk_load(void*, const void*, uint32_t, uint64_t*) {}
void fence_proxy_async() {}
void tmem_st4(uint32_t, const float4&) { t_stores = true; }
void tmem_wait_st() { t_stores = false; }
void tmem_ld4x4(const uint32_t (&)[4], float4 (&)[4]) {}

}  // namespace
}  // namespace lamb

#include "stash_cut.inc"

using namespace lamb;

namespace {

Shared g_sh;
int g_pending = 0;   // lanes that left with stores to tensor memory in flight
std::mutex g_mutex;

void run_warp(int first_thread, const std::function<void()>& body) {
  std::vector<std::thread> lanes;
  for (int i = 0; i < 32; ++i)
    lanes.emplace_back([&, i] {
      threadIdx.x = (unsigned)(first_thread + i);
      try {
        body();
      } catch (const Left&) {
      }
      if (t_stores) {
        std::lock_guard<std::mutex> lock(g_mutex);
        ++g_pending;
      }
      g_warp.leave(i);
    });
  for (auto& t : lanes) t.join();
}

void pause_until(const std::function<bool()>& done) {
  for (int i = 0; i < 400 && !done(); ++i)
    std::this_thread::sleep_for(std::chrono::microseconds(500));
}
volatile int* abort_flag() { return &g_sh.abort; }

}  // namespace

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  StepParams p = {};
  StashParams q = {};
  std::vector<StashRec> recs(64);
  std::vector<uint32_t> bar(kStashBarWords, 0u);
  std::vector<float> arrays(4 * 8192, 0.f);
  for (int i = 0; i < 64; ++i) {   // kept chunks of four tiles, a tensor each
    recs[(size_t)i] = StashRec{};
    recs[(size_t)i].len_bits = 4096u | kStashVec | (kStashKeep << 30);
    recs[(size_t)i].tensor = i;
    recs[(size_t)i].chunk = i;
    recs[(size_t)i].n_chunks = 1;
    recs[(size_t)i].keep_end = i + 1;
    recs[(size_t)i].w = arrays.data();
    recs[(size_t)i].m = arrays.data() + 8192;
    recs[(size_t)i].v = arrays.data() + 2 * 8192;
    recs[(size_t)i].g = arrays.data() + 3 * 8192;
  }
  q.recs = recs.data();
  q.bar = bar.data();
  q.n_items = 64;
  q.slots = 23;
  q.wslots = 0;
  q.max_keep = 4;
  std::memset(&g_sh, 0, sizeof g_sh);
  g_sh.issued = 1 << 30;
  g_sh.end_seq = g_sh.end_kept = 0x7fffffff;

  // one barrier whose phase the lower lanes see complete and the others not
  auto split = [&](uint64_t* b) {
    *abort_flag() = 1;
    g_passed = [b](uint64_t* x) { return x != b || !upper(); };
  };
  auto drawer = [&] { draw(p, q, g_sh); };
  auto closer = [&] { close_chunks(p, q, g_sh, 1.0); };
  std::vector<char> smem((size_t)(kStages * kStageBytes<float>), 0);
  auto worker = [&] {
    Worker<0, float, false> w(p, q, g_sh, smem.data(), 0u);
    w.run();
  };

  if (what == "drawer_record") {
    split(&g_sh.free[0]);
    run_warp(0, drawer);
  } else if (what == "drawer_kept_record") {
    split(&g_sh.kfree[0]);
    run_warp(0, drawer);
  } else if (what == "drawer_issued") {
    // the loader's count arrives as the launch gives up
    g_sh.issued = -1;
    g_sleep = [] {
      if (upper()) {
        *abort_flag() = 1;
      } else {
        pause_until([] { return g_warp.upper_gone(); });
        *reinterpret_cast<volatile int*>(&g_sh.issued) = 1 << 30;
      }
    };
    run_warp(0, drawer);
  } else if (what == "drawer_kept_tensor") {
    q.max_keep = 1;
    *abort_flag() = 1;
    g_counter = [] { return upper() ? 0u : 1u << 20; };
    run_warp(0, drawer);
  } else if (what == "closer_record") {
    split(&g_sh.full[0]);
    run_warp(0, closer);
  } else if (what == "closer_done") {
    split(&g_sh.done[0]);
    run_warp(0, closer);
  } else if (what == "worker_wait") {
    // the flag is set between two lanes' looks at it
    g_passed = [](uint64_t*) { return false; };
    g_sleep = [] { *abort_flag() = 1; };
    g_voted = [] {
      if (!upper()) return;
      pause_until([] { return *abort_flag() != 0; });
      *abort_flag() = 1;
    };
    run_warp(0, worker);
  } else if (what == "worker_stores") {
    // one chunk is kept, then the launch gives up
    static_cast<StashRec&>(g_sh.rec[0]) = recs[0];
    g_sh.rec[0].len = 4096;
    g_sh.rec[0].kind = kStashKeep;
    g_sh.rec[0].vec = kStashVec;
    g_sh.rec[0].tiles = 4;
    *abort_flag() = 1;
    g_passed = [](uint64_t* b) {
      return b == &g_sh.full[0] || (b >= g_sh.sfull && b < g_sh.sfull + kStages);
    };
    run_warp(0, worker);
  } else {
    std::fprintf(stderr, "unknown scenario\n");
    return 2;
  }
  if (g_warp.fault) {
    std::fprintf(stderr, "lanes left while others of the warp waited\n");
    return 1;
  }
  if (g_pending) {
    std::fprintf(stderr, "%d lanes left with tensor memory stores in flight\n",
                 g_pending);
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
