// Harness of the C entry points' host code (test infrastructure, built by
// tests/test_capi_routes.py): lamb_capi.cu and planner.cpp as they stand, on a
// stand-in for the CUDA runtime whose device memory is host memory, with
// launchers that only write down that they were called.  So what a step launches
// can be seen for any layout, and a launch can be refused.  Prints one line per
// step: the launches, in order.
//   capi_routes <algorithm> <opt> <flags> <sizes> [<option>=<value> ...]
// sizes: n or nxm (m tensors of n elements), separated by commas.  Options:
// those of lamb_plan_options_t by name, and refuse=<cudaError_t> (what the
// one-launch kernel's launch returns).
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "lamb.h"
#include "lamb_internal.h"
#include "lamb_onchip.h"
#include "lamb_stash.h"

namespace {
std::vector<std::string> g_launches;
int g_refuse = 0, g_last_error = 0, g_events = 0;
int64_t g_plan_chunks = 0;   // the plan's own chunk table
int g_wrong_table = 0;

int seen(const std::string& name) {
  g_launches.push_back(name);
  return 0;
}
// a two-pass launch works on the plan's own chunks, not on the one launch's
int two_pass(const std::string& name, const lamb::StepParams& p) {
  if (p.n_chunks != g_plan_chunks) g_wrong_table = 1;
  return seen(name + ((p.flags & (LAMB_FLAG_GRAD_NORM |
                                  LAMB_FLAG_SKIP_NONFINITE)) ? "+gn" : ""));
}
bool seen_any(const char* prefix) {
  for (const std::string& x : g_launches)
    if (x.rfind(prefix, 0) == 0) return true;
  return false;
}
const char* kNames[4] = {"lamb", "nlamb", "nnlamb", "lars"};
}  // namespace

namespace lamb {
int launch_lamb_pass1(const StepParams& p, int nest, int, int, void*) {
  return two_pass(std::string(kNames[nest]) + "1", p);
}
int launch_lamb_pass2(const StepParams& p, int nest, int, int, int, void*) {
  return two_pass(std::string(kNames[nest]) + "2", p);
}
int launch_lars_pass1(const StepParams& p, int, int, void*) {
  return two_pass("lars1", p);
}
int launch_lars_pass2(const StepParams& p, int, int, int, void*) {
  return two_pass("lars2", p);
}
int launch_finalize_all(const StepParams&, double, void*) {
  return seen("finalize");
}
int launch_onchip(const StepParams&, const OcParams&, int opt, int, int, int,
                  int, void*) {
  return seen(std::string("onchip_") + kNames[opt]);
}
int launch_grad_check(const StepParams&, int, int, int, void*) {
  return seen("check");
}
int launch_stash_records(const StashItem*, const ChunkDesc*, const TensorDesc*,
                         const TensorPtrs*, int, StashRec*, int, void*) {
  return 0;
}
int launch_stash(const StepParams&, const StashParams&, int opt, int, int, int,
                 void*) {
  seen(std::string(g_refuse ? "refused_" : "stash_") + kNames[opt]);
  g_last_error = g_refuse;
  return g_refuse;
}
int occupancy_lamb_pass1(int, int* b) { return *b = 3, 0; }
int occupancy_lamb_pass2(int, int* b) { return *b = 3, 0; }
int occupancy_lars_pass1(int, int* b) { return *b = 4, 0; }
int occupancy_lars_pass2(int, int* b) { return *b = 3, 0; }
int onchip_prepare(int, int* rows) { return *rows = 216, 0; }
int stash_prepare(int, int grad_bf16, int* slots, int* wslots) {
  *slots = grad_bf16 ? 24 : 23;
  *wslots = 2 * *slots - 32;
  return 0;
}
}  // namespace lamb

// ---- the runtime ------------------------------------------------------------
extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  return *v = 152, cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  return *p = std::calloc(n, 1), *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind,
                            cudaStream_t) {
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  return std::memset(d, v, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  return std::memset(d, v, n), cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const int e = g_last_error;
  g_last_error = 0;
  return (cudaError_t)e;
}
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  return *e = reinterpret_cast<cudaEvent_t>((intptr_t)++g_events), cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  return *ms = 1.f, cudaSuccess;
}
}

static int die(const char* what) {
  std::fprintf(stderr, "%s: %s\n", what, lamb_last_error());
  return 1;
}

int main(int argc, char** argv) {
  if (argc < 5) return 2;
  lamb_plan_options_t o;
  std::memset(&o, 0, sizeof o);
  o.algorithm = std::atoi(argv[1]);
  const std::string opt = argv[2];
  const uint32_t flags = (uint32_t)std::atoi(argv[3]);
  std::vector<int64_t> sizes;
  for (char* s = std::strtok(argv[4], ","); s; s = std::strtok(nullptr, ",")) {
    char* end = nullptr;
    const int64_t n = std::strtoll(s, &end, 10);
    sizes.insert(sizes.end(), *end == 'x' ? (size_t)std::atoll(end + 1) : 1, n);
  }
  for (int i = 5; i < argc; ++i) {
    const std::string a = argv[i];
    const std::string key = a.substr(0, a.find('='));
    const int v = std::atoi(a.c_str() + key.size() + 1);
    if (key == "chunk_elems") o.chunk_elems = v;
    else if (key == "blocks_per_sm") o.blocks_per_sm = v;
    else if (key == "tail_elems") o.tail_elems = v;
    else if (key == "onchip_rows") o.onchip_rows = v;
    else if (key == "onchip_max_ctas") o.onchip_max_ctas = v;
    else if (key == "wait_limit_ms") o.wait_limit_ms = v;
    else if (key == "shard_world") o.shard_world = v;
    else if (key == "refuse") g_refuse = v;
    else return 2;
  }
  lamb_plan_t plan = nullptr;
  if (lamb_plan_create(sizes.data(), (int32_t)sizes.size(), nullptr, LAMB_F32,
                       LAMB_DTYPE_NONE, 0, &o, &plan))
    return die("create");
  // any aligned address does: nothing reads or writes it
  std::vector<void*> ptr(sizes.size(), reinterpret_cast<void*>(0x10000));
  if (lamb_plan_bind(plan, ptr.data(), ptr.data(), ptr.data(), ptr.data(),
                     nullptr, nullptr))
    return die("bind");
  lamb_plan_info_t info;
  if (lamb_plan_get_info(plan, &info)) return die("info");
  g_plan_chunks = info.n_chunks;
  lamb_hyper_t h;
  std::memset(&h, 0, sizeof h);
  h.beta1 = .9;
  h.beta2 = .999;
  h.eps = 1e-6;
  h.trust_coef = 1.;
  h.flags = flags;
  const int32_t optimizer = opt == "lamb" ? LAMB_OPT_LAMB
                            : opt == "lars" ? LAMB_OPT_LARS
                            : opt == "nlamb" ? LAMB_OPT_NLAMB : LAMB_OPT_NNLAMB;
  int32_t form = 0;
  if (lamb_plan_step_form(plan, &h, optimizer, &form) ||
      !lamb_plan_step_form(plan, &h, 4, &form) ||
      !lamb_plan_step_form(plan, &h, optimizer, nullptr))
    return die("form");
  int64_t step = 1;
  float lr = .1f;
  double prod = 1.;
  if (lamb_plan_set_timing(plan, 1)) return die("timing");
  const lamb_status_t st =
      opt == "lars" ? lars_step(plan, &h, &step, &lr, nullptr)
      : opt == "lamb"
          ? lamb_step(plan, &h, &step, &lr, nullptr)
          : nlamb_step(plan, &h, .004, opt == "nnlamb", &step, &lr, &prod,
                       nullptr);
  int32_t timed = 0;
  double ms[3] = {0., 0., 0.};
  if (lamb_plan_read_timing(plan, &timed, ms, 3)) return die("read timing");
  // what the step launched is what the plan said it would
  const bool one = seen_any("stash_") || seen_any("refused_");
  if (form != (one ? LAMB_FORM_ONE_LAUNCH
               : seen_any("onchip_") ? LAMB_FORM_ON_CHIP : LAMB_FORM_TWO_PASS))
    return die("form of the step");
  std::string line = "algo " + std::to_string(info.algorithm) + " status " +
                     std::to_string((int)st) + ":";
  for (const std::string& x : g_launches) line += " " + x;
  line += " timed " + std::to_string((int)(ms[0] + ms[1] + ms[2]));
  line += " left " + std::to_string((int)cudaGetLastError());
  if (g_wrong_table) line += " wrong chunk table";
  std::printf("%s\n", line.c_str());
  if (lamb_plan_destroy(plan)) return die("destroy");
  return 0;
}
