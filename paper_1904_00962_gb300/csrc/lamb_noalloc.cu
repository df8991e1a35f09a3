// lamb_step_noalloc: one LAMB step that never allocates device memory.
//
// Who needs this: callers that must not call cudaMalloc -- code running
// under an allocator that owns all device memory (a framework caching
// allocator, a memory pool sized up front), code that must not hit the
// implicit device synchronisation a cudaMalloc/cudaFree can cause, or
// plugins that are handed a stream and buffers but no right to allocate.
// The plan API (lamb_plan_create) allocates its tables once with cudaMalloc;
// this entry point instead keeps every table, partial sum and counter in one
// fixed, file-scope device array that exists in every process that loads
// the library, on every GPU it runs on, until the process exits.
//
// The array is shared by all calls: calls that overlap on the GPU (different
// streams, or different host threads without ordering) race on it.  Each
// call rebuilds the tables and clears its counters, so it does not depend on
// what an earlier call left there.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "lamb.h"
#include "lamb_internal.h"

namespace lamb {
namespace {

// ---- limits and layout of the scratch array --------------------------------
constexpr int kNaMaxTensors = 4096;
constexpr int kNaMaxChunks = 131072;          // 2^31 elements at 16384/chunk
constexpr int kNaChunk = kDefaultChunk;       // same chunking as the plan API

constexpr size_t na_align(size_t x) { return (x + 255) / 256 * 256; }
constexpr size_t kOffSizes = 0;
constexpr size_t kOffMask = na_align(kOffSizes + 8ull * kNaMaxTensors);
constexpr size_t kOffRaw = na_align(kOffMask + 1ull * kNaMaxTensors);  // 5 arrays
constexpr size_t kOffTensors = na_align(kOffRaw + 5ull * 8 * kNaMaxTensors);
constexpr size_t kOffPtrs = na_align(kOffTensors + sizeof(TensorDesc) * kNaMaxTensors);
constexpr size_t kOffChunks = na_align(kOffPtrs + sizeof(TensorPtrs) * kNaMaxTensors);
constexpr size_t kOffSlots = na_align(kOffChunks + sizeof(ChunkDesc) * (size_t)kNaMaxChunks);
constexpr size_t kOffTickets = na_align(kOffSlots + 8ull * kNaMaxChunks);
constexpr size_t kOffRatio = na_align(kOffTickets + 4ull * kNaMaxTensors);
constexpr size_t kOffWnorm = na_align(kOffRatio + 8ull * kNaMaxTensors);
constexpr size_t kOffUnorm = na_align(kOffWnorm + 8ull * kNaMaxTensors);
constexpr size_t kOffScal = na_align(kOffUnorm + 8ull * kNaMaxTensors);
constexpr size_t kOffStatus = na_align(kOffScal + sizeof(StepScalars));
constexpr size_t kOffCounters = na_align(kOffStatus + 4);
constexpr size_t kNaScratchBytes = na_align(kOffCounters + 16);
static_assert(kNaScratchBytes <= (4u << 20), "scratch layout exceeds 4 MiB");

// The scratch itself: 4 MiB per GPU, for the life of the process.
static __device__ __align__(256) unsigned char g_noalloc_scratch[4u << 20];

// Failures are reported through lamb_last_error() like every other call.
lamb_status_t na_fail(lamb_status_t st, const char* fmt, ...) {
  char msg[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(msg, sizeof(msg), fmt, ap);
  va_end(ap);
  set_last_error(msg);
  return st;
}

// ---- per-device set-up (symbol address, SM count, grid sizes) --------------
constexpr int kNaMaxDevices = 64;
struct NaDevice {
  unsigned char* scratch = nullptr;   // device address of g_noalloc_scratch
  int num_sms = 0;
  int occ[4] = {0, 0, 0, 0};          // pass1 f32/bf16 g, pass2 no copy/copy
};
NaDevice g_na_dev[kNaMaxDevices];
std::atomic<int> g_na_ready[kNaMaxDevices];
std::mutex g_na_mutex;

// Runs once per device, with that device current.
cudaError_t na_setup(int dev, NaDevice** out) {
  if (g_na_ready[dev].load(std::memory_order_acquire)) {
    *out = &g_na_dev[dev];
    return cudaSuccess;
  }
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ready[dev].load(std::memory_order_relaxed)) {
    NaDevice d;
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    d.scratch = static_cast<unsigned char*>(ptr);
    e = cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int rc = occupancy_lamb_pass1(0, &d.occ[0]);
    if (!rc) rc = occupancy_lamb_pass1(1, &d.occ[1]);
    if (!rc) rc = occupancy_lamb_pass2(0, &d.occ[2]);
    if (!rc) rc = occupancy_lamb_pass2(1, &d.occ[3]);
    if (rc) return (cudaError_t)rc;
    g_na_dev[dev] = d;
    g_na_ready[dev].store(1, std::memory_order_release);
  }
  *out = &g_na_dev[dev];
  return cudaSuccess;
}

// ---- set-up kernel: builds the tables inside the scratch array -------------
// The caller's host arrays, for the tensors of one call.
struct NaSource {
  const int64_t* sizes;
  const uint8_t* mask;      // NULL: every tensor decays
  void* const* ptr[5];      // w, g, m, v, copy (NULL: no copies)
};

// The same arrays as a kernel parameter: up to kCap tensors go to the device
// with the set-up launch itself.
template <int kCap>
struct NaArgs {
  int64_t sizes[kCap];
  void* ptr[5][kCap];
  uint8_t mask[kCap];
};
// A launch takes at most 32764 bytes of parameters; a small step should not
// carry all of them, so there are two sizes (161 tensors are a ResNet-50).
constexpr int kNaArgsSmall = 192, kNaArgsLarge = 640;
static_assert(sizeof(NaArgs<kNaArgsLarge>) + 16 <= 32764, "kernel parameters");

// CTAs of 1024 threads.  Each scans the tensors' chunk counts for itself
// (the first chunk and the last chunk's length of every tensor stay in its
// shared memory); the tensors' tables (with the 128-bit alignment flag),
// tickets and default results (ratio 1, norms 0) are written by whole warps
// dealt over the CTAs, and every thread writes the chunk table's entries of
// its grid-wide index, finding their tensor by a binary search.  The CTAs
// share nothing, so none waits.
//
// What bounds it: latency -- the launch, the scan's few barriers and the
// stores; hence one tensor a thread up to 1024 tensors, a scan by shuffles,
// and kSetupChunks entries per CTA.  ResNet-50's 161 tensors and 1,643
// chunks: 7.6 us by one CTA with a scan in shared memory, 5.9 us so; the
// whole step 183 us with the arrays copied first, 173 us with the arrays in
// the launch (171 since pass 2 is launched early; the passes take 157).
constexpr int kSetupThreads = 1024;
constexpr int kSetupWarps = kSetupThreads / 32;
constexpr int kSetupChunks = 256;

__device__ __forceinline__ void build_tables(const NaSource& src, int n,
                                             int grad_bf16) {
  unsigned char* s = g_noalloc_scratch;
  TensorDesc* tens = reinterpret_cast<TensorDesc*>(s + kOffTensors);
  TensorPtrs* ptrs = reinterpret_cast<TensorPtrs*>(s + kOffPtrs);
  ChunkDesc* chunks = reinterpret_cast<ChunkDesc*>(s + kOffChunks);
  uint32_t* tickets = reinterpret_cast<uint32_t*>(s + kOffTickets);
  double* ratio = reinterpret_cast<double*>(s + kOffRatio);
  double* wnorm = reinterpret_cast<double*>(s + kOffWnorm);
  double* unorm = reinterpret_cast<double*>(s + kOffUnorm);
  uint32_t* status = reinterpret_cast<uint32_t*>(s + kOffStatus);
  uint32_t* counters = reinterpret_cast<uint32_t*>(s + kOffCounters);

  __shared__ int32_t s_warp[kSetupWarps];
  __shared__ int32_t s_first[kNaMaxTensors];     // first chunk of tensor k
  __shared__ int32_t s_lastlen[kNaMaxTensors];   // length of its last chunk
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // thread t owns the tensors [t * per, (t + 1) * per)
  const int per = (n + kSetupThreads - 1) / kSetupThreads;
  int32_t sum = 0;              // at most kNaMaxChunks chunks in all
  for (int i = 0; i < per; ++i) {
    const int k = t * per + i;
    if (k < n) sum += (int32_t)((src.sizes[k] + kNaChunk - 1) / kNaChunk);
  }
  int32_t incl = sum;           // inclusive scan in the warp, then of warps
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int32_t before = 0, n_chunks = 0;
  for (int w = 0; w < kSetupWarps; ++w) {
    const int32_t x = s_warp[w];
    if (w < warp) before += x;
    n_chunks += x;
  }
  const bool mine = (uint32_t)warp % gridDim.x == blockIdx.x;
  int32_t first = before + incl - sum;
  for (int i = 0; i < per; ++i) {
    const int k = t * per + i;
    if (k >= n) break;
    const int64_t d = src.sizes[k];
    const int32_t nc = (int32_t)((d + kNaChunk - 1) / kNaChunk);
    s_first[k] = first;
    s_lastlen[k] = (int32_t)(d - (int64_t)(nc - 1) * kNaChunk);
    if (mine) {
      TensorDesc td{};
      td.numel = d;
      td.first_chunk = first;
      td.n_chunks = nc;
      td.decay = (!src.mask || src.mask[k]) ? 1.0f : 0.0f;
      tens[k] = td;
      TensorPtrs tp{};
      tp.w = static_cast<float*>(src.ptr[0][k]);
      tp.g = src.ptr[1][k];
      tp.m = static_cast<float*>(src.ptr[2][k]);
      tp.v = static_cast<float*>(src.ptr[3][k]);
      tp.copy = src.ptr[4] ? src.ptr[4][k] : nullptr;
      const uintptr_t ga = grad_bf16 ? 8 : 16;
      const bool ok = (uintptr_t)tp.w % 16 == 0 && (uintptr_t)tp.m % 16 == 0 &&
                      (uintptr_t)tp.v % 16 == 0 && (uintptr_t)tp.g % ga == 0 &&
                      (uintptr_t)tp.copy % 8 == 0;
      tp.vec_ok = ok ? 1u : 0u;
      ptrs[k] = tp;
      tickets[k] = 0u;
      ratio[k] = 1.0;
      wnorm[k] = 0.0;
      unorm[k] = 0.0;
    }
    first += nc;
  }
  if (t == 0 && blockIdx.x == 0) {
    *status = 0u;
    counters[0] = counters[1] = counters[2] = counters[3] = 0u;
  }
  __syncthreads();   // the tensors' first chunks are complete
  for (int32_t c = (int32_t)blockIdx.x + t * (int32_t)gridDim.x; c < n_chunks;
       c += kSetupThreads * (int32_t)gridDim.x) {
    // the last tensor whose first chunk is <= c (a 0-chunk tensor shares its
    // first chunk with the next one, which comes later and wins)
    int lo = 0, hi = n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (s_first[mid] <= c) lo = mid;
      else hi = mid - 1;
    }
    // tensor lo holds chunk c; its chunks end where the next tensor's begin
    const int32_t end = lo + 1 < n ? s_first[lo + 1] : n_chunks;
    ChunkDesc cd;
    cd.offset = (int64_t)(c - s_first[lo]) * kNaChunk;
    cd.tensor = lo;
    cd.len = c + 1 == end ? s_lastlen[lo] : kNaChunk;
    chunks[c] = cd;
  }
}

// The arrays come with the launch (at most kCap tensors).
template <int kCap>
__global__ void __launch_bounds__(kSetupThreads)
    noalloc_setup_args_kernel(const __grid_constant__ NaArgs<kCap> a, int n,
                              int has_mask, int grad_bf16, int copy_bf16) {
  NaSource src;
  src.sizes = a.sizes;
  src.mask = has_mask ? a.mask : nullptr;
  for (int i = 0; i < 4; ++i) src.ptr[i] = a.ptr[i];
  src.ptr[4] = copy_bf16 ? a.ptr[4] : nullptr;
  build_tables(src, n, grad_bf16);
}

// The arrays were copied into the scratch (any number of tensors).
__global__ void __launch_bounds__(kSetupThreads)
    noalloc_setup_kernel(int n, int has_mask, int grad_bf16, int copy_bf16) {
  unsigned char* s = g_noalloc_scratch;
  NaSource src;
  src.sizes = reinterpret_cast<const int64_t*>(s + kOffSizes);
  src.mask = has_mask ? s + kOffMask : nullptr;
  for (int i = 0; i < 5; ++i)
    src.ptr[i] = reinterpret_cast<void* const*>(s + kOffRaw) +
                 (size_t)i * kNaMaxTensors;
  if (!copy_bf16) src.ptr[4] = nullptr;
  build_tables(src, n, grad_bf16);
}

// The caller's arrays, as the host sees them.
struct NaHost {
  const int64_t* sizes;
  const uint8_t* mask;
  const void* const* ptr[5];
};

template <int kCap>
cudaError_t setup_from_args(const NaHost& a, int n, int grad_bf16, int grid,
                            cudaStream_t stream) {
  NaArgs<kCap> args;   // the launch copies it; entries past n are not read
  std::memcpy(args.sizes, a.sizes, (size_t)n * 8);
  for (int i = 0; i < 5; ++i)
    if (a.ptr[i]) std::memcpy(args.ptr[i], a.ptr[i], (size_t)n * 8);
  if (a.mask) std::memcpy(args.mask, a.mask, (size_t)n);
  noalloc_setup_args_kernel<kCap><<<grid, kSetupThreads, 0, stream>>>(
      args, n, a.mask ? 1 : 0, grad_bf16, a.ptr[4] ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t setup_from_copies(unsigned char* s, const NaHost& a, int n,
                              int grad_bf16, int grid, cudaStream_t stream) {
  const size_t nb = (size_t)n * 8;
  cudaError_t e = cudaMemcpyAsync(s + kOffSizes, a.sizes, nb,
                                  cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess && a.mask)
    e = cudaMemcpyAsync(s + kOffMask, a.mask, (size_t)n,
                        cudaMemcpyHostToDevice, stream);
  for (int i = 0; i < 5 && e == cudaSuccess; ++i)
    if (a.ptr[i])
      e = cudaMemcpyAsync(s + kOffRaw + (size_t)i * 8 * kNaMaxTensors,
                          a.ptr[i], nb, cudaMemcpyHostToDevice, stream);
  if (e != cudaSuccess) return e;
  noalloc_setup_kernel<<<grid, kSetupThreads, 0, stream>>>(
      n, a.mask ? 1 : 0, grad_bf16, a.ptr[4] ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace
}  // namespace lamb

using namespace lamb;

extern "C" LAMB_API lamb_status_t lamb_step_noalloc(
    const int64_t* sizes, int32_t n_tensors, const uint8_t* decay_mask,
    int32_t grad_dtype, int32_t copy_dtype, void* const* w,
    const void* const* g, void* const* m, void* const* v,
    void* const* w_copy, const lamb_hyper_t* hyper, int64_t* d_step,
    const float* d_lr, double* d_ratio, cudaStream_t stream) {
  // ---- host-side checks (no device work yet) -----------------------------
  if (n_tensors < 1 || n_tensors > kNaMaxTensors)
    return na_fail(LAMB_ERR_INVALID_ARG,
                   "lamb_step_noalloc: n_tensors must be in [1, %d] (got %d)",
                   kNaMaxTensors, n_tensors);
  if (!sizes || !w || !g || !m || !v || !hyper || !d_lr)
    return na_fail(LAMB_ERR_INVALID_ARG,
                   "lamb_step_noalloc: sizes, w, g, m, v, hyper and d_lr are "
                   "required");
  if (grad_dtype != LAMB_F32 && grad_dtype != LAMB_BF16)
    return na_fail(LAMB_ERR_UNSUPPORTED_DTYPE,
                   "lamb_step_noalloc: grad_dtype %d unsupported", grad_dtype);
  if (copy_dtype != LAMB_DTYPE_NONE && copy_dtype != LAMB_BF16)
    return na_fail(LAMB_ERR_UNSUPPORTED_DTYPE,
                   "lamb_step_noalloc: copy_dtype %d unsupported", copy_dtype);
  const bool copy = copy_dtype == LAMB_BF16;
  if (copy && !w_copy)
    return na_fail(LAMB_ERR_INVALID_ARG,
                   "lamb_step_noalloc: w_copy is required with a bf16 copy");
  const lamb_hyper_t& h = *hyper;
  if (!(h.beta1 >= 0.0 && h.beta1 < 1.0) || !(h.beta2 >= 0.0 && h.beta2 < 1.0) ||
      !(h.eps >= 0.0 && std::isfinite(h.eps)) || !std::isfinite(h.weight_decay) ||
      (h.phi != LAMB_PHI_IDENTITY && h.phi != LAMB_PHI_CLIP) ||
      (h.phi == LAMB_PHI_CLIP && !(h.gamma_l <= h.gamma_u)) ||
      (h.flags & ~(uint32_t)(LAMB_FLAG_BIAS_CORRECTION | LAMB_FLAG_INCREMENT_STEP)))
    return na_fail(LAMB_ERR_INVALID_ARG, "lamb_step_noalloc: bad hyper");
  if (!d_step && (h.flags & (LAMB_FLAG_BIAS_CORRECTION | LAMB_FLAG_INCREMENT_STEP)))
    return na_fail(LAMB_ERR_INVALID_ARG,
                   "lamb_step_noalloc: d_step is NULL but the flags need it");
  int64_t n_chunks = 0;
  for (int k = 0; k < n_tensors; ++k) {
    const int64_t d = sizes[k];
    if (d < 0)
      return na_fail(LAMB_ERR_INVALID_ARG,
                     "lamb_step_noalloc: sizes[%d] is negative", k);
    if (d > (int64_t)kNaMaxChunks * kNaChunk)   // before any rounding sum
      return na_fail(LAMB_ERR_INVALID_ARG,
                     "lamb_step_noalloc: sizes[%d] = %lld exceeds the %lld "
                     "parameters the scratch holds", k, (long long)d,
                     (long long)kNaMaxChunks * kNaChunk);
    n_chunks += (d + kNaChunk - 1) / kNaChunk;
    if (n_chunks > kNaMaxChunks)
      return na_fail(LAMB_ERR_INVALID_ARG,
                     "lamb_step_noalloc: more than %d chunks of %d elements "
                     "(at most %lld parameters in total)",
                     kNaMaxChunks, kNaChunk,
                     (long long)kNaMaxChunks * kNaChunk);
    if (d > 0) {
      if (!w[k] || !g[k] || !m[k] || !v[k] || (copy && !w_copy[k]))
        return na_fail(LAMB_ERR_INVALID_ARG,
                       "lamb_step_noalloc: tensor %d has a NULL pointer", k);
      if ((uintptr_t)w[k] % 4 || (uintptr_t)m[k] % 4 || (uintptr_t)v[k] % 4 ||
          (uintptr_t)g[k] % (grad_dtype == LAMB_BF16 ? 2 : 4) ||
          (copy && (uintptr_t)w_copy[k] % 2))
        return na_fail(LAMB_ERR_INVALID_ARG,
                       "lamb_step_noalloc: tensor %d pointer not aligned to "
                       "its element size", k);
    }
  }

  // ---- per-device set-up (first call on a device) --------------------------
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kNaMaxDevices)
    return na_fail(LAMB_ERR_CUDA, "lamb_step_noalloc: cudaGetDevice: %s",
                   cudaGetErrorString(e));
  NaDevice* nd = nullptr;
  e = na_setup(dev, &nd);
  if (e != cudaSuccess)
    return na_fail(LAMB_ERR_CUDA, "lamb_step_noalloc: set-up: %s",
                   cudaGetErrorString(e));
  unsigned char* s = nd->scratch;

  // ---- the tables, from the caller's host arrays ---------------------------
  // As a parameter of the set-up launch as far as they fit: one launch in
  // place of six or seven copies and a launch.
  const int gbf = grad_dtype == LAMB_BF16 ? 1 : 0;
  const NaHost host = {sizes, decay_mask, {w, g, m, v, copy ? w_copy : nullptr}};
  int sgrid = (int)((n_chunks + kSetupChunks - 1) / kSetupChunks);
  if (sgrid > nd->num_sms) sgrid = nd->num_sms;
  if (sgrid < 1) sgrid = 1;
  if (n_tensors <= kNaArgsSmall)
    e = setup_from_args<kNaArgsSmall>(host, n_tensors, gbf, sgrid, stream);
  else if (n_tensors <= kNaArgsLarge)
    e = setup_from_args<kNaArgsLarge>(host, n_tensors, gbf, sgrid, stream);
  else
    e = setup_from_copies(s, host, n_tensors, gbf, sgrid, stream);
  if (e != cudaSuccess)
    return na_fail(LAMB_ERR_CUDA, "lamb_step_noalloc: set-up: %s",
                   cudaGetErrorString(e));

  // ---- the two LAMB passes on tables inside the scratch --------------------
  // The flags check above admits BIAS_CORRECTION and INCREMENT_STEP only:
  // the fields of the schedule, the gradient check and the N-LAMB product
  // stay zero / NULL here, which is what those two flags need.
  StepParams sp;
  std::memset(&sp, 0, sizeof(sp));
  fill_hyper(h, &sp);
  sp.chunks = reinterpret_cast<const ChunkDesc*>(s + kOffChunks);
  sp.tensors = reinterpret_cast<const TensorDesc*>(s + kOffTensors);
  sp.ptrs = reinterpret_cast<const TensorPtrs*>(s + kOffPtrs);
  sp.slots = reinterpret_cast<float2*>(s + kOffSlots);
  sp.tickets = reinterpret_cast<uint32_t*>(s + kOffTickets);
  sp.counters = reinterpret_cast<uint32_t*>(s + kOffCounters);
  sp.ratio = reinterpret_cast<double*>(s + kOffRatio);
  sp.wnorm = reinterpret_cast<double*>(s + kOffWnorm);
  sp.unorm = reinterpret_cast<double*>(s + kOffUnorm);
  sp.scal = reinterpret_cast<StepScalars*>(s + kOffScal);
  sp.status = reinterpret_cast<uint32_t*>(s + kOffStatus);
  sp.d_step = d_step;
  sp.d_lr = d_lr;
  sp.n_chunks = (int32_t)n_chunks;
  auto grid_of = [&](int occ) {
    int64_t gsz = (int64_t)nd->num_sms * (occ < 1 ? 1 : occ);
    if (gsz > n_chunks) gsz = n_chunks;
    return (int)(gsz < 1 ? 1 : gsz);
  };
  int rc = launch_lamb_pass1(sp, 0, gbf, grid_of(nd->occ[gbf]), stream);
  if (!rc)
    rc = launch_lamb_pass2(sp, 0, gbf, copy ? 1 : 0,
                           grid_of(nd->occ[2 + (copy ? 1 : 0)]), stream);
  if (!rc && d_ratio)
    rc = (int)cudaMemcpyAsync(d_ratio, s + kOffRatio, (size_t)n_tensors * 8,
                              cudaMemcpyDeviceToDevice, stream);
  if (rc)
    return na_fail(LAMB_ERR_CUDA, "lamb_step_noalloc: %s",
                   cudaGetErrorString((cudaError_t)rc));
  return LAMB_OK;
}
