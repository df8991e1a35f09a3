// sm_103a kernel of the two-pass step as one launch that reads and writes
// every operand once.
//
// The two-pass kernels read m, v and w a second time because the trust ratio
// of a tensor needs all of it (40 B per parameter with bf16 g and a bf16
// copy).  Here the SM that forms a chunk's u keeps it, with w, until the
// tensor's ratio is known, and then writes the new w: 28 B.  The element
// arithmetic is the two-pass kernels' (m, v and u are theirs bit for bit); the
// norms are summed in another fixed order (fp32 over four elements of a thread,
// two floats over the thread's tiles and the chunk's warps, fp64 over chunks), so
// every run gives the same bits, and a norm is within some 2e-9 of the exact one.
//
// One cooperative launch, one CTA per SM, 20 warps:
//   workers (16 warps)  A TILE is 1,024 elements of a chunk, one float4 for
//     each of 256 threads; workers 0-7 take a chunk's even tiles and 8-15 its
//     odd ones (8 warps alone were bound by the latency of the square root and
//     the division: 2.5 ms on BERT-large).  A pair of tiles arrives in a stage
//     of shared memory; after pass 1 w and u go to the thread's place in a ring
//     of tiles, u in tensor memory, w in shared memory or, past its end, in
//     tensor memory too (a warp reaches its own quarter of the lanes, which is
//     all it needs: a thread's elements are read by nobody else).  Workers never
//     meet: a warp has its own positions in the chunk sequence and in the ring,
//     and updates w from the ring once a chunk's ratio is there, between the
//     tiles of a later chunk.
//   loader   copies the pairs of tiles, one cp.async.bulk per array (issuing a
//     copy takes ~100 cycles of the one warp), as far ahead as there are
//     stages.  It copies whole 16-byte granules, so a tensor at any address
//     streams in; the workers read at the remainder.
//   drawer   takes items (chunks) from the work counter and writes their
//     records, about a chunk ahead of the workers; a chunk that is kept gets a
//     second record, for its update.
//   closer   combines a finished chunk's sixteen warp sums, publishes them and
//     takes the tensor's ticket; for a tensor's last chunk it forms the norms
//     and the ratio (the two-pass finaliser's sums, in its order) and
//     publishes eta rho_k in a 64-bit word tagged with the launch.
//   poller   reloads those words for the chunks that wait (one lane for each
//     record) and hands eta rho_k to the workers.
//
// Storage: w and u of a tile take 4 KB each.  Shared memory holds three stages
// and 28 tiles of w next to the records (32 with bf16 g), tensor memory 64
// tiles: a ring of 46 tiles (48), half of them even ones.  A CTA can always keep
// four chunks of 10,240 elements of one tensor: 6.2M parameters over 152 SMs.
// A larger tensor (a word embedding) keeps its first chunks; the rest goes
// through pass 1 only and is read again, last chunk first, when its ratio is
// known (12 B more).
//
// No wait can close a circle.  Items are drawn in order; a worker waits only
// for the ratio of a chunk it holds, and all chunks of that tensor are either
// drawn or will be: a CTA that holds max_keep chunks of a tensor draws again
// only after the counter has passed that tensor's kept chunks, so a chunk in
// work always finds room once older tensors are updated, and the oldest
// tensor with an unfinished chunk waits for nothing.  All CTAs are resident
// (cooperative launch).  The waits are bounded all the same: a poller that
// waits longer than the plan's limit sets LAMB_STATUS_WAIT_TIMEOUT and an
// abort word, and every CTA returns.
//
// Measured (us per step, the two kernels / this one): BERT-large LAMB with bf16
// g and copy 1924 / 1496, N-LAMB 2039 / 1499, BERT-base LAMB 638 / 518, 4,000
// ragged tensors (1.1e9 parameters) 6416 / 4590.  That is 0.93 of a copy's rate
// on BERT-large's 28 B per parameter.  What is left there: the embedding's
// second read, rings that are full while a 4096 x 1024 tensor is finished (13%
// of the workers' time), and the last chunks' ratios.
//
// The work counter is reset by the CTA that draws last, the epoch behind the
// words' tags by the last CTA to finish, which also closes the step: nothing
// is reset by the host, so the launch can be replayed from a CUDA graph.
#include "lamb_device.cuh"
#include "lamb_stash.h"
#include "lamb_sync.cuh"

namespace lamb {
namespace {

constexpr int kOptLars = 3;
constexpr int kWorkers = 2 * kWarps;
constexpr int kDrawer = kWorkers, kCloser = kWorkers + 1,
              kPoller = kWorkers + 2, kLoader = kWorkers + 3;
constexpr int kStashThreads = (kWorkers + 4) * 32;
constexpr uint32_t kAllLanes = 0xffffffffu;
constexpr int kStages = 3;       // pairs of tiles in flight
constexpr int kTmemSlots = 32;   // float4s a thread has in tensor memory: 512
                                 // columns, 4 warps per quarter, 4 each
// an array's part of a stage, with the granule that an unaligned one needs more
constexpr int kPairBytes = 2 * kStashTile * 4 + 16;
template <typename GT>
constexpr int kStageBytes = 3 * kPairBytes + 2 * kStashTile * (int)sizeof(GT) +
                            16;

// ---------------------------------------------------------------------------
// Sums of squares in two floats (the error of each addition is kept: ~48
// significant bits), as in the on-chip kernel, whose plans run here too.  Not
// renormalised on the way, so that hi alone is the fp32 sum, infinities
// included.  Against plain fp32 sums, us: BERT-base 515 / 518, BERT-large 1512 /
// 1496 (with more loads in flight in `combine`), 4,000 ragged tensors 4562 /
// 4590.
// ---------------------------------------------------------------------------
struct Sum2 {
  float hi, lo;
};
__device__ __forceinline__ void sum2_add(Sum2& a, float x) {
  const float s = __fadd_rn(a.hi, x);
  const float y = __fsub_rn(s, a.hi);
  a.lo = __fadd_rn(a.lo, __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, y)),
                                   __fsub_rn(x, y)));
  a.hi = s;
}
__device__ __forceinline__ void sum2_add(Sum2& a, const Sum2& b) {
  sum2_add(a, b.hi);
  a.lo = __fadd_rn(a.lo, b.lo);
}
// Each half of the warp's lanes by itself: valid in lanes 0 and 16.
__device__ __forceinline__ void sum2_half_warps(Sum2& a) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const Sum2 b{__shfl_xor_sync(kAllLanes, a.hi, o),
                 __shfl_xor_sync(kAllLanes, a.lo, o)};
    sum2_add(a, b);
  }
}
// (the error term of a sum that is not finite is not a number)
__device__ __forceinline__ double sum2_value(const Sum2& a) {
  return isfinite(a.hi) ? (double)a.hi + (double)a.lo : (double)a.hi;
}

// A kept chunk that waits for its update.
struct __align__(16) Kept {
  float* w;             // at the chunk's first element
  void* copy;
  int32_t len;
  uint32_t vec;
  int32_t tiles;
  int32_t tensor;
  float dd;             // eta lambda_k (decoupled decay) or 0
  float s;              // eta rho_k, set when it is known
};

// A drawn chunk.
struct __align__(16) Rec : StashRec {
  int32_t len;
  uint32_t kind;        // kStash*
  uint32_t vec;         // arrays aligned for float4 accesses
  int32_t tiles;
  float lam;            // lambda_k inside u
  float dd;             // eta lambda_k outside it (decoupled decay) or 0
  float s;              // eta rho_k, set when it is known (kStashReread)
};

struct Shared {
  Rec rec[kStashRecs];
  Kept kept[kStashRecs];
  Sum2 red[kStashRecs][2][kWorkers];   // sum w^2, sum u^2 of each worker
  uint64_t full[kStashRecs];     // record written
  uint64_t done[kStashRecs];     // the workers finished pass 1 (or pass 2 of
                                 // a re-read chunk)
  uint64_t ready[kStashRecs];    // rec.s is set
  uint64_t free[kStashRecs];     // nobody reads the record any more
  uint64_t kfull[kStashRecs];    // the same of the kept chunks' records
  uint64_t kready[kStashRecs];
  uint64_t kfree[kStashRecs];
  uint64_t sfull[kStages];       // a stage's pair of tiles has arrived
  uint64_t sfree[kStages];       // and has been read
  LambConsts k;
  int64_t t;
  float lr;
  int skip;
  uint32_t unused_draw;
  uint32_t epoch, abort_word;
  uint32_t tmem;
  int abort;             // leave at once
  int dry;               // a step that is skipped: norms only
  int issued;            // tiles whose copies have been started
  int end_seq;           // chunks this CTA drew, once known
  int end_kept;          // kept chunks among them
};

__device__ __forceinline__ bool aborted(const Shared& sh) {
  return *reinterpret_cast<const volatile int*>(&sh.abort) != 0;
}
// Waits for a phase; false if the launch gives up.
__device__ __forceinline__ bool wait_phase(const Shared& sh, uint64_t* b,
                                           uint32_t parity) {
  while (!mbar_try(b, parity))
    if (aborted(sh)) return false;
  return true;
}
// The same, and whether the launch gives up, with one answer for a warp: its
// lanes look at the flag one by one, and lanes that left alone would be waited
// for in the next warp-wide operation.
__device__ __forceinline__ bool warp_wait(const Shared& sh, uint64_t* b,
                                          uint32_t parity) {
  return __all_sync(kAllLanes, wait_phase(sh, b, parity));
}
__device__ __forceinline__ bool warp_aborted(const Shared& sh) {
  return __any_sync(kAllLanes, aborted(sh));
}
__device__ __forceinline__ uint32_t phase_of(int seq) {
  return (uint32_t)(seq / kStashRecs) & 1u;
}

// ---------------------------------------------------------------------------
// Tiles.  Aligned chunks: tile i holds the float4s 256 i .. 256 i + 255, one
// per thread t; the len mod 4 last elements form one more tile.  Others: tile
// i holds elements 1024 i .. + 1023, thread t those at t + 256 c.
// ---------------------------------------------------------------------------
struct Span {
  int at, n;       // first element inside the chunk, elements
};
template <typename R>
__device__ __forceinline__ int full_tiles(const R& r) {
  return r.vec ? r.len / kStashTile : 0;
}
template <typename R>
__device__ __forceinline__ Span tile_span(const R& r, int tile) {
  const int at = tile * kStashTile;
  if (!r.vec) return Span{at, min(kStashTile, r.len - at)};
  const int whole = r.len & ~3;
  if (at < whole) return Span{at, min(kStashTile, whole - at)};
  return Span{whole, r.len - whole};
}
__device__ __forceinline__ int chunk_tiles(int len, bool vec) {
  if (!vec) return (len + kStashTile - 1) / kStashTile;
  const int nv = len >> 2;
  return (nv + kThreads - 1) / kThreads + ((len & 3) ? 1 : 0);
}
// The elements that a pair of tiles spans: tiles 2 i and 2 i + 1 are adjacent.
template <typename R>
__device__ __forceinline__ Span pair_span(const R& r, int pair) {
  const Span a = tile_span(r, 2 * pair);
  return Span{a.at, 2 * pair + 1 < r.tiles ? a.n + tile_span(r, 2 * pair + 1).n
                                           : a.n};
}
// A thread's elements of a tile that is not full: n of them from `at` in
// steps of `step`, relative to the tile.
struct Part {
  int at, step, n;
};
template <typename R>
__device__ __forceinline__ Part tile_part(const R& r, const Span& s, int t) {
  if (r.vec && s.n >= 4) return Part{4 * t, 1, 4 * t < s.n ? 4 : 0};
  const int left = s.n - t;
  return Part{t, kThreads,
              left <= 0 ? 0 : min(4, (left + kThreads - 1) / kThreads)};
}
__device__ __forceinline__ uint32_t skew(const void* p) {
  return (uint32_t)(uintptr_t)p & 15u;
}

// Four gradients at 8 (bf16) or 16 bytes alignment in shared memory.
__device__ __forceinline__ float4 grad4(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 grad4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16),
                     __uint_as_float(u.x & 0xffff0000u),
                     __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float grad1(const float* p) { return *p; }
__device__ __forceinline__ float grad1(const __nv_bfloat16* p) {
  return __uint_as_float(
      (uint32_t)*reinterpret_cast<const unsigned short*>(p) << 16);
}

__device__ __forceinline__ float4 new_w(const float4& w, const float4& u,
                                        float s, float dd) {
  float4 o;
  o.x = __fmaf_rn(-s, u.x, w.x);
  o.y = __fmaf_rn(-s, u.y, w.y);
  o.z = __fmaf_rn(-s, u.z, w.z);
  o.w = __fmaf_rn(-s, u.w, w.w);
  if (dd != 0.f) {   // skipped, not added as a zero (signed zeros)
    o.x = __fmaf_rn(-dd, w.x, o.x);
    o.y = __fmaf_rn(-dd, w.y, o.y);
    o.z = __fmaf_rn(-dd, w.z, o.z);
    o.w = __fmaf_rn(-dd, w.w, o.w);
  }
  return o;
}

// The new w (and its copy) of a tile that is not full; w and copy at the tile.
template <bool kCopy>
__device__ __forceinline__ void store_new_w(float* w, void* copy, const Part& q,
                                            const float4& o) {
  const float x[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (c < q.n) {
      w[q.at + c * q.step] = x[c];
      if (kCopy) st_copy1(copy, q.at + c * q.step, x[c]);
    }
  }
}
template <int kOpt>
__device__ __forceinline__ float direction(float m, float v, float g, float w,
                                           float lam, const LambConsts& k) {
  if (kOpt == kOptLars) return m;
  return kOpt ? nlamb_direction<kOpt>(m, v, g, w, lam, k)
              : lamb_direction(m, v, w, lam, k);
}

// ---------------------------------------------------------------------------
// Workers
// ---------------------------------------------------------------------------
// Shared memory: stages (w, m, v, g of a pair of tiles), ring of the even
// tiles' w, of the odd tiles'.
template <int kOpt, typename GT, bool kCopy>
struct Worker {
  static constexpr bool kV = kOpt != kOptLars;
  Shared& sh;
  char* smem;
  float4* ring;            // this thread's w of slot x at x * kThreads
  const uint32_t tm;       // this warp's u of slot 0 in tensor memory
  const int slots;         // ring slots of this half of the tiles
  const int wslots;        // those whose w is in shared memory
  const int t, half, lane;
  const bool store;        // false: a skipped step, which forms its norms only
  const LambConsts k;
  int count = 0;                 // pairs taken
  int wslot = 0, held = 0;       // next ring slot, slots held
  int kseq = 0;                  // kept chunks formed
  int hseq = 0, htile, hslot = 0;   // oldest held one, its next tile
  Sum2 aw{0.f, 0.f}, au{0.f, 0.f};

  __device__ Worker(const StepParams& p, const StashParams& q, Shared& s,
                    char* m, uint32_t tmem)
      : sh(s), smem(m),
        ring(reinterpret_cast<float4*>(m + kStages * kStageBytes<GT>) +
             (threadIdx.x / kThreads) * q.wslots * kThreads +
             threadIdx.x % kThreads),
        tm(tmem + (((threadIdx.x >> 5) & 3u) << 21) +
           (threadIdx.x >> 7) * (4u * kTmemSlots)),
        slots(q.slots), wslots(q.wslots), t((int)threadIdx.x % kThreads),
        half((int)threadIdx.x / kThreads), lane((int)threadIdx.x & 31),
        store(s.dry == 0),
        k{p.b1, p.omb1, p.b2, p.omb2, s.k.c1, s.k.c2, p.eps,
          s.k.am, s.k.ag, s.k.bv, s.k.bg} {
    htile = half;
  }

  __device__ __forceinline__ bool all_test(uint64_t* b, uint32_t parity) {
    return __all_sync(kAllLanes, mbar_test(b, parity));
  }
  __device__ __forceinline__ bool head_ready() {
    return hseq < kseq &&
           all_test(&sh.kready[hseq % kStashRecs], phase_of(hseq));
  }
  __device__ __forceinline__ bool head_wait() {
    return warp_wait(sh, &sh.kready[hseq % kStashRecs], phase_of(hseq));
  }

  // Where slot x has its u, and its w if that is in tensor memory.
  __device__ __forceinline__ uint32_t u_at(int x) {
    return tm + (uint32_t)(4 * x);
  }
  __device__ __forceinline__ uint32_t w_at(int x) {
    return tm + (uint32_t)(4 * (slots + x - wslots));
  }

  // Up to two tiles of the oldest held chunk, whose ratio is known.
  __device__ __forceinline__ void update_some() {
    const int rs = hseq % kStashRecs;
    const Kept& r = sh.kept[rs];
    const int tiles = r.tiles, full = full_tiles(r);
    const float s = r.s, dd = r.dd;
    const int n = min(2, (tiles - htile + 1) / 2);
    if (n > 0) {
      tmem_wait_st();
      const int x0 = hslot, x1 = hslot + 1 == slots ? 0 : hslot + 1;
      const uint32_t a[4] = {u_at(x0), u_at(x1),
                             x0 < wslots ? u_at(x0) : w_at(x0),
                             x1 < wslots ? u_at(x1) : w_at(x1)};
      float4 y[4];
      tmem_ld4x4(a, y);
      if (x0 < wslots) y[2] = ring[x0 * kThreads];
      if (x1 < wslots) y[3] = ring[x1 * kThreads];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i < n) {
          const int tile = htile + 2 * i;
          const float4 o = new_w(y[2 + i], y[i], s, dd);
          if (tile < full) {
            const int at = 4 * (tile * kThreads + t);
            st4_last(r.w + at, o);
            if (kCopy) st_copy4(r.copy, at, o);
          } else {
            const Span sp = tile_span(r, tile);
            store_new_w<kCopy>(r.w + sp.at,
                               static_cast<__nv_bfloat16*>(r.copy) + sp.at,
                               tile_part(r, sp, t), o);
          }
        }
      }
      htile += 2 * n;
      held -= n;
      hslot += n;
      if (hslot >= slots) hslot -= slots;
    }
    if (htile >= tiles) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.kfree[rs]);
      htile = half;
      ++hseq;
    }
  }

  // Keeps w and u of a tile; false if the launch gives up.
  __device__ __forceinline__ bool keep(const float4& w, const float4& u) {
    while (held >= slots) {   // room comes from the oldest held chunk
      if (!head_wait()) return false;
      update_some();
    }
    if (wslot < wslots)
      ring[wslot * kThreads] = w;
    else
      tmem_st4(w_at(wslot), w);
    tmem_st4(u_at(wslot), u);
    ++held;
    if (++wslot == slots) wslot = 0;
    return true;
  }

  // The squares of a thread's elements of a tile.
  __device__ __forceinline__ void add_squares(const float (&w)[4],
                                              const float (&u)[4]) {
    float qw = 0.f, qu = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      qw = __fmaf_rn(w[c], w[c], qw);
      qu = __fmaf_rn(u[c], u[c], qu);
    }
    sum2_add(aw, qw);
    sum2_add(au, qu);
  }

  // The full tile of the pair in stage `st`; false if the launch gives up.
  __device__ __forceinline__ bool full_tile(const Rec& r, int tile,
                                            const char* st, uint64_t* freed) {
    const int at = 4 * (tile * kThreads + t);
    const uint32_t kind = r.kind;
    const float lam = r.lam;
    const int x = half * kThreads + t;   // float4 of the pair
    const float4 w4 = reinterpret_cast<const float4*>(st)[x];
    const float4 m4 = reinterpret_cast<const float4*>(st + kPairBytes)[x];
    const float4 v4 =
        kV ? reinterpret_cast<const float4*>(st + 2 * kPairBytes)[x]
           : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 g4 = grad4(
        reinterpret_cast<const GT*>(st + 3 * kPairBytes + skew(r.g)) + 4 * x);
    __syncwarp();
    if (lane == 0) mbar_arrive(freed);
    const float g[4] = {g4.x, g4.y, g4.z, g4.w};
    const float w[4] = {w4.x, w4.y, w4.z, w4.w};
    float m[4] = {m4.x, m4.y, m4.z, m4.w};
    float v[4] = {v4.x, v4.y, v4.z, v4.w};
    float u[4];
    if (kind != kStashReread) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (kOpt == kOptLars)
          m[c] = lars_momentum(g[c], m[c], w[c], lam, k.b1, k.omb1);
        else
          lamb_moments(g[c], m[c], v[c], k);
      }
      if (store) {
        st4(r.m + at, make_float4(m[0], m[1], m[2], m[3]));
        if (kV) st4(r.v + at, make_float4(v[0], v[1], v[2], v[3]));
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      u[c] = direction<kOpt>(m[c], v[c], g[c], w[c], lam, k);
    const float4 u4 = make_float4(u[0], u[1], u[2], u[3]);
    if (kind == kStashReread) {
      const float4 o = new_w(w4, u4, r.s, r.dd);
      st4_last(r.w + at, o);
      if (kCopy) st_copy4(r.copy, at, o);
      return true;
    }
    add_squares(w, u);
    return kind != kStashKeep || keep(w4, u4);
  }

  // The same for a tile that is not full (kVec) or of an unaligned chunk.  The
  // stage is read before anything is formed, and an unaligned chunk's offsets are
  // known while compiling: 362 / 349 us on a packed ragged list.
  template <bool kVec>
  __device__ __forceinline__ bool part_tile(const Rec& r, int tile,
                                            const char* st, uint64_t* freed) {
    const Span sp = tile_span(r, tile);
    Part q = tile_part(r, sp, t);
    if (!kVec) {   // known while compiling: the offsets go into the accesses
      q.at = t;
      q.step = kThreads;
    }
    const uint32_t kind = r.kind;
    const int pair = tile_span(r, tile & ~1).at;   // where the pair begins
    const int off = sp.at - pair;
    float* gw = r.w + sp.at;
    float* gm = r.m + sp.at;
    float* gv = kV ? r.v + sp.at : nullptr;
    const float* sw =
        reinterpret_cast<const float*>(st + skew(r.w + pair)) + off;
    const float* sm = reinterpret_cast<const float*>(
                          st + kPairBytes + skew(r.m + pair)) + off;
    const float* sv = reinterpret_cast<const float*>(
                          st + 2 * kPairBytes + skew(r.v + pair)) + off;
    const GT* sg = reinterpret_cast<const GT*>(
                       st + 3 * kPairBytes +
                       skew(static_cast<const GT*>(r.g) + pair)) + off;
    float g[4], m[4], v[4], w[4], u[4];   // zeros past the tile's end
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = q.at + c * q.step;
      const bool in = c < q.n;
      w[c] = in ? sw[i] : 0.f;
      m[c] = in ? sm[i] : 0.f;
      v[c] = kV && in ? sv[i] : 0.f;
      g[c] = in ? grad1(sg + i) : 0.f;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(freed);
    if (kind != kStashReread) {
      const int n_store = store ? q.n : 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (kOpt == kOptLars)
          m[c] = lars_momentum(g[c], m[c], w[c], r.lam, k.b1, k.omb1);
        else
          lamb_moments(g[c], m[c], v[c], k);
        if (c < n_store) {
          const int i = q.at + c * q.step;
          gm[i] = m[c];
          if (kV) gv[i] = v[c];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      u[c] = c < q.n ? direction<kOpt>(m[c], v[c], g[c], w[c], r.lam, k) : 0.f;
    add_squares(w, u);
    const float4 w4 = make_float4(w[0], w[1], w[2], w[3]);
    const float4 u4 = make_float4(u[0], u[1], u[2], u[3]);
    if (kind == kStashReread)
      store_new_w<kCopy>(gw, static_cast<__nv_bfloat16*>(r.copy) + sp.at, q,
                         new_w(w4, u4, r.s, r.dd));
    return kind != kStashKeep || keep(w4, u4);
  }

  // Waits for a barrier, updating what can be updated in the meantime.
  __device__ __forceinline__ bool wait_working(uint64_t* b, uint32_t parity) {
    while (!all_test(b, parity)) {
      if (head_ready())
        update_some();
      else if (warp_aborted(sh))
        return false;
      else
        __nanosleep(32);
    }
    return true;
  }

  // All the work; early if the launch gives up, with tiles still in the ring.
  __device__ __forceinline__ void run() {
    take_all();
    __syncwarp();
    tmem_wait_st();   // no store may outlive the allocation
  }

  __device__ __forceinline__ void take_all() {
    for (int seq = 0;; ++seq) {
      const int rs = seq % kStashRecs;
      const Rec& r = sh.rec[rs];
      if (!wait_working(&sh.full[rs], phase_of(seq))) return;
      const uint32_t kind = r.kind;
      if (kind == kStashEnd) break;
      const int tiles = r.tiles, full = full_tiles(r);
      for (int tile = half; tile - half < tiles; tile += 2) {
        const int st = count % kStages;
        uint64_t* freed = &sh.sfree[st];
        if (!wait_working(&sh.sfull[st], (uint32_t)(count / kStages) & 1u))
          return;
        const char* stage = smem + st * kStageBytes<GT>;
        if (tile >= tiles) {   // the last pair has no odd tile
          if (lane == 0) mbar_arrive(freed);
        } else if (!(tile < full ? full_tile(r, tile, stage, freed)
                     : r.vec     ? part_tile<true>(r, tile, stage, freed)
                                 : part_tile<false>(r, tile, stage, freed))) {
          return;
        }
        ++count;
        // as many tiles are updated as are formed, so that the writes of one
        // chunk mix with the reads of the next
        if ((tile & 2) && head_ready()) update_some();
      }
      if (kind != kStashReread) {
        // the lower lanes add w^2, the upper ones u^2
        const bool up = lane >= 16;
        Sum2 x = up ? au : aw;
        const Sum2 y = up ? aw : au;
        const Sum2 z{__shfl_xor_sync(kAllLanes, y.hi, 16),
                     __shfl_xor_sync(kAllLanes, y.lo, 16)};
        sum2_add(x, z);
        sum2_half_warps(x);
        if ((lane & 15) == 0) sh.red[rs][lane >> 4][threadIdx.x >> 5] = x;
      }
      if (kind == kStashKeep) ++kseq;
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sh.done[rs]);
        mbar_arrive(&sh.free[rs]);
      }
      aw = au = Sum2{0.f, 0.f};
    }
    while (hseq < kseq) {
      if (!head_wait()) return;
      update_some();
    }
  }
};

// ---------------------------------------------------------------------------
// Loader: lanes 0-3 copy w, m, v and g of a pair of tiles.
// ---------------------------------------------------------------------------
constexpr uint32_t kLoadLanes = 0xfu;

// wait_phase with one answer for the loader's lanes.
__device__ __forceinline__ bool load_wait(const Shared& sh, uint64_t* b,
                                          uint32_t parity) {
  return __all_sync(kLoadLanes, wait_phase(sh, b, parity));
}

template <int kOpt, typename GT>
__device__ __forceinline__ void load_chunks(Shared& sh, char* smem) {
  constexpr bool kG2 = kOpt == 1 || kOpt == 2;   // u holds g
  const int lane = threadIdx.x & 31;
  const int elem = lane == 3 ? (int)sizeof(GT) : 4;
  int count = 0;        // pairs
  int issued = 0;       // tiles
  bool go = true;
  for (int seq = 0; go; ++seq) {
    const int rs = seq % kStashRecs;
    if (!load_wait(sh, &sh.full[rs], phase_of(seq))) break;
    const Rec& r = sh.rec[rs];
    const uint32_t kind = r.kind;
    if (kind == kStashEnd) break;
    const bool again = kind == kStashReread;
    if (again) {   // other SMs' pass 1 wrote what is read now
      if (!load_wait(sh, &sh.ready[rs], phase_of(seq))) break;
      fence_proxy_async();
    }
    const int tiles = r.tiles;
    const char* base = static_cast<const char*>(
        lane == 0 ? (const void*)r.w : lane == 1 ? (const void*)r.m
        : lane == 2 ? (const void*)r.v : r.g);
    const bool copied = lane < 2 || (lane == 2 && kOpt != kOptLars) ||
                        (lane == 3 && (kG2 || !again));
    for (int pair = 0; 2 * pair < tiles; ++pair) {
      const int st = count % kStages;
      // whole 16-byte granules: the workers read at the remainder
      const Span sp = pair_span(r, pair);
      const char* from = base + (int64_t)sp.at * elem;
      const uint32_t off = skew(from);
      const uint32_t bytes =
          copied ? (off + (uint32_t)(sp.n * elem) + 15u) & ~15u : 0u;
      uint32_t sum = bytes + __shfl_xor_sync(kLoadLanes, bytes, 1);
      sum += __shfl_xor_sync(kLoadLanes, sum, 2);
      // a stage used before must have been read
      if (count >= kStages &&
          !load_wait(sh, &sh.sfree[st], (uint32_t)(count / kStages - 1) & 1u)) {
        go = false;
        break;
      }
      if (lane == 0) mbar_expect(&sh.sfull[st], sum);
      __syncwarp(kLoadLanes);
      if (copied)
        bulk_load(smem + st * kStageBytes<GT> + lane * kPairBytes, from - off,
                  bytes, &sh.sfull[st]);
      ++count;
      issued += min(2, tiles - 2 * pair);
      if (lane == 0) *reinterpret_cast<volatile int*>(&sh.issued) = issued;
    }
    __syncwarp(kLoadLanes);
    if (go && lane == 0) mbar_arrive(&sh.free[rs]);
  }
  // no copy may outlive the CTA, whatever ended the loop
  for (int i = max(0, count - kStages); i < count; ++i)
    for (int tries = 0; tries < (1 << 20); ++tries)
      if (mbar_try(&sh.sfull[i % kStages], (uint32_t)(i / kStages) & 1u))
        break;
}

// ---------------------------------------------------------------------------
// Drawer
// ---------------------------------------------------------------------------
__device__ __forceinline__ void draw(const StepParams& p, const StashParams& q,
                                     Shared& sh) {
  const int lane = threadIdx.x & 31;
  const bool decoupled = (p.flags & kFlagDecoupledDecay) != 0;
  int drawn = 0;                          // tiles
  int kseq = 0;                           // kept chunks drawn
  int kt = -1, kept = 0, keep_end = 0;    // newest kept tensor
  for (int seq = 0;; ++seq) {
    const int slot = seq % kStashRecs;
    if (seq >= kStashRecs &&
        !warp_wait(sh, &sh.free[slot], phase_of(seq - kStashRecs)))
      return;
    // Drawn only when all that was drawn before is on its way in: work that a
    // CTA holds while its ring is full delays its tensor for every other CTA
    // (BERT-large, drawing 0 / 2 / 6 tiles early: 1503 / 1570 / 1632 us).
    while (__any_sync(kAllLanes,
                      drawn - *reinterpret_cast<volatile int*>(&sh.issued) >
                          0)) {
      if (warp_aborted(sh)) return;
      __nanosleep(32);
    }
    // a CTA full of one tensor's chunks draws no more of them
    if (kept >= q.max_keep) {
      while (__any_sync(kAllLanes, (int)ld_relaxed_u32(q.bar + kStashCounter) <
                                       keep_end)) {
        if (warp_aborted(sh)) return;
        __nanosleep(100);
      }
    }
    uint32_t idx = 0;
    if (lane == 0) idx = atomicAdd(q.bar + kStashCounter, 1u);
    idx = __shfl_sync(0xffffffffu, idx, 0);
    if (idx >= (uint32_t)q.n_items) {
      if (lane == 0) {
        // every CTA draws one index past the end; the last of them resets
        if (idx == (uint32_t)q.n_items + gridDim.x - 1u)
          atomicExch(q.bar + kStashCounter, 0u);
        *reinterpret_cast<volatile int*>(&sh.end_seq) = seq;
        *reinterpret_cast<volatile int*>(&sh.end_kept) = kseq;
        sh.rec[slot].kind = kStashEnd;
        mbar_arrive(&sh.full[slot]);
      }
      return;
    }
    Rec& r = sh.rec[slot];
    if (lane < 4)
      reinterpret_cast<int4*>(static_cast<StashRec*>(&r))[lane] =
          __ldcg(reinterpret_cast<const int4*>(q.recs + idx) + lane);
    __syncwarp();
    const uint32_t bits = r.len_bits;
    const int len = (int)(bits & kStashLen), k = r.tensor;
    uint32_t kind = bits >> 30;
    if (sh.dry) {   // nothing is updated
      if (kind == kStashReread) {
        --seq;
        continue;
      }
      kind = kStashPlain;
    }
    const int n = chunk_tiles(len, (bits & kStashVec) != 0);
    const int ks = kseq % kStashRecs;
    if (kind == kStashKeep && kseq >= kStashRecs &&
        !warp_wait(sh, &sh.kfree[ks], phase_of(kseq - kStashRecs)))
      return;
    if (kind == kStashKeep) {
      ++kseq;
      kept = k == kt ? kept + 1 : 1;
      kt = k;
      keep_end = r.keep_end;
    }
    drawn += n;
    __syncwarp();
    if (lane == 0) {
      const float lamk = bits & kStashDecay ? p.wd : 0.f * p.wd;
      r.len = len;
      r.kind = kind;
      r.vec = bits & kStashVec;
      r.tiles = n;
      r.lam = decoupled ? 0.f : lamk;
      r.dd = decoupled
                 ? __double2float_rn((double)sh.lr * (double)lamk) : 0.f;
      if (kind == kStashKeep) {
        Kept& kp = sh.kept[ks];
        kp.w = r.w;
        kp.copy = r.copy;
        kp.len = len;
        kp.vec = r.vec;
        kp.tiles = n;
        kp.tensor = k;
        kp.dd = r.dd;
        mbar_arrive(&sh.kfull[ks]);
      }
      mbar_arrive(&sh.full[slot]);
    }
  }
}

// ---------------------------------------------------------------------------
// Closer
// ---------------------------------------------------------------------------
// Warp-wide sums of a tensor's chunk sums (of w^2 in lane 0, of u^2 in lane 16)
// in a fixed order, in fp64; two rounds of 16 loads per lane are in flight
// (BERT-base / BERT-large, us: 8 loads 519.6 / 1500, 16 loads 518.0 / 1491).  A
// half warp for each of the two: fp64 adds are slow, so no lane adds both, and
// none adds the zeros past the last chunk (a packed ragged list: 349 / 344 us).
__device__ __forceinline__ double combine(const double2* sums, int n) {
  constexpr int kLoads = 16;
  const int lane = threadIdx.x & 31;
  const double* from = &sums->x + (lane >> 4);
  double x[kLoads], y[kLoads];
  auto fetch = [&](double (&z)[kLoads], int base) {
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int at = base + 16 * i + (lane & 15);
      z[i] = at < n ? __ldcg(from + 2 * at) : 0.0;
    }
  };
  double a = 0.0;
  fetch(x, 0);
  for (int base = 0; base < n; base += 16 * kLoads) {
    fetch(y, base + 16 * kLoads);
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      if (base + 16 * i < n) a += x[i];
      x[i] = y[i];
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(kAllLanes, a, o);
  return a;
}

static_assert(kWorkers == 16, "half a warp adds the workers' sums");
__device__ __forceinline__ void close_chunks(const StepParams& p,
                                             const StashParams& q, Shared& sh,
                                             double coef) {
  const int lane = threadIdx.x & 31;
  for (int seq = 0;; ++seq) {
    const int slot = seq % kStashRecs;
    if (!warp_wait(sh, &sh.full[slot], phase_of(seq))) return;
    const uint32_t kind = sh.rec[slot].kind;
    if (kind == kStashEnd) return;
    if (!warp_wait(sh, &sh.done[slot], phase_of(seq))) return;
    const Rec& r = sh.rec[slot];
    const int k = r.tensor, c = r.chunk, first = r.first, n = r.n_chunks;
    const bool again = n > (int)gridDim.x * q.max_keep;
    Sum2 z = sh.red[slot][lane >> 4][lane & 15];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.free[slot]);
    if (kind == kStashReread) continue;
    sum2_half_warps(z);
    double sum = sum2_value(z);   // of w^2 in lane 0, of u^2 in lane 16
    if (n > 1) {
      const double u2 = __shfl_sync(kAllLanes, sum, 16);
      int last = 0;
      if (lane == 0) {
        // releases the slot and, through the workers' barrier, their m and v
        q.sums[c] = make_double2(sum, u2);
        last = atom_add_acq_rel(&p.tickets[k], 1u) + 1u == (uint32_t)n;
        if (last) p.tickets[k] = 0u;
      }
      if (!__shfl_sync(0xffffffffu, last, 0)) continue;
      sum = combine(q.sums + first, n);
    }
    const double root = sqrt(sum);   // both at once
    const double un = __shfl_sync(kAllLanes, root, 16);
    if (lane == 0) {
      const double wn = root;
      double rho = 1.0;                                // zero-norm rule
      if (!(wn == 0.0 || un == 0.0)) rho = coef * phi_of(wn, p) / un;
      const float s = __double2float_rn((double)sh.lr * rho);
      if (again) __threadfence();   // the tensor's other chunks are read
      st_relaxed_u64(q.words + k, (uint64_t)__float_as_uint(s) |
                                      ((uint64_t)(sh.epoch + 1u) << 32));
      p.ratio[k] = rho;
      p.wnorm[k] = wn;
      p.unorm[k] = un;
      if (!isfinite(wn) || !isfinite(un)) atomicOr(p.status, kStatusNonfinite);
    }
  }
}

// ---------------------------------------------------------------------------
// Poller: lane i hands out eta rho_k for the kept chunks' record i, lane
// kStashRecs + i for the drawn chunks' record i (chunks read again).
// ---------------------------------------------------------------------------
static_assert(2 * kStashRecs == 32, "one lane per record");

__device__ __forceinline__ void poll(const StepParams& p, const StashParams& q,
                                     Shared& sh) {
  const int lane = threadIdx.x & 31, slot = lane % kStashRecs;
  const bool kept = lane < kStashRecs;
  const uint32_t tag = sh.epoch + 1u + (uint32_t)q.extra_tag;
  uint64_t* full = kept ? &sh.kfull[slot] : &sh.full[slot];
  uint64_t* ready = kept ? &sh.kready[slot] : &sh.ready[slot];
  uint64_t* done = kept ? &sh.kfree[slot] : &sh.free[slot];
  float* s = kept ? &sh.kept[slot].s : &sh.rec[slot].s;
  const volatile int* end = kept ? &sh.end_kept : &sh.end_seq;
  bool active = true;
  int seq = slot;
  uint64_t since = 0;
  for (uint32_t turn = 0;; ++turn) {
    if (active) {
      if (seq >= *end) {
        active = false;
      } else if (mbar_test(full, phase_of(seq))) {
        const uint32_t kind = kept ? kStashReread : sh.rec[slot].kind;
        if (kind == kStashEnd) {
          active = false;
        } else {
          bool out = kind != kStashReread;   // nothing to hand out
          if (!out) {
            const int k = kept ? sh.kept[slot].tensor : sh.rec[slot].tensor;
            const uint64_t x = ld_relaxed_u64(q.words + k);
            if ((uint32_t)(x >> 32) == tag) {
              out = true;
              *s = __uint_as_float((uint32_t)x);
              // the workers will read what other SMs' pass 1 wrote
              if (!kept) __threadfence();
            }
          }
          if (out) {
            mbar_arrive(ready);
            mbar_arrive(done);
            seq += kStashRecs;
            since = 0;
          } else if (since == 0) {
            since = global_ns();
          } else if ((turn & 63u) == 0u &&
                     global_ns() - since > (uint64_t)q.wait_limit_ns) {
            atomicOr(p.status, kStatusWaitTimeout);
            atomicExch(q.bar + kStashAbort, 1u);
          }
        }
      }
    }
    if (!__any_sync(0xffffffffu, active)) return;
    if ((turn & 63u) == 63u) {
      const uint32_t gone = ld_acquire_u32(q.bar + kStashAbort);
      if (__any_sync(0xffffffffu, gone != 0u)) {
        if (lane == 0) *reinterpret_cast<volatile int*>(&sh.abort) = 1;
        return;
      }
    }
    __nanosleep(60);
  }
}

// ---------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------
template <int kOpt, typename GT, bool kCopy>
__global__ void __launch_bounds__(kStashThreads, 1)
    stash_step_kernel(const StepParams p, const StashParams q) {
  extern __shared__ float4 s_tiles[];   // stages, then the ring's w
  __shared__ Shared sh;
  constexpr bool kLars = kOpt == kOptLars;
  constexpr int kNest = kLars ? 0 : kOpt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (warp == kPoller && lane == 0) {
    sh.abort_word = ld_acquire_u32(q.bar + kStashAbort);
    sh.epoch = ld_acquire_u32(q.bar + kStashEpoch);
  }
  if (warp == kDrawer && lane == 0) {
    sh.lr = (p.flags & kFlagLrSchedule) ? 0.f : *p.d_lr;
    sh.abort = 0;
    sh.dry = (p.flags & kFlagSkipNonfinite) && p.gcheck->nonfinite;
    sh.issued = 0;
    sh.end_seq = sh.end_kept = 0x7fffffff;
  }
  if (warp == kCloser && lane < kStashRecs) {
    mbar_init(&sh.full[lane], 1);
    mbar_init(&sh.done[lane], kWorkers);
    mbar_init(&sh.ready[lane], 1);
    // read by the workers, the closer, the poller and the loader
    mbar_init(&sh.free[lane], kWorkers + 3);
    mbar_init(&sh.kfull[lane], 1);
    mbar_init(&sh.kready[lane], 1);
    mbar_init(&sh.kfree[lane], kWorkers + 1);   // the workers and the poller
  }
  if (warp == kLoader) {
    if (lane < kStages) {
      mbar_init(&sh.sfull[lane], 1);
      mbar_init(&sh.sfree[lane], kWorkers);
    }
    // the bulk copies count on barriers that were set up like this
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!kLars) {
    step_constants<kNest, false>(p, &sh.unused_draw, &sh.skip, &sh.k, &sh.t);
  } else if (threadIdx.x == 0) {
    const int64_t t = p.d_step ? *p.d_step : int64_t(0);
    sh.t = t;
    sh.skip = 0;
    sh.k = LambConsts{p.b1, p.omb1, p.b2, p.omb2, 1.f, 1.f, p.eps,
                      0.f, 0.f, 0.f, 0.f};
    if (blockIdx.x == 0) {
      StepScalars sc{};
      sc.t = t;
      sc.c1 = 1.f;
      sc.c2 = 1.f;
      sc.lr = step_lr(p, t);
      *p.scal = sc;
    }
  }
  __syncthreads();
  // a launch after one that gave up does nothing; a step count < 1 is skipped
  // (status set by CTA 0)
  if (sh.abort_word || sh.skip) return;
  if (threadIdx.x == 0 && (p.flags & kFlagLrSchedule)) sh.lr = step_lr(p, sh.t);
  if (warp == kCloser) {
    tmem_alloc_all(&sh.tmem);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (warp < kWorkers) {
    Worker<kOpt, GT, kCopy> work(p, q, sh, reinterpret_cast<char*>(s_tiles),
                                 sh.tmem);
    work.run();
  } else if (warp == kDrawer) {
    draw(p, q, sh);
  } else if (warp == kCloser) {
    close_chunks(p, q, sh, kLars ? p.trust : 1.0);
  } else if (warp == kPoller) {
    poll(p, q, sh);
  } else if (lane < 4) {
    load_chunks<kOpt, GT>(sh, reinterpret_cast<char*>(s_tiles));
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kCloser) tmem_free_all(sh.tmem);
  if (sh.abort) return;
  // the last CTA to finish advances the epoch and closes the step
  if (threadIdx.x == 0 &&
      atom_add_acq_rel(q.bar + kStashTicket, 1u) == gridDim.x - 1u) {
    st_relaxed_u32(q.bar + kStashTicket, 0u);
    st_relaxed_u32(q.bar + kStashEpoch, sh.epoch + 1u);
    if (!sh.dry) {
      const StepScalars sc = *p.scal;
      if (kNest && p.d_mu_product) *p.d_mu_product = sc.mu_prod;
      close_step(p, sc);
    }
  }
}

// ---------------------------------------------------------------------------
// Gradient check before the step: reads g alone (2 or 4 B per parameter), so
// that the step's decision is known before anything is written and the step can
// run as one launch: 30 B per parameter with bf16 g and copy, where the two
// kernels' skip mode moves 42 (BERT-large: 2096 us).  One warp per chunk; a lane
// keeps 10 loads of 16 bytes in flight and adds in 8 accumulators (40 elements
// each): 117 us of BERT-large's 1630, 5.7 TB/s.  The tensor's last
// warp forms ||g_k||, the last tensor's the global norm and the decision, both
// in a fixed order.
// ---------------------------------------------------------------------------
constexpr int kCheckLoads = 10;

// 16 or 8 bytes of gradients, widened: n of them.
__device__ __forceinline__ void widen(const float4& x, float (&g)[4]) {
  g[0] = x.x;
  g[1] = x.y;
  g[2] = x.z;
  g[3] = x.w;
}
__device__ __forceinline__ void widen(const uint2& x, float (&g)[4]) {
  g[0] = __uint_as_float(x.x << 16);
  g[1] = __uint_as_float(x.x & 0xffff0000u);
  g[2] = __uint_as_float(x.y << 16);
  g[3] = __uint_as_float(x.y & 0xffff0000u);
}
__device__ __forceinline__ void widen(const uint4& x, float (&g)[8]) {
  float a[4], b[4];
  widen(make_uint2(x.x, x.y), a);
  widen(make_uint2(x.z, x.w), b);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g[i] = a[i];
    g[4 + i] = b[i];
  }
}

// Adds the squares of n loads of type V at p, kN gradients each.
template <typename V, int kN>
__device__ __forceinline__ void check_run(const void* p, int n, float (&a)[8],
                                          float& z) {
  const V* v = static_cast<const V*>(p);
  for (int base = (int)(threadIdx.x & 31); base < n;
       base += 32 * kCheckLoads) {
    V x[kCheckLoads];
#pragma unroll
    for (int i = 0; i < kCheckLoads; ++i) {
      x[i] = V{};
      if (base + 32 * i < n) x[i] = __ldcs(v + base + 32 * i);
    }
#pragma unroll
    for (int i = 0; i < kCheckLoads; ++i) {
      float g[kN];
      widen(x[i], g);
#pragma unroll
      for (int e = 0; e < kN; ++e) {
        float& b = a[kN == 8 ? e : 4 * (i & 1) + e];
        b = __fmaf_rn(g[e], g[e], b);
        z = __fmaf_rn(g[e], 0.f, z);
      }
    }
  }
}
// Returns how many elements it took.
__device__ __forceinline__ int check_vec(const float* g, int len,
                                         float (&a)[8], float& z) {
  check_run<float4, 4>(g, len >> 2, a, z);
  return len & ~3;
}
__device__ __forceinline__ int check_vec(const __nv_bfloat16* g, int len,
                                         float (&a)[8], float& z) {
  if ((uintptr_t)g % 16 == 0) {
    check_run<uint4, 8>(g, len >> 3, a, z);
    return len & ~7;
  }
  check_run<uint2, 4>(g, len >> 2, a, z);
  return len & ~3;
}

// Warp-wide sums of a tensor's slots in a fixed order, in fp64 as in the
// two-pass finaliser; two rounds of eight slots per lane are in flight.  (With
// `combine` above in its place the kernel gets fewer registers, and with fp32 g
// it waits for its loads one by one: 31 / 48 us on 6M parameters.)
__device__ __forceinline__ void combine_slots(const float2* slots, int n,
                                              double* sum, double* nan) {
  constexpr int kLoads = 8;
  const int lane = threadIdx.x & 31;
  float2 x[kLoads], y[kLoads];
  auto fetch = [&](float2 (&z)[kLoads], int base) {
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int at = base + 32 * i + lane;
      z[i] = at < n ? __ldcg(slots + at) : make_float2(0.f, 0.f);
    }
  };
  double a = 0.0, b = 0.0;
  fetch(x, 0);
  for (int base = 0; base < n; base += 32 * kLoads) {
    fetch(y, base + 32 * kLoads);
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      a += (double)x[i].x;
      b += (double)x[i].y;
      x[i] = y[i];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(kAllLanes, a, o);
    b += __shfl_xor_sync(kAllLanes, b, o);
  }
  *sum = a;
  *nan = b;
}

template <typename GT>
__global__ void __launch_bounds__(kThreads)
    grad_check_kernel(const StepParams p, int needs_t) {
  const int lane = threadIdx.x & 31;
  // a step that is skipped for its step count checks nothing
  if (needs_t && *p.d_step < 1) return;
  const int n_warps = (int)gridDim.x * kWarps;
  for (int c = (int)blockIdx.x * kWarps + (int)(threadIdx.x >> 5);
       c < p.n_chunks; c += n_warps) {
    const ChunkDesc ch = p.chunks[c];
    const TensorDesc td = p.tensors[ch.tensor];
    const TensorPtrs tp = p.ptrs[ch.tensor];
    const GT* g = static_cast<const GT*>(tp.g) + ch.offset;
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, z = 0.f;
    const int from = tp.vec_ok ? check_vec(g, ch.len, a, z) : 0;
    for (int base = from + lane; base < ch.len; base += 32 * 8) {
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        x[i] = base + 32 * i < ch.len ? ld_grad1(g + base + 32 * i) : 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        a[i] = __fmaf_rn(x[i], x[i], a[i]);
        z = __fmaf_rn(x[i], 0.f, z);
      }
    }
    const float s = warp_sum(((a[0] + a[1]) + (a[2] + a[3])) +
                             ((a[4] + a[5]) + (a[6] + a[7])));
    z = warp_sum(z);
    int last = 0;
    if (lane == 0) {
      p.grad_slots[c] = make_float2(s, z);
      last = atom_add_acq_rel(&p.tickets[ch.tensor], 1u) + 1u ==
             (uint32_t)td.n_chunks;
      if (last) p.tickets[ch.tensor] = 0u;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) continue;
    double sum, nan;
    combine_slots(p.grad_slots + td.first_chunk, td.n_chunks, &sum, &nan);
    int last_tensor = 0;
    if (lane == 0) {
      p.gsq[ch.tensor] = sum;
      p.gnorm[ch.tensor] = sqrt(sum);
      if (isnan(nan)) atomicOr(&p.gcheck->acc, 1u);
      __threadfence();
      last_tensor =
          atomicAdd(&p.gcheck->done, 1u) + 1u == (uint32_t)p.n_live;
    }
    if (__shfl_sync(0xffffffffu, last_tensor, 0)) finalize_grad(p);
  }
}

__global__ void __launch_bounds__(256)
    stash_records_kernel(const StashItem* items, const ChunkDesc* chunks,
                         const TensorDesc* tensors, const TensorPtrs* ptrs,
                         int grad_size, StashRec* recs, int n) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  const StashItem it = items[i];
  const int c = (int)(it.chunk & 0x3fffffffu);
  const ChunkDesc ch = chunks[c];
  const TensorDesc td = tensors[ch.tensor];
  const TensorPtrs tp = ptrs[ch.tensor];
  StashRec r;
  r.w = tp.w + ch.offset;
  r.g = static_cast<const char*>(tp.g) + ch.offset * grad_size;
  r.m = tp.m + ch.offset;
  r.v = tp.v ? tp.v + ch.offset : nullptr;
  r.copy = tp.copy ? static_cast<__nv_bfloat16*>(tp.copy) + ch.offset : nullptr;
  r.len_bits = (uint32_t)ch.len | (tp.vec_ok ? kStashVec : 0u) |
               (td.decay != 0.f ? kStashDecay : 0u) | (it.chunk & 0xc0000000u);
  r.tensor = ch.tensor;
  r.chunk = c;
  r.first = td.first_chunk;
  r.n_chunks = td.n_chunks;
  r.keep_end = it.keep_end;
  recs[i] = r;
}

template <int kOpt, typename GT, bool kCopy>
int launch_one(const StepParams& p, const StashParams& q, int grid,
               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kStashThreads);
  cfg.dynamicSmemBytes = (size_t)(kStages * kStageBytes<GT> +
                                  2 * q.wslots * kThreads * 16);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, stash_step_kernel<kOpt, GT, kCopy>, p,
                                 q);
}

// f(kernel) for every instantiation, until one returns non-zero.
template <int kOpt, typename F>
int each_type(const F& f) {
  int rc = f(stash_step_kernel<kOpt, float, false>);
  if (!rc) rc = f(stash_step_kernel<kOpt, float, true>);
  if (!rc) rc = f(stash_step_kernel<kOpt, __nv_bfloat16, false>);
  if (!rc) rc = f(stash_step_kernel<kOpt, __nv_bfloat16, true>);
  return rc;
}
template <typename F>
int each_kernel(const F& f) {
  int rc = each_type<0>(f);
  if (!rc) rc = each_type<1>(f);
  if (!rc) rc = each_type<2>(f);
  if (!rc) rc = each_type<3>(f);
  return rc;
}

template <int kOpt>
int launch_opt(const StepParams& p, const StashParams& q, int g_bf16, int copy,
               int grid, cudaStream_t s) {
  if (g_bf16)
    return copy ? launch_one<kOpt, __nv_bfloat16, true>(p, q, grid, s)
                : launch_one<kOpt, __nv_bfloat16, false>(p, q, grid, s);
  return copy ? launch_one<kOpt, float, true>(p, q, grid, s)
              : launch_one<kOpt, float, false>(p, q, grid, s);
}

}  // namespace

int stash_prepare(int device, int grad_bf16, int* slots, int* wslots) {
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(
      &optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return (int)e;
  int stat = 0;
  int rc = each_kernel([&](auto* f) {
    cudaFuncAttributes a;
    const cudaError_t x = cudaFuncGetAttributes(&a, f);
    if (x == cudaSuccess && (int)a.sharedSizeBytes > stat)
      stat = (int)a.sharedSizeBytes;
    return (int)x;
  });
  if (rc) return rc;
  const int dyn = (optin - stat) & ~15;
  rc = each_kernel([&](auto* f) {
    return (int)cudaFuncSetAttribute(
        f, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
  });
  if (rc) return rc;
  const int stages = kStages * (grad_bf16 ? kStageBytes<__nv_bfloat16>
                                          : kStageBytes<float>);
  // per half of the tiles: a slot's u takes one of the thread's places in
  // tensor memory, its w another one or, for the first slots, shared memory
  int w = (dyn - stages) / (2 * kThreads * 16);
  int n = (kTmemSlots + w) / 2;
  if (n > kTmemSlots) n = kTmemSlots;
  w = 2 * n - kTmemSlots;
  if (w < 0) return (int)cudaErrorInvalidConfiguration;
  int blocks = 0;   // the launch needs one resident CTA per SM
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &blocks, stash_step_kernel<0, __nv_bfloat16, true>, kStashThreads,
      (size_t)dyn);
  if (e != cudaSuccess) return (int)e;
  if (blocks < 1) return (int)cudaErrorInvalidConfiguration;
  *slots = n;
  *wslots = w;
  return 0;
}

int launch_stash_records(const StashItem* items, const ChunkDesc* chunks,
                         const TensorDesc* tensors, const TensorPtrs* ptrs,
                         int grad_bf16, StashRec* recs, int n_items,
                         void* stream) {
  if (n_items < 1) return 0;
  stash_records_kernel<<<(n_items + 255) / 256, 256, 0,
                         static_cast<cudaStream_t>(stream)>>>(
      items, chunks, tensors, ptrs, grad_bf16 ? 2 : 4, recs, n_items);
  return (int)cudaGetLastError();
}

int launch_grad_check(const StepParams& p, int opt, int grad_bf16, int num_sms,
                      void* stream) {
  const int needs_t =
      opt == 1 || opt == 2 ||
      (opt == 0 && (p.flags & kFlagBiasCorrection)) ? 1 : 0;
  // more CTAs than are resident: a warp's chunk is short, and the scheduler
  // evens them out (BERT-large: 5 per SM 142 us, 8 127, 16 and more 120)
  const int64_t want = ((int64_t)p.n_chunks + kWarps - 1) / kWarps;
  const int64_t most = (int64_t)num_sms * 16;
  const unsigned grid = (unsigned)(want < 1 ? 1 : want < most ? want : most);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (grad_bf16)
    grad_check_kernel<__nv_bfloat16><<<grid, kThreads, 0, s>>>(p, needs_t);
  else
    grad_check_kernel<float><<<grid, kThreads, 0, s>>>(p, needs_t);
  return (int)cudaGetLastError();
}

int launch_stash(const StepParams& p, const StashParams& q, int opt,
                 int grad_bf16, int copy_bf16, int grid, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (opt) {
    case 0: return launch_opt<0>(p, q, grad_bf16, copy_bf16, grid, s);
    case 1: return launch_opt<1>(p, q, grad_bf16, copy_bf16, grid, s);
    case 2: return launch_opt<2>(p, q, grad_bf16, copy_bf16, grid, s);
    default: return launch_opt<3>(p, q, grad_bf16, copy_bf16, grid, s);
  }
}

}  // namespace lamb
