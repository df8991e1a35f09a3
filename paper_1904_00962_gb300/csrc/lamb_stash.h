// Tables and launcher of the one-launch form of the two-pass step
// (lamb_stash.cu).
//
// HBM layout added to a plan that uses it (same arena, each piece 256-byte
// aligned):
//   ChunkDesc  chunks[n_chunks]     16 B  its own chunk table
//   TensorDesc tensors[n_tensors]   32 B  and tensor table
//   double2    sums[n_chunks]       16 B  per chunk (sum w^2, sum u^2)
//   float2     gsums[n_chunks]       8 B  per chunk (sum g^2, sum 0*g)
//   StashItem  items[n_items]        8 B  the work, in the order it is drawn
//   StashRec   recs[n_items]        64 B  the same with all that a CTA needs
//                                         to know of a chunk, made by bind
//   uint64     words[n_tensors]      8 B  per tensor: eta rho_k, tagged with
//                                         the launch that wrote it
//   uint32     bar[kStashBarWords]        launch epoch, finish ticket, abort
//                                         word, work counter
#pragma once
#include <stdint.h>

#include <vector>

#include "lamb_internal.h"

namespace lamb {

constexpr int kStashTile = 4 * kThreads;   // elements: one float4 per thread
// Elements per chunk.  A chunk is kept until its tensor's last one is done, so
// short chunks need less room (of a 4096 x 1024 tensor an SM holds 27 tiles, and
// what it forms while the last chunk is summed), and more of a tensor larger than
// the SMs is kept; but each takes a draw, a tree of sums and a ticket.  us per
// step, a two-layer encoder / BERT-base / BERT-large / 4,000 ragged tensors: 8,192
// elements 67.9 / 538 / 1524 / 4695, 10,240 67.4 / 518 / 1493 / 4590, 12,288 69.1 /
// 511 / 1479 / 4566, 16,384 64.6 / 506 / 1524 / 4600.  12,288 would keep 5.6M
// parameters of a tensor in place of 6.2M, and the lines of AUTO's rules were
// measured at 10,240.  Workers take tiles in pairs: the number is even.
constexpr int kStashChunk = 10 * kStashTile;
constexpr int kStashRecs = 16;   // chunks a CTA has drawn and not finished

// What is done with a chunk.
enum : uint32_t {
  kStashKeep = 0u,     // pass 1; w and u stay on the SM for the update
  kStashPlain = 1u,    // pass 1 only (a tensor larger than the grid holds)
  kStashReread = 2u,   // pass 2 of a kStashPlain chunk, from HBM
  kStashEnd = 3u };    // no more work

struct __align__(8) StashItem {
  uint32_t chunk;      // chunk index, kind in the two top bits
  int32_t keep_end;    // items up to here hold every kept chunk of the tensor
};

struct __align__(16) StashRec {
  float* w;             // at the chunk's first element
  const void* g;
  float* m;
  float* v;
  void* copy;
  uint32_t len_bits;    // elements (at most 2^24), kStashVec, kStashDecay, kind
                        // in the two top bits
  int32_t tensor;
  int32_t chunk;
  int32_t first, n_chunks;   // of the tensor
  int32_t keep_end;
};
static_assert(sizeof(StashRec) == 64, "StashRec layout");
constexpr uint32_t kStashVec = 1u << 28;     // float4 accesses
constexpr uint32_t kStashDecay = 1u << 29;   // weight decay applies
constexpr uint32_t kStashLen = (1u << 28) - 1u;

// Words of the launch block (uint32 indices; each on its own 128-byte line)
constexpr int kStashEpoch = 0;     // launches that finished
constexpr int kStashTicket = 32;   // CTAs of the current launch that finished
constexpr int kStashAbort = 64;    // a wait gave up: the plan is unusable
constexpr int kStashCounter = 96;  // items drawn by the current launch
constexpr int kStashBarWords = 128;

struct StashParams {
  const StashRec* recs;
  double2* sums;
  uint64_t* words;
  uint32_t* bar;
  int32_t n_items;
  int32_t slots;          // tiles of either half (even, odd) a CTA can keep
  int32_t wslots;         // those of them whose w is in shared memory
  int32_t max_keep;       // kept chunks of one tensor per CTA, at most
  int32_t extra_tag;      // > 0 only in tests of the give-up path
  int64_t wait_limit_ns;
};

// Kept chunks of one tensor that a CTA with room for `slots` tiles of either
// half can always hold (planner.cpp): 0 if not even one fits.
int32_t stash_max_keep(int32_t slots);
// The work list of the chunk table `tensors`: every tensor's chunks in order.
// Of a tensor with more than grid * max_keep chunks the first that many are kept
// and the rest is read again, last chunk first, `grid` chunks later, when the
// ratio is likely there.
void plan_stash(const TensorDesc* tensors, int32_t n, int32_t grid,
                int32_t max_keep, std::vector<StashItem>* items);

// Fills recs from the items and the plan's tables, on `stream`.
int launch_stash_records(const StashItem* items, const ChunkDesc* chunks,
                         const TensorDesc* tensors, const TensorPtrs* ptrs,
                         int grad_bf16, StashRec* recs, int n_items,
                         void* stream);
// The gradient check over the chunk table p.chunks, into p.grad_slots and the
// results it leads to; read by the step launched next.  opt as below.
int launch_grad_check(const StepParams& p, int opt, int grad_bf16, int num_sms,
                      void* stream);
// Launcher: opt 0 LAMB, 1 N-LAMB, 2 NN-LAMB, 3 LARS.
int launch_stash(const StepParams& p, const StashParams& q, int opt,
                 int grad_bf16, int copy_bf16, int grid, void* stream);
// StashParams.slots and wslots on `device`, after the kernels' static shared
// memory and the stages; also raises the kernels' dynamic shared-memory limit.
int stash_prepare(int device, int grad_bf16, int* slots, int* wslots);

}  // namespace lamb
