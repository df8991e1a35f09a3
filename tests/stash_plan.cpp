// Harness of the work list of the one-launch two-pass step (test
// infrastructure, built by tests/test_stash_plan.py with sanitizers): random
// layouts through plan_chunks and plan_stash.  Checks the list against the rule
// its declaration states, then runs it through a model of the kernel's CTAs --
// what they draw, hold and wait for, in random turns -- and checks that it ends
// whatever the turns.  Exit status 0: every layout passed.
#include <cstdio>
#include <cstdlib>
#include <deque>
#include <vector>

#include "lamb_internal.h"
#include "lamb_stash.h"

using namespace lamb;

namespace {

uint64_t g_state = 0x9E3779B97F4A7C15ull;
int64_t below(int64_t n) {   // splitmix64
  uint64_t z = (g_state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (int64_t)((z ^ (z >> 31)) % (uint64_t)n);
}

#define CHECK(x)                                                        \
  do {                                                                  \
    if (!(x)) {                                                         \
      std::fprintf(stderr, "%s:%d: %s\n", __FILE__, __LINE__, #x);      \
      return false;                                                     \
    }                                                                   \
  } while (0)

int tiles_of(int len) {   // of an aligned chunk
  return (len / 4 + kThreads - 1) / kThreads + (len % 4 ? 1 : 0);
}

struct Cta {
  std::deque<int> drawn;            // item indices not begun
  std::deque<std::pair<int, int>> held;   // tensor, tiles
  int tensor = -1, kept = 0, keep_end = 0;
  bool done = false;
};

bool run(const std::vector<int64_t>& sizes, int grid, int slots) {
  const int n = (int)sizes.size();
  const int max_keep = stash_max_keep(slots);
  std::vector<TensorDesc> td((size_t)n);
  char err[256];
  int64_t count = 0;
  CHECK(plan_chunks(sizes.data(), n, kStashChunk, nullptr, 0, &count,
                    td.data(), nullptr, err, sizeof err) == 0);
  std::vector<ChunkDesc> chunks((size_t)count);
  CHECK(count == 0 ||
        plan_chunks(sizes.data(), n, kStashChunk, chunks.data(), count, &count,
                    td.data(), nullptr, err, sizeof err) == 0);
  std::vector<StashItem> items;
  plan_stash(td.data(), n, grid, max_keep, &items);

  // every chunk once, in order; what is not kept once more, after its tensor
  int64_t next = 0;
  std::vector<int> keep((size_t)n, 0), last_keep((size_t)n, -1);
  std::vector<int> seen((size_t)n, 0), plain((size_t)count, 0);
  for (size_t i = 0; i < items.size(); ++i) {
    const uint32_t c = items[i].chunk & 0x3fffffffu, kind = items[i].chunk >> 30;
    CHECK((int64_t)c < count && kind <= kStashReread);
    const int k = chunks[c].tensor;
    if (kind == kStashReread) {
      CHECK(seen[(size_t)k] == td[(size_t)k].n_chunks && plain[c] == 1);
      plain[c] = 2;
      continue;
    }
    CHECK((int64_t)c == next++);
    ++seen[(size_t)k];
    if (kind == kStashKeep) {
      ++keep[(size_t)k];
      last_keep[(size_t)k] = (int)i;
    } else {
      plain[c] = 1;
    }
  }
  CHECK(next == count);
  for (int64_t c = 0; c < count; ++c) CHECK(plain[(size_t)c] != 1);
  for (size_t i = 0; i < items.size(); ++i)
    if (items[i].chunk >> 30 == kStashKeep) {
      const int k = chunks[items[i].chunk & 0x3fffffffu].tensor;
      CHECK(items[i].keep_end == last_keep[(size_t)k] + 1);
      CHECK(keep[(size_t)k] <= grid * max_keep);
    }

  // the kernel's CTAs, a random one at a time; `idle` turns without progress
  std::vector<Cta> cta((size_t)grid);
  std::vector<int> formed((size_t)n, 0);
  size_t counter = 0;
  int left = grid;
  auto ready = [&](int k) {
    return formed[(size_t)k] == td[(size_t)k].n_chunks;
  };
  while (left > 0) {
    bool progress = false;
    const int at = (int)below(grid);
    for (int j = 0; j < grid && !progress; ++j) {
      Cta& c = cta[(size_t)((at + j) % grid)];
      if (c.done) continue;
      int room = 2 * slots;
      for (auto& h : c.held) room -= h.second;
      if (!c.held.empty() && ready(c.held.front().first) && below(2)) {
        c.held.pop_front();
        progress = true;
        continue;
      }
      // one item in work, one drawn ahead
      if (c.drawn.size() < 2 &&
          !(c.kept >= max_keep && (int)counter < c.keep_end)) {
        if (counter >= items.size()) {
          if (c.drawn.empty() && c.held.empty()) {
            c.done = true;
            --left;
            progress = true;
            continue;
          }
        } else {
          const int i = (int)counter++;
          c.drawn.push_back(i);
          progress = true;
          if (items[(size_t)i].chunk >> 30 == kStashKeep) {
            const int k = chunks[items[(size_t)i].chunk & 0x3fffffffu].tensor;
            c.kept = k == c.tensor ? c.kept + 1 : 1;
            c.tensor = k;
            c.keep_end = items[(size_t)i].keep_end;
          }
          continue;
        }
      }
      if (!c.drawn.empty()) {
        const StashItem it = items[(size_t)c.drawn.front()];
        const ChunkDesc& ch = chunks[it.chunk & 0x3fffffffu];
        const uint32_t kind = it.chunk >> 30;
        if (kind == kStashReread) {
          if (ready(ch.tensor)) {
            c.drawn.pop_front();
            progress = true;
          }
        } else {
          // a half takes a tile more than the other of an odd number
          const int need = (tiles_of(ch.len) + 1) / 2 * 2;
          if (kind == kStashPlain || need <= room) {
            c.drawn.pop_front();
            ++formed[(size_t)ch.tensor];
            if (kind == kStashKeep) c.held.push_back({ch.tensor, need});
            progress = true;
          } else {
            CHECK(!c.held.empty());
          }
        }
        if (progress) continue;
      }
      if (!c.held.empty() && ready(c.held.front().first)) {
        c.held.pop_front();
        progress = true;
      }
    }
    CHECK(progress);
  }
  return true;
}

}  // namespace

int main(int argc, char** argv) {
  const int layouts = argc > 1 ? std::atoi(argv[1]) : 500;
  for (int i = 0; i < layouts; ++i) {
    const int grid = 1 + (int)below(8);
    const int slots = 6 + (int)below(27);
    std::vector<int64_t> sizes((size_t)(1 + below(12)));
    for (auto& s : sizes)
      s = below(4) == 0 ? below(5) :
          below(3) == 0 ? (1 + below(60)) * kStashChunk + below(7) - 3
                        : below(200000);
    if (!run(sizes, grid, slots)) return 1;
  }
  std::printf("%d layouts\n", layouts);
  return 0;
}
