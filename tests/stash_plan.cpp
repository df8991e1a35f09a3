// Harness of the work list of the one-launch two-pass step (test
// infrastructure, built by tests/test_stash_plan.py with sanitizers): random
// layouts through plan_chunks and plan_stash.  Checks the list against the rule
// its declaration states, then runs it through a model of the kernel's CTAs --
// the records, stages and ring places that each warp role takes and what it
// waits for, in random turns -- and checks that it ends whatever the turns.
// Exit status 0: every layout passed.
#include <cstdio>
#include <cstdlib>
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

// A chunk that a CTA has drawn.
struct Rec {
  uint32_t kind;
  int tensor, tiles;
  int kept = -1;            // its number among the CTA's kept chunks
  bool done[2] = {false, false};   // formed (or read again) by a half's workers
};

// What limits a CTA: the records of drawn and of kept chunks, the stages, and a
// ring of tiles for each half of the workers (even and odd tiles).
struct Half {
  int seq = 0, tile = 0;    // next tile of the record `seq`
  int pairs = 0;            // stages read
  bool to_keep = false;     // a tile has been read and waits for room
  int held = 0;             // tiles in the ring
  int kseq = 0;             // kept chunks formed
  int hseq = 0, htile = 0;  // oldest of them not updated, tiles of it updated
  bool ended = false;
};

struct Cta {
  std::vector<Rec> recs;            // published
  std::vector<int> kept;            // records of the kept chunks
  // drawer
  int drawn_tiles = 0;
  int tensor = -1, n_kept = 0, keep_end = 0;
  int held_item = -1;               // drawn, waits for a kept record
  bool last = false;                // has drawn past the end
  // loader
  int load_rec = 0, load_pair = 0, pairs = 0, issued_tiles = 0;
  Half half[2];
};

// tiles of a chunk that a half takes
int half_tiles(int tiles, int h) { return (tiles - h + 1) / 2; }

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

  // the kernel's CTAs: drawer, loader and the two halves of the workers, one of
  // them at a time in random order.  (A chunk is closed as soon as both halves
  // are done: the closer waits for nothing else.)
  const int stages = 1 + (int)below(3);
  std::vector<Cta> cta((size_t)grid);
  std::vector<int> formed((size_t)n, 0);
  size_t counter = 0;
  auto ready = [&](int k) {
    return formed[(size_t)k] == td[(size_t)k].n_chunks;
  };
  auto publish = [&](Cta& c, const StashItem& it) {
    const ChunkDesc& ch = chunks[it.chunk & 0x3fffffffu];
    Rec r;
    r.kind = it.chunk >> 30;
    r.tensor = ch.tensor;
    r.tiles = tiles_of(ch.len);
    if (r.kind == kStashKeep) {
      r.kept = (int)c.kept.size();
      c.kept.push_back((int)c.recs.size());
    }
    c.drawn_tiles += r.tiles;
    c.recs.push_back(r);
  };
  auto kept_free = [&](const Cta& c) {   // the record that the next one takes
    const int old = (int)c.kept.size() - kStashRecs;
    return old < 0 || (c.half[0].hseq > old && c.half[1].hseq > old);
  };
  auto drawer = [&](Cta& c) {
    if (c.held_item >= 0) {
      if (!kept_free(c)) return false;
      publish(c, items[(size_t)c.held_item]);
      c.held_item = -1;
      return true;
    }
    if (c.last) return false;
    const int old = (int)c.recs.size() - kStashRecs;
    if (old >= 0 && !(c.recs[(size_t)old].done[0] &&
                      c.recs[(size_t)old].done[1]))
      return false;
    if (c.drawn_tiles > c.issued_tiles) return false;
    if (c.n_kept >= max_keep && (int)counter < c.keep_end) return false;
    if (counter >= items.size()) return c.last = true;
    const int i = (int)counter++;
    if (items[(size_t)i].chunk >> 30 == kStashKeep) {
      const int k = chunks[items[(size_t)i].chunk & 0x3fffffffu].tensor;
      c.n_kept = k == c.tensor ? c.n_kept + 1 : 1;
      c.tensor = k;
      c.keep_end = items[(size_t)i].keep_end;
      if (!kept_free(c)) {
        c.held_item = i;
        return true;
      }
    }
    publish(c, items[(size_t)i]);
    return true;
  };
  auto loader = [&](Cta& c) {
    if (c.load_rec >= (int)c.recs.size()) return false;
    const Rec& r = c.recs[(size_t)c.load_rec];
    if (r.kind == kStashReread && !ready(r.tensor)) return false;
    const int read = c.half[0].pairs < c.half[1].pairs ? c.half[0].pairs
                                                       : c.half[1].pairs;
    if (c.pairs - read >= stages) return false;
    ++c.pairs;
    c.issued_tiles += r.tiles - 2 * c.load_pair < 2 ? 1 : 2;
    if (2 * ++c.load_pair >= r.tiles) {
      c.load_pair = 0;
      ++c.load_rec;
    }
    return true;
  };
  // up to two tiles of the oldest kept chunk, if its ratio is there
  auto update = [&](Cta& c, int h) {
    Half& w = c.half[h];
    const Rec& r = c.recs[(size_t)c.kept[(size_t)w.hseq]];
    if (!ready(r.tensor)) return false;
    const int left = half_tiles(r.tiles, h) - w.htile;
    const int now = left < 2 ? left : 2;
    w.htile += now;
    w.held -= now;
    if (w.htile == half_tiles(r.tiles, h)) {
      w.htile = 0;
      ++w.hseq;
    }
    return true;
  };
  bool broken = false;   // a wait for the chunk that is being formed
  auto worker = [&](Cta& c, int h) {
    Half& w = c.half[h];
    if (w.to_keep) {
      if (w.held >= slots) {
        if (w.hseq >= w.kseq) return broken = true;
        return update(c, h);
      }
      ++w.held;
      w.to_keep = false;
      return true;
    }
    if (w.hseq < w.kseq && below(2) && update(c, h)) return true;
    if (w.seq >= (int)c.recs.size()) {
      if (w.hseq < w.kseq) return update(c, h);
      if (c.last && c.held_item < 0 && !w.ended) return w.ended = true;
      return false;
    }
    Rec& r = c.recs[(size_t)w.seq];
    if (2 * w.tile < r.tiles) {      // a pair of tiles; the odd one may be none
      if (w.pairs >= c.pairs)
        return w.hseq < w.kseq && update(c, h);
      ++w.pairs;
      w.to_keep = r.kind == kStashKeep && w.tile < half_tiles(r.tiles, h);
      ++w.tile;
      return true;
    }
    if (r.kind == kStashKeep) ++w.kseq;
    r.done[h] = true;
    if (r.kind != kStashReread && r.done[1 - h]) ++formed[(size_t)r.tensor];
    w.tile = 0;
    ++w.seq;
    return true;
  };
  for (;;) {
    bool progress = false, all = true;
    const int at = (int)below(4 * grid);
    for (int j = 0; j < 4 * grid && !progress; ++j) {
      const int a = (at + j) % (4 * grid);
      Cta& c = cta[(size_t)(a / 4)];
      progress = a % 4 == 0 ? drawer(c)
                 : a % 4 == 1 ? loader(c) : worker(c, a % 4 - 2);
      CHECK(!broken);
    }
    for (const Cta& c : cta) all = all && c.half[0].ended && c.half[1].ended;
    if (all) break;
    CHECK(progress);
  }
  CHECK(counter == items.size());
  for (int k = 0; k < n; ++k) CHECK(ready(k));
  for (const Cta& c : cta)
    for (const Half& w : c.half) CHECK(w.held == 0 && w.seq == (int)c.recs.size());
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
    if (i % 4 == 0)   // hundreds of one-chunk tensors among the others
      for (int j = (int)below(300); j > 0; --j)
        sizes.insert(sizes.begin() + below((int64_t)sizes.size() + 1),
                     1 + below(below(2) ? 3000 : 20000));
    if (!run(sizes, grid, slots)) return 1;
  }
  std::printf("%d layouts\n", layouts);
  return 0;
}
