// Scratch memory lent from regions that a step leaves unused, and the size of the batches that fit it.
// Host code without CUDA.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

// A few regions, handed out in 256-byte units from the region with most left.  `full`: something did
// not fit (its pointer is null), nothing of the placement may be used.
struct Scratch {
  struct Region {
    unsigned char* p;
    size_t bytes, used;
  };
  std::vector<Region> r;
  bool full = false;
  void add(void* p, int64_t bytes) {
    if (bytes > 0) r.push_back(Region{(unsigned char*)p, (size_t)bytes, 0});
  }
  void reset() {
    for (Region& g : r) g.used = 0;
    full = false;
  }
  template <typename P> P* take(size_t bytes) {
    bytes = (bytes + 255) & ~(size_t)255;
    Region* best = nullptr;
    for (Region& g : r)
      if (g.bytes - g.used >= bytes && (!best || g.bytes - g.used > best->bytes - best->used)) best = &g;
    if (!best) {
      full = true;
      return nullptr;
    }
    unsigned char* q = best->p + best->used;
    best->used += bytes;
    return reinterpret_cast<P*>(q);
  }
};

// The size of equal batches of `want` blocks, as large as their buffers fit (place(n) takes those of n
// blocks, none larger for fewer); 0: none.  Whatever fits n blocks fits fewer, so bisection finds the
// largest, and the equal size and the last batch's remainder fit too: if region by region, in the order
// of what they have left, one placement has no less than another, that stays so when the first takes no
// more than the second from its largest rest (the others compare as before, and so do the two rests).
template <typename Place>
int batch_of(Scratch& w, int want, Place place) {
  auto fits = [&](int c) {
    w.reset();
    place(c);
    return !w.full;
  };
  int lo = 0, hi = std::min(want, 32768);
  if (want < 1) return 0;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (fits(mid)) lo = mid;
    else hi = mid - 1;
  }
  if (lo == 0) return 0;
  const int batches = (want + lo - 1) / lo;
  return (want + batches - 1) / batches;
}
