// The sizes of batches whose buffers are placed in several regions: whatever the regions and buffers,
// every batch that is made of the size returned has to fit.  Prints "scratch ok" on success.
#include <cstdio>
#include <random>

#include "../../paper_2207_10701_gb300/csrc/scratch.h"

static unsigned char base[1];

static int check(const std::vector<int64_t>& regions, const std::vector<int64_t>& per, const std::vector<int64_t>& once,
                 int want) {
  Scratch w;
  for (int64_t r : regions) w.add(base, r);
  auto place = [&](int c) {
    for (size_t i = 0; i < per.size(); ++i) w.take<char>((size_t)(c * per[i] + once[i]));
  };
  const int c = batch_of(w, want, place);
  if (c < 0 || c > want) return std::printf("scratch FAIL: %d of %d\n", c, want), 1;
  for (int k = 0; c > 0 && k < want; k += c) {
    w.reset();
    place(std::min(c, want - k));
    if (w.full) return std::printf("scratch FAIL: a batch of %d (size %d of %d)\n", std::min(c, want - k), c, want), 1;
  }
  return 0;
}

int main() {
  std::mt19937_64 rng(7);
  auto upto = [&](int64_t n) { return (int64_t)(rng() % (uint64_t)n); };
  for (int t = 0; t < 200000; ++t) {
    std::vector<int64_t> regions(2 + upto(4)), per(2 + upto(5)), once;
    for (int64_t& r : regions) r = 256 * (1 + upto(60));
    for (int64_t& p : per) {
      p = 256 * (1 + upto(6));
      once.push_back(upto(3) ? 0 : p);
    }
    if (check(regions, per, once, 1 + (int)upto(24))) return 1;
  }
  std::printf("scratch ok\n");
  return 0;
}
