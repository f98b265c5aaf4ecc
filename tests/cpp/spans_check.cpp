// spans_cross (mg_spans.h) against the comparison of every pair.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2302_13903_gb300/csrc/mg_spans.h"

int main() {
  std::mt19937 rng(7);
  int found = 0;
  for (int trial = 0; trial < 20000; ++trial) {
    const int range = 10 + (int)(rng() % 400);
    auto spans = [&](int n) {
      std::vector<mg::Span> v;
      for (int q = 0; q < n; ++q) {
        const uintptr_t lo = 16 + rng() % range;
        v.push_back({lo, lo + 1 + rng() % 24, (int)(rng() % 3)});
      }
      return v;
    };
    const auto out = spans(rng() % 8), in = spans(rng() % 8);
    bool want = false;
    for (const auto& a : out)
      for (const auto& b : in) want = want || (a.group != b.group && a.lo < b.hi && b.lo < a.hi);
    if (mg::spans_cross(out, in) != want) {
      std::printf("trial %d: %d wanted\n", trial, want);
      return 1;
    }
    found += want;
  }
  std::printf("%d of 20000 cross\n", found);
  return found < 1000 || found > 19000;
}
