// mg_spans.h -- whether arrays written by one group of grids overlap arrays read
// by another (host code, tested on the host).
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace mg {

struct Span {
  uintptr_t lo, hi;  // [lo, hi)
  int group;
};

// Whether a span of `out` overlaps one of `in` of another group.
inline bool spans_cross(const std::vector<Span>& out, std::vector<Span> in) {
  if (out.empty() || in.empty()) return false;
  uintptr_t ol = UINTPTR_MAX, oh = 0, il = UINTPTR_MAX, ih = 0;
  for (const Span& s : out) ol = std::min(ol, s.lo), oh = std::max(oh, s.hi);
  for (const Span& s : in) il = std::min(il, s.lo), ih = std::max(ih, s.hi);
  if (oh <= il || ih <= ol) return false;  // outputs and inputs apart as a whole
  std::sort(in.begin(), in.end(), [](const Span& a, const Span& b) { return a.lo < b.lo; });
  std::vector<uintptr_t> reach(in.size());  // the largest end up to each span (they may overlap)
  uintptr_t far = 0;
  for (size_t q = 0; q < in.size(); ++q) reach[q] = far = std::max(far, in[q].hi);
  for (const Span& s : out) {
    size_t q = (size_t)(std::lower_bound(in.begin(), in.end(), s.hi,
                                         [](const Span& a, uintptr_t v) { return a.lo < v; }) -
                        in.begin());
    while (q > 0 && reach[q - 1] > s.lo) {
      --q;
      if (in[q].hi > s.lo && in[q].group != s.group) return true;
    }
  }
  return false;
}

}  // namespace mg
