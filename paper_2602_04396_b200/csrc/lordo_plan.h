// Rules by which work is dealt out, on the host and free of CUDA: tests compile this file on its own.
#pragma once
#include <algorithm>

namespace lordo {

// Ranges of k that a product of the refresh with few output tiles is dealt out in: the count with the shortest last wave on
// `pairs` CTA pairs, a range costing about four steps of 64 k on top of its own (start of the pipeline, epilogue), and
// left four steps at least. A range has at most 64 steps, whatever their count: the tensor cores' fp32 accumulation truncates, and
// the ranges meet in fp64. Above that, no more than `most`.
inline int k_ranges(long long tiles, long long steps, long long most, long long pairs) {
  const long long least = (steps + 63) / 64;
  long long best = least, best_cost = -1;
  for (long long ns = least; ns == least || (ns <= most && steps / ns >= 4); ++ns) {
    const long long cost = ((tiles * ns + pairs - 1) / pairs) * ((steps + ns - 1) / ns + 4);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = ns; }
  }
  return (int)best;
}

}  // namespace lordo
