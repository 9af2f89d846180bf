// Rules by which work is dealt out, on the host and free of CUDA: tests compile this file on its own.
#pragma once
#include <algorithm>
#include <utility>
#include <vector>

namespace lordo {

// SMs that sizes in the workspace are planned for: lordo_query_workspace makes no CUDA call and lordo_init has to agree with it. With
// fewer at hand the same ranges and chunks take more waves. Lists that lordo_init alone makes go by the device's own count.
constexpr int kPlannedSms = 148;

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

// A piece of work of one CTA (update) or CTA pair (projection) of the TMA-fed kernels: steps [t0, t1) of 64 rows of one
// strip, or one pair of strips. Workers walk their own part of a list, [start[w], start[w + 1]), dealt out by lordo_init so
// that all of them end together.
struct TcSeg {
  int prob, strip, t0, t1;
};
struct WorkItem {  // a strip (or a pair of strips) of `len` steps that costs `cost`, which is `len` where strips may be cut
  int prob, strip, len;
  double cost;
};
constexpr int kMinPiece = 8;   // steps of a piece of a cut strip
constexpr int kPieceHead = 4;  // steps that a piece costs on top of its own: its operands are fetched anew

// Deals items out, longest first, each to the worker with the least so far. With `split` no worker gets more than `share`: a
// strip that would take its worker past it is cut there and the rest dealt on, a remainder that would be too short being
// made long enough at the cost of the piece before it. False where something has no place.
// A worker is cut at most once: it is left with less room than a piece needs. So there are at most items + workers pieces.
inline bool deal_within(const std::vector<WorkItem>& items, bool split, int head, double share, std::vector<std::vector<TcSeg>>& lists) {
  typedef std::pair<double, int> Load;  // what a worker has, the worker
  std::vector<Load> heap;
  for (int w = 0; w < (int)lists.size(); ++w) { lists[w].clear(); heap.push_back(Load(0.0, w)); }
  const auto later = [](const Load& a, const Load& b) { return a > b; };
  for (const WorkItem& it : items) {
    for (int t0 = 0; t0 < it.len;) {
      std::pop_heap(heap.begin(), heap.end(), later);
      Load& ld = heap.back();
      int n = it.len - t0;
      if (split) {
        const int room = (int)(share - ld.first) - head;
        if (n > room) {
          n = std::min(room, n - kMinPiece);
          if (n < kMinPiece) return false;
        }
      }
      lists[ld.second].push_back({it.prob, it.strip, t0, t0 + n});
      ld.first += it.cost * n / it.len + head;
      t0 += n;
      std::push_heap(heap.begin(), heap.end(), later);
    }
  }
  return true;
}

// How long the workers of a cut or uncut list take, in steps of a worker that has the memory to itself: up to `busy` of them run at that
// pace, more share what the memory gives.
inline double time_of(const std::vector<std::vector<TcSeg>>& lists, int head, int busy) {
  std::vector<double> load;
  for (const std::vector<TcSeg>& l : lists) {
    double x = 0.0;
    for (const TcSeg& s : l) x += s.t1 - s.t0 + head;
    if (x > 0.0) load.push_back(x);
  }
  std::sort(load.begin(), load.end());
  double t = 0.0, before = 0.0;
  for (size_t i = 0; i < load.size(); ++i) {
    t += (load[i] - before) * std::max(1.0, (double)(load.size() - i) / busy);
    before = load[i];
  }
  return t;
}

// `list` comes back with every worker's pieces, `start` with their offsets; workers at the end without work are left out. The
// share is the smallest, in steps of 2 %, in which everything has a place. Strips dealt round the grid ended apart wherever
// they were few or of different lengths: 7 layers of 768 (r = 128, K = 8) update 183 us, dealt out 137 us.
// Strips are cut only where that ends sooner by time_of: with most of the SMs at work the memory is busy anyway, and every
// piece fetches its operands. Update of 4096 rows, r = 256: 40 strips 83 us whole, 43 us cut; 110 strips 101 and 110 us,
// 128 strips 114 and 127 us, 156 strips 199 and 147 us, 256 strips 241 and 245 us.
inline void deal_out(std::vector<WorkItem> items, int workers, bool split, int head, int busy, std::vector<TcSeg>& list, std::vector<int>& start) {
  std::stable_sort(items.begin(), items.end(), [](const WorkItem& a, const WorkItem& b) { return a.cost > b.cost; });
  std::vector<std::vector<TcSeg>> lists(workers);
  deal_within(items, false, head, 0.0, lists);
  if (split) {
    std::vector<std::vector<TcSeg>> cut(workers);
    double total = 0.0;
    for (const WorkItem& it : items) total += it.cost + head;
    double share = std::max(total / workers, (double)(kMinPiece + head));
    while (!deal_within(items, true, head, share, cut)) share += std::max(0.02 * share, 0.5);
    if (time_of(cut, head, busy) < time_of(lists, head, busy)) lists.swap(cut);
  }
  list.clear();
  start.assign(1, 0);
  for (const std::vector<TcSeg>& l : lists) {
    list.insert(list.end(), l.begin(), l.end());
    start.push_back((int)list.size());
  }
  while (start.size() > 1 && start[start.size() - 2] == (int)list.size()) start.pop_back();
}

}  // namespace lordo
