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

// Deals items out, longest first, each to the worker with the least so far. Returns the longest worker's.
//   WHOLE  strips are not cut
//   EVEN   a strip that would take its worker past `share` is cut there and the rest dealt on; what finds no room is dealt on
//          top, in the shortest pieces, and a remainder that would be too short stays with the piece before it
//   WITHIN no worker gets more than `share`: a remainder that would be too short is made long enough at the cost of the piece
//          before it. Returns -1 where something has no place. A worker is cut at most once, being left with less room
//          than a piece needs, so there are at most items + workers pieces.
enum Dealing { WHOLE, EVEN, WITHIN };
inline int deal(const std::vector<WorkItem>& items, Dealing how, int head, double share, std::vector<std::vector<TcSeg>>& lists) {
  typedef std::pair<double, int> Load;  // what a worker has, the worker
  std::vector<Load> heap;
  for (int w = 0; w < (int)lists.size(); ++w) { lists[w].clear(); heap.push_back(Load(0.0, w)); }
  const auto later = [](const Load& a, const Load& b) { return a > b; };
  double longest = 0.0;
  for (const WorkItem& it : items) {
    for (int t0 = 0; t0 < it.len;) {
      std::pop_heap(heap.begin(), heap.end(), later);
      Load& ld = heap.back();
      const int rest = it.len - t0, room = (int)(share - ld.first - head + 0.5);
      int n = rest;
      if (how == EVEN && n > room) {
        n = std::min(n, std::max(room, kMinPiece));
        if (rest - n < kMinPiece) n = rest;
      } else if (how == WITHIN && n > room) {
        n = std::min(room, rest - kMinPiece);
        if (n < kMinPiece) return -1;
      }
      lists[ld.second].push_back({it.prob, it.strip, t0, t0 + n});
      ld.first += how == WHOLE ? it.cost + head : n + head;
      longest = std::max(longest, ld.first);
      t0 += n;
      std::push_heap(heap.begin(), heap.end(), later);
    }
  }
  return (int)(longest + 0.5);
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

// `list` comes back with every worker's pieces, `start` with their offsets; workers at the end without work are left out. Strips dealt
// round the grid ended apart wherever they were few or of different lengths: 7 layers of 768 (r = 128, K = 8) update 183 us,
// dealt out 137 us.
// With `split` strips are dealt out by EVEN, with half a head of slack per worker. Where cuts cost more than that (few long strips: one
// of 2004 steps ended with a longest worker of 1.75 times the mean), the smallest share that WITHIN finds a place for is better, and where
// most SMs have a whole strip the memory is busy anyway and WHOLE is, since every piece fetches its operands. Either is taken where
// it ends sooner than EVEN by a tenth by time_of, which is about how well that tells: update of 4096 rows, r = 256, EVEN, WHOLE and WITHIN:
// 40 strips 50, 83, 43 us; 120 strips 122, 107, 121 us; 256 strips 241, 241, 245 us; mixes that it called 4 to 8 % better were 2 to 5 % slower.
inline void deal_out(std::vector<WorkItem> items, int workers, bool split, int head, int busy, std::vector<TcSeg>& list, std::vector<int>& start) {
  std::stable_sort(items.begin(), items.end(), [](const WorkItem& a, const WorkItem& b) { return a.cost > b.cost; });
  std::vector<std::vector<TcSeg>> lists(workers);
  const int longest = deal(items, WHOLE, head, 0.0, lists);
  if (split) {
    double total = 0.0;
    for (const WorkItem& it : items) total += it.cost + head;
    std::vector<std::vector<TcSeg>> even(workers), cut(workers), within;
    deal(items, EVEN, head, std::max(total / workers + head / 2.0, (double)(kMinPiece + head)), even);
    size_t pieces = 0;
    for (const std::vector<TcSeg>& l : even) pieces += l.size();
    int least = std::max((int)(total / workers), kMinPiece + head) - 1, share = longest;  // nothing below, everything at WHOLE's longest
    while (share - least > 1) {
      const int mid = least + (share - least) / 2;
      if (deal(items, WITHIN, head, mid, cut) < 0) least = mid;
      else { share = mid; within.swap(cut); cut.resize(workers); }
    }
    if (!within.empty() && time_of(within, head, busy) < time_of(lists, head, busy)) lists.swap(within);
    const bool fits = pieces <= items.size() + workers;  // the room that the table has; either of the others does
    if (fits && time_of(lists, head, busy) > 0.9 * time_of(even, head, busy)) lists.swap(even);
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
