// Rules by which work is dealt out, on the host and free of CUDA: tests compile this file on its own.
#pragma once
#include <algorithm>
#include <functional>
#include <queue>
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

// CTAs per matrix of the factorisation: as many, up to the portable cluster size, as leave every matrix a place on the device at once (`fits`:
// clusters of that many CTAs that the device holds) and every CTA about two row blocks. r = 512, 16 matrices, us: one CTA each 828, two 499,
// four 301, six 275; seven or eight, of which fifteen clusters fit, 504 and 392. r = 256, 7 matrices: 150, 97, with four 76. Above 74 matrices
// one CTA each: 148 of r = 192 take 128 us that way, 152 in two, 300 of r = 256 488 and 480.
inline int factor_ctas(int panels, int matrices, const int* fits) {
  int c = 8;
  while (c > 1 && (2 * c > panels + 1 || matrices > fits[c])) --c;
  return c;
}

// A piece of work of one CTA (update) or CTA pair (projection) of the TMA-fed kernels: steps [t0, t1) of one strip, of 64 rows
// each with bf16 storage and of 32 with fp32 (as many bytes), or one pair of strips. Workers walk their own part of a list,
// [start[w], start[w + 1]), dealt out by lordo_init so that all of them end together.
struct TcSeg {
  int prob, strip, t0, t1;
};
struct WorkItem {  // a strip (or a pair of strips) of `len` steps that costs `cost`, which is `len` where strips may be cut
  int prob, strip, len;
  double cost;
};
// Steps of a piece of a cut strip. With fp32 storage short ones pay: the products of a step are half as long, and with pieces of eight 1064 x 72,
// r = 8 went to 5 CTAs (a round of four steps 170 us, with pieces of four 154, of two 146; the kernel before this one 161),
// 456 x 592, r = 32 and two workers to 10 (38.9, 30.7, 28.7; 36.4). 190 steps and rounds of random shapes: 1.04 times as fast on average with pieces
// of two as of eight, at worst 0.97. A smaller kPieceHead cost up to 4 % of some, a larger one changed nothing, nor did other shares of busy SMs.
constexpr int kMinPiece = 8, kMinPiece32 = 2;
constexpr int kPieceHead = 4;  // steps that a piece costs on top of its own: its operands are fetched anew

// Deals items out, longest first, each to the worker with the least so far. Returns the longest worker's.
//   WHOLE  strips are not cut
//   EVEN   a strip that would take its worker past `share` is cut there and the rest dealt on; what finds no room is dealt on
//          top, in the shortest pieces (of `least` steps), and a remainder that would be too short stays with the piece before it
//   WITHIN no worker gets more than `share`: a remainder that would be too short is made long enough at the cost of the piece
//          before it. Returns -1 where something has no place. A worker is cut at most once, being left with less room
//          than a piece needs, so there are at most items + workers pieces.
enum Dealing { WHOLE, EVEN, WITHIN };
struct Dealt {
  typedef std::pair<double, int> Load;  // what a worker has, the worker
  std::vector<TcSeg> piece;
  std::vector<int> worker;    // of a piece
  std::vector<Load> least;    // a heap, the worker with the least first
};
inline int deal(const std::vector<WorkItem>& items, Dealing how, int head, int least, double share, int workers, Dealt& d) {
  d.piece.clear();
  d.worker.clear();
  d.least.clear();
  for (int w = 0; w < workers; ++w) d.least.push_back(Dealt::Load(0.0, w));
  double longest = 0.0;
  for (const WorkItem& it : items) {
    for (int t0 = 0; t0 < it.len;) {
      Dealt::Load ld = d.least.front();
      const int rest = it.len - t0, room = (int)(share - ld.first - head + 0.5);
      int n = rest;
      if (how == EVEN && n > room) {
        n = std::min(n, std::max(room, least));
        if (rest - n < least) n = rest;
      } else if (how == WITHIN && n > room) {
        n = std::min(room, rest - least);
        if (n < least) return -1;
      }
      d.piece.push_back({it.prob, it.strip, t0, t0 + n});
      d.worker.push_back(ld.second);
      ld.first += how == WHOLE ? it.cost + head : n + head;
      longest = std::max(longest, ld.first);
      t0 += n;
      int at = 0;
      for (int c = 1; c < workers; c = 2 * at + 1) {
        if (c + 1 < workers && d.least[c + 1] < d.least[c]) ++c;
        if (ld < d.least[c]) break;
        d.least[at] = d.least[c];
        at = c;
      }
      d.least[at] = ld;
    }
  }
  return (int)(longest + 0.5);
}

// How long the workers of a cut or uncut list take, in steps of a worker that has the memory to itself: up to `busy` of them run at that
// pace, more share what the memory gives.
inline double time_of(const Dealt& d, int busy) {
  std::vector<double> load;
  for (const Dealt::Load& l : d.least)
    if (l.first > 0.0) load.push_back(l.first);
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
inline void deal_out(std::vector<WorkItem> items, int workers, bool split, int head, int shortest, int busy, std::vector<TcSeg>& list, std::vector<int>& start) {
  std::stable_sort(items.begin(), items.end(), [](const WorkItem& a, const WorkItem& b) { return a.cost > b.cost; });
  Dealt dealt;
  const int longest = deal(items, WHOLE, head, shortest, 0.0, workers, dealt);
  if (split) {
    double total = 0.0;
    for (const WorkItem& it : items) total += it.cost + head;
    Dealt even, cut, within;
    deal(items, EVEN, head, shortest, std::max(total / workers + head / 2.0, (double)(shortest + head)), workers, even);
    int least = std::max((int)(total / workers), shortest + head) - 1, share = longest;  // nothing below, everything at WHOLE's longest
    while (share - least > 1) {
      const int mid = least + (share - least) / 2;
      if (deal(items, WITHIN, head, shortest, mid, workers, cut) < 0) least = mid;
      else { share = mid; std::swap(within, cut); }
    }
    if (!within.piece.empty() && time_of(within, busy) < time_of(dealt, busy)) std::swap(dealt, within);
    const bool fits = even.piece.size() <= items.size() + workers;  // the room that the table has; either of the others does
    if (fits && time_of(dealt, busy) > 0.9 * time_of(even, busy)) std::swap(dealt, even);
  }
  start.assign(workers + 1, 0);
  for (int w : dealt.worker) ++start[w + 1];
  for (int w = 0; w < workers; ++w) start[w + 1] += start[w];
  list.resize(dealt.piece.size());
  std::vector<int> next(start.begin(), start.end() - 1);
  for (size_t i = 0; i < dealt.piece.size(); ++i) list[next[dealt.worker[i]]++] = dealt.piece[i];
  while (start.size() > 1 && start[start.size() - 2] == (int)list.size()) start.pop_back();
}

// ---- fp32 products: rows per thread and CTAs per output tile ------------------------------------
// Consecutive tiles of a launch whose contraction takes `slices` slices of 16 k.
struct ProductRun {
  int slices;
  long long tiles;
};
struct ProductSplit {
  int rows = 4, ctas = 1;  // rows per thread (4 or 8); CTAs per tile, a cluster that shares the slices
};
inline int longest_run(const std::vector<ProductRun>& runs) {
  int longest = 1;
  for (const ProductRun& r : runs) longest = std::max(longest, r.slices);
  return longest;
}

// How long a launch takes, in slices of a CTA of four rows that has an SM to itself. CTAs take their places in the order of the tiles; what
// a slice takes depends on how many share an SM: four rows 1 and, two on an SM, 1.2, eight rows 1.375, 1.4 and, three, 1.475
// (a slice of one CTA is latency: 0.85 us). A CTA takes some four slices more for its start and end, and the meeting of a cluster one
// and 0.45 for each of its CTAs.
inline double product_time(const std::vector<ProductRun>& runs, int rows, int ctas, int sms) {
  typedef std::pair<double, long long> Group;  // when they end, at the pace of one to an SM, and how many
  std::priority_queue<Group, std::vector<Group>, std::greater<Group>> running;
  const long long room = (long long)sms * (rows == 4 ? 2 : 3);  // by registers
  const double extra = (rows == 4 ? 4.5 : 4.0) + (ctas > 1 ? 1.0 + 0.45 * ctas : 0.0);
  const auto pace = [&](double per_sm) {
    if (rows == 4) return 1.0 + 0.2 * std::max(0.0, per_sm - 1.0);
    return per_sm <= 2.0 ? 1.375 + 0.025 * std::max(0.0, per_sm - 1.0) : 1.4 + 0.075 * (per_sm - 2.0);
  };
  double at = 0.0, time = 0.0;
  long long resident = 0;
  size_t next = 0;
  long long left = runs.empty() ? 0 : runs[0].tiles * ctas;
  for (;;) {
    while (next < runs.size() && resident < room) {
      const long long n = std::min(left, room - resident);
      if (n > 0) running.push(Group(at + (runs[next].slices + ctas - 1) / ctas + extra, n));
      resident += n;
      left -= n;
      if (left == 0 && ++next < runs.size()) left = runs[next].tiles * ctas;
    }
    if (running.empty()) return time;
    const double end = running.top().first;
    time += (end - at) * pace((double)resident / sms);
    at = end;
    while (!running.empty() && running.top().first <= at) { resident -= running.top().second; running.pop(); }
  }
}

// Sums carried in fp32 (fast mode): four rows, and the count of CTAs whose turns on the device times the slices of k of each, with about three
// more for its start and end, are least; each is left two slices. A product with few tiles is a chain of slices, each about a
// trip to memory long: 256 x 256, r = 16, two replicas, P^T (c G + E) in 8 CTAs 44 us, in 64 10.5; Gram matrices of 1000 rows and
// r up to 136 in 14 CTAs 105 us, in 112 17.
inline ProductSplit split_by_turns(const std::vector<ProductRun>& runs, int sms) {
  const int slices = longest_run(runs);
  long long tiles = 0, best = -1;
  for (const ProductRun& r : runs) tiles += r.tiles;
  ProductSplit s;
  for (int x = 1; x <= 8 && (x == 1 || slices >= 2 * x); x *= 2) {
    const long long cost = ((tiles * x + 2 * sms - 1) / (2 * sms)) * ((slices + x - 1) / x + 3);
    if (best < 0 || cost < best) { best = cost; s.ctas = x; }
  }
  return s;
}

// Sums carried in fp64 (check mode): the rows and CTAs whose launch is over first by product_time. Turns of CTAs as long as the longest contraction
// told eight rows from four only where the contractions are alike: matrices of 5472 rows, r = 120 and of 64 to 3704 rows, r <= 40
// took 209 us in pairs of eight rows by that rule, 87 in fours of four rows, and take 71 now. Over 790 launches of parity runs of random
// shapes the choice takes at most 1.02 of the best split's time for nine of ten, and 1.3 for the worst (by turns 1.2 and 3.2).
// A launch of more than 2048 tiles is timed as one of that many: the same choice, and a bounded time to make it in.
inline ProductSplit split_by_time(std::vector<ProductRun> runs, int sms) {
  const int slices = longest_run(runs);
  long long tiles = 0;
  for (const ProductRun& r : runs) tiles += r.tiles;
  if (tiles > 2048)
    for (ProductRun& r : runs) r.tiles = (r.tiles * 2048 + tiles - 1) / tiles;
  ProductSplit best;
  double least = -1.0;
  for (int rows = 4; rows <= 8; rows += 4)
    for (int x = 1; x <= 8 && (x == 1 || slices >= 2 * x); x *= 2) {
      const double t = product_time(runs, rows, x, sms);
      if (least < 0.0 || t < least) { least = t; best.rows = rows; best.ctas = x; }
    }
  return best;
}

}  // namespace lordo
