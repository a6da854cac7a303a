// Key-range splitting of the tensor-memory attention launch: the host-side choice of how many pieces every
// head's key range is cut into.  Pure host code (no CUDA): the launch is described by the key tiles of its
// heads in dispatch order (descending), the query tile pairs per head, the sequences of the call and the SMs.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"

namespace heatkv {

SplitShape split_shape(const std::vector<int>& tiles, const std::vector<int>& ns, int n_qp, int n_qt) {
  SplitShape r;
  for (size_t i = 0; i < tiles.size(); ++i) {
    r.items += ns[i] > 0 ? n_qp * ns[i] : n_qt;
    if (ns[i] > 1) { r.slots += n_qp * ns[i]; r.ctrs += n_qp; }
  }
  return r;
}

// Estimated makespan (in units of one 128-key tile) of the launch.  Items are taken by the resident CTAs in
// dispatch order (heads by descending key count, pieces, query tile pairs, sequences interleaved); for very
// large launches the list-scheduling bound total / SMs + longest is used.  The per-item constants were fitted
// to clock stamps of the kernel: an item costs its tiles plus the result's way out and the next item's start;
// a piece writes fp32 partials instead, and the piece that arrives last reads the others.
// The items of a piece are all alike and the SMs that finish at the same moment are kept as one entry, so an entry takes
// as many items at once as it has SMs: the search on a new context (a thousand launches of hundreds of items, on the way
// of a model's first image) takes 1.3 ms where a heap of single SMs took 75 (32 heads, 2 layers, 13 scales).
// `give_up`: any value at or above it may be returned as soon as the launch cannot end before it.
struct ItemRun {
  double cost;
  int n;                                                   // items of that cost, per sequence
};
static void add(std::vector<ItemRun>& items, double cost, int n) {
  if (!items.empty() && items.back().cost == cost) items.back().n += n;       // neighbours that are alike
  else items.push_back({cost, n});
}
constexpr double FIXED = 2.0, PUBLISH = 1.0, MERGE_PER_PIECE = 1.5;
static double finish(const std::vector<ItemRun>& items, int n_seq, int n_sm, double give_up) {
  double total = 0.0, longest = 0.0;
  size_t n_items = 0;
  for (const ItemRun& it : items) {
    total += it.cost * it.n;
    longest = std::max(longest, it.cost);
    n_items += it.n;
  }
  n_items *= (size_t)n_seq;
  if (n_items > 8192) return total * n_seq / n_sm + longest;
  const double at_least = std::max(total * n_seq / n_sm, longest);
  if (at_least >= give_up) return at_least;
  struct Run {
    double t;                                              // finish time
    int sms;                                               // SMs that share it
  };
  std::vector<Run> runs;                                   // binary min-heap
  runs.reserve(2 * items.size() + 2);
  runs.push_back({0.0, n_sm});
  auto later = [](const Run& a, const Run& b) { return a.t > b.t; };
  double end = 0.0;
  for (const ItemRun& it : items)
    for (int left = it.n * n_seq; left > 0;) {
      std::pop_heap(runs.begin(), runs.end(), later);
      Run& r = runs.back();
      const int n = std::min(left, r.sms);
      const double t = r.t + it.cost;
      left -= n;
      end = std::max(end, t);
      if (n < r.sms) {
        r.sms -= n;
        std::push_heap(runs.begin(), runs.end(), later);
        runs.push_back({t, n});
      } else {
        r.t = t;
      }
      std::push_heap(runs.begin(), runs.end(), later);
    }
  return end;
}

static double makespan(const std::vector<int>& tiles, const std::vector<int>& ns, int n_qp, int n_seq, int n_sm, double give_up) {
  std::vector<ItemRun> items;
  items.reserve(2 * tiles.size());
  for (size_t i = 0; i < tiles.size(); ++i)
    for (int pc = 0; pc < ns[i]; ++pc) {
      const int piece = (tiles[i] + ns[i] - 1) / ns[i];
      const int len = std::min(tiles[i], (pc + 1) * piece) - pc * piece;
      add(items, len + FIXED + (ns[i] > 1 ? PUBLISH + MERGE_PER_PIECE * (ns[i] - 1) / ns[i] : 0.0), n_qp);
    }
  return finish(items, n_seq, n_sm, give_up);
}

double split_makespan(const std::vector<int>& tiles, const std::vector<int>& ns, int n_qp, int n_seq, int n_sm) {
  return makespan(tiles, ns, n_qp, n_seq, n_sm, HUGE_VAL);
}

// The search.  Long heads are cut to a common longest run (candidates: the longest head divided by 2..16), and,
// when `per_head` allows a piece count of its own for every head, the heads dispatched last may be cut two or
// three times finer so that the last round of items fills the SMs.  A cut is taken when it shortens the estimate of the
// launch with whole heads by 5 % and that of the best cut so far by 2 % (28 uncompressed heads: 2.16 ms a pass with 5 % for
// both, 2.12 with 2 %; image pair 2.319 and 2.311; any gain at all measured no better); pieces are never shorter than
// SPLIT_MIN_PIECE tiles, and the partial slots and arrival counters the cut needs per sequence (times n_seq) must fit
// max_slots / max_ctrs.
constexpr double WORTH = 0.95, BETTER = 0.98;
SplitChoice split_search(const std::vector<int>& tiles, int n_qp, int n_seq, int n_sm, bool per_head, uint64_t max_slots,
                         uint64_t max_ctrs) {
  const int H = (int)tiles.size();
  SplitChoice best;
  best.ns.assign(H, 1);
  if (H == 0) return best;
  double best_t = split_makespan(tiles, best.ns, n_qp, n_seq, n_sm);
  const double whole_t = best_t;
  auto fits = [&](const SplitShape& sh) {
    return (uint64_t)sh.slots * n_seq <= max_slots && (uint64_t)sh.ctrs * n_seq * SPLIT_CTRS_PER_GROUP <= max_ctrs;
  };
  const int max_tiles = *std::max_element(tiles.begin(), tiles.end());
  std::vector<int> lmaxes = {0};
  for (int div : {2, 3, 4, 6, 8, 12, 16}) {
    const int cand = (max_tiles + div - 1) / div;
    if (cand < SPLIT_MIN_PIECE) break;
    lmaxes.push_back(cand);
  }
  for (int lmax : lmaxes) {
    std::vector<int> base(H);
    for (int i = 0; i < H; ++i) base[i] = split_pieces_for(tiles[i], lmax);
    for (int extra = 1; extra <= (per_head ? 3 : 1); ++extra)
      for (int tail = (extra == 1 ? 0 : 1); tail <= (extra == 1 ? 0 : H); ++tail) {
        std::vector<int> ns = base;
        bool ok = true;
        for (int i = H - tail; i < H; ++i) {
          ns[i] = base[i] * extra;
          ok = ok && (tiles[i] + ns[i] - 1) / ns[i] >= SPLIT_MIN_PIECE;
        }
        for (int i = 0; i < H; ++i) ok = ok && split_cut_ok(tiles[i], ns[i]);
        if (!ok || (lmax == 0 && tail == 0)) continue;
        if (!fits(split_shape(tiles, ns, n_qp, 0))) continue;
        const double take = std::min(BETTER * best_t, WORTH * whole_t);
        const double t = makespan(tiles, ns, n_qp, n_seq, n_sm, take);
        if (t < take) { best_t = t; best.ns = ns; best.lmax = tail == 0 ? lmax : -1; }
      }
  }
  return best;
}

// Should the launch take query tiles one by one instead (SplitChoice::lone)?  Such an item takes its key tiles two at a time, so it is
// half as long as a pair's without the partial results of a cut, at the price of keys and values read once per tile instead of once
// per pair: per key tile 1.02 us where a pair takes 1.83 (1024 queries, 12 to 40 key tiles, 296 heads) and 0.80 where a pair takes 1.52
// (28 heads x 576 queries).  Candidates: the longest heads, the ones dispatched last, both, all, or none but the odd last tiles.  Back
// to back: 32 heads x 576 queries, two of 12 and thirty of 5 to 7 tiles, 22.5 -> 16.8 us; 28 x 576, 12 tiles, 25.9 -> 18.5; 28 x 1024,
// 20 tiles, all by themselves 44 against 39 (not taken); 128 x 1600 queries, last tiles alone, 224.5 -> 218.8.  Launches with cuts are
// longer than their estimate by what the last piece's way through memory takes and no other item hides (14 launches of 80 to
// 288 items: whole heads and lone tiles 1.58 us per unit and 2.3, cuts 3.4 to 5.8 us more): 102 items of 256 queries, 30 of 12 tiles, cut
// in three 20.6 us, lone 15.9; 32 heads x 1024 queries, 4 of 19 tiles, cut in two 27.4, lone 22.6.
constexpr double TILE_SINGLE = 0.55;        // a key tile of such an item
constexpr double TILE_PADDED = 0.81;        // of a lone query tile run as the first of a pair
constexpr double LONE_LAUNCH = 0.8;         // a kernel of its own: its code is fetched anew between launches of the other
constexpr double CUT_LAUNCH = 3.0;
void single_search(const std::vector<int>& tiles, int t_q, int n_seq, int n_sm, bool per_head, SplitChoice* choice) {
  const int H = (int)tiles.size(), n_qp = (t_q + 255) / 256, n_qt = (t_q + 127) / 128, odd = n_qt & 1;
  if (H == 0) return;
  std::vector<ItemRun> items;
  auto list = [&](const std::vector<int>& ns, bool lone) {
    items.clear();
    for (int i = 0, m; i < H; i += m) {
      for (m = 1; i + m < H && tiles[i + m] == tiles[i] && ns[i + m] == ns[i];) ++m;       // heads that are alike
      if (ns[i] == 0) {
        add(items, TILE_SINGLE * tiles[i] + FIXED, m * n_qt);
        continue;
      }
      const int k = ns[i], piece = (tiles[i] + k - 1) / k;
      const double fixed = FIXED + (k > 1 ? PUBLISH + MERGE_PER_PIECE * (k - 1) / k : 0.0);
      for (int pc = 0; pc < k; ++pc) {
        const int len = std::min(tiles[i], (pc + 1) * piece) - pc * piece;
        if (n_qp > odd) add(items, len + fixed, m * (n_qp - odd));
        if (odd) add(items, (lone ? TILE_SINGLE : TILE_PADDED) * len + fixed, m);
      }
    }
  };
  list(choice->ns, false);
  const bool is_cut = std::any_of(choice->ns.begin(), choice->ns.end(), [](int n) { return n > 1; });
  double take = BETTER * (finish(items, n_seq, n_sm, HUGE_VAL) + (is_cut ? CUT_LAUNCH : 0.0)) - LONE_LAUNCH;
  std::vector<int> ns(H);
  auto attempt = [&](int first, int last) {
    ns.assign(H, 1);
    std::fill(ns.begin(), ns.begin() + first, 0);
    std::fill(ns.end() - last, ns.end(), 0);
    list(ns, true);
    const double t = finish(items, n_seq, n_sm, take);
    if (t >= take) return;
    take = BETTER * t;
    choice->lone = ns;
  };
  attempt(H, 0);
  if (odd) attempt(0, 0);
  if (!per_head) return;
  for (int first = 0, tried = 0; first < H && tried < 4; ++tried) {
    for (int last = first == 0 ? 1 : 0; first + last < H; last = last ? 2 * last : 1) attempt(first, last);
    const int longest = tiles[first];
    while (first < H && tiles[first] == longest) ++first;
  }
}

}  // namespace heatkv

extern "C" int heatkv_split_plan(const int32_t* tiles, int n_heads, int n_qp, int n_seq, int n_sm, int per_head,
                                 uint64_t max_slots, uint64_t max_ctrs, int32_t* pieces, double* makespan_whole,
                                 double* makespan_cut) {
  if (!tiles || !pieces || n_heads < 1 || n_qp < 1 || n_seq < 1 || n_sm < 1) return HEATKV_ERR_INVALID_ARG;
  for (int i = 0; i < n_heads; ++i)
    if (tiles[i] < 1 || (i > 0 && tiles[i] > tiles[i - 1])) return HEATKV_ERR_INVALID_ARG;
  try {
    const std::vector<int> t(tiles, tiles + n_heads);
    const heatkv::SplitChoice ch = heatkv::split_search(t, n_qp, n_seq, n_sm, per_head != 0, max_slots, max_ctrs);
    for (int i = 0; i < n_heads; ++i) pieces[i] = ch.ns[i];
    if (makespan_whole) *makespan_whole = heatkv::split_makespan(t, std::vector<int>(n_heads, 1), n_qp, n_seq, n_sm);
    if (makespan_cut) *makespan_cut = heatkv::split_makespan(t, ch.ns, n_qp, n_seq, n_sm);
  } catch (const std::bad_alloc&) {
    return HEATKV_ERR_HOST_MEMORY;
  }
  return HEATKV_OK;
}
