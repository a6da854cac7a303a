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
// as many items at once as it has SMs.  The searches look at a thousand launches of hundreds of items on the way of a model's first
// image, so a candidate's total and longest item come from sums per head, and its items are only listed and simulated (in buffers that
// the whole search shares) where that bound is below the best so far: both searches for every step and layer of a pair of images at 20x
// (16 heads, 4 layers) take 0.49 ms where listing every candidate took 1.55, with 32 heads of 64 (2 layers) 0.45 and 2.1.
constexpr double FIXED = 2.0, PUBLISH = 1.0, MERGE_PER_PIECE = 1.5;
constexpr size_t SIMULATED_ITEMS = 8192;
struct ItemRun {
  double cost;
  int n;                                                   // items of that cost, per sequence
};
// What every estimate needs of a number of heads.
struct Load {
  double total = 0.0, longest = 0.0;
  size_t items = 0;
  uint64_t slots = 0, ctrs = 0;
  Load operator+(const Load& o) const {
    return {total + o.total, std::max(longest, o.longest), items + o.items, slots + o.slots, ctrs + o.ctrs};
  }
  Load items_of(double cost, int n) const { return *this + Load{cost * n, n > 0 ? cost : 0.0, (size_t)n, 0, 0}; }
};
struct Launch {
  int n_seq, n_sm;
  std::vector<ItemRun> items;
  struct Run {
    double t;                                              // finish time
    int sms;                                               // SMs that share it
  };
  std::vector<Run> runs;                                   // binary min-heap

  void add(double cost, int n) {
    if (!items.empty() && items.back().cost == cost) items.back().n += n;     // neighbours that are alike
    else items.push_back({cost, n});
  }
  // The estimate of a launch whose items `list` adds; any value at or above `give_up` if it cannot end before that.
  template <typename F>
  double estimate(const Load& sum, double give_up, F list) {
    if (sum.items * n_seq > SIMULATED_ITEMS) return sum.total * n_seq / n_sm + sum.longest;
    const double at_least = std::max(sum.total * n_seq / n_sm, sum.longest);
    if (at_least >= give_up) return at_least;
    items.clear();
    list();
    return finish(give_up);
  }
  double finish(double give_up) {
    runs.clear();
    runs.push_back({0.0, n_sm});
    auto later = [](const Run& a, const Run& b) { return a.t > b.t; };
    double end = 0.0;
    for (const ItemRun& it : items)
      for (int left = it.n * n_seq; left > 0;) {
        const double t = runs[0].t + it.cost;
        const int n = std::min(left, runs[0].sms);
        left -= n;
        end = std::max(end, t);
        if (end >= give_up) return end;
        if (n < runs[0].sms) {
          runs[0].sms -= n;                                // (it stays the earliest)
          runs.push_back({t, n});
          std::push_heap(runs.begin(), runs.end(), later);
          continue;
        }
        size_t at = 0;                                     // the earliest entry ends at t now: down to its place
        for (size_t below; (below = 2 * at + 1) < runs.size(); at = below) {
          if (below + 1 < runs.size() && runs[below + 1].t < runs[below].t) ++below;
          if (runs[below].t >= t) break;
          runs[at] = runs[below];
        }
        runs[at] = {t, n};
      }
    return end;
  }
};

// Pieces of a head: all but the last as long as the first.
struct Cut {
  int full, last;
  double fixed;
  Cut(int tiles, int ns) : full((tiles + ns - 1) / ns), last(tiles - (ns - 1) * full),
                           fixed(FIXED + (ns > 1 ? PUBLISH + MERGE_PER_PIECE * (ns - 1) / ns : 0.0)) {}
};
static Load head_load(int tiles, int ns, int n_qp) {
  const Cut c(tiles, ns);
  Load r = Load().items_of(c.full + c.fixed, n_qp * (ns - 1)).items_of(c.last + c.fixed, n_qp);
  if (ns > 1) { r.slots = (uint64_t)n_qp * ns; r.ctrs = n_qp; }
  return r;
}
static void add_head(Launch& launch, int tiles, int ns, int n_qp) {
  const Cut c(tiles, ns);
  if (ns > 1) launch.add(c.full + c.fixed, n_qp * (ns - 1));
  launch.add(c.last + c.fixed, n_qp);
}

double split_makespan(const std::vector<int>& tiles, const std::vector<int>& ns, int n_qp, int n_seq, int n_sm) {
  Launch launch{n_seq, n_sm};
  Load sum;
  for (size_t i = 0; i < tiles.size(); ++i) sum = sum + head_load(tiles[i], ns[i], n_qp);
  return launch.estimate(sum, HUGE_VAL, [&] {
    for (size_t i = 0; i < tiles.size(); ++i) add_head(launch, tiles[i], ns[i], n_qp);
  });
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
  Launch launch{n_seq, n_sm};
  double best_t = split_makespan(tiles, best.ns, n_qp, n_seq, n_sm);
  const double whole_t = best_t;
  const int max_tiles = *std::max_element(tiles.begin(), tiles.end());
  std::vector<int> lmaxes = {0};
  for (int div : {2, 3, 4, 6, 8, 12, 16}) {
    const int cand = (max_tiles + div - 1) / div;
    if (cand < SPLIT_MIN_PIECE) break;
    lmaxes.push_back(cand);
  }
  std::vector<int> base(H);
  std::vector<Load> before(H + 1);                         // of the heads before this one
  for (int lmax : lmaxes) {
    int base_ok = 0;                                       // heads before the first whose equal cut would leave a piece empty
    for (int i = 0; i < H; ++i) {
      base[i] = split_pieces_for(tiles[i], lmax);
      before[i + 1] = before[i] + head_load(tiles[i], base[i], n_qp);
      if (base_ok == i && split_cut_ok(tiles[i], base[i])) ++base_ok;
    }
    // the last `tail` heads in `extra` times as many pieces
    auto attempt = [&](int extra, int tail, const Load& sum) {
      if (sum.slots * n_seq > max_slots || sum.ctrs * n_seq * SPLIT_CTRS_PER_GROUP > max_ctrs) return;
      const double take = std::min(BETTER * best_t, WORTH * whole_t);
      const double t = launch.estimate(sum, take, [&] {
        for (int i = 0; i < H; ++i) add_head(launch, tiles[i], i < H - tail ? base[i] : base[i] * extra, n_qp);
      });
      if (t >= take) return;
      best_t = t;
      best.lmax = tail == 0 ? lmax : -1;
      best.ns = base;
      for (int i = H - tail; i < H; ++i) best.ns[i] *= extra;
    };
    if (lmax > 0 && base_ok == H) attempt(1, 0, before[H]);
    for (int extra = 2; extra <= (per_head ? 3 : 1); ++extra) {
      Load finer;
      for (int i = H - 1; i >= 0; --i) {
        const int ns = base[i] * extra;
        if ((tiles[i] + ns - 1) / ns < SPLIT_MIN_PIECE || !split_cut_ok(tiles[i], ns)) break;
        finer = finer + head_load(tiles[i], ns, n_qp);
        if (base_ok >= i) attempt(extra, H - i, before[i] + finer);
      }
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
// Items are simulated in the kernel's own order, head by head: with the odd last tiles of equal heads behind all their pairs the estimate was
// up to a third too short, and 72 heads x 576 queries over 25 key tiles ran lone in 82.9 us (64-wide 74.7) where cut heads take 72.3 (62.0);
// now 72.5 (61.4), over 15 tiles 54.0 -> 47.2, 136 heads 89.5 -> 76.5.
constexpr double TILE_SINGLE = 0.55;        // a key tile of such an item
constexpr double TILE_PADDED = 0.81;        // of a lone query tile run as the first of a pair
constexpr double LONE_LAUNCH = 0.8;         // a kernel of its own: its code is fetched anew between launches of the other
// Of 64-wide heads cuts are that much longer by 1.7 units, not by 3 (152 launches under 45 units against 130 of whole heads, 1.28 us a unit; lone
// ones 0.2 shorter than those; 128-wide: 3.3, 1.66 us, 0.4 longer), cold launches the same within 0.5.
constexpr double CUT_LAUNCH_128 = 3.0, CUT_LAUNCH_64 = 1.7;
void single_search(const std::vector<int>& tiles, int t_q, int n_seq, int n_sm, int d, bool per_head, SplitChoice* choice) {
  const int H = (int)tiles.size(), n_qp = (t_q + 255) / 256, n_qt = (t_q + 127) / 128, odd = n_qt & 1;
  if (H == 0) return;
  Launch launch{n_seq, n_sm};
  std::vector<Load> pairs(H + 1), singles(H + 1);          // of the heads before this one: whole, and with their query tiles one by one
  Load as_chosen;
  for (int i = 0; i < H; ++i) {
    const double one = TILE_SINGLE * tiles[i] + FIXED;
    singles[i + 1] = singles[i].items_of(one, n_qt);
    pairs[i + 1] = pairs[i].items_of(tiles[i] + FIXED, n_qp - odd).items_of(one, odd);
    const int ns = choice->ns[i];
    const Cut c(tiles[i], ns);
    as_chosen = as_chosen.items_of(c.full + c.fixed, (ns - 1) * (n_qp - odd)).items_of(c.last + c.fixed, n_qp - odd);
    if (odd)
      as_chosen = as_chosen.items_of(TILE_PADDED * c.full + c.fixed, ns - 1).items_of(TILE_PADDED * c.last + c.fixed, 1);
  }
  const double chosen_t = launch.estimate(as_chosen, HUGE_VAL, [&] {
    for (int i = 0; i < H; ++i) {
      const int ns = choice->ns[i];
      const Cut c(tiles[i], ns);
      for (int pc = 0; pc < ns; ++pc) {
        const int len = pc + 1 < ns ? c.full : c.last;
        if (n_qp > odd) launch.add(len + c.fixed, n_qp - odd);
        if (odd) launch.add(TILE_PADDED * len + c.fixed, 1);
      }
    }
  });
  const bool is_cut = std::any_of(choice->ns.begin(), choice->ns.end(), [](int n) { return n > 1; });
  double take = BETTER * (chosen_t + (!is_cut ? 0.0 : d == 64 ? CUT_LAUNCH_64 : CUT_LAUNCH_128)) - LONE_LAUNCH;
  auto attempt = [&](int first, int last) {
    // (a sum of differences: the bound it gives may be an ulp off, the simulation decides)
    Load sum = singles[first];
    const Load &mid0 = pairs[first], &mid1 = pairs[H - last], &end0 = singles[H - last], &end1 = singles[H];
    sum.total += mid1.total - mid0.total + end1.total - end0.total;
    sum.items += mid1.items - mid0.items + end1.items - end0.items;
    // (the plan's order is by tokens: among heads of nearly as many a later one may have a tile more)
    for (int i = first; i < H; ++i)
      sum.longest = std::max(sum.longest, (i < H - last && n_qp > odd ? 1.0 : TILE_SINGLE) * tiles[i] + FIXED);
    const double t = launch.estimate(sum, take, [&] {
      for (int i = 0; i < H; ++i) {
        if (i < first || i >= H - last) {
          launch.add(TILE_SINGLE * tiles[i] + FIXED, n_qt);
          continue;
        }
        if (n_qp > odd) launch.add(tiles[i] + FIXED, n_qp - odd);
        if (odd) launch.add(TILE_SINGLE * tiles[i] + FIXED, 1);
      }
    });
    if (t >= take) return;
    take = BETTER * t;
    choice->lone.assign(H, 1);
    std::fill(choice->lone.begin(), choice->lone.begin() + first, 0);
    std::fill(choice->lone.end() - last, choice->lone.end(), 0);
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

static bool valid(const int32_t* tiles, int n_heads, int queries, int n_seq, int n_sm) {
  if (!tiles || n_heads < 1 || queries < 1 || n_seq < 1 || n_sm < 1) return false;
  for (int i = 0; i < n_heads; ++i)
    if (tiles[i] < 1 || (i > 0 && tiles[i] > tiles[i - 1])) return false;
  return true;
}

extern "C" int heatkv_split_plan(const int32_t* tiles, int n_heads, int n_qp, int n_seq, int n_sm, int per_head,
                                 uint64_t max_slots, uint64_t max_ctrs, int32_t* pieces, double* makespan_whole,
                                 double* makespan_cut) {
  if (!pieces || !valid(tiles, n_heads, n_qp, n_seq, n_sm)) return HEATKV_ERR_INVALID_ARG;
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

extern "C" int heatkv_lone_plan(const int32_t* tiles, int n_heads, int t_q, int n_seq, int n_sm, int d, int per_head,
                                uint64_t max_slots, uint64_t max_ctrs, int32_t* pieces, int32_t* singles, int32_t* lone) {
  if (!pieces || !singles || !lone || (d != 64 && d != 128) || !valid(tiles, n_heads, t_q, n_seq, n_sm))
    return HEATKV_ERR_INVALID_ARG;
  try {
    const std::vector<int> t(tiles, tiles + n_heads);
    heatkv::SplitChoice ch = heatkv::split_search(t, (t_q + 255) / 256, n_seq, n_sm, per_head != 0, max_slots, max_ctrs);
    heatkv::single_search(t, t_q, n_seq, n_sm, d, per_head != 0, &ch);
    *lone = !ch.lone.empty();
    for (int i = 0; i < n_heads; ++i) {
      pieces[i] = ch.ns[i];
      singles[i] = *lone && ch.lone[i] == 0;
    }
  } catch (const std::bad_alloc&) {
    return HEATKV_ERR_HOST_MEMORY;
  }
  return HEATKV_OK;
}
