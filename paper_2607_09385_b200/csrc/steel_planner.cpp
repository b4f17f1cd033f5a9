// Host planner: mask descriptor -> executed-tile lists -> work items -> per-CTA assignment.
// Pure host C++ (no CUDA calls), so it is testable on a machine without a GPU.
#include "steel_planner.h"

#include <algorithm>
#include <cmath>
#include <limits>
#include <queue>

namespace steel {
namespace {

constexpr int64_t kInf = std::numeric_limits<int64_t>::max() / 4;

// Geometry of the causal / window terms of the predicate, on token rectangles with inclusive
// bounds that lie inside the problem.  `p = i + off` is the key position aligned with query i.
struct Geom {
  int64_t seq_q, seq_kv, off, window;
  bool causal, windowed;

  bool any_visible(int64_t i0, int64_t i1, int64_t j0, int64_t j1) const {
    // row p sees keys (p - W, p]; it meets [j0, j1] iff j0 <= p (causal) and p <= j1 + W - 1 (window)
    int64_t lb = causal ? j0 : -kInf, ub = windowed ? j1 + window - 1 : kInf;
    return std::max(lb, i0 + off) <= std::min(ub, i1 + off);
  }
  bool all_visible(int64_t i0, int64_t i1, int64_t j0, int64_t j1) const {
    if (causal && !(j1 <= i0 + off)) return false;
    if (windowed && !((i1 + off) - j0 < window)) return false;
    return true;
  }
  int64_t visible_pairs(int64_t i0, int64_t i1, int64_t j0, int64_t j1) const {
    if (all_visible(i0, i1, j0, j1)) return (i1 - i0 + 1) * (j1 - j0 + 1);
    int64_t n = 0;
    for (int64_t i = i0; i <= i1; ++i) {
      int64_t p = i + off;
      int64_t a = std::max(j0, windowed ? p - window + 1 : -kInf), b = std::min(j1, causal ? p : kInf);
      if (b >= a) n += b - a + 1;
    }
    return n;
  }
};

// First and last query position in tile I of a matrix of `rows` rows whose row r holds position r mod seq_q.
void tile_positions(int64_t seq_q, int64_t rows, int64_t I, int64_t *i0, int64_t *i1) {
  const int64_t r0 = I * kTile, r1 = std::min<int64_t>(r0 + kTile, rows) - 1;
  const bool one_head = r0 / seq_q == r1 / seq_q;
  *i0 = one_head ? r0 % seq_q : 0;
  *i1 = one_head ? r1 % seq_q : seq_q - 1;
}

struct Ctx {
  const steel_attn_params_t *p;
  Geom g;
  int64_t bq, bkv;         // descriptor block sizes (64 or 128)
  int64_t tq128, tkv128;   // kernel tiles
  int64_t tqb, tkvb, words;  // descriptor blocks
  bool bitmap;

  bool bit(int h, int64_t I, int64_t J) const {
    if (I >= tqb || J >= tkvb) return false;
    return (p->mask.bitmap[(int64_t(h) * tqb + I) * words + (J >> 5)] >> (J & 31)) & 1u;
  }
  void rows(int64_t I, int64_t size, int64_t &i0, int64_t &i1) const {
    i0 = I * size;
    i1 = std::min<int64_t>(i0 + size - 1, p->seq_q - 1);
  }
  void keys(int64_t J, int64_t size, int64_t &j0, int64_t &j1) const {
    j0 = J * size;
    j1 = std::min<int64_t>(j0 + size - 1, p->seq_kv - 1);
  }
  // First and last tile of `size` keys that queries i0 .. i1 see, and that they see whole, under the causal
  // and window terms (each set is a range; empty if first > last).
  void seen_range(int64_t i0, int64_t i1, int64_t size, int64_t tiles, int64_t *first, int64_t *last) const {
    const int64_t top = g.causal ? i1 + g.off : kInf, bottom = g.windowed ? i0 + g.off - g.window + 1 : 0;
    *last = top < 0 ? -1 : std::min(tiles - 1, top / size);
    *first = bottom > 0 ? bottom / size : 0;
  }
  void whole_range(int64_t i0, int64_t i1, int64_t size, int64_t *first, int64_t *last) const {
    const int64_t top = g.causal ? i0 + g.off : kInf, bottom = g.windowed ? i1 + g.off - g.window + 1 : 0;
    *last = top < 0 ? -1 : (std::min<int64_t>(top, p->seq_kv - 1) + 1) / size - 1;
    if (top >= p->seq_kv - 1) *last = (p->seq_kv - 1) / size;  // a ragged last tile is seen whole
    *first = bottom > 0 ? (bottom + size - 1) / size : 0;
  }
  // Bits first .. last of the word that holds bits 32 w .. 32 w + 31.
  static uint32_t range_bits(int64_t w, int64_t first, int64_t last) {
    const int64_t a = std::max<int64_t>(first - 32 * w, 0), b = std::min<int64_t>(last - 32 * w, 31);
    return a > b ? 0u : (0xFFFFFFFFu >> (31 - (b - a))) << a;
  }

  // Bitmap masks: the entries of query tile I of head h, fully masked tiles (case i) left out.  Word by word:
  // one tile at a time took most of the planning (8 heads x 4096 tokens, 64-token blocks, plan of the allocation-free
  // call without statistics, on the host of a B200: 416 us in all, now 75).
  void entries(int h, int64_t I, std::vector<uint32_t> *out) const {
    int64_t i0, i1, whole_lo, whole_hi;
    rows(I, kTile, i0, i1);
    whole_range(i0, i1, kTile, &whole_lo, &whole_hi);
    const bool ragged = p->seq_kv % kTile != 0;
    kept_words(h, I, [&](int64_t w, uint32_t inside, const uint32_t (&set)[2], bool two_rows, uint32_t kept) {
      const int per = int(kTile / bq);
      for (; kept; kept &= kept - 1) {
        const int bit0 = __builtin_ctz(kept);
        const int64_t J = (32 * w + bit0) / per;
        uint32_t sub = 0xF;
        bool full = J >= whole_lo && J <= whole_hi;
        if (per == 2) {  // sub-blocks TL, TR, BL, BR; those outside the problem do not make a tile partial
          const uint32_t a = (set[0] >> bit0) & 3u, b = (set[1] >> bit0) & 3u, in = (inside >> bit0) & 3u;
          sub = a | b << 2;
          full = full && a == in && (!two_rows || b == in);
        }
        uint32_t e = uint32_t(J) | kEntryPresent | (sub << kEntrySubShift);
        if (!full || (ragged && J == tkv128 - 1)) e |= kEntryPartial;
        out->push_back(e);
      }
    });
  }
  // Their number.
  int64_t count_entries(int h, int64_t I) const {
    int64_t n = 0;
    kept_words(h, I, [&](int64_t, uint32_t, const uint32_t (&)[2], bool, uint32_t kept) { n += __builtin_popcount(kept); });
    return n;
  }

  // The words of query tile I's blocks that hold visible ones: visit(word, bits inside the problem, bits of the tile's
  // rows of blocks, whether there are two, one bit per visible key tile).
  template <class Visit>
  void kept_words(int h, int64_t I, Visit &&visit) const {
    const int per = int(kTile / bq);  // blocks of a tile in each direction: 1 or 2
    const uint32_t *row[2] = {nullptr, nullptr};
    int64_t lo[2] = {0, 0}, hi[2] = {-1, -1};
    for (int a = 0; a < per && per * I + a < tqb; ++a) {
      row[a] = p->mask.bitmap + (int64_t(h) * tqb + per * I + a) * words;
      int64_t r0, r1;
      rows(per * I + a, bq, r0, r1);
      seen_range(r0, r1, bq, tkvb, &lo[a], &hi[a]);
    }
    const int64_t w_first = (per == 1 ? lo[0] : std::min(lo[0], row[1] ? lo[1] : lo[0])) / 32;
    const int64_t w_last = std::max(hi[0], hi[1]) / 32;
    if (std::max(hi[0], hi[1]) < 0) return;
    for (int64_t w = w_first; w <= w_last; ++w) {
      const uint32_t inside = range_bits(w, 0, tkvb - 1);
      uint32_t set[2] = {0u, 0u}, kept = 0u;
      for (int a = 0; a < per; ++a)
        if (row[a]) {
          set[a] = row[a][w] & inside;
          kept |= set[a] & range_bits(w, lo[a], hi[a]);
        }
      if (per == 2) kept = (kept | kept >> 1) & 0x55555555u;
      visit(w, inside, set, row[1] != nullptr, kept);
    }
  }
};

// Key tiles lo .. hi (empty if lo > hi) that query tile I of a matrix of `rows` rows sees under the causal
// and window terms; `rows` is seq_q, or a multiple of it where the matrix holds several heads.
void key_range(const Ctx &c, int64_t rows, int64_t I, int64_t *lo, int64_t *hi) {
  int64_t i0, i1;
  tile_positions(c.p->seq_q, rows, I, &i0, &i1);
  const int64_t p0 = i0 + c.g.off, p1 = i1 + c.g.off;
  *hi = c.g.causal ? std::min<int64_t>(c.tkv128 - 1, p1 >= 0 ? p1 / kTile : -1) : c.tkv128 - 1;
  *lo = 0;
  if (c.g.windowed) {
    const int64_t first_key = p0 - c.g.window + 1;
    *lo = first_key > 0 ? first_key / kTile : 0;
  }
  auto seen = [&](int64_t J) {
    return c.g.any_visible(i0, i1, J * kTile, std::min<int64_t>(J * kTile + kTile, c.p->seq_kv) - 1);
  };
  while (*lo <= *hi && !seen(*lo)) ++*lo;
  while (*hi >= *lo && !seen(*hi)) --*hi;
}

struct Task {  // one query tile of one head (packed: of one group of heads)
  int h;
  int64_t I;
  int64_t jlo = 0, jhi = -1;      // range kind
  // list kind: the task's stretch of one array for all tasks (a heap block each took longer than the rest)
  struct Entries {
    const uint32_t *first = nullptr;
    size_t n = 0, at = 0;  // `at`: offset in the array, while that grows
    size_t size() const { return n; }
    bool empty() const { return n == 0; }
    uint32_t operator[](size_t i) const { return first[i]; }
    const uint32_t *begin() const { return first; }
    const uint32_t *end() const { return first + n; }
  } entries;
  int64_t count() const { return entries.empty() ? jhi - jlo + 1 : int64_t(entries.size()); }
};

bool slot_used(const WorkItem &w, int s) { return w.head[s] >= 0 && w.hi[s] >= w.lo[s]; }

double step_cost(const WorkItem &w) { return slot_used(w, 0) && slot_used(w, 1) ? 1.0 : kSingleStep; }

// Load of the busiest CTA, in steps of two slots, with the longest item first to the least loaded CTA.
double makespan(std::vector<double> cost, int num_ctas) {
  std::sort(cost.begin(), cost.end(), std::greater<double>());
  std::priority_queue<double, std::vector<double>, std::greater<double>> load;
  for (int n = 0; n < num_ctas; ++n) load.push(0.0);
  double most = 0.0;
  for (double x : cost) {
    x += load.top();
    load.pop();
    load.push(x);
    most = std::max(most, x);
  }
  return most;
}

double makespan(const std::vector<Draft> &drafts, int num_ctas) {
  std::vector<double> cost;
  cost.reserve(drafts.size());
  for (const Draft &d : drafts) cost.push_back(step_cost(d.w) * d.w.n_steps + kItemOverheadSteps);
  return makespan(std::move(cost), num_ctas);
}

// Steps [t0, t1) of `d`.  A draft of one query tile becomes a piece whose slots walk the two halves of the
// range, so that one slot's softmax runs beside the other's products.
Draft cut_piece(const Draft &d, int t0, int t1) {
  Draft r;
  r.w = d.w;
  r.group = d.group;
  WorkItem &w = r.w;
  if (!slot_used(d.w, 1)) {
    const int n0 = (t1 - t0 + 1) / 2, n1 = t1 - t0 - n0;
    w.head[1] = n1 ? d.w.head[0] : -1;
    w.qtile[1] = d.w.qtile[0];
    w.lo[0] = 0;
    w.hi[0] = n0 - 1;
    w.lo[1] = n1 ? 0 : 1;
    w.hi[1] = n1 ? n1 - 1 : 0;
    w.n_steps = n0;
    if (d.w.kind == 0) {
      w.j0[0] = d.w.j0[0] + t0;
      w.j0[1] = d.w.j0[0] + t0 + n0;
    } else {
      for (int t = 0; t < n0; ++t)
        r.list.push_back(StepPair{{d.list[t0 + t].e[0], t < n1 ? d.list[t0 + n0 + t].e[0] : 0u}});
    }
    return r;
  }
  int n = 0;
  for (int s = 0; s < 2; ++s) {  // a slot absent from these steps drops out; the other one is then slot 0
    const int lo = std::max(d.w.lo[s], t0), hi = std::min(d.w.hi[s], t1 - 1);
    if (lo > hi) continue;
    w.head[n] = d.w.head[s];
    w.qtile[n] = d.w.qtile[s];
    w.lo[n] = lo - t0;
    w.hi[n] = hi - t0;
    if (d.w.kind == 0) w.j0[n] = d.w.j0[s] + t0;
    for (int t = t0; d.w.kind == 1 && t < t1; ++t) {
      if (n == 0) r.list.push_back(StepPair{{d.list[t].e[s], 0u}});
      else r.list[t - t0].e[1] = d.list[t].e[s];
    }
    ++n;
  }
  if (n == 1) {
    w.head[1] = -1;
    w.lo[1] = 1;
    w.hi[1] = 0;
  }
  w.n_steps = std::max(w.hi[0], n == 2 ? w.hi[1] : 0) + 1;
  return r;
}

// Steps [t0, t1) of a draft, or all of it as it is, for one CTA.
struct Share {
  int32_t draft, t0, t1, cta;
  bool whole;
};

// Deal the drafts' steps, in order, into one share of at most `quota` per CTA (a piece of a draft at either end
// of a share).  False if the shares do not suffice.  Only the numbers: the pieces are made once the quota is found
// (made at every step of the search they took half of the planning: bitmap, 4 heads x 8192, 749 us in all, now 392).
bool deal_shares(const std::vector<Draft> &drafts, int num_ctas, double quota, double fill, std::vector<Share> *shares) {
  const double overhead = kPieceOverheadSteps + part_write_steps(fill);
  int cta = 0;
  double left = quota;
  auto next_share = [&] {
    ++cta;
    left = quota;
  };
  for (size_t id = 0; id < drafts.size(); ++id) {
    const Draft &d = drafts[id];
    const bool one = !slot_used(d.w, 1);
    const double w = one ? 0.5 : 1.0;
    const int n = d.w.n_steps, per_step = one ? 1 : 2;
    // at most kMaxParts parts of one query tile (two per piece)
    const int least = std::max<int>(min_piece_tiles(fill) / per_step, (n + kMaxParts / 2 - 1) / (kMaxParts / 2));
    int t = 0;
    do {
      int take = std::max(0, int((left - overhead) / w));
      if (take < std::min(least, n - t) && left < quota) {  // the rest of this share is too short
        next_share();
        continue;
      }
      take = std::max(take, least);
      if (n - t - take < least) take = n - t;
      if (cta >= num_ctas) return false;
      // a tile with few rows in use is worth two parts even within one CTA
      const bool whole = take == n && !(one && fill <= 0.25 && n >= 2 * least);
      shares->push_back(Share{int32_t(id), t, t + take, cta, whole});
      left -= (whole && one ? kSingleStep : w) * take + (whole ? kPieceOverheadSteps : overhead);
      if (left <= overhead) next_share();
      t += take;
    } while (t < n);
  }
  return true;
}

// The pieces of dealt drafts, and the numbers of the parts of the query tiles that were cut.
void make_pieces(const std::vector<Draft> &drafts, const std::vector<Share> &shares, std::vector<Draft> *pieces,
                 Plan *plan) {
  pieces->reserve(shares.size());
  for (size_t k = 0; k < shares.size();) {
    const size_t first = pieces->size();
    const Draft &d = drafts[shares[k].draft];
    const bool one = !slot_used(d.w, 1);
    for (const int32_t id = shares[k].draft; k < shares.size() && shares[k].draft == id; ++k) {
      pieces->push_back(shares[k].whole ? d : cut_piece(d, shares[k].t0, shares[k].t1));
      pieces->back().cta = shares[k].cta;
    }
    if (pieces->size() == first + 1 && !(one && slot_used(pieces->back().w, 1))) continue;
    // the parts of each query tile are all slots of its pieces that hold it
    for (int s = 0; s < (one ? 1 : 2); ++s) {
      SplitTile tile{plan->n_parts, 0};
      const int32_t id = int32_t(plan->split_tiles.size());
      int32_t *only = nullptr;
      for (size_t n = first; n < pieces->size(); ++n)
        for (int u = 0; u < 2; ++u) {
          WorkItem &x = (*pieces)[n].w;
          if (slot_used(x, u) && x.head[u] == d.w.head[s] && x.qtile[u] == d.w.qtile[s]) {
            only = &x.split[u];
            *only = split_code(id, tile.n_parts++);
          }
        }
      if (tile.n_parts > 1) {
        plan->split_tiles.push_back(tile);
        plan->n_parts += tile.n_parts;
      } else if (only) {
        *only = -1;
      }
    }
  }
}

// Cut the drafts over the CTAs with the smallest share that works, to 3 %.  Returns the load of the busiest CTA, or
// infinity where nothing was cut.
double cut_over_ctas(const std::vector<Draft> &drafts, int num_ctas, double fill, std::vector<Draft> *pieces,
                     Plan *plan) {
  double work = 0.0;
  size_t live = 0;
  for (const Draft &d : drafts) {
    work += (slot_used(d.w, 1) ? 1.0 : 0.5) * d.w.n_steps;
    live += d.w.n_steps > 0;
  }
  double quota = (work + kPieceOverheadSteps * double(std::max<size_t>(live, num_ctas))) / num_ctas;
  std::vector<Share> shares;
  while (!deal_shares(drafts, num_ctas, quota, fill, &shares)) {
    quota *= 1.03;
    shares.clear();
  }
  make_pieces(drafts, shares, pieces, plan);
  if (plan->split_tiles.empty()) return std::numeric_limits<double>::infinity();
  std::vector<double> load(num_ctas, 0.0);
  int most_parts = 0;
  for (const Draft &d : *pieces)
    load[d.cta] += step_cost(d.w) * d.w.n_steps + kPieceOverheadSteps +
                   (d.w.split[0] >= 0 || d.w.split[1] >= 0 ? part_write_steps(fill) : 0.0);
  for (const SplitTile &t : plan->split_tiles) most_parts = std::max(most_parts, t.n_parts);
  return *std::max_element(load.begin(), load.end()) + combine_steps(fill, most_parts);
}

// Statistics of the executed tiles.  Ranges are counted as such: visiting every tile of them took most of the
// planning of long sequences (32/8 heads x 131072: 143 ms in all, now 4).
void count_tiles(const Ctx &c, const Plan &plan, int64_t rows, steel_attn_stats_t *s) {
  for (const WorkItem &w : plan.items) {
    if (w.kind == 1) {
      for (int t = 0; t < w.n_steps; ++t) {
        const StepPair &pair = plan.steps[size_t(w.j0[0]) + size_t(t)];
        const bool in0 = pair.e[0] != 0, in1 = pair.e[1] != 0;
        const bool shared = in0 && in1 && (pair.e[0] & kEntryTileMask) == (pair.e[1] & kEntryTileMask);
        s->exec_tiles += in0 + in1;
        s->exec_partial += ((pair.e[0] & kEntryPartial) != 0) + ((pair.e[1] & kEntryPartial) != 0);
        s->kv_tile_loads += in0 + in1 - shared;
      }
      continue;
    }
    int64_t tiles = 0, shared = 0;
    for (int u = 0; u < 2; ++u) {
      if (!slot_used(w, u)) continue;
      tiles += w.hi[u] - w.lo[u] + 1;
      // those seen whole, and not ragged
      int64_t i0, i1, first, last;
      tile_positions(c.p->seq_q, rows, w.qtile[u], &i0, &i1);
      c.whole_range(i0, i1, kTile, &first, &last);
      if (c.p->seq_kv % kTile) last = std::min(last, c.tkv128 - 2);
      first = std::max<int64_t>(first, int64_t(w.j0[u]) + w.lo[u]);
      last = std::min<int64_t>(last, int64_t(w.j0[u]) + w.hi[u]);
      s->exec_partial += w.hi[u] - w.lo[u] + 1 - std::max<int64_t>(0, last - first + 1);
    }
    if (slot_used(w, 0) && slot_used(w, 1) && w.j0[0] == w.j0[1])
      shared = std::max(0, std::min(w.hi[0], w.hi[1]) - std::max(w.lo[0], w.lo[1]) + 1);
    s->exec_tiles += tiles;
    s->kv_tile_loads += tiles - shared;
  }
}

// Order the drafts, assign them to CTAs and write the plan's lists and the statistics of its items.
steel_status_t place_items(const steel_attn_params_t &p, int num_ctas, std::vector<Draft> &drafts, Plan *plan) {
  // ---- order: waves of KV heads whose K and V fit comfortably in L2, longest item first inside
  // a wave (policy 0); natural order (policy 1)
  std::vector<int> order(drafts.size());
  for (size_t n = 0; n < order.size(); ++n) order[n] = int(n);
  const int policy = p.policy;
  if (policy == 0) {
    const double kv_bytes_per_head = 2.0 * double(p.seq_kv) * p.head_dim * 2.0;
    int heads_per_wave = int(std::max(1.0, std::floor(double(kL2WaveBytes) / kv_bytes_per_head)));
    struct Key {
      int64_t wave;
      int32_t n_steps, id;
    };
    std::vector<Key> keys(drafts.size());
    for (size_t n = 0; n < keys.size(); ++n) {
      const Draft &d = drafts[n];
      keys[n] = Key{(int64_t(d.w.batch) * p.heads_kv + d.group) / heads_per_wave, d.w.n_steps, int32_t(n)};
    }
    std::sort(keys.begin(), keys.end(), [](const Key &a, const Key &b) {
      if (a.wave != b.wave) return a.wave < b.wave;
      if (a.n_steps != b.n_steps) return a.n_steps > b.n_steps;
      return a.id < b.id;
    });
    for (size_t n = 0; n < keys.size(); ++n) order[n] = keys[n].id;
  }

  // ---- assignment to persistent CTAs
  int grid = int(std::min<size_t>(size_t(num_ctas), std::max<size_t>(drafts.size(), 1)));
  std::vector<std::vector<int>> per_cta(grid);
  std::vector<int64_t> load(grid, 0);
  if (!plan->split_tiles.empty()) {
    grid = num_ctas;
    per_cta.resize(grid);
    load.resize(grid, 0);
    for (size_t id = 0; id < drafts.size(); ++id) per_cta[drafts[id].cta].push_back(int(id));
  } else if (policy == 0) {
    // greedy longest-processing-time: next item goes to the least loaded CTA
    typedef std::pair<int64_t, int> Slot;
    std::priority_queue<Slot, std::vector<Slot>, std::greater<Slot>> heap;
    for (int cta = 0; cta < grid; ++cta) heap.push(Slot(0, cta));
    for (int id : order) {
      Slot sl = heap.top();
      heap.pop();
      per_cta[sl.second].push_back(id);
      sl.first += drafts[id].w.n_steps + kItemOverheadSteps;
      load[sl.second] = sl.first;
      heap.push(sl);
    }
  } else if (policy == 1) {
    // uniform placement: contiguous chunks of the natural order
    size_t n = order.size();
    for (size_t k = 0; k < n; ++k) {
      int cta = int(k * size_t(grid) / std::max<size_t>(n, 1));
      per_cta[cta].push_back(order[k]);
      load[cta] += drafts[order[k]].w.n_steps + kItemOverheadSteps;
    }
  } else {
    // interleaved placement: consecutive items of the natural order go to consecutive CTAs, so
    // that CTAs working side by side hold query tiles of similar sparsity
    for (size_t k = 0; k < order.size(); ++k) {
      int cta = int(k % size_t(grid));
      per_cta[cta].push_back(order[k]);
      load[cta] += drafts[order[k]].w.n_steps + kItemOverheadSteps;
    }
  }

  size_t n_steps = 0;
  for (const Draft &d : drafts) n_steps += d.list.size();
  plan->steps.reserve(n_steps);
  plan->items.reserve(drafts.size());
  plan->grid = grid;
  plan->cta_begin.push_back(0);
  for (int cta = 0; cta < grid; ++cta) {
    for (int id : per_cta[cta]) {
      Draft &d = drafts[id];
      if (d.w.kind == 1) {
        d.w.j0[0] = int32_t(plan->n_steps);
        plan->n_steps += d.list.empty() ? int64_t(d.w.n_steps) : int64_t(d.list.size());
        plan->steps.insert(plan->steps.end(), d.list.begin(), d.list.end());
      }
      plan->items.push_back(d.w);
    }
    plan->cta_begin.push_back(int32_t(plan->items.size()));
  }
  if (plan->n_steps >= (int64_t(1) << 31)) return STEEL_ERR_UNSUPPORTED;

  // ---- statistics of the executed plan
  steel_attn_stats_t &s = plan->stats;
  s.work_items = int64_t(plan->items.size());
  s.grid = grid;
  s.list_entries = plan->n_steps;
  s.max_cta_steps = 0;
  for (int cta = 0; cta < grid; ++cta) {
    int64_t st_sum = 0;
    for (int id : per_cta[cta]) st_sum += drafts[id].w.n_steps;
    s.max_cta_steps = std::max(s.max_cta_steps, st_sum);
  }
  for (const WorkItem &w : plan->items) s.steps += w.n_steps;
  return STEEL_OK;
}

}  // namespace

steel_status_t validate_params(const steel_attn_params_t *p) {
  if (!p) return STEEL_ERR_INVALID_ARG;
  if (p->batch <= 0 || p->heads_q <= 0 || p->heads_kv <= 0 || p->seq_q <= 0 || p->seq_kv <= 0 || p->head_dim <= 0)
    return STEEL_ERR_INVALID_ARG;
  if (p->heads_q % p->heads_kv != 0) return STEEL_ERR_INVALID_ARG;
  if (!(p->scale > 0.0f) || !std::isfinite(p->scale)) return STEEL_ERR_INVALID_ARG;
  const uint32_t known = STEEL_MASK_CAUSAL | STEEL_MASK_WINDOW | STEEL_MASK_BITMAP;
  if (p->mask.flags & ~known) return STEEL_ERR_INVALID_ARG;
  if ((p->mask.flags & STEEL_MASK_WINDOW) && p->mask.window <= 0) return STEEL_ERR_INVALID_ARG;
  if ((p->mask.flags & STEEL_MASK_BITMAP) && !p->mask.bitmap) return STEEL_ERR_INVALID_ARG;
  if (p->mask.block_q < 0 || p->mask.block_kv < 0) return STEEL_ERR_INVALID_ARG;
  if (p->policy < 0 || p->policy > 2 || p->exp_emulation < 0 || p->exp_emulation > 3) return STEEL_ERR_INVALID_ARG;
  if (p->head_dim != 64 && p->head_dim != 128) return STEEL_ERR_UNSUPPORTED;
  int bq = p->mask.block_q ? p->mask.block_q : kTile, bkv = p->mask.block_kv ? p->mask.block_kv : kTile;
  if (bq != bkv || (bq != 64 && bq != 128)) return STEEL_ERR_UNSUPPORTED;
  if ((int64_t(p->seq_kv) + kTile - 1) / kTile > (int64_t(1) << 24)) return STEEL_ERR_UNSUPPORTED;
  if (p->seq_q > (1 << 30) || p->seq_kv > (1 << 30)) return STEEL_ERR_UNSUPPORTED;
  if (int64_t(p->batch) * p->heads_q * p->seq_q >= (int64_t(1) << 31)) return STEEL_ERR_UNSUPPORTED;
  if (int64_t(p->batch) * p->heads_kv * p->seq_kv >= (int64_t(1) << 31)) return STEEL_ERR_UNSUPPORTED;
  return STEEL_OK;
}

steel_status_t build_plan(const steel_attn_params_t *p, int num_ctas, Plan *plan, bool stats, Spread spread,
                          Plan *whole, bool device_lists) {
  steel_status_t st = validate_params(p);
  if (st != STEEL_OK) return st;
  const int policy = p->policy;
  if (num_ctas <= 0 || !plan) return STEEL_ERR_INVALID_ARG;

  Ctx c;
  c.p = p;
  c.bitmap = (p->mask.flags & STEEL_MASK_BITMAP) != 0;
  c.g = Geom{p->seq_q, p->seq_kv, int64_t(p->seq_kv) - p->seq_q, p->mask.window,
             (p->mask.flags & STEEL_MASK_CAUSAL) != 0, (p->mask.flags & STEEL_MASK_WINDOW) != 0};
  c.bq = p->mask.block_q ? p->mask.block_q : kTile;
  c.bkv = p->mask.block_kv ? p->mask.block_kv : kTile;
  c.tq128 = (p->seq_q + kTile - 1) / kTile;
  c.tkv128 = (p->seq_kv + kTile - 1) / kTile;
  c.tqb = (p->seq_q + c.bq - 1) / c.bq;
  c.tkvb = (p->seq_kv + c.bkv - 1) / c.bkv;
  c.words = (c.tkvb + 31) / 32;
  int G = p->heads_q / p->heads_kv;  // heads (matrices of Q) that share a KV head
  int heads = p->heads_q;
  if (policy != 0) spread = Spread::kNone;

  plan->items.clear();
  plan->steps.clear();
  plan->n_steps = 0;
  plan->split_tiles.clear();
  plan->n_parts = 0;
  plan->packed = false;
  plan->cta_begin.clear();
  steel_attn_stats_t &s = plan->stats;
  s = steel_attn_stats_t{};

  // ---- statistics at the descriptor's block granularity (what "kept tiles" means to a caller)
  if (stats) {
    int64_t kept = 0, partial = 0;
    double pairs = 0.0;
    for (int h = 0; h < p->heads_q; ++h) {
      if (!c.bitmap && h > 0) break;  // range masks are identical for every head
      for (int64_t I = 0; I < c.tqb; ++I) {
        int64_t i0, i1;
        c.rows(I, c.bq, i0, i1);
        for (int64_t J = 0; J < c.tkvb; ++J) {
          if (c.bitmap && !c.bit(h, I, J)) continue;
          int64_t j0, j1;
          c.keys(J, c.bkv, j0, j1);
          if (!c.g.any_visible(i0, i1, j0, j1)) {
            if (!c.bitmap && c.g.causal && j0 > i1 + c.g.off) break;  // rest of the row is empty
            continue;
          }
          ++kept;
          bool full = c.g.all_visible(i0, i1, j0, j1);
          partial += !full;
          pairs += full ? double((i1 - i0 + 1) * (j1 - j0 + 1)) : double(c.g.visible_pairs(i0, i1, j0, j1));
        }
      }
    }
    int64_t mult = int64_t(p->batch) * (c.bitmap ? 1 : p->heads_q);
    s.kept_tiles = kept * mult;
    s.partial_tiles = partial * mult;
    s.total_tiles = int64_t(p->batch) * p->heads_q * c.tqb * c.tkvb;
    s.effective_flop = 4.0 * double(c.bq) * double(c.bkv) * p->head_dim * double(s.kept_tiles);
    s.useful_flop = 4.0 * p->head_dim * pairs * double(mult);
  }

  // ---- per (head, query tile) executed key tiles
  // Heads of a group lie one behind the other in Q, O and LSE, so their rows form one matrix of G * seq_q
  // rows.  Few queries per head leave most of a head's last tile empty (a decode step: 127 of 128 rows);
  // tiles over that matrix are then fewer.  A tile that holds the end of one head and the start of the next
  // spans all positions, which costs key tiles under a causal mask: taken only where the total is smaller.
  if (spread != Spread::kNone && !c.bitmap && G > 1) {
    auto executed = [&](bool packed) {
      const int64_t rows = packed ? int64_t(G) * p->seq_q : p->seq_q;
      int64_t n = 0, lo, hi;
      for (int64_t I = 0; I * kTile < rows; ++I) {
        key_range(c, rows, I, &lo, &hi);
        n += std::max<int64_t>(0, hi - lo + 1);
      }
      return packed ? n : n * G;
    };
    // with more than 8 tiles per head a shared tile saves less than one in eight
    if (c.tq128 <= 8 && executed(true) < executed(false)) {
      plan->packed = true;
      c.tq128 = (int64_t(G) * p->seq_q + kTile - 1) / kTile;
      heads = p->heads_kv;
      G = 1;
    }
  }
  const int64_t rows_q = plan_rows_q(*p, *plan);
  std::vector<std::vector<Task>> tasks(heads);  // [h][I]
  // Bitmap masks: the search for partners takes most of the planning, so where no key range may be cut the
  // choice between pairs and single tiles is made on the lengths alone (partners are of similar length).
  const bool on_lengths = spread == Spread::kTiles && c.bitmap && int64_t(p->batch) * heads * c.tq128 < 8 * num_ctas;
  for (int h = 0; h < heads; ++h) {
    tasks[h].resize(c.tq128);
    for (int64_t I = 0; I < c.tq128; ++I) {
      Task &t = tasks[h][I];
      t.h = h;
      t.I = I;
      if (on_lengths) {
        t.entries.n = size_t(c.count_entries(h, I));
      } else if (!c.bitmap && h > 0) {
        t.jlo = tasks[0][I].jlo;
        t.jhi = tasks[0][I].jhi;
      } else if (!c.bitmap) {
        // kept key tiles of a row of tiles form one contiguous range under causal / window masks
        key_range(c, rows_q, I, &t.jlo, &t.jhi);
      }
    }
  }
  bool pair = true;
  int64_t n_lists = 0, n_entries = 0;  // of single query tiles
  if (on_lengths) {
    std::vector<double> paired, single;
    double work = 0.0;
    std::vector<int64_t> count;
    for (int g = 0; g < p->heads_kv; ++g) {
      count.clear();
      for (int h = g * G; h < (g + 1) * G; ++h)
        for (const Task &t : tasks[h])
          if (t.count() > 0) count.push_back(t.count());
      std::sort(count.begin(), count.end(), std::greater<int64_t>());
      for (int batch = 0; batch < p->batch; ++batch)
        for (size_t n = 0; n < count.size(); ++n) {
          single.push_back(kSingleStep * double(count[n]) + kItemOverheadSteps);
          ++n_lists;
          n_entries += count[n];
          if (n % 2) continue;
          paired.push_back((n + 1 < count.size() ? 1.0 : kSingleStep) * double(count[n]) + kItemOverheadSteps);
          work += paired.back();
        }
    }
    const double load = makespan(std::move(paired), num_ctas);
    pair = !(load > 1.1 * work / num_ctas && makespan(std::move(single), num_ctas) < 0.95 * load);
  }
  device_lists = device_lists && on_lengths && !pair && !stats && lists_on_device(n_lists, n_entries);
  const size_t key_words = size_t(c.tkv128 + 63) / 64;
  std::vector<uint32_t> entries;
  std::vector<uint64_t> keys;  // the key tiles of each task as bits
  if (c.bitmap && !device_lists) {
    keys.assign(size_t(heads) * size_t(c.tq128) * key_words, 0);
    for (int h = 0; h < heads; ++h)
      for (int64_t I = 0; I < c.tq128; ++I) {
        Task &t = tasks[h][I];
        t.entries.at = entries.size();
        c.entries(h, I, &entries);
        t.entries.n = entries.size() - t.entries.at;
        for (size_t n = t.entries.at; n < entries.size(); ++n) {
          const uint32_t J = entries[n] & kEntryTileMask;
          keys[size_t(h * c.tq128 + I) * key_words + J / 64] |= uint64_t(1) << (J % 64);
        }
      }
    for (std::vector<Task> &row : tasks)
      for (Task &t : row) t.entries.first = entries.data() + t.entries.at;
  }

  // ---- work items: pair query tiles that can share K/V loads
  std::vector<Draft> drafts, uncut;  // `uncut`: for `whole`
  auto finish_range = [&](const Task *a, const Task *b, int batch, int g) {
    Draft d{};
    d.group = g;
    WorkItem &w = d.w;
    w.batch = batch;
    w.kv_head = g;
    w.kind = 0;
    w.head[0] = a->h;
    w.qtile[0] = int32_t(a->I);
    w.head[1] = b ? b->h : -1;
    w.qtile[1] = b ? int32_t(b->I) : 0;
    w.j0[0] = w.j0[1] = int32_t(a->jlo);
    w.split[0] = w.split[1] = -1;
    w.lo[0] = 0;
    w.hi[0] = int32_t(a->jhi - a->jlo);
    w.lo[1] = 1;
    w.hi[1] = 0;
    if (b) {
      w.lo[1] = int32_t(b->jlo - a->jlo);
      w.hi[1] = int32_t(b->jhi - a->jlo);
    }
    w.n_steps = std::max(w.hi[0], w.hi[1]) + 1;
    drafts.push_back(std::move(d));
  };
  std::vector<uint32_t> ea, eb, rest_a, rest_b;  // of finish_list
  auto finish_list = [&](const Task *a, const Task *b, int batch, int g) {
    Draft d{};
    d.group = g;
    WorkItem &w = d.w;
    w.batch = batch;
    w.kv_head = g;
    w.kind = 1;
    w.head[0] = a->h;
    w.qtile[0] = int32_t(a->I);
    w.head[1] = b ? b->h : -1;
    w.qtile[1] = b ? int32_t(b->I) : 0;
    w.split[0] = w.split[1] = -1;
    size_t na = a->entries.size(), nb = b ? b->entries.size() : 0;
    w.lo[0] = 0;
    w.hi[0] = int32_t(na) - 1;
    w.lo[1] = b ? 0 : 1;
    w.hi[1] = b ? int32_t(nb) - 1 : 0;
    w.n_steps = int32_t(std::max(na, nb));
    // Key tiles may be visited in any order (the online softmax does not care), so the tiles both
    // query tiles want come first, in the same steps: each of those steps needs one K/V load, not two.
    ea.clear();
    eb.clear();
    if (b) {
      rest_a.clear();
      rest_b.clear();
      size_t ia = 0, ib = 0;
      while (ia < na || ib < nb) {
        const uint32_t ta = ia < na ? (a->entries[ia] & kEntryTileMask) : 0xFFFFFFFFu;
        const uint32_t tb = ib < nb ? (b->entries[ib] & kEntryTileMask) : 0xFFFFFFFFu;
        if (ta == tb) {
          ea.push_back(a->entries[ia++]);
          eb.push_back(b->entries[ib++]);
        } else if (ta < tb) {
          rest_a.push_back(a->entries[ia++]);
        } else {
          rest_b.push_back(b->entries[ib++]);
        }
      }
      ea.insert(ea.end(), rest_a.begin(), rest_a.end());
      eb.insert(eb.end(), rest_b.begin(), rest_b.end());
    } else {
      if (!device_lists) {
        d.list.reserve(na);
        for (uint32_t e : a->entries) d.list.push_back(StepPair{{e, 0u}});
      }
      drafts.push_back(std::move(d));
      return;
    }
    d.list.reserve(size_t(w.n_steps));
    for (size_t t = 0; t < size_t(w.n_steps); ++t)
      d.list.push_back(StepPair{{t < na ? ea[t] : 0u, t < nb ? eb[t] : 0u}});
    drafts.push_back(std::move(d));
  };
  auto empty_item = [&](const Task *a, int batch, int g) {  // no visible key: rows get O = 0, LSE = -inf
    Draft d{};
    d.group = g;
    WorkItem &w = d.w;
    w.batch = batch;
    w.kv_head = g;
    w.kind = 0;
    w.head[0] = a->h;
    w.qtile[0] = int32_t(a->I);
    w.head[1] = -1;
    w.split[0] = w.split[1] = -1;
    w.lo[0] = 0;
    w.hi[0] = -1;
    w.lo[1] = 1;
    w.hi[1] = 0;
    w.n_steps = 0;
    drafts.push_back(std::move(d));
  };

  auto build_drafts = [&] {
    drafts.clear();
    for (int batch = 0; batch < p->batch; ++batch) {
      for (int g = 0; g < p->heads_kv; ++g) {
        std::vector<const Task *> live;
        for (int h = g * G; h < (g + 1) * G; ++h)
          for (int64_t I = 0; I < c.tq128; ++I) {
            const Task *t = &tasks[h][I];
            if (t->count() <= 0) empty_item(t, batch, g);
            else live.push_back(t);
          }
        if (c.bitmap) {
          // similar lengths pair best: both tiles of an item then finish together
          struct Length {
            int64_t n;
            const uint64_t *keys;
            const Task *task;
          };
          std::vector<Length> by_length;
          by_length.reserve(live.size());
          for (const Task *t : live)
            by_length.push_back({t->count(), pair ? &keys[size_t(t->h * c.tq128 + t->I) * key_words] : nullptr, t});
          if (pair)
            std::stable_sort(by_length.begin(), by_length.end(), [](const Length &a, const Length &b) { return a.n > b.n; });
          // among the next few tasks of similar length, take the partner with the most key tiles in common
          std::vector<char> used(live.size(), 0);
          for (size_t n = 0; n < live.size(); ++n) {
            if (used[n]) continue;
            used[n] = 1;
            const Length &a = by_length[n];
            size_t best = live.size(), seen = 0;
            int64_t best_common = 0;
            for (size_t m = n + 1; pair && m < live.size() && seen < kPartnerWindow; ++m) {
              if (used[m]) continue;
              ++seen;
              const Length &b = by_length[m];
              int64_t common = 0;
              for (size_t w = 0; w < key_words; ++w) common += __builtin_popcountll(a.keys[w] & b.keys[w]);
              // a step with one idle slot costs far more than a shared load saves
              const int64_t score = common - 16 * (a.n - b.n);
              if (score > best_common || best == live.size()) { best_common = score; best = m; }
            }
            if (best < live.size()) used[best] = 1;
            finish_list(a.task, best < live.size() ? by_length[best].task : nullptr, batch, g);
          }
        } else if (!pair) {
          for (const Task *t : live) finish_range(t, nullptr, batch, g);
        } else if (G % 2 == 0) {
          // two query heads of the group on the same query tile: identical key ranges
          for (int h = g * G; h < (g + 1) * G; h += 2)
            for (int64_t I = 0; I < c.tq128; ++I)
              if (tasks[h][I].count() > 0) finish_range(&tasks[h][I], &tasks[h + 1][I], batch, g);
        } else {
          // adjacent query tiles of one head: ranges differ by at most one tile at each end
          for (int h = g * G; h < (g + 1) * G; ++h) {
            int64_t I = 0;
            while (I < c.tq128) {
              const Task *a = &tasks[h][I];
              if (a->count() <= 0) { ++I; continue; }
              const Task *b = (I + 1 < c.tq128 && tasks[h][I + 1].count() > 0) ? &tasks[h][I + 1] : nullptr;
              if (b && (b->jlo < a->jlo || b->jlo > a->jhi + 1)) b = nullptr;
              finish_range(a, b, batch, g);
              I += b ? 2 : 1;
            }
          }
        }
      }
    }
  };
  drafts.reserve(size_t(p->batch) * size_t(heads) * size_t(c.tq128));
  build_drafts();

  // ---- few items: one query tile per item, or key ranges cut over all CTAs, where that ends earlier.
  // (Many items spread evenly by themselves: the paired plan stands where its busiest CTA has at most a
  // tenth more than the mean.)  Kernel time, paired -> chosen plan: 500 queries on 12500 keys, 32/8 heads,
  // 161 -> 96 us (cut); a decode step of batch 8 on 6001 keys, 32/8 heads, 82 -> 39 us (packed and cut);
  // 12 heads x 512 d64 11.8 -> 9.6 us, 16/4 heads x 2048 d128 35.2 -> 30.7 us (one query tile per item).
  if (spread != Spread::kNone && !on_lengths && drafts.size() < size_t(8 * num_ctas)) {
    const double fill = double(std::min<int64_t>(rows_q, kTile)) / kTile;
    double work = 0.0;
    for (const Draft &d : drafts) work += step_cost(d.w) * d.w.n_steps + kItemOverheadSteps;
    const double paired = makespan(drafts, num_ctas);
    if (paired > 1.1 * work / num_ctas) {
      std::vector<Draft> paired_drafts;
      paired_drafts.swap(drafts);
      double best = 0.95 * paired;
      pair = false;
      build_drafts();
      std::vector<Draft> singles;
      singles.swap(drafts);
      for (const std::vector<Draft> *from : {&paired_drafts, &singles}) {
        if (spread != Spread::kCut) break;
        Plan cut;
        std::vector<Draft> pieces;
        const double t = cut_over_ctas(*from, num_ctas, fill, &pieces, &cut);
        if (t < best) {
          best = t;
          drafts.swap(pieces);
          plan->split_tiles.swap(cut.split_tiles);
          plan->n_parts = cut.n_parts;
        }
      }
      const double single = makespan(singles, num_ctas);
      if (single < best) {
        drafts.swap(singles);
        plan->split_tiles.clear();
        plan->n_parts = 0;
      } else if (drafts.empty()) {
        drafts.swap(paired_drafts);
      } else {
        uncut.swap(single < 0.95 * paired ? singles : paired_drafts);
      }
    }
  }

  st = place_items(*p, num_ctas, drafts, plan);
  if (st == STEEL_OK && whole && !plan->split_tiles.empty()) {
    whole->packed = plan->packed;
    st = place_items(*p, num_ctas, uncut, whole);
  }
  if (st != STEEL_OK) return st;
  if (stats) count_tiles(c, *plan, rows_q, &s);
  return STEEL_OK;
}

BitmapMask bitmap_mask(const steel_attn_params_t &p) {
  BitmapMask m;
  m.seq_q = p.seq_q;
  m.seq_kv = p.seq_kv;
  m.off = int64_t(p.seq_kv) - p.seq_q;
  m.window = p.mask.window;
  m.block = p.mask.block_q ? p.mask.block_q : kTile;
  m.blocks_q = (p.seq_q + m.block - 1) / m.block;
  m.blocks_kv = (p.seq_kv + m.block - 1) / m.block;
  m.words = (m.blocks_kv + 31) / 32;
  m.causal = (p.mask.flags & STEEL_MASK_CAUSAL) != 0;
  m.windowed = (p.mask.flags & STEEL_MASK_WINDOW) != 0;
  return m;
}

steel_status_t plan_noalloc(const steel_attn_params_t *p, int num_ctas, NoallocPlan *np) {
  const BitmapMask mask = bitmap_mask(*p);
  const size_t bitmap_bytes =
      (p->mask.flags & STEEL_MASK_BITMAP) ? size_t(p->heads_q) * mask.blocks_q * mask.words * sizeof(uint32_t) : 0;
  Plan &plan = np->plan;
  bool fits = false;
  auto plan_as = [&](Spread spread, bool on_device) {
    const steel_status_t st = build_plan(p, num_ctas, &plan, /*stats=*/false, spread, nullptr, on_device);
    if (st != STEEL_OK) return st;
    fits = plan.items.size() <= kNoallocItems && size_t(plan.n_steps) <= kNoallocSteps &&
           plan.cta_begin.size() <= kNoallocCtas + 1;
    np->device_lists = plan.steps.empty() && plan.n_steps > 0;
    np->bitmap_bytes = np->device_lists ? bitmap_bytes : 0;
    np->off_cta_begin = kNoallocStatusBytes;
    // items start on 64 bytes, so that each lies in one cache line
    np->off_items = round_up(np->off_cta_begin + plan.cta_begin.size() * sizeof(int32_t), 64);
    np->off_bitmap = np->off_items + plan.items.size() * sizeof(WorkItem);
    np->off_steps = np->off_bitmap + round_up(np->bitmap_bytes, 16);
    np->end = np->off_steps + size_t(plan.n_steps) * sizeof(StepPair);
    np->copy_bytes = np->device_lists ? np->off_bitmap + np->bitmap_bytes : np->end;
    return STEEL_OK;
  };
  // One query tile per item can need more list entries than pairs: where the array has no room for it, the paired plan
  // is taken.  Where the items of a bitmap mask are single query tiles, their lists are written on the device if the
  // bitmap fits into the array beside them; else by the host.  What fits in no way is refused, not truncated.
  steel_status_t st = plan_as(Spread::kTiles, bitmap_bytes > 0);
  if (st == STEEL_OK && fits && np->device_lists && np->end > kNoallocBytes) st = plan_as(Spread::kTiles, false);
  if (st == STEEL_OK && !fits) st = plan_as(Spread::kNone, false);
  if (st != STEEL_OK) return st;
  return fits ? STEEL_OK : STEEL_ERR_UNSUPPORTED;
}

int64_t plan_rows_q(const steel_attn_params_t &p, const Plan &plan) {
  return plan.packed ? int64_t(p.heads_q / p.heads_kv) * p.seq_q : p.seq_q;
}

void set_query_view(const steel_attn_params_t &p, bool packed, KernelParams *kp) {
  kp->heads_q = packed ? p.heads_kv : p.heads_q;
  kp->rows_q = packed ? p.heads_q / p.heads_kv * p.seq_q : p.seq_q;
}

// Entry of slot `slot` at step t of an item, as the kernel derives it.
uint32_t item_entry(const Plan &plan, const WorkItem &w, int slot, int t, const steel_attn_params_t *p) {
  if (w.head[slot] < 0 || t < w.lo[slot] || t > w.hi[slot]) return 0;
  if (w.kind == 1) return plan.steps[size_t(w.j0[0]) + size_t(t)].e[slot];
  // range kind: geometry decides whether the element-wise mask is needed
  Geom g{p->seq_q, p->seq_kv, int64_t(p->seq_kv) - p->seq_q, p->mask.window,
         (p->mask.flags & STEEL_MASK_CAUSAL) != 0, (p->mask.flags & STEEL_MASK_WINDOW) != 0};
  int64_t J = int64_t(w.j0[slot]) + t;
  int64_t i0, i1;
  tile_positions(p->seq_q, plan_rows_q(*p, plan), w.qtile[slot], &i0, &i1);
  int64_t j0 = J * kTile, j1 = std::min<int64_t>(j0 + kTile - 1, p->seq_kv - 1);
  uint32_t e = uint32_t(J) | kEntryPresent | kEntrySubAll;
  if (!g.all_visible(i0, i1, j0, j1) || (j1 - j0 + 1) < kTile) e |= kEntryPartial;
  return e;
}

void walk_plan(const Plan &plan, const std::function<void(int, const WorkItem &, int, int, uint32_t, bool)> &visit,
               const steel_attn_params_t *p) {
  for (size_t n = 0; n < plan.items.size(); ++n) {
    const WorkItem &w = plan.items[n];
    for (int t = 0; t < w.n_steps; ++t) {
      uint32_t e0 = item_entry(plan, w, 0, t, p), e1 = item_entry(plan, w, 1, t, p);
      bool shared = e0 && e1 && ((e0 & kEntryTileMask) == (e1 & kEntryTileMask));
      if (e0) visit(int(n), w, 0, t, e0, false);
      if (e1) visit(int(n), w, 1, t, e1, shared);
    }
  }
}

}  // namespace steel
