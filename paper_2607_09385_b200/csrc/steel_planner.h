// Host planner interface: turns a validated problem description into the work items, step lists
// and per-CTA assignment the kernel consumes, and the statistics reported to callers.
#pragma once
#include <functional>
#include <vector>

#include "../../include/steel_attn.h"
#include "steel_bitmap.h"
#include "steel_plan.h"

namespace steel {

// K + V bytes of the KV heads scheduled together.  Data that every SM reads ends up in both halves
// of the 126 MB L2, so about half of it is usable: with 64 MiB waves the 32K bitmap workload read its
// K/V from DRAM 1.5 times, with 32 MiB waves 1.02 times (and ran 2 % faster).
constexpr int64_t kL2WaveBytes = 32ll << 20;
// Fixed cost of an item (Q load, first-tile latency, epilogue) in units of one key-tile step.
constexpr int kItemOverheadSteps = 2;
// Bitmap masks: how many tasks of similar length are examined when choosing a query tile's partner.
constexpr size_t kPartnerWindow = 16;
// CTA count assumed by the host-only planning entry point (the SM count of a B200).
constexpr int kPlanHostCtas = 148;

// Cutting key ranges over CTAs, in key-tile steps of two slots (1.75 us).  `fill`: share of a query tile's
// 128 rows in use, 1 except where all rows of a matrix are fewer.
constexpr double kSingleStep = 0.65;  // a step of which one slot takes part (1.2 us)
constexpr double kPieceOverheadSteps = 1.5;
// A part writes 64 KB of O (head_dim 128) before its CTA goes on; the last one reads those of all parts at an
// SM's 64 bytes per cycle.
constexpr double part_write_steps(double fill) { return 2.5 * fill; }
constexpr double combine_steps(double fill, int parts) { return 1.5 + 0.7 * fill * parts; }
// Shorter pieces (in key tiles) cost more to start and combine than they take.
constexpr int min_piece_tiles(double fill) { return int(4 + 8 * fill); }

// Whether a small kernel writes the lists of single query tiles, `entries` in all: its launch costs 2.5 us, and it saves
// the host 0.06 us per list and 0.01 us per entry (steel_attn_run_noalloc at 110 shapes).  Us, lists from the host /
// from the device: 4 lists of 10 entries 33.7 / 35.7, 16 of 37 36.7 / 37.8, 24 of 36 37.8 / 37.8, 24 of 117 51.0 / 51.0,
// 32 of 73 39.8 / 38.8, 48 of 110 44.0 / 42.8, 128 of 825 79.8 / 67.2, 32 of 391 67.4 / 64.6.
constexpr bool lists_on_device(int64_t lists, int64_t entries) { return 6 * lists + entries >= 240; }

struct Draft {  // a work item before it is placed
  WorkItem w;
  std::vector<StepPair> list;
  int group;
  int cta = -1;  // placed already (make_pieces)
};

struct Plan {
  std::vector<WorkItem> items;     // in CTA order
  std::vector<int32_t> cta_begin;  // grid + 1
  std::vector<StepPair> steps;     // list-kind entries
  int64_t n_steps = 0;             // their number; `steps` is empty where the lists are left to the device
  std::vector<SplitTile> split_tiles;
  int32_t n_parts = 0;             // part buffers of all split tiles
  bool packed = false;             // query tiles hold rows of all heads of a group (KernelParams::rows_q)
  steel_attn_stats_t stats;
  int grid = 0;
};

steel_status_t validate_params(const steel_attn_params_t *p);
// What a plan may do beyond pairing query tiles (policy 0 only; build_plan takes what ends earliest).
enum class Spread {
  kNone,
  kTiles,  // query tiles over the heads of a group, one query tile per item
  kCut,    // also key ranges cut over CTAs, which needs part buffers
};
// Scheduling policy and the other options come from `p`.  Without `stats` the plan's statistics stay 0 (they
// take a walk over every block).  Where `plan` cuts key ranges, `whole` (if not null)
// becomes the plan that would be taken without cuts: items, steps and the statistics of its items.
// `device_lists`: where the items of a bitmap mask are single query tiles and lists_on_device says so, the plan holds the
// lengths and places of their lists only; the entry of tile J is BitmapMask::entry, in ascending order of J (Spread::kTiles, no `stats`).
steel_status_t build_plan(const steel_attn_params_t *p, int num_ctas, Plan *plan, bool stats = true,
                          Spread spread = Spread::kNone, Plan *whole = nullptr, bool device_lists = false);

BitmapMask bitmap_mask(const steel_attn_params_t &p);

// steel_attn_run_noalloc: the fixed array, and a call's plan and places in it, one behind the other so that one copy
// brings them: status word, per-CTA ranges, items, then the bitmap where the device writes the step lists, then those.
constexpr size_t kNoallocItems = 16384;   // work items (64 bytes each)
constexpr size_t kNoallocCtas = 1024;     // persistent CTAs (+1 range entry)
constexpr size_t kNoallocSteps = 131072;  // explicit step-list entries of bitmap masks (8 bytes each)
constexpr size_t round_up(size_t n, size_t to) { return (n + to - 1) / to * to; }
constexpr size_t kNoallocStatusBytes = 256;
constexpr size_t kNoallocBytes = kNoallocStatusBytes + round_up((kNoallocCtas + 1) * sizeof(int32_t), 64) +
                                 kNoallocItems * sizeof(WorkItem) + kNoallocSteps * sizeof(StepPair);  // about 2.0 MiB
struct NoallocPlan {
  Plan plan;
  bool device_lists = false;
  size_t off_cta_begin = 0, off_items = 0, off_bitmap = 0, off_steps = 0;
  size_t bitmap_bytes = 0;  // 0 unless device_lists
  size_t copy_bytes = 0;    // from the array's start, host -> device
  size_t end = 0;           // of all that the call keeps in the array
};
// STEEL_ERR_UNSUPPORTED: no plan fits.  Host only; may throw std::bad_alloc.
steel_status_t plan_noalloc(const steel_attn_params_t *p, int num_ctas, NoallocPlan *np);

// steel_attn_create with a limit on what the plan may do (implemented in steel_attn.cu).
steel_status_t create_attention(const steel_attn_params_t *params, Spread most, steel_attn_t **out);

// Launches of at most this many steps on the busiest CTA overlap their set-up with the launch before them on
// the stream (kernel time, without -> with: 1 head x 256 7.6 -> 6.4 us, 12 heads x 512 9.7 -> 8.9 us, a decode step
// of batch 8 38.0 -> 37.1 us); longer ones do not gain (32 heads x 4096, 60 steps: 123 -> 126 us; 500 queries on
// 12500 keys, 46 steps: 99 -> 104 to 117 us).
constexpr int64_t kOverlapSteps = 32;

// Rows of one matrix of Q as the plan's query tiles see it, and the kernel's fields for that view.
int64_t plan_rows_q(const steel_attn_params_t &p, const Plan &plan);
void set_query_view(const steel_attn_params_t &p, bool packed, KernelParams *kp);

// Entry (tile index and flags, 0 if absent) of `slot` at step `t`, derived exactly as on the device.
uint32_t item_entry(const Plan &plan, const WorkItem &w, int slot, int t, const steel_attn_params_t *p);

// Visit every executed tile: (item index, item, slot, step, entry, shares the other slot's load).
void walk_plan(const Plan &plan, const std::function<void(int, const WorkItem &, int, int, uint32_t, bool)> &visit,
               const steel_attn_params_t *p);

}  // namespace steel
