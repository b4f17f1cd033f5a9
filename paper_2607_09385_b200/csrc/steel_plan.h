// Plain-data structures shared by the host planner and the device kernel: work items, step
// entries and kernel parameters.  The planner turns the mask descriptor into these (the three
// mask cases of the paper's Sec. "The STEEL Pipeline" at 128 x 128 tile granularity); the kernel
// only ever sees tiles that must be executed.
#pragma once
#include <stdint.h>

namespace steel {

constexpr int kTile = 128;  // query rows per tile and keys per tile
constexpr long long kDefaultTimeoutCycles = 4000000000ll;  // about two seconds of SM clock
constexpr long long kMaxTimeoutCycles = 1ll << 46;       // about ten hours: waits may keep time in 32 bits of 65 536 cycles

// One step entry of one query tile ("slot") in a list-kind item.
constexpr uint32_t kEntryTileMask = 0x00FFFFFFu;  // key-tile index
constexpr uint32_t kEntryPresent = 1u << 24;
constexpr uint32_t kEntryPartial = 1u << 25;      // element-wise mask needed
constexpr uint32_t kEntrySubShift = 26;           // 4 bits: 64x64 sub-blocks TL, TR, BL, BR enabled
constexpr uint32_t kEntrySubAll = 0xFu << kEntrySubShift;

// A work item: one or two query tiles ("slots") of the same batch and KV head that walk their key
// tiles in lock-step, sharing a K/V load whenever both want the same key tile at the same step.
// Slot s is present on steps lo[s]..hi[s] (inclusive; lo > hi means the slot is unused), and
// lo[0] <= lo[1] whenever both are used.
struct WorkItem {
  int32_t batch;
  int32_t kv_head;
  int32_t head[2];   // query head of each slot
  int32_t qtile[2];  // query tile index (rows qtile*128 ...) of each slot
  int32_t lo[2];
  int32_t hi[2];
  int32_t n_steps;
  int32_t kind;      // 0: range (key tile of step t is j0[s] + t for slot s), 1: list
  int32_t j0[2];     // range kind; list kind: j0[0] is the index of the item's first StepPair
  int32_t split[2];  // slot s holds one of several key ranges of its query tile: split_code; else -1
};
static_assert(sizeof(WorkItem) == 64, "WorkItem layout");

// A query tile whose key tiles are cut over several items: each part leaves its unnormalised O and its
// row statistics in a buffer of its own, and the part that finishes last combines them.
constexpr int kMaxParts = 64;
struct SplitTile {
  int32_t first;    // buffer of part 0; the parts' buffers are consecutive
  int32_t n_parts;
};
constexpr int32_t split_code(int32_t tile, int32_t part) { return tile << 6 | part; }
static_assert(kMaxParts <= 64, "split_code keeps the part in 6 bits");

// Entries of both slots for one step of a list-kind item.
struct StepPair {
  uint32_t e[2];
};

struct KernelParams {
  const WorkItem *items;     // ordered so that CTA c owns items cta_begin[c] .. cta_begin[c+1]-1
  const int32_t *cta_begin;  // gridDim.x + 1 entries
  const StepPair *steps;       // list-kind step entries
  void *o;                   // bf16 [batch, heads_q, seq_q, head_dim]
  float *lse;                // fp32 [batch, heads_q, seq_q] or null
  bool o_aligned32;          // `o` is a multiple of 32 (16 is what callers promise)
  int32_t *status;           // device status word (0 ok, else STEEL_ERR_TIMEOUT)
  const SplitTile *split_tiles;  // null: no query tile is split
  float *parts;              // per part: O as float4 [head_dim / 4][part_rows], then (m, l) [part_rows]
  int32_t part_rows;         // rows of a query tile that can be used (128, or those of a shorter matrix), a multiple of 4
  int32_t *arrivals;         // per split tile and row quarter: parts finished; zero between launches
  // Q as [batch][heads_q][rows_q][head_dim]: `heads_q` matrices of rows_q = seq_q rows or, where a query
  // tile holds rows of several heads of a group, heads_kv matrices of group * seq_q rows
  int32_t heads_q, heads_kv, rows_q, seq_q, seq_kv;
  uint32_t mask_flags;
  int32_t window;            // clamped to int32 range
  float scale_log2;          // scale * log2(e)
  long long *clock_probe;    // measurement hook: CTA 0 stores {SM cycles, nanoseconds} of its run here, else null
  long long timeout_cycles;  // bound of every device-side wait
  bool overlap_launch;       // host side: start beside the end of the launch before it on the stream
  int32_t stall_cta;         // test hook: this CTA's producer withholds its commands (-1: none)
};

}  // namespace steel
