// The step entry of one (query tile, key tile) pair under a bitmap mask, from the mask's words, and the list of a query
// tile made of them: what the kernel does that writes the step lists of steel_attn_run_noalloc.  The planner counts, and
// makes its own lists, word by word (Ctx::kept_words); tests/list_entries.cpp compares the two, and a list that is not as
// long as the planner has counted is reported (ListWriter::finish).
#pragma once
#include <stdint.h>

#include "steel_plan.h"

#ifdef __CUDACC__
#define STEEL_HOST_DEVICE __host__ __device__
#else
#define STEEL_HOST_DEVICE
#endif

namespace steel {

struct BitmapMask {
  int64_t seq_q, seq_kv, off, window;  // off = seq_kv - seq_q
  int32_t block;                       // 64 or 128
  int32_t blocks_q, blocks_kv, words;  // descriptor blocks in each direction, words per row of blocks
  bool causal, windowed;

  STEEL_HOST_DEVICE int32_t key_tiles() const { return int32_t((seq_kv + kTile - 1) / kTile); }

  // Entry of key tile J for query tile I, 0 if no key of it is visible.  `rows`: the words of the tile's head.
  STEEL_HOST_DEVICE uint32_t entry(const uint32_t *rows, int64_t I, int64_t J) const {
    const int per = kTile / block;  // blocks of a tile in each direction
    uint32_t sub = 0, in = 0;
    bool any = false, full = true;
    for (int a = 0; a < per; ++a) {
      const int64_t row = per * I + a;
      if (row >= blocks_q) break;
      const int64_t i0 = row * block, i1 = i0 + block < seq_q ? i0 + block - 1 : seq_q - 1;
      for (int b = 0; b < per; ++b) {
        const int64_t col = per * J + b;
        if (col >= blocks_kv) continue;
        in |= 1u << (2 * a + b);
        if (!((rows[row * words + (col >> 5)] >> (col & 31)) & 1u)) continue;
        sub |= 1u << (2 * a + b);
        // row p sees keys (p - window, p]
        const int64_t j0 = col * block, j1 = j0 + block < seq_kv ? j0 + block - 1 : seq_kv - 1;
        if ((!causal || j0 <= i1 + off) && (!windowed || i0 + off - j1 < window)) any = true;
      }
    }
    if (!any) return 0;
    const int64_t i0 = I * kTile, i1 = i0 + kTile < seq_q ? i0 + kTile - 1 : seq_q - 1;
    const int64_t j0 = J * kTile, j1 = j0 + kTile < seq_kv ? j0 + kTile - 1 : seq_kv - 1;
    if (sub != in) full = false;
    if (causal && j1 > i0 + off) full = false;
    if (windowed && i1 + off - j0 >= window) full = false;
    if (j1 - j0 + 1 < kTile) full = false;  // a ragged last tile is masked element by element
    if (per == 1) sub = 0xFu;
    return uint32_t(J) | kEntryPresent | (sub << kEntrySubShift) | (full ? 0u : kEntryPartial);
  }
};

STEEL_HOST_DEVICE inline int bits(uint32_t word) {
#ifdef __CUDA_ARCH__
  return __popc(word);
#else
  return __builtin_popcount(word);
#endif
}

// One lane's part in writing a query tile's list, 32 key tiles at a time in ascending order.  Only the list's own
// `n_steps` places are written.
struct ListWriter {
  StepPair *out;
  int n_steps;
  int at = 0;  // entries found so far, by all lanes

  // `e`: the lane's entry (0 if its tile is not visible), `seen`: the lanes that have one.
  STEEL_HOST_DEVICE void place(int lane, uint32_t e, uint32_t seen) {
    const int here = at + bits(seen & ((1u << lane) - 1u));
    if (e != 0 && here < n_steps) out[here] = StepPair{{e, 0u}};
    at += bits(seen);
  }
  // After the last key tile: whether the list is as long as planned.  Places without an entry become key tile 0, so that
  // the steps that the attention kernel expects are there whatever has gone wrong.
  STEEL_HOST_DEVICE bool finish(int lane) {
    for (int n = at + lane; n < n_steps; n += 32) out[n] = StepPair{{kEntryPresent | (0xFu << kEntrySubShift) | kEntryPartial, 0u}};
    return at == n_steps;
  }
};

}  // namespace steel
