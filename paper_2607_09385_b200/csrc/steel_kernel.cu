// Fused block-sparse attention kernel for sm_100a (paper Algorithm 1 on one persistent CTA per SM).
//
// A CTA processes work items; an item is one or two query tiles (128 rows each, "slots") that walk
// the same sequence of key-tile steps.  Roles (three warpgroups, register file re-split between them):
//   warps 0-3 / 4-7 : softmax warpgroup of slot 0 / 1.  Thread r owns query row r: it reads the
//                     score row S (fp32) from TMEM into registers and hands the S buffer back,
//                     applies scale and (partial tiles only) the mask computed from coordinates,
//                     keeps the running maximum m and sum l, writes P = 2^(S*scale*log2e - m) as
//                     bf16 into the slot's own P columns, rescales O when the maximum has grown, and
//                     at the end writes O / l and LSE.  (Algorithm 1: scale_and_mask and rowmax of
//                     the First Stage, the Second Stage, and the rescale of the Third.)
//   warp 8          : TMA producer and scheduler.  Walks the items, loads Q once per item and K_j / V_j
//                     for executed tiles only into a shared-memory ring (a tile wanted by both slots
//                     in the same step is loaded once), and publishes one command word per product
//                     for its MMA issuer, with ring slots, barrier phases and release flags worked out.
//   warps 9-11      : MMA issuers on tcgen05 with fp32 accumulators in TMEM: warp 9 issues S = Q K^T of
//                     both slots (both operands in shared memory), warp 10 / 11 O += P V of slot 0 / 1 (P
//                     from TMEM, V from shared memory).
// Tensor memory (512 columns): one S buffer that the slots use in turn (128), P of each slot
// (2 x 64), O of each slot (2 x head_dim).  S(s, t + 1) does not wait for PV(s, t), so a slot's next
// scores are computed while its softmax warps still work on the current tile.  (At head_dim 64 the
// columns would allow an S buffer per slot; measured, that layout is slower: 32 heads of 8192 tokens
// 419 us against 382 us.  The shared buffer keeps the slots half a tile apart, so that one computes
// exponentials while the other reads scores and searches its maximum.)
//
// What bounds it: the chain S -> registers -> hand-back of the S buffer -> next S, and the softmax warps'
// instruction stream (16 384 exponentials per tile: 1 024 cycles of the special-function unit at best, as
// much as the tile's two products take on the tensor core at head_dim 128).  Three issuers instead of one,
// because a tcgen05.commit returns only when the products before it have nearly drained: one thread that
// issues everything spends 1 450 to 1 700 cycles per pair of products that take 1 024.  Measured, one
// issuer -> three (kernel time): 32 heads x 4096 causal, head_dim 128: 136.5 -> 125.6 us; 16 heads x 32768,
// bitmap 25 %: 1 027 -> 954 us; 32/8 heads x 16384 causal: 1 753 -> 1 635 us; 32 heads x 8192 causal,
// head_dim 64: 408 -> 382 us.  Two issuers, one per slot with both its products: 126 / 968 / 1 636 / 395 us.
// Every mbarrier and queue wait is bounded; on expiry the CTA sets the status word and all roles leave.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include "sm100_ptx.cuh"
#include "steel_kernel.h"
#include "steel_plan.h"
#include "steel_wait.cuh"

namespace steel {

constexpr int kThreads = 384;        // softmax slot 0, softmax slot 1, {producer, 3 MMA issuers}
// Registers per thread after the warpgroups re-split the file.  2 * 128 * kRegsSoftmax + 128 *
// kRegsOther must stay below the 65 536 registers of an SM with room to spare: setmaxnreg.inc waits,
// without any bound, until the increase can be granted.
constexpr int kRegsSoftmax = 216;
constexpr int kRegsOther = 72;
static_assert(2 * 128 * kRegsSoftmax + 128 * kRegsOther <= 65536 - 1024, "register re-split needs slack");
constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;  // first of three: S of both slots, PV of slot 0, PV of slot 1
constexpr float kRescaleThreshold = 8.0f;           // lazy rescale: P stays below 2^8
constexpr int kMaxStages = 10;
constexpr int kFifoDepth = 32;
constexpr uint32_t kMaskCausal = 1u, kMaskWindow = 2u, kMaskBitmap = 4u;

template <int D>
struct Cfg {
  static constexpr int kTileBytes = kTile * D * 2;  // one Q, K or V tile
  static constexpr int kBoxes = D / 64;             // 64-column (128-byte) TMA boxes per tile
  static constexpr int kBoxBytes = kTile * 128;
  static constexpr int kStages = (D == 128) ? 5 : 10;
  static constexpr int kSmemBytes = 1024 + (2 + kStages) * kTileBytes;
  // Tensor-memory columns: S (fp32, 128 columns), one buffer that the slots use in turn; P of slot s
  // (bf16 pairs, 64 columns) at kColP + 64 s; O of slot s (D columns) at kColO + D s.
  static constexpr uint32_t kColS = 0, kColP = 128, kColO = 256;
};

struct Ctrl {
  uint64_t ring_full[kMaxStages], ring_empty[kMaxStages];
  uint64_t q_full[2], q_empty[2], s_full[2], p_full[2], p_free[2], o_full[2], o_empty[2];
  uint64_t s_free;     // the softmax warps that own the S buffer's content have it in registers
  uint64_t drain[3];   // an MMA issuer's last commit when it leaves on an expired wait
  uint32_t fifo[3][kFifoDepth];  // command words from the producer to the MMA issuers (0 = empty)
  uint32_t tmem_base;
  int abort;
  long long timeout_cycles;
};

// Command word (producer -> MMA issuer): one product, S(s, t) or PV(s, t).  In the queue its 16 bits stand beside
// their complement: the issuing warp puts a word together from what each of its lanes has read (warp_uniform), and
// nothing in the language makes the lanes read at the same moment.  A word that only some lanes have seen fails the
// check and is read again.
constexpr uint32_t kCmdValid = 1u << 0, kCmdSlot1 = 1u << 1,
                   kCmdFirst = 1u << 2, kCmdLast = 1u << 3,  // of the slot's steps in this item
                   kCmdRingShift = 4,  // 4 bits: ring slot of the K or V tile
                   kCmdRingPhase = 1u << 8,
                   kCmdUsePhase = 1u << 9,    // Q full (S), O empty (PV); read with kCmdFirst
                   kCmdDepPhase = 1u << 10,   // S buffer free (S), P full (PV)
                   kCmdWaitSFree = 1u << 11,  // not the CTA's first S
                   kCmdFinal = 1u << 12,      // S: last reader of the K tile, release the ring slot
                   kCmdExit = 1u << 13;
__device__ __forceinline__ bool cmd_complete(uint32_t word) { return ((word ^ (word >> 16)) & 0xFFFFu) == 0xFFFFu; }

__device__ __forceinline__ bool bounded_wait(uint64_t *bar, uint32_t parity, Ctrl &ctrl, int32_t *status) {
  if (mbar_test_wait(bar, parity)) return true;  // the common case: already complete, no suspension
  const long long start = clock64();
  uint32_t n = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++n & 63u) == 0) {
      if (*reinterpret_cast<volatile int *>(&ctrl.abort)) return false;
      if (clock64() - start > ctrl.timeout_cycles) {
        *reinterpret_cast<volatile int *>(&ctrl.abort) = 1;
        atomicExch(status, 5);
        return false;
      }
    }
  }
}

// A work item unpacked into scalars (no indexable arrays, so everything stays in registers).
struct Item {
  int batch, kv_head, head0, head1, qtile0, qtile1, lo0, lo1, hi0, hi1, n_steps, kind, j00, j01, split0, split1;
  __device__ __forceinline__ int lo(int s) const { return s ? lo1 : lo0; }
  __device__ __forceinline__ int hi(int s) const { return s ? hi1 : hi0; }
  __device__ __forceinline__ int head(int s) const { return s ? head1 : head0; }
  __device__ __forceinline__ int qtile(int s) const { return s ? qtile1 : qtile0; }
  __device__ __forceinline__ int j0(int s) const { return s ? j01 : j00; }
  __device__ __forceinline__ int split(int s) const { return s ? split1 : split0; }
  __device__ __forceinline__ int list_off() const { return j00; }
  __device__ __forceinline__ bool active(int s) const { return head(s) >= 0 && hi(s) >= lo(s); }
};

__device__ __forceinline__ Item load_item(const WorkItem *items, int k) {
  const int4 *src = reinterpret_cast<const int4 *>(items + k);
  const int4 a = __ldg(src), b = __ldg(src + 1), c = __ldg(src + 2), d = __ldg(src + 3);
  Item w;
  w.batch = a.x;  w.kv_head = a.y;  w.head0 = a.z;  w.head1 = a.w;
  w.qtile0 = b.x; w.qtile1 = b.y;   w.lo0 = b.z;    w.lo1 = b.w;
  w.hi0 = c.x;    w.hi1 = c.y;      w.n_steps = c.z; w.kind = c.w;
  w.j00 = d.x;    w.j01 = d.y;      w.split0 = d.z; w.split1 = d.w;
  return w;
}

// Entries {slot 0, slot 1} of step t: key-tile index plus the present bit (0 when the slot is absent).
template <bool kList>
__device__ __forceinline__ uint2 load_step(const Item &w, const StepPair *steps, int t) {
  uint2 e = make_uint2(0u, 0u);
  if (t >= w.n_steps) return e;
  if (!kList || w.kind == 0) {
    if (w.active(0) && t >= w.lo0 && t <= w.hi0) e.x = uint32_t(w.j00 + t) | kEntryPresent;
    if (w.active(1) && t >= w.lo1 && t <= w.hi1) e.y = uint32_t(w.j01 + t) | kEntryPresent;
  } else {
    e = __ldg(reinterpret_cast<const uint2 *>(steps + w.list_off() + t));
  }
  return e;
}

// The canonical order of an item's tensor-core operations S(s, t) = Q_s K_j^T and PV(s, t):
// O_s += P_s V_j: the order in which the producer loads tiles (at their first use) and publishes
// commands, and therefore the order in which each MMA issuer executes its own.
// For each step t: first S(s, t) of slots that start at t, then for each present slot S(s, t + 1)
// followed by PV(s, t): the first product runs one step ahead of the second, so a slot's next scores
// are computed while its softmax warps still work on the current ones (they hold them in registers;
// the S buffer in TMEM is free again as soon as they are loaded).  A tile wanted by both slots in
// one step is one ring fill: slot 0 uses it first, slot 1 last (the planner guarantees lo0 <= lo1).
// `ring` counts fills.
// op(s, t, j, is_s, fill, first, last) returns false to stop.
struct RingPos {
  uint32_t slot, phase;  // next fill goes to `slot`; `phase` flips each time the ring wraps
};
struct Fill {
  uint32_t slot, phase;
};

template <int kStages, bool kList, class Op>
__device__ __forceinline__ bool walk_item(const Item &w, const StepPair *steps, RingPos &ring, Op &&op) {
  Fill last_k{0, 0}, last_v{0, 0};
  auto take = [&]() {
    Fill f{ring.slot, ring.phase};
    if (++ring.slot == uint32_t(kStages)) {
      ring.slot = 0;
      ring.phase ^= 1u;
    }
    return f;
  };
  auto visit = [&](const uint2 &e, int s, int t, bool is_s) -> bool {
    const uint32_t mine = s ? e.y : e.x, other = s ? e.x : e.y;
    const bool shared = other != 0 && ((mine ^ other) & kEntryTileMask) == 0;
    Fill &last = is_s ? last_k : last_v;
    Fill f;
    bool first = true, final_use = true;
    if (s == 1 && shared) {
      f = last;
      first = false;
    } else {
      f = take();
      if (s == 0) {
        last = f;
        final_use = !shared;
      }
    }
    return op(s, t, int(mine & kEntryTileMask), is_s, f, first, final_use);
  };
  uint2 cur = load_step<kList>(w, steps, 0);
  for (int t = 0; t < w.n_steps; ++t) {
    const uint2 nxt = load_step<kList>(w, steps, t + 1);
    if (cur.x != 0 && t == w.lo0 && !visit(cur, 0, t, true)) return false;
    if (cur.y != 0 && t == w.lo1 && !visit(cur, 1, t, true)) return false;
    if (cur.x != 0) {
      if (t < w.hi0 && !visit(nxt, 0, t + 1, true)) return false;
      if (!visit(cur, 0, t, false)) return false;
    }
    if (cur.y != 0) {
      if (t < w.hi1 && !visit(nxt, 1, t + 1, true)) return false;
      if (!visit(cur, 1, t, false)) return false;
    }
    cur = nxt;
  }
  return true;
}

// ------------------------------------------------------------------------------------------------
// Bounded push into the single-producer single-consumer command queue in shared memory (the pop is
// with the MMA issuer below).
__device__ __forceinline__ bool fifo_push(Ctrl &ctrl, int s, uint32_t &tail, uint32_t word, int32_t *status) {
  volatile uint32_t *cell = &ctrl.fifo[s][tail];
  if (*cell != 0) {
    const long long start = clock64();
    uint32_t n = 0;
    while (*cell != 0) {
      if ((++n & 63u) == 0) {
        if (*reinterpret_cast<volatile int *>(&ctrl.abort)) return false;
        if (clock64() - start > ctrl.timeout_cycles) {
          *reinterpret_cast<volatile int *>(&ctrl.abort) = 1;
          atomicExch(status, 5);
          return false;
        }
      }
    }
  }
  *cell = word | ~word << 16;
  tail = (tail + 1) & (kFifoDepth - 1);
  return true;
}
// The producer is also the scheduler: it walks the items, issues the TMA loads and publishes one
// command word per product, so the MMA issuers' own loops stay a few instructions long.
template <int D, bool kList>
__device__ void producer_role(const KernelParams &p, const CUtensorMap *map_q, const CUtensorMap *map_k,
                              const CUtensorMap *map_v, Ctrl &ctrl, uint8_t *smem_q, uint8_t *smem_ring) {
  using C = Cfg<D>;
  // measurement hook: the SM clock this CTA really ran at is cycles / nanoseconds over its run
  const bool probe = p.clock_probe != nullptr && blockIdx.x == 0;
  long long probe_c0 = 0;
  unsigned long long probe_t0 = 0;
  if (probe) {
    probe_c0 = clock64();
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(probe_t0));
  }
  RingPos ring{0, 0};
  uint32_t n_use0 = 0, n_use1 = 0, n_sp0 = 0, n_sp1 = 0, n_s = 0, fills = 0, tail_s = 0, tail_pv0 = 0, tail_pv1 = 0;
  bool ok = true;
  const bool stalled = p.stall_cta == int(blockIdx.x);
  const int k_end = p.cta_begin[blockIdx.x + 1];
  for (int k = p.cta_begin[blockIdx.x]; k < k_end && ok; ++k) {
    const Item w = load_item(p.items, k);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!ok || !w.active(s)) continue;
      uint32_t &n_use = s ? n_use1 : n_use0;
      ok = bounded_wait(&ctrl.q_empty[s], (n_use & 1u) ^ 1u, ctrl, p.status);
      if (!ok) break;
      mbar_arrive_expect_tx(&ctrl.q_full[s], C::kTileBytes);
#pragma unroll
      for (int b = 0; b < C::kBoxes; ++b)
        tma_load_3d(smem_q + s * C::kTileBytes + b * C::kBoxBytes, map_q, &ctrl.q_full[s], b * 64,
                    w.qtile(s) * kTile, w.batch * p.heads_q + w.head(s));
      ++n_use;
    }
    if (!ok) break;
    const int z = w.batch * p.heads_kv + w.kv_head;
    ok = walk_item<C::kStages, kList>(w, p.steps, ring, [&](int s, int t, int j, bool is_s, Fill f, bool first, bool final_use) -> bool {
      if (first) {
        if (!bounded_wait(&ctrl.ring_empty[f.slot], f.phase ^ 1u, ctrl, p.status)) return false;
        // a ring slot is free again after two arrivals: the issuers of both slots release a V tile that both
        // want; K has one issuer, and a tile that one slot wants one reader
        if (is_s || final_use) mbar_arrive(&ctrl.ring_empty[f.slot]);
        mbar_arrive_expect_tx(&ctrl.ring_full[f.slot], C::kTileBytes);
        const CUtensorMap *map = is_s ? map_k : map_v;
#pragma unroll
        for (int b = 0; b < C::kBoxes; ++b)
          tma_load_3d(smem_ring + f.slot * C::kTileBytes + b * C::kBoxBytes, map, &ctrl.ring_full[f.slot], b * 64,
                      j * kTile, z);
        ++fills;
      }
      // phase of this item's use of the slot: Q-full for S, O-empty (inverted) for PV
      const uint32_t use_phase = ((s ? n_use1 : n_use0) - 1u) & 1u;
      uint32_t cmd = kCmdValid | (f.slot << kCmdRingShift) | (f.phase ? kCmdRingPhase : 0u) |
                     (t == w.lo(s) ? kCmdFirst : 0u) | (t == w.hi(s) ? kCmdLast : 0u);
      if (is_s) {
        // the S buffer is shared: S number n may be issued once S number n - 1 has been loaded into registers
        cmd |= (s ? kCmdSlot1 : 0u) | (use_phase ? kCmdUsePhase : 0u) | (final_use ? kCmdFinal : 0u) |
               (n_s > 0 ? kCmdWaitSFree : 0u) | (((n_s - 1u) & 1u) ? kCmdDepPhase : 0u);
        ++n_s;
        if (stalled) return true;  // test hook: the issuer's bounded wait for this command must expire
        return fifo_push(ctrl, 0, tail_s, cmd, p.status);
      }
      uint32_t &n_sp = s ? n_sp1 : n_sp0;
      cmd |= ((use_phase ^ 1u) ? kCmdUsePhase : 0u) | ((n_sp & 1u) ? kCmdDepPhase : 0u);
      ++n_sp;
      if (stalled) return true;
      return fifo_push(ctrl, 1 + s, s ? tail_pv1 : tail_pv0, cmd, p.status);
    });
  }
  if (ok) ok = fifo_push(ctrl, 0, tail_s, kCmdValid | kCmdExit, p.status);
  if (ok) ok = fifo_push(ctrl, 1, tail_pv0, kCmdValid | kCmdExit, p.status);
  if (ok) ok = fifo_push(ctrl, 2, tail_pv1, kCmdValid | kCmdExit, p.status);
  if (probe) {
    unsigned long long t1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    p.clock_probe[0] = clock64() - probe_c0;
    p.clock_probe[1] = (long long)(t1 - probe_t0);
  }
  if (!ok) {
    // leave only after the copies already issued have landed (bounded), so none writes into
    // shared memory of a later CTA: the last min(fills, stages) fills end at ring.slot - 1
    const uint32_t pending = fills < uint32_t(C::kStages) ? fills : uint32_t(C::kStages);
    uint32_t slot = ring.slot, phase = ring.phase;
    for (uint32_t e = 0; e < pending; ++e) {
      if (slot == 0) {
        slot = C::kStages;
        phase ^= 1u;
      }
      --slot;
      const long long start = clock64();
      while (!mbar_try_wait(&ctrl.ring_full[slot], phase) && clock64() - start < ctrl.timeout_cycles / 8) {
      }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint32_t n_use = s ? n_use1 : n_use0;
      if (n_use) {
        const long long start = clock64();
        while (!mbar_try_wait(&ctrl.q_full[s], (n_use - 1) & 1u) && clock64() - start < ctrl.timeout_cycles / 8) {
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// tcgen05.mma, tcgen05.commit and mbarrier tests take their operands from the warp's uniform
// registers, so the issuing warp keeps everything it derives from a command word provably uniform:
// all 32 lanes run the loop and read the same queue cell, and the word is rebuilt by a warp vote
// (lane i contributes bit i).  A value loaded from shared memory by one lane is not uniform as far
// as the compiler can tell, and every operand derived from it would be copied into a uniform
// register again before each instruction that needs it.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t word, int lane) {
  return __ballot_sync(0xffffffffu, (word >> lane) & 1u);
}

// Pop by the whole warp: every lane polls the same cell; the decision to leave is taken on the
// voted word, so the lanes stay together.  Lane 0 empties the cell.
__device__ __forceinline__ uint32_t fifo_pop_warp(Ctrl &ctrl, int s, uint32_t &head, int32_t *status, int lane) {
  volatile uint32_t *cell = &ctrl.fifo[s][head];
  __syncwarp();
  uint32_t word = warp_uniform(*cell, lane);
  if (!cmd_complete(word)) {
    const long long start = clock64();
    uint32_t n = 0;
    while (true) {
      __syncwarp();
      word = warp_uniform(*cell, lane);
      if (cmd_complete(word)) break;
      if ((++n & 63u) == 0) {
        const bool stop = *reinterpret_cast<volatile int *>(&ctrl.abort) != 0 || clock64() - start > ctrl.timeout_cycles;
        if (__any_sync(0xffffffffu, stop)) {
          if (lane == 0 && *reinterpret_cast<volatile int *>(&ctrl.abort) == 0) {
            *reinterpret_cast<volatile int *>(&ctrl.abort) = 1;
            atomicExch(status, 5);
          }
          return kCmdExit;
        }
      }
    }
  }
  if (lane == 0) *cell = 0;
  head = (head + 1) & (kFifoDepth - 1);
  return word;
}

// Three issuing warps: one for the first products of both slots, one for the second products of each
// slot.  None of them waits for anything but the inputs of its own next product.  Accumulation chains
// (O of a slot) stay within one thread, which is what tcgen05 orders.
template <int D>
__device__ void mma_role(const KernelParams &p, Ctrl &ctrl, uint8_t *smem_q, uint8_t *smem_ring, const int who,
                         const int lane) {
  using C = Cfg<D>;
  const uint32_t tmem = warp_uniform(ctrl.tmem_base, lane);
  const uint32_t idesc_s = make_idesc_bf16(kTile, kTile, 0, 0);
  const uint32_t idesc_pv = make_idesc_bf16(kTile, D, 0, 1);
  const uint64_t desc_q0 = make_smem_desc(smem_u32(smem_q), 16, 1024);
  const uint64_t desc_k0 = make_smem_desc(smem_u32(smem_ring), 16, 1024);
  const uint64_t desc_v0 = make_smem_desc(smem_u32(smem_ring), C::kBoxBytes, 1024);
  uint32_t head = 0;
  bool ok = true;
  auto wait = [&](uint64_t *bar, uint32_t parity) {
    if (ok) ok = bounded_wait(bar, parity, ctrl, p.status);
  };
  uint32_t cmd = fifo_pop_warp(ctrl, who, head, p.status, lane);
  while (!(cmd & kCmdExit)) {
    // look at the next command now, so that its shared-memory latency hides behind this one's issue
    volatile uint32_t *next_cell = &ctrl.fifo[who][head];
    __syncwarp();
    const uint32_t next_raw = *next_cell;
    const uint32_t slot = (cmd >> kCmdRingShift) & 0xFu;
    const uint32_t ring_phase = (cmd & kCmdRingPhase) ? 1u : 0u, use_phase = (cmd & kCmdUsePhase) ? 1u : 0u,
                   dep_phase = (cmd & kCmdDepPhase) ? 1u : 0u;
    if (elect_one()) {
      if (who == 0) {
        const uint32_t s = (cmd & kCmdSlot1) ? 1u : 0u;
        if (cmd & kCmdFirst) wait(&ctrl.q_full[s], use_phase);
        wait(&ctrl.ring_full[slot], ring_phase);
        if (cmd & kCmdWaitSFree) wait(&ctrl.s_free, dep_phase);
        if (ok) {
          tc_fence_after();
          const uint64_t dq = desc_q0 + uint64_t((s * C::kTileBytes) >> 4);
          const uint64_t dk = desc_k0 + uint64_t((slot * C::kTileBytes) >> 4);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t off = uint64_t(((kk / 4) * C::kBoxBytes + (kk % 4) * 32) >> 4);
            mma_ss(tmem + C::kColS, dq + off, dk + off, idesc_s, kk > 0);
          }
          tc_commit(&ctrl.s_full[s]);
          tc_commit_if(&ctrl.ring_empty[slot], cmd & kCmdFinal);
          tc_commit_if(&ctrl.q_empty[s], cmd & kCmdLast);
        }
      } else {
        const uint32_t s = who - 1;
        if (cmd & kCmdFirst) wait(&ctrl.o_empty[s], use_phase);
        wait(&ctrl.ring_full[slot], ring_phase);
        wait(&ctrl.p_full[s], dep_phase);
        if (ok) {
          // O_s += P_s V: P from its own TMEM columns, written by the softmax warps of slot s
          tc_fence_after();
          const uint64_t dv = desc_v0 + uint64_t((slot * C::kTileBytes) >> 4);
          const uint32_t t_p = tmem + C::kColP + s * (kTile / 2), t_o = tmem + C::kColO + s * D;
          const uint32_t acc0 = (cmd & kCmdFirst) ? 0u : 1u;
#pragma unroll
          for (int kk = 0; kk < kTile / 16; ++kk)
            mma_ts(t_o, t_p + kk * 8, dv + uint64_t((kk * 2048) >> 4), idesc_pv, kk > 0 ? 1u : acc0);
          tc_commit(&ctrl.p_free[s]);
          tc_commit(&ctrl.ring_empty[slot]);
          tc_commit_if(&ctrl.o_full[s], cmd & kCmdLast);
        }
      }
    }
    const uint32_t next = warp_uniform(next_raw, lane);
    if (__any_sync(0xffffffffu, !ok)) break;
    if (cmd_complete(next)) {
      if (lane == 0) *next_cell = 0;
      head = (head + 1) & (kFifoDepth - 1);
      cmd = next;
    } else {
      cmd = fifo_pop_warp(ctrl, who, head, p.status, lane);
    }
  }
  // Leaving on an expired wait: everything this warp issued must have retired before the CTA frees
  // its tensor memory, so commit to a spare barrier and wait for it (bounded).
  if (warp_aborted(ctrl)) {
    if (elect_one()) {
      tc_commit(&ctrl.drain[who]);
      const long long start = clock64();
      while (!mbar_try_wait(&ctrl.drain[who], 0) && clock64() - start < ctrl.timeout_cycles / 8) {
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// 2^y for a pair of exponents on the FMA pipe instead of the special-function unit: y = n + f with
// n = round(y), f in [-0.5, 0.5]; 2^f by a cubic with 7.5e-5 relative error (far below bf16's
// 2^-9), scaled by adding n to the exponent field.  Inputs must be finite or -inf; they are clamped
// at -125 so the exponent field stays positive (the result is then at most 2^-125).
__device__ __forceinline__ float2 exp2_poly(float2 y) {
  const float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to the nearest integer
  y.x = fmaxf(y.x, -125.0f);
  y.y = fmaxf(y.y, -125.0f);
  const float2 t = fadd2(y, make_float2(kMagic, kMagic));
  const float2 f = fadd2(y, fadd2(make_float2(kMagic, kMagic), make_float2(-t.x, -t.y)));
  float2 q = ffma2(make_float2(5.517166907e-02f, 5.517166907e-02f), f, make_float2(2.426111222e-01f, 2.426111222e-01f));
  q = ffma2(q, f, make_float2(6.932609855e-01f, 6.932609855e-01f));
  q = ffma2(q, f, make_float2(9.999280735e-01f, 9.999280735e-01f));
  q.x = __int_as_float(__float_as_int(q.x) + (__float_as_int(t.x) << 23));
  q.y = __int_as_float(__float_as_int(q.y) + (__float_as_int(t.y) << 23));
  return q;
}

// 2^y for a pair, on the FMA pipe, more exact than ex2.approx (relative error against 64 bits on [-30, 8]: at most
// 7.9e-8, root mean square 2.7e-8; ex2.approx 1.45e-7 and 5.7e-8): y = n + f as above, 2^f by a polynomial of degree 6
// with 2^0 = 1 (minimax for the relative error on [-0.5, 0.5], fitted by Lawson's iteration), times 2^n built in the
// exponent field.  Below -125.5 the result is 0, so a masked (-inf) score gives exactly 0; NaN stays NaN.  From 128 up it
// is +inf, which scores beyond 2^31 need: there the rounding of the maximum leaves such exponents.  That bound costs no
// instruction, because the number that rounds y stands 128 units below the largest float: t overflows to +inf by itself
// (n = +inf, f = -inf).  Its low nine bits are 0x17f, so t's are 0x17f + n; less one unit and shifted into sign and
// exponent they give -2^(n-1), and -inf for t = +inf, to go with -2 * 2^f, which is -inf then.  (A second comparison per
// exponent: 32 heads x 8192 339.5 -> 343.0 us, 12 heads x 512 8.81 -> 9.01; as here 338.4 -> 336.7, 8.81 -> 8.81.)
__device__ __forceinline__ float2 exp2_full(float2 y) {
  const float kRound = __uint_as_float(0x7f7fff7fu), kUnit = 0x1p104f;  // adding kRound rounds to multiples of kUnit
  y.x = fmax_nan(y.x, -126.0f);
  y.y = fmax_nan(y.y, -126.0f);
  const float2 t = ffma2(y, make_float2(kUnit, kUnit), make_float2(kRound, kRound));
  const float2 n = fadd2(t, make_float2(-kRound, -kRound));  // times kUnit
  const float2 f = ffma2(n, make_float2(-1.0f / kUnit, -1.0f / kUnit), y);
  float2 q = ffma2(make_float2(-3.07067240e-04f, -3.07067240e-04f), f, make_float2(-2.67977500e-03f, -2.67977500e-03f));
  q = ffma2(q, f, make_float2(-1.92368738e-02f, -1.92368738e-02f));
  q = ffma2(q, f, make_float2(-1.11006647e-01f, -1.11006647e-01f));
  q = ffma2(q, f, make_float2(-4.80452954e-01f, -4.80452954e-01f));
  q = ffma2(q, f, make_float2(-1.38629436e+00f, -1.38629436e+00f));
  q = ffma2(q, f, make_float2(-2.0f, -2.0f));
  const float2 power = make_float2(__uint_as_float((__float_as_uint(t.x) << 23) + 0xff800000u),
                                   __uint_as_float((__float_as_uint(t.y) << 23) + 0xff800000u));
  return fmul2(q, power);
}

// exp2 of 64 scaled scores -> 32 packed bf16x2 registers; accumulates the row sum in two lane pairs.
// With kEmu > 0, one pair in every 2^(3 - kEmu) is evaluated by exp2_poly (12.5 %, 25 %, 50 % of the
// exponentials leave the special-function unit for the FMA pipe: the counterpart of the lookup-table
// exponent the paper uses on the NPU generation that has no exponent unit).
// kShare: one pair in eight by exp2_full.  At head_dim 64 the special-function unit is what a tile waits for (2 048
// cycles for two tiles, their products take 1 024): 32 heads x 8192 340 -> 330 us, 2 x 12 heads x 4096 147 -> 144 us
// (one in six: 335, 145.6; degree 5, as exact as ex2.approx but no more: 328, 143).  At head_dim 128 the products take
// as long as the exponentials and it is slower (32 heads x 4096 121 -> 131 us).
template <int kEmu, bool kShare>
__device__ __forceinline__ void exp_half(const float (&x)[kTile], int base, float2 scale2, float2 neg_m2,
                                         float2 &acc_a, float2 &acc_b, uint32_t (&packed)[32]) {
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    const int e = base + 2 * i;
    float2 y0 = ffma2(make_float2(x[e], x[e + 1]), scale2, neg_m2);
    float2 y1 = ffma2(make_float2(x[e + 2], x[e + 3]), scale2, neg_m2);
    y0.x = ex2_approx(y0.x);
    y0.y = ex2_approx(y0.y);
    const bool emulate = kEmu > 0 && ((i / 2) % (1 << (3 - kEmu)) == (1 << (3 - kEmu)) - 1);
    if (emulate) {
      y1 = exp2_poly(y1);
    } else if (kEmu == 0 && kShare && (i / 2) % 4 == 3) {
      y1 = exp2_full(y1);
    } else {
      y1.x = ex2_approx(y1.x);
      y1.y = ex2_approx(y1.y);
    }
    acc_a = fadd2(acc_a, y0);
    acc_b = fadd2(acc_b, y1);
    packed[i] = pack_bf16x2(y0.x, y0.y);
    packed[i + 1] = pack_bf16x2(y1.x, y1.y);
  }
}

// ------------------------------------------------------------------------------------------------
// Split query tiles.  Every part counts its arrival per warp (32 rows); the warp that arrives last combines
// the parts of its rows, always in the order of the parts, so the result does not depend on who was last:
//   O = sum_i w_i O_i / sum_i w_i l_i,  w_i = 2^(m_i - max m).
// In fp32 throughout, as in TMEM.  Bound by the latency of its loads from L2 and, with full tiles, by what one
// SM can read, so a batch of loads is in flight together and lanes beyond the rows in use take a share of the
// columns.  (Loops over single parts: 500 queries on 12500 keys 103 us, as here 97 us.)
template <int D>
__device__ __forceinline__ float *part_buffer(const KernelParams &p, int n) {
  return p.parts + size_t(n) * size_t(p.part_rows) * (D + 2);
}

// Columns c0, c0 + step, ... of one row (in units of four columns): kCols of them from kBatch parts at a time.
// Returns sum_i w_i l_i.
template <int D, int kCols, int kBatch>
__device__ __forceinline__ float combine_columns(const float4 *col, const float2 *stat, size_t stride, int part_rows,
                                                 int n_parts, int c0, int step, float m, __nv_bfloat16 *o_row) {
  float4 acc[kCols] = {};
  float l = 0.0f;
#pragma unroll 1
  for (int i0 = 0; i0 < n_parts; i0 += kBatch) {
    float2 ml[kBatch];
    float4 v[kBatch][kCols];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      // beyond the last part zeros, not another part with weight 0: where its O is infinite, that is a NaN
      const bool in = i0 + b < n_parts;
      ml[b] = in ? __ldcg(stat + (i0 + b) * (stride / 2)) : make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < kCols; ++k)
        v[b][k] = in ? __ldcg(col + (i0 + b) * (stride / 4) + size_t(min(c0 + k * step, D / 4 - 1)) * part_rows)
                     : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const float w = ml[b].y > 0.0f ? ex2_approx(ml[b].x - m) : 0.0f;
      l = fmaf(w, ml[b].y, l);
#pragma unroll
      for (int k = 0; k < kCols; ++k) {
        acc[k].x = fmaf(w, v[b][k].x, acc[k].x);
        acc[k].y = fmaf(w, v[b][k].y, acc[k].y);
        acc[k].z = fmaf(w, v[b][k].z, acc[k].z);
        acc[k].w = fmaf(w, v[b][k].w, acc[k].w);
      }
    }
  }
  const float inv = l > 0.0f ? 1.0f / l : 0.0f;
#pragma unroll
  for (int k = 0; k < kCols; ++k)
    if (c0 + k * step < D / 4)
      *reinterpret_cast<uint2 *>(o_row + (c0 + k * step) * 4) =
          make_uint2(pack_bf16x2(acc[k].x * inv, acc[k].y * inv), pack_bf16x2(acc[k].z * inv, acc[k].w * inv));
  return l;
}

// Count one part of a split tile as ended for this warp's 32 rows.  True for the warp that ends last, which sets
// the counter back for the next launch.  Rows beyond the matrix are not counted (`used` <= 0).
__device__ __forceinline__ bool count_part(const KernelParams &p, int split, int n_parts, int used, int warp, int lane) {
  if (used <= 0) return false;
  int32_t *counter = p.arrivals + (split >> 6) * 4 + warp;
  __syncwarp();
  int before = 0;
  if (lane == 0) before = atomic_add_acq_rel(counter, 1);
  before = __shfl_sync(0xffffffffu, before, 0);
  __syncwarp();
  if (before != n_parts - 1) return false;
  if (lane == 0) *counter = 0;
  return true;
}

// A warp that leaves on an expired wait counts the parts of its items from k on all the same: every launch then
// counts every part once, and the counters are back at 0 for the next launch without any help from the host.
// (What is combined in this launch is undefined, as its status says.)
__device__ __noinline__ void count_abandoned_parts(const KernelParams &p, int k, int s, int warp, int lane) {
  for (const int k_end = p.cta_begin[blockIdx.x + 1]; k < k_end; ++k) {
    const Item w = load_item(p.items, k);
    if (!w.active(s) || w.split(s) < 0) continue;
    count_part(p, w.split(s), p.split_tiles[w.split(s) >> 6].n_parts, p.rows_q - w.qtile(s) * kTile - warp * 32, warp,
               lane);
  }
}

template <int D>
__device__ __forceinline__ void finish_part(const KernelParams &p, int split, int tile_row0, size_t tile_out_row,
                                            int warp, int lane) {
  const int used = min(32, p.rows_q - tile_row0 - warp * 32);
  const SplitTile tile = p.split_tiles[split >> 6];
  if (!count_part(p, split, tile.n_parts, used, warp, lane)) return;
  // `lanes` lanes share a row: lane = row + rows * share
  const int rows = used > 16 ? 32 : used > 8 ? 16 : used > 4 ? 8 : used > 2 ? 4 : used > 1 ? 2 : 1, lanes = 32 / rows;
  const int share = lane / rows;
  const bool valid = (lane & (rows - 1)) < used;
  const int r = warp * 32 + min(lane & (rows - 1), used - 1);
  const size_t stride = size_t(p.part_rows) * (D + 2);
  const float *base = part_buffer<D>(p, tile.first);
  const float2 *stat = reinterpret_cast<const float2 *>(base + size_t(D) * p.part_rows) + r;
  // max m: each lane of a row over its share of the parts, then over the lanes
  float m = -CUDART_INF_F;
#pragma unroll 1
  for (int i0 = share; i0 < tile.n_parts; i0 += 4 * lanes) {
    float top[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) top[b] = __ldcg(stat + min(i0 + b * lanes, tile.n_parts - 1) * (stride / 2)).x;
    m = fmax3(fmax3(m, top[0], top[1]), top[2], top[3]);
  }
#pragma unroll 1
  for (int step = rows; step < 32; step *= 2) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, step));
  if (valid) {
    float l = 0.0f;
    const size_t out_row = tile_out_row + size_t(r);
    __nv_bfloat16 *o_row = static_cast<__nv_bfloat16 *>(p.o) + out_row * D;
    const float4 *col = reinterpret_cast<const float4 *>(base) + r;
    // few rows: the shorter loop body, whose first pass through the instruction cache counts (a decode step with
    // 4 rows per tile: 41.1 -> 38.9 us)
    if (lanes <= 4) {
#pragma unroll 1
      for (int c0 = share; c0 < D / 4; c0 += 8 * lanes)
        l = combine_columns<D, 8, 4>(col, stat, stride, p.part_rows, tile.n_parts, c0, lanes, m, o_row);
    } else {
#pragma unroll 1
      for (int c0 = share; c0 < D / 4; c0 += 4 * lanes)
        l = combine_columns<D, 4, 4>(col, stat, stride, p.part_rows, tile.n_parts, c0, lanes, m, o_row);
    }
    if (p.lse != nullptr && share == 0)
      p.lse[out_row] = l > 0.0f ? 0.6931471805599453f * (m + log2f(l)) : -CUDART_INF_F;
  }
  __syncwarp();
}

// Returns -1, or the item in which a wait expired.
template <int D, int kEmu, bool kSplit, bool kList>
__device__ int softmax_role(const KernelParams &p, Ctrl &ctrl, const int s, const int r) {
  using C = Cfg<D>;
  const int lane = r % 32;
  const uint32_t lane_base = uint32_t((r / 32) * 32) << 16;
  const uint32_t t_s = ctrl.tmem_base + lane_base + C::kColS;
  const uint32_t t_p = ctrl.tmem_base + lane_base + C::kColP + s * (kTile / 2);
  const uint32_t t_o = ctrl.tmem_base + lane_base + C::kColO + s * D;
  const bool causal = (p.mask_flags & kMaskCausal) != 0, windowed = (p.mask_flags & kMaskWindow) != 0;
  const int off = p.seq_kv - p.seq_q;
  const float scale_log2 = p.scale_log2;
  const float2 scale2 = make_float2(scale_log2, scale_log2);
  __nv_bfloat16 *o_base = static_cast<__nv_bfloat16 *>(p.o);
  uint32_t n_sp = 0, n_use = 0;

  const int k_end = p.cta_begin[blockIdx.x + 1];
  for (int k = p.cta_begin[blockIdx.x]; k < k_end; ++k) {
    const Item w = load_item(p.items, k);
    if (k + 1 < k_end) prefetch_l1(p.items + k + 1);  // a miss at the start of an item costs 1 000 cycles
    if (w.head(s) < 0) continue;
    const int row = w.qtile(s) * kTile + r;
    const size_t out_row = (size_t(w.batch) * p.heads_q + w.head(s)) * size_t(p.rows_q) + size_t(row);
    float m_ref = -CUDART_INF_F, l = 0.0f;
    const int lo = w.lo(s), hi = w.hi(s);
    const bool active = hi >= lo;

    // Range items: tiles f_lo .. f_hi need no element-wise mask (case ii).  List items carry it in the entry.
    int f_lo = 0, f_hi = p.seq_kv / kTile - 1;
    const int r0 = w.qtile(s) * kTile, r1 = min(r0 + kTile, p.rows_q) - 1;
    // first and last position in the tile; one that spans several heads spans all positions.  (Divisions only where rows
    // of several heads are packed: 100 cycles each, and one per partial tile.)
    int pos0 = r0, pos1 = r1, pos_row = row;
    if (p.rows_q != p.seq_q) {
      const bool one_head = r0 / p.seq_q == r1 / p.seq_q;
      pos0 = one_head ? r0 % p.seq_q : 0;
      pos1 = one_head ? r1 % p.seq_q : p.seq_q - 1;
      pos_row = row % p.seq_q;
    }
    if (causal) f_hi = min(f_hi, (pos0 + off + 1) / kTile - 1);
    if (windowed) {
      const int first = pos1 + off - p.window + 1;
      f_lo = first > 0 ? (first + kTile - 1) / kTile : 0;
    }
    const uint32_t *entries = reinterpret_cast<const uint32_t *>(p.steps + w.list_off()) + s;
    uint32_t next_entry = (kList && w.kind != 0 && active) ? __ldg(entries + 2 * lo) : 0u;

    for (int t = lo; t <= hi; ++t) {
      // which key tile, and does it need the element-wise mask (case iii)?
      int j = w.j0(s) + t;
      bool partial = j < f_lo || j > f_hi;
      uint32_t sub = 0xF;
      if (kList && w.kind != 0) {
        const uint32_t e = next_entry;
        next_entry = t < hi ? __ldg(entries + 2 * (t + 1)) : 0u;
        j = int(e & kEntryTileMask);
        partial = (e & kEntryPartial) != 0;
        sub = (e >> kEntrySubShift) & 0xF;
      }

      bool ok;
      {
        ok = warp_wait(&ctrl.s_full[s], n_sp & 1u, ctrl);
      }
      if (!ok) return k;
      tc_fence_after();

      float x[kTile];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t regs[32];
        tmem_ld32(t_s + c * 32, regs);
#pragma unroll
        for (int i = 0; i < 32; ++i) x[c * 32 + i] = __uint_as_float(regs[i]);
      }
      tc_wait_ld();
      // the scores are in registers: hand the S buffer back for the next QK^T (of either slot)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl.s_free);

      if (partial) {
        // visible columns of this row form one interval [c_lo, c_hi] of the tile
        const int pos = pos_row + off, jb = j * kTile;  // key position aligned with the row's query
        int c_hi = min(kTile - 1, p.seq_kv - 1 - jb), c_lo = 0;
        if (causal) c_hi = min(c_hi, pos - jb);
        if (windowed) c_lo = max(c_lo, pos - p.window + 1 - jb);
        const uint32_t half = (sub >> (2 * (r / 64))) & 3u;  // bit 0: keys 0-63 enabled, bit 1: keys 64-127
        if (!(half & 1u)) c_lo = max(c_lo, 64);
        if (!(half & 2u)) c_hi = min(c_hi, 63);
        // As bits c_lo .. c_hi of four words: a bit test and a select per score instead of two comparisons
        // and a select.  The code sits in the tile loop, so every tile gains (the instruction stream is what
        // the softmax warps wait for most): 32 heads x 8192 causal d64 382 -> 367 us, batch 4 x 1777 92.5 ->
        // 87 us, 64-token bitmap blocks (every tile partial), 4 heads x 2048: 30.5 -> 25.8 us.
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int a = min(max(c_lo - 32 * q, 0), 32), b = min(max(c_hi + 1 - 32 * q, 0), 32);
          const uint32_t keep = (b < 32 ? (1u << b) - 1u : 0xffffffffu) & ~(a < 32 ? (1u << a) - 1u : 0xffffffffu);
#pragma unroll
          for (int c = 0; c < 32; ++c) x[32 * q + c] = (keep >> c) & 1u ? x[32 * q + c] : -CUDART_INF_F;
        }
      }

      float mx0 = fmax3(x[0], x[1], x[2]), mx1 = fmax3(x[3], x[4], x[5]);
      float mx2 = fmax3(x[6], x[7], x[8]), mx3 = fmax3(x[9], x[10], x[11]);
#pragma unroll
      for (int c = 12; c < 124; c += 8) {
        mx0 = fmax3(mx0, x[c], x[c + 1]);
        mx1 = fmax3(mx1, x[c + 2], x[c + 3]);
        mx2 = fmax3(mx2, x[c + 4], x[c + 5]);
        mx3 = fmax3(mx3, x[c + 6], x[c + 7]);
      }
      mx0 = fmax3(mx0, x[124], x[125]);
      mx1 = fmax3(mx1, x[126], x[127]);
      const float ms = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * scale_log2;

      // the running maximum only has to bound the exponents: O is rescaled lazily, once PV(s, t - 1) has finished
      const float m_old = m_ref;
      const bool grown = ms > m_ref + kRescaleThreshold;
      if (grown) m_ref = ms;
      const bool need = grown && t > lo;
      const float m_use = (m_ref == -CUDART_INF_F) ? 0.0f : m_ref;
      const float2 neg_m2 = make_float2(-m_use, -m_use);

      float2 acc_a = make_float2(0.f, 0.f), acc_b = make_float2(0.f, 0.f);
      uint32_t p_lo[32], p_hi[32];
      exp_half<kEmu, D == 64>(x, 0, scale2, neg_m2, acc_a, acc_b, p_lo);
      exp_half<kEmu, D == 64>(x, 64, scale2, neg_m2, acc_a, acc_b, p_hi);
      // PV(s, t - 1) reads the P columns and accumulates into O: it must have finished before either is written.  P
      // stays in registers until here, because products that are issued at the same time share the tensor core:
      // with an S beside it PV takes up to 1 024 cycles, and a softmax warp that waits for it halfway through its
      // exponentials stands still.  (At a slot's first step the barrier is complete or in its initial phase.)  One vote
      // decides about both, the wait and the rare rescale: each vote and branch in this loop costs the warp about
      // 100 cycles of its 2 700 per tile.  P stored in halves -> here: 32 heads x 8192 d64 352 -> 337 us, 32 heads x
      // 4096 d128 123.4 -> 119.3 us, window 4096 of 16384 796 -> 755 us, 500 queries on 12500 keys 95.1 -> 90.5 us.
      if (!__all_sync(0xffffffffu, mbar_test_wait(&ctrl.p_free[s], (n_sp - 1u) & 1u) && !need)) {
        if (!warp_wait(&ctrl.p_free[s], (n_sp - 1u) & 1u, ctrl)) return k;
        if (__any_sync(0xffffffffu, need)) {
          tc_fence_after();
          // kept short, so that the loop around it needs fewer instructions from the cache
          const float v = need ? ex2_approx(m_old - m_ref) : 1.0f;
          l *= v;
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {
            uint32_t regs[16];
            tmem_ld16(t_o + c * 16, regs);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) regs[i] = __float_as_uint(__uint_as_float(regs[i]) * v);
            tmem_st16(t_o + c * 16, regs);
          }
        }
      }
      tc_fence_after();
      tmem_st32(t_p, p_lo);
      tmem_st32(t_p + 32, p_hi);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl.p_full[s]);
      ++n_sp;
      const float2 acc = fadd2(acc_a, acc_b);
      // The polynomial path returns 2^-125 rather than 0 for a masked (-inf) score: a row that has
      // not seen a visible key yet (m = -inf) must keep l = 0 exactly, so that it ends as O = 0.
      if (kEmu == 0 || m_ref != -CUDART_INF_F) l += acc.x + acc.y;
    }

    // epilogue: O / l and LSE = ln2 * (m + log2 l)
    if (active) {
      bool ok;
      {
        ok = warp_wait(&ctrl.o_full[s], n_use & 1u, ctrl);
      }
      if (!ok) return k;
      ++n_use;
      tc_fence_after();
      const bool valid = row < p.rows_q;
      const int split = kSplit ? w.split(s) : -1;
      if (kSplit && split >= 0) {
        // one of several key ranges of this query tile: leave O and (m, l) for the part that ends last
        float *part = part_buffer<D>(p, p.split_tiles[split >> 6].first + (split & 63));
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t regs[32];
          tmem_ld32(t_o + c * 32, regs);
          tc_wait_ld();
          if (valid) {
            uint4 *dst = reinterpret_cast<uint4 *>(part) + size_t(c) * 8 * p.part_rows + r;
#pragma unroll
            for (int i = 0; i < 8; ++i)
              dst[i * p.part_rows] = make_uint4(regs[4 * i], regs[4 * i + 1], regs[4 * i + 2], regs[4 * i + 3]);
          }
        }
        if (valid) reinterpret_cast<float2 *>(part + size_t(D) * p.part_rows)[r] = make_float2(m_ref, l);
      } else {
        const float inv = l > 0.0f ? 1.0f / l : 0.0f;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t regs[32];
          tmem_ld32(t_o + c * 32, regs);
          tc_wait_ld();
          if (valid) {
            // A row's 64 bytes as two 32-byte stores: whole sectors, and half as many passes through L1 (each lane
            // writes a line of its own, and what bounds the epilogue is one line per cycle).  16-byte stores ->
            // here: batch 4 24/8 x 1777 79.8 -> 77.8 us, window 4096 of 16384 744 -> 731 us.  Turning pieces
            // among four lanes by shuffles, for whole lines, took longer than it saved (95 us).
            __nv_bfloat16 *dst = o_base + out_row * D + c * 32;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t v[8];
#pragma unroll
              for (int e = 0; e < 8; ++e)
                v[e] = pack_bf16x2(__uint_as_float(regs[16 * i + 2 * e]) * inv, __uint_as_float(regs[16 * i + 2 * e + 1]) * inv);
              if (p.o_aligned32) {
                store_global32(dst + 16 * i, v);
              } else {
                reinterpret_cast<uint4 *>(dst)[2 * i] = make_uint4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<uint4 *>(dst)[2 * i + 1] = make_uint4(v[4], v[5], v[6], v[7]);
              }
            }
          }
        }
        if (p.lse != nullptr && valid)
          p.lse[out_row] = l > 0.0f ? 0.6931471805599453f * (m_ref + log2f(l)) : -CUDART_INF_F;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl.o_empty[s]);
      if (kSplit && split >= 0) finish_part<D>(p, split, w.qtile(s) * kTile, out_row - size_t(r), r / 32, lane);
    } else if (row < p.rows_q) {
      // no key tile is visible to this query tile
      uint4 *dst = reinterpret_cast<uint4 *>(o_base + out_row * D);
#pragma unroll
      for (int i = 0; i < D / 8; ++i) dst[i] = make_uint4(0u, 0u, 0u, 0u);
      if (p.lse != nullptr) p.lse[out_row] = -CUDART_INF_F;
    }
  }
  return -1;
}

// ------------------------------------------------------------------------------------------------
template <int D, int kEmu, bool kSplit, bool kList>
__global__ void __launch_bounds__(kThreads, 1)
steel_attn_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const __grid_constant__ CUtensorMap map_v, const __grid_constant__ KernelParams p) {
  using C = Cfg<D>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Ctrl ctrl;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *smem_q = smem;
  uint8_t *smem_ring = smem + 2 * C::kTileBytes;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int i = 0; i < C::kStages; ++i) {
      mbar_init(&ctrl.ring_full[i], 1);
      mbar_init(&ctrl.ring_empty[i], 2);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&ctrl.q_full[s], 1);
      mbar_init(&ctrl.q_empty[s], 1);
      mbar_init(&ctrl.s_full[s], 1);
      mbar_init(&ctrl.p_full[s], 4);  // one arrival per softmax warp
      mbar_init(&ctrl.p_free[s], 1);
      mbar_init(&ctrl.o_full[s], 1);
      mbar_init(&ctrl.o_empty[s], 4);
    }
    mbar_init(&ctrl.s_free, 4);
    for (int i = 0; i < 3; ++i) mbar_init(&ctrl.drain[i], 1);
    for (int i = 0; i < 3 * kFifoDepth; ++i) ctrl.fifo[0][i] = 0;
    ctrl.abort = 0;
    ctrl.timeout_cycles = p.timeout_cycles;
    fence_barrier_init();
  }
  if (warp == kProducerWarp && lane == 0) {
    prefetch_tensormap(&map_q);
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&ctrl.tmem_base, 512);
    tmem_relinquish();
  }
  // From here on the next launch on the stream may set itself up on SMs that this one leaves; this launch in
  // turn touches global memory only after the one before it has completed.
  grid_launch_dependents();
  grid_dependency_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  if (warp < 8) {
    setmaxnreg_inc<kRegsSoftmax>();
    const int left = softmax_role<D, kEmu, kSplit, kList>(p, ctrl, warp / 4, threadIdx.x % kTile);
    if (left >= 0 && lane == 0 && *reinterpret_cast<volatile int *>(&ctrl.abort) == 0) {
      *reinterpret_cast<volatile int *>(&ctrl.abort) = 1;
      atomicExch(p.status, 5);
    }
    if (kSplit && left >= 0) count_abandoned_parts(p, left, warp / 4, warp % 4, lane);
  } else {
    setmaxnreg_dec<kRegsOther>();
    if (warp == kProducerWarp) {
      if (lane == 0) producer_role<D, kList>(p, &map_q, &map_k, &map_v, ctrl, smem_q, smem_ring);
    } else if (warp >= kMmaWarp) {
      mma_role<D>(p, ctrl, smem_q, smem_ring, warp - kMmaWarp, lane);
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(ctrl.tmem_base, 512);
}

namespace {

// Builds.  kSplit: combines split query tiles.  kList: items may be lists (bitmap masks).  Each is a kernel of
// its own because the tile loop is bound by its instruction stream: without the list code the range masks take
// 32 heads x 8192 d64 371 -> 364 us, 32 heads x 4096 125.3 -> 123.1 us, 12 heads x 512 d64 8.9 -> 8.65 us.
// Software exponents are built with the list code only.
template <int D, int kEmu, bool kSplit, bool kList>
cudaError_t configure_build() {
  return cudaFuncSetAttribute(steel_attn_kernel<D, kEmu, kSplit, kList>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              Cfg<D>::kSmemBytes);
}

template <int D, int kEmu>
cudaError_t configure_one() {
  cudaError_t e = configure_build<D, kEmu, false, true>();
  if (e == cudaSuccess) e = configure_build<D, kEmu, true, true>();
  if (kEmu == 0 && e == cudaSuccess) e = configure_build<D, kEmu, false, kEmu != 0>();
  if (kEmu == 0 && e == cudaSuccess) e = configure_build<D, kEmu, true, kEmu != 0>();
  return e;
}

template <int D, int kEmu>
void launch_one(const CUtensorMap &map_q, const CUtensorMap &map_k, const CUtensorMap &map_v,
                const KernelParams &params, int grid, cudaStream_t stream) {
  cudaLaunchConfig_t config = {};
  config.gridDim = dim3(grid);
  config.blockDim = dim3(kThreads);
  config.dynamicSmemBytes = Cfg<D>::kSmemBytes;
  config.stream = stream;
  cudaLaunchAttribute overlap;
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  config.attrs = &overlap;
  config.numAttrs = params.overlap_launch ? 1 : 0;
  const bool split = params.split_tiles != nullptr, list = kEmu != 0 || (params.mask_flags & kMaskBitmap) != 0;
  auto *kernel = split ? (list ? steel_attn_kernel<D, kEmu, true, true> : steel_attn_kernel<D, kEmu, true, kEmu != 0>)
                       : (list ? steel_attn_kernel<D, kEmu, false, true> : steel_attn_kernel<D, kEmu, false, kEmu != 0>);
  cudaLaunchKernelEx(&config, kernel, map_q, map_k, map_v, params);
}

template <int D>
void launch_dim(int exp_emulation, const CUtensorMap &map_q, const CUtensorMap &map_k, const CUtensorMap &map_v,
                const KernelParams &params, int grid, cudaStream_t stream) {
  switch (exp_emulation) {
    case 1: launch_one<D, 1>(map_q, map_k, map_v, params, grid, stream); break;
    case 2: launch_one<D, 2>(map_q, map_k, map_v, params, grid, stream); break;
    case 3: launch_one<D, 3>(map_q, map_k, map_v, params, grid, stream); break;
    default: launch_one<D, 0>(map_q, map_k, map_v, params, grid, stream); break;
  }
}

}  // namespace

cudaError_t configure_kernels(int head_dim, int exp_emulation) {
  const bool wide = head_dim == 128;
  switch (exp_emulation) {
    case 1: return wide ? configure_one<128, 1>() : configure_one<64, 1>();
    case 2: return wide ? configure_one<128, 2>() : configure_one<64, 2>();
    case 3: return wide ? configure_one<128, 3>() : configure_one<64, 3>();
    default: return wide ? configure_one<128, 0>() : configure_one<64, 0>();
  }
}

cudaError_t configure_kernels() {
  cudaError_t e = cudaSuccess;
  for (int emulation = 0; emulation <= 3; ++emulation)
    for (int head_dim : {64, 128})
      if (e == cudaSuccess) e = configure_kernels(head_dim, emulation);
  return e;
}

cudaError_t launch_attention(int head_dim, int exp_emulation, const CUtensorMap &map_q, const CUtensorMap &map_k,
                             const CUtensorMap &map_v, const KernelParams &params, int grid, cudaStream_t stream) {
  if (head_dim == 128)
    launch_dim<128>(exp_emulation, map_q, map_k, map_v, params, grid, stream);
  else
    launch_dim<64>(exp_emulation, map_q, map_k, map_v, params, grid, stream);
  return cudaGetLastError();
}

}  // namespace steel
