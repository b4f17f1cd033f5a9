// Compares the two ways to the step lists of single query tiles under a bitmap mask, for tests/test_plan_spread_lists.py:
// the planner's own, and BitmapMask::entry over all key tiles in ascending order, as the device writes them.  Host code
// only.  usage: list_entries cases seed; prints the number of plans of single tiles, or the first difference.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "../paper_2607_09385_b200/csrc/steel_planner.h"

using namespace steel;

int main(int argc, char **argv) {
  if (argc < 3) return 2;
  std::mt19937 g(std::atoi(argv[2]));
  auto pick = [&](int lo, int hi) { return lo + int(g() % unsigned(hi - lo + 1)); };
  int compared = 0;
  for (int n = 0; n < std::atoi(argv[1]); ++n) {
    steel_attn_params_t p{};
    p.batch = pick(1, 2);
    p.heads_kv = pick(1, 3);
    p.heads_q = p.heads_kv * pick(1, 3);
    p.seq_q = pick(1, 1500);
    p.seq_kv = pick(1, 2600);
    p.head_dim = 64;
    p.scale = 1.0f;
    p.mask.flags = STEEL_MASK_BITMAP | (pick(0, 1) ? STEEL_MASK_CAUSAL : 0u) | (pick(0, 2) == 0 ? STEEL_MASK_WINDOW : 0u);
    p.mask.window = pick(1, 1200);
    p.mask.block_q = p.mask.block_kv = pick(0, 1) ? 64 : 128;
    const BitmapMask m = bitmap_mask(p);
    std::vector<uint32_t> words(size_t(p.heads_q) * m.blocks_q * m.words);
    const int dense = pick(0, 4);  // bits outside the problem are set, too
    for (uint32_t &w : words) w = dense == 0 ? 0u : dense == 4 ? 0xFFFFFFFFu : g() & (dense > 1 ? 0xFFFFFFFFu : g());
    p.mask.bitmap = words.data();
    Plan host, device;
    if (build_plan(&p, 148, &host, false, Spread::kTiles) != STEEL_OK ||
        build_plan(&p, 148, &device, false, Spread::kTiles, nullptr, true) != STEEL_OK)
      return 3;
    if (device.steps.empty() && device.n_steps > 0) {
      ++compared;
      device.steps.assign(size_t(device.n_steps), StepPair{{0u, 0u}});
      for (const WorkItem &w : device.items) {
        if (w.kind != 1) continue;
        const uint32_t *rows = words.data() + size_t(w.head[0]) * m.blocks_q * m.words;
        int at = 0;
        for (int J = 0; J < m.key_tiles(); ++J)
          if (const uint32_t e = m.entry(rows, w.qtile[0], J)) {
            if (at < w.n_steps) device.steps[size_t(w.j0[0] + at)].e[0] = e;
            ++at;
          }
        if (at != w.n_steps) return std::printf("case %d: %d entries for a list of %d\n", n, at, w.n_steps), 1;
      }
    }
    if (host.items.size() != device.items.size() || host.cta_begin != device.cta_begin ||
        host.n_steps != device.n_steps || host.steps.size() != device.steps.size() ||
        std::memcmp(host.items.data(), device.items.data(), host.items.size() * sizeof(WorkItem)) != 0 ||
        (!host.steps.empty() &&
         std::memcmp(host.steps.data(), device.steps.data(), host.steps.size() * sizeof(StepPair)) != 0))
      return std::printf("case %d differs: %d x %d/%d heads, %d x %d, flags %u window %lld block %d\n", n, p.batch, p.heads_q,
                         p.heads_kv, p.seq_q, p.seq_kv, p.mask.flags, (long long)p.mask.window, p.mask.block_q), 1;
  }
  std::printf("%d\n", compared);
  return 0;
}
