// Prints the plan that steel_attn_create builds, for tests/test_plan_spread.py and tests/test_gpu_spread.py.  Host code
// only.  usage: plan_dump ctas batch heads_q heads_kv seq_q seq_kv flags window block [bitmap words in hex ...]
#include <cstdio>
#include <cstdlib>

#include "../paper_2607_09385_b200/csrc/steel_planner.h"

int main(int argc, char **argv) {
  if (argc < 10) return 2;
  std::vector<uint32_t> bitmap;
  for (int n = 10; n < argc; ++n) bitmap.push_back(uint32_t(std::strtoul(argv[n], nullptr, 16)));
  steel_attn_params_t p{};
  p.batch = std::atoi(argv[2]);
  p.heads_q = std::atoi(argv[3]);
  p.heads_kv = std::atoi(argv[4]);
  p.seq_q = std::atoi(argv[5]);
  p.seq_kv = std::atoi(argv[6]);
  p.head_dim = 64;
  p.scale = 1.0f;
  p.mask.flags = uint32_t(std::atoi(argv[7]));
  p.mask.window = std::atoi(argv[8]);
  p.mask.block_q = p.mask.block_kv = std::atoi(argv[9]);
  p.mask.bitmap = bitmap.empty() ? nullptr : bitmap.data();
  steel::Plan plan;
  if (steel::build_plan(&p, std::atoi(argv[1]), &plan, true, steel::Spread::kCut) != STEEL_OK) return 3;
  std::printf("plan %d %d %d %d\n", plan.grid, int(plan.packed), plan.n_parts, int(plan.items.size()));
  for (const steel::SplitTile &t : plan.split_tiles) std::printf("split %d %d\n", t.first, t.n_parts);
  for (size_t c = 0; c + 1 < plan.cta_begin.size(); ++c)
    for (int n = plan.cta_begin[c]; n < plan.cta_begin[c + 1]; ++n) {
      const steel::WorkItem &w = plan.items[n];
      std::printf("item %d %d %d %d %d %d %d\n", int(c), w.n_steps, w.kind, w.lo[0], w.hi[0], w.lo[1], w.hi[1]);
      for (int s = 0; s < 2; ++s) {
        if (w.head[s] < 0) continue;
        std::printf("slot %d %d %d %d %d", s, w.batch, w.head[s], w.qtile[s], w.split[s]);
        for (int t = w.lo[s]; t <= w.hi[s]; ++t) {
          const uint32_t e = steel::item_entry(plan, w, s, t, &p);
          std::printf(" %u:%d", e & steel::kEntryTileMask, (e & steel::kEntryPartial) != 0);
        }
        std::printf("\n");
      }
    }
  return 0;
}
