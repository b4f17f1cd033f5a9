// Prints where the step lists of steel_attn_run_noalloc are written, for tests/test_noalloc_plan.py.  Host code only.
// usage: noalloc_plan batch heads_q heads_kv seq_q seq_kv flags window block words-value (hex, for every word)
// prints: items, list entries, 1 if the device writes them
#include <cstdio>
#include <cstdlib>

#include "../paper_2607_09385_b200/csrc/steel_planner.h"

int main(int argc, char **argv) {
  if (argc != 10) return 2;
  steel_attn_params_t p{};
  p.batch = std::atoi(argv[1]);
  p.heads_q = std::atoi(argv[2]);
  p.heads_kv = std::atoi(argv[3]);
  p.seq_q = std::atoi(argv[4]);
  p.seq_kv = std::atoi(argv[5]);
  p.head_dim = 64;
  p.scale = 1.0f;
  p.mask.flags = uint32_t(std::atoi(argv[6]));
  p.mask.window = std::atoi(argv[7]);
  p.mask.block_q = p.mask.block_kv = std::atoi(argv[8]);
  const steel::BitmapMask m = steel::bitmap_mask(p);
  const std::vector<uint32_t> words(size_t(p.heads_q) * m.blocks_q * m.words, uint32_t(std::strtoul(argv[9], nullptr, 16)));
  p.mask.bitmap = words.data();
  steel::Plan plan;
  const steel_status_t st = steel::build_plan(&p, 148, &plan, false, steel::Spread::kTiles, nullptr, true);
  if (st != STEEL_OK) return 3;
  std::printf("%zu %lld %d\n", plan.items.size(), (long long)plan.n_steps, int(plan.steps.empty() && plan.n_steps > 0));
  return 0;
}
