// Prints how steel_attn_run_noalloc lays out a call, for tests/test_noalloc_plan.py, after checking that what it keeps
// lies in the fixed array in order, aligned and without overlap.  Host code only.
// usage: noalloc_plan batch heads_q heads_kv seq_q seq_kv flags window block words-value (hex, for every word)
// prints: items, list entries, 1 if the device writes them; or "refused"
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
  steel::NoallocPlan np;
  const steel_status_t st = steel::plan_noalloc(&p, 148, &np);
  if (st == STEEL_ERR_UNSUPPORTED) return std::puts("refused"), 0;
  if (st != STEEL_OK) return 3;
  const steel::Plan &plan = np.plan;
  const size_t steps = size_t(plan.n_steps) * sizeof(steel::StepPair), bitmap = words.size() * sizeof(uint32_t);
  const bool in_order = np.off_cta_begin >= sizeof(int32_t) &&
                        np.off_items >= np.off_cta_begin + plan.cta_begin.size() * sizeof(int32_t) &&
                        np.off_bitmap >= np.off_items + plan.items.size() * sizeof(steel::WorkItem) &&
                        np.off_steps >= np.off_bitmap + np.bitmap_bytes && np.end >= np.off_steps + steps &&
                        np.end <= steel::kNoallocBytes && np.copy_bytes <= np.end;
  const bool aligned = np.off_cta_begin % 4 == 0 && np.off_items % 64 == 0 && np.off_bitmap % 4 == 0 && np.off_steps % 16 == 0;
  const bool copied = np.device_lists ? np.bitmap_bytes == bitmap && np.copy_bytes == np.off_bitmap + bitmap && plan.steps.empty()
                                      : np.bitmap_bytes == 0 && np.copy_bytes >= np.off_steps + steps &&
                                            plan.steps.size() == size_t(plan.n_steps);
  if (!in_order || !aligned || !copied) return std::printf("layout %d %d %d\n", in_order, aligned, copied), 4;
  std::printf("%zu %lld %d\n", plan.items.size(), (long long)plan.n_steps, int(np.device_lists));
  return 0;
}
