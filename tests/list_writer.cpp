// Runs the writing of a query tile's step list (ListWriter) with 32 lanes in turn, for tests/test_noalloc_plan.py: the
// list's length as planned, too short and too long by some entries.  Host code only.
#include <cstdio>
#include <random>

#include "../paper_2607_09385_b200/csrc/steel_planner.h"

using namespace steel;

int main() {
  std::mt19937 g(7);
  const StepPair untouched{{0x12345678u, 0x9abcdef0u}};
  for (int n = 0; n < 300; ++n) {
    BitmapMask m{};
    m.block = n % 2 ? 64 : 128;
    m.seq_q = kTile;
    m.seq_kv = 1 + int(g() % 20000);
    m.off = m.seq_kv - m.seq_q;
    m.blocks_q = int32_t(kTile / m.block);
    m.blocks_kv = int32_t((m.seq_kv + m.block - 1) / m.block);
    m.words = (m.blocks_kv + 31) / 32;
    std::vector<uint32_t> words(size_t(m.blocks_q) * m.words), entries;
    for (uint32_t &w : words) w = g() & (n % 3 ? g() : 0xFFFFFFFFu);
    for (int J = 0; J < m.key_tiles(); ++J)
      if (const uint32_t e = m.entry(words.data(), 0, J)) entries.push_back(e);
    const int found = int(entries.size());
    for (int planned : {found, found + 1, found + 40, found - 1, found / 2, 0}) {
      if (planned < 0) continue;
      std::vector<StepPair> out(size_t(planned) + 64, untouched);
      ListWriter lane[32];
      for (ListWriter &l : lane) l = ListWriter{out.data(), planned};
      for (int j0 = 0; j0 < m.key_tiles(); j0 += 32) {
        uint32_t e[32], seen = 0;
        for (int i = 0; i < 32; ++i) {
          e[i] = j0 + i < m.key_tiles() ? m.entry(words.data(), 0, j0 + i) : 0u;
          seen |= uint32_t(e[i] != 0) << i;
        }
        for (int i = 0; i < 32; ++i) lane[i].place(i, e[i], seen);
      }
      for (int i = 0; i < 32; ++i)
        if (lane[i].finish(i) != (planned == found)) return std::printf("%d of %d entries: not noticed\n", found, planned), 1;
      for (int k = 0; k < planned + 64; ++k) {
        const StepPair &s = out[size_t(k)];
        if (k >= planned ? s.e[0] != untouched.e[0] || s.e[1] != untouched.e[1]
            : k < found  ? s.e[0] != entries[size_t(k)] || s.e[1] != 0
                         : !(s.e[0] & kEntryPresent) || (s.e[0] & kEntryTileMask) != 0 || s.e[1] != 0)
          return std::printf("place %d of %d, %d entries\n", k, planned, found), 1;
      }
    }
  }
  return 0;
}
