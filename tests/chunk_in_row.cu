// Host check of the hub sweep's test that a chunk lies inside its row, at the
// last positions that 32 bits hold, against 64-bit sums. Chunks that the walk
// reaches start at or before the end of a row of at least a chunk.
#include <cstdio>

#include "../paper_2609_21848_gb300/csrc/sweep_device.cuh"

int main() {
  const uint32_t ends[] = {0u, 1u, 127u, 128u, 0x7FFFFFFFu, 0x80000000u, 0xFFFFFF80u, 0xFFFFFFFDu, 0xFFFFFFFEu};
  int wrong = 0;
  for (uint32_t en : ends)
    for (uint32_t back = 0; back <= 300 && back <= en; back++)
      for (uint32_t n = 4; n <= 128 && n <= en; n *= 2) {
        const uint32_t c = en - back;
        wrong += (c <= dbbc::last_chunk(en, n)) != ((uint64_t)c + n <= (uint64_t)en);
      }
  std::printf("%d wrong\n", wrong);
  return wrong ? 1 : 0;
}
