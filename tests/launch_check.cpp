// Host-side check of the update's launch arithmetic
// (paper_1805_07920_gb300/csrc/amh_launch.h).
#include <cstdio>

#include "../paper_1805_07920_gb300/csrc/amh_launch.h"

using namespace amh;

static int fails = 0;
#define CHECK(cond, ...)                                                   \
  do {                                                                     \
    if (!(cond)) {                                                         \
      std::printf("FAIL %s: ", #cond), std::printf(__VA_ARGS__), fails++; \
      std::printf("\n");                                                   \
    }                                                                      \
  } while (0)

int main() {
  long n = 0;
  for (int sm : {1, 2, 78, 148, 152, 160})
    for (int most = 1; most <= 4; most++)
      for (int64_t tiles = 1; tiles < 6000; tiles += tiles < 3000 ? 1 : 97, n++) {
        const int k = blocks_per_sm(tiles, sm, most);
        const int64_t grid = std::min<int64_t>(tiles, (int64_t)k * sm);
        const int64_t rounds = (tiles + grid - 1) / grid, full = (tiles + (int64_t)most * sm - 1) / ((int64_t)most * sm);
        CHECK(k >= 1 && k <= most && grid >= 1 && grid <= tiles, "sm %d most %d tiles %ld: %d", sm, most, (long)tiles, k);
        CHECK(rounds == full, "sm %d most %d tiles %ld: %ld rounds, %ld with all blocks", sm, most, (long)tiles, (long)rounds, (long)full);
        // one or two rounds: fewer blocks per SM would need more rounds; longer: all of them
        CHECK(full > 2 ? k == most : k == 1 || (int64_t)(k - 1) * sm * full < tiles, "sm %d most %d tiles %ld: %d", sm, most, (long)tiles, k);
        // fewer tiles than SMs: one block per tile
        CHECK(tiles > sm || (k == 1 && grid == tiles), "sm %d most %d tiles %ld", sm, most, (long)tiles);
      }
  // window weights in registers: never more rounds at three blocks than at four, at most two
  for (int sm : {1, 78, 152})
    for (int64_t tiles = 1; tiles < 3000; tiles++, n++) {
      const bool r = registers_pay(tiles, sm, 3, 4);
      const int64_t r3 = (tiles + 3 * sm - 1) / (3 * sm), r4 = (tiles + 4 * sm - 1) / (4 * sm);
      CHECK(r == (r3 <= 2 && r3 == r4), "sm %d tiles %ld", sm, (long)tiles);
    }
  // the carve-out holds the blocks in the sizes the device offers (it takes the next one up)
  const int sizes[] = {0, 8, 16, 32, 64, 100, 132, 164, 196, 228}, smem_sm = 228 * 1024;
  for (int smem : {SMEM})
    for (int blocks = 1; blocks <= 4; blocks++, n++) {
      if ((int64_t)blocks * (smem + 1024) > smem_sm) continue;
      const int pct = carveout_percent(blocks, smem, smem_sm);
      int got = 0, least = 0;
      for (int s : sizes) {
        if (!got && s * 1024ll * 100 >= (int64_t)pct * smem_sm) got = s;
        if (!least && s * 1024 >= blocks * (smem + 1024)) least = s;
      }
      CHECK(got == least && pct <= 100, "%d blocks of %d bytes: %d %%, %d KB for %d", blocks, smem, pct, got, least);
    }
  CHECK(carveout_percent(4, 70000, smem_sm) == 100 && carveout_percent(1, 40000, 0) == 100, "limits");
  std::printf("%ld launches checked, %d failures\n", n, fails);
  return fails ? 1 : 0;
}
