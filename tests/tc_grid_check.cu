// Host-side check of the convolutions' launch grids
// (paper_1805_07920_gb300/csrc/amh_conv_tc.cuh): for every channel pair, device
// size and number of tiles, and for as many resident CTAs as the plan allows
// (the register file may allow fewer), a gradient's CTAs have a row of partial
// sums each per quarter, no CTA is without a tile, and otherwise the resident
// CTAs are used.
#include <cstdio>

#include "../paper_1805_07920_gb300/csrc/amh_conv_tc.cuh"

using namespace amh::tc;

int main() {
  const int cins[] = {16, 32, 64, 96, 128}, sms[] = {1, 78, 132, 148, 152, 160, 304};
  int n = 0, fails = 0;
  for (int cin : cins)
    for (int cout = 16; cout <= kMaxCout; cout += 16) {
      const ConvPlan p = conv_plan(cin, cout);
      const int nblk = cout / p.Nb;
      for (int sm : sms)
        for (int cps = 1; cps <= p.ctas_per_sm; cps++)
          for (int tiles = 1; tiles < 40000; tiles = 2 * tiles + 1)
            for (int grad = 0; grad < 2; grad++, n++) {
              const int g = conv_grid(tiles, sm, cps, nblk, grad != 0), resident = sm * cps / nblk;
              const bool ok = g >= 1 && g <= tiles && (g <= resident || g == 1) && (!grad || 4 * g <= kBiasRows) &&
                              (g == tiles || g >= resident || (grad && 4 * g == kBiasRows));
              if (!ok) std::printf("FAIL cin %d cout %d sm %d ctas %d tiles %d gradient %d: %d\n", cin, cout, sm, cps, tiles, grad, g), fails++;
            }
    }
  std::printf("%d grids checked, %d failures\n", n, fails);
  return fails ? 1 : 0;
}
