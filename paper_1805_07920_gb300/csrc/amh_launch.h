// amh_launch.h -- how the update's launches are laid out on the device (host
// arithmetic only).
#pragma once
#include <algorithm>
#include <cstdint>

namespace amh {

struct DeviceShape {
  int n_sm = 0;                           // multiprocessors
  int smem_sm = 0;                        // bytes of shared memory of each
};

// Blocks an SM is given, at most `most`, by a launch over `tiles` tiles of about
// the same work.  A tile takes longer the more blocks share its SM, so a launch
// of one or two rounds takes the fewest blocks that need no more rounds than
// `most` would; in longer ones the rounds even out and more warps in flight count.
inline int blocks_per_sm(int64_t tiles, int n_sm, int most) {
  const int64_t rounds = (tiles + (int64_t)most * n_sm - 1) / ((int64_t)most * n_sm);
  if (rounds > 2) return most;
  return (int)std::max<int64_t>(1, (tiles + rounds * n_sm - 1) / std::max<int64_t>(1, rounds * n_sm));
}

// The update through the texture unit's filter has so little arithmetic per
// sample that the shared-memory reads of its window weights show where warps are
// few.  With the weights in registers an SM takes `three` blocks instead of
// `four`; that pays while it needs no more rounds for them, one or two.  Two
// sources, four iterations, weights in shared memory (carve-out for the blocks
// in use) / in registers / one kernel for all sizes before, in us: 320 x 240 394 /
// 381 / 407, 360 x 270 505 / 488 / 509, 440 x 330 (one round or two) 635 / 830 / 636,
// 520 x 390 960 / 939 / 1013, 640 x 480 (two or three) 1287 / 1363 / 1287.
inline bool registers_pay(int64_t tiles, int n_sm, int three, int four) {
  const int64_t r3 = (tiles + (int64_t)three * n_sm - 1) / ((int64_t)three * n_sm);
  const int64_t r4 = (tiles + (int64_t)four * n_sm - 1) / ((int64_t)four * n_sm);
  return r3 <= r4 && r3 <= 2;
}

// The shared-memory carve-out that holds `blocks` blocks of `smem` bytes (and the
// 1 KB each that the system keeps), as a percentage; the rest of the unified L1
// is texture and local-memory cache.  Rounded down: the device has a few sizes
// and takes the next one up, and rounded up four blocks of the batch (162.9 KB)
// ask for 164.2 of 164 KB and get the size after.
inline int carveout_percent(int blocks, int smem, int smem_sm) {
  if (smem_sm <= 0) return 100;
  return (int)std::min<int64_t>(100, (int64_t)100 * blocks * (smem + 1024) / smem_sm);
}

}  // namespace amh
