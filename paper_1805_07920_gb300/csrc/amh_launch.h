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

// Groups of 32 pixels of a team's launch: 16 x 4 tiles of one colour, 8 x 4 tiles
// of the initialisation.
inline int64_t phase_groups(int W, int H) { return (int64_t)((W + 15) / 16) * ((H + 3) / 4); }
inline int64_t init_groups(int W, int H) { return (int64_t)((W + 7) / 8) * ((H + 3) / 4); }

// Warps per 32 pixels for a launch over `groups` of them: 16, 8 or 4 (a team), or
// 1 (one thread per pixel).  A team's fixed work (propagation, window, view
// selection, barriers) is repeated or waited for by its warps, so it pays while
// the GPU has room for it: 16 or 8 warps while all teams fit at once with 16 warps
// per SM; 4 while the groups are at most a share of those warps that grows with the
// number of sources, over which the fixed work spreads.  Four iterations, uint8 /
// filter form, one thread / 4 warps / (8 warps) in us, on 2432 warps:
//   1 source   220x165 (0.24) 267 / 182, filter 227 / 169; 240x180 (0.28) 277 / 297, filter 245 / 267
//   2          240x180 415 / 381, filter 361 / 338; 260x195 (0.34) 424 / 410, filter 369 / 373
//   3          280x210 (0.39) 570 / 547, filter 496 / 491; 320x240 (0.49) 583 / 613, filter 514 / 540
//   4          280x210 713 / 651, filter 610 / 590; 320x240 731 / 734, filter 627 / 651
//   6          320x240 1011 / 1016 (1058), 400x300 (0.77) 1604 / 1566 (1616), 440x330 (0.96) 1661 / 1869
//   16         160x120 1729 / 1083 (610), 400x300 3633 / 3123, 440x330 3742 / 3712
// The initialisation evaluates one plane per pixel, so a team of few sources has
// little to share: 1 source 200x150 (0.39) 8.2 / 10.3, 4 sources 240x180 (0.56)
// 16.5 / 18.5, 16 sources 400x300 (1.54) 145 / 117, 440x330 (1.88) 152 / 141.
inline int team_warps(int64_t groups, int n_src, int n_sm, bool init) {
  const int64_t warps = (int64_t)16 * n_sm;
  if (groups * 16 <= warps) return 16;
  if (groups * 8 <= warps) return 8;
  const int percent = init ? (n_src < 4 ? 25 : n_src < 8 ? 35 : 160)
                           : (n_src < 2 ? 25 : n_src < 3 ? 30 : n_src < 4 ? 40 : n_src < 6 ? 45 : 80);
  return groups * 100 <= warps * percent ? 4 : 1;
}

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
