// amh_team.cuh -- the checkerboard update of 32 pixels by a team of T warps,
// for images with too few pixels to fill the GPU with one thread per pixel
// (amh_update.cuh: a pixel's ~20 .. 300 evaluations run one after another
// there).  The lanes of every warp are the team's 32 pixels and the work of a
// pixel is split over the warps: warp 0 loads the reference window while the
// others take the propagation regions; the (view, hypothesis) pairs of the
// matrix, the views of the joint selection and of the own plane, and the
// refinement candidates (or, when there are at most two, their views) are
// dealt to the warps, so every texture fetch still has one view per warp.
// What one warp computes and another reads goes through shared memory.  Each
// value is computed by the same expressions in the same order as by one
// thread, so the results are the same bits.
#pragma once
#include "amh_update.cuh"

namespace amh {
namespace upd {

// one team per block
template <int T>
struct TeamShared {
  float4 win[kWinPairs * kTeamPixels];    // bilateral weights (TeamWin)
  float4 c[kRegions * kTeamPixels];       // propagated planes, then candidate planes, as (K^-T n / d, 1 / D)
  float stat[3 * kTeamPixels];            // TeamWin's inv_sw, sum_wr, var_r
  float hD[kRegions * kTeamPixels];       // depth of propagated row g at the pixel
  int pick[kRegions * kTeamPixels];       // its packed offset, -1 none
  float row[kRegions * kTeamPixels];      // unified costs of the rows
  float cand[kRegions * kTeamPixels];     // unified costs of the candidates (infinite: lost)
  uint32_t bits[3][T * kTeamPixels];      // per warp: valid rows, good views, kept (or lowest) views
  int vtop[kTeamPixels];                  // the most important good view
};
// dynamic shared memory of a team with N views, in floats: the matrix (entry
// 8 j + g), psi_mod and one cost per view of 32 pixels.  With the static part a team
// of four warps takes 19456 + 1280 N bytes: four fit an SM up to 29 views, then
// three.
__host__ __device__ constexpr int team_floats(int N) { return kTeamPixels * 10 * N; }

// The launch before this one on the stream has finished and its state is
// visible (the window depends on the image only, so it is loaded before); the
// next launch may be set up from here on.
__device__ __forceinline__ void phase_before_done() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One colour phase's update of the team's 32 pixels; lane l's pixel is (x, y),
// w the warp's index in the team (warp-uniform).  The whole block calls it.
template <bool kHalf, bool kTex, int T, class A>
__device__ __forceinline__ void update_team(const A& a, TeamShared<T>& sh, float* dyn, int w, int x, int y,
                                            int* npairs) {
  const int lane = threadIdx.x & 31;
  const int N = a.N;
  const bool live = x < a.W && y < a.H;
  x = min(x, a.W - 1);                    // lanes outside the image read a pixel inside
  y = min(y, a.H - 1);
  const int pi = (int)checked_index(a, state_index(x, y, a.W), state_size(a.W, a.H), kBadPixel);
  const float3 ray = ref_ray(a.Kinv, (float)x, (float)y);
  auto at = [&](int i) { return i * kTeamPixels + lane; };
  auto all_bits = [&](int k) {
    uint32_t b = 0;
#pragma unroll
    for (int t = 0; t < T; t++) b |= sh.bits[k][at(t)];
    return b;
  };
  auto pick_index = [&](int off) {
    return checked_index(a, state_index(x + (off & 255) - 32, y + (off >> 8) - 32, a.W), state_size(a.W, a.H),
                         kBadNeighbour);
  };
  float* M = dyn;
  float* psim = dyn + 8 * N * kTeamPixels;
  float* per_view = psim + N * kTeamPixels;

  // --- warp 0: the reference window; the others: Sec. 3.1, asymmetric
  // checkerboard propagation (update_pixel, with the regions' geometry computed)
  TeamWin rw;
  rw.q = sh.win + lane;
  uint32_t valid = 0;
  if (w == 0) {
    load_ref_window<kHalf>(a, x, y, rw);
    sh.stat[at(0)] = rw.inv_sw;
    sh.stat[at(1)] = rw.sum_wr;
    sh.stat[at(2)] = rw.var_r;
    phase_before_done();
  } else {
    phase_before_done();
    const int srow = 2 * ((a.W + 1) >> 1), xodd = x & 1;
    const int qbase = y * srow + (((x + y) & 1) ? 0 : (srow >> 1)) + (x >> 1);
    for (int g = w - 1; g < kRegions; g += T - 1) {
      int best = -1;
      float bc = 0.f;
      if (live) {
        const int dir = g & 3;
#pragma unroll
        for (int i = 0; i < 11; i++) {
          if (g < 4 && i >= 7) continue;
          const int dep = g < 4 ? (i + 1) / 2 + 1 : 3 + 2 * i;
          const int lat = g < 4 && i > 0 ? ((i & 1) ? -1 : 1) * ((i + 1) / 2) : 0;
          const int dx = dir == 2 ? -dep : dir == 3 ? dep : lat, dy = dir == 0 ? -dep : dir == 1 ? dep : lat;
          const int qx = x + dx, qy = y + dy;
          if (qx < 0 || qy < 0 || qx >= a.W || qy >= a.H) continue;
          const int q = (int)checked_index(a, (size_t)(qbase + dy * srow + ((xodd + dx) >> 1)), state_size(a.W, a.H),
                                           kBadNeighbour);
          const float cq = a.cost[q];         // not a read-only load: the launch before may still write when this one starts
          if (best < 0 || cq < bc) { best = (dx + 32) | (dy + 32) << 8; bc = cq; }
        }
      }
      sh.pick[at(g)] = best;
      if (best < 0) continue;
      float Dx;
      float4 c;
      if (!propagate(a, a.plane[pick_index(best)], x + (best & 255) - 32, y + (best >> 8) - 32, ray, &Dx, &c)) continue;
      sh.c[at(g)] = c;
      sh.hD[at(g)] = Dx;
      valid |= 1u << g;
    }
  }
  sh.bits[0][at(w)] = valid;
  const uint32_t S_prev = a.sel[pi];
  const int v_prev = a.vbest[pi];         // 255: none
  float4 best = a.plane[pi];
  __syncthreads();
  rw.inv_sw = sh.stat[at(0)];
  rw.sum_wr = sh.stat[at(1)];
  rw.var_r = sh.stat[at(2)];
  valid = all_bits(0);

  // --- Eq. (1): the 8 x N cost matrix, (view, row) pairs in equal runs
  {
    const int per = (8 * N + T - 1) / T, t1 = min(8 * N, (w + 1) * per);
#pragma unroll 1
    for (int t = w * per; t < t1; t++) {
      const int g = t & 7;
      const bool ok = valid >> g & 1u;
      const float4 c = ok ? sh.c[at(g)] : make_float4(0.f, 0.f, 0.f, 0.f);
      M[at(t)] = ncc_cost<kHalf, kTex>(a.v[t >> 3], c, ok, ray, rw, npairs);
    }
  }
  __syncthreads();

  // --- Eqs. (2)-(6), the views split over the warps (joint_view_selection)
  const int nvalid = __popc(valid);
  const int k = a.k < N ? a.k : N;
  uint32_t S = 0;
  for (int j = w; j < N; j += T) {
    ViewScore score;
#pragma unroll
    for (int i = 0; i < kRegions; i++)
      if (valid >> i & 1u) score.add(a, M[at(8 * j + i)]);
    float pm;
    if (score.weigh(a, nvalid, j == v_prev, &pm)) S |= 1u << j;
    psim[at(j)] = pm;
  }
  sh.bits[1][at(w)] = S;
  __syncthreads();
  S = all_bits(1);
  uint32_t kept = 0;
  for (int j = w; j < N; j += T) {
    if (!(S >> j & 1u)) continue;
    const float pj = psim[at(j)];
    int rank = 0;
    for (int q = 0; q < N; q++) {
      const float pq = psim[at(q)];
      rank += (S >> q & 1u) && (pq > pj || (pq == pj && q < j));
    }
    if (rank < k) kept |= 1u << j;                 // at most k views keep weight
    if (rank == 0) sh.vtop[lane] = j;
  }
  sh.bits[2][at(w)] = kept;
  __syncthreads();
  kept = all_bits(2);
  const int v = S ? sh.vtop[lane] : -1;
  float sw = 0.f;
  uint32_t wm = 0;
  for (int j = 0; j < N; j++) {
    const float wj = (S >> j & 1u) ? ((kept >> j & 1u) ? psim[at(j)] : 0.f) : (S_prev >> j & 1u) ? 0.2f : 0.f;
    sw += wj;
    wm |= (wj > 0.f ? 1u : 0u) << j;
  }
  const bool none = wm == 0;              // no weight at all: the k views of smallest mean cost get 1
  if (__any_sync(0xffffffffu, none)) {    // the same answer in every warp
    for (int j = w; j < N; j += T) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < kRegions; i++)
        if (valid >> i & 1u) s += M[at(8 * j + i)];
      per_view[at(j)] = nvalid ? s / (float)nvalid : 0.f;
    }
    __syncthreads();
    uint32_t low = 0;
    for (int j = w; j < N; j += T) {
      const float cj = per_view[at(j)];
      int rank = 0;
      for (int q = 0; q < N; q++) {
        const float cq = per_view[at(q)];
        rank += cq < cj || (cq == cj && q < j);
      }
      if (rank < k) low |= 1u << j;
    }
    sh.bits[1][at(w)] = low;
    __syncthreads();
    low = all_bits(1);
    if (none) {
      wm = low;
      sw = 0.f;
      for (int j = 0; j < N; j++) sw += (low >> j & 1u) ? 1.f : 0.f;
    }
  }
  const float inv_sw = 1.f / sw;
  // weight of a view of the mask wm
  auto weight = [&](int j) { return none ? 1.f : (S >> j & 1u) ? psim[at(j)] : 0.2f; };

  // --- Eq. (7): unified costs of the own plane (its views split over the warps)
  // and of the rows; the own plane wins ties
  float4 c;
  bool ok = plane_c(a.Kinv, best, ray, &c);
  const uint32_t views = __reduce_or_sync(0xffffffffu, live ? wm : 0u);   // the team's views of some weight
  {
    int i = 0;
#pragma unroll 1
    for (uint32_t u = views; u; u &= u - 1, i++) {
      if (i % T != w) continue;
      const int j = __ffs(u) - 1;
      if (live && (wm >> j & 1u)) per_view[at(j)] = ncc_cost<kHalf, kTex>(a.v[j], c, ok, ray, rw, npairs);
    }
  }
  for (int g = T - 1 - w; g < kRegions; g += T) {
    float r = 0.f;
    for (int j = 0; j < N; j++)
      if (wm >> j & 1u) r = fmaf(weight(j), M[at(8 * j + g)], r);
    sh.row[at(g)] = r * inv_sw;
  }
  __syncthreads();
  float bm = 0.f;
  for (int j = 0; j < N; j++)
    if (wm >> j & 1u) bm = fmaf(weight(j), per_view[at(j)], bm);
  bm *= inv_sw;
  int choice = 8;
  for (int g = 0; g < kRegions; g++) {
    if (!(valid >> g & 1u)) continue;
    const float r = sh.row[at(g)];
    if (r < bm) { bm = r; choice = g; }
  }
  if (choice < 8) {
    const float4 pq = a.plane[pick_index(sh.pick[at(choice)])];
    best = make_float4(pq.x, pq.y, pq.z, sh.hD[at(choice)]);
  }

  // --- Sec. 3.3: refinement with the same weights (update_pixel); the
  // candidates' planes take the rows' slots
  const int nc = a.t < 3 ? 1 : kMaxRefine;
  float4 prop;
  const bool has_prop = learned_plane(a, x, y, ray, &prop);
  const int ncand = nc + (a.prop ? 1 : 0);
  if (ncand <= 2) {
    // the (view, candidate) pairs are dealt to the warps; the costs take the
    // matrix's place, entry 2 j + ci
    int i = 0;
#pragma unroll 1
    for (int ci = 0; ci < ncand; ci++) {
      const bool cand_ok = plane_c<true>(a.Kinv, ci < nc ? refine_candidate(a, x, y, best, ray, ci) : prop, ray, &c);
#pragma unroll 1
      for (uint32_t u = views; u; u &= u - 1, i++) {
        if (i % T != w) continue;
        const int j = __ffs(u) - 1;
        if (live && (wm >> j & 1u) && (ci < nc || has_prop))
          M[at(2 * j + ci)] = ncc_cost<kHalf, kTex>(a.v[j], c, cand_ok, ray, rw, npairs);
      }
    }
  } else {
    uint32_t okm = 0u, cand_live = 0u;
#pragma unroll 1
    for (int ci = w; ci < ncand; ci += T) {
      float4 cc;
      if (plane_c<true>(a.Kinv, ci < nc ? refine_candidate(a, x, y, best, ray, ci) : prop, ray, &cc)) okm |= 1u << ci;
      sh.c[at(ci)] = cc;
      sh.cand[at(ci)] = 0.f;
      if (live && (ci < nc || has_prop)) cand_live |= 1u << ci;
    }
#pragma unroll 1
    for (uint32_t u = views; u; u &= u - 1) {
      const int j = __ffs(u) - 1;
      uint32_t todo = (wm >> j & 1u) ? cand_live : 0u;
      while (todo) {
        const int ci = __ffs(todo) - 1;
        todo &= todo - 1u;
        const float m = fmaf(weight(j), ncc_cost<kHalf, kTex>(a.v[j], sh.c[at(ci)], (okm >> ci) & 1u, ray, rw, npairs),
                             sh.cand[at(ci)]);
        sh.cand[at(ci)] = m;
        if (!(m * inv_sw < bm)) cand_live &= ~(1u << ci);
      }
    }
    for (int ci = w; ci < ncand; ci += T)
      sh.cand[at(ci)] = (cand_live >> ci & 1u) ? sh.cand[at(ci)] * inv_sw : __int_as_float(0x7f800000);
  }
  __syncthreads();
  if (w != 0 || !live) return;
  int bc = -1;
  float bcm = 0.f;
  for (int ci = 0; ci < ncand; ci++) {
    float m;
    if (ncand <= 2) {
      if (ci >= nc && !has_prop) continue;
      m = 0.f;
      for (int j = 0; j < N; j++)
        if (wm >> j & 1u) m = fmaf(weight(j), M[at(2 * j + ci)], m);
      m *= inv_sw;
    } else {
      m = sh.cand[at(ci)];
    }
    if (bc < 0 || m < bcm) { bc = ci; bcm = m; }
  }
  if (bc >= 0 && bcm < bm) {
    bm = bcm;
    best = bc < nc ? refine_candidate(a, x, y, best, ray, bc) : prop;
    choice = bc < nc ? 9 + bc : 15;
  }
  __stcs(&a.plane[pi], best);
  __stcs(&a.cost[pi], bm);
  __stcs(&a.sel[pi], S);
  __stcs(&a.vbest[pi], v < 0 ? (uint8_t)255 : (uint8_t)v);
  __stcs(&a.wmask[pi], wm);
  __stcs(&a.choice[pi], (uint8_t)choice);
}

// Random initialisation of the team's 32 pixels (init_pixel): the views split
// over the warps.
template <bool kHalf, bool kTex, int T, class A>
__device__ __forceinline__ void init_team(const A& a, TeamShared<T>& sh, float* per_view, int w, int x, int y,
                                          int* npairs) {
  const int lane = threadIdx.x & 31;
  const int N = a.N;
  phase_before_done();                    // launched without overlap: only lets the first phase's blocks in
  const bool live = x < a.W && y < a.H;
  x = min(x, a.W - 1);
  y = min(y, a.H - 1);
  const float3 ray = ref_ray(a.Kinv, (float)x, (float)y);
  auto at = [&](int i) { return i * kTeamPixels + lane; };
  const float4 pl = random_plane(a, x, y, ray);
  float4 c;
  const bool ok = plane_c(a.Kinv, pl, ray, &c) && live;
  TeamWin rw;
  rw.q = sh.win + lane;
  if (w == 0) {
    load_ref_window<kHalf>(a, x, y, rw);
    sh.stat[at(0)] = rw.inv_sw;
    sh.stat[at(1)] = rw.sum_wr;
    sh.stat[at(2)] = rw.var_r;
  }
  __syncthreads();
  rw.inv_sw = sh.stat[at(0)];
  rw.sum_wr = sh.stat[at(1)];
  rw.var_r = sh.stat[at(2)];
#pragma unroll 1
  for (int j = w; j < N; j += T) per_view[at(j)] = ncc_cost<kHalf, kTex>(a.v[j], c, ok, ray, rw, npairs);
  __syncthreads();
  if (w == 0 && live) init_state(a, x, y, pl, kbest_mean<kTeamPixels>(per_view + lane, N, min(a.k, N)));
}

}  // namespace upd
}  // namespace amh
