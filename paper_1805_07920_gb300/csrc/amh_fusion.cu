// amh_fusion.cu -- post-processing of the depth maps (Sec. 3.3, last two
// paragraphs): the 4x4 median filter, and the fusion of several views'
// depth / normal maps by Gipuma's consistency check (the paper's reference
// [9]) with the thresholds f_eps (disparity difference), f_ang (normal
// difference) and f_con (consistent views).  Readings (the paper leaves the
// details to [9]):
//   median: offsets -2..+1 in x and y, clamped borders, mean of the 8th and
//     9th smallest of the 16 values;
//   fusion: pixel p of view i with depth D > 0 back-projects to the world
//     point X with world normal n; view j agrees when X is in front of it,
//     projects to the pixel q = floor(u + 0.5), floor(v + 0.5) inside it with
//     D_j(q) > 0, f_j |C_i - C_j| |1 / z_j(X) - 1 / D_j(q)| <= f_eps and the
//     angle between n and view j's world normal at q is <= f_ang; with at
//     least f_con agreeing views the point is the mean of X and their
//     back-projected points, the normal the normalised sum of the normals.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "amh.h"
#include "amh_ctx.h"
#include "amh_device.cuh"

namespace amh {
namespace {

constexpr int kFuseMaxViews = 32;

__device__ __forceinline__ void cswap(float& a, float& b) {
  const float lo = fminf(a, b), hi = fmaxf(a, b);
  a = lo;
  b = hi;
}
// the median of one window by a full insertion sort (the loops unroll: no
// local memory); it also fixes what a NaN does to its window
__device__ __noinline__ float median16_sorted(const float* __restrict__ in, int x, int y, int W, int H) {
  float v[16];
#pragma unroll
  for (int k = 0; k < 16; k++) {
    const int xx = min(max(x + (k & 3) - 2, 0), W - 1), yy = min(max(y + (k >> 2) - 2, 0), H - 1);
    v[k] = __ldg(&in[(size_t)yy * W + xx]);
  }
#pragma unroll
  for (int a = 1; a < 16; a++) {
#pragma unroll
    for (int b = a; b > 0; b--) cswap(v[b - 1], v[b]);
  }
  // both halves are exact: one rounding, as the exact mean rounded to FP32
  return 0.5f * v[7] + 0.5f * v[8];
}

// 4x4 median.  A warp takes 32 columns and kMedRows output rows; lane l loads
// its column once (clamped) and gives the 29 outputs whose four columns the
// warp holds.  What neighbouring windows share is sorted once: vertical pairs
// (shared by two windows), columns of four (3 more comparators; shared by four
// lanes through shuffles), pairs of columns merged to sorted eights A and B
// (9 comparators); then the 8th and 9th smallest of the 16 are max_i min(A_i,
// B_7-i) and min_i max(A_i, B_7-i).  About 56 min / max per output instead of
// the 240 of a sort of its own, which bound it (3200 x 2112: 102 us before,
// 31 us now; reading and writing the map once takes 8).  A warp whose columns
// hold a NaN sorts each window in full: with a NaN the result depends on the
// order of the comparisons.
constexpr int kMedRows = 16, kMedCols = 29, kMedWarps = 4;
__global__ void __launch_bounds__(32 * kMedWarps) median4_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                                 int W, int H) {
  const int lane = threadIdx.x & 31;
  const int strips = (W + kMedCols - 1) / kMedCols, bands = (H + kMedRows - 1) / kMedRows;
  const int item = blockIdx.x * kMedWarps + (threadIdx.x >> 5);
  if (item >= strips * bands) return;
  // this lane's output column, first row (unsigned: past the last ones without overflow)
  const unsigned x = (unsigned)(item % strips) * kMedCols + lane, y0 = (unsigned)(item / strips) * kMedRows;
  const float* col = in + min(max(x, 2u) - 2u, (unsigned)W - 1u);
  float v[kMedRows + 3];
  bool nan = false;
#pragma unroll
  for (int r = 0; r < kMedRows + 3; r++) {
    v[r] = __ldg(col + (size_t)min(max(y0 + r, 2u) - 2u, (unsigned)H - 1u) * W);
    nan |= v[r] != v[r];
  }
  const bool mine = lane < kMedCols && x < (unsigned)W;
  const bool sort_all = __any_sync(0xffffffffu, nan);
  float lo0 = fminf(v[0], v[1]), hi0 = fmaxf(v[0], v[1]);      // rows r, r + 1
  float lo1 = fminf(v[1], v[2]), hi1 = fmaxf(v[1], v[2]);      // rows r + 1, r + 2
#pragma unroll
  for (int r = 0; r < kMedRows; r++) {
    const float lo2 = fminf(v[r + 2], v[r + 3]), hi2 = fmaxf(v[r + 2], v[r + 3]);
    // the column of rows r .. r + 3
    float c[8] = {lo0, hi0, lo2, hi2};
    cswap(c[0], c[2]);
    cswap(c[1], c[3]);
    cswap(c[1], c[2]);
    // columns l and l + 1: odd-even merge of c[0..3] and c[4..7]
#pragma unroll
    for (int k = 0; k < 4; k++) c[4 + k] = __shfl_down_sync(0xffffffffu, c[k], 1);
    cswap(c[0], c[4]);
    cswap(c[2], c[6]);
    cswap(c[2], c[4]);
    cswap(c[1], c[5]);
    cswap(c[3], c[7]);
    cswap(c[3], c[5]);
    cswap(c[1], c[2]);
    cswap(c[3], c[4]);
    cswap(c[5], c[6]);
    // and columns l + 2, l + 3
    float lo[8], hi[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const float d = __shfl_down_sync(0xffffffffu, c[7 - k], 2);
      lo[k] = fminf(c[k], d);
      hi[k] = fmaxf(c[k], d);
    }
    float m8 = lo[0], m9 = hi[0];
#pragma unroll
    for (int k = 1; k < 8; k++) {
      m8 = fmaxf(m8, lo[k]);
      m9 = fminf(m9, hi[k]);
    }
    if (mine && y0 + r < (unsigned)H)
      out[(size_t)(y0 + r) * W + x] = sort_all ? median16_sorted(in, (int)x, (int)(y0 + r), W, H) : 0.5f * m8 + 0.5f * m9;
    lo0 = lo1;
    hi0 = hi1;
    lo1 = lo2;
    hi1 = hi2;
  }
}

struct FuseView {
  float Kinv[9];
  float K[9];
  float R[9];
  float t[3];
  float C[3];
  int W, H;
  const float* depth;
  const float* normal;
  float* points;
  uint8_t* count;
};

struct FuseArgs {
  int n;
  float f_eps, cos_ang;
  int f_con;
  int tiles_x, bands;
  FuseView v[kFuseMaxViews];
};

// What the fusion decides (the pixel q, the two thresholds) it decides as the
// correctly rounded quotients and roots would.  A check is evaluated without
// branches from the hardware reciprocal and reciprocal root (about 1 ulp);
// where one of its decisions comes within its error of the boundary, or a
// value is outside the range the estimates hold for, the whole check is
// repeated with the correctly rounded operations (check_exactly).
constexpr float kTiny = 1e-30f, kHuge = 1e30f;

// A block takes 32 x 16 pixels of one view, a warp 32 pixels of a row;
// neighbouring blocks take the same tile of all views, so that what they gather
// from the other views is in L2.  What bounds it: instruction issue, about 200
// per check and warp, then the gathers.  Ten 1600 x 1056 views take 1007 us,
// twenty views around a ring, where most checks fail, 7.1 ms; with five correctly
// rounded divisions and three roots per check and their branches, the views'
// constants by indexed loads, a 64-bit division per pixel and 24-byte strided
// stores 1790 us and 8.5 ms.  On the way, with four rows per block instead of 16
// (the set-up of the constants shows: 1116 us, 10.3 ms): one view after another
// 1384 us where tile after tile took 1171; two or four pixels per thread 1566 /
// 1827 (registers), the next view's fetches issued ahead 1289, five blocks of 8
// warps (48 registers) 1322.  Points leave through shared memory as rows of 768
// bytes.
constexpr int kFuseWarps = 4, kFuseRows = 4 * kFuseWarps, kFuseBlocksPerSM = 8;   // 64 registers
// a view's constants in shared memory, read as float4
struct FuseShared {
  float4 R[3];          // rows of R, t in w
  float4 K[2];          // rows 0 and 1 of K; the width and height in w
  float4 Kinv[3];       // rows of K^-1; in row 0 the baseline to view i times the focal length in w
  const float *depth, *normal;
  int W;
  float lim;            // a pixel coordinate beyond it is outside
};
struct FuseExact {
  float uf, vf, D, m0, m1, m2;
  bool agree;
};
// The check in full: floor(num / z + 0.5) inside the view, a depth there, the
// disparity and the angle.
__device__ __noinline__ FuseExact check_exactly(const FuseShared& S, float nu, float nv, float z, float n0, float n1,
                                                float n2, float nn, float eps, float cos_ang) {
  FuseExact c = {};
  c.uf = floorf(nu / z + 0.5f);
  c.vf = floorf(nv / z + 0.5f);
  if (!(c.uf >= 0.f && c.uf < S.K[0].w && c.vf >= 0.f && c.vf < S.K[1].w)) return c;
  const size_t q = (size_t)(int)c.vf * S.W + (int)c.uf;
  c.D = S.depth[q];
  if (!(c.D > 0.f)) return c;
  if (!(S.Kinv[0].w * fabsf(1.f / z - 1.f / c.D) <= eps)) return c;
  c.m0 = S.normal[3 * q];
  c.m1 = S.normal[3 * q + 1];
  c.m2 = S.normal[3 * q + 2];
  const float4 r0 = S.R[0], r1 = S.R[1], r2 = S.R[2];
  const float a0 = r0.x * c.m0 + r1.x * c.m1 + r2.x * c.m2, a1 = r0.y * c.m0 + r1.y * c.m1 + r2.y * c.m2,
              a2 = r0.z * c.m0 + r1.z * c.m1 + r2.z * c.m2;
  const float dn = sqrtf(a0 * a0 + a1 * a1 + a2 * a2) * nn;
  c.agree = (n0 * a0 + n1 * a1 + n2 * a2) / fmaxf(dn, 1e-30f) >= cos_ang;
  return c;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__global__ void __launch_bounds__(32 * kFuseWarps, kFuseBlocksPerSM) fuse_kernel(const __grid_constant__ FuseArgs a) {
  __shared__ float stage[kFuseWarps][32 * 6];
  __shared__ FuseShared view[kFuseMaxViews];
  const int i = (int)(blockIdx.x % (unsigned)a.n), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = (int)(blockIdx.x / (unsigned)a.n);
  const FuseView& Vi = a.v[i];
  const int x0 = tile % a.tiles_x * 32, px = x0 + lane;
  if (x0 >= Vi.W || (int64_t)(tile / a.tiles_x) * kFuseRows >= Vi.H) return;   // views smaller than the largest
  if (threadIdx.x < a.n) {
    const FuseView& V = a.v[threadIdx.x];
    FuseShared& S = view[threadIdx.x];
    const float bx = Vi.C[0] - V.C[0], by = Vi.C[1] - V.C[1], bz = Vi.C[2] - V.C[2];
    for (int r = 0; r < 3; r++) S.R[r] = make_float4(V.R[3 * r], V.R[3 * r + 1], V.R[3 * r + 2], V.t[r]);
    S.K[0] = make_float4(V.K[0], V.K[1], V.K[2], (float)V.W);
    S.K[1] = make_float4(V.K[3], V.K[4], V.K[5], (float)V.H);
    for (int r = 0; r < 3; r++)
      S.Kinv[r] = make_float4(V.Kinv[3 * r], V.Kinv[3 * r + 1], V.Kinv[3 * r + 2],
                              r ? 0.f : V.K[0] * sqrtf(bx * bx + by * by + bz * bz));
    S.W = V.W;
    S.lim = (float)max(V.W, V.H) + 1.f;
    S.depth = V.depth;
    S.normal = V.normal;
  }
  __syncthreads();
  const int cols = min(32, Vi.W - x0);
  // rows of the tile (with fewer bands than the rows need, of every bands-th one)
  for (int64_t k = warp;; k += kFuseWarps) {
    const int64_t row = ((int64_t)(tile / a.tiles_x) + k / kFuseRows * a.bands) * kFuseRows + k % kFuseRows;
    if (row >= Vi.H) break;
    const size_t p = (size_t)row * Vi.W + px;
    const float x = (float)px, y = (float)row;
    const float D = lane < cols ? Vi.depth[p] : 0.f;
    float out[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int cnt = 0;
    if (D > 0.f) {
      // X = R^T (D K^-1 [x y 1] - t), n = R^T n_cam
      const float rx = Vi.Kinv[0] * x + Vi.Kinv[1] * y + Vi.Kinv[2];
      const float ry = Vi.Kinv[3] * x + Vi.Kinv[4] * y + Vi.Kinv[5];
      const float rz = Vi.Kinv[6] * x + Vi.Kinv[7] * y + Vi.Kinv[8];
      const float cx = D * rx - Vi.t[0], cy = D * ry - Vi.t[1], cz = D * rz - Vi.t[2];
      float X[3], n[3];
      const float* nc = Vi.normal + 3 * p;
#pragma unroll
      for (int r = 0; r < 3; r++) {
        X[r] = Vi.R[r] * cx + Vi.R[3 + r] * cy + Vi.R[6 + r] * cz;
        n[r] = Vi.R[r] * nc[0] + Vi.R[3 + r] * nc[1] + Vi.R[6 + r] * nc[2];
      }
      const float nn = sqrtf(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
      float sX[3] = {X[0], X[1], X[2]}, sN[3] = {n[0], n[1], n[2]};
      const float rnn = rcp_approx(nn);
      const bool nn_ok = nn > 1e-5f && nn < 1e5f;
#pragma unroll 1
      for (int j = 0; j < a.n; j++) {
        if (j == i) continue;
        const FuseShared& S = view[j];
        const float4 r0 = S.R[0], r1 = S.R[1], r2 = S.R[2];
        const float z = r2.x * X[0] + r2.y * X[1] + r2.z * X[2] + r2.w;
        if (!(z > 0.f)) continue;
        const float4 k0 = S.K[0], k1 = S.K[1];
        const float X0 = r0.x * X[0] + r0.y * X[1] + r0.z * X[2] + r0.w;
        const float X1 = r1.x * X[0] + r1.y * X[1] + r1.z * X[2] + r1.w;
        const float iz = rcp_approx(z);
        const float nu = k0.x * X0 + k0.y * X1 + k0.z * z, nv = k1.x * X0 + k1.y * X1 + k1.z * z;
        const float u = nu * iz, v = nv * iz;
        float uf = floorf(u + 0.5f), vf = floorf(v + 0.5f);
        // The quotients are within 2^-22 |u| of the rounded ones, whose sums with
        // 0.5 round by 2^-24 (|u| + 0.5): u - uf within 2^-21 (|u| + 1) of -0.5 or
        // 0.5 leaves the pixel open, unless both images of it lie outside (|u| or
        // |v| beyond lim, the larger size + 1).
        const float off = fmaxf(fabsf(u - uf), fabsf(v - vf));
        const float big = fmaxf(fabsf(u), fabsf(v)), m = fmaf(-4.76837158203125e-7f, big, 0.5f - 4.76837158203125e-7f);
        const bool z_ok = z > kTiny && z < kHuge;
        const bool in = z_ok && uf >= 0.f && uf < k0.w && vf >= 0.f && vf < k1.w;
        bool unsure = (!(off <= m) && big <= S.lim) || !z_ok;
        if (!in && !unsure) continue;
        const int64_t q = in ? (int64_t)(int)vf * S.W + (int)uf : 0;
        const float* ncj = S.normal + 3 * q;
        float D2 = __ldg(S.depth + q);
        const float m0 = __ldg(ncj), m1 = __ldg(ncj + 1), m2 = __ldg(ncj + 2);
        const float4 i0 = S.Kinv[0];
        const bool has = in && D2 > 0.f;
        const float rd = rcp_approx(D2), dd = fmaf(i0.w, fabsf(iz - rd), -a.f_eps);
        const float md = fmaf(2.384185791015625e-7f * i0.w, iz + rd, 1e-6f * a.f_eps);      // 2^-22
        float nj0 = r0.x * m0 + r1.x * m1 + r2.x * m2, nj1 = r0.y * m0 + r1.y * m1 + r2.y * m2,
              nj2 = r0.z * m0 + r1.z * m1 + r2.z * m2;
        const float q2 = nj0 * nj0 + nj1 * nj1 + nj2 * nj2;
        const float da = fmaf(n[0] * nj0 + n[1] * nj1 + n[2] * nj2, rsqrt_approx(q2) * rnn, -a.cos_ang);
        bool agree = has && dd <= 0.f && da >= 0.f;
        // sure: the disparity further from the threshold than its error and, if it
        // passes, the cosine too (|cosine| <= 1 + 1e-6: 4e-6 covers its error);
        // comparisons with NaN are not
        const bool sure = D2 > kTiny && fabsf(dd) > md && (dd > 0.f || (nn_ok && q2 > kTiny && fabsf(da) > 4e-6f));
        unsure |= has && !sure;
        if (unsure) {
          const FuseExact e = check_exactly(S, nu, nv, z, n[0], n[1], n[2], nn, a.f_eps, a.cos_ang);
          agree = e.agree;
          uf = e.uf;
          vf = e.vf;
          D2 = e.D;
          nj0 = r0.x * e.m0 + r1.x * e.m1 + r2.x * e.m2;
          nj1 = r0.y * e.m0 + r1.y * e.m1 + r2.y * e.m2;
          nj2 = r0.z * e.m0 + r1.z * e.m1 + r2.z * e.m2;
        }
        if (!agree) continue;
        // the agreeing view's own point at q
        const float4 i1 = S.Kinv[1], i2 = S.Kinv[2];
        const float qx = i0.x * uf + i0.y * vf + i0.z;
        const float qy = i1.x * uf + i1.y * vf + i1.z;
        const float qz = i2.x * uf + i2.y * vf + i2.z;
        const float ex = D2 * qx - r0.w, ey = D2 * qy - r1.w, ez = D2 * qz - r2.w;
        sX[0] += r0.x * ex + r1.x * ey + r2.x * ez;
        sX[1] += r0.y * ex + r1.y * ey + r2.y * ez;
        sX[2] += r0.z * ex + r1.z * ey + r2.z * ez;
        sN[0] += nj0;
        sN[1] += nj1;
        sN[2] += nj2;
        cnt++;
      }
      if (cnt >= a.f_con) {
        const float inv = 1.f / (float)(1 + cnt);
        const float ln = sqrtf(sN[0] * sN[0] + sN[1] * sN[1] + sN[2] * sN[2]);
#pragma unroll
        for (int r = 0; r < 3; r++) {
          out[r] = sX[r] * inv;
          out[3 + r] = sN[r] / fmaxf(ln, 1e-30f);
        }
      }
    }
    __syncwarp();
    float* st = stage[warp];
#pragma unroll
    for (int r = 0; r < 6; r++) st[6 * lane + r] = out[r];
    __syncwarp();
    float* o = Vi.points + 6 * ((size_t)row * Vi.W + x0);
    for (int e = lane; e < 6 * cols; e += 32) __stcs(o + e, st[e]);
    if (lane < cols) Vi.count[p] = (uint8_t)cnt;
  }
}

bool inv3f(const double* A, double* I) {
  const double c00 = A[4] * A[8] - A[5] * A[7], c01 = A[5] * A[6] - A[3] * A[8],
               c02 = A[3] * A[7] - A[4] * A[6];
  const double det = A[0] * c00 + A[1] * c01 + A[2] * c02;
  if (!(std::fabs(det) > 0) || !std::isfinite(det)) return false;
  const double id = 1.0 / det;
  I[0] = c00 * id; I[1] = (A[2] * A[7] - A[1] * A[8]) * id; I[2] = (A[1] * A[5] - A[2] * A[4]) * id;
  I[3] = c01 * id; I[4] = (A[0] * A[8] - A[2] * A[6]) * id; I[5] = (A[2] * A[3] - A[0] * A[5]) * id;
  I[6] = c02 * id; I[7] = (A[1] * A[6] - A[0] * A[7]) * id; I[8] = (A[0] * A[4] - A[1] * A[3]) * id;
  return true;
}

int launch_status(const char* what) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? AMH_OK : fail_no_context(AMH_ECUDA, "%s launch: %s", what, cudaGetErrorString(e));
}

}  // namespace
}  // namespace amh

using namespace amh;

extern "C" {

AMH_API int amh_median4(const float* depth_in, float* depth_out, int32_t width, int32_t height, void* stream) {
  if (!depth_in || !depth_out || width < 1 || height < 1 || depth_in == depth_out)
    return fail_no_context(AMH_EINVAL, "amh_median4: NULL or aliased buffers, or an empty image");
  const int64_t items = (int64_t)((width + (int64_t)kMedCols - 1) / kMedCols) * ((height + (int64_t)kMedRows - 1) / kMedRows);
  const int64_t blocks = (items + kMedWarps - 1) / kMedWarps;
  if (blocks * kMedWarps > INT32_MAX) return fail_no_context(AMH_EINVAL, "amh_median4: image too large");
  median4_kernel<<<(unsigned)blocks, 32 * kMedWarps, 0, (cudaStream_t)stream>>>(depth_in, depth_out, width, height);
  return launch_status("amh_median4");
}

AMH_API int amh_fuse(int32_t n_views, const amh_camera* cams, const float* const* depth, const float* const* normal3,
                     float f_eps, float f_ang_deg, int32_t f_con, float* const* points6, uint8_t* const* count,
                     void* stream) {
  if (n_views < 2 || n_views > kFuseMaxViews || !cams || !depth || !normal3 || !points6 || !count)
    return fail_no_context(AMH_EINVAL, "amh_fuse: 2..%d views with non-NULL arrays required", kFuseMaxViews);
  if (!(f_eps >= 0.f) || !(f_ang_deg >= 0.f && f_ang_deg <= 180.f) || f_con < 1)
    return fail_no_context(AMH_EINVAL, "amh_fuse: thresholds out of range");
  FuseArgs a;
  std::memset(&a, 0, sizeof a);
  a.n = n_views;
  a.f_eps = f_eps;
  a.cos_ang = (float)std::cos((double)f_ang_deg * 3.14159265358979323846 / 180.0);
  a.f_con = f_con;
  int most_w = 0, most_h = 0;
  for (int v = 0; v < n_views; v++) {
    const amh_camera& c = cams[v];
    if (!depth[v] || !normal3[v] || !points6[v] || !count[v] || c.width < 1 || c.height < 1)
      return fail_no_context(AMH_EINVAL, "amh_fuse: view %d has a NULL array or an empty image", v);
    double Ki[9];
    if (!inv3f(c.K, Ki)) return fail_no_context(AMH_EINVAL, "amh_fuse: K of view %d is singular", v);
    FuseView& F = a.v[v];
    for (int k = 0; k < 9; k++) {
      F.Kinv[k] = (float)Ki[k];
      F.K[k] = (float)c.K[k];
      F.R[k] = (float)c.R[k];
    }
    for (int r = 0; r < 3; r++) {
      F.t[r] = (float)c.t[r];
      F.C[r] = (float)-(c.R[r] * c.t[0] + c.R[3 + r] * c.t[1] + c.R[6 + r] * c.t[2]);   // -R^T t
    }
    F.W = c.width;
    F.H = c.height;
    F.depth = depth[v];
    F.normal = normal3[v];
    F.points = points6[v];
    F.count = count[v];
    most_w = std::max(most_w, c.width);
    most_h = std::max(most_h, c.height);
  }
  // at most 2^31 - 1 blocks; with fewer bands than the rows need, each takes more rows
  a.tiles_x = (int)((most_w + (int64_t)31) / 32);
  a.bands = (int)std::max<int64_t>(1, std::min((most_h + (int64_t)kFuseRows - 1) / kFuseRows,
                                               INT32_MAX / ((int64_t)a.tiles_x * n_views)));
  const unsigned grid = (unsigned)((int64_t)a.tiles_x * a.bands * n_views);
  fuse_kernel<<<grid, 32 * kFuseWarps, 0, (cudaStream_t)stream>>>(a);
  return launch_status("amh_fuse");
}

}  // extern "C"
