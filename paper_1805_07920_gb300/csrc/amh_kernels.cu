// amh_kernels.cu -- kernels of the single-reference context: random
// initialisation and one colour phase over a 16 x 16 tile per block (the
// update itself is in amh_update.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "amh_device.cuh"
#include "amh_kernels.h"
#include "amh_team.cuh"
#include "amh_update.cuh"

namespace amh {
namespace {
using namespace upd;

constexpr int kTile = 16;
constexpr int kThreads = 128;
// 128 registers per thread; the window weights are 36 KB of shared memory per
// block, so 4 blocks leave 92 KB of L1.  Five blocks (96 registers): the
// learned form at 1600 x 1056 32.2 ms against 31.9, 640 x 480 3.99 against 3.65.
// The staged sweep's boxes and the window weights in registers (168) allow 3.
constexpr int kPhaseBlocksPerSM = 4, kThreeBlocksPerSM = 3;
constexpr int phase_blocks_per_sm(int mode) { return mode & (kStage | kRegs) ? kThreeBlocksPerSM : kPhaseBlocksPerSM; }

// npairs: evaluations of this thread, plus 2^16 for each one sampled from a
// shared-memory box (fewer than 2^11 per thread and launch); the two totals
// go to the first and the second kPairCounters counters
__device__ __forceinline__ void count_pairs(const PhaseArgs& a, int npairs) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)npairs & 0xFFFFu);
  const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)npairs >> 16);
  const int k = (blockIdx.x * 4 + (threadIdx.x >> 5) + blockIdx.y * 7) % kPairCounters;
  if ((threadIdx.x & 31) == 0 && lo) atomicAdd(&a.pairs[k], (unsigned long long)lo);
  if ((threadIdx.x & 31) == 0 && hi) atomicAdd(&a.pairs[kPairCounters + k], (unsigned long long)hi);
}

template <bool kHalf, int kMode>
__global__ void __launch_bounds__(kThreads, phase_blocks_per_sm(kMode)) phase_kernel(const __grid_constant__ PhaseArgs a) {
  PixelArrays sm;
  const int tid = threadIdx.x;
  int npairs = 0;
  if constexpr ((kMode & kRegs) != 0) {
    const int y = blockIdx.y * kTile + (tid >> 3);
    const int x = blockIdx.x * kTile + 2 * (tid & 7) + ((y + a.color) & 1);
    update_pixel<kHalf, kMode>(a, sm, x, y, &npairs, nullptr, nullptr, x < a.W && y < a.H);
  } else if constexpr ((kMode & kStage) != 0) {
    __shared__ WinShared ws;
    // Warp w updates rows 4w .. 4w + 3 of the tile (8 pixels of the colour
    // per row); each quarter-warp takes 4 pixels of two neighbouring rows, so
    // the 8 lanes of a 16-byte shared load sample 8 distinct columns modulo
    // 8 of the box where the view maps the tile at unit scale.
    const int lane = tid & 31, q = lane >> 3;
    const int y = blockIdx.y * kTile + 4 * (tid >> 5) + 2 * (q >> 1) + ((lane >> 2) & 1);
    const int x = blockIdx.x * kTile + 2 * (4 * (q & 1) + (lane & 3)) + ((y + a.color) & 1);
    // the whole block takes part in the staged sweep, pixels outside the image too
    extern __shared__ __align__(16) unsigned char stage_dyn[];
    update_pixel<kHalf, kMode>(a, sm, x, y, &npairs, ws.q + tid, ws.slots[tid >> 5], x < a.W && y < a.H,
                               reinterpret_cast<StageShared*>(stage_dyn));
  } else {
    __shared__ WinShared ws;
    const int y = blockIdx.y * kTile + (tid >> 3);
    const int x = blockIdx.x * kTile + 2 * (tid & 7) + ((y + a.color) & 1);
    update_pixel<kHalf, kMode>(a, sm, x, y, &npairs, ws.q + tid, ws.slots[tid >> 5], x < a.W && y < a.H);
  }
  count_pairs(a, npairs);
}

// Random initialisation: one thread per pixel over the whole image.
template <bool kHalf, bool kTex>
__global__ void __launch_bounds__(kThreads, kPhaseBlocksPerSM) init_kernel(const __grid_constant__ PhaseArgs a) {
  PixelArrays sm;
  __shared__ WinShared ws;
  const int x = blockIdx.x * kTile + (threadIdx.x & 15), y = blockIdx.y * 8 + (threadIdx.x >> 4);
  int npairs = 0;
  if (x < a.W && y < a.H) init_pixel<kHalf, kTex>(a, sm, x, y, &npairs, ws.q + threadIdx.x);
  count_pairs(a, npairs);
}

// Small images: a team of T warps per 16 x 4 tile (32 pixels of the colour), or
// per 8 x 4 tile of the initialisation.
template <int T>
constexpr int kTeamBlocksPerSM = 16 / T;      // 16 warps, 128 registers per thread, as phase_kernel
template <bool kHalf, bool kTex, int T>
__global__ void __launch_bounds__(32 * T, kTeamBlocksPerSM<T>) phase_team_kernel(const __grid_constant__ PhaseArgs a) {
  extern __shared__ float dyn[];
  __shared__ TeamShared<T> sh;
  const int w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  int npairs = 0;
  const int y = blockIdx.y * 4 + (lane >> 3);
  update_team<kHalf, kTex, T>(a, sh, dyn, w, blockIdx.x * 16 + 2 * (lane & 7) + ((y + a.color) & 1), y, &npairs);
  count_pairs(a, npairs);
}
template <bool kHalf, bool kTex, int T>
__global__ void __launch_bounds__(32 * T, kTeamBlocksPerSM<T>) init_team_kernel(const __grid_constant__ PhaseArgs a) {
  extern __shared__ float dyn[];
  __shared__ TeamShared<T> sh;
  const int w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  int npairs = 0;
  init_team<kHalf, kTex, T>(a, sh, dyn, w, blockIdx.x * 8 + (lane & 7), blockIdx.y * 4 + (lane >> 3), &npairs);
  count_pairs(a, npairs);
}

}  // namespace

// A launch of one thread per pixel, with the carve-out for the blocks an SM gets.
// Four iterations in us, with the carve-out for all four blocks and now: two
// sources 320 x 240 447 -> 430, three 520 x 390 1494 -> 1430; the same at full size.
template <typename K>
int launch_blocks(K kernel, dim3 grid, int most, int smem, int dynamic, const PhaseArgs& a, const DeviceShape& dev,
                  cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = dynamic;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  at.val.sharedMemCarveout =
      carveout_percent(blocks_per_sm((int64_t)grid.x * grid.y, dev.n_sm, most), smem + dynamic, dev.smem_sm);
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, a);
  return (int)cudaGetLastError();
}

// Static and dynamic shared memory together go past the default limit of 48 KB:
// the team kernels' with many views, the staged sweep's boxes beside the window
// weights.  Allowed once per device.
template <typename K>
void allow_dynamic(K kernel, int bytes, std::once_flag* once) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::call_once(once[dev & 63], [=] { cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}
constexpr int kTeamDynamic = team_floats(kMaxSrc) * (int)sizeof(float);   // most of a team kernel
template <bool kHalf, bool kTex, int T>
int launch_init_team(const PhaseArgs& a, cudaStream_t s) {
  static std::once_flag once[64];
  allow_dynamic(init_team_kernel<kHalf, kTex, T>, kTeamDynamic, once);
  const dim3 grid((a.W + 7) / 8, (a.H + 3) / 4);
  init_team_kernel<kHalf, kTex, T><<<grid, 32 * T, kTeamPixels * a.N * sizeof(float), s>>>(a);
  return (int)cudaGetLastError();
}
template <bool kHalf, bool kTex, int T>
int launch_phase_team(const PhaseArgs& a, cudaStream_t s) {
  static std::once_flag once[64];
  allow_dynamic(phase_team_kernel<kHalf, kTex, T>, kTeamDynamic, once);
  const dim3 grid((a.W + 15) / 16, (a.H + 3) / 4);
  // Small phases are short (10 - 20 us): the next one's blocks start loading their
  // windows while this one's last blocks run.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(32 * T);
  cfg.dynamicSmemBytes = team_floats(a.N) * sizeof(float);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, phase_team_kernel<kHalf, kTex, T>, a);
  return (int)cudaGetLastError();
}

template <bool kHalf, bool kTex>
int launch_init_t(const PhaseArgs& a, const DeviceShape& dev, cudaStream_t s) {
  switch (team_warps(init_groups(a.W, a.H), a.N, dev.n_sm, true)) {
    case 16: return launch_init_team<kHalf, kTex, 16>(a, s);
    case 8: return launch_init_team<kHalf, kTex, 8>(a, s);
    case 4: return launch_init_team<kHalf, kTex, 4>(a, s);
    default: break;
  }
  const dim3 grid((a.W + kTile - 1) / kTile, (a.H + 7) / 8);
  return launch_blocks(init_kernel<kHalf, kTex>, grid, kPhaseBlocksPerSM, (int)sizeof(WinShared), 0, a, dev, s);
}
// the texture-filter form exists for uint8 images only (the context refuses
// it with FP16 images and with the ablations)
int launch_init(const PhaseArgs& a, const DeviceShape& dev, cudaStream_t s) {
  if (a.tex_filter) return launch_init_t<false, true>(a, dev, s);
  return a.img_half ? launch_init_t<true, false>(a, dev, s) : launch_init_t<false, false>(a, dev, s);
}

template <bool kHalf, int kMode>
int launch_phase_t(const PhaseArgs& a, const DeviceShape& dev, cudaStream_t s) {
  if constexpr (kMode == 0 || kMode == kTexture) {   // the ablations and the staged sweep: one thread per pixel
    switch (team_warps(phase_groups(a.W, a.H), a.N, dev.n_sm, false)) {
      case 16: return launch_phase_team<kHalf, kMode == kTexture, 16>(a, s);
      case 8: return launch_phase_team<kHalf, kMode == kTexture, 8>(a, s);
      case 4: return launch_phase_team<kHalf, kMode == kTexture, 4>(a, s);
      default: break;
    }
  }
  const dim3 grid((a.W + kTile - 1) / kTile, (a.H + kTile - 1) / kTile);
  if constexpr (kMode == kTexture) {
    if (registers_pay((int64_t)grid.x * grid.y, dev.n_sm, kThreeBlocksPerSM, kPhaseBlocksPerSM))
      return launch_blocks(phase_kernel<kHalf, kMode | kRegs>, grid, kThreeBlocksPerSM, 0, 0, a, dev, s);
  }
  constexpr bool kStaged = (kMode & kStage) != 0;
  constexpr int kDynamic = kStaged ? (int)sizeof(StageShared) : 0;
  if constexpr (kStaged) {
    static std::once_flag once[64];
    allow_dynamic(phase_kernel<kHalf, kMode>, kDynamic, once);
  }
  return launch_blocks(phase_kernel<kHalf, kMode>, grid, phase_blocks_per_sm(kMode), (int)sizeof(WinShared), kDynamic, a,
                       dev, s);
}
template <int kMode>
int launch_phase_m(const PhaseArgs& a, const DeviceShape& dev, cudaStream_t s) {
  // staged sweep on request; at t = 0 the planes are the random ones of the
  // initialisation and no window set fits a box, so those phases fetch
  // through the texture unit
  if (a.staged && a.t > 0)
    return a.img_half ? launch_phase_t<true, kMode | kStage>(a, dev, s) : launch_phase_t<false, kMode | kStage>(a, dev, s);
  return a.img_half ? launch_phase_t<true, kMode>(a, dev, s) : launch_phase_t<false, kMode>(a, dev, s);
}
// the method, or one of the ablations of Sec. 4 (a.ablation: bit 0 symmetric
// propagation, bit 1 heuristic view selection)
int launch_phase(const PhaseArgs& a, const DeviceShape& dev, cudaStream_t s) {
  if (a.tex_filter) return launch_phase_t<false, kTexture>(a, dev, s);
  switch (a.ablation & 3) {
    case kSymmetric: return launch_phase_m<kSymmetric>(a, dev, s);
    case kHeuristic: return launch_phase_m<kHeuristic>(a, dev, s);
    case kSymmetric | kHeuristic: return launch_phase_m<kSymmetric | kHeuristic>(a, dev, s);
    default: return launch_phase_m<0>(a, dev, s);
  }
}

namespace {
// conversion between the state layout and row-major maps
template <class T>
__global__ void __launch_bounds__(256) state_to_rows_kernel(const T* __restrict__ st, T* __restrict__ rows, int W, int H) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x >= W) return;
  for (int y = blockIdx.y; y < H; y += gridDim.y) rows[(size_t)y * W + x] = st[state_index(x, y, W)];
}
template <class T>
__global__ void __launch_bounds__(256) rows_to_state_kernel(const T* __restrict__ rows, T* __restrict__ st, int W, int H) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x >= W) return;
  for (int y = blockIdx.y; y < H; y += gridDim.y) st[state_index(x, y, W)] = rows[(size_t)y * W + x];
}
template <class T>
void launch_convert(const void* src, void* dst, int W, int H, bool to_rows, cudaStream_t s) {
  const dim3 grid((W + 255) / 256, H < 65535 ? H : 65535);
  if (to_rows)
    state_to_rows_kernel<T><<<grid, 256, 0, s>>>(static_cast<const T*>(src), static_cast<T*>(dst), W, H);
  else
    rows_to_state_kernel<T><<<grid, 256, 0, s>>>(static_cast<const T*>(src), static_cast<T*>(dst), W, H);
}
cudaError_t convert(const void* src, void* dst, int W, int H, int elem, bool to_rows, cudaStream_t s) {
  switch (elem) {
    case 16: launch_convert<float4>(src, dst, W, H, to_rows, s); break;
    case 4: launch_convert<uint32_t>(src, dst, W, H, to_rows, s); break;
    case 1: launch_convert<uint8_t>(src, dst, W, H, to_rows, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
}  // namespace

namespace {
// the maps of amh_read_maps in one launch, row-major; any of them may be null
__global__ void __launch_bounds__(256) export_maps_kernel(const float4* __restrict__ plane, const float* __restrict__ cost,
                                                          const uint32_t* __restrict__ wmask, int W, int H,
                                                          float* __restrict__ depth, float* __restrict__ normal3,
                                                          float* __restrict__ cost_out, uint32_t* __restrict__ sel_out) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x >= W) return;
  for (int y = blockIdx.y; y < H; y += gridDim.y) {
    const size_t i = (size_t)y * W + x, q = state_index(x, y, W);
    if (depth || normal3) {
      const float4 p = plane[q];
      if (depth) depth[i] = p.w;
      if (normal3) {
        normal3[3 * i] = p.x;
        normal3[3 * i + 1] = p.y;
        normal3[3 * i + 2] = p.z;
      }
    }
    if (cost_out) cost_out[i] = cost[q];
    if (sel_out) sel_out[i] = wmask[q];
  }
}
}  // namespace
cudaError_t export_maps(const float4* plane, const float* cost, const uint32_t* wmask, int W, int H, float* depth,
                        float* normal3, float* cost_out, uint32_t* sel_out, cudaStream_t s) {
  if (!depth && !normal3 && !cost_out && !sel_out) return cudaSuccess;
  const dim3 grid((W + 255) / 256, H < 65535 ? H : 65535);
  export_maps_kernel<<<grid, 256, 0, s>>>(plane, cost, wmask, W, H, depth, normal3, cost_out, sel_out);
  return cudaGetLastError();
}

cudaError_t export_state_field(const void* state, void* rows, int W, int H, int elem, bool host, cudaStream_t s) {
  if (!host) return convert(state, rows, W, H, elem, true, s);
  const size_t bytes = (size_t)W * H * elem;
  void* tmp = nullptr;
  cudaError_t e = cudaMallocAsync(&tmp, bytes, s);
  if (e != cudaSuccess) return e;
  e = convert(state, tmp, W, H, elem, true, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(rows, tmp, bytes, cudaMemcpyDeviceToHost, s);
  const cudaError_t f = cudaFreeAsync(tmp, s);
  return e != cudaSuccess ? e : f;
}
cudaError_t import_state_field(const void* rows, void* state, int W, int H, int elem, bool host, cudaStream_t s) {
  if (!host) return convert(rows, state, W, H, elem, false, s);
  const size_t bytes = (size_t)W * H * elem;
  void* tmp = nullptr;
  cudaError_t e = cudaMallocAsync(&tmp, bytes, s);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(tmp, rows, bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = convert(tmp, state, W, H, elem, false, s);
  const cudaError_t f = cudaFreeAsync(tmp, s);
  return e != cudaSuccess ? e : f;
}
}  // namespace amh
