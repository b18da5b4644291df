// amh_learned.cu -- the learned proposal network (this project's extension):
// a 4-level convolutional encoder-decoder that reads the half-resolution
// state of the checkerboard update (reference intensity, log depth, normal,
// cost) and proposes one plane per pixel; the phase kernel scores that plane
// with the unchanged matching cost (Eq. 8) and view weights (Eqs. 2-7) as one
// more candidate, so the plain method stays the arbiter.
//
// Kernels: 3x3 convolution forward on the fifth-generation tensor cores
// (tcgen05.mma, FP32 accumulator in tensor memory, BF16 operands brought in by
// the tensor memory accelerator), bias, ReLU, skip addition, 2x2 average pooling
// and nearest upsampling in its epilogue; the data gradient as the same
// convolution with flipped, transposed weights, the adjoints of pooling and
// upsampling, the ReLU masks and the bias sums in its epilogue; the weight
// gradient on the same tensor-core path, reading the pixel-major operands
// directly (amh_conv_tc.cuh); the L1 loss, Adam, and the feature / head /
// proposal conversions.
//
// Layout: activations (H, W, C) with C a multiple of 16, BF16 between
// layers; conv weights (9, Cout, Cin) BF16 (FP32 master copy for Adam), tap
// t = 3 (dy + 1) + (dx + 1).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include <cudaTypedefs.h>

#include "amh.h"
#include "amh_conv_tc.cuh"
#include "amh_ctx.h"
#include "amh_device.cuh"

namespace amh {
namespace {

constexpr int kLayers = 8;
constexpr int kMaxBands = 4;            // bands of rows of the last two layers (amh_net_forward with an output)
struct LayerDef { int cin, cout, relu; };
// e1 e2 e3 e4 d3 d2 d1 out
constexpr LayerDef kNet[kLayers] = {{16, 32, 1}, {32, 64, 1}, {64, 96, 1}, {96, 128, 1},
                                    {128, 96, 1}, {96, 64, 1}, {64, 32, 1}, {32, 16, 0}};

// Bias gradients: db of a layer is the sum of the rows of its partial sums
// (written by the kernels that produce dy), one block per channel and layer.
using tc::kBiasRows;                  // most rows of partial sums of a layer
struct BiasArgs {
  const float* part[kLayers];
  float* db[kLayers];
  int rows[kLayers], C[kLayers];
};
__global__ void __launch_bounds__(256) bias_sum_kernel(BiasArgs a) {
  __shared__ float red[256];
  const int c = blockIdx.x, L = blockIdx.y, C = a.C[L];
  if (c >= C) return;
  float s = 0.f;
  for (int b = threadIdx.x; b < a.rows[L]; b += 256) s += a.part[L][(size_t)b * C + c];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) a.db[L][c] = red[0];
}

// weights (9, Cout, Cin) -> data-gradient weights (9, Cin, Cout), taps flipped
__global__ void flip_transpose_kernel(const __nv_bfloat16* w, __nv_bfloat16* wd, int Cin, int Cout) {
  const int n = 9 * Cin * Cout;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int t = i / (Cin * Cout), ci = (i / Cout) % Cin, co = i % Cout;
    wd[i] = w[((size_t)(8 - t) * Cout + co) * Cin + ci];
  }
}

__global__ void bf16_to_f32_kernel(const __nv_bfloat16* g, float* o, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    o[i] = __bfloat162float(g[i]);
}
// out (H, W, C) FP32: pixels (2 x, 2 y) of the BF16 tensor x (2 H, 2 W, C)
__global__ void subsample_kernel(const __nv_bfloat16* x, float* o, int H, int W, int C) {
  const size_t n = (size_t)H * W * C;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t p = i / C;
    o[i] = __bfloat162float(x[((2 * (p / W)) * (2 * W) + 2 * (p % W)) * C + i % C]);
  }
}
__global__ void to_bf16_kernel(const float* g, __nv_bfloat16* o, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    o[i] = __float2bfloat16(g[i]);
}

// sum of the mask's bytes into *count (zeroed before)
__global__ void __launch_bounds__(256) mask_count_kernel(const uint8_t* __restrict__ mask, int np, unsigned int* count) {
  unsigned int s = 0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < np / 16; i += gridDim.x * 256) {
    const uint4 v = reinterpret_cast<const uint4*>(mask)[i];   // np is a multiple of 64
    s = __dp4a(v.x, 0x01010101u, s);
    s = __dp4a(v.y, 0x01010101u, s);
    s = __dp4a(v.z, 0x01010101u, s);
    s = __dp4a(v.w, 0x01010101u, s);
  }
  s = __reduce_add_sync(0xffffffffu, s);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(count, s);
}
// L1 loss over the 4 used output channels of the masked pixels, divided by the
// mask's sum, and its gradient (zero on the other 12 channels) in FP32 and
// BF16, with its sums per block for the bias gradient; the loss goes to *loss
// (zeroed before), one addition per block
__global__ void __launch_bounds__(256) l1_loss_kernel(const float* __restrict__ out, const float* __restrict__ target,
                                                      const uint8_t* __restrict__ mask,
                                                      const unsigned int* __restrict__ count, float* __restrict__ dout,
                                                      __nv_bfloat16* __restrict__ dout16, float* __restrict__ part,
                                                      float* loss, int np) {
  const float inv_n = 1.f / (float)max(1u, *count);
  float s = 0.f, gs[4] = {0.f, 0.f, 0.f, 0.f};
  // four threads per pixel, each a quarter of its channels: the first has the
  // used ones, the others store zeros
  const int q = threadIdx.x & 3;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 4 * (int64_t)np; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(i >> 2);
    float g[4] = {0.f, 0.f, 0.f, 0.f};
    if (q == 0) {
      const float4 o = reinterpret_cast<const float4*>(out)[(size_t)p * 4];
      const float4 t = reinterpret_cast<const float4*>(target)[p];
      const bool on = mask[p] != 0;
      const float d[4] = {o.x - t.x, o.y - t.y, o.z - t.z, o.w - t.w};
#pragma unroll
      for (int c = 0; c < 4; c++) {
        if (on) {
          s += fabsf(d[c]);
          g[c] = (d[c] > 0.f ? 1.f : (d[c] < 0.f ? -1.f : 0.f)) * inv_n;
        }
        gs[c] += g[c];
      }
    }
    reinterpret_cast<float4*>(dout)[i] = make_float4(g[0], g[1], g[2], g[3]);
    reinterpret_cast<uint2*>(dout16)[i] = make_uint2(tc::pack_bf16(g[0], g[1]), tc::pack_bf16(g[2], g[3]));
  }
  __shared__ float red[8][5];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
    for (int c = 0; c < 4; c++) gs[c] += __shfl_xor_sync(0xffffffffu, gs[c], o);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[warp][4] = s;
    for (int c = 0; c < 4; c++) red[warp][c] = gs[c];
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    float v = 0.f;
    if (threadIdx.x < 4)
      for (int w = 0; w < 8; w++) v += red[w][threadIdx.x];
    part[(size_t)blockIdx.x * 16 + threadIdx.x] = v;
  }
  if (threadIdx.x == 32) {
    float v = 0.f;
    for (int w = 0; w < 8; w++) v += red[w][4];
    atomicAdd(loss, v * inv_n);
  }
}

// One Adam step of every layer (the layers' weights lie one after another, then
// their biases), the weights' BF16 copy and its flipped transpose for the data
// gradients (flip_transpose_kernel).
struct AdamArgs {
  float *w, *m, *v;
  const float* g;
  __nv_bfloat16 *w16, *wd16;
  int n_weights, n;
  int start[kLayers], cin[kLayers], cout[kLayers];
  float lr, b1, b2, eps, c1, c2;
};
__global__ void __launch_bounds__(256) adam_kernel(const __grid_constant__ AdamArgs a) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
    const float gi = a.g[i];
    const float mi = a.b1 * a.m[i] + (1.f - a.b1) * gi, vi = a.b2 * a.v[i] + (1.f - a.b2) * gi * gi;
    a.m[i] = mi;
    a.v[i] = vi;
    const float wi = a.w[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    a.w[i] = wi;
    if (i < a.n_weights) {
      int L = 0;
#pragma unroll
      for (int l = 1; l < kLayers; l++) L += i >= a.start[l];
      const int q = i - a.start[L], cin = a.cin[L], cout = a.cout[L];
      const int ci = q % cin, co = q / cin % cout, t = q / (cin * cout);
      const __nv_bfloat16 h = __float2bfloat16(wi);
      a.w16[i] = h;
      a.wd16[a.start[L] + ((8 - t) * cin + ci) * cout + co] = h;
    }
  }
}

// Features of half-resolution pixel (X, Y), read at full-resolution pixel
// (2X, 2Y): intensity / 255 - 0.5, normalised log depth, normal, cost / 2,
// zeros up to 16 channels.  Also keeps the input plane for the head.  The
// plane and cost come from the context's state (state_index layout).
__global__ void features_kernel(const void* ref, int ref_half, const float4* plane, const float* cost, int W, int H,
                                int w2, int h2, float lmid, float lscale, __nv_bfloat16* x0, float4* pin) {
  const int n = w2 * h2;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int X = p % w2, Y = p / w2;
    const int x = min(2 * X, W - 1), y = min(2 * Y, H - 1);
    const size_t q = (size_t)y * W + x, qs = state_index(x, y, W);   // image, state
    const float I = ref_half ? __half2float(reinterpret_cast<const __half*>(ref)[q])
                             : (float)reinterpret_cast<const uint8_t*>(ref)[q];
    const float4 pl = plane[qs];
    const float f[6] = {I / 255.f - 0.5f, (logf(fmaxf(pl.w, 1e-6f)) - lmid) * lscale, pl.x, pl.y, pl.z,
                        cost[qs] * 0.5f};
    uint4* xr = reinterpret_cast<uint4*>(x0) + (size_t)p * 2;
    xr[0] = make_uint4(tc::pack_bf16(f[0], f[1]), tc::pack_bf16(f[2], f[3]), tc::pack_bf16(f[4], f[5]), 0u);
    xr[1] = make_uint4(0u, 0u, 0u, 0u);
    pin[p] = pl;
  }
}
// one training example, mirrored: output pixel (X, Y) reads source pixel
// (w2 - 1 - X or X, h2 - 1 - Y or Y); an x mirror negates the normal's x
// (feature 2, target 1), a y mirror its y (feature 3, target 2); features
// padded to 16 channels and stored as BF16
__global__ void example_kernel(const float* __restrict__ x, int C, const float* __restrict__ t,
                               const uint8_t* __restrict__ m, int w2, int h2, int mirror, __nv_bfloat16* x0,
                               float* target, uint8_t* mask) {
  const int n = w2 * h2;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int X = p % w2, Y = p / w2;
    const int sx = (mirror & 1) ? w2 - 1 - X : X, sy = (mirror & 2) ? h2 - 1 - Y : Y;
    const size_t q = (size_t)sy * w2 + sx;
    __align__(16) __nv_bfloat16 row[16];
#pragma unroll
    for (int c = 0; c < 16; c++) {
      float v = c < C ? x[q * C + c] : 0.f;
      if ((c == 2 && (mirror & 1)) || (c == 3 && (mirror & 2))) v = -v;
      row[c] = __float2bfloat16(v);
    }
    reinterpret_cast<uint4*>(x0)[(size_t)p * 2] = reinterpret_cast<const uint4*>(row)[0];
    reinterpret_cast<uint4*>(x0)[(size_t)p * 2 + 1] = reinterpret_cast<const uint4*>(row)[1];
    float4 tv = reinterpret_cast<const float4*>(t)[q];
    if (mirror & 1) tv.y = -tv.y;
    if (mirror & 2) tv.z = -tv.z;
    reinterpret_cast<float4*>(target)[p] = tv;
    mask[p] = m[q];
  }
}
// targets: (log D_final - log D_in, n_final - n_in) where the final cost is
// below cmax (confident pixels)
__global__ void targets_kernel(const float4* plane, const float* cost, const float4* pin, int W, int H, int w2,
                               int h2, float cmax, float* target, uint8_t* mask) {
  const int n = w2 * h2;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int X = p % w2, Y = p / w2;
    const int x = min(2 * X, W - 1), y = min(2 * Y, H - 1);
    const size_t q = state_index(x, y, W);
    const float4 pf = plane[q], pi = pin[p];
    const bool ok = cost[q] < cmax && pf.w > 0.f && pi.w > 0.f;
    target[(size_t)p * 4 + 0] = ok ? logf(pf.w) - logf(pi.w) : 0.f;
    target[(size_t)p * 4 + 1] = ok ? pf.x - pi.x : 0.f;
    target[(size_t)p * 4 + 2] = ok ? pf.y - pi.y : 0.f;
    target[(size_t)p * 4 + 3] = ok ? pf.z - pi.z : 0.f;
    mask[p] = ok ? 1 : 0;
  }
}
// head: proposal plane of half-resolution pixel (X, Y) as (n, d) with
// n . X + d = 0, from the input plane and the predicted residuals, valid when
// it faces the camera at full-resolution pixel (2X, 2Y)
__global__ void head_kernel(const float* out, const float4* pin, int W, int H, int w2, int h2, PhaseArgs geo,
                            float4* prop) {
  const int n = w2 * h2;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int X = p % w2, Y = p / w2;
    const float x = (float)min(2 * X, W - 1), y = (float)min(2 * Y, H - 1);
    const float4 pi = pin[p];
    const float* o = out + (size_t)p * 16;
    const float D = pi.w * expf(fminf(fmaxf(o[0], -3.f), 3.f));
    float3 nn = make_float3(pi.x + o[1], pi.y + o[2], pi.z + o[3]);
    const float l = sqrtf(dot3(nn, nn));
    const float3 ray = ref_ray(geo.Kinv, x, y);
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (l > 1e-6f && pi.w > 0.f && isfinite(D)) {
      nn = face_camera(make_float3(nn.x / l, nn.y / l, nn.z / l), ray);
      const float d = -D * dot3(nn, ray);
      if (d > 0.f && isfinite(d)) r = make_float4(nn.x, nn.y, nn.z, d);
    }
    prop[p] = r;
  }
}

int blocks_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 4096); }

}  // namespace
}  // namespace amh

using namespace amh;

// ===========================================================================
// host side
// ===========================================================================
// One convolution of the network, laid out once: its tensor maps, arguments
// and launch shape depend only on the network's own buffers.
struct ConvOp {
  CUtensorMap mx[2], mw[2];
  tc::ConvTcArgs a;
  int epi;
  dim3 grid;
  int threads;
  size_t smem;
};
struct WgradOp {
  CUtensorMap mdy, mx;
  tc::WgradTcArgs a;
  dim3 grid;
  size_t smem;
};
struct amh_net {
  int w2 = 0, h2 = 0;                     // network input size (half resolution)
  cudaStream_t stream = nullptr;
  // parameters per layer: FP32 master, BF16 copy, Adam moments, gradients
  float* wm[kLayers] = {};
  float* bm[kLayers] = {};
  __nv_bfloat16* w16[kLayers] = {};
  __nv_bfloat16* wd16[kLayers] = {};      // data-gradient weights
  float *mw[kLayers] = {}, *vw[kLayers] = {}, *mb[kLayers] = {}, *vb[kLayers] = {};
  float *gw[kLayers] = {}, *gb[kLayers] = {};
  // the layers' arrays lie one after another (weights, then biases): wm, mw,
  // vw and gw of layer 0 start the whole; the loss and the mask's sum follow the
  // gradients
  size_t n_weights = 0, n_params = 0;
  float* bpart[kLayers] = {};             // partial sums of the bias gradients
  int brows[kLayers] = {};                // and their rows
  int step = 0;
  // activations (BF16) and gradient buffers (FP32)
  __nv_bfloat16 *x0 = nullptr, *e1 = nullptr, *in_e2 = nullptr, *e2 = nullptr, *in_e3 = nullptr, *e3 = nullptr,
                *in_e4 = nullptr, *e4 = nullptr, *in_d3 = nullptr, *r3 = nullptr, *in_d2 = nullptr,
                *r2 = nullptr, *in_d1 = nullptr, *r1 = nullptr, *d1 = nullptr;
  float* out = nullptr;
  float* target = nullptr;
  uint8_t* mask = nullptr;
  float4* pin = nullptr;
  float4* prop = nullptr;
  // backward: dy[L] = gradient at layer L's output after its ReLU mask (FP32,
  // and a BF16 copy the tensor cores read), gE1..gE3 gradients arriving at
  // e1..e3 through the skips
  float* dy[kLayers] = {};
  __nv_bfloat16* dy16[kLayers] = {};
  float *gE1 = nullptr, *gE2 = nullptr, *gE3 = nullptr;
  float* scratch = nullptr;               // 64 floats per pixel: host examples, tensors read back
  ConvOp fwd[kLayers], dgr[kLayers];      // forward; data gradients (layer 0 has none)
  WgradOp wgr[kLayers];
  // the output's copy to the host, beside the layers that compute its later rows
  cudaStream_t side = nullptr;
  cudaEvent_t ready = nullptr, done = nullptr;
  int n_bands = 0;
  ConvOp band[2 * kMaxBands];             // the last two layers in bands of rows
  float* loss = nullptr;
  unsigned int* count = nullptr;          // sum of the mask
  unsigned int* status = nullptr;         // bit 0: a convolution's barrier wait gave up
  std::vector<void*> allocs;
  std::string err;
};

namespace {
thread_local std::string g_net_err;
int nfail(amh_net* n, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (n) n->err = buf; else g_net_err = buf;
  return code;
}
template <typename T>
cudaError_t nalloc(amh_net* n, T** p, size_t count) {
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e == cudaSuccess) {
    n->allocs.push_back((void*)*p);
    e = cudaMemsetAsync(*p, 0, count * sizeof(T), n->stream);
  }
  return e;
}
#define NTRY(n, call)                                                                          \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess)                                                                     \
      return nfail(n, e_ == cudaErrorMemoryAllocation ? AMH_ENOMEM : AMH_ECUDA, "%s: %s", #call, \
                   cudaGetErrorString(e_));                                                    \
  } while (0)

void free_net(amh_net* n) {
  if (n->side) cudaStreamDestroy(n->side);
  if (n->ready) cudaEventDestroy(n->ready);
  if (n->done) cudaEventDestroy(n->done);
  for (void* p : n->allocs) cudaFree(p);
  delete n;
}
// the driver's tensor-map encoder, looked up once through the runtime
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}
// tensor map of a BF16 tensor of dims (d0, d1, d2), d0 contiguous, rows of
// pitch0 elements (>= d0), read in boxes of (b0, b1, b2); reads outside the
// tensor return zeros
bool bf16_map(CUtensorMap* m, const void* p, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t b0, uint32_t b1,
              uint32_t b2 = 1, uint64_t pitch0 = 0, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_NONE) {
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return false;
  if (!pitch0) pitch0 = d0;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {pitch0 * 2, pitch0 * d1 * 2};
  cuuint32_t box[3] = {b0, b1, b2};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(p), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// the swizzle of a channel block of conv3x3_tc_kernel: rows of 2 x nch bytes
CUtensorMapSwizzle block_swizzle(int nch) {
  return nch == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : nch == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}

// the convolution kernels, by epilogue
const void* conv_kernel(int epi) {
  switch (epi) {
    case tc::kEpiPool: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiPool>);
    case tc::kEpiUp: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiUp>);
    case tc::kEpiSkip: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiSkip>);
    case tc::kEpiSkipUp: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiSkipUp>);
    case tc::kEpiMask: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiMask>);
    case tc::kEpiDown: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiDown>);
    case tc::kEpiSpread: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiSpread>);
    default: return reinterpret_cast<const void*>(tc::conv3x3_tc_kernel<tc::kEpiPlain>);
  }
}
// Launch of a tensor-core kernel.  overlap: its set-up (barriers, tensor memory,
// weights) may start while the kernel before it on the stream is still running;
// the kernel itself waits for that one before it reads or writes anything else.
// The weights are read during set-up, so they must be complete one ordinary
// launch earlier: the first convolution after they may have changed does not
// overlap.
cudaError_t launch_conv(const void* kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, bool overlap, void** args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, kernel, args);
}

// Lay out a 3x3 convolution on the tensor cores (amh_conv_tc.cuh): x (H, W,
// Cin), w (9, Cout, Cin), Cin and Cout multiples of 16, Cout at most 128; a
// holds the other tensors of the epilogue.
int plan_conv(amh_net* n, ConvOp& op, const __nv_bfloat16* x, const __nv_bfloat16* w, int H, int W, int Cin, int Cout,
              int epi, tc::ConvTcArgs a) {
  if (Cin % 16 || Cin > 128 || Cin % 64 == 48 || Cout % 16 || Cout > tc::kMaxCout)
    return nfail(n, AMH_EINVAL, "conv: channel counts");
  const tc::ConvPlan p = tc::conv_plan(Cin, Cout);
  // one map per kind of channel block (64 channels; the 16 or 32 of the
  // tail); a kind the layer lacks gets a copy of the other
  const int tail = Cin % 64;
  bool ok = true;
  if (Cin >= 64)
    ok = bf16_map(&op.mx[0], x, Cin, W, H, 64, tc::kHalo, 1, 0, block_swizzle(64)) &&
         bf16_map(&op.mw[0], w, Cin, Cout, 9, 64, p.Nb, 1, 0, block_swizzle(64));
  if (ok && tail)
    ok = bf16_map(&op.mx[1], x, Cin, W, H, tail, tc::kHalo, 1, 0, block_swizzle(tail)) &&
         bf16_map(&op.mw[1], w, Cin, Cout, 9, tail, p.Nb, 1, 0, block_swizzle(tail));
  if (!ok) return nfail(n, AMH_ECUDA, "conv: tensor map encoding failed");
  if (Cin < 64) op.mx[0] = op.mx[1], op.mw[0] = op.mw[1];
  if (!tail) op.mx[1] = op.mx[0], op.mw[1] = op.mw[0];
  a.status = n->status;
  if (!a.rows) a.rows = H;                  // all rows
  a.H = H;
  a.W = W;
  a.Cin = Cin;
  a.Cout = Cout;
  a.Nb = p.Nb;
  a.S = p.S;
  op.a = a;
  op.epi = epi;
  op.threads = tc::conv_threads(p.Nb);
  op.smem = p.smem;
  if (p.smem > tc::kConvSmemCap) return nfail(n, AMH_EINVAL, "conv: shared memory plan too large");
  cudaFuncAttributes fa;
  int dev = 0, n_sm = 0;
  cudaError_t e = cudaFuncSetAttribute(conv_kernel(epi), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kConvSmemCap);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, conv_kernel(epi));
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return nfail(n, AMH_ECUDA, "conv: kernel attributes: %s", cudaGetErrorString(e));
  // persistent grid: per channel block, as many CTAs as fit on the SMs at
  // once (every CTA holds its tensor memory until it exits), by the plan and by
  // the register file; at most one per tile (or pair of tiles)
  const int by_regs = 65536 / (((fa.numRegs + 7) & ~7) * op.threads);
  const int cps = std::max(1, std::min(p.ctas_per_sm, by_regs));
  const int nblk = Cout / p.Nb, ntiles = a.rows * ((W + tc::kM - 1) / tc::kM) / (tc::epi_row_pairs(epi) ? 2 : 1);
  op.grid = dim3(tc::conv_grid(ntiles, n_sm, cps, nblk, tc::epi_gradient(epi)), nblk);
  return AMH_OK;
}
int conv(amh_net* n, ConvOp& op, bool overlap) {
  void* args[] = {&op.mx[0], &op.mx[1], &op.mw[0], &op.mw[1], &op.a};
  const cudaError_t e = launch_conv(conv_kernel(op.epi), op.grid, op.threads, op.smem, n->stream, overlap, args);
  if (e != cudaSuccess) return nfail(n, AMH_ECUDA, "conv launch: %s", cudaGetErrorString(e));
  return AMH_OK;
}
int plan_wgrad(amh_net* n, WgradOp& op, int L, const __nv_bfloat16* x, int H, int W);
// every convolution of the forward and backward pass
int plan_network(amh_net* n) {
  const int W0 = n->w2, H0 = n->h2, W1 = W0 / 2, H1 = H0 / 2, W2 = W1 / 2, H2 = H1 / 2, W3 = W2 / 2, H3 = H2 / 2;
  struct F {
    const __nv_bfloat16* x;
    int H, W, epi;
    const __nv_bfloat16* skip;
    __nv_bfloat16 *y16, *r16, *res16;
    float* y32;
  };
  const F f[kLayers] = {{n->x0, H0, W0, tc::kEpiPool, nullptr, n->e1, nullptr, n->in_e2, nullptr},
                        {n->in_e2, H1, W1, tc::kEpiPool, nullptr, n->e2, nullptr, n->in_e3, nullptr},
                        {n->in_e3, H2, W2, tc::kEpiPool, nullptr, n->e3, nullptr, n->in_e4, nullptr},
                        {n->in_e4, H3, W3, tc::kEpiUp, nullptr, n->e4, nullptr, n->in_d3, nullptr},
                        {n->in_d3, H2, W2, tc::kEpiSkipUp, n->e3, nullptr, n->r3, n->in_d2, nullptr},
                        {n->in_d2, H1, W1, tc::kEpiSkipUp, n->e2, nullptr, n->r2, n->in_d1, nullptr},
                        {n->in_d1, H0, W0, tc::kEpiSkip, n->e1, n->d1, n->r1, nullptr, nullptr},
                        {n->d1, H0, W0, tc::kEpiPlain, nullptr, nullptr, nullptr, nullptr, n->out}};
  int rc = AMH_OK;
  for (int L = 0; L < kLayers && !rc; L++) {
    tc::ConvTcArgs a{};
    a.bias = n->bm[L];
    a.skip = f[L].skip;
    a.y16 = f[L].y16;
    a.r16 = f[L].r16;
    a.res16 = f[L].res16;
    a.y32 = f[L].y32;
    a.relu = kNet[L].relu;
    rc = plan_conv(n, n->fwd[L], f[L].x, n->w16[L], f[L].H, f[L].W, kNet[L].cin, kNet[L].cout, f[L].epi, a);
  }
  // data gradients, from dy16[L] to dy[L - 1] (or, through the pooling and the
  // skips, to the layer the gradient passes on to)
  struct D {
    int epi, to;
    const __nv_bfloat16* mask;
    const float* add;
    float* raw;
  };
  const D d[kLayers] = {{},
                        {tc::kEpiSpread, 0, n->e1, n->gE1, nullptr},
                        {tc::kEpiSpread, 1, n->e2, n->gE2, nullptr},
                        {tc::kEpiSpread, 2, n->e3, n->gE3, nullptr},
                        {tc::kEpiDown, 3, n->e4, nullptr, nullptr},      // in_d3 = up(e4)
                        {tc::kEpiDown, 4, n->r3, nullptr, n->gE3},       // in_d2 = up(d3), d3 = r3 + e3
                        {tc::kEpiDown, 5, n->r2, nullptr, n->gE2},       // in_d1 = up(d2), d2 = r2 + e2
                        {tc::kEpiMask, 6, n->r1, nullptr, n->gE1}};      // d1 = r1 + e1
  for (int L = 1; L < kLayers && !rc; L++) {
    tc::ConvTcArgs a{};
    a.mask = d[L].mask;
    a.add32 = d[L].add;
    a.raw32 = d[L].raw;
    a.dy32 = n->dy[d[L].to];
    a.dy16 = n->dy16[d[L].to];
    a.bpart = n->bpart[d[L].to];
    rc = plan_conv(n, n->dgr[L], n->dy16[L], n->wd16[L], f[L].H, f[L].W, kNet[L].cout, kNet[L].cin, d[L].epi, a);
    n->brows[d[L].to] = 4 * (int)n->dgr[L].grid.x;
  }
  // band b of the last layer: rows [H0 b / n, H0 (b + 1) / n); of the layer before
  // it: the rows those need that no earlier band computed (one row ahead)
  n->n_bands = std::max(1, std::min(kMaxBands, H0 / 32));
  for (int b = 0; b < n->n_bands && !rc; b++) {
    const int r0 = H0 * b / n->n_bands, r1 = H0 * (b + 1) / n->n_bands;
    for (int l = 0; l < 2 && !rc; l++) {
      const int L = kLayers - 2 + l;
      tc::ConvTcArgs a = n->fwd[L].a;
      a.row0 = l ? r0 : b ? r0 + 1 : 0;
      a.rows = (l || r1 == H0 ? r1 : r1 + 1) - a.row0;
      rc = plan_conv(n, n->band[2 * b + l], f[L].x, n->w16[L], H0, W0, kNet[L].cin, kNet[L].cout, f[L].epi, a);
    }
  }
  for (int L = 0; L < kLayers && !rc; L++) rc = plan_wgrad(n, n->wgr[L], L, f[L].x, f[L].H, f[L].W);
  return rc;
}
// weight gradient of layer L from its input x and its output gradient (BF16
// dy16): the tensor-core kernel reads both pixel-major and sums a band of rows
// per CTA (all nine taps when Cout <= 32, else the three of one vertical tap)
// into gw
int plan_wgrad(amh_net* n, WgradOp& op, int L, const __nv_bfloat16* x, int H, int W) {
  const int Cin = kNet[L].cin, Cout = kNet[L].cout;
  const int stacked = Cout <= 32 ? 1 : 0, cba = stacked ? Cout : 64, cbb = tc::wgrad_xbox(Cin);
  if (!bf16_map(&op.mdy, n->dy16[L], Cout, W, H, cba, 64, 1, 0, block_swizzle(cba)) ||
      !bf16_map(&op.mx, x, Cin, W, H, cbb, 66, 1, 0, block_swizzle(cbb)))
    return nfail(n, AMH_ECUDA, "wgrad: tensor map encoding failed");
  const int S = tc::wgrad_stages(Cin);
  op.smem = (size_t)S * tc::wgrad_stage_bytes(Cin) + tc::kWgSlack;
  int dev = 0, n_sm = 0;
  cudaError_t e = cudaFuncSetAttribute(tc::wgrad3x3_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(tc::kWgSmemCap + tc::kWgSlack));
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return nfail(n, AMH_ECUDA, "wgrad: kernel attributes: %s", cudaGetErrorString(e));
  // one CTA per SM (the ring takes most of the shared memory), each an equal
  // share of the (row, 64-pixel chunk) steps
  const int gy = stacked ? 1 : 3, steps = H * ((W + 63) / 64);
  const int per_cta = (steps + std::max(1, n_sm / gy) - 1) / std::max(1, n_sm / gy);
  op.a = tc::WgradTcArgs{n->gw[L], n->status, H, W, Cin, Cout, per_cta, stacked, S};
  op.grid = dim3((steps + per_cta - 1) / per_cta, gy);
  return AMH_OK;
}
int wgrad(amh_net* n, WgradOp& op) {
  void* args[] = {&op.mdy, &op.mx, &op.a};
  const cudaError_t e = launch_conv(reinterpret_cast<const void*>(tc::wgrad3x3_tc_kernel), op.grid, tc::kThreads, op.smem,
                                    n->stream, true, args);
  if (e != cudaSuccess) return nfail(n, AMH_ECUDA, "wgrad launch: %s", cudaGetErrorString(e));
  return AMH_OK;
}
// the last two layers in bands, each band's output on its way to the host's
// pinned memory as soon as it is there; the main stream waits for the copies.
// After a failure no copy is left in flight.
int forward_bands(amh_net* n, float* out_host) {
  cudaError_t e = cudaSuccess;
  int rc = AMH_OK;
  for (int b = 0; b < n->n_bands && !rc && e == cudaSuccess; b++) {
    rc = conv(n, n->band[2 * b], true);
    if (!rc) rc = conv(n, n->band[2 * b + 1], true);
    if (rc) break;
    const tc::ConvTcArgs& a = n->band[2 * b + 1].a;
    const size_t first = (size_t)a.row0 * a.W * 16, count = (size_t)a.rows * a.W * 16;
    e = cudaEventRecord(n->ready, n->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(n->side, n->ready, 0);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(out_host + first, n->out + first, count * 4, cudaMemcpyDeviceToHost, n->side);
  }
  if (!rc && e == cudaSuccess) e = cudaEventRecord(n->done, n->side);
  if (!rc && e == cudaSuccess) e = cudaStreamWaitEvent(n->stream, n->done, 0);
  if (rc || e != cudaSuccess) cudaStreamSynchronize(n->side);
  return rc ? rc : e == cudaSuccess ? AMH_OK : nfail(n, AMH_ECUDA, "output copy: %s", cudaGetErrorString(e));
}
}  // namespace

extern "C" {

AMH_API int amh_net_create(amh_net** out, int32_t width2, int32_t height2, uint64_t seed, void* stream) {
  g_net_err.clear();
  if (!out) return nfail(nullptr, AMH_EINVAL, "out is NULL");
  *out = nullptr;
  if (width2 < 8 || height2 < 8 || width2 % 8 || height2 % 8 || (size_t)width2 * height2 > (1u << 24))
    return nfail(nullptr, AMH_EINVAL, "network size must be positive multiples of 8 (at most 2^24 pixels)");
  amh_net* n = new (std::nothrow) amh_net();
  if (!n) return nfail(nullptr, AMH_ENOMEM, "host allocation failed");
  n->w2 = width2;
  n->h2 = height2;
  n->stream = (cudaStream_t)stream;
  auto bail = [&](int code) {
    g_net_err = n->err;
    free_net(n);
    return code;
  };
#define NA(p, c)                                                  \
  do {                                                            \
    cudaError_t e_ = nalloc(n, &(p), (c));                        \
    if (e_ != cudaSuccess) {                                      \
      nfail(n, AMH_ENOMEM, "allocation: %s", cudaGetErrorString(e_)); \
      return bail(AMH_ENOMEM);                                    \
    }                                                             \
  } while (0)
  // He-normal initial weights from a seeded host generator (Box-Muller over
  // a 64-bit LCG), zero biases
  uint64_t s = seed * 6364136223846793005ull + 1442695040888963407ull;
  auto uni = [&]() {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return ((s >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  };
  for (const LayerDef& d : kNet) {
    n->n_weights += (size_t)9 * d.cin * d.cout;
    n->n_params += (size_t)9 * d.cin * d.cout + d.cout;
  }
  float *pw, *pm, *pv, *pg;
  __nv_bfloat16 *p16, *pd16;
  NA(pw, n->n_params); NA(pm, n->n_params); NA(pv, n->n_params); NA(pg, n->n_params + 2);
  NA(p16, n->n_weights); NA(pd16, n->n_weights);
  n->loss = pg + n->n_params;
  n->count = reinterpret_cast<unsigned int*>(n->loss + 1);
  size_t ow = 0, ob = n->n_weights;
  for (int L = 0; L < kLayers; L++) {
    const int Cin = kNet[L].cin, Cout = kNet[L].cout;
    const size_t nw = (size_t)9 * Cin * Cout;
    n->wm[L] = pw + ow; n->mw[L] = pm + ow; n->vw[L] = pv + ow; n->gw[L] = pg + ow;
    n->w16[L] = p16 + ow; n->wd16[L] = pd16 + ow;
    n->bm[L] = pw + ob; n->mb[L] = pm + ob; n->vb[L] = pv + ob; n->gb[L] = pg + ob;
    ow += nw;
    ob += Cout;
    NA(n->bpart[L], (size_t)kBiasRows * Cout);
    std::vector<float> w(nw);
    const double sd = std::sqrt(2.0 / (9.0 * Cin)) * (L == kLayers - 1 ? 0.1 : 1.0);
    for (size_t i = 0; i < nw; i++) w[i] = (float)(sd * std::sqrt(-2.0 * std::log(uni())) * std::cos(6.283185307179586 * uni()));
    cudaMemcpyAsync(n->wm[L], w.data(), nw * sizeof(float), cudaMemcpyHostToDevice, n->stream);
    cudaStreamSynchronize(n->stream);
  }
  NA(n->status, 1);
  const size_t P0 = (size_t)width2 * height2, P1 = P0 / 4, P2 = P0 / 16, P3 = P0 / 64;
  NA(n->x0, P0 * 16); NA(n->e1, P0 * 32); NA(n->in_e2, P1 * 32); NA(n->e2, P1 * 64); NA(n->in_e3, P2 * 64);
  NA(n->e3, P2 * 96); NA(n->in_e4, P3 * 96); NA(n->e4, P3 * 128); NA(n->in_d3, P2 * 128); NA(n->r3, P2 * 96);
  NA(n->in_d2, P1 * 96); NA(n->r2, P1 * 64); NA(n->in_d1, P0 * 64);
  NA(n->r1, P0 * 32); NA(n->d1, P0 * 32);
  NA(n->scratch, P0 * 64);
  {
    const size_t lp[kLayers] = {P0, P1, P2, P3, P2, P1, P0, P0};   // output size of each layer
    for (int L = 0; L < kLayers; L++) {
      NA(n->dy[L], lp[L] * kNet[L].cout);
      NA(n->dy16[L], lp[L] * kNet[L].cout);
    }
  }
  NA(n->gE1, P0 * 32); NA(n->gE2, P1 * 64); NA(n->gE3, P2 * 96);
  NA(n->out, P0 * 16); NA(n->target, P0 * 4); NA(n->mask, P0); NA(n->pin, P0); NA(n->prop, P0);
#undef NA
  cudaError_t se = cudaStreamCreateWithFlags(&n->side, cudaStreamNonBlocking);
  if (se == cudaSuccess) se = cudaEventCreateWithFlags(&n->ready, cudaEventDisableTiming);
  if (se == cudaSuccess) se = cudaEventCreateWithFlags(&n->done, cudaEventDisableTiming);
  if (se != cudaSuccess) {
    nfail(n, AMH_ECUDA, "side stream: %s", cudaGetErrorString(se));
    return bail(AMH_ECUDA);
  }
  if (const int rc = plan_network(n)) return bail(rc);
  for (int L = 0; L < kLayers; L++) {
    const size_t nw = (size_t)9 * kNet[L].cin * kNet[L].cout;
    to_bf16_kernel<<<blocks_for(nw), 256, 0, n->stream>>>(n->wm[L], n->w16[L], nw);
    flip_transpose_kernel<<<blocks_for(nw), 256, 0, n->stream>>>(n->w16[L], n->wd16[L], kNet[L].cin, kNet[L].cout);
  }
  cudaError_t e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) {
    nfail(n, AMH_ECUDA, "net init: %s", cudaGetErrorString(e));
    return bail(AMH_ECUDA);
  }
  *out = n;
  return AMH_OK;
}

AMH_API int amh_net_params(amh_net* n, int32_t layer, float* w, float* b, int32_t set) {
  if (!n || layer < 0 || layer >= kLayers) return AMH_EINVAL;
  const size_t nw = (size_t)9 * kNet[layer].cin * kNet[layer].cout, nb = kNet[layer].cout;
  if (set) {
    if (w) NTRY(n, cudaMemcpyAsync(n->wm[layer], w, nw * 4, cudaMemcpyHostToDevice, n->stream));
    if (b) NTRY(n, cudaMemcpyAsync(n->bm[layer], b, nb * 4, cudaMemcpyHostToDevice, n->stream));
    to_bf16_kernel<<<blocks_for(nw), 256, 0, n->stream>>>(n->wm[layer], n->w16[layer], nw);
    flip_transpose_kernel<<<blocks_for(nw), 256, 0, n->stream>>>(n->w16[layer], n->wd16[layer], kNet[layer].cin,
                                                                kNet[layer].cout);
  } else {
    if (w) NTRY(n, cudaMemcpyAsync(w, n->wm[layer], nw * 4, cudaMemcpyDeviceToHost, n->stream));
    if (b) NTRY(n, cudaMemcpyAsync(b, n->bm[layer], nb * 4, cudaMemcpyDeviceToHost, n->stream));
  }
  NTRY(n, cudaStreamSynchronize(n->stream));
  return AMH_OK;
}

AMH_API int amh_net_grads(amh_net* n, int32_t layer, float* gw, float* gb) {
  if (!n || layer < 0 || layer >= kLayers) return AMH_EINVAL;
  const size_t nw = (size_t)9 * kNet[layer].cin * kNet[layer].cout, nb = kNet[layer].cout;
  if (gw) NTRY(n, cudaMemcpyAsync(gw, n->gw[layer], nw * 4, cudaMemcpyDeviceToHost, n->stream));
  if (gb) NTRY(n, cudaMemcpyAsync(gb, n->gb[layer], nb * 4, cudaMemcpyDeviceToHost, n->stream));
  NTRY(n, cudaStreamSynchronize(n->stream));
  return AMH_OK;
}

// input features (H2 x W2 x 16) from the host (tests), or from a context
AMH_API int amh_net_set_input(amh_net* n, const float* x0_host) {
  if (!n || !x0_host) return AMH_EINVAL;
  const size_t ne = (size_t)n->w2 * n->h2 * 16;
  std::vector<__nv_bfloat16> h(ne);
  for (size_t i = 0; i < ne; i++) h[i] = __float2bfloat16(x0_host[i]);
  NTRY(n, cudaMemcpyAsync(n->x0, h.data(), ne * 2, cudaMemcpyHostToDevice, n->stream));
  NTRY(n, cudaStreamSynchronize(n->stream));
  return AMH_OK;
}

AMH_API int amh_net_set_example(amh_net* n, const float* x, int32_t channels, const float* target,
                                const uint8_t* mask, int32_t mirror, int32_t mem) {
  if (!n || !x || !target || !mask) return AMH_EINVAL;
  if (channels < 1 || channels > 16) return nfail(n, AMH_EINVAL, "channels must be 1..16");
  if (mem != AMH_MEM_HOST && mem != AMH_MEM_DEVICE) return nfail(n, AMH_EINVAL, "bad memory kind");
  const size_t np = (size_t)n->w2 * n->h2;
  const float *dx = x, *dt = target;
  const uint8_t* dm = mask;
  float* const ts = n->scratch;           // targets, then the features, then the mask
  if (mem == AMH_MEM_HOST) {
    float* xs = ts + np * 4;
    uint8_t* ms = reinterpret_cast<uint8_t*>(xs + np * 16);
    NTRY(n, cudaMemcpyAsync(xs, x, np * channels * 4, cudaMemcpyHostToDevice, n->stream));
    NTRY(n, cudaMemcpyAsync(ts, target, np * 16, cudaMemcpyHostToDevice, n->stream));
    NTRY(n, cudaMemcpyAsync(ms, mask, np, cudaMemcpyHostToDevice, n->stream));
    dx = xs;
    dt = ts;
    dm = ms;
  }
  if (reinterpret_cast<uintptr_t>(dt) & 15) {   // the kernel reads each pixel's targets as one float4
    NTRY(n, cudaMemcpyAsync(ts, dt, np * 16, cudaMemcpyDeviceToDevice, n->stream));
    dt = ts;
  }
  example_kernel<<<blocks_for(np), 256, 0, n->stream>>>(dx, channels, dt, dm, n->w2, n->h2, mirror & 3, n->x0,
                                                        n->target, n->mask);
  NTRY(n, cudaGetLastError());
  return AMH_OK;
}

AMH_API int amh_net_features(amh_net* n, amh_ctx* c) {
  if (!n || !c) return AMH_EINVAL;
  if ((c->W + 1) / 2 > n->w2 || (c->H + 1) / 2 > n->h2) return nfail(n, AMH_EINVAL, "context larger than the network");
  const float lmid = 0.5f * (std::log(c->p.depth_min) + std::log(c->p.depth_max));
  const float lscale = 2.f / std::max(1e-6f, std::log(c->p.depth_max / c->p.depth_min));
  features_kernel<<<blocks_for((size_t)n->w2 * n->h2), 256, 0, n->stream>>>(
      c->d_ref, c->args.img_half, c->d_plane, c->d_cost, c->W, c->H, n->w2, n->h2, lmid, lscale, n->x0, n->pin);
  NTRY(n, cudaGetLastError());
  return AMH_OK;
}

AMH_API int amh_net_targets(amh_net* n, amh_ctx* c, float cost_max) {
  if (!n || !c) return AMH_EINVAL;
  targets_kernel<<<blocks_for((size_t)n->w2 * n->h2), 256, 0, n->stream>>>(
      c->d_plane, c->d_cost, n->pin, c->W, c->H, n->w2, n->h2, cost_max, n->target, n->mask);
  NTRY(n, cudaGetLastError());
  return AMH_OK;
}

AMH_API int amh_net_set_targets(amh_net* n, const float* target_host, const uint8_t* mask_host) {
  if (!n || !target_host || !mask_host) return AMH_EINVAL;
  const size_t np = (size_t)n->w2 * n->h2;
  NTRY(n, cudaMemcpyAsync(n->target, target_host, np * 16, cudaMemcpyHostToDevice, n->stream));
  NTRY(n, cudaMemcpyAsync(n->mask, mask_host, np, cudaMemcpyHostToDevice, n->stream));
  NTRY(n, cudaStreamSynchronize(n->stream));
  return AMH_OK;
}

AMH_API int amh_net_forward(amh_net* n, float* out_host) {
  if (!n) return AMH_EINVAL;
  const cudaStream_t s = n->stream;
  int rc = AMH_OK;
  // An output to pinned memory is copied in bands of rows while the next band of
  // the last two layers runs (the copy of 800 x 528 takes 142 us on the link,
  // the two layers 55; with 1, 2, 3, 4, 6 bands 312, 292, 286, 284, 286 us).  A
  // copy to pageable memory holds the host until it is done and goes last.
  bool bands = false;
  if (out_host) {
    cudaPointerAttributes at;
    const cudaError_t e = cudaPointerGetAttributes(&at, out_host);
    if (e != cudaSuccess) cudaGetLastError();
    bands = e == cudaSuccess && at.type == cudaMemoryTypeHost;
  }
  for (int L = 0; L < (bands ? kLayers - 2 : kLayers) && !rc; L++) rc = conv(n, n->fwd[L], L > 0);
  if (bands) {
    if (!rc) rc = forward_bands(n, out_host);
    if (rc) return rc;
    NTRY(n, cudaGetLastError());
    NTRY(n, cudaStreamSynchronize(s));
    return AMH_OK;
  }
  if (rc) return rc;
  NTRY(n, cudaGetLastError());
  if (out_host) {
    NTRY(n, cudaMemcpyAsync(out_host, n->out, (size_t)n->w2 * n->h2 * 16 * 4, cudaMemcpyDeviceToHost, s));
    NTRY(n, cudaStreamSynchronize(s));
  }
  return AMH_OK;
}

// loss of the last forward against the targets, and all gradients
AMH_API int amh_net_backward(amh_net* n, float* loss_out) {
  if (!n) return AMH_EINVAL;
  const size_t P0 = (size_t)n->w2 * n->h2;
  const cudaStream_t s = n->stream;
  // gradients, loss and the mask's sum
  NTRY(n, cudaMemsetAsync(n->gw[0], 0, (n->n_params + 2) * sizeof(float), s));
  mask_count_kernel<<<(int)std::min<size_t>((P0 / 16 + 255) / 256, 152), 256, 0, s>>>(n->mask, (int)P0, n->count);
  const int lb = (int)std::min<size_t>((P0 * 4 + 255) / 256, kBiasRows);
  l1_loss_kernel<<<lb, 256, 0, s>>>(n->out, n->target, n->mask, n->count, n->dy[7], n->dy16[7], n->bpart[7], n->loss, (int)P0);
  n->brows[7] = lb;
  int rc = AMH_OK;
  for (int L = kLayers - 1; L >= 0 && !rc; L--) {
    rc = wgrad(n, n->wgr[L]);
    if (!rc && L > 0) rc = conv(n, n->dgr[L], true);
  }
  BiasArgs ba;
  for (int L = 0; L < kLayers; L++) {
    ba.part[L] = n->bpart[L];
    ba.db[L] = n->gb[L];
    ba.rows[L] = n->brows[L];
    ba.C[L] = kNet[L].cout;
  }
  bias_sum_kernel<<<dim3(128, kLayers), 256, 0, s>>>(ba);
  if (rc) return rc;
  NTRY(n, cudaGetLastError());
  if (loss_out) {
    NTRY(n, cudaMemcpyAsync(loss_out, n->loss, 4, cudaMemcpyDeviceToHost, s));
    NTRY(n, cudaStreamSynchronize(s));
  }
  return AMH_OK;
}

AMH_API int amh_net_adam(amh_net* n, float lr) {
  if (!n) return AMH_EINVAL;
  n->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n->step), c2 = 1.f - std::pow(b2, (float)n->step);
  AdamArgs a;
  a.w = n->wm[0];
  a.m = n->mw[0];
  a.v = n->vw[0];
  a.g = n->gw[0];
  a.w16 = n->w16[0];
  a.wd16 = n->wd16[0];
  a.n_weights = (int)n->n_weights;
  a.n = (int)n->n_params;
  for (int L = 0; L < kLayers; L++) {
    a.start[L] = (int)(n->wm[L] - n->wm[0]);
    a.cin[L] = kNet[L].cin;
    a.cout[L] = kNet[L].cout;
  }
  a.lr = lr;
  a.b1 = b1;
  a.b2 = b2;
  a.eps = 1e-8f;
  a.c1 = c1;
  a.c2 = c2;
  adam_kernel<<<blocks_for(n->n_params), 256, 0, n->stream>>>(a);
  NTRY(n, cudaGetLastError());
  return AMH_OK;
}

// the proposal planes of the last forward, handed to the context's phases
AMH_API int amh_net_propose(amh_net* n, amh_ctx* c) {
  if (!n || !c) return AMH_EINVAL;
  head_kernel<<<blocks_for((size_t)n->w2 * n->h2), 256, 0, n->stream>>>(n->out, n->pin, c->W, c->H, n->w2, n->h2,
                                                                        c->args, n->prop);
  NTRY(n, cudaGetLastError());
  c->args.prop = n->prop;
  c->args.prop_w = n->w2;
  c->args.prop_h = n->h2;
  return AMH_OK;
}

AMH_API int amh_clear_proposal(amh_ctx* c) {
  if (!c) return AMH_EINVAL;
  c->args.prop = nullptr;
  return AMH_OK;
}

// internal tensors for element-wise checks of every operation
AMH_API int amh_net_read(amh_net* n, int32_t which, float* out, int64_t* count) {
  if (!n || !count) return AMH_EINVAL;
  const size_t P0 = (size_t)n->w2 * n->h2, P1 = P0 / 4, P2 = P0 / 16, P3 = P0 / 64;
  struct B { const __nv_bfloat16* b; const float* f; size_t n; };
  const B act[] = {{n->x0, nullptr, P0 * 16},   {n->e1, nullptr, P0 * 32},    {n->in_e2, nullptr, P1 * 32},
                   {n->e2, nullptr, P1 * 64},   {n->in_e3, nullptr, P2 * 64}, {n->e3, nullptr, P2 * 96},
                   {n->in_e4, nullptr, P3 * 96}, {n->e4, nullptr, P3 * 128},  {n->in_d3, nullptr, P2 * 128},
                   {n->r3, nullptr, P2 * 96},   {n->in_d2, nullptr, P2 * 96},  {n->in_d2, nullptr, P1 * 96},
                   {n->r2, nullptr, P1 * 64},   {n->in_d1, nullptr, P1 * 64},  {n->in_d1, nullptr, P0 * 64},
                   {n->r1, nullptr, P0 * 32},   {n->d1, nullptr, P0 * 32},    {nullptr, n->out, P0 * 16}};
  constexpr int kAct = (int)(sizeof(act) / sizeof(act[0]));
  const size_t lp[kLayers] = {P0, P1, P2, P3, P2, P1, P0, P0};
  B src{};
  if (which == 65) {   // the mask, as 0 / 1
    if (!out) {
      *count = (int64_t)P0;
      return AMH_OK;
    }
    if (*count != (int64_t)P0) return nfail(n, AMH_EINVAL, "the mask has %zu elements", P0);
    std::vector<uint8_t> h(P0);
    NTRY(n, cudaMemcpyAsync(h.data(), n->mask, P0, cudaMemcpyDeviceToHost, n->stream));
    NTRY(n, cudaStreamSynchronize(n->stream));
    for (size_t i = 0; i < P0; i++) out[i] = (float)h[i];
    return AMH_OK;
  }
  if (which >= 0 && which < kAct) src = act[which];
  else if (which >= 32 && which < 32 + kLayers) src = B{nullptr, n->dy[which - 32], lp[which - 32] * kNet[which - 32].cout};
  else if (which == 64) src = B{nullptr, n->target, P0 * 4};
  else return nfail(n, AMH_EINVAL, "unknown tensor %d", which);
  if (!out) {
    *count = (int64_t)src.n;
    return AMH_OK;
  }
  if (*count != (int64_t)src.n) return nfail(n, AMH_EINVAL, "tensor %d has %zu elements, not %lld", which, src.n, (long long)*count);
  const float* dev = src.f;
  if (src.b) {   // BF16 -> FP32 in the scratch buffer (the largest tensor fits)
    // d3 and d2 exist upsampled only: every other pixel and row of in_d2, in_d1
    const int sub = which == 10 ? 4 : which == 13 ? 2 : 0;
    const int C = which == 10 ? 96 : 64;
    if (sub)
      subsample_kernel<<<blocks_for(src.n), 256, 0, n->stream>>>(src.b, n->scratch, n->h2 / sub, n->w2 / sub, C);
    else
      bf16_to_f32_kernel<<<blocks_for(src.n), 256, 0, n->stream>>>(src.b, n->scratch, src.n);
    NTRY(n, cudaGetLastError());
    dev = n->scratch;
  }
  NTRY(n, cudaMemcpyAsync(out, dev, src.n * 4, cudaMemcpyDeviceToHost, n->stream));
  NTRY(n, cudaStreamSynchronize(n->stream));
  return AMH_OK;
}

AMH_API int amh_net_synchronize(amh_net* n) {
  if (!n) return AMH_EINVAL;
  NTRY(n, cudaStreamSynchronize(n->stream));
  unsigned int st = 0;
  NTRY(n, cudaMemcpy(&st, n->status, sizeof st, cudaMemcpyDeviceToHost));
  if (st) return nfail(n, AMH_EDEVICE, "a convolution's barrier wait gave up (status 0x%x)", st);
  return AMH_OK;
}

AMH_API const char* amh_net_last_error(const amh_net* n) { return n ? n->err.c_str() : g_net_err.c_str(); }

AMH_API void amh_net_destroy(amh_net* n) {
  if (!n) return;
  cudaStreamSynchronize(n->stream);
  cudaStreamSynchronize(n->side);
  free_net(n);
}

}  // extern "C"
