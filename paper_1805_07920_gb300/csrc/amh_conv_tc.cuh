// amh_conv_tc.cuh -- 3x3 convolution (stride 1, zero padding) of the learned
// proposal network on the fifth-generation tensor cores: tcgen05.mma with the
// FP32 accumulator in tensor memory, BF16 operands brought into shared memory
// by the tensor memory accelerator (cp.async.bulk.tensor).
//
// Implicit GEMM: D (pixels x Cout) = sum over the 9 taps t and the input
// channels ci of X (pixel + off(t), ci) W (t, co, ci), one MMA per tap and 16
// input channels (M = 128 pixels of one row, N = a block of output channels,
// K = 16).  Both operands sit in shared memory in the tensor cores' K-major
// layout, in blocks of 64 channels (128-byte rows, 128-byte swizzle; a 16- or
// 32-channel remainder in 32- or 64-byte rows).  The forward / data-gradient
// kernel keeps its block of weights resident and streams input rows with a
// one-pixel halo, each row loaded once per run of vertically adjacent tiles
// (its comment below gives the schedule); the weight-gradient kernel streams
// 64-pixel chunks of the same pixel-major tensors as MN-major operands.  A
// producer warp issues the TMA copies, an MMA warp consumes them and recycles
// each buffer once the MMAs that read it have committed, and the epilogue
// warps read the accumulator with tcgen05.ld and apply bias, ReLU, skip
// addition and the BF16 / FP32 stores.
//
// Layout: activations (H, W, C) BF16 with C a multiple of 16; weights (9,
// Cout, Cin) BF16, tap t = 3 (dy + 1) + (dx + 1); Cout a multiple of 16, at
// most 128.  Every wait on a barrier gives up after a bounded number of
// tries and sets the status word instead of hanging.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace amh {
namespace tc {

constexpr int kM = 128;          // pixels per CTA (rows of the accumulator)
constexpr int kMaxCout = 128;
constexpr uint32_t kWaitTries = 1u << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// true once the barrier's phase with the given parity has completed; false
// after kWaitTries unsuccessful tries.  A waiter that is not on the critical
// path passes sleep_ns, so that between tries it leaves the issue slots of its
// SM sub-partition to the warps that are.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, uint32_t sleep_ns = 0) {
  uint32_t done = 0;
  for (uint32_t it = 0; it < kWaitTries; it++) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    if (done) break;
    if (sleep_ns) __nanosleep(sleep_ns);
  }
  return done != 0;
}
// TMA: one box of a 3-D tensor into shared memory, completion counted on bar
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}
// Shared-memory matrix descriptor of a tcgen05 operand, as two 32-bit words.
// Low word: start address >> 4 (bits 0-13) and the leading byte offset >> 4
// (bits 16-29; ignored for swizzled K-major operands, set to 16 bytes;
// for MN-major operands the step between blocks along M / N, see
// desc_lo_mn).  High word: the stride byte offset >> 4 (between 8-row groups:
// along M / N for K-major, along K for MN-major; 8 rows of `pitch` bytes
// either way), descriptor version 1 (bit 46 of the whole), base offset 0 and
// the layout in bits 61-63 (2, 4, 6: rows of 128, 64, 32 bytes with the
// matching swizzle).  The swizzle pattern follows the shared-memory address
// bits, so a start moved by whole rows stays consistent with what the TMA
// wrote.  The low word moves with the operand; the high word is fixed per
// channel block.
__host__ __device__ constexpr uint32_t swizzle_layout(int pitch) { return pitch == 128 ? 2u : pitch == 64 ? 4u : 6u; }
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_hi(uint32_t pitch) {
  return ((8u * pitch) >> 4) | (1u << 14) | (swizzle_layout((int)pitch) << 29);
}
__device__ __forceinline__ uint64_t desc_pack(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

// position in a ring of S buffers: the slot and the parity of its current use
struct RingPos {
  uint32_t slot, phase;
  __device__ __forceinline__ RingPos next(uint32_t S) const {
    return slot + 1 == S ? RingPos{0u, phase ^ 1u} : RingPos{slot + 1, phase};
  }
};
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t mma_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// The MMA warps run their issue loops with all 32 lanes converged, so that
// the descriptor arithmetic is warp-uniform; one lane chosen by elect.sync
// (the same lane every time, the warp being converged) issues each MMA and
// each commit.  Measured: 39-48 cycles per M = 128, K = 16 MMA (N <= 64)
// with the descriptors computed in the loop this way, 63-68 cycles when a
// single lane runs the loop.
__device__ __forceinline__ void mma_bf16_elect(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit_elect(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar))
      : "memory");
}
// a barrier wait by the whole warp, with one answer for all its lanes
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(b, parity));
}
// 16 consecutive accumulator columns of this thread's TMEM lane (the warp
// reads its lane quarter); the caller waits with tcgen05.wait::ld
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// Both kernels are persistent and warp-specialised: epilogue warps drain the
// accumulator (a warp reads the TMEM lanes of its SM sub-partition, lanes
// 32 (w % 4) .. 32 (w % 4) + 31), one warp produces (TMA), one allocates the
// tensor memory and issues the MMAs.  Two accumulators in tensor memory let
// the epilogue of one tile overlap the MMAs of the next.  The weight-gradient
// kernel has 4 epilogue warps (kThreads); the convolution kernel has 4 per
// 16 output channels of its block (conv_threads), so that the chunks of a
// tile drain in parallel.
constexpr int kThreads = 192;

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

// Lane pairs (2k, 2k + 1) hold neighbouring pixels, each lane its pixel's
// 32-byte sector (16 BF16 channels) as two 16-byte halves lo, hi.  After the
// exchange the even lane holds both pixels' lo, the odd lane both pixels' hi
// (a of the even pixel, b of the odd one), so that storing a and then b at the
// lane's half writes whole sectors with each instruction.  All 32 lanes call it.
struct SectorPair {
  uint4 a, b;
};
__device__ __forceinline__ uint4 shfl_xor1(uint4 v) {
  return make_uint4(__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1),
                    __shfl_xor_sync(0xffffffffu, v.z, 1), __shfl_xor_sync(0xffffffffu, v.w, 1));
}
__device__ __forceinline__ SectorPair pair_exchange(uint4 lo, uint4 hi, bool odd) {
  const uint4 recv = shfl_xor1(odd ? lo : hi);
  return odd ? SectorPair{recv, hi} : SectorPair{lo, recv};
}
// the programmatic dependent launch: the next kernel of the stream may start
// its set-up once every block has called pdl_launch; pdl_wait returns when the
// kernel before has finished and its writes are visible
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t v) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v));
}
// eight values as BF16 (16 bytes), and back
__device__ __forceinline__ uint4 pack8(const float* f) {
  return make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
}
__device__ __forceinline__ void unpack8(uint4 v, float* f) {
  const float2 a = unpack_bf16(v.x), b = unpack_bf16(v.y), c = unpack_bf16(v.z), d = unpack_bf16(v.w);
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y; f[4] = c.x; f[5] = c.y; f[6] = d.x; f[7] = d.y;
}
// Transpose within each group of four lanes (four neighbouring pixels, 16 FP32
// channels each): t[k] becomes channels 4 (lane % 4) .. + 3 of pixel k of the
// group, so that one 16-byte access per lane covers 64 contiguous bytes of
// eight pixels instead of 16 bytes of 32.  All 32 lanes call it.
__device__ __forceinline__ void quad_transpose(float (&t)[4][4], int lane) {
#pragma unroll
  for (int s = 1; s <= 2; s <<= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (k & s) continue;
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const float r = __shfl_xor_sync(0xffffffffu, up ? t[k][e] : t[k + s][e], s);
        if (up) t[k][e] = r;
        else t[k + s][e] = r;
      }
    }
  }
}
__device__ __forceinline__ void store4(float* p, const float* f) {
  *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
}

// Forward / data-gradient kernel.  A tile is 128 consecutive pixels of one
// output row and one block of Nb output channels; CTA (bx, by) owns channel
// block by and a contiguous range of the tiles ordered (128-pixel column
// segment, row), i.e. runs of vertically adjacent tiles.  Its Nb x Cin x 9
// weights are loaded into shared memory once.  The input enters as slabs:
// one input row, 130 pixels (the tile's 128 and one halo pixel on each side)
// x all Cin channels.  Channels are split into blocks of 64 (128-byte rows)
// and a tail of 16 or 32 (32- or 64-byte rows); each block is one TMA box
// with the swizzle of its row length, 1024-byte aligned, and the weights of
// a tap use the same blocks.  Output row y reads the slabs of input rows
// y - 1, y, y + 1, and the tap (dx, dy) of slab y + dy is the same block seen
// from row 1 + dx: its matrix descriptor starts 1 + dx rows later (the
// swizzle pattern follows the address, so the shifted view reads what the
// TMA wrote).  So each input row of a run is loaded once and feeds
// 9 Cin / 16 MMAs (M = 128, N = Nb, K = 16) for three output rows.  The slabs
// sit in a ring of S stages; slab k is released when output row k + 1 (the
// last one reading it) has committed its MMAs.
constexpr int kHalo = kM + 2;               // pixels per slab row
constexpr int kMaxStages = 8;
constexpr int kConvMaxNb = 64;              // output channels per CTA
// threads of conv3x3_tc_kernel: 4 epilogue warps per 16 output channels of the
// block (one per TMEM lane quarter and 16-channel chunk), the producer and the
// MMA warp
__host__ __device__ constexpr int conv_threads(int nb) { return 32 * (4 * (nb / 16) + 2); }
constexpr int kConvMaxThreads = 32 * (4 * (kConvMaxNb / 16) + 2);

// What the epilogue does with a pixel's accumulator.  The encoder layers also
// write the 2 x 2 mean the next level reads, the decoder layers the nearest
// upsampling the next layer reads (instead of, or beside, their own output):
// as passes of their own these took 70 of the forward's 225 us of kernels at
// 800 x 528.
enum ConvEpi {
  kEpiPlain,    // y32
  kEpiPool,     // y16, and up / down: its 2 x 2 mean (H / 2, W / 2)
  kEpiUp,       // y16, and its nearest upsampling (2 H, 2 W)
  kEpiSkip,     // r16 before the skip addition, y16 after
  kEpiSkipUp,   // r16 before the skip addition, the upsampling of the sum
  // Data gradients, on to the gradient dy of the layer below (after its ReLU
  // mask; FP32 and BF16, with its sums over the pixels for the bias gradient):
  // as separate passes these moved 600 MB and took 170 us of a backward pass at
  // 800 x 528.
  kEpiMask,     // raw32 = the gradient; dy = it where mask > 0
  kEpiDown,     // adjoint of the upsampling: sums of 2 x 2 pixels into raw32 (or null) and dy, (H / 2, W / 2)
  kEpiSpread    // adjoint of the pooling: add32 + gradient / 4 on 2 x 2 pixels, into dy, (2 H, 2 W)
};
__host__ __device__ constexpr bool epi_row_pairs(int epi) { return epi == kEpiPool || epi == kEpiDown; }   // tiles come in vertical pairs
__host__ __device__ constexpr bool epi_gradient(int epi) { return epi == kEpiMask || epi == kEpiDown || epi == kEpiSpread; }

struct ConvTcArgs {
  const float* bias;          // Cout or null
  const __nv_bfloat16* skip;  // (H, W, Cout) added after the ReLU
  __nv_bfloat16* y16;         // (H, W, Cout) BF16 output (after ReLU + skip)
  __nv_bfloat16* r16;         // (H, W, Cout) ReLU output before the skip
  __nv_bfloat16* res16;       // the 2 x 2 mean or the upsampling of the output
  float* y32;                 // (H, W, Cout) FP32 output
  const __nv_bfloat16* mask;  // data gradients: the ReLU output of the layer below
  const float* add32;
  float *raw32, *dy32;
  __nv_bfloat16* dy16;
  float* bpart;               // sums of dy per CTA and lane quarter: row 4 blockIdx.x + quarter, Cout channels
  unsigned int* status;       // bit 0: a barrier wait gave up
  int H, W, Cin, Cout, relu;
  int row0, rows;             // output rows row0 .. row0 + rows - 1
  int Nb;                     // output channels per CTA (a multiple of 16 dividing Cout, at most kConvMaxNb)
  int S;                      // slab stages (3 .. kMaxStages)
};

// channel blocks of a Cin-channel operand: cin / 64 blocks of 64 channels,
// then a tail of cin % 64 (0, 16 or 32) channels; each block's region is
// rows x (2 x its channels) bytes rounded up to 1 KB
__host__ __device__ constexpr size_t round_1k(size_t b) { return (b + 1023) & ~(size_t)1023; }
__host__ __device__ constexpr size_t conv_block_bytes(int cin, int rows) {
  return (size_t)(cin / 64) * round_1k((size_t)rows * 128) + (cin % 64 ? round_1k((size_t)rows * 2 * (cin % 64)) : 0);
}
// dynamic shared memory of conv3x3_tc_kernel: alignment slack, the weights
// (9 taps of Nb rows), the slab ring (rows of kHalo pixels)
__host__ __device__ constexpr size_t conv_wtap_bytes(int cin, int nb) { return conv_block_bytes(cin, nb); }
__host__ __device__ constexpr size_t conv_weight_bytes(int cin, int nb) { return 9 * conv_wtap_bytes(cin, nb); }
__host__ __device__ constexpr size_t conv_slab_bytes(int cin) { return conv_block_bytes(cin, kHalo); }
__host__ __device__ constexpr size_t conv_smem_bytes(int cin, int nb, int s) {
  return 1024 + conv_weight_bytes(cin, nb) + (size_t)s * conv_slab_bytes(cin);
}
// tensor-memory columns of one accumulator (allocations are powers of two >= 32)
__host__ __device__ constexpr uint32_t conv_acc_cols(int nb) { return nb <= 32 ? 32u : nb <= 64 ? 64u : 128u; }

// run r of the CTA's tile range: tiles u .. u + len - 1 of one column segment
struct TileRun {
  int seg, y0, len;
};
__device__ __forceinline__ bool next_run(int& u, int hi, int H, TileRun& r) {
  if (u >= hi) return false;
  r.seg = u / H;
  r.y0 = u % H;
  r.len = min(hi - u, H - r.y0);
  u += r.len;
  return true;
}

// tx_main / tw_main: boxes of 64 channels x (kHalo pixels | Nb output
// channels), 128-byte swizzle; tx_tail / tw_tail: the same for the tail
// channels (unused when Cin is a multiple of 64)
template <int kEpi>
__global__ void __launch_bounds__(kConvMaxThreads, 1) conv3x3_tc_kernel(const __grid_constant__ CUtensorMap tx_main,
                                                              const __grid_constant__ CUtensorMap tx_tail,
                                                              const __grid_constant__ CUtensorMap tw_main,
                                                              const __grid_constant__ CUtensorMap tw_tail,
                                                              const ConvTcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* wsm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = a.S, Nb = a.Nb, nmain = a.Cin / 64, tail = a.Cin % 64, nblk = nmain + (tail ? 1 : 0);
  uint8_t* slabs = wsm + conv_weight_bytes(a.Cin, Nb);
  const uint32_t slab_bytes = (uint32_t)conv_slab_bytes(a.Cin), wtap_bytes = (uint32_t)conv_wtap_bytes(a.Cin, Nb);
  // per channel block: byte offset in a slab / a tap's weights
  const uint32_t sblk = (uint32_t)round_1k((size_t)kHalo * 128), wblk = (uint32_t)round_1k((size_t)Nb * 128);
  __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], wbar;
  __shared__ uint32_t tmem_slot;
  __shared__ float bias_s[kMaxCout];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int w_prod = 4 * (Nb / 16), w_mma = w_prod + 1;
  const int co0 = blockIdx.y * Nb;
  const int nseg = (a.W + kM - 1) / kM, ntiles = a.rows * nseg;
  // with row pairs (rows even, row0 = 0) every range starts and ends at an even row
  constexpr int kUnit = epi_row_pairs(kEpi) ? 2 : 1;
  const int lo = kUnit * (int)((int64_t)(ntiles / kUnit) * blockIdx.x / gridDim.x);
  const int hi = kUnit * (int)((int64_t)(ntiles / kUnit) * (blockIdx.x + 1) / gridDim.x);
  const uint32_t ncols = conv_acc_cols(Nb);

  if (warp == w_mma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(2 * ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < S; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], (uint32_t)w_prod);    // one arrival per epilogue warp
    }
    mbar_init(&wbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int c = tid; c < Nb; c += (int)blockDim.x) bias_s[c] = a.bias ? a.bias[co0 + c] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  bool ok = true;

  if (warp == w_prod) {
    // producer: the weights once, then the slabs of every run in order
    if (lane == 0) {
      // the weights are no output of the kernel before
      mbar_expect_tx(&wbar, 9u * (uint32_t)Nb * 2u * (uint32_t)a.Cin);
      for (int t = 0; t < 9; t++)
        for (int bk = 0; bk < nblk; bk++)
          tma_load_3d(wsm + (size_t)t * wtap_bytes + (size_t)bk * wblk, bk < nmain ? &tw_main : &tw_tail, 64 * bk, co0, t,
                      &wbar);
      pdl_wait();
      pdl_launch();
      RingPos q{0u, 0u};
      TileRun r;
      for (int u = lo; ok && next_run(u, hi, a.rows, r);) {
        const int x0 = r.seg * kM;
        for (int k = 0; k < r.len + 2 && ok; k++, q = q.next((uint32_t)S)) {
          if (!(ok = mbar_wait(&empty[q.slot], q.phase ^ 1u))) break;
          mbar_expect_tx(&full[q.slot], (uint32_t)kHalo * 2u * (uint32_t)a.Cin);
          uint8_t* dst = slabs + (size_t)q.slot * slab_bytes;
          for (int bk = 0; bk < nblk; bk++)
            tma_load_3d(dst + (size_t)bk * sblk, bk < nmain ? &tx_main : &tx_tail, 64 * bk, x0 - 1, a.row0 + r.y0 - 1 + k,
                        &full[q.slot]);
        }
      }
    }
  } else if (warp == w_mma) {
    // MMA issuer: output row i of a run accumulates 9 Cin / 16 MMAs over the
    // slabs i, i + 1, i + 2 of the run into accumulator buffer (tile count % 2)
    {   // all 32 lanes: warp-uniform descriptors, elected issue
      const uint32_t idesc = mma_idesc(kM, Nb);
      const uint32_t hi_main = desc_hi(128u), hi_tail = desc_hi(2u * (uint32_t)tail);
      const uint32_t w_lo = desc_lo(smem_u32(wsm)), s_lo = desc_lo(smem_u32(slabs));
      const uint32_t wtap16 = wtap_bytes >> 4, slab16 = slab_bytes >> 4, sblk16 = sblk >> 4, wblk16 = wblk >> 4;
      const uint32_t tail16 = (2u * (uint32_t)tail) >> 4;      // the tail's row pitch, in 16-byte units
      ok = mbar_wait_warp(&wbar, 0);
      uint32_t tc = 0;
      RingPos q{0u, 0u};    // ring position of the next slab
      TileRun r;
      for (int u = lo; ok && next_run(u, hi, a.rows, r);) {
        RingPos q0 = q, q1 = q.next((uint32_t)S);    // slabs i and i + 1 of the run
        for (int i = 0; i < r.len && ok; i++, tc++) {
          const uint32_t b = tc & 1u;
          const RingPos q2 = q1.next((uint32_t)S);
          if (!(ok = mbar_wait_warp(&acc_empty[b], ((tc >> 1) & 1u) ^ 1u))) break;
          if (i == 0) ok = mbar_wait_warp(&full[q0.slot], q0.phase) && mbar_wait_warp(&full[q1.slot], q1.phase);
          if (!(ok = ok && mbar_wait_warp(&full[q2.slot], q2.phase))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d = tmem + b * ncols;
          uint32_t acc = 0;
#pragma unroll
          for (int dy = 0; dy < 3; dy++) {
            const uint32_t slot = dy == 0 ? q0.slot : dy == 1 ? q1.slot : q2.slot;
            const uint32_t xs = s_lo + slot * slab16, ws = w_lo + (uint32_t)(3 * dy) * wtap16;
            for (int bk = 0; bk < nmain; bk++) {
              const uint32_t xb = xs + (uint32_t)bk * sblk16, wb = ws + (uint32_t)bk * wblk16;
#pragma unroll
              for (int c = 0; c < 4; c++)
#pragma unroll
                for (int dx = 0; dx < 3; dx++) {
                  mma_bf16_elect(d, desc_pack(xb + 8u * dx + 2u * c, hi_main), desc_pack(wb + dx * wtap16 + 2u * c, hi_main),
                           idesc, acc);
                  acc = 1;
                }
            }
            if (tail) {
              const uint32_t xb = xs + (uint32_t)nmain * sblk16, wb = ws + (uint32_t)nmain * wblk16;
              for (uint32_t c = 0; c < tail16 / 2; c++)
#pragma unroll
                for (int dx = 0; dx < 3; dx++) {
                  mma_bf16_elect(d, desc_pack(xb + tail16 * dx + 2u * c, hi_tail), desc_pack(wb + dx * wtap16 + 2u * c, hi_tail),
                           idesc, acc);
                  acc = 1;
                }
            }
          }
          mma_commit_elect(&acc_full[b]);
          mma_commit_elect(&empty[q0.slot]);    // slab i is read by no later row
          q0 = q1;
          q1 = q2;
        }
        if (!ok) break;
        // the run's last two slabs
        mma_commit_elect(&empty[q0.slot]);
        mma_commit_elect(&empty[q1.slot]);
        q = q1.next((uint32_t)S);
      }
    }
  } else {
    // epilogue: warp w drains TMEM lanes (pixels) 32 qw .. 32 qw + 31, qw =
    // w % 4, of output channels c0 .. c0 + 15, c0 = 16 (w / 4), of each tile
    pdl_wait();
    pdl_launch();
    const int qw = warp & 3, c0 = 16 * (warp >> 2);
    constexpr bool kSkipIn = kEpi == kEpiSkip || kEpi == kEpiSkipUp;
    uint32_t tc = 0;
    [[maybe_unused]] uint4 plo, phi;      // kEpiPool: the even row's output of this pixel
    [[maybe_unused]] float prow[4][4];    // kEpiDown: the even row's gradient (quad_transpose)
    // sums of dy, channels 4 (lane % 4) .. + 3: of a few pixels, of all of this
    // CTA's tiles, and what the latter's roundings lost
    [[maybe_unused]] float part[4] = {0.f, 0.f, 0.f, 0.f}, bsum[4] = {0.f, 0.f, 0.f, 0.f}, lost[4] = {0.f, 0.f, 0.f, 0.f};
    [[maybe_unused]] const int c4 = co0 + c0 + 4 * (lane & 3);
    // dy of four channels at offset q where the ReLU output m passed
    [[maybe_unused]] auto emit = [&](float* g, uint2 m, size_t q) {
      const float2 m0 = unpack_bf16(m.x), m1 = unpack_bf16(m.y);
      g[0] = m0.x > 0.f ? g[0] : 0.f;
      g[1] = m0.y > 0.f ? g[1] : 0.f;
      g[2] = m1.x > 0.f ? g[2] : 0.f;
      g[3] = m1.y > 0.f ? g[3] : 0.f;
#pragma unroll
      for (int e = 0; e < 4; e++) part[e] += g[e];
      store4(a.dy32 + q, g);
      *reinterpret_cast<uint2*>(a.dy16 + q) = make_uint2(pack_bf16(g[0], g[1]), pack_bf16(g[2], g[3]));
    };
    // Neighbouring gradients are often the same value, whose running sum rounds
    // the same way in every lane; so the long sum keeps its rounding errors
    // (two-sum, Knuth).  Bias gradients of the 64 -> 32 layer, error against 64
    // bits in units of 2^-24 of the summed magnitudes (rms over the channels):
    // 800 x 528 1.05 -> 0.51, 1600 x 1056 1.57 -> 0.52; the step takes 695 us as before.
    [[maybe_unused]] auto fold = [&] {
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const float s = bsum[e] + part[e], d = s - bsum[e];
        lost[e] += (bsum[e] - (s - d)) + (part[e] - d);
        bsum[e] = s;
        part[e] = 0.f;
      }
    };
    TileRun r;
    for (int u = lo; ok && next_run(u, hi, a.rows, r);) {
      for (int i = 0; i < r.len && ok; i++, tc++) {
        const uint32_t b = tc & 1u;
        const int y = a.row0 + r.y0 + i, px = r.seg * kM + qw * 32 + lane;
        const bool in = px < a.W;
        const size_t o = ((size_t)y * a.W + (in ? px : 0)) * a.Cout + co0 + c0;
        // this lane's skip values, fetched while the tile's MMAs run
        [[maybe_unused]] uint4 sk0, sk1;
        if constexpr (kSkipIn) {
          sk0 = __ldg(reinterpret_cast<const uint4*>(a.skip + o));
          sk1 = __ldg(reinterpret_cast<const uint4*>(a.skip + o) + 1);
        }
        // the masks of the quad's four pixels (kEpiDown: of its two pixel pairs, on odd rows)
        const int p0 = r.seg * kM + qw * 32 + (lane & ~3);
        [[maybe_unused]] uint2 mk[4];
        if constexpr (kEpi == kEpiMask) {
#pragma unroll
          for (int k = 0; k < 4; k++)
            mk[k] = __ldg(reinterpret_cast<const uint2*>(a.mask + ((size_t)y * a.W + min(p0 + k, a.W - 1)) * a.Cout + c4));
        }
        if constexpr (kEpi == kEpiDown) {
          if (y & 1) {
#pragma unroll
            for (int k = 0; k < 2; k++)
              mk[k] = __ldg(reinterpret_cast<const uint2*>(
                  a.mask + ((size_t)(y >> 1) * (a.W >> 1) + min((p0 >> 1) + k, (a.W >> 1) - 1)) * a.Cout + c4));
          }
        }
        if (!(ok = mbar_wait(&acc_full[b], (tc >> 1) & 1u, 64))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t v[16];
        tmem_ld16(tmem + b * ncols + ((uint32_t)(qw * 32) << 16) + (uint32_t)c0, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        // buffer b may be overwritten by the next tile's MMAs once every
        // epilogue warp has its values
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[b]);
        float f[16];
#pragma unroll
        for (int e = 0; e < 16; e++) {
          const float val = __uint_as_float(v[e]) + bias_s[c0 + e];
          f[e] = a.relu ? fmaxf(val, 0.f) : val;
        }
        if constexpr (kEpi == kEpiPlain || epi_gradient(kEpi)) {
          float t[4][4];
#pragma unroll
          for (int e = 0; e < 16; e++) t[e >> 2][e & 3] = f[e];
          quad_transpose(t, lane);
          if constexpr (kEpi == kEpiPlain || kEpi == kEpiMask) {
#pragma unroll
            for (int k = 0; k < 4; k++) {
              if (p0 + k >= a.W) continue;
              const size_t q = ((size_t)y * a.W + p0 + k) * a.Cout + c4;
              store4((kEpi == kEpiPlain ? a.y32 : a.raw32) + q, t[k]);
              if constexpr (kEpi == kEpiMask) emit(t[k], mk[k], q);
            }
          } else if constexpr (kEpi == kEpiDown) {
            if (y & 1) {
#pragma unroll
              for (int k = 0; k < 2; k++) {
                if (p0 + 2 * k >= a.W) continue;      // W is even
                float g[4];
#pragma unroll
                for (int e = 0; e < 4; e++)
                  g[e] = ((prow[2 * k][e] + prow[2 * k + 1][e]) + t[2 * k][e]) + t[2 * k + 1][e];
                const size_t q = ((size_t)(y >> 1) * (a.W >> 1) + (p0 >> 1) + k) * a.Cout + c4;
                if (a.raw32) store4(a.raw32 + q, g);
                emit(g, mk[k], q);
              }
            } else {
#pragma unroll
              for (int e = 0; e < 16; e++) prow[e >> 2][e & 3] = t[e >> 2][e & 3];
            }
          } else {
#pragma unroll
            for (int k = 0; k < 4; k++) {
              if (p0 + k >= a.W) continue;
#pragma unroll
              for (int d = 0; d < 4; d++) {
                const size_t q = ((size_t)(2 * y + (d >> 1)) * (2 * a.W) + 2 * (p0 + k) + (d & 1)) * a.Cout + c4;
                const uint2 m = __ldg(reinterpret_cast<const uint2*>(a.mask + q));
                const float4 u = __ldg(reinterpret_cast<const float4*>(a.add32 + q));
                float g[4] = {u.x + 0.25f * t[k][0], u.y + 0.25f * t[k][1], u.z + 0.25f * t[k][2], u.w + 0.25f * t[k][3]};
                emit(g, m, q);
              }
              fold();
            }
          }
          if constexpr (epi_gradient(kEpi) && kEpi != kEpiSpread) fold();
          continue;
        }
        // Lanes past the row's end compute on their TMEM rows and take part in
        // the exchanges; they store only their partner's pixel.
        const bool odd = (lane & 1) != 0;
        uint4 h0 = pack8(f), h1 = pack8(f + 8);
        if constexpr (kEpi == kEpiPool) {
          // W and H are even: both pixels and both rows of a pair are inside.
          // The even lane averages channels 0-7, the odd lane 8-15.
          if (in) {
            reinterpret_cast<uint4*>(a.y16 + o)[0] = h0;
            reinterpret_cast<uint4*>(a.y16 + o)[1] = h1;
          }
          if (y & 1) {
            const uint4 r0 = shfl_xor1(odd ? plo : phi), r1 = shfl_xor1(odd ? h0 : h1);
            float x00[8], x01[8], x10[8], x11[8], m[8];
            unpack8(odd ? r0 : plo, x00);
            unpack8(odd ? phi : r0, x01);
            unpack8(odd ? r1 : h0, x10);
            unpack8(odd ? h1 : r1, x11);
#pragma unroll
            for (int e = 0; e < 8; e++) m[e] = 0.25f * (((x00[e] + x01[e]) + x10[e]) + x11[e]);
            if (in)
              *reinterpret_cast<uint4*>(a.res16 + ((size_t)(y >> 1) * (a.W >> 1) + (px >> 1)) * a.Cout + co0 + c0 +
                                        (odd ? 8 : 0)) = pack8(m);
          } else {
            plo = h0;
            phi = h1;
          }
        } else {
          // the lane's half (lo: even lanes, hi: odd lanes) of the sectors of the
          // pair's two pixels
          const bool in_partner = __shfl_xor_sync(0xffffffffu, in ? 1 : 0, 1) != 0;
          const bool in_a = odd ? in_partner : in, in_b = odd ? in : in_partner;
          const int xa = px & ~1, half = odd ? 8 : 0;
          const size_t oa = ((size_t)y * a.W + xa) * a.Cout + co0 + c0 + half;
          SectorPair q = pair_exchange(h0, h1, odd);
          if constexpr (kSkipIn) {
            if (in_a) *reinterpret_cast<uint4*>(a.r16 + oa) = q.a;
            if (in_b) *reinterpret_cast<uint4*>(a.r16 + oa + a.Cout) = q.b;
            float s[16];
            unpack8(h0, f);
            unpack8(h1, f + 8);
            unpack8(sk0, s);
            unpack8(sk1, s + 8);
#pragma unroll
            for (int e = 0; e < 16; e++) f[e] = f[e] + s[e];
            h0 = pack8(f);
            h1 = pack8(f + 8);
            q = pair_exchange(h0, h1, odd);
          }
          if constexpr (kEpi == kEpiUp || kEpi == kEpiSkip) {
            if (in_a) *reinterpret_cast<uint4*>(a.y16 + oa) = q.a;
            if (in_b) *reinterpret_cast<uint4*>(a.y16 + oa + a.Cout) = q.b;
          }
          if constexpr (kEpi == kEpiUp || kEpi == kEpiSkipUp) {
#pragma unroll
            for (int dy = 0; dy < 2; dy++) {
              __nv_bfloat16* d = a.res16 + ((size_t)(2 * y + dy) * (2 * a.W) + 2 * xa) * a.Cout + co0 + c0 + half;
              if (in_a) {
                *reinterpret_cast<uint4*>(d) = q.a;
                *reinterpret_cast<uint4*>(d + a.Cout) = q.a;
              }
              if (in_b) {
                *reinterpret_cast<uint4*>(d + 2 * a.Cout) = q.b;
                *reinterpret_cast<uint4*>(d + 3 * a.Cout) = q.b;
              }
            }
          }
        }
      }
    }
    if constexpr (epi_gradient(kEpi)) {
#pragma unroll
      for (int e = 0; e < 4; e++)
        if (isfinite(lost[e])) bsum[e] += lost[e];      // a sum that overflowed stays as it is
#pragma unroll
      for (int e = 0; e < 4; e++)
#pragma unroll
        for (int m = 16; m >= 4; m >>= 1) bsum[e] += __shfl_xor_sync(0xffffffffu, bsum[e], m);
      if (lane < 4) store4(a.bpart + (size_t)(4 * blockIdx.x + qw) * a.Cout + c4, bsum);
    }
  }
  if (!ok && (lane == 0)) atomicOr(a.status, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == w_mma) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * ncols));
  }
}

// Weight gradient of a 3x3 convolution on the tensor cores:
// dW (t, co, ci) = sum over pixels p of dy (p, co) x (p + off(t), ci), as
// GEMMs with K = pixels, read straight from the pixel-major BF16 tensors
// dy (H, W, Cout) and x (H, W, Cin): both operands are MN-major (the channel
// is the contiguous dimension, a pixel is a row of the shared-memory tile).
// Substituting y' = y + dy, dW (dy, dx) = sum over (y', x) of
// dy (y' - dy, x, co) x (y', x + dx, ci): a K step is 64 pixels x .. x + 63
// of one row y'.  B is one box of x at row y', pixels x - 1 .. x + 64, read
// by three MMAs whose start rows differ by one pixel (dx = -1, 0, 1: one
// accumulator each; the swizzle follows the shared-memory address bits, so
// a start moved by whole rows reads what the TMA wrote); A the box(es) of
// dy at rows y' - dy.  Rows and pixels outside the image read zeros.
// With Cout <= 32 the three vertical taps share one MMA: A's rows 32 g + co
// hold dy at row y' - (g - 1), so one CTA computes all nine taps from one
// load of each operand per step (rows past Cout in each group are left over
// and ignored); otherwise blockIdx.y is the vertical tap and A is one or two
// boxes of 64 channels.  blockIdx.x is a band of rows y'.  Per step 4 x 3
// MMAs of 16 pixels.  The band's sums are added into dw (FP32) by the
// epilogue warps with vector atomics.  blockIdx.x takes an equal share of
// the (row, 64-pixel chunk) steps, in row order.
//
// Channel boxes: Cout (stacked) or 64 channels of dy, min(Cin, 64) channels
// of x, rows of 2 x channels bytes with the matching swizzle; a box of dy is
// 64 pixel rows, one of x 66 (72 reserved, a whole number of swizzle
// atoms); boxes along the channels lie one box apart (the MN stride of the
// descriptor), groups of 8 pixels one 8-row group apart.
constexpr int kWgMaxStages = 8;
constexpr size_t kWgA = 128 * 128;                        // A: 128 channel rows x 64 pixels
__host__ __device__ constexpr int wgrad_xbox(int cin) { return cin < 64 ? cin : 64; }
constexpr int kWgXRows = 72;                              // x box: 66 pixels, 72 rows reserved
__host__ __device__ constexpr size_t wgrad_xbox_bytes(int cin) { return (size_t)kWgXRows * 2 * wgrad_xbox(cin); }
__host__ __device__ constexpr size_t wgrad_stage_bytes(int cin) {
  return (kWgA + (size_t)((cin + 63) / 64) * wgrad_xbox_bytes(cin) + 1023) & ~size_t(1023);
}
__host__ __device__ constexpr uint32_t wgrad_acc_stride(int cin) { return cin <= 32 ? 32u : (uint32_t)cin; }
__host__ __device__ constexpr uint32_t wgrad_tmem_cols(int cin) {
  return 3 * wgrad_acc_stride(cin) <= 128 ? 128u : 3 * wgrad_acc_stride(cin) <= 256 ? 256u : 512u;
}
constexpr size_t kWgSmemCap = 200 * 1024;
constexpr size_t kWgSlack = 1024;               // alignment of the ring
__host__ __device__ constexpr int wgrad_stages(int cin) {
  return (int)(kWgSmemCap / wgrad_stage_bytes(cin)) < kWgMaxStages ? (int)(kWgSmemCap / wgrad_stage_bytes(cin))
                                                                      : kWgMaxStages;
}
struct WgradTcArgs {
  float* dw;                 // (9, Cout, Cin), accumulated into
  unsigned int* status;      // bit 0: a barrier wait gave up
  int H, W, Cin, Cout;
  int steps_per_cta;         // (row, 64-pixel chunk) steps of one CTA
  int stacked;               // Cout <= 32: the three vertical taps in one MMA
  int S;                     // stages
};
// the low descriptor word of an MN-major operand: start address and the
// stride between boxes along the channels
__device__ __forceinline__ uint32_t desc_lo_mn(uint32_t addr, uint32_t box_bytes) {
  return ((addr >> 4) & 0x3FFFu) | (((box_bytes >> 4) & 0x3FFFu) << 16);
}

__global__ void __launch_bounds__(kThreads) wgrad3x3_tc_kernel(const __grid_constant__ CUtensorMap tdy,
                                                               const __grid_constant__ CUtensorMap tx,
                                                               const WgradTcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[kWgMaxStages], empty[kWgMaxStages], acc_full;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = a.S;
  const uint32_t stage_bytes = (uint32_t)wgrad_stage_bytes(a.Cin), xb_bytes = (uint32_t)wgrad_xbox_bytes(a.Cin);
  const int cba = a.stacked ? a.Cout : 64, cbb = wgrad_xbox(a.Cin);     // channels per box
  const int dy_cta = a.stacked ? 0 : (int)blockIdx.y - 1;               // this CTA's vertical tap (not stacked)
  const int nseg = (a.W + 63) / 64, k0 = blockIdx.x * a.steps_per_cta;
  const int nk = max(0, min(a.H * nseg, k0 + a.steps_per_cta) - k0);
  const uint32_t stride = wgrad_acc_stride(a.Cin), ncols = wgrad_tmem_cols(a.Cin);

  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < S; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  bool ok = true;

  if (warp == 4) {
    if (lane == 0) {
      const int na = a.stacked ? 3 : (a.Cout + 63) / 64, nbx = (a.Cin + 63) / 64;
      const uint32_t bytes = (uint32_t)na * 128u * (uint32_t)cba + (uint32_t)nbx * 132u * (uint32_t)cbb;
      pdl_wait();
      pdl_launch();
      RingPos q{0u, 0u};
      for (int k = 0; k < nk && ok; k++, q = q.next((uint32_t)S)) {
        if (!(ok = mbar_wait(&empty[q.slot], q.phase ^ 1u))) break;
        const int y = (k0 + k) / nseg, x0 = ((k0 + k) % nseg) * 64;
        uint8_t* st = ring + (size_t)q.slot * stage_bytes;
        mbar_expect_tx(&full[q.slot], bytes);
        if (a.stacked) {   // vertical tap g - 1 at A rows 32 g ..
          for (int g = 0; g < 3; g++) tma_load_3d(st + (size_t)g * 4096, &tdy, 0, x0, y - (g - 1), &full[q.slot]);
        } else {
          for (int b = 0; b < na; b++) tma_load_3d(st + (size_t)b * 8192, &tdy, 64 * b, x0, y - dy_cta, &full[q.slot]);
        }
        for (int b = 0; b < nbx; b++) tma_load_3d(st + kWgA + (size_t)b * xb_bytes, &tx, 64 * b, x0 - 1, y, &full[q.slot]);
      }
    }
  } else if (warp == 5) {
    {   // all 32 lanes: warp-uniform descriptors, elected issue
      const uint32_t idesc = mma_idesc(kM, a.Cin) | (1u << 15) | (1u << 16);   // A and B MN-major
      const uint32_t a_hi = desc_hi(2u * (uint32_t)cba), b_hi = desc_hi(2u * (uint32_t)cbb);
      const uint32_t a_lo = desc_lo_mn(smem_u32(ring), 128u * (uint32_t)cba);
      const uint32_t b_lo = desc_lo_mn(smem_u32(ring) + (uint32_t)kWgA, xb_bytes);
      // one pixel = one row of 2 x channels bytes, in 16-byte units
      const uint32_t a_row = (uint32_t)cba >> 3, b_row = (uint32_t)cbb >> 3;
      const uint32_t stage16 = stage_bytes >> 4;
      RingPos q{0u, 0u};
      for (int k = 0; k < nk && ok; k++, q = q.next((uint32_t)S)) {
        if (!(ok = mbar_wait_warp(&full[q.slot], q.phase))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
          for (int dx = 0; dx < 3; dx++)
            mma_bf16_elect(tmem + (uint32_t)dx * stride, desc_pack(a_lo + q.slot * stage16 + 16u * a_row * c, a_hi),
                     desc_pack(b_lo + q.slot * stage16 + (16u * c + (uint32_t)dx) * b_row, b_hi), idesc,
                     (k > 0 || c > 0) ? 1u : 0u);
        mma_commit_elect(&empty[q.slot]);
      }
      if (ok) mma_commit_elect(&acc_full);
    }
  } else if (nk > 0) {
    // epilogue: TMEM lane 32 w + l is A's row: (vertical tap w - 1, output
    // channel l) when stacked, else output channel 32 w + l
    const int g = a.stacked ? warp : dy_cta + 1, co = a.stacked ? lane : warp * 32 + lane;
    const bool rows_used = a.stacked ? warp < 3 : warp * 32 < a.Cout;
    pdl_wait();
    if (rows_used && (ok = mbar_wait(&acc_full, 0, 64))) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int dx = 0; dx < 3; dx++) {
        float* d = a.dw + ((size_t)(3 * g + dx) * a.Cout + co) * a.Cin;
        for (int c0 = 0; c0 < a.Cin; c0 += 16) {
          uint32_t v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)dx * stride + (uint32_t)c0, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (co >= a.Cout) continue;
#pragma unroll
          for (int e = 0; e < 4; e++)
            atomicAdd(reinterpret_cast<float4*>(d + c0) + e,
                      make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]), __uint_as_float(v[4 * e + 2]),
                                  __uint_as_float(v[4 * e + 3])));
        }
      }
    }
  }
  if (!ok && lane == 0) atomicOr(a.status, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 5) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
  }
}

// Launch plan of conv3x3_tc_kernel for one layer: the largest channel block
// Nb (a multiple of 16 dividing Cout) whose weights and four slabs fit in
// 220 KB of shared memory; then as many slab stages (at most kMaxStages) as
// fit in 110 KB, so that two CTAs share an SM, or else in 220 KB; and the
// CTAs that fit on one SM by shared memory and by tensor memory (512
// columns, two accumulators per CTA).
struct ConvPlan {
  int Nb, S, ctas_per_sm;
  size_t smem;
};
constexpr size_t kConvSmemCap = 220 * 1024;   // dynamic; the kernel's static shared memory comes on top
inline ConvPlan conv_plan(int cin, int cout) {
  const size_t cap = kConvSmemCap, half = kConvSmemCap / 2, slab = conv_slab_bytes(cin);
  int nb = 16;
  for (int d = 1; d <= cout / 16; d++) {
    if (cout % d || (cout / d) % 16 || cout / d > kConvMaxNb) continue;
    if (conv_smem_bytes(cin, cout / d, 4) <= cap) {
      nb = cout / d;
      break;
    }
  }
  const size_t budget = conv_smem_bytes(cin, nb, 4) <= half ? half : cap;
  int s = (int)((budget - conv_smem_bytes(cin, nb, 0)) / slab);
  s = s < kMaxStages ? s : kMaxStages;
  ConvPlan p{nb, s, 1, conv_smem_bytes(cin, nb, s)};
  const int by_tmem = 512 / (int)(2 * conv_acc_cols(nb)), by_smem = (int)((228 * 1024) / (p.smem + 2048));   // + reserved and static
  p.ctas_per_sm = by_tmem < by_smem ? by_tmem : by_smem;
  if (p.ctas_per_sm < 1) p.ctas_per_sm = 1;
  return p;
}

// CTAs of a convolution along its tiles: per channel block (nblk of them) as
// many as are resident at once, at most one per tile (or pair of tiles).  The
// gradients' CTAs write four rows of bias partial sums each and have kBiasRows
// of them; with fewer CTAs each takes more tiles.
constexpr int kBiasRows = 2048;
__host__ constexpr int conv_grid(int ntiles, int n_sm, int ctas_per_sm, int nblk, bool gradient) {
  int g = n_sm * ctas_per_sm / nblk;
  if (gradient && g > kBiasRows / 4) g = kBiasRows / 4;
  if (g > ntiles) g = ntiles;
  return g < 1 ? 1 : g;
}

}  // namespace tc
}  // namespace amh
