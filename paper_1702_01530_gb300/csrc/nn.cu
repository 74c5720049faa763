// Retrace-probability network: 4 layers of 3x3 convolutions
// (10 -> 32 -> 32 -> 32 -> 1, zero padding 1, ReLU, sigmoid), BF16 operands
// (E4M3 for layers 2-4 in FP8 inference) and FP32 accumulation on the
// 5th-generation tensor cores (sm_103a).
//
// Forward pass: k_net_fused, all four layers in one kernel; activations are
// written only where training or calibration asks for them.
//
// Backward pass: data gradients are convolutions with the 3x3 taps flipped and
// Cin/Cout swapped (k_bwd_fused, all three in one kernel); weight gradients are
// contractions over the pixels (k_wgrad); BCE on the sigmoid output; Adam on FP32
// master weights.
//
// Convolution as implicit GEMM on tcgen05: 128 pixels of a row are the M of an
// MMA. A row's input sits in shared memory as 16-byte channel chunks ordered
// [chunk][pixel], so kernel column dx is the same K-major, non-swizzled operand
// (8-row core matrices 128 B apart, SBO; chunk planes apart by LBO) moved by dx
// pixels. An MMA of N = Cout costs the tensor core as much as one of N = 64 (about
// 45 cycles on GB300, measured; N = 96 about 56, N = 256 about 128, the full rate),
// so the three vertical taps of a kernel column are stacked along N; weights are
// packed in this stacked core-matrix layout, [dx][chunk][3 Cout][chunk elements].
// Every mbarrier wait has an iteration bound; on expiry the kernel sets the error
// word, waits (bounded) for what it has in flight and frees its TMEM.
//
// Layouts in HBM: the network input features are interleaved [P][16]; the BCE
// gradient is one chunk per pixel [P][8]; the 32-channel activations and data
// gradients are chunk-planar [4][P][8] BF16 (plane k holds one 16-byte chunk of
// channels of every pixel), so a halo row of one chunk is one contiguous run
// and each warp's epilogue store a contiguous 512-byte run per plane.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstdlib>

#include "rt_internal.cuh"

namespace rt {
namespace nn {

constexpr uint32_t kSmemBudget = 220u * 1024u;
constexpr uint32_t kWaitBound = 1u << 26;

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// instruction descriptor: kind::f16, D = F32, A = B = BF16, both K-major
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// Low and high words of a no-swizzle descriptor. A descriptor of the same
// operand at byte offset k from its base is the base's low word plus k >> 4
// (the start-address field cannot carry: shared addresses stay below 2^18),
// so the unrolled MMA loops below pay one integer add per descriptor.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo) {
  return ((saddr >> 4) & 0x3FFFu) | (((lbo >> 4) & 0x3FFFu) << 16);
}
__host__ __device__ constexpr uint32_t desc_hi(uint32_t sbo) {
  return ((sbo >> 4) & 0x3FFFu) | (1u << 14);   // bit 46 of the descriptor: tcgen05 version
}
__device__ __forceinline__ uint64_t desc_join(uint32_t lo, uint32_t hi) {
  return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase) {
  const uint32_t a = smem_u32(bar);
#pragma unroll 1
  for (uint32_t i = 0; i < kWaitBound; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// true in one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// waits for two barriers' phases; with OVERLAP their first polls overlap
template <bool OVERLAP>
__device__ __forceinline__ bool mbar_wait2(uint64_t* bar0, uint32_t phase0, uint64_t* bar1, uint32_t phase1) {
  if (!OVERLAP) return mbar_wait(bar0, phase0) && mbar_wait(bar1, phase1);
  uint32_t d0, d1;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%2], %3;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 q, [%4], %5;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "selp.u32 %1, 1, 0, q;\n\t}"
      : "=r"(d0), "=r"(d1)
      : "r"(smem_u32(bar0)), "r"(phase0), "r"(smem_u32(bar1)), "r"(phase1)
      : "memory");
  return (d0 || mbar_wait(bar0, phase0)) && (d1 || mbar_wait(bar1, phase1));
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// instruction descriptor: kind::f8f6f4, D = F32, A = B = E4M3 (format 0), both K-major
__host__ __device__ constexpr uint32_t make_idesc_e4m3(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_e4m3(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// 4-D tiled TMA load of one box into shared memory, completion counted in
// bytes on the mbarrier; out-of-range elements are written as zeros
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}

// 3-D tiled TMA load (the same)
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}

// 5-D tiled TMA load (the same, with an image index among the coordinates)
__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, int c4, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
      "r"(smem_u32(bar))
      : "memory");
}

// 16 consecutive TMEM columns of this warp's 32 lanes, without the wait:
// several loads share one tcgen05.wait::ld
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t r[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// A pixel's ReLU mask of 32 channels in one word: pair j of channels (2 j, 2 j + 1)
// has bits j and 16 + j. Adds pair j of BF16 values.
__device__ __forceinline__ uint32_t mask_bits(uint32_t word, uint32_t pair, int j) {
  const __nv_bfloat162 zero = __float2bfloat162_rn(0.f);
  return word | (__hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&pair), zero) & (0x00010001u << j));
}
// BF16 of (a, b), each zero where its bit of pair j is not set
__device__ __forceinline__ uint32_t masked_pair(uint32_t word, int j, uint32_t a, uint32_t b) {
  uint32_t m;                          // bits 15 and 31 after the shift: signs of bytes 1 and 3, over their halves
  asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(m) : "r"(word << (15 - j)));
  return pack_bf16(__uint_as_float(a), __uint_as_float(b)) & m;
}

// (a0, a1) += (b0, b1) in one instruction, each sum rounded to nearest
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1) {
  asm("{\n\t.reg .b64 x, y;\n\t"
      "mov.b64 x, {%0, %1};\n\t"
      "mov.b64 y, {%2, %3};\n\t"
      "add.rn.f32x2 x, x, y;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}

// (a0, a1) = fma((a0, a1), (m0, m1), (b0, b1))
__device__ __forceinline__ void fma2(float& a0, float& a1, float m0, float m1, float b0, float b1) {
  asm("{\n\t.reg .b64 x, m, y;\n\t"
      "mov.b64 x, {%0, %1};\n\t"
      "mov.b64 m, {%2, %3};\n\t"
      "mov.b64 y, {%4, %5};\n\t"
      "fma.rn.f32x2 x, x, m, y;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(m0), "f"(m1), "f"(b0), "f"(b1));
}
// max(x, 0) of two BF16 (0 for a NaN, as fmaxf gives)
__device__ __forceinline__ uint32_t relu_bf16(uint32_t x) {
  uint32_t y;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(y) : "r"(x), "r"(0u));
  return y;
}

// e4m3(max(x, 0)) of four values, round to nearest even, saturating (a NaN
// stays a NaN)
__device__ __forceinline__ uint32_t relu_e4m3x4(float x0, float x1, float x2, float x3) {
  uint32_t d;
  asm("{\n\t.reg .b16 lo, hi;\n\t"
      "cvt.rn.satfinite.relu.e4m3x2.f32 lo, %2, %1;\n\t"
      "cvt.rn.satfinite.relu.e4m3x2.f32 hi, %4, %3;\n\t"
      "mov.b32 %0, {lo, hi};\n\t}"
      : "=r"(d)
      : "f"(x0), "f"(x1), "f"(x2), "f"(x3));
  return d;
}

// zeroes 16 consecutive TMEM columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
          taddr),
      "r"(0u)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------ fused forward
// The whole network in one kernel: a strip of 122 output pixels streams down
// the image, one input row at a time, through the four layers; the
// activations between them never leave the SM (32 bytes of features in and 4
// of probability out per pixel, against 420 when each layer wrote its output).
//
// Streaming and stacked taps: input row h of a layer adds tap dy = 2 to output
// row h - 2, dy = 1 to h - 1 and dy = 0 to h. The three rows' accumulators are
// three 32-column TMEM slots, row r in slot r % 3, so one MMA of N = 96 per
// kernel column and K step serves all three vertical taps, every input row is
// read once, and no product falls outside the tile. Which tap a slot takes
// rotates with the row: the weights of a (dx, chunk) lie in shared memory as
// five blocks [dy 2 | 1 | 0 | 2 | 1], and the window of three blocks that
// starts at block 2 - row % 3 has the right order. After input row h the epilogue
// reads the finished row h - 2 and zeroes its slot, which becomes row h + 1's.
// An MMA of N = 96 takes ~56 cycles, one of N <= 32 ~45 (measured): a row of
// 122 pixels takes 3 (layer 1) + 6 + 6 (layers 2, 3, BF16) MMAs of N = 96.
// Layer 4 (one output channel) puts its 9 taps along N = 16 instead: 2 MMAs a
// row, no shift of A; its epilogue adds the three vertical taps of each kernel
// column in registers while the rows pass and exchanges two values with the
// neighbouring pixels: 930 cycles a row in all (BF16), 548 (E4M3 layers 2-4).
//
// Pixels: lane m of layer k's accumulators (k = 0 .. 3) is the image column
// x_strip - 3 + min(k, 2) + m; each layer's output row is stored at pixel m of
// the next one's input row (16-byte channel chunks [chunk][130 pixels]), so
// kernel column dx is the A operand moved by dx pixels. Lanes past the strip
// (126, 127 of layer 2, ...) hold what they hold and are never used. Outputs
// outside the image are stored as zeros, the next layer's padding.
//
// Roles: per layer one thread issues the MMAs (layer 1's also loads the feature
// rows, kFuF - 1 ahead) and one warpgroup runs the epilogue, so rows of all
// four layers are in flight. One thread for the MMAs of all layers spent more
// time waiting for their barriers in turn than the tensor core needs: 3490
// cycles a row.
// The warp of an issuing thread walks its loop as a whole and elects the thread,
// which keeps the descriptors in uniform registers (107 -> 71 us, BF16 1080p).
//
// Measured: 1920x1080 0.206 -> 0.074 ms (BF16), 8 images of 3840x2160 3.185 ->
// 1.83 ms (FP8), against one launch per layer. A BF16 row takes ~960 cycles,
// 890 of shared-memory reads by the MMAs (4 KB of A and 3 KB of weights each,
// at 128 bytes a cycle) and 930 of tensor issue: both are nearly full. An FP8
// row takes as long: half the MMAs, but each layer's next row waits for the
// epilogue's read of its accumulators (~700 cycles from MMA to MMA).
//   full[k][d]      input row in slot d of layer k's ring has arrived (TMA
//                   bytes for k = 0, the 4 epilogue warps of layer k - 1 else)
//   done[k][d]      the MMAs that read it completed (commit): its slot may be
//                   refilled, and the accumulators are up to date
//   acc_empty[k]    layer k's epilogue has read and zeroed its slot (k < 3)
//   acc4_empty[b]   layer 4's epilogue has read TMEM buffer b
constexpr int kFuW = 122;                     // output pixels of a strip
constexpr int kFuPx = 130;                    // pixels of a row buffer
constexpr uint32_t kFuPitch = kFuPx * 16u;    // one chunk of a row buffer
constexpr int kFuF = 6, kFuD = 3;             // ring depths: feature rows, activation rows
constexpr int kFuThreads = 32 * (16 + 4);

template <bool FP8>
struct FusedLayout {
  static constexpr int kCh = FP8 ? 2 : 4;                                  // chunks of an activation pixel
  static constexpr uint32_t kRowF = (2 * kFuPitch + 127u) & ~127u, kRowA = kCh * kFuPitch;
  static constexpr uint32_t kW1 = 3u * 2 * 160 * 16, kWk = 3u * kCh * 160 * 16, kW4 = kCh * 16u * 16;
  static constexpr uint32_t kOffA = kFuF * kRowF;                          // 3 rings of kFuD rows
  static constexpr uint32_t kOffW = kOffA + 3 * kFuD * kRowA;              // W1, W2, W3, W4
  static constexpr uint32_t kOffC = kOffW + kW1 + 2 * kWk + kW4;           // scale[4][32], bias[4][32]
  static constexpr uint32_t kOffX = kOffC + 2 * 4 * 32 * 4;                // layer 4's exchange, [2][2][128] floats
  static constexpr uint32_t kOffB = kOffX + 2 * 2 * 128 * 4;               // barriers
  static constexpr uint32_t kBars = 2 * 4 * kFuF + 3 + 3 + 1;
  static constexpr uint32_t kSmem = kOffB + kBars * 8 + 16;
};

struct FusedArgs {
  const void* w[4];              // packed weights (pack_weights, pack_weights_fp8)
  const float* bias[4];
  const float* inv[4];           // E4M3 inputs: inverse scale per output channel (null: 1)
  float out_scale[4];            // E4M3 outputs (1 otherwise)
  __nv_bfloat16* act[3];         // hidden activations to keep, BF16 planar [4][P][8] (null: none)
  uint32_t* mask;                // training: ReLU masks of the hidden layers, [3][P] words
  __nv_bfloat16* dz[3];          // (data gradients) of layers 3, 2, 1, BF16 planar
  float* prob;                   // output (null: none)
  // training: labels in, the BCE's gradient out and the loss' partial sums,
  // one per warp of layer 4's epilogue (see "BCE and d(logit)")
  const float* label;
  uint4* g8;
  float* loss_part;
  uint32_t W, H, n_img, strips, segs, rows;   // rows: output rows of a segment
  uint32_t* err;
};

// a unit of work: `rows` output rows (fewer at the bottom) of one strip
struct FusedItem {
  int img, x0, y0, rows;         // x0: image column of the first layer's lane 0
};
// LAYERS convolutions in a row: every one but the last loses a pixel at either
// end of the strip
template <int LAYERS>
__host__ __device__ constexpr int strip_width() { return 128 - 2 * (LAYERS - 1); }
template <int LAYERS>
__device__ __forceinline__ FusedItem fused_item(const FusedArgs& a, uint32_t item) {
  const uint32_t strip = item % a.strips, q = item / a.strips, seg = q % a.segs;
  FusedItem it;
  it.img = (int)(q / a.segs);
  it.x0 = (int)strip * strip_width<LAYERS>() - (LAYERS - 1);
  it.y0 = (int)(seg * a.rows);
  it.rows = (int)min(a.rows, a.H - seg * a.rows);
  return it;
}

// One row of a stacked layer: for kernel column dx and 32-byte K step, the
// input row moved by dx pixels times the window of weight blocks at wbase.
template <int CH, bool E4M3>
__device__ __forceinline__ void issue_row_mmas(uint32_t abase, uint32_t wbase, uint32_t dtmem) {
  constexpr uint32_t idesc = E4M3 ? make_idesc_e4m3(128, 96) : make_idesc(128, 96);
  const uint32_t a_lo = desc_lo(abase, kFuPitch), b_lo = desc_lo(wbase, 160u * 16u);
  constexpr uint32_t hi = desc_hi(128u);
#pragma unroll
  for (int dx = 0; dx < 3; ++dx)
#pragma unroll
    for (int ks = 0; ks < CH / 2; ++ks) {
      const uint32_t a_off = 2u * ks * kFuPitch + dx * 16u, b_off = (uint32_t)(dx * CH + 2 * ks) * 160u * 16u;
      const uint64_t da = desc_join(a_lo + (a_off >> 4), hi), db = desc_join(b_lo + (b_off >> 4), hi);
      if (E4M3) mma_e4m3(dtmem, da, db, idesc, 1u);
      else mma_bf16(dtmem, da, db, idesc, 1u);
    }
}

// ring position of a layer's rows: slot and the parity of its current use
struct Ring {
  uint32_t slot = 0, par = 0;
  __device__ __forceinline__ void next(uint32_t depth) {
    if (++slot == depth) { slot = 0; par ^= 1u; }
  }
};

// The feature rows of a CTA's items in order: one TMA box per row into the
// ring, zeros outside the image.
template <int LAYERS>
struct FeatureLoader {
  uint32_t item, n_loaded;
  int i;
  FusedItem it;
  __device__ __forceinline__ void load(const FusedArgs& a, const CUtensorMap* map, unsigned char* smem,
                                       uint32_t row_bytes, uint64_t* full, uint32_t n_items) {
    if (item >= n_items) return;
    if (i == 0) it = fused_item<LAYERS>(a, item);
    const uint32_t d = n_loaded % kFuF;
    if (elect_one()) {
      mbar_arrive_expect_tx(full + d, 2 * kFuPitch);
      tma_load_5d(smem + d * row_bytes, map, 0, it.x0 - 1, 0, it.y0 - LAYERS + i, it.img, full + d);
    }
    ++n_loaded;
    if (++i == it.rows + 2 * LAYERS) { i = 0; item += gridDim.x; }
  }
};

// MMAs of layer K's rows (one thread): a row is issued once it has arrived and
// the epilogue has read and zeroed the slot it will finish. Layer 1's thread
// also loads the feature rows: when the epilogue has read row r - 1's sums,
// that row's MMAs are done and its slot takes row r - 1 + kFuF.
// KIND: 0 layer 1, 1 layers 2 and 3 (K = 1, 2), 2 layer 4.
template <int KIND, bool FP8, int LAYERS>
__device__ __forceinline__ bool fused_mmas(const int K, const FusedArgs& a, const CUtensorMap* map,
                                           unsigned char* smem, uint64_t* full, uint64_t* done,
                                           uint64_t* empty, uint32_t tmem) {
  using Lt = FusedLayout<FP8>;
  const uint32_t sbase = smem_u32(smem);
  constexpr uint32_t kDepth = KIND == 0 ? kFuF : kFuD;
  constexpr uint32_t kRow = KIND == 0 ? Lt::kRowF : Lt::kRowA;
  const uint32_t rows0 = sbase + (KIND == 0 ? 0u : Lt::kOffA + (uint32_t)(K - 1) * kFuD * Lt::kRowA);
  const uint32_t w0 = sbase + Lt::kOffW + (K > 0 ? Lt::kW1 : 0u) + (K > 1 ? (uint32_t)(K - 1) * Lt::kWk : 0u);
  const uint32_t n_items = a.strips * a.segs * a.n_img;
  uint64_t* full_k = full + K * kFuF;
  uint64_t* done_k = done + K * kFuF;
  Ring ring;
  uint32_t row3 = 0, n_row = 0;
  bool ok = true;
  FeatureLoader<LAYERS> ld = {blockIdx.x, 0u, 0, {}};
  if (KIND == 0)
    for (int i = 0; i < kFuF - 1; ++i) ld.load(a, map, smem, Lt::kRowF, full, n_items);
  for (uint32_t item = blockIdx.x; ok && item < n_items; item += gridDim.x) {
    const int n = fused_item<LAYERS>(a, item).rows + 2 * (LAYERS - K);
    for (int i = 0; i < n; ++i) {
      if (KIND < 2)
        ok = n_row == 0 ? mbar_wait(full_k + ring.slot, ring.par)
                        : mbar_wait2<FP8>(full_k + ring.slot, ring.par, empty + K, (n_row - 1) & 1u);
      else
        ok = n_row < 3 ? mbar_wait(full_k + ring.slot, ring.par)
                       : mbar_wait2<FP8>(full_k + ring.slot, ring.par, empty + row3, (n_row / 3 - 1) & 1u);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) break;
      fence_after();
      if (elect_one()) {
        const uint32_t abase = rows0 + ring.slot * kRow;
        if (KIND < 2) {
          issue_row_mmas<KIND == 0 ? 2 : Lt::kCh, (KIND > 0 && FP8)>(abase, w0 + (2u - row3) * 512u, tmem + 96u * K);
        } else {
          constexpr uint32_t idesc = FP8 ? make_idesc_e4m3(128, 16) : make_idesc(128, 16);
          constexpr uint32_t hi = desc_hi(128u);
          const uint32_t a_lo = desc_lo(abase, kFuPitch), b_lo = desc_lo(w0, 256u);
#pragma unroll
          for (int ks = 0; ks < Lt::kCh / 2; ++ks) {
            const uint64_t da = desc_join(a_lo + ((2u * ks * kFuPitch) >> 4), hi);
            const uint64_t db = desc_join(b_lo + ((2u * ks * 256u) >> 4), hi);
            if (FP8) mma_e4m3(tmem + 288u + 16u * row3, da, db, idesc, ks > 0);
            else mma_bf16(tmem + 288u + 16u * row3, da, db, idesc, ks > 0);
          }
        }
        mma_commit(done_k + ring.slot);
      }
      if (KIND == 0) ld.load(a, map, smem, Lt::kRowF, full, n_items);
      __syncwarp();
      ring.next(kDepth);
      row3 = row3 == 2u ? 0u : row3 + 1u;
      ++n_row;
    }
  }
  // drain: the last copy into each slot has landed before the CTA exits
  if (KIND == 0)
    for (uint32_t j = ld.n_loaded > (uint32_t)kFuF ? ld.n_loaded - kFuF : 0; j < ld.n_loaded; ++j)
      mbar_wait(full + j % kFuF, (j / kFuF) & 1u);
  // drain: the last MMAs complete (and signal) before TMEM is freed
  for (uint32_t r = n_row > kDepth ? n_row - kDepth : 0; r < n_row; ++r)
    mbar_wait(done_k + r % kDepth, (r / kDepth) & 1u);
  return ok;
}

// Epilogue of layers 1-3 (K = 0 .. 2): one warpgroup, lane = pixel. K is no
// template argument: three copies of the loop, each run by one warp per
// scheduler, kept missing the instruction cache.
template <int KT, bool FP8, bool STORE>
__device__ __forceinline__ bool fused_epilogue(const int KR, const FusedArgs& a, unsigned char* smem, uint64_t* full,
                                               uint64_t* done, uint64_t* acc_empty, uint32_t tmem) {
  using Lt = FusedLayout<FP8>;
  const int K = KT < 0 ? KR : KT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, m = quarter * 32 + lane;
  // Biases and (E4M3 output) scales stay in registers: shared memory is what
  // bounds this kernel, and reading them there for every pixel took 190 (BF16)
  // to 640 (FP8) of its cycles a row.
  const float* cst = reinterpret_cast<const float*>(smem + Lt::kOffC) + K * 32;
  float bi[32];
  float sc[FP8 ? 32 : 1];
#pragma unroll
  for (int c = 0; c < 32; ++c) bi[c] = cst[4 * 32 + c];
  if (FP8)
#pragma unroll
    for (int c = 0; c < 32; ++c) sc[c % (FP8 ? 32 : 1)] = cst[c];
  const uint32_t slots = tmem + ((uint32_t)(quarter * 32) << 16) + 96u * K;
  unsigned char* ring = smem + Lt::kOffA + (uint32_t)K * kFuD * Lt::kRowA + (uint32_t)m * 16u;
  const uint32_t n_items = a.strips * a.segs * a.n_img;
  const uint32_t depth = K == 0 ? kFuF : kFuD;
  uint64_t* full_n = full + (K + 1) * kFuF;
  uint64_t* done_k = done + K * kFuF;
  uint64_t* done_n = done + (K + 1) * kFuF;
  Ring in, out;                       // rows read from this layer's ring / written to the next one's
  bool out_wrapped = false;
  uint32_t fin = 1;                   // slot of the finished row: (row - 2) % 3
  for (uint32_t item = blockIdx.x; item < n_items; item += gridDim.x) {
    const FusedItem it = fused_item<4>(a, item);
    const int n = it.rows + 8 - 2 * K;
    const int x = it.x0 + K + m;
    const bool col_in = x >= 0 && x < (int)a.W;
    for (int i = 0; i < n; ++i) {
      // the sums, and (from the first reuse on) the output row's slot
      const bool ok = i >= 2 && out_wrapped ? mbar_wait2<FP8>(done_n + out.slot, out.par ^ 1u, done_k + in.slot, in.par)
                                            : mbar_wait(done_k + in.slot, in.par);
      if (!__all_sync(0xFFFFFFFFu, ok)) return false;
      in.next(depth);
      fence_after();
      uint32_t r[2][16];
      const uint32_t at = slots + fin * 32u;
      tmem_ld16_nowait(at, r[0]);
      tmem_ld16_nowait(at + 16u, r[1]);
      tmem_wait_ld();
      tmem_zero16(at);
      tmem_zero16(at + 16u);
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + K);
      fin = fin == 2u ? 0u : fin + 1u;
      if (i < 2) continue;            // rows above the segment: never read
      const int y = it.y0 - 3 + K + (i - 2);
      const bool inside = col_in && y >= 0 && y < (int)a.H;
      unsigned char* dst = ring + out.slot * Lt::kRowA;
      uint4 v[Lt::kCh];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t packed[8];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          const int c0 = h * 16 + 2 * j;
          float y0 = __uint_as_float(r[h][2 * j]), y1 = __uint_as_float(r[h][2 * j + 1]);
          float y2 = __uint_as_float(r[h][2 * j + 2]), y3 = __uint_as_float(r[h][2 * j + 3]);
          if (FP8) {
            constexpr int kS = FP8 ? 32 : 1;
            fma2(y0, y1, sc[c0 % kS], sc[(c0 + 1) % kS], bi[c0], bi[c0 + 1]);
            fma2(y2, y3, sc[(c0 + 2) % kS], sc[(c0 + 3) % kS], bi[c0 + 2], bi[c0 + 3]);
            if (K == 0) { y0 = fmaxf(y0, 0.f); y1 = fmaxf(y1, 0.f); y2 = fmaxf(y2, 0.f); y3 = fmaxf(y3, 0.f); }
            packed[j >> 1] = relu_e4m3x4(y0, y1, y2, y3);
          } else {
            add2(y0, y1, bi[c0], bi[c0 + 1]);
            add2(y2, y3, bi[c0 + 2], bi[c0 + 3]);
            packed[j] = relu_bf16(pack_bf16(y0, y1));
            packed[j + 1] = relu_bf16(pack_bf16(y2, y3));
          }
        }
        if (FP8) {
          v[h] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        } else {
          v[(2 * h) % Lt::kCh] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
          v[(2 * h + 1) % Lt::kCh] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
        }
      }
      if (!__all_sync(0xFFFFFFFFu, inside)) {
        if (!inside)
#pragma unroll
          for (int c = 0; c < Lt::kCh; ++c) v[c] = make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int c = 0; c < Lt::kCh; ++c) *reinterpret_cast<uint4*>(dst + (uint32_t)c * kFuPitch) = v[c];
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full_n + out.slot);
      out.next(kFuD);
      if (out.slot == 0) out_wrapped = true;
      if (STORE && !FP8) {            // the segment's own pixels: image columns x0 + 3 .. x0 + 3 + 121
        const int own = m + K - 3;
        if (inside && own >= 0 && own < kFuW && y >= it.y0 && y < it.y0 + it.rows) {
          const size_t P = (size_t)a.W * a.H * a.n_img, p = ((size_t)it.img * a.H + y) * a.W + x;
#pragma unroll
          for (int c = 0; c < Lt::kCh; ++c) *reinterpret_cast<uint4*>(a.act[K] + ((size_t)c * P + p) * 8) = v[c];
          if (a.mask) {
            uint32_t word = 0u;
#pragma unroll
            for (int c = 0; c < Lt::kCh; ++c) {
              word = mask_bits(word, v[c].x, 4 * c);
              word = mask_bits(word, v[c].y, 4 * c + 1);
              word = mask_bits(word, v[c].z, 4 * c + 2);
              word = mask_bits(word, v[c].w, 4 * c + 3);
            }
            a.mask[K * P + p] = word;
          }
        }
      }
    }
  }
  return true;
}

// ------------------------------------------------------- BCE and d(logit)
// loss = mean(-(y log p + (1-y) log(1-p))), dlogit g = p - y (the 1/P factor
// is applied in the weight-gradient reduction). g goes out as one 16-byte
// channel chunk per pixel, [P][8] BF16: channel 0 = bf16(g), the input of the
// layer-4 data-gradient conv, and channels 1, 2 = the two BF16 remainders, so
// that the three add up to the FP32 g exactly and the layer-4 weight gradient
// keeps all its bits on the tensor cores. Returns the pixel's loss.
__device__ __forceinline__ float bce_gradient(float p, float y, uint4& g8) {
  const float q = fminf(fmaxf(p, 1e-7f), 1.f - 1e-7f);
  const float g = p - y;
  const float hi = __bfloat162float(__float2bfloat16_rn(g));
  const float mid = __bfloat162float(__float2bfloat16_rn(g - hi));
  g8 = make_uint4(pack_bf16(hi, mid), pack_bf16(g - hi - mid, 0.f), 0u, 0u);
  return -(y * __logf(q) + (1.f - y) * __logf(1.f - q));
}

template <bool FP8, bool STORE>
__global__ void __launch_bounds__(kFuThreads, 1)
    k_net_fused(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ FusedArgs a) {
  using Lt = FusedLayout<FP8>;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lt::kOffB);
  uint64_t* full = bars;                         // [4][kFuF]
  uint64_t* done = bars + 4 * kFuF;              // [4][kFuF]
  uint64_t* acc_empty = bars + 8 * kFuF;         // [3]
  uint64_t* acc4_empty = acc_empty + 3;          // [3]
  uint64_t* xbar = acc4_empty + 3;               // layer 4's exchange
  uint32_t* tslot = reinterpret_cast<uint32_t*>(xbar + 1);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // known to be uniform
  const uint32_t n_items = a.strips * a.segs * a.n_img;

  // the two pixels past every activation row feed unused lanes only: finite
  for (uint32_t i = tid; i < 3u * kFuD * Lt::kRowA / 16u; i += kFuThreads)
    reinterpret_cast<uint4*>(smem + Lt::kOffA)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    for (int k = 0; k < 4; ++k)
      for (int d = 0; d < kFuF; ++d) {
        mbar_init(full + k * kFuF + d, k == 0 ? 1 : 4);
        mbar_init(done + k * kFuF + d, 1);
      }
    for (int k = 0; k < 3; ++k) {
      mbar_init(acc_empty + k, 4);
      mbar_init(acc4_empty + k, 4);
    }
    mbar_init(xbar, 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap)) : "memory");
  }
  if (warp == 0) tmem_alloc(tslot, 512);
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);
  if (warp < 4) {
    for (uint32_t c = 0; c < 288u; c += 16) tmem_zero16(tmem + ((uint32_t)(warp * 32) << 16) + c);
    tmem_wait_st();
  }
  after_previous();              // the weights may come from the kernel before

  // weights: three stacked blocks per (dx, chunk) become five
  uint32_t off_w[4] = {Lt::kOffW, Lt::kOffW + Lt::kW1, Lt::kOffW + Lt::kW1 + Lt::kWk,
                       Lt::kOffW + Lt::kW1 + 2 * Lt::kWk};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t groups = 3u * (k == 0 ? 2u : (uint32_t)Lt::kCh);
    const uint4* src = static_cast<const uint4*>(a.w[k]);
    uint4* dst = reinterpret_cast<uint4*>(smem + off_w[k]);
    for (uint32_t i = tid; i < groups * 160u; i += kFuThreads) {
      const uint32_t g = i / 160u, r = i - g * 160u;
      dst[i] = src[g * 96u + (r >= 96u ? r - 96u : r)];
    }
  }
  for (uint32_t i = tid; i < Lt::kW4 / 16u; i += kFuThreads)
    reinterpret_cast<uint4*>(smem + off_w[3])[i] = static_cast<const uint4*>(a.w[3])[i];
  float* cst = reinterpret_cast<float*>(smem + Lt::kOffC);
  for (uint32_t i = tid; i < 4u * 32u; i += kFuThreads) {
    const uint32_t k = i / 32u, c = i % 32u;
    const bool real = k < 3u || c == 0u;
    // powers of two: the folded form rounds like scaling the rounded sum
    cst[i] = real ? (a.inv[k] ? a.inv[k][c] : 1.f) * a.out_scale[k] : 0.f;
    cst[4 * 32 + i] = real ? a.bias[k][c] * a.out_scale[k] : 0.f;
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();

  // registers by role: 128 x (3 x 120 + 64 + 40) of the 640 x 96 launched with
  if (warp >= 16) {
    // ---- MMA issue, one thread per layer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    const bool ok = warp == 16  ? fused_mmas<0, FP8, 4>(0, a, &tmap, smem, full, done, acc_empty, tmem)
                    : warp < 19 ? fused_mmas<1, FP8, 4>(warp - 16, a, &tmap, smem, full, done, acc_empty, tmem)
                                : fused_mmas<2, FP8, 4>(3, a, &tmap, smem, full, done, acc4_empty, tmem);
    if (!ok && lane == 0) atomicOr(a.err, ERR_ITER);
  } else if (warp < 12) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 120;");
    bool ok;
    if (FP8)
      ok = warp < 4   ? fused_epilogue<0, FP8, STORE>(0, a, smem, full, done, acc_empty, tmem)
           : warp < 8 ? fused_epilogue<1, FP8, STORE>(1, a, smem, full, done, acc_empty, tmem)
                      : fused_epilogue<2, FP8, STORE>(2, a, smem, full, done, acc_empty, tmem);
    else
      ok = fused_epilogue<-1, FP8, STORE>(warp >> 2, a, smem, full, done, acc_empty, tmem);
    if (!ok && lane == 0) atomicOr(a.err, ERR_ITER);
  } else {
    // ---- layer 4: sums[dx] of the three vertical taps, then the neighbours'
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const int quarter = warp & 3, m = quarter * 32 + lane;
    float* xs = reinterpret_cast<float*>(smem + Lt::kOffX);      // [parity][dx 0 or 2][pixel]
    const float sc = cst[3 * 32], bi = cst[7 * 32];
    Ring in;
    uint32_t buf = 0, n_row = 0;
    float loss = 0.f;
    float s1[3] = {0.f, 0.f, 0.f}, s2[3] = {0.f, 0.f, 0.f};      // rows with one and with two taps added
    bool ok = true;
    for (uint32_t item = blockIdx.x; ok && item < n_items; item += gridDim.x) {
      const FusedItem it = fused_item<4>(a, item);
      const int x = it.x0 + 2 + m;
      for (int i = 0; i < it.rows + 2; ++i, ++n_row) {
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(done + 3 * kFuF + in.slot, in.par))) { ok = false; break; }
        in.next(kFuD);
        fence_after();
        uint32_t r[16];
        tmem_ld16_nowait(tmem + ((uint32_t)(quarter * 32) << 16) + 288u + 16u * buf, r);
        tmem_wait_ld();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc4_empty + buf);
        buf = buf == 2u ? 0u : buf + 1u;
        float z[3];
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          z[dx] = s2[dx] + __uint_as_float(r[6 + dx]);
          s2[dx] = s1[dx] + __uint_as_float(r[3 + dx]);
          s1[dx] = __uint_as_float(r[dx]);
        }
        float* px = xs + (n_row & 1u) * 256u;
        px[m] = z[0];
        px[128 + m] = z[2];
        __syncwarp();
        if (lane == 0) mbar_arrive(xbar);
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(xbar, n_row & 1u))) { ok = false; break; }
        if (i < 2) continue;
        const int y = it.y0 + i - 2;
        if (m >= 1 && m <= kFuW && x < (int)a.W) {
          const float v = fmaf((px[m - 1] + z[1]) + px[128 + m + 1], sc, bi);
          const float prob = 1.f / (1.f + __expf(-v));
          const size_t p = ((size_t)it.img * a.H + y) * a.W + x;
          if (!STORE || a.prob) a.prob[p] = prob;
          if (STORE && a.label) loss += bce_gradient(prob, a.label[p], a.g8[p]);
        }
      }
    }
    if (STORE && a.label) {
      for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, off);
      if (lane == 0) a.loss_part[blockIdx.x * 4 + quarter] = loss;
    }
    if (!ok && lane == 0) atomicOr(a.err, ERR_ITER);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------- data gradients
// The three data-gradient convolutions (weights flipped, channels swapped, each
// followed by the ReLU mask of the layer's activations) in one kernel, streamed
// like the forward pass: BCE gradient in, the gradients of layers 3, 2 and 1
// stay on the SM on their way to the next one and go to memory once, for the
// weight gradients. Same MMAs in the same order as one launch per layer: same
// bits. A strip is 124 pixels wide. Bound by memory: 64 bytes of gradient per
// pixel and layer, and 4 of mask (one bit a channel, written by the forward pass;
// loaded before the wait for the row's sums). Measured at 960x540: three launches
// 21 + 26 + 26 us; one with the activations themselves as masks (64 bytes) 54, with
// bits 42. Training step 180 -> 169 -> 153 us, 251x143 49.3 -> 44.1 -> 43.5.
// (149 and 39.9 since the kernels set up before they wait for the one before.)
constexpr int kBwThreads = 32 * (12 + 4);

// Epilogue of gradient K (one warpgroup, lane = pixel)
__device__ __forceinline__ bool bwd_epilogue(const int K, const FusedArgs& a, unsigned char* smem, uint64_t* full,
                                             uint64_t* done, uint64_t* acc_empty, uint32_t tmem) {
  using Lt = FusedLayout<false>;
  constexpr int kLayers = 3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, m = quarter * 32 + lane;
  const uint32_t slots = tmem + ((uint32_t)(quarter * 32) << 16) + 96u * K;
  unsigned char* ring = smem + Lt::kOffA + (uint32_t)K * kFuD * Lt::kRowA + (uint32_t)m * 16u;
  const uint32_t n_items = a.strips * a.segs;
  const uint32_t depth = K == 0 ? kFuF : kFuD;
  const bool to_next = K + 1 < kLayers;
  uint64_t* full_n = full + (K + 1) * kFuF;
  uint64_t* done_k = done + K * kFuF;
  uint64_t* done_n = done + (K + 1) * kFuF;
  uint4* const out = reinterpret_cast<uint4*>(a.dz[K]);
  const size_t P = (size_t)a.W * a.H;
  const uint32_t* const mask = a.mask + (2 - K) * P;
  Ring in, next;
  bool wrapped = false;
  uint32_t fin = 1;
  for (uint32_t item = blockIdx.x; item < n_items; item += gridDim.x) {
    const FusedItem it = fused_item<kLayers>(a, item);
    const int n = it.rows + 2 * (kLayers - K);
    const int x = it.x0 + K + m;
    const bool col_in = x >= 0 && x < (int)a.W, col_own = m + K - 2 >= 0 && m + K - 2 < strip_width<kLayers>();
    for (int i = 0; i < n; ++i) {
      const int y = it.y0 - 2 + K + (i - 2);
      const bool inside = i >= 2 && col_in && y >= 0 && y < (int)a.H;
      const size_t p = inside ? (size_t)y * a.W + x : 0;
      const uint32_t mk = inside ? __ldcg(mask + p) : 0u;   // written by the kernel before
      const bool ok = i >= 2 && to_next && wrapped
                          ? mbar_wait2<false>(done_n + next.slot, next.par ^ 1u, done_k + in.slot, in.par)
                          : mbar_wait(done_k + in.slot, in.par);
      if (!__all_sync(0xFFFFFFFFu, ok)) return false;
      in.next(depth);
      fence_after();
      uint32_t r[2][16];
      const uint32_t at = slots + fin * 32u;
      tmem_ld16_nowait(at, r[0]);
      tmem_ld16_nowait(at + 16u, r[1]);
      tmem_wait_ld();
      tmem_zero16(at);
      tmem_zero16(at + 16u);
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + K);
      fin = fin == 2u ? 0u : fin + 1u;
      if (i < 2) continue;
      uint4 v[4];                       // a zero mask (outside the image too) gives zeros
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t* q = &r[c >> 1][(c & 1) * 8];
        v[c].x = masked_pair(mk, 4 * c + 0, q[0], q[1]);
        v[c].y = masked_pair(mk, 4 * c + 1, q[2], q[3]);
        v[c].z = masked_pair(mk, 4 * c + 2, q[4], q[5]);
        v[c].w = masked_pair(mk, 4 * c + 3, q[6], q[7]);
      }
      if (to_next) {
        unsigned char* dst = ring + next.slot * Lt::kRowA;
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(dst + (uint32_t)c * kFuPitch) = v[c];
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_n + next.slot);
        next.next(kFuD);
        if (next.slot == 0) wrapped = true;
      }
      if (inside && col_own && y >= it.y0 && y < it.y0 + it.rows)
#pragma unroll
        for (int c = 0; c < 4; ++c) out[c * P + p] = v[c];
    }
  }
  return true;
}

__global__ void __launch_bounds__(kBwThreads, 1)
    k_bwd_fused(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ FusedArgs a) {
  using Lt = FusedLayout<false>;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lt::kOffB);
  uint64_t* full = bars;                         // [4][kFuF]
  uint64_t* done = bars + 4 * kFuF;              // [4][kFuF]
  uint64_t* acc_empty = bars + 8 * kFuF;         // [3]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(acc_empty + 3);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // known to be uniform
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t groups = 3u * (k == 0 ? 2u : 4u);
    const uint4* src = static_cast<const uint4*>(a.w[k]);
    uint4* dst = reinterpret_cast<uint4*>(smem + Lt::kOffW + (k > 0 ? Lt::kW1 : 0u) + (k > 1 ? Lt::kWk : 0u));
    for (uint32_t i = tid; i < groups * 160u; i += kBwThreads) {
      const uint32_t g = i / 160u, r = i - g * 160u;
      dst[i] = src[g * 96u + (r >= 96u ? r - 96u : r)];
    }
  }
  // the two pixels past every gradient row feed unused lanes only: finite
  for (uint32_t i = tid; i < 2u * kFuD * Lt::kRowA / 16u; i += kBwThreads)
    reinterpret_cast<uint4*>(smem + Lt::kOffA)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    for (int k = 0; k < 3; ++k) {
      for (int d = 0; d < kFuF; ++d) {
        mbar_init(full + k * kFuF + d, k == 0 ? 1 : 4);
        mbar_init(done + k * kFuF + d, 1);
      }
      mbar_init(acc_empty + k, 4);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap)) : "memory");
  }
  if (warp == 0) tmem_alloc(tslot, 512);
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);
  if (warp < 4) {
    for (uint32_t c = 0; c < 288u; c += 16) tmem_zero16(tmem + ((uint32_t)(warp * 32) << 16) + c);
    tmem_wait_st();
  }
  fence_before();
  __syncthreads();
  fence_after();
  // the weights are older than the kernel before: it began after they were written
  after_previous();
  bool ok = true;
  if (warp < 12)
    ok = bwd_epilogue(warp >> 2, a, smem, full, done, acc_empty, tmem);
  else if (warp == 12)
    ok = fused_mmas<0, false, 3>(0, a, &tmap, smem, full, done, acc_empty, tmem);
  else if (warp < 15)
    ok = fused_mmas<1, false, 3>(warp - 12, a, &tmap, smem, full, done, acc_empty, tmem);
  if (!ok && lane == 0) atomicOr(a.err, ERR_ITER);
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------ weight packing (FP32 -> BF16)
// Canonical parameter layout of a layer: W[Cout][Cin][3][3] then b[Cout].
// Packed (stacked taps): element i of a conv with output
// channels cout_p and input channels cin_p, chunks of `per` elements, is
// [dx][ci / per][j * cout_p + co][ci % per] with tap (dy = 2 - j, dx).
struct StackedIndex {
  int co, ci, tap;
};
__device__ __forceinline__ StackedIndex stacked_index(int i, int per, int cout_p, int cin_p) {
  const int e = i % per, rest = i / per;
  const int n = rest % (3 * cout_p), rest2 = rest / (3 * cout_p);
  const int chunk = rest2 % (cin_p / per), dx = rest2 / (cin_p / per);
  const int j = n / cout_p;
  return {n - j * cout_p, chunk * per + e, (2 - j) * 3 + dx};
}

// forward pack: W[co][ci][tap] with ci < cin_pad, co < cout_pad (zero fill)
__global__ void k_pack_fwd(const float* __restrict__ Wt, int cout, int cin, int cout_pad,
                           int cin_pad, __nv_bfloat16* __restrict__ out) {
  const int n = 9 * cin_pad * cout_pad;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const StackedIndex x = stacked_index(i, 8, cout_pad, cin_pad);
    float v = 0.f;
    if (x.co < cout && x.ci < cin) v = Wt[((size_t)x.co * cin + x.ci) * 9 + x.tap];
    out[i] = __float2bfloat16_rn(v);
  }
}

// backward-data pack: a conv whose output channel o is forward input channel
// ci and whose input channel c is forward output channel co, taps flipped:
// W'[o][c][tap] = W[c][o][8 - tap]
__global__ void k_pack_bwd(const float* __restrict__ Wt, int cout, int cin, int cout_pad,
                           int cin_pad, __nv_bfloat16* __restrict__ out) {
  // as a conv: CIN' = cout_pad, COUT' = cin_pad
  const int n = 9 * cout_pad * cin_pad;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const StackedIndex x = stacked_index(i, 8, cin_pad, cout_pad);   // x.co: forward ci, x.ci: forward co
    float v = 0.f;
    if (x.ci < cout && x.co < cin) v = Wt[((size_t)x.ci * cin + x.co) * 9 + (8 - x.tap)];
    out[i] = __float2bfloat16_rn(v);
  }
}

// FP8 forward pack of layers 2-4: E4M3 of W[co][ci][tap] * scale[co] (round
// to nearest even, saturating), chunks of 16 elements, zero fill
__global__ void k_pack_fwd_fp8(const float* __restrict__ Wt, int cout, int cin, int cout_pad,
                               int cin_pad, const float* __restrict__ scale, uint8_t* __restrict__ out) {
  const int n = 9 * cin_pad * cout_pad;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const StackedIndex x = stacked_index(i, 16, cout_pad, cin_pad);
    float v = 0.f;
    if (x.co < cout && x.ci < cin) v = Wt[((size_t)x.co * cin + x.ci) * 9 + x.tap] * scale[x.co];
    out[i] = (uint8_t)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
  }
}

// Layer 4 of the fused forward pass: its 9 taps along N, [chunk][16][chunk
// elements] with W[0][ci][tap] at n = tap < 9 (BF16, or E4M3 scaled like the
// other layers), zero fill
__global__ void k_pack_taps(const float* __restrict__ Wt, int cin, __nv_bfloat16* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 16 * cin; i += gridDim.x * blockDim.x) {
    const int ci = i / (16 * 8) * 8 + i % 8, n = i / 8 % 16;
    out[i] = __float2bfloat16_rn(n < 9 ? Wt[ci * 9 + n] : 0.f);
  }
}
__global__ void k_pack_taps_fp8(const float* __restrict__ Wt, int cin, const float* __restrict__ scale,
                                uint8_t* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 16 * cin; i += gridDim.x * blockDim.x) {
    const int ci = i / (16 * 16) * 16 + i % 16, n = i / 16 % 16;
    const float v = n < 9 ? Wt[ci * 9 + n] * scale[0] : 0.f;
    out[i] = (uint8_t)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
  }
}

// largest element of a non-negative BF16 map (ReLU outputs): float bits of
// non-negative values order like unsigned integers
__global__ void k_amax(const __nv_bfloat16* __restrict__ a, size_t n, unsigned* __restrict__ out) {
  float m = 0.f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    m = fmaxf(m, __bfloat162float(a[i]));
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_down_sync(0xFFFFFFFFu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// ------------------------------------------------------ weight gradients
// dW[co][ci][ky][kx] = scale * sum_x dZ[y][x][co] * A[y+ky-1][x+kx-1][ci],
// db[co] = scale * sum_x dZ[y][x][co]: a contraction over the pixels, on the
// tensor cores (tcgen05, BF16 operands whose products are exact in FP32).
// A is the layer's input (AC 16-byte channel chunks per pixel: 4 planar, or 2
// interleaved for the features), dZ its data gradient (ZC planar chunks: 4,
// or the BCE gradient's single chunk, whose three parts are added at the end).
// All four layers run in one launch, each on its share of the SMs.
//
// A persistent CTA takes tiles of 4 rows x 112 pixels. TMA boxes bring the
// halo of A (6 rows x 114 pixels) and dZ into shared memory as [row][chunk]
// [pixel][8 channels]: with the pixel as K that is the MN-major, non-swizzled
// operand layout (core matrices of 8 pixels x 8 channels, 128 B apart along
// K), and (row, chunk) is one uniform stride along M and N. So an MMA of
// M = 128 multiplies 4 halo rows (8 of the 16-channel features) at once with
// N = two rows of dZ: block (h, r) of D is the tap ky = h - r of dZ row r.
// Three accumulators, one per kx (the A start moves by kx pixels), 7 K steps
// of 16 pixels and 2 row pairs: 42 MMAs for the 448 pixels of a tile.
// The tensor core truncates when it adds a product to its accumulator, the
// more the longer the sum. So after every CHAIN K steps 8 epilogue warps add
// the useful blocks to FP32 registers, rounding to nearest (warp w: TMEM lanes
// 32 (w % 4), dZ row r = w / 4 of a pair), from one of two accumulator sets
// while the next group's MMAs fill the other; two more warps add up dZ for the
// bias. After every kWgFlush tiles (more in large images) the registers go out as two rows of unscaled
// partial sums (one per r) and start again; k_update adds the rows in a fixed
// order, compensated: the gradient, and training, is the same bit for bit from
// run to run.
// Measured (all four layers and the reduction, hot L2): 0.231 ms at 1920x1080,
// 0.066 at 960x540, 0.017 at 251x143. A tile takes ~2980 cycles, 2190 of them the
// tensor core's 42 MMAs. The FP32 loop through shared memory took 24 ms for one
// 32 x 32 layer at 1920x1080, and 14.4 of a 960x540 training step's 14.5 ms.
// CHAIN = 4 (groups of 4 and 3), or 2 where a CTA has at most kWgFewTiles
// tiles. Error of a 32 x 32 layer's dW against 64 bits, 2-norm, for dZ of random
// sign / of one sign, and what that FP32 loop had:
//   3840x2160  2.8e-7 / 4.4e-8   loop 3.2e-7 / 6.8e-8
//   1920x1080  1.5e-7 / 4.3e-8        2.2e-7 / 6.7e-8
//   960x540    1.5e-7 / 4.4e-8        1.9e-7 / 6.3e-8
//   251x143    7.3e-8 / 4.0e-8        1.1e-7 / 4.8e-8
//   113x5      6.0e-8 / 4.2e-8        5.9e-8 / 4.3e-8   (CHAIN 2; 4: 6.0e-8 / 5.2e-8)
// (whole tiles inside the tensor core, CHAIN 7: 2.0e-7 with one sign).
constexpr int kWgRows = 4, kWgW = 112;                // dZ rows and pixels of a tile
constexpr uint32_t kWgFewTiles = 2;
// tiles between flushes of a CTA, and flushes at most (they bound the partial
// rows: 90 MB for any image)
constexpr uint32_t kWgFlush = 16, kWgFlushes = 8;
// 8 epilogue warps, the MMA warp, the TMA warp and two bias warps
constexpr int kWgEpiWarps = 8, kWgBiasWarps = 2, kWgThreads = 32 * (kWgEpiWarps + 2 + kWgBiasWarps);
static_assert(kWgRows % 2 == 0 && kWgW % 16 == 0, "row pairs, K steps of 16 pixels");

template <int AC, int ZC>
struct WgradLayout {
  static constexpr uint32_t kPitchA = (kWgW + 2) * 16u, kPitchZ = kWgW * 16u;   // one row of one chunk
  static constexpr uint32_t kRowA = AC * kPitchA, kRowZ = ZC * kPitchZ;
  static constexpr uint32_t kBoxA = (kWgRows + 2) * kRowA, kBoxZ = kWgRows * kRowZ;
  static constexpr uint32_t kOffZ = (kBoxA + 127u) & ~127u;
  static constexpr uint32_t kSpanA = (16u / AC) * kRowA;                // bytes an MMA's M = 128 rows span
  // a stage also covers what the last row pair's MMAs read past the halo
  // (AC = 2: M rows that no tap uses)
  static constexpr uint32_t kEndA = (kWgRows - 2) * kRowA + kSpanA + 32u, kEndZ = kOffZ + kBoxZ;
  static constexpr uint32_t kStage = ((kEndA > kEndZ ? kEndA : kEndZ) + 1023u) & ~1023u;
  static constexpr uint32_t kFit = (kSmemBudget - 2048u) / kStage;
  static constexpr int kSt = kFit > 4u ? 4 : (int)kFit;
  static constexpr int kN = 2 * 8 * ZC;                                 // MMA N: two dZ rows
  static constexpr uint32_t kSet = 3 * kN;                              // TMEM columns of one accumulator set
  static constexpr size_t kSmem = kSt * (size_t)kStage + 4 * 8 * 4 + 20 * 8 + 16;
  static constexpr int kCo = ZC == 4 ? 32 : 1;                          // output channels
  static constexpr int kOuts = 9 * kCo * 8 * AC;                        // partial sums of a row, without the biases
};

// instruction descriptor: kind::f16, D = F32, A = B = BF16, both MN-major
__host__ __device__ constexpr uint32_t make_idesc_mn(int M, int N) {
  return make_idesc(M, N) | (1u << 15) | (1u << 16);
}

// 8 consecutive TMEM columns of this warp's 32 lanes, without the wait
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t r[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
}

// (s, c) += x with the rounding error of the sum kept in c (Knuth's TwoSum)
__device__ __forceinline__ void two_sum(float& s, float& c, float x) {
  const float t = s + x, b = t - s;
  c += (s - (t - b)) + (x - b);
  s = t;
}

constexpr uint32_t kWgTmemCols = 512;

// a layer's share of the launch: CTAs blk0 .. blk0 + nblk - 1, and the partial
// rows they write (2 nblk flushes of them, from element part0 on)
struct WgradShare {
  uint32_t blk0, nblk, flush_every, flushes;   // a flush every so many tiles of a CTA
  uint64_t part0;
};
struct WgradArgs {
  CUtensorMap a[4], z[4];        // layers 1 .. 4: input activations, data gradients
  WgradShare share[4];
  uint32_t W, H;
  float* part;
  uint32_t* err;
};

// One CTA's tiles of one layer. Barriers: full[b] TMA bytes of stage b;
// empty[b] its MMAs (commit) and the bias warps' sums are done;
// acc_full[s]: the sums are complete (commit); acc_empty[s]: the epilogue has
// read and zeroed them. A partial row is kOuts + kCo floats, [tap][co][ci] then
// [co].
template <int AC, int ZC, int CHAIN>
__device__ __forceinline__ void wgrad_body(const WgradArgs& args, const int layer, unsigned char* smem) {
  using Lt = WgradLayout<AC, ZC>;
  constexpr int kGroupsRow = (kWgW / 16 + CHAIN - 1) / CHAIN;   // accumulator groups of a row pair
  constexpr int kGroups = kWgRows / 2 * kGroupsRow;             // ... of a tile
  const CUtensorMap& map_a = args.a[layer];
  const CUtensorMap& map_z = args.z[layer];
  const uint32_t W = args.W, H = args.H, nblk = args.share[layer].nblk;
  const uint32_t blk = blockIdx.x - args.share[layer].blk0;
  float* part = args.part + args.share[layer].part0;
  uint32_t* err = args.err;
  float* bias_s = reinterpret_cast<float*>(smem + Lt::kSt * (size_t)Lt::kStage);   // [4][8]
  uint64_t* bars = reinterpret_cast<uint64_t*>(bias_s + 4 * 8);
  uint64_t* full = bars;            // [kSt]
  uint64_t* empty = bars + 8;       // [kSt]
  uint64_t* acc_full = bars + 16;   // [2]
  uint64_t* acc_empty = bars + 18;  // [2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 20);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // known to be uniform
  const uint32_t tiles_x = (W + kWgW - 1) / kWgW;
  const uint32_t n_tiles = tiles_x * ((H + kWgRows - 1) / kWgRows);
  if (tid == 0) {
    for (int b = 0; b < Lt::kSt; ++b) {
      mbar_init(full + b, 1);
      mbar_init(empty + b, 1 + kWgBiasWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full + b, 1);
      mbar_init(acc_empty + b, 32 * kWgEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tslot, kWgTmemCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tslot, 0);
  after_previous();
  const uint32_t my_tiles = blk < n_tiles ? (n_tiles - 1 - blk) / nblk + 1 : 0;

  if (warp == kWgEpiWarps) {
    // ---- MMA issue (the whole warp walks the loop, an elected lane issues)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
    constexpr uint32_t idesc = make_idesc_mn(128, Lt::kN);
    // LBO: from one group of 8 pixels (K) to the next; SBO: from one
    // (row, chunk) group of 8 channels (M or N) to the next
    constexpr uint32_t hi_a = desc_hi(Lt::kPitchA), hi_z = desc_hi(Lt::kPitchZ);
    uint32_t n_mma = 0, grp = 0;       // tiles and accumulator groups issued
    bool ok = true;
    for (uint32_t it = 0; it < my_tiles && ok; ++it) {
      const uint32_t b = it % Lt::kSt;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(full + b, (it / Lt::kSt) & 1u));
      if (!ok) break;
      const uint32_t base = smem_u32(smem) + b * Lt::kStage;
      const uint32_t a_lo = desc_lo(base, 128u), z_lo = desc_lo(base + Lt::kOffZ, 128u);
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        const uint32_t sa = grp & 1u;
        if (grp >= 2) ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_empty + sa, ((grp >> 1) - 1) & 1u));
        if (!ok) break;
        fence_after();
        if (elect_one()) {
          const int rp = g / kGroupsRow, ks0 = (g % kGroupsRow) * CHAIN;
#pragma unroll
          for (int ks = ks0; ks < ks0 + CHAIN && ks < kWgW / 16; ++ks)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              const uint32_t a_off = (2u * rp) * Lt::kRowA + (uint32_t)(16 * ks + dx) * 16u;
              const uint32_t z_off = (2u * rp) * Lt::kRowZ + (uint32_t)(16 * ks) * 16u;
              mma_bf16(tmem + sa * Lt::kSet + (uint32_t)(dx * Lt::kN),
                       desc_join(a_lo + (a_off >> 4), hi_a), desc_join(z_lo + (z_off >> 4), hi_z), idesc,
                       ks == ks0 ? 0u : 1u);
            }
          mma_commit(acc_full + sa);
          if (g == kGroups - 1) mma_commit(empty + b);
        }
        __syncwarp();
        ++grp;
      }
      if (ok) n_mma = it + 1;
    }
    if (!ok && lane == 0) atomicOr(err, ERR_ITER);
    // drain: the MMAs issued here complete (and signal) before TMEM is freed
    for (uint32_t k = grp > 2 ? grp - 2 : 0; k < grp; ++k) mbar_wait(acc_full + (k & 1u), (k >> 1) & 1u);
    for (uint32_t it = n_mma > (uint32_t)Lt::kSt ? n_mma - Lt::kSt : 0; it < n_mma; ++it)
      mbar_wait(empty + (it % Lt::kSt), (it / Lt::kSt) & 1u);
  } else if (warp == kWgEpiWarps + 1) {
    // ---- TMA loads
    asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
    if (lane == 0) {
      bool ok = true;
      uint32_t n_loaded = 0;
      for (uint32_t j = 0; j < my_tiles; ++j) {
        const int b = (int)(j % Lt::kSt);
        if (j >= (uint32_t)Lt::kSt && !mbar_wait(empty + b, ((j / Lt::kSt) - 1) & 1u)) { ok = false; break; }
        const uint32_t tile = blk + j * nblk;
        const int ty = (int)(tile / tiles_x);
        const int y = ty * kWgRows, x0 = (int)(tile - (uint32_t)ty * tiles_x) * kWgW;
        unsigned char* st = smem + (size_t)b * Lt::kStage;
        mbar_arrive_expect_tx(full + b, Lt::kBoxA + Lt::kBoxZ);
        if (AC == 2) tma_load_4d(st, &map_a, 0, x0 - 1, 0, y - 1, full + b);   // {8 channels, W, chunks, H}
        else tma_load_3d(st, &map_a, 2 * (x0 - 1), 0, y - 1, full + b);        // {8-byte halves (2 W), chunks, H}
        tma_load_3d(st + Lt::kOffZ, &map_z, 2 * x0, 0, y, full + b);
        n_loaded = j + 1;
      }
      if (!ok) atomicOr(err, ERR_ITER);
      // drain: the last copy into each stage has landed before the CTA exits
      for (uint32_t j = n_loaded > (uint32_t)Lt::kSt ? n_loaded - Lt::kSt : 0; j < n_loaded; ++j)
        mbar_wait(full + (j % Lt::kSt), (j / Lt::kSt) & 1u);
    }
    __syncwarp();
  } else if (warp > kWgEpiWarps + 1) {
    // ---- bias warps: dZ summed over the tile's pixels, tile after tile
    // compensated (by the epilogue warps it held up the accumulators: 1400 of
    // 4000 cycles a tile)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
    constexpr int kPer = 32 * kWgBiasWarps / ZC;       // threads that add up one chunk of dZ
    const int t = tid - 32 * (kWgEpiWarps + 2), zc = t / kPer, zt = t % kPer;
    float sum[8], comp[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c] = comp[c] = 0.f;
    bool ok = true;
    for (uint32_t it = 0; it < my_tiles && ok; ++it) {
      const int b = (int)(it % Lt::kSt);
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(full + b, (it / Lt::kSt) & 1u));
      if (!ok) break;
      const unsigned char* z = smem + (size_t)b * Lt::kStage + Lt::kOffZ + (uint32_t)zc * Lt::kPitchZ;
      float part8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      constexpr int kLoads = (kWgW + kPer - 1) / kPer;   // of a row
#pragma unroll 1
      for (int row = 0; row < kWgRows; ++row) {
        uint4 v[kLoads];
#pragma unroll
        for (int k = 0; k < kLoads; ++k) {
          const int px = zt + k * kPer;
          v[k] = px < kWgW ? *reinterpret_cast<const uint4*>(z + (uint32_t)row * Lt::kRowZ + (uint32_t)px * 16u)
                           : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < kLoads; ++k) {
          const uint32_t w4[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
            add2(part8[2 * i], part8[2 * i + 1], __uint_as_float(w4[i] << 16), __uint_as_float(w4[i] & 0xFFFF0000u));
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + b);
#pragma unroll
      for (int c = 0; c < 8; ++c) two_sum(sum[c], comp[c], part8[c]);
    }
    if (!ok && lane == 0) atomicOr(err, ERR_ITER);
    // lanes of a chunk (16, or the warp's 32 when there is one chunk), in a fixed order
    constexpr int kLanes = kPer < 32 ? kPer : 32;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      sum[c] += comp[c];
      for (int off = kLanes / 2; off > 0; off >>= 1) sum[c] += __shfl_xor_sync(0xFFFFFFFFu, sum[c], off);
    }
    if (lane % kLanes == 0)
#pragma unroll
      for (int c = 0; c < 8; ++c) bias_s[(t / kLanes) * 8 + c] = sum[c];
  } else {
    // ---- epilogue warps: 256 x 208 + 128 x 80 of the 384 x 168 registers launched with
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    constexpr int kCo = Lt::kCo;                        // output channels a thread accumulates
    const int q = warp & 3, r = warp >> 2;
    const int m = q * 32 + lane, h = m / (8 * AC), ci = m % (8 * AC), dy = h - r;
    const bool useful = dy >= 0 && dy <= 2;
    const bool warp_useful = __any_sync(0xFFFFFFFFu, useful);
    float acc[3][kCo];
    uint32_t grp = 0, it = 0;
    bool ok = true;
    for (uint32_t f = 0; f < args.share[layer].flushes; ++f) {
#pragma unroll
      for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int c = 0; c < kCo; ++c) acc[dx][c] = 0.f;
      const uint32_t end = min(my_tiles, (f + 1) * args.share[layer].flush_every);
      for (; it < end && ok; ++it) {
        // warp-uniform outcomes: tcgen05.ld below is a warp-collective instruction
#pragma unroll 1
        for (int g = 0; g < kGroups; ++g, ++grp) {
          const uint32_t s = grp & 1u;
          if (!__all_sync(0xFFFFFFFFu, mbar_wait(acc_full + s, (grp >> 1) & 1u))) { ok = false; break; }
          fence_after();
          // every column of the group first, then hand the set back, then add
          uint32_t v[3][ZC == 4 ? 32 : 8];
          if (warp_useful) {
            const uint32_t at = tmem + ((uint32_t)(q * 32) << 16) + s * Lt::kSet + (uint32_t)(r * 8 * ZC);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              if (ZC == 4) {
                tmem_ld16_nowait(at + (uint32_t)(dx * Lt::kN), v[dx]);
                tmem_ld16_nowait(at + (uint32_t)(dx * Lt::kN + 16), v[dx] + (ZC == 4 ? 16 : 0));
              } else {
                tmem_ld8_nowait(at + (uint32_t)(dx * Lt::kN), v[dx]);
              }
            }
            tmem_wait_ld();
          }
          fence_before();
          mbar_arrive(acc_empty + s);
          if (warp_useful) {
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              if (ZC == 4) {
#pragma unroll
                for (int c = 0; c < kCo; c += 2)
                  add2(acc[dx][c], acc[dx][(c + 1) % kCo], __uint_as_float(v[dx][c]), __uint_as_float(v[dx][c + 1]));
              } else {
                acc[dx][0] += (__uint_as_float(v[dx][2]) + __uint_as_float(v[dx][1])) + __uint_as_float(v[dx][0]);
              }
            }
          }
        }
      }
      // partial sums since the last flush (zeros where a CTA has fewer than
      // others): row 2 (f nblk + blk) + r, [tap][co][ci]
      if (useful) {
        float* row = part + (2 * ((size_t)f * nblk + blk) + r) * (Lt::kOuts + kCo) +
                     (size_t)(dy * 3 * kCo) * (8 * AC) + ci;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
          for (int c = 0; c < kCo; ++c) row[(dx * kCo + c) * (8 * AC)] = acc[dx][c];
      }
    }
    if (!ok && lane == 0) atomicOr(err, ERR_ITER);
  }
  fence_before();
  __syncthreads();
  fence_after();
  constexpr int kCo = Lt::kCo, kBiasAt = Lt::kOuts;
  if (tid < kCo) {
    // four chunks of 8 channels, or the two halves of the one chunk's pixels
    const float t = ZC == 4 ? bias_s[tid]
                            : ((bias_s[2] + bias_s[10]) + (bias_s[1] + bias_s[9])) + (bias_s[0] + bias_s[8]);
    for (uint32_t f = 0; f < args.share[layer].flushes; ++f)
      for (uint32_t r = 0; r < 2; ++r)
        part[(2 * ((size_t)f * nblk + blk) + r) * (kBiasAt + kCo) + kBiasAt + tid] = f + r == 0 ? t : 0.f;
  }
  if (warp == 0) tmem_dealloc(tmem, kWgTmemCols);
}

template <int CHAIN>
__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad(const __grid_constant__ WgradArgs args) {
  extern __shared__ __align__(1024) unsigned char smem[];
  if (blockIdx.x < args.share[1].blk0) wgrad_body<2, 4, CHAIN>(args, 0, smem);
  else if (blockIdx.x < args.share[2].blk0) wgrad_body<4, 4, CHAIN>(args, 1, smem);
  else if (blockIdx.x < args.share[3].blk0) wgrad_body<4, 4, CHAIN>(args, 2, smem);
  else wgrad_body<4, 1, CHAIN>(args, 3, smem);
}

// ------------------------------------------ reduction, Adam and packing
// One launch for everything after the gradients' contractions, all layers:
// 32 columns of a layer's partial rows per block. grad = scale * the rows' sum,
// in a fixed order and compensated (the FP32 rounding of some hundred rows
// would cost more precision than the tensor cores do): warp w adds rows w,
// w + 8, w + 16, ..., then threads 0..31 add the 8 warp sums in warp order.
// Column j is [tap][co][cin_p] (or, from n_w on, a bias). With an update, Adam
// on the parameter, whose new value goes into the packed weights of the forward
// and the data-gradient kernels (their zero padding never changes). Block 0
// also adds up the loss.
struct UpdateLayer {
  uint32_t block0;               // first block of the layer
  uint32_t nrow, cout, cin, cin_p, off_w, off_b;
  uint64_t part0;
  __nv_bfloat16* wf;
  __nv_bfloat16* wb;             // null: none (layer 1)
};
struct UpdateArgs {
  UpdateLayer layer[4];
  const float* part;
  float scale;                   // 1 / P
  float* grads;                  // null: not wanted
  float *w, *m, *v;              // m null: no update
  float lr, c1, c2;              // step size and Adam's bias corrections
  const float* loss_part;
  uint32_t n_loss;
  float* loss;
};

__global__ void __launch_bounds__(256) k_update(const __grid_constant__ UpdateArgs a) {
  after_previous();
  __shared__ float s[8][32], sc[8][32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int l = 3;
  while (l > 0 && blockIdx.x < a.layer[l].block0) --l;
  const UpdateLayer& y = a.layer[l];
  const uint32_t n_w = 9 * y.cout * y.cin_p, n = n_w + y.cout;
  const uint32_t j = (blockIdx.x - y.block0) * 32 + lane;
  float t = 0.f, c = 0.f;
  if (j < n) {
    const float* part = a.part + y.part0 + j;
#pragma unroll 8
    for (uint32_t b = warp; b < y.nrow; b += 8) two_sum(t, c, part[(size_t)b * n]);
  }
  s[warp][lane] = t;
  sc[warp][lane] = c;
  __syncthreads();
  if (warp == 1 && blockIdx.x == 0) {
    float acc = 0.f, e = 0.f;
    for (uint32_t i = lane; i < a.n_loss; i += 32) two_sum(acc, e, a.loss_part[i]);
    acc += e;
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (lane == 0) *a.loss = acc;
  }
  if (warp != 0 || j >= n) return;
#pragma unroll
  for (int w = 1; w < 8; ++w) {
    c += sc[w][lane];
    two_sum(t, c, s[w][lane]);
  }
  const float g = (t + c) * a.scale;
  const uint32_t ci = j % y.cin_p, co = j < n_w ? (j / y.cin_p) % y.cout : j - n_w, tap = j / (y.cin_p * y.cout);
  if (j < n_w && ci >= y.cin) return;                   // a padding channel
  const uint32_t at = j < n_w ? y.off_w + (co * y.cin + ci) * 9 + tap : y.off_b + co;
  if (a.grads) a.grads[at] = g;
  if (!a.m) return;
  constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mi = b1 * a.m[at] + (1.f - b1) * g;
  const float vi = b2 * a.v[at] + (1.f - b2) * g * g;
  a.m[at] = mi;
  a.v[at] = vi;
  const float w = a.w[at] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + eps);
  a.w[at] = w;
  if (j >= n_w) return;
  const __nv_bfloat16 wb = __float2bfloat16_rn(w);
  const uint32_t dy = tap / 3, dx = tap - 3 * dy;
  if (l < 3)   // stacked taps, as k_pack_fwd
    y.wf[((dx * (y.cin_p / 8) + ci / 8) * (3 * y.cout) + (2 - dy) * y.cout + co) * 8 + ci % 8] = wb;
  else         // taps along N, as k_pack_taps
    y.wf[(ci / 8) * 128 + tap * 8 + ci % 8] = wb;
  if (y.wb) {  // flipped taps, channels swapped, as k_pack_bwd
    const uint32_t cout_p = l == 3 ? 16u : 32u, fy = 2 - dy, fx = 2 - dx;
    y.wb[((fx * (cout_p / 8) + co / 8) * (3 * y.cin_p) + (2 - fy) * y.cin_p + ci) * 8 + co % 8] = wb;
  }
}

}  // namespace nn
}  // namespace rt

// ===================================================================== host
namespace rt {
namespace nn {

namespace {
// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
// (no link-time dependency on libcuda)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    else
      cudaGetLastError();
  }
  return fn;
}

// One map of W x H pixels for k_wgrad: `chunks` 16-byte channel chunks per
// pixel, interleaved ([P][16], 2 chunks) as {8 channels, W, chunks, H} or
// planar ([chunks][P][8]) as 8-byte elements {2 W, chunks, H}; the box is
// `px` pixels of every chunk in `rows` rows, in shared memory [row][chunk][px].
cudaError_t make_wgrad_map(CUtensorMap* map, const void* in, uint32_t W, uint32_t H, uint32_t chunks,
                           bool interleaved, uint32_t px, uint32_t rows) {
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return cudaErrorNotSupported;
  if (reinterpret_cast<uintptr_t>(in) & 15u) return cudaErrorInvalidValue;
  const cuuint64_t P = (cuuint64_t)W * H;
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r;
  if (interleaved) {
    const cuuint64_t d[4] = {8, W, chunks, H}, st[3] = {16ull * chunks, 16, 16ull * chunks * W};
    const cuuint32_t bx[4] = {8, px, chunks, rows};
    r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(in), d, st, bx, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    const cuuint64_t d[3] = {2ull * W, chunks, H}, st[2] = {P * 16, 16ull * W};
    const cuuint32_t bx[3] = {2 * px, chunks, rows};
    r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<void*>(in), d, st, bx, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

uint64_t wgrad_tiles(uint32_t W, uint32_t H) {
  return (uint64_t)((W + kWgW - 1) / kWgW) * ((H + kWgRows - 1) / kWgRows);
}

// Shares of the SMs: the next CTA always goes to the layer that would take
// longest (tiles a CTA times a tile's cost; at most one CTA per tile)
void wgrad_shares(uint32_t W, uint32_t H, WgradShare share[4], uint64_t* part_floats) {
  // Between a tile's bytes (the first and last layer load 0.70 of a middle one's)
  // and its MMAs (the same number in every layer). Training step at 251x143 / 640x360
  // / 960x540 / 1400x800, us: 39.5 / 80.5 / 148.1 / 288.6; with 0.7 for both 42.8 /
  // 82.7 / 152.0 / 301.7, with 0.6 42.9 / 85.8 / 157.1 / 313.3, with 0.9 39.5 / 79.2 /
  // 145.7 / 285.0, with 1 39.6 / 79.3 / 142.8 / 282.3: the MMAs decide.
  static const float kCost[4] = {0.8f, 1.f, 1.f, 0.8f};
  const uint64_t tiles = wgrad_tiles(W, H);
  uint32_t nb[4] = {1, 1, 1, 1};
  for (int used = 4; used < num_sms(); ++used) {
    int at = -1;
    float most = 0.f;
    for (int l = 0; l < 4; ++l) {
      const float t = (float)((tiles + nb[l] - 1) / nb[l]) * kCost[l];
      if (nb[l] < tiles && t > most) { most = t; at = l; }
    }
    if (at < 0) break;
    ++nb[at];
  }
  static const uint32_t kRow[4] = {WgradLayout<2, 4>::kOuts + 32, WgradLayout<4, 4>::kOuts + 32,
                                   WgradLayout<4, 4>::kOuts + 32, WgradLayout<4, 1>::kOuts + 1};
  uint32_t blk = 0;
  uint64_t at = 0;
  for (int l = 0; l < 4; ++l) {
    const uint32_t most = (uint32_t)((tiles + nb[l] - 1) / nb[l]);   // tiles of a CTA
    const uint32_t every = std::max(kWgFlush, (most + kWgFlushes - 1) / kWgFlushes);
    const uint32_t flushes = (most + every - 1) / every;
    share[l] = {blk, nb[l], every, flushes, at};
    blk += nb[l];
    at += 2ull * nb[l] * flushes * kRow[l];
  }
  *part_floats = at;
}

}  // namespace

// parameter offsets (canonical layout W[Cout][Cin][3][3], b[Cout] per layer)
constexpr uint32_t kOffW[4] = {0, 2912, 12160, 21408};
constexpr uint32_t kOffB[4] = {2880, 12128, 21376, 21696};
constexpr int kCout[4] = {32, 32, 32, 1};
constexpr int kCin[4] = {10, 32, 32, 32};
constexpr int kCinPad[4] = {16, 32, 32, 32};
constexpr int kCoutPad[4] = {32, 32, 32, 16};

// layers 1-3 stacked for the fused forward pass, layer 4 taps along N
size_t packed_fwd_elems(int l) { return l == 3 ? 16ull * kCinPad[l] : 9ull * kCinPad[l] * kCoutPad[l]; }
size_t packed_bwd_elems(int l) { return 9ull * kCoutPad[l] * kCinPad[l]; }

cudaError_t pack_weights(const float* params, __nv_bfloat16* const wf[4], __nv_bfloat16* const wb[4],
                         cudaStream_t st) {
  for (int l = 0; l < 4; ++l) {
    if (l < 3)
      k_pack_fwd<<<64, 256, 0, st>>>(params + kOffW[l], kCout[l], kCin[l], kCoutPad[l], kCinPad[l], wf[l]);
    else
      k_pack_taps<<<2, 256, 0, st>>>(params + kOffW[l], kCin[l], wf[l]);
    if (l > 0 && wb[l])
      k_pack_bwd<<<64, 256, 0, st>>>(params + kOffW[l], kCout[l], kCin[l], kCoutPad[l], kCinPad[l], wb[l]);
  }
  return cudaGetLastError();
}

namespace {
// feature maps [n_img][H][W][8 chunks] BF16, chunks = 2, or the BCE gradient with
// one (the second is zero fill), as {8 channels, W, chunks, H, images}: one box is
// one row of a strip, in shared memory [chunk][130 pixels]
cudaError_t make_feature_map(CUtensorMap* map, const void* in, uint32_t chunks, uint32_t W, uint32_t H,
                             uint32_t n_img) {
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return cudaErrorNotSupported;
  if (reinterpret_cast<uintptr_t>(in) & 15u) return cudaErrorInvalidValue;
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const cuuint64_t px = 16ull * chunks;
  const cuuint64_t d[5] = {8, W, chunks, H, n_img}, st[4] = {px, 16, px * W, px * W * H};
  const cuuint32_t bx[5] = {8, (cuuint32_t)kFuPx, 2, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(in), d, st, bx, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Segments per strip: a segment of R rows costs R + 2 LAYERS steps (the rows above
// and below it that its first layers recompute), and the CTAs take the segments in
// whole rounds, so the fewest steps over all rounds. Returns the grid.
template <int LAYERS>
int choose_segments(FusedArgs& a, uint32_t W, uint32_t H, uint32_t n_img) {
  a.W = W; a.H = H; a.n_img = n_img;
  a.strips = (W + strip_width<LAYERS>() - 1) / strip_width<LAYERS>();
  uint64_t best = ~0ull;
  const uint64_t strips = (uint64_t)a.strips * n_img, sms = (uint64_t)num_sms();
  for (uint32_t rows = H;;) {
    const uint32_t segs = (H + rows - 1) / rows;
    const uint64_t cost = (strips * segs + sms - 1) / sms * (rows + 2u * LAYERS);
    if (cost < best) { best = cost; a.segs = segs; a.rows = rows; }
    if (rows == 1) break;
    rows = std::min(rows - 1, (H + segs) / (segs + 1));   // one more segment, shorter by a row at least
  }
  return (int)std::min(strips * a.segs, sms);
}

// Dynamic shared memory of a kernel. An attribute of the current device, so set
// before every launch (0.2 us), not once in a process.
template <typename Kernel>
cudaError_t allow_smem(Kernel* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <bool FP8, bool STORE>
cudaError_t launch_fused(const __nv_bfloat16* feat16, FusedArgs& a, uint32_t W, uint32_t H,
                         uint32_t n_img, cudaStream_t st, int* grid_out = nullptr) {
  using Lt = FusedLayout<FP8>;
  // a CTA takes all TMEM columns: more than half of an SM's shared memory, so
  // that no second one can be placed beside it
  constexpr uint32_t smem = Lt::kSmem < 116u * 1024u ? 116u * 1024u : Lt::kSmem;
  CUtensorMap map;
  cudaError_t e = allow_smem(k_net_fused<FP8, STORE>, smem);
  if (e == cudaSuccess) e = make_feature_map(&map, feat16, 2, W, H, n_img);
  if (e != cudaSuccess) return e;
  const int grid = choose_segments<4>(a, W, H, n_img);
  if (grid_out) *grid_out = grid;
  launch_after(k_net_fused<FP8, STORE>, grid, kFuThreads, smem, st, map, a);
  return cudaGetLastError();
}

// gradients of layers 3, 2, 1 (dz[0..2]) from the BCE gradient g8
cudaError_t launch_bwd(const void* g8, __nv_bfloat16* const wb[4], uint32_t* mask,
                       __nv_bfloat16* const dz[3], uint32_t W, uint32_t H, uint32_t* err, cudaStream_t st) {
  constexpr uint32_t smem = FusedLayout<false>::kSmem;
  static_assert(smem > 116u * 1024u, "a CTA takes all TMEM columns: one on an SM");
  CUtensorMap map;
  cudaError_t e = allow_smem(k_bwd_fused, smem);
  if (e == cudaSuccess) e = make_feature_map(&map, g8, 1, W, H, 1);
  if (e != cudaSuccess) return e;
  FusedArgs a = {};
  for (int k = 0; k < 3; ++k) {
    a.w[k] = wb[3 - k];
    a.dz[k] = dz[k];
  }
  a.mask = mask;
  a.err = err;
  const int grid = choose_segments<3>(a, W, H, 1);
  launch_after(k_bwd_fused, grid, kBwThreads, smem, st, map, a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t forward(const __nv_bfloat16* feat16, const float* params, __nv_bfloat16* const wf[4],
                    __nv_bfloat16* const act[3], float* prob, uint32_t W, uint32_t H, uint32_t* err,
                    cudaStream_t st, uint32_t n_img) {
  FusedArgs a = {};
  for (int l = 0; l < 4; ++l) {
    a.w[l] = wf[l];
    a.bias[l] = params + kOffB[l];
    a.out_scale[l] = 1.f;
  }
  a.prob = prob;
  a.err = err;
  if (!act) return launch_fused<false, false>(feat16, a, W, H, n_img, st);
  for (int l = 0; l < 3; ++l) a.act[l] = act[l];
  return launch_fused<false, true>(feat16, a, W, H, n_img, st);
}

cudaError_t pack_weights_fp8(const float* params, const float* const scale[3], uint8_t* const w8[3],
                             cudaStream_t st) {
  for (int l = 1; l < 3; ++l)
    k_pack_fwd_fp8<<<64, 256, 0, st>>>(params + kOffW[l], kCout[l], kCin[l], kCoutPad[l], kCinPad[l],
                                       scale[l - 1], w8[l - 1]);
  k_pack_taps_fp8<<<2, 256, 0, st>>>(params + kOffW[3], kCin[3], scale[2], w8[2]);
  return cudaGetLastError();
}

size_t packed_fp8_bytes(int l) { return packed_fwd_elems(l); }

// the FP8 network: layer 1 in BF16 with E4M3 output, layers 2-4 on E4M3
// operands (kind::f8f6f4)
cudaError_t forward_fp8(const __nv_bfloat16* feat16, const float* params, __nv_bfloat16* const wf[4],
                        uint8_t* const w8[3], const float* const inv[3], const float act_scale[3],
                        float* prob, uint32_t W, uint32_t H, uint32_t* err, cudaStream_t st,
                        uint32_t n_img) {
  FusedArgs a = {};
  for (int l = 0; l < 4; ++l) {
    a.w[l] = l == 0 ? static_cast<const void*>(wf[0]) : w8[l - 1];
    a.bias[l] = params + kOffB[l];
    a.inv[l] = l == 0 ? nullptr : inv[l - 1];
    a.out_scale[l] = l < 3 ? act_scale[l] : 1.f;
  }
  a.prob = prob;
  a.err = err;
  return launch_fused<true, false>(feat16, a, W, H, n_img, st);
}

// raises amax3[l] to the largest value of hidden activation l (the caller
// clears amax3 before the first map it measures)
cudaError_t activation_amax(const __nv_bfloat16* const act[3], uint64_t P, unsigned* amax3,
                            cudaStream_t st) {
  for (int l = 0; l < 3; ++l) k_amax<<<num_sms() * 4, 256, 0, st>>>(act[l], P * 32, amax3 + l);
  return cudaGetLastError();
}

size_t wgrad_part_floats(uint32_t W, uint32_t H) {
  WgradShare share[4];
  uint64_t floats = 0;
  wgrad_shares(W, H, share, &floats);
  return (size_t)floats;
}

int loss_parts() { return 4 * num_sms(); }

// One training step on the mean BCE: forward with its activations kept, data
// gradients of layers 4 to 2, weight gradients of all layers, and the update.
cudaError_t train_step(const __nv_bfloat16* feat16, const float* label, const TrainBuffers& t, uint32_t W,
                       uint32_t H, float lr, uint32_t step, float* grads, uint32_t* err, cudaStream_t st) {
  FusedArgs f = {};
  for (int l = 0; l < 4; ++l) {
    f.w[l] = t.wf[l];
    f.bias[l] = t.params + kOffB[l];
    f.out_scale[l] = 1.f;
  }
  for (int l = 0; l < 3; ++l) f.act[l] = t.act[l];
  f.mask = t.mask;
  f.label = label;
  f.g8 = reinterpret_cast<uint4*>(t.g8);
  f.loss_part = t.loss_part;
  f.err = err;
  int fwd_grid = 0;
  cudaError_t e = launch_fused<false, true>(feat16, f, W, H, 1, st, &fwd_grid);
  if (e == cudaSuccess) e = launch_bwd(t.g8, t.wb, t.mask, t.dz, W, H, err, st);
  if (e != cudaSuccess) return e;

  // weight gradients: layer l + 1 from its input and its data gradient
  WgradArgs g;
  const void* in[4] = {feat16, t.act[0], t.act[1], t.act[2]};
  const void* dz[4] = {t.dz[2], t.dz[1], t.dz[0], t.g8};
  for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
    const uint32_t zc = l == 3 ? 1 : 4;
    e = make_wgrad_map(&g.a[l], in[l], W, H, l == 0 ? 2 : 4, l == 0, kWgW + 2, kWgRows + 2);
    if (e == cudaSuccess) e = make_wgrad_map(&g.z[l], dz[l], W, H, zc, false, kWgW, kWgRows);
  }
  if (e != cudaSuccess) return e;
  uint64_t floats = 0;
  wgrad_shares(W, H, g.share, &floats);
  g.W = W;
  g.H = H;
  g.part = t.wpart;
  g.err = err;
  // the largest layer's stages; one CTA (and its TMEM) per SM
  constexpr size_t smem = std::max(std::max(WgradLayout<2, 4>::kSmem, WgradLayout<4, 4>::kSmem),
                                   std::max(WgradLayout<4, 1>::kSmem, (size_t)116 * 1024));
  const uint32_t grid = g.share[3].blk0 + g.share[3].nblk;
  const bool few = wgrad_tiles(W, H) <= (uint64_t)kWgFewTiles * g.share[1].nblk;
  const auto wgrad = few ? k_wgrad<2> : k_wgrad<4>;
  e = allow_smem(wgrad, smem);
  if (e != cudaSuccess) return e;
  launch_after(wgrad, grid, kWgThreads, smem, st, g);
  // no update from partial sums that were not made
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;

  UpdateArgs u = {};
  uint32_t block = 0;
  for (int l = 0; l < 4; ++l) {
    const uint32_t n = 9u * (uint32_t)(kCout[l] * kCinPad[l]) + (uint32_t)kCout[l];
    u.layer[l] = {block, 2u * g.share[l].nblk * g.share[l].flushes, (uint32_t)kCout[l], (uint32_t)kCin[l],
                  (uint32_t)kCinPad[l], kOffW[l], kOffB[l], g.share[l].part0, t.wf[l], l ? t.wb[l] : nullptr};
    block += (n + 31) / 32;
  }
  u.part = t.wpart;
  u.scale = 1.f / (float)(W * H);
  u.grads = grads;
  u.w = t.params;
  u.v = t.v;
  if (lr > 0.f) u.m = t.m;
  u.lr = lr;
  u.c1 = 1.f - powf(0.9f, (float)step);
  u.c2 = 1.f - powf(0.999f, (float)step);
  u.loss_part = t.loss_part;
  u.n_loss = 4u * (uint32_t)fwd_grid;
  u.loss = t.loss;
  launch_after(k_update, block, 256, 0, st, u);
  return cudaGetLastError();
}

}  // namespace nn
}  // namespace rt
