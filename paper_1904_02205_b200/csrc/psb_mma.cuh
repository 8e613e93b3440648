// Dense contraction on the 5th-generation tensor cores (tcgen05, sm_100a).
//
// acc[m, o] = sum_i X[m, i] * W_k[o, i]  (paper Eq. 1 with Eq. 9 summed over the
// draws) is an integer matrix product: M = output locations, N = output channels,
// K = taps x input channels.  |W_k| needs up to 22 bits, an MMA operand holds 8, so
// W_k is split into P signed 7-bit digit planes, W_k = sum_p D_p * 2^(7p).  One
// tcgen05.mma (kind::i8, s8 x s8 -> s32) of shape 128 x (P*64) x 32 multiplies an
// activation tile with all planes of 64 output channels at once; each plane owns
// 64 accumulator columns in tensor memory (TMEM) and the epilogue recombines them
// exactly (Recombine).
//
// Structure of one CTA (one per SM, persistent over tiles):
//   warps 0-1 producers (one thread each, taking the stages in turns): TMA loads of the activation tile (im2col mode for
//            filters with taps, stride or padding; plain 2-D tiles otherwise) and
//            of the digit-plane tile into a ring of shared-memory stages
//   warp 2 issues the MMAs
//   warp 3 allocates TMEM; issues half of the MMAs in band mode and where a tile is one stage; flips the top bit of
//            unsigned activations; staged outputs: moves shortcut tiles in and output tiles out of shared memory
//   warps 4-19 epilogue: TMEM -> registers, recombine planes, dequantise, bias,
//            shortcut, ReLU, re-quantise, vectorised stores; overlaps the next
//            tile's MMAs through two TMEM accumulator buffers
// Per-location draw counts (Sec. 4.5): the caller sorts the output locations by level and
// gathers the activation rows in that order (psb_sort.cu); every tile then has one level, and
// the epilogue scatters each row back to its location.
// Every wait is bounded; on a timeout the kernel raises the device error word and
// leaves through the common exit that frees TMEM.
#pragma once

#include <cuda.h>

#include <cstring>

#include "psb_common.cuh"

namespace psb {

namespace {

constexpr int kTileM = 128;
constexpr int kProducerWarps = 2;    // one issuing thread each: their barrier waits overlap
constexpr int kMmaWarp0 = kProducerWarps;          // issues the MMAs
constexpr int kMmaWarp1 = kMmaWarp0 + 1;           // band mode: issues half of them; flips unsigned activations; owns the
                                                   // TMEM allocation
constexpr int kFirstEpilogueWarp = kMmaWarp1 + 1;  // a multiple of 4: warp & 3 = TMEM lane quarter
constexpr int kPlaneBars = 4;        // resident digit planes arrive in this many parts, each with its barrier
constexpr int kEpilogueWarps = 16;
constexpr int kThreadsTensor = 32 * (kFirstEpilogueWarp + kEpilogueWarps);   // five warps of 96 registers per scheduler: no room for another
constexpr int kIoSlots = 4;                          // staged outputs: a tile being loaded, two worked on, one stored
constexpr uint32_t kIoTileBytes = kTileM * kTileN;   // a tile of codes: 128 rows x 64 bytes
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemBufStride = 256;
constexpr int kMaxStages = 12;
constexpr uint32_t kResidentMaxBytes = 112 * 1024;          // digit planes kept in shared memory
constexpr size_t kSmemBudget = 227 * 1024;

}  // namespace

struct TmapSet {
  CUtensorMap a;     // activations; the digit planes need none: their tiles are contiguous
  CUtensorMap out, res;   // staged outputs: codes and shortcut as [M][O] bytes, boxes of a tile
};

struct TensorParams {
  ConvArgs a;
  uint32_t M;           // N * OH * OW
  uint32_t m_tiles, o_tiles;
  uint32_t n_cb;        // channel blocks per tap
  uint32_t im2col;      // 1: activation tile through the im2col tensor map
  uint32_t stages;
  uint32_t group;       // K blocks per pipeline stage (one barrier hand-over per group)
  uint32_t stage_bytes_a, stage_bytes_b_max;
  uint32_t planes[kMaxLevels];
  const uint8_t* tile_mask;   // per row tile: levels present (bit l = level l), or null without a map
  uint32_t unit;        // widest store (bytes: 16, 8, 4, 2, 1) that every channels-last output row allows
  uint32_t tail_ksteps; // MMA K steps of a tap's last channel block (the rest of the block lies beyond the channels)
  uint32_t staged;      // 1: codes and shortcut bytes pass through shared memory (epilogue_staged, epilogue_sorted)
  uint32_t flip;        // 1: the activations are unsigned bytes; their top bit is flipped in shared memory (x - 128)
                        // and `corr` restores the sum.  Positions the copy engine fills with zeros become -128, i.e.
                        // x = 0, so padding needs no case of its own
  uint32_t resident;    // 1: the CTA keeps the digit planes of its channel tile in shared memory
  uint32_t ctas_per_otile;
  uint32_t alternate;   // 1: one pipeline stage per tile, and two warps issue the MMAs of alternate tiles
  uint32_t resident_bytes;
  const uint32_t* rowsum256;   // [level][O] row sums of |W_k| in units of 256 (rounded up), or null
  uint32_t amax;        // largest activation magnitude the caller vouches for
  uint32_t real_slots;  // 1: real-valued rows pass through shared memory (epilogue_chunk_real), 2 KB per epilogue warp
  uint32_t mid;         // 1: two digit planes fit 32 bits together (kRecMid)
  const long long* corr[kMaxLevels];  // per-channel integer addend, or null
  const int8_t* planes_ptr[kMaxLevels];  // digit planes: [o_tile][K block][P * 64 rows][BK], pre-swizzled tiles
  // Band mode (stride-1 filters with taps, one channel block, resident planes): a tile is 128
  // consecutive positions of one image's output in "padded-linear" order t = oy * Wp + ox with
  // Wp = W + 2 * pad (positions with ox >= OW are computed and dropped).  In that order the
  // input pixel of tap (kh, kw) for position t is pixel t + kh * Wp + kw of the zero-padded
  // image, so one copy of a band of padded input rows serves every tap: the activation operand
  // of a tap is the same shared-memory band read from a start address moved by
  // (kh * Wp + kw) pixels.  (The swizzle of a K-major operand is a function of the
  // shared-memory address bits, so a start address moved by whole rows reads correctly.)
  uint32_t band;        // 1: band mode
  uint32_t Wp;          // padded row length
  uint32_t tpi;         // tiles per image: ceil(OH * Wp / 128)
  uint32_t band_rows;   // padded input rows per band
  uint32_t band_bytes;  // stage size (band_rows * Wp * C rounded up to 1024)
  // Per-location draw counts: the rows of the activation matrix are sorted by level (psb_sort.cu), every tile
  // has one level (tile_mask holds one bit), and row r of the matrix is output location perm[r]
  const uint32_t* perm;  // or null
  uint32_t Wp_magic, tpi_magic;   // ceil(2^32 / Wp), ceil(2^32 / tpi): quotients by multiply-high (exact in the
                                  // ranges band mode is restricted to)
  unsigned long long wait_limit;  // bound of every wait in SM clocks
};

namespace {

// ---- thin PTX wrappers -------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// What a bounded wait consults on its slow path: the CTA-wide give-up flag and the bound in SM clocks.
struct WaitCtl {
  volatile uint32_t abort;
  uint32_t pad;
  volatile unsigned long long limit;
};

constexpr uint32_t kNoSleep = 0xFFFFFFFFu;   // backoff value of a wait that is about to end: poll without sleeping

// Bounded wait.  Returns false after wc->limit SM clocks without completion, or as soon
// as another thread of the CTA has given up.  (The SM cycle counter is cheap to read.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, WaitCtl* wc,
                                          uint32_t backoff_ns = 0) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    // a thread that has to wait long should not eat the issue slots of the warps doing the
    // arithmetic: poll a few times at full speed, then sleep between polls
    ++spins;
    if (backoff_ns != kNoSleep && (backoff_ns || spins > 4u))
      __nanosleep(backoff_ns ? backoff_ns : (spins > 32u ? 256u : 64u));
    if ((spins & 15u) == 0u) {
      if (wc->abort) return false;
      if ((unsigned long long)(clock64() - t0) > wc->limit) return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}

// Plain bulk copy of a contiguous, 16-byte aligned run of global memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c, int w, int h,
                                            int n) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n)
      : "memory");
}

__device__ __forceinline__ void tma_load_im2col_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                   int c, int w, int h, int n, uint16_t off_w,
                                                   uint16_t off_h) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

// One lane of the (converged) warp.  The MMA role runs with all 32 lanes and lets one of them issue: its addresses are
// then warp-uniform values, which is where the instruction wants its descriptors.  In code that only one lane enters,
// every descriptor word is moved from a vector register first, about 100 clocks per MMA.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0u;
}

// Descriptors given as (low word, high word); `acc` 0 overwrites the accumulator.
__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                          uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The two words of that descriptor.  Only the low word depends on the address (bits 0..13 = address / 16;
// shared memory ends below 2^18, so adding a byte offset / 16 to the low word moves the start address and
// touches nothing else).
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t smem_desc_hi(uint32_t bk) {
  const uint32_t layout = bk == 128 ? 2u : (bk == 64 ? 4u : 6u);
  return ((8u * bk) >> 4) | (1u << 14) | (layout << 29);
}

// Levels (log2 k) of a tile as a bit mask: one byte per row tile, written by the level sort just before the
// contraction kernel (rows are sorted by level, so exactly one bit is set).
__device__ __forceinline__ uint32_t tile_levels(const TensorParams& p, uint32_t m_tile) {
  if (!p.tile_mask) return 1u << p.a.uniform_log2k;
  return (uint32_t)p.tile_mask[m_tile];
}

// Walks the tiles of this CTA without divisions in the loop.  Resident mode: the CTA owns one
// channel tile and strides over the row tiles; streaming mode: tiles are dealt round-robin with
// the channel tile fastest.
struct TileIter {
  uint32_t m_tile, o_tile, step_m, step_o, o_tiles, m_tiles;
  __device__ __forceinline__ void init(const TensorParams& p) {
    o_tiles = p.o_tiles;
    m_tiles = p.m_tiles;
    if (p.resident) {
      o_tile = blockIdx.x / p.ctas_per_otile;
      m_tile = blockIdx.x % p.ctas_per_otile;
      step_m = p.ctas_per_otile;
      step_o = 0;
    } else {
      m_tile = blockIdx.x / p.o_tiles;
      o_tile = blockIdx.x % p.o_tiles;
      step_m = gridDim.x / p.o_tiles;
      step_o = gridDim.x % p.o_tiles;
    }
  }
  __device__ __forceinline__ bool valid() const { return m_tile < m_tiles; }
  __device__ __forceinline__ void next() {
    m_tile += step_m;
    o_tile += step_o;
    if (o_tile >= o_tiles) { o_tile -= o_tiles; ++m_tile; }
  }
};

struct SharedCtl {
  unsigned long long full[kMaxStages];
  unsigned long long empty[kMaxStages];
  unsigned long long acc_full[2];
  unsigned long long acc_empty[2];
  unsigned long long planes_full[kPlaneBars];
  unsigned long long slot_ready[kIoSlots];  // staged outputs: the shortcut tile has landed
  unsigned long long slot_done[kIoSlots];   // the codes of the tile are in the slot
  unsigned long long started[2];        // band mode, per accumulator buffer: the overwriting MMA of the tile has been issued
  unsigned long long flipped[kMaxStages];   // full, and the top bits flipped (unsigned activations)
  uint32_t tmem_base;
  uint32_t rowmax[kMaxLevels];          // largest row sum of |W_k| per level (units of 256), see find_row_maxima
  WaitCtl wait;
  alignas(16) int32_t corr32[kEpilogueWarps][16];   // low words of the integer addends
  alignas(16) float2 scb[kEpilogueWarps][32];   // per epilogue warp: (scale * 2^(e_base - log2 k), bias), read two
                                                // channels (16 bytes) at a time
  long long corr[kEpilogueWarps][32];   // per epilogue warp: integer addend per channel
};

// Output arithmetic of one 16-channel chunk held in registers (v[plane][channel]), common case:
// only re-quantised bytes are wanted.  Same arithmetic as dequant()/requant(), with as few issued
// instructions per output as the definition allows (the output stage of a layer with few input
// channels is bound by instruction issue, and every slot it takes is one the MMA-issuing thread of
// the same scheduler does not get):
//   W32: the accumulator itself is known to stay below 2^31 in magnitude (the sampler keeps the
//        largest row sum of |W_k|, the caller vouches for the largest activation): the planes are
//        recombined in 32 bits (wrap-around in the partial sums is harmless) and one conversion
//        instruction rounds to nearest even, as the 64-bit conversion would.  Otherwise 64-bit
//        recombination plus the per-channel integer addend, converted in two exact halves.  Between the two (Recombine).
//   y = fma(a, sc, bias); optional shortcut fma on a byte converted by the conversion unit.
//   t = y * inv_step, clamped above in fp32; cvt.rni (round half to even, saturating) gives the
//   integer; cvt.pack.sat packs two integers at a time into bytes, saturating to the byte's range.
//   FAST_U8: unsigned codes whose lower bound is 0 (the ReLU, if any, folded into it): the byte
//   saturation is the lower clamp.  Otherwise both clamps are applied in fp32 first.
// How the plane sums of a layer become its accumulators' floats.
//   kRec32:    in 32 bits, see above.  kRec32Add: plus an integer addend per channel (x - 128 fed for unsigned x).
//   kRecMid:   three planes whose lower two fit 32 bits together (the host knows: 16383 x channels and taps x largest byte fed).
//              With t = v0 + 2^7 v1 the accumulator is 2^14 (v2 + (t >> 14)) + (t mod 2^14), the upper part below 2^24 in
//              magnitude: both parts are exact floats and one fma rounds their sum.  2^23 + the lower part is a bit
//              pattern, and the 2^23 is taken off the upper part, as 512.  kRecMidAdd: plus an addend per channel, split alike.
//   kRec64:    everything else.  (Of the networks' layers the classifier of the MobileNet-v2 shape, 1280 inputs with bytes to 255.)
// An output costs a warp about 12 clocks of dispatch beside this; in 32 bits it adds 5, kRecMid 9, in 64 bits 23 (two 64-bit
// multiply-adds, the addend's 64 bits, two conversions).  Maps of five levels, ResNet-50 shape,
// batch 128: 4753 -> 4645 us; MobileNet-v2 shape, 8 bits, batch 64: 1042 -> 1013.
enum Recombine { kRec64, kRec32, kRec32Add, kRecMid, kRecMidAdd };
__host__ __device__ constexpr bool folds_all(int W) { return W == kRec32 || W == kRec32Add; }
__host__ __device__ constexpr bool is_mid(int W) { return W == kRecMid || W == kRecMidAdd; }
__host__ __device__ constexpr bool has_addend(int W) { return W == kRec32Add || W == kRecMidAdd || W == kRec64; }
// The recombinations that an instance of the kernel carries, chosen on the host: kRec32 and kRec64 for two to four planes;
// kRec32 and kRecMid for three whose lower two fit 32 bits; kRec32Add, kRecMidAdd and kRec64 for three with an addend.  (All in
// one instance, codes: 1x1 64 -> 256 @56 batch 16 12.8 -> 13.8 us, 3x3 64 -> 64 @56 batch 32 with a map 32.1 -> 33.2.)
constexpr int kPlainSums = 0, kMidSums = 1, kAddSums = 2;

// A channel's addend as the output loop of the kind wants it in its eight bytes: 64 bits, or two words.
template <int W>
__device__ __forceinline__ long long addend_words(long long c) {
  if (W == kRecMidAdd) return (long long)(((unsigned long long)(uint32_t)((int)(c >> 14) - 512) << 32) | (uint32_t)(c & 0x3FFF));
  return c;
}

struct EpiConst {
  float res_scale, inv_step, lo_f, hi_f;   // lo_f already holds the relu (see the epilogue set-up)
  uint32_t out_signed;
};

// d = bytes (sat(b), sat(a), c.b0, c.b1), saturation to the unsigned / signed byte range
__device__ __forceinline__ uint32_t pack_sat_u8(int a, int b, uint32_t c) {
  uint32_t d;
  asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t pack_sat_s8(int a, int b, uint32_t c) {
  uint32_t d;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// RES: 0 no shortcut, 1 unsigned shortcut bytes, 2 signed ones.
template <int P, int W, int RES, bool FAST_U8>
__device__ __forceinline__ uint4 chunk_math(const uint32_t (&v)[P][16], const uint4& r4, const float2* scb,
                                            const long long* corr, const EpiConst& c) {
  const uint32_t rw[4] = {r4.x, r4.y, r4.z, r4.w};
  const float4* scb2 = reinterpret_cast<const float4*>(scb);   // two channels' (scale, bias) per load
  uint32_t qw[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    int q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = 4 * g + e;
      float af;
      if (folds_all(W)) {
        int acc = (int)v[0][j];
#pragma unroll
        for (int pl = 1; pl < P; ++pl) acc += (int)v[pl][j] << (kDigitBits * pl);
        if (W == kRec32Add) acc += reinterpret_cast<const int2*>(corr)[j].x;
        af = __int2float_rn(acc);
      } else if (is_mid(W)) {          // v[0] = v0 + 2^7 v1 (load_chunk)
        constexpr int top = P > 2 ? 2 : 0;
        int t = (int)v[0][j], hi = (int)v[top][j] - 512;
        if (W == kRecMidAdd) {
          const int2 c2 = reinterpret_cast<const int2*>(corr)[j];
          t += c2.x;
          hi = (int)v[top][j] + c2.y;
        }
        hi += t >> 14;
        af = __fmaf_rn(__int2float_rn(hi), 16384.0f, __uint_as_float(((uint32_t)t & 0x3FFFu) | 0x4B000000u));
      } else {
        long long acc = (long long)(int)v[0][j];
#pragma unroll
        for (int pl = 1; pl < P; ++pl) acc += (long long)(int)v[pl][j] * (long long)(1 << (kDigitBits * pl));
        acc += corr[j];
        af = acc_to_float(acc);
      }
      const float4 sb2 = scb2[j >> 1];
      float y = (j & 1) ? __fmaf_rn(af, sb2.z, sb2.w) : __fmaf_rn(af, sb2.x, sb2.y);
      if (RES == 1) y = __fmaf_rn((float)((rw[g] >> (8 * e)) & 0xFFu), c.res_scale, y);
      if (RES == 2) y = __fmaf_rn((float)(int)(signed char)(rw[g] >> (8 * e)), c.res_scale, y);
      float t = fminf(__fmul_rn(y, c.inv_step), c.hi_f);
      if (!FAST_U8) t = fmaxf(t, c.lo_f);
      q[e] = __float2int_rn(t);
    }
    if (FAST_U8) {
      qw[g] = pack_sat_u8(q[1], q[0], pack_sat_u8(q[3], q[2], 0u));
    } else {
      const uint32_t u = pack_sat_u8(q[1], q[0], pack_sat_u8(q[3], q[2], 0u));
      const uint32_t sg = pack_sat_s8(q[1], q[0], pack_sat_s8(q[3], q[2], 0u));
      qw[g] = c.out_signed ? sg : u;
    }
  }
  return make_uint4(qw[0], qw[1], qw[2], qw[3]);
}

// 16 bytes of a channels-last row.  Rows that are only 8-byte aligned (channel counts that are odd
// multiples of 8) move as two halves; `both` is false for the last 8 channels of such a row.
// The loads are volatile asm so that they stay where they are written (a tile ahead of their use, before
// the wait for the accumulator) instead of being sunk to the first use of the value.  Shortcut bytes are the output of an
// earlier kernel: ordinary loads (the rule at pdl_prologue).
__device__ __forceinline__ uint4 load_row16(const uint8_t* src, bool vec16, bool both) {
  uint4 r = make_uint4(0u, 0u, 0u, 0u);
  if (vec16) {
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(src));
    return r;
  }
  asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(src));
  if (both) asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(r.z), "=r"(r.w) : "l"(src + 8));
  return r;
}
__device__ __forceinline__ void store_row16(uint8_t* dst, uint4 v, bool vec16, bool both) {
  if (vec16) {
    *reinterpret_cast<uint4*>(dst) = v;
  } else {
    *reinterpret_cast<uint2*>(dst) = make_uint2(v.x, v.y);
    if (both) *reinterpret_cast<uint2*>(dst + 8) = make_uint2(v.z, v.w);
  }
}

// The same 16 channels of one output location in a planar ([n][o][oy][ox]) tensor: byte j sits
// j * plane further on.  Lanes of a warp hold consecutive locations, so each of the 16 accesses
// is a contiguous run of 32 bytes per warp.
// (Out of line to keep the callers' loops small.  The registers such a function may use are what all
// of its callers can spare, so each caller family gets its own instance, selected by TAG: when the
// plain output-stage loop, which holds more live values, shared one instance with the band-mode loop,
// the byte loop of the store spilled and band mode with planar output lost a third of its speed.)
template <int TAG>
__device__ __noinline__ uint4 load_planar16(const uint8_t* src, size_t plane, uint32_t count) {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if ((uint32_t)j < count) w[j >> 2] |= (uint32_t)__ldcg(src + (size_t)j * plane) << (8 * (j & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}
template <int TAG>
__device__ __noinline__ void store_planar16(uint8_t* dst, size_t plane, uint32_t count, uint4 v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if ((uint32_t)j < count) dst[(size_t)j * plane] = (uint8_t)(w[j >> 2] >> (8 * (j & 3)));
}

// Channels-last rows whose alignment allows no 8-byte access: loads and stores of `unit` (4, 2 or 1) bytes.
__device__ __noinline__ uint4 load_narrow16(const uint8_t* src, uint32_t unit, uint32_t count) {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (unit == 4u) {
      if ((uint32_t)(4 * j) < count) w[j] = *reinterpret_cast<const uint32_t*>(src + 4 * j);
    } else if (unit == 2u) {
      if ((uint32_t)(4 * j) < count) w[j] = *reinterpret_cast<const uint16_t*>(src + 4 * j);
      if ((uint32_t)(4 * j + 2) < count) w[j] |= (uint32_t)*reinterpret_cast<const uint16_t*>(src + 4 * j + 2) << 16;
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if ((uint32_t)(4 * j + b) < count) w[j] |= (uint32_t)src[4 * j + b] << (8 * b);
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// The stores are warp-collective: every lane brings its row's 16 bytes, and 16 / unit neighbouring lanes write the
// pieces of one row, so that a store instruction covers 2 * unit rows in contiguous 16-byte runs instead of 32 rows
// in single pieces.  `off`: byte offset of the lane's row, negative for a row that is not stored.
__device__ __noinline__ void store_narrow16(uint8_t* base, long long off, uint32_t unit, uint32_t count, uint4 v) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t per_row = 16u / unit, part = lane & (per_row - 1u), at = part * unit;
  const uint32_t shift = (at & 3u) * 8u, word = at >> 2;
  for (uint32_t r0 = 0; r0 < 32u; r0 += 2u * unit) {
    const int row = (int)(r0 + lane / per_row);
    const uint32_t a0 = __shfl_sync(0xFFFFFFFFu, v.x, row), a1 = __shfl_sync(0xFFFFFFFFu, v.y, row);
    const uint32_t a2 = __shfl_sync(0xFFFFFFFFu, v.z, row), a3 = __shfl_sync(0xFFFFFFFFu, v.w, row);
    const long long o = __shfl_sync(0xFFFFFFFFu, off, row);
    const uint32_t d = (word == 0u ? a0 : word == 1u ? a1 : word == 2u ? a2 : a3) >> shift;
    if (o < 0 || at >= count) continue;
    uint8_t* dst = base + o + at;
    if (unit == 4u) *reinterpret_cast<uint32_t*>(dst) = d;
    else if (unit == 2u) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)d;
    else *dst = (uint8_t)d;
  }
}

// The P plane sums of a 16-channel chunk, TMEM -> registers.  With 32-bit recombination the planes are
// folded as they arrive (v0 + 2^7 v1 + ..., what chunk_math computes first anyway): 32 registers at the
// peak instead of 16 P, which is what the loop around it was spilling.  The folded planes are left as
// literal zeros, so the arithmetic after them drops out.
template <int P, int W>
__device__ __forceinline__ void load_chunk(uint32_t taddr, uint32_t (&v)[P][16]) {
  if (P >= 3 && is_mid(W)) {
    tc_ld16(taddr, v[0]);
    tc_ld16(taddr + kTileN, v[1]);
    tc_wait_ld();
    tc_ld16(taddr + 2 * kTileN, v[2]);
#pragma unroll
    for (int j = 0; j < 16; ++j) v[0][j] = (uint32_t)((int)v[0][j] + ((int)v[1][j] << kDigitBits));
    tc_wait_ld();
  } else if (P >= 3 && folds_all(W)) {
    tc_ld16(taddr, v[0]);
    tc_ld16(taddr + kTileN, v[1]);
    tc_wait_ld();
#pragma unroll
    for (int pl = 2; pl < P; ++pl) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        v[0][j] = (uint32_t)((int)v[0][j] + ((int)v[pl - 1][j] << (kDigitBits * (pl - 1))));
        v[pl - 1][j] = 0u;
      }
      tc_ld16(taddr + pl * kTileN, v[pl]);
      tc_wait_ld();
    }
  } else {
#pragma unroll
    for (int pl = 0; pl < P; ++pl) tc_ld16(taddr + pl * kTileN, v[pl]);
    tc_wait_ld();
  }
}

// Integer addend of the 32-bit recombination, added to the lowest plane (the sum is taken modulo 2^32 anyway).
__device__ __forceinline__ void add_corr32(const int32_t* corr32, uint32_t (&v)[16]) {
  const int4* c4 = reinterpret_cast<const int4*>(corr32);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int4 c = c4[g];
    v[4 * g] += (uint32_t)c.x;
    v[4 * g + 1] += (uint32_t)c.y;
    v[4 * g + 2] += (uint32_t)c.z;
    v[4 * g + 3] += (uint32_t)c.w;
  }
}

template <int P, bool W32, int RES>
__device__ __noinline__ void epilogue_chunk_q(uint32_t taddr, bool valid, uint8_t* q_out, size_t off, uint4 r4,
                                              uint32_t unit, uint32_t count, const float2* scb, const long long* corr,
                                              const int32_t* corr32, EpiConst c) {
  uint32_t v[P][16];
  constexpr int W = W32 ? kRec32 : kRec64;
  load_chunk<P, W>(taddr, v);
  if (W32 && corr32) add_corr32(corr32, v[0]);
  const uint4 q = chunk_math<P, W, RES, false>(v, r4, scb, corr, c);
  if (unit < 8u) store_narrow16(q_out, valid ? (long long)off : -1ll, unit, count, q);
  else if (valid) store_row16(q_out + off, q, unit == 16u, count >= 16u);
}

// General output stage: accumulators with any other outputs beside them, and codes that no other loop takes; any layout and
// channel count.
template <int P>
__device__ __noinline__ void epilogue_chunk(const TensorParams& p, uint32_t taddr, uint32_t o_base,
                                            uint32_t m, bool valid, uint32_t n, uint32_t pix,
                                            const float2* scb, const long long* corr, bool use_corr) {
  uint32_t v[P][16];
#pragma unroll
  for (int pl = 0; pl < P; ++pl) tc_ld16(taddr + pl * kTileN, v[pl]);
  tc_wait_ld();
  if (!valid) return;
  const ConvArgs& a = p.a;
  const uint32_t ohow = a.OH * a.OW;
  const bool vec = p.unit == 16u && o_base + 16u <= a.O && !a.out_nchw;
  uint32_t rw[4] = {0, 0, 0, 0};
  if (vec && a.residual) {
    uint4 r4 = *reinterpret_cast<const uint4*>((const uint8_t*)a.residual + (size_t)m * a.O + o_base);
    rw[0] = r4.x; rw[1] = r4.y; rw[2] = r4.z; rw[3] = r4.w;
  }
  uint32_t qw[4] = {0, 0, 0, 0};
#pragma unroll 1
  for (int j = 0; j < 16; ++j) {
    const uint32_t o = o_base + j;
    if (o >= a.O) break;
    long long acc = (long long)(int)v[0][j];
#pragma unroll
    for (int pl = 1; pl < P; ++pl) acc += (long long)(int)v[pl][j] * (long long)(1 << (kDigitBits * pl));
    if (use_corr) acc += corr[j];
    const size_t oidx = a.out_nchw ? ((size_t)n * a.O + o) * ohow + pix : (size_t)m * a.O + o;
    if (a.acc_out) a.acc_out[oidx] = acc;
    if (a.q_out || a.f32_out) {
      int rb = 0;
      if (a.residual) {
        if (vec) rb = (int)((rw[j >> 2] >> (8 * (j & 3))) & 0xFFu);
        else rb = (int)((const uint8_t*)a.residual)[oidx];
        if (a.residual_dtype == PSB_DT_S8) rb = (int)(int8_t)rb;
      }
      const float y = dequant(acc, scb[j].x, scb[j].y, a.residual != nullptr, rb, a.residual_scale, a.relu != 0);
      if (a.f32_out) a.f32_out[oidx] = y;
      if (a.q_out) {
        const int q = requant(y, a.inv_step, a.qmin, a.qmax);
        if (vec) qw[j >> 2] |= ((uint32_t)q & 0xFFu) << (8 * (j & 3));
        else ((uint8_t*)a.q_out)[oidx] = (uint8_t)q;
      }
    }
  }
  if (vec && a.q_out)
    *reinterpret_cast<uint4*>((uint8_t*)a.q_out + (size_t)m * a.O + o_base) = make_uint4(qw[0], qw[1], qw[2], qw[3]);
}

// Real-valued outputs, codes beside them if wanted, any layout and channel count: 16 channels of one location per lane, the same
// arithmetic as dequant() and requant() (the clamp to whole numbers before the rounding instead of after it).  Channels-last rows
// of whole 16-byte pieces pass through a slot of the warp's own in shared memory, so that four lanes store the 64 bytes of
// a row together (a row per lane touches 32 cache lines per instruction).
// us, one output at a time in a rolled loop / so, codes and fp32: 3x3 64->64 @56 batch 32 142 / 27.7 (codes only 11.8), 3x3
// stride 2 120->544 @89 batch 26 519 / 161, 1x1 336->176 planar 38 / 16; fp32 alone, 2048->1000 features, 512 rows 25 / 11.
struct RealOut {
  float* f32;
  uint8_t* q;            // or null
  const uint8_t* res;    // or null
  uint32_t O, ohow, slot;
  bool planar, vec, relu, res_signed;
  float res_scale, inv_step, lo, hi;
  __device__ __forceinline__ RealOut(const TensorParams& p, uint32_t warp_slot) {
    const ConvArgs& a = p.a;
    f32 = a.f32_out; q = (uint8_t*)a.q_out; res = (const uint8_t*)a.residual;
    O = a.O; ohow = a.OH * a.OW; slot = warp_slot;
    planar = a.out_nchw != 0u; vec = p.real_slots != 0u; relu = a.relu != 0u; res_signed = a.residual_dtype == PSB_DT_S8;
    res_scale = a.residual_scale; inv_step = a.inv_step; lo = (float)a.qmin; hi = (float)a.qmax;
  }
  __device__ __forceinline__ size_t offset(uint32_t m, uint32_t o_base) const {
    if (!planar) return (size_t)m * O + o_base;
    const uint32_t n = m / ohow;
    return ((size_t)n * O + o_base) * ohow + (m - n * ohow);
  }
};

// The shortcut bytes of a lane's 16 channels.
__device__ __forceinline__ void load_real_shortcut(const RealOut& r, size_t at, uint32_t count, uint32_t (&rw)[4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    rw[g] = 0u;
    if ((uint32_t)(4 * g) >= count) break;
    if (r.vec) {
      rw[g] = *reinterpret_cast<const uint32_t*>(r.res + at + 4 * g);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if ((uint32_t)(4 * g + e) < count) rw[g] |= (uint32_t)r.res[at + (size_t)(4 * g + e) * (r.planar ? r.ohow : 1u)] << (8 * e);
    }
  }
}

template <int P, int W>
__device__ __forceinline__ void store_real(const RealOut& r, const uint32_t (&v)[P][16], const uint32_t (&rw)[4], uint32_t o_base, uint32_t m,
                                           bool valid, const float2* scb, const long long* corr) {
  const uint32_t count = min(16u, r.O - o_base), lane = threadIdx.x & 31u;
  const size_t at = r.offset(m, o_base), step = r.planar ? r.ohow : 1u;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if ((uint32_t)(4 * g) >= count) break;
    float y[4];
    uint32_t code = 0u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = 4 * g + e;
      float af;
      if (is_mid(W)) {
        const int2 c2 = reinterpret_cast<const int2*>(corr)[j];
        const int t = (int)v[0][j] + c2.x;
        af = __fmaf_rn(__int2float_rn((int)v[P > 2 ? 2 : 0][j] + (t >> 14) + c2.y), 16384.0f,
                       __uint_as_float(((uint32_t)t & 0x3FFFu) | 0x4B000000u));
      } else {
        long long acc = (long long)(int)v[0][j] + corr[j];
#pragma unroll
        for (int pl = 1; pl < P; ++pl) acc += (long long)(int)v[pl][j] * (long long)(1 << (kDigitBits * pl));
        af = __ll2float_rn(acc);
      }
      const float2 sb = scb[j];
      y[e] = __fmaf_rn(af, sb.x, sb.y);
      if (r.res) {
        const uint32_t rb = (rw[g] >> (8 * e)) & 0xFFu;
        y[e] = __fmaf_rn(r.res_signed ? (float)(int)(signed char)rb : (float)rb, r.res_scale, y[e]);
      }
      if (r.relu) y[e] = fmaxf(y[e], 0.0f);
      code |= ((uint32_t)__float2int_rn(fminf(fmaxf(__fmul_rn(y[e], r.inv_step), r.lo), r.hi)) & 0xFFu) << (8 * e);
    }
    if (r.vec) {
      // pieces permuted by the row, against bank conflicts both ways
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(r.slot + lane * 64u + (((uint32_t)g ^ (lane >> 1)) & 3u) * 16u),
                   "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]) : "memory");
      if (r.q && valid) *reinterpret_cast<uint32_t*>(r.q + at + 4 * g) = code;
    } else if (valid) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if ((uint32_t)(4 * g + e) < count) {
          r.f32[at + (size_t)(4 * g + e) * step] = y[e];
          if (r.q) r.q[at + (size_t)(4 * g + e) * step] = (uint8_t)(code >> (8 * e));
        }
    }
  }
  if (r.vec) {
    __syncwarp();
    const uint32_t piece = lane & 3u;
#pragma unroll
    for (uint32_t i = 0; i < 4u; ++i) {
      const uint32_t row = 8u * i + (lane >> 2);
      const uint32_t mm = __shfl_sync(0xFFFFFFFFu, m, (int)row);
      const int ok = __shfl_sync(0xFFFFFFFFu, valid ? 1 : 0, (int)row);
      float4 y;
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w)
                   : "r"(r.slot + row * 64u + ((piece ^ (row >> 1)) & 3u) * 16u) : "memory");
      if (ok && piece * 4u < count) *reinterpret_cast<float4*>(r.f32 + (size_t)mm * r.O + o_base + piece * 4u) = y;
    }
    __syncwarp();
  }
}

// One chunk of the general loop (draw-count maps).
template <int P, int W>
__device__ __noinline__ void epilogue_chunk_real(const TensorParams& p, uint32_t taddr, uint32_t slot, uint32_t o_base, uint32_t m,
                                                 bool valid, const float2* scb, const long long* corr) {
  const RealOut r(p, slot);
  uint32_t v[P][16], rw[4] = {0u, 0u, 0u, 0u};
  load_chunk<P, W>(taddr, v);
  if (r.res && valid) load_real_shortcut(r, r.offset(m, o_base), min(16u, r.O - o_base), rw);
  store_real<P, W>(r, v, rw, o_base, m, valid, scb, corr);
}

// True when the layer takes the specialised epilogue loop below.
__host__ __device__ __forceinline__ bool uniform_epilogue(const TensorParams& p) {
  const ConvArgs& a = p.a;
  const bool q_only = a.q_out && !a.f32_out && !a.acc_out && (p.unit >= 8u || a.out_nchw) && a.inv_step > 0.0f;
  if (a.kmap) {
    // rows sorted by level: the same loop serves if every sampled level has the same number of digit planes
    uint32_t P0 = 0;
    for (uint32_t lv = 0; lv < (uint32_t)kMaxLevels; ++lv)
      if ((a.level_mask >> lv) & 1u) {
        if (P0 && p.planes[lv] != P0) return false;
        P0 = p.planes[lv];
      }
    return p.perm && q_only && P0 >= 2u && P0 <= 4u;
  }
  const uint32_t P0 = p.planes[a.uniform_log2k < (uint32_t)kMaxLevels ? a.uniform_log2k : 0u];
  return q_only && P0 >= 2u && P0 <= 4u;
}

// The same two functions on register copies of the few parameters they need.  Inside an out-of-line
// function the kernel's parameter block is reached through a generic pointer, and every asm statement
// with a memory clobber (barrier waits, TMEM loads) makes the compiler fetch such fields again: a
// dozen dependent loads per tile in the output-stage loop before the copies were made.  (Plain mode.)
struct RowMap {
  static constexpr int kTag = 1;     // distinguishes the row maps in template tags
  uint32_t M, O, ohow, planar;
  __device__ __forceinline__ void init(const TensorParams& p) {
    M = p.M; O = p.a.O; ohow = p.a.OH * p.a.OW; planar = p.a.out_nchw;
  }
  __device__ __forceinline__ uint32_t row_index(uint32_t m_tile, uint32_t row, bool* valid) const {
    const uint32_t m = m_tile * kTileM + row;
    *valid = m < M;
    return m;
  }
  __device__ __forceinline__ size_t offset(uint32_t m, uint32_t o_base) const {
    if (!planar) return (size_t)m * O + o_base;
    const uint32_t n = m / ohow;
    return ((size_t)n * O + o_base) * ohow + (m - n * ohow);
  }
};

// Band mode: rows of a tile are padded-linear positions of one image (tile_row_index above).
struct RowMapBand {
  static constexpr int kTag = 0;
  uint32_t tpi, tpi_magic, Wp, Wp_magic, OH, OW, O, ohow, planar;
  __device__ __forceinline__ void init(const TensorParams& p) {
    tpi = p.tpi; tpi_magic = p.tpi_magic; Wp = p.Wp; Wp_magic = p.Wp_magic;
    OH = p.a.OH; OW = p.a.OW; O = p.a.O; ohow = p.a.OH * p.a.OW; planar = p.a.out_nchw;
  }
  __device__ __forceinline__ uint32_t row_index(uint32_t m_tile, uint32_t row, bool* valid) const {
    const uint32_t n = __umulhi(m_tile, tpi_magic);
    const uint32_t t = (m_tile - n * tpi) * kTileM + row;
    const uint32_t oy = __umulhi(t, Wp_magic), ox = t - oy * Wp;
    *valid = oy < OH && ox < OW;
    return (n * OH + oy) * OW + ox;
  }
  __device__ __forceinline__ size_t offset(uint32_t m, uint32_t o_base) const {
    if (!planar) return (size_t)m * O + o_base;
    const uint32_t n = m / ohow;
    return ((size_t)n * O + o_base) * ohow + (m - n * ohow);
  }
};

// Largest row sum of |W_k| (kept by the sampler in units of 256, each contribution rounded up) of every sampled level the
// call may use, by all epilogue warps together: one warp alone scans 2048 rows in 16 rounds of L2 latency, once per
// level.  (Draw-count maps with five levels, ResNet-50 shape, batch 128: 5541 -> 5512 us.)
__device__ __forceinline__ void find_row_maxima(const TensorParams& p, SharedCtl* ctl, uint32_t levels) {
  const uint32_t et = threadIdx.x - 32u * (uint32_t)kFirstEpilogueWarp;
  for (uint32_t l = 0; l < (uint32_t)kMaxLevels; ++l) {
    if (!((levels >> l) & 1u)) continue;
    const uint32_t* sums = p.rowsum256 + (size_t)l * p.a.O;
    uint32_t best = 0;
#pragma unroll 4
    for (uint32_t o = et; o < p.a.O; o += 32u * (uint32_t)kEpilogueWarps) best = max(best, sums[o]);
    best = __reduce_max_sync(0xFFFFFFFFu, best);
    if ((threadIdx.x & 31u) == 0u && best) atomicMax(&ctl->rowmax[l], best);
  }
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpilogueWarps) : "memory");
}

// Whether the accumulators of level l stay below 2^31 in magnitude: row sum x largest activation magnitude (with an
// integer addend the magnitude before the offset, since the sum that counts is the one after the addend).
__device__ __forceinline__ bool fits_32_bits(const TensorParams& p, const SharedCtl* ctl, uint32_t l) {
  const uint32_t best = ctl->rowmax[l];
  // (a sum that wrapped reads as huge)
  return (unsigned long long)best * 256ull * (unsigned long long)p.amax < (1ull << 31) && best < (1u << 24);
}

// Rows sorted by level (per-location draw counts): row r of the matrix is location perm[r].
struct RowMapSorted {
  static constexpr int kTag = 2;
  const uint32_t* perm;
  uint32_t O, ohow, planar;
  __device__ __forceinline__ void init(const TensorParams& p) {
    perm = p.perm; O = p.a.O; ohow = p.a.OH * p.a.OW; planar = p.a.out_nchw;
  }
  __device__ __forceinline__ uint32_t row_index(uint32_t m_tile, uint32_t row, bool* valid) const {
    const uint32_t m = __ldcg(perm + (size_t)m_tile * kTileM + row);
    *valid = m != 0xFFFFFFFFu;
    return m;
  }
  __device__ __forceinline__ size_t offset(uint32_t m, uint32_t o_base) const {
    if (!planar) return (size_t)m * O + o_base;
    const uint32_t n = m / ohow;
    return ((size_t)n * O + o_base) * ohow + (m - n * ohow);
  }
};

// Epilogue loop of one warp for the common case: one draw count for the whole layer, only
// re-quantised bytes wanted.  The warp owns 32 rows (its TMEM lane quarter) x 16 channels of
// every tile.  Per tile: wait for the accumulator, pull the chunk into registers, hand the TMEM
// buffer back at once (the MMA of the tile after next can start), then do the arithmetic and
// the store.  Shortcut bytes are fetched one tile ahead.  RM maps the rows of a tile to output
// locations (plain tiles or band mode).  Returns true if a wait timed out.
template <int P, int W, int RES, bool FAST_U8, typename RM>
__device__ __noinline__ bool epilogue_uniform(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base,
                                              uint32_t ew, uint32_t lane, EpiConst c) {
  constexpr bool HAS_RES = RES != 0;
  // every instance of this loop gets its own instance of the out-of-line planar helpers (see load_planar16)
  constexpr int TAG = (((P * 5 + W) * 3 + RES) * 2 + (FAST_U8 ? 1 : 0)) * 3 + RM::kTag;
  const ConvArgs& a = p.a;
  const uint32_t quarter = ew & 3u, sub = ew >> 2;
  const uint32_t row = quarter * 32u + lane;
  constexpr bool kSorted = RM::kTag == 2;      // one level per tile, taken from the tile's mask
  uint32_t l = a.uniform_log2k;
  const bool use_corr = p.corr[kSorted ? (uint32_t)__ffs((int)(a.level_mask & 0x7Fu)) - 1u : l] != nullptr;
  WaitCtl* abort = &ctl->wait;
  const uint8_t* const res_base = (const uint8_t*)a.residual;
  uint8_t* const q_base = (uint8_t*)a.q_out;
  RM rm;
  rm.init(p);
  const float2* scb = ctl->scb[ew];
  const long long* corr = ctl->corr[ew];
  const bool vec16 = p.unit == 16u, planar = rm.planar != 0u;
  const uint32_t ohow = rm.ohow;
  TileIter ti;
  ti.init(p);
  uint32_t pass = 0, cur_o_tile = 0xFFFFFFFFu;
  uint4 r_next = make_uint4(0, 0, 0, 0);
  // Sorted rows: the location of this thread's row and the tile's level are lookups in global memory.  They are
  // made one tile ahead (nx_*) and the shortcut fetch of the next tile, whose address depends on them, is issued
  // after the accumulator wait instead of before it, so that no address waits for a lookup.
  // (Without a shortcut nothing but the final store depends on the row's location, and looking ahead only
  // costs registers: measured slower.)
  constexpr bool kAhead = kSorted && HAS_RES;
  uint32_t nx_m = 0, nx_levels = 0;
  bool nx_ok = false;
  if (kSorted && ti.valid()) {
    if (kAhead) nx_m = rm.row_index(ti.m_tile, row, &nx_ok);
    nx_levels = tile_levels(p, ti.m_tile);
  }
  if (HAS_RES && ti.valid()) {
    bool ok_row;
    uint32_t m = nx_m;
    if (kAhead) ok_row = nx_ok; else m = rm.row_index(ti.m_tile, row, &ok_row);
    const uint32_t ob = ti.o_tile * kTileN + sub * 16u;
    if (ok_row && ob < rm.O) {
      const uint8_t* src = res_base + rm.offset(m, ob);
      r_next = planar ? load_planar16<TAG>(src, ohow, rm.O - ob) : load_row16(src, vec16, ob + 16u <= rm.O);
    }
  }
  while (ti.valid()) {
    bool row_valid = nx_ok;
    uint32_t m = nx_m;
    if (!kAhead) m = rm.row_index(ti.m_tile, row, &row_valid);
    const uint32_t o_tile = ti.o_tile;
    const uint32_t o_base = o_tile * kTileN + sub * 16u;
    const bool active = o_base < rm.O;          // warp-uniform
    if (kSorted) {
      // the tile's level; a tile without a sampled level gets no pass from the other roles either
      const uint32_t levels = nx_levels;
      if (!(levels & a.level_mask & 0x7Fu)) {
        if (row_valid) atomicOr(a.err, kDevErrBadLevel);     // a location asks for a level that was not sampled
        ti.next();
        if (ti.valid()) {
          if (kAhead) nx_m = rm.row_index(ti.m_tile, row, &nx_ok);
          nx_levels = tile_levels(p, ti.m_tile);
        }
        if (HAS_RES && ti.valid()) {
          const bool ok_row = nx_ok;
          const uint32_t mn = nx_m, ob = ti.o_tile * kTileN + sub * 16u;
          r_next = make_uint4(0, 0, 0, 0);
          if (ok_row && ob < rm.O) {
            const uint8_t* src = res_base + rm.offset(mn, ob);
            r_next = planar ? load_planar16<TAG>(src, ohow, rm.O - ob) : load_row16(src, vec16, ob + 16u <= rm.O);
          }
        }
        continue;
      }
      l = (uint32_t)__ffs((int)(levels & a.level_mask & 0x7Fu)) - 1u;
    }
    ti.next();
    if (kSorted && ti.valid()) {
      if (kAhead) nx_m = rm.row_index(ti.m_tile, row, &nx_ok);
      nx_levels = tile_levels(p, ti.m_tile);
    }
    if ((kSorted ? o_tile * 8u + l : o_tile) != cur_o_tile) {
      // per-channel constants of this channel tile: the warp keeps its own copy of its 16 channels
      __syncwarp();
      if (lane < 16u) {
        const uint32_t o = o_base + lane;
        float2 sb = make_float2(0.f, 0.f);
        long long cr = 0;
        if (o < a.O) {
          sb.x = ldexpf(a.scale[o], a.e_base[o] - (int)l);
          sb.y = a.bias[o];
          if (use_corr) cr = p.corr[l][o];
        }
        ctl->scb[ew][lane] = sb;
        // (also where nothing reads it: without the store 1x1 64 -> 256 @56 batch 16 took 13.3 us, not 12.6, by the compiler's schedule)
        ctl->corr[ew][lane] = addend_words<W>(cr);
      }
      cur_o_tile = kSorted ? o_tile * 8u + l : o_tile;
      __syncwarp();
    }
    const uint4 r_cur = r_next;
    if (HAS_RES && !kAhead && ti.valid()) {
      bool ok_row;
      const uint32_t mn = rm.row_index(ti.m_tile, row, &ok_row), ob = ti.o_tile * kTileN + sub * 16u;
      r_next = make_uint4(0, 0, 0, 0);
      if (ok_row && ob < rm.O) {
        const uint8_t* src = res_base + rm.offset(mn, ob);
        r_next = planar ? load_planar16<TAG>(src, ohow, rm.O - ob) : load_row16(src, vec16, ob + 16u <= rm.O);
      }
    }
    const uint32_t buf = pass & 1u, aph = (pass >> 1) & 1u;
    const bool ok = mbar_wait(smem_u32(&ctl->acc_full[buf]), aph, abort, 32);
    if (__any_sync(0xFFFFFFFFu, !ok)) return true;
    tc_fence_after();
    uint32_t v[P][16];
    if (active) {
      const uint32_t taddr = tmem_base + buf * kTmemBufStride + ((quarter * 32u) << 16) + sub * 16u;
      load_chunk<P, W>(taddr, v);
    }
    // the chunk is in registers: give the accumulator buffer back before doing the arithmetic
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[buf]));
    if (kAhead && ti.valid()) {
      const uint32_t ob = ti.o_tile * kTileN + sub * 16u;
      r_next = make_uint4(0, 0, 0, 0);
      if (nx_ok && ob < rm.O) {
        const uint8_t* src = res_base + rm.offset(nx_m, ob);
        r_next = planar ? load_planar16<TAG>(src, ohow, rm.O - ob) : load_row16(src, vec16, ob + 16u <= rm.O);
      }
    }
    if (active && row_valid) {
      const uint4 q16 = chunk_math<P, W, RES, FAST_U8>(v, r_cur, scb, corr, c);
      uint8_t* dst = q_base + rm.offset(m, o_base);
      if (planar) store_planar16<TAG>(dst, ohow, rm.O - o_base, q16);
      else store_row16(dst, q16, vec16, o_base + 16u <= rm.O);
    }
    ++pass;
  }
  return false;
}

// The loop for real-valued outputs under one draw count: as epilogue_uniform, the accumulator handed back before the arithmetic.
// Inlined into its instance: out of line, four planes spill 552 bytes and not 196 (1x1 64 -> 256 @56 batch 16 planar, k = 64,
// 54.0 -> 38.0 us).
template <int P, int W>
__device__ __forceinline__ bool epilogue_real(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t slots_addr,
                                           uint32_t ew, uint32_t lane) {
  const ConvArgs& a = p.a;
  const RealOut r(p, slots_addr + ew * 2048u);
  const uint32_t quarter = ew & 3u, sub = ew >> 2, row = quarter * 32u + lane, l = a.uniform_log2k, M = p.M;
  const bool use_corr = p.corr[l] != nullptr;
  WaitCtl* abort = &ctl->wait;
  const float2* scb = ctl->scb[ew];
  const long long* corr = ctl->corr[ew];
  TileIter ti;
  ti.init(p);
  uint32_t pass = 0, cur_o_tile = 0xFFFFFFFFu;
  while (ti.valid()) {
    const uint32_t m = ti.m_tile * kTileM + row, o_tile = ti.o_tile, o_base = o_tile * kTileN + sub * 16u;
    const bool valid = m < M, active = o_base < r.O;
    ti.next();
    if (o_tile != cur_o_tile) {
      // per-channel constants of this channel tile: the warp keeps its own copy of its 16 channels
      __syncwarp();
      if (lane < 16u) {
        const uint32_t o = o_base + lane;
        float2 sb = make_float2(0.f, 0.f);
        long long cr = 0;
        if (o < r.O) {
          sb.x = ldexpf(a.scale[o], a.e_base[o] - (int)l);
          sb.y = a.bias[o];
          if (use_corr) cr = p.corr[l][o];
        }
        ctl->scb[ew][lane] = sb;
        ctl->corr[ew][lane] = addend_words<W>(cr);
      }
      cur_o_tile = o_tile;
      __syncwarp();
    }
    uint32_t rw[4] = {0u, 0u, 0u, 0u};
    if (r.res && valid && active) load_real_shortcut(r, r.offset(m, o_base), min(16u, r.O - o_base), rw);
    const uint32_t buf = pass & 1u, aph = (pass >> 1) & 1u;
    const bool ok = mbar_wait(smem_u32(&ctl->acc_full[buf]), aph, abort, 32);
    if (__any_sync(0xFFFFFFFFu, !ok)) return true;
    tc_fence_after();
    uint32_t v[P][16];
    if (active) load_chunk<P, W>(tmem_base + buf * kTmemBufStride + ((quarter * 32u) << 16) + sub * 16u, v);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[buf]));
    if (active) store_real<P, W>(r, v, rw, o_base, m, valid, scb, corr);
    ++pass;
  }
  return false;
}

// 16 channels with the planes recombined in 32 bits.
template <int P>
__device__ __forceinline__ void load_folded(uint32_t taddr, uint32_t (&a)[1][16]) {
  uint32_t v[P][16];
#pragma unroll
  for (int pl = 0; pl < P; ++pl) tc_ld16(taddr + pl * kTileN, v[pl]);
  tc_wait_ld();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    int acc = (int)v[0][j];
#pragma unroll
    for (int pl = 1; pl < P; ++pl) acc += (int)v[pl][j] << (kDigitBits * pl);
    a[0][j] = (uint32_t)acc;
  }
}

// The loop for layers with a shortcut and several tiles per CTA, channels-last rows of whole 16-byte pieces in tile order (p.staged).
// Two things differ.  Codes and shortcut bytes pass through slots of shared memory, moved as one box per tile by the
// copy engine (io_role): direct accesses, 16 bytes of a different row per lane, cost 32 cache-line look-ups and half-used
// sectors per instruction.  And the sixteen warps form two groups that take alternate tiles, each with the accumulator
// buffer of its parity, a warp taking 32 rows x 32 channels, so that the bookkeeping of a tile is spent on twice as many
// outputs.  1x1 64 -> 256 channels @56 with a shortcut, batch 64: 55.4 -> 40.3 us (staged without the groups 48.4; 17.7 us
// at memory rate).
template <int P, int W, int RES, bool FAST_U8>
__device__ __noinline__ bool epilogue_staged(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t slots_addr,
                                             uint32_t ew, uint32_t lane, EpiConst c) {
  const ConvArgs& a = p.a;
  const uint32_t quarter = ew & 3u, half = (ew >> 2) & 1u, group = ew >> 3, row = quarter * 32u + lane;
  const uint32_t l = a.uniform_log2k, O = a.O;
  const bool use_corr = p.corr[l] != nullptr;
  WaitCtl* abort = &ctl->wait;
  const float2* scb = ctl->scb[ew];
  const long long* corr = ctl->corr[ew];
  // this lane's two 16-byte pieces of a slot: rows of 64 bytes, pieces permuted by the copy engine's 64-byte swizzle
  const uint32_t sw = (row >> 1) & 3u, row_addr = slots_addr + group * kIoTileBytes + row * (uint32_t)kTileN;
  const uint32_t piece[2] = {((2u * half) ^ sw) << 4, ((2u * half + 1u) ^ sw) << 4};
  const uint32_t ready0 = smem_u32(&ctl->slot_ready[group]), done0 = smem_u32(&ctl->slot_done[group]);
  const uint32_t acc_full = smem_u32(&ctl->acc_full[group]), acc_empty = smem_u32(&ctl->acc_empty[group]);
  const uint32_t taddr = tmem_base + group * kTmemBufStride + ((quarter * 32u) << 16) + half * 32u;
  TileIter ti;
  ti.init(p);
  if (group) ti.next();
  uint32_t n = 0, cur_o_tile = 0xFFFFFFFFu;      // n: tiles of this group so far; their slots alternate
  while (ti.valid()) {
    const uint32_t o_tile = ti.o_tile, o_base = o_tile * kTileN + half * 32u;
    const bool active = o_base < O;             // warp-uniform
    ti.next();
    ti.next();
    if (o_tile != cur_o_tile) {
      // per-channel constants of this channel tile: the warp keeps its own copy of its 32 channels
      __syncwarp();
      const uint32_t o = o_base + lane;
      float2 sb = make_float2(0.f, 0.f);
      long long cr = 0;
      if (o < O) {
        sb.x = ldexpf(a.scale[o], a.e_base[o] - (int)l);
        sb.y = a.bias[o];
        if (use_corr) cr = p.corr[l][o];
      }
      ctl->scb[ew][lane] = sb;
      // (also where nothing reads it, as in epilogue_uniform: 1x1 64 -> 256 @56 with a shortcut, batch 64, 41.2 -> 40.8 us)
      ctl->corr[ew][lane] = addend_words<W>(cr);
      cur_o_tile = o_tile;
      __syncwarp();
    }
    bool ok = mbar_wait(acc_full, n & 1u, abort, 32);
    if (__any_sync(0xFFFFFFFFu, !ok)) return true;
    tc_fence_after();
    const uint32_t slot = (n & 1u) * 2u, addr = row_addr + slot * kIoTileBytes;
    auto release = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    };
    auto shortcut = [&](uint32_t at) {
      uint4 r;
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(at));
      return r;
    };
    auto store = [&](uint32_t at, uint4 q) {
      asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w) : "memory");
    };
    if (folds_all(W)) {
      uint32_t a0[1][16], a1[1][16];
      if (active) {
        load_folded<P>(taddr, a0);
        load_folded<P>(taddr + 16u, a1);
      }
      release();
      ok = mbar_wait(ready0 + 8u * slot, (n >> 1) & 1u, abort, 32);
      if (__any_sync(0xFFFFFFFFu, !ok)) return true;
      if (active) {
        store(addr + piece[0], chunk_math<1, W, RES, FAST_U8>(a0, shortcut(addr + piece[0]), scb, corr, c));
        store(addr + piece[1], chunk_math<1, W, RES, FAST_U8>(a1, shortcut(addr + piece[1]), scb + 16, corr + 16, c));
      }
    } else {
      ok = mbar_wait(ready0 + 8u * slot, (n >> 1) & 1u, abort, 32);
      if (__any_sync(0xFFFFFFFFu, !ok)) return true;
      uint32_t v[P][16];
      if (active) {
        load_chunk<P, W>(taddr, v);
        store(addr + piece[0], chunk_math<P, W, RES, FAST_U8>(v, shortcut(addr + piece[0]), scb, corr, c));
        load_chunk<P, W>(taddr + 16u, v);
      }
      release();
      if (active) store(addr + piece[1], chunk_math<P, W, RES, FAST_U8>(v, shortcut(addr + piece[1]), scb + 16, corr + 16, c));
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(done0 + 8u * slot);
    ++n;
  }
  return false;
}

// The loop for rows sorted by level (per-location draw counts), several tiles per CTA, rows of whole 16-byte pieces: the
// two groups of warps of epilogue_staged, but the rows of a tile lie anywhere in the tensors, so every warp moves its own
// 32 rows x 32 bytes, two lanes per row (whole sectors, 16 cache lines per instruction instead of 32): the shortcut of its
// next tile into a slot of its own by asynchronous copies, the codes from the slot to the tensor.  Bound
// by instruction issue and by L2 sectors; with a row per lane, every load and store touched 32 lines for 16 bytes each (ResNet-50 shape, batch 128, maps of five levels: 5401 -> 4853 us, layers with a shortcut and
// without; its attention mode, batch 32 in the second pass: 3109 -> 2980 us).
template <int P, int W, int RES, bool FAST_U8>
__device__ __noinline__ bool epilogue_sorted(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t slots_addr,
                                             uint32_t ew, uint32_t lane, EpiConst c) {
  const ConvArgs& a = p.a;
  const uint32_t quarter = ew & 3u, half = (ew >> 2) & 1u, group = ew >> 3, row = quarter * 32u + lane;
  const uint32_t O = a.O, sampled = a.level_mask & 0x7Fu;
  const bool use_corr = p.corr[(uint32_t)__ffs((int)sampled) - 1u] != nullptr;
  WaitCtl* abort = &ctl->wait;
  const float2* scb = ctl->scb[ew];
  const long long* corr = ctl->corr[ew];
  const uint8_t* const res_base = (const uint8_t*)a.residual;
  uint8_t* const q_base = (uint8_t*)a.q_out;
  const uint32_t* const perm = p.perm;
  // two slots of 32 rows x 32 bytes; the pieces of rows 4 .. 7 of every eight are swapped, so that neither the accesses
  // of a row per lane nor those of two lanes per row conflict
  const uint32_t my_slots = slots_addr + ew * 2048u;
  const uint32_t sw = (lane >> 2) & 1u, own[2] = {lane * 32u + (sw << 4), lane * 32u + ((sw ^ 1u) << 4)};
  const uint32_t r_mov = lane >> 1, piece = lane & 1u;       // moved rows r_mov and r_mov + 16, this 16-byte piece
  const uint32_t mov = r_mov * 32u + ((piece ^ ((r_mov >> 2) & 1u)) << 4);      // (+ 512 for the second row: same swap)
  const uint32_t acc_full = smem_u32(&ctl->acc_full[group]), acc_empty = smem_u32(&ctl->acc_empty[group]);
  const uint32_t taddr = tmem_base + group * kTmemBufStride + ((quarter * 32u) << 16) + half * 32u;
  TileIter ti;
  ti.init(p);
  uint32_t n = 0, cur_key = 0xFFFFFFFFu;
  uint32_t nx_m = 0xFFFFFFFFu, nx_levels = 0;
  auto levels_of = [&](const TileIter& t) { return t.valid() ? tile_levels(p, t.m_tile) : 0u; };
  // Moves ti from tile `pass` of those that run (a level was sampled) to tile `to`, one step at a time; locations on the
  // way that ask for a level that was not sampled are reported.
  auto walk = [&](uint32_t pass, uint32_t to, uint32_t levels) {
    while (levels && (!(levels & sampled) || pass != to)) {
      if (levels & sampled) ++pass;
      else if (__ldcg(perm + (size_t)ti.m_tile * kTileM + row) != 0xFFFFFFFFu) atomicOr(a.err, kDevErrBadLevel);
      ti.next();
      levels = levels_of(ti);
    }
    nx_levels = levels;
  };
  auto look_ahead = [&]() { nx_m = nx_levels ? __ldcg(perm + (size_t)ti.m_tile * kTileM + row) : 0xFFFFFFFFu; };
  auto advance = [&]() {                        // the next tile of this group: two on, as a rule
    TileIter t1 = ti, t2;
    t1.next();
    t2 = t1;
    t2.next();
    const uint32_t l1 = levels_of(t1), l2 = levels_of(t2);
    if ((l1 & sampled) && (l2 & sampled)) {
      ti = t2;
      nx_levels = l2;
    } else {
      ti = t1;
      walk(0u, 1u, l1);
    }
    look_ahead();
  };
  walk(0u, group, levels_of(ti));
  auto fetch_shortcut = [&](uint32_t slot) {        // of the tile at ti, into the warp's slot
    const uint32_t ob = ti.o_tile * kTileN + half * 32u + piece * 16u;
#pragma unroll
    for (uint32_t i = 0; i < 2u; ++i) {
      const uint32_t m = __shfl_sync(0xFFFFFFFFu, nx_m, (int)(r_mov + 16u * i));
      if (m != 0xFFFFFFFFu && ob < O)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(my_slots + slot * 1024u + mov + 512u * i),
                     "l"(res_base + (size_t)m * O + ob) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  look_ahead();
  if (RES) fetch_shortcut(0u);
  while (nx_levels) {
    const uint32_t o_tile = ti.o_tile, o_base = o_tile * kTileN + half * 32u, m = nx_m;
    const uint32_t l = (uint32_t)__ffs((int)(nx_levels & sampled)) - 1u;
    const bool active = o_base < O;             // warp-uniform
    advance();
    if (o_tile * 8u + l != cur_key) {
      // per-channel constants of this channel tile and level: the warp keeps its own copy of its 32 channels
      __syncwarp();
      const uint32_t o = o_base + lane;
      float2 sb = make_float2(0.f, 0.f);
      long long cr = 0;
      if (o < O) {
        sb.x = ldexpf(a.scale[o], a.e_base[o] - (int)l);
        sb.y = a.bias[o];
        if (has_addend(W) && use_corr) cr = p.corr[l][o];
      }
      ctl->scb[ew][lane] = sb;
      if (has_addend(W)) ctl->corr[ew][lane] = addend_words<W>(cr);
      cur_key = o_tile * 8u + l;
      __syncwarp();
    }
    const bool ok = mbar_wait(acc_full, n & 1u, abort, 32);
    if (__any_sync(0xFFFFFFFFu, !ok)) return true;
    tc_fence_after();
    const uint32_t slot_addr = my_slots + (n & 1u) * 1024u;
    auto release = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    };
    auto shortcut = [&](uint32_t at) {
      uint4 r = make_uint4(0u, 0u, 0u, 0u);
      if (RES) asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(at) : "memory");
      return r;
    };
    auto put = [&](uint32_t at, uint4 q) {
      asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w) : "memory");
    };
    // Every lane has read the other slot's codes (the barrier orders those reads before the copies): the next tile's
    // shortcut may come in.
    auto arrive_shortcut = [&]() {
      if (!RES) return;
      __syncwarp();
      fetch_shortcut((n & 1u) ^ 1u);
      asm volatile("cp.async.wait_group 1;" ::: "memory");       // this tile's
      __syncwarp();
    };
    if (folds_all(W)) {
      uint32_t a0[1][16], a1[1][16];
      if (active) {
        load_folded<P>(taddr, a0);
        load_folded<P>(taddr + 16u, a1);
      }
      release();
      arrive_shortcut();
      if (active) {
        put(slot_addr + own[0], chunk_math<1, W, RES, FAST_U8>(a0, shortcut(slot_addr + own[0]), scb, corr, c));
        put(slot_addr + own[1], chunk_math<1, W, RES, FAST_U8>(a1, shortcut(slot_addr + own[1]), scb + 16, corr + 16, c));
      }
    } else {
      arrive_shortcut();
      uint32_t v[P][16];
      if (active) {
        load_chunk<P, W>(taddr, v);
        put(slot_addr + own[0], chunk_math<P, W, RES, FAST_U8>(v, shortcut(slot_addr + own[0]), scb, corr, c));
        load_chunk<P, W>(taddr + 16u, v);
      }
      release();
      if (active) put(slot_addr + own[1], chunk_math<P, W, RES, FAST_U8>(v, shortcut(slot_addr + own[1]), scb + 16, corr + 16, c));
    }
    __syncwarp();
#pragma unroll
    for (uint32_t i = 0; i < 2u; ++i) {
      const uint32_t mm = __shfl_sync(0xFFFFFFFFu, m, (int)(r_mov + 16u * i)), ob = o_base + piece * 16u;
      uint4 q;
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                   : "r"(slot_addr + mov + 512u * i) : "memory");
      if (mm != 0xFFFFFFFFu && ob < O) *reinterpret_cast<uint4*>(q_base + (size_t)mm * O + ob) = q;
    }
    ++n;
  }
  if (RES) asm volatile("cp.async.wait_group 0;" ::: "memory");
  return false;
}

// One thread moves the tiles of epilogue_staged: the shortcuts of up to three tiles ahead in, the codes out.  Rows and channels
// beyond the tensor read as zeros and are not written.
__device__ __noinline__ bool io_role(const TensorParams& p, const TmapSet& maps, SharedCtl* ctl, uint32_t slots_addr) {
  TileIter out, in;
  out.init(p);
  in.init(p);
  auto prepare = [&](uint32_t slot) {
    if (!in.valid()) return;
    const uint32_t bar = smem_u32(&ctl->slot_ready[slot]);
    mbar_expect_tx(bar, kIoTileBytes);
    tma_load_2d(slots_addr + slot * kIoTileBytes, &maps.res, bar, (int)(in.o_tile * kTileN), (int)(in.m_tile * kTileM));
    in.next();
  };
  prepare(0u);
  prepare(1u);
  prepare(2u);
  bool ok = true;
  uint32_t slot = 0, phase = 0;
  for (; out.valid(); out.next()) {
    ok = mbar_wait(smem_u32(&ctl->slot_done[slot]), phase, &ctl->wait);
    if (!ok) break;
    tma_store_2d(&maps.out, slots_addr + slot * kIoTileBytes, (int)(out.o_tile * kTileN), (int)(out.m_tile * kTileM));
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    // all but this store have read their slots: the one of the tile before is free
    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
    prepare((slot + (uint32_t)kIoSlots - 1u) % (uint32_t)kIoSlots);
    if (++slot == (uint32_t)kIoSlots) { slot = 0; phase ^= 1u; }
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  return !ok;
}

// Run-time options of the uniform output stage -> template instance.
struct EpiChoice {
  bool fast_u8;
  uint32_t res;       // 0 no shortcut, 1 unsigned, 2 signed bytes
  bool fits, mid;     // the sums fit 32 bits (and, in kPlainSums, have no addend); p.mid
};
template <int P, int W, int RES, bool kSorted>
__device__ __forceinline__ bool uniform_dispatch_tail(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base,
                                                      uint32_t slots_addr, uint32_t ew, uint32_t lane, const EpiConst& c,
                                                      bool fast_u8) {
  // An addend comes with flipped activations, which are never in band mode and never staged in tile order, or with the gathered
  // rows of a flat K axis, which are never in band mode but may be staged.
  constexpr bool kAddend = W == kRec32Add || W == kRecMidAdd;
  if constexpr (kSorted) {
    if (p.staged)
      return fast_u8 ? epilogue_sorted<P, W, RES, true>(p, ctl, tmem_base, slots_addr, ew, lane, c)
                     : epilogue_sorted<P, W, RES, false>(p, ctl, tmem_base, slots_addr, ew, lane, c);
    return fast_u8 ? epilogue_uniform<P, W, RES, true, RowMapSorted>(p, ctl, tmem_base, ew, lane, c)
                   : epilogue_uniform<P, W, RES, false, RowMapSorted>(p, ctl, tmem_base, ew, lane, c);
  }
  if (RES && p.staged)
    return fast_u8 ? epilogue_staged<P, W, RES ? RES : 1, true>(p, ctl, tmem_base, slots_addr, ew, lane, c)
                   : epilogue_staged<P, W, RES ? RES : 1, false>(p, ctl, tmem_base, slots_addr, ew, lane, c);
  if constexpr (!kAddend) {
    if (p.band)
      return fast_u8 ? epilogue_uniform<P, W, RES, true, RowMapBand>(p, ctl, tmem_base, ew, lane, c)
                     : epilogue_uniform<P, W, RES, false, RowMapBand>(p, ctl, tmem_base, ew, lane, c);
  }
  return fast_u8 ? epilogue_uniform<P, W, RES, true, RowMap>(p, ctl, tmem_base, ew, lane, c)
                 : epilogue_uniform<P, W, RES, false, RowMap>(p, ctl, tmem_base, ew, lane, c);
}
template <int P, int W, bool kSorted>
__device__ __forceinline__ bool uniform_dispatch_res(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t slots_addr,
                                                     uint32_t ew, uint32_t lane, const EpiConst& c, const EpiChoice& how) {
  if (how.res == 0u) return uniform_dispatch_tail<P, W, 0, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how.fast_u8);
  if (how.res == 1u) return uniform_dispatch_tail<P, W, 1, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how.fast_u8);
  return uniform_dispatch_tail<P, W, 2, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how.fast_u8);
}
template <int P, int kRec, bool kSorted>
__device__ __forceinline__ bool uniform_dispatch(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t slots_addr,
                                                 uint32_t ew, uint32_t lane, const EpiConst& c, const EpiChoice& how) {
  constexpr int kSmall = kRec == kAddSums ? kRec32Add : kRec32;
  constexpr int kLarge = kRec == kAddSums ? kRecMidAdd : kRec == kMidSums ? kRecMid : kRec64;
  if (how.fits) return uniform_dispatch_res<P, kSmall, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how);
  if constexpr (kRec == kAddSums)
    if (!how.mid) return uniform_dispatch_res<P, kRec64, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how);
  return uniform_dispatch_res<P, kLarge, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, c, how);
}

// All lanes of the warp wait together; false when a wait ran out.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, WaitCtl* wc) {
  return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, wc, kNoSleep)) != 0;
}

// The MMA issuing role: one warp, inlined into the kernel so that its parameters come from the constant bank and its
// addresses stay uniform.  Two single threads taking turns, out of line, as there were before, needed 100 to 250 clocks
// per MMA and hand-overs between them (K block of 4 MMAs, streamed planes, 3x3 256 -> 256 channels: 753 -> 640 clocks;
// the copies of a K block, 40 KB at the 68 bytes per clock and SM that L2 delivers to all SMs at once, take 600).
// Tiles of a single stage alternate between two warps (p.alternate): what a warp does per tile beside its MMAs (waits,
// descriptors, commits) takes about 1300 clocks, more than the tile's copies: 1x1 96 -> 16 channels
// @112, batch 64: 34.6 -> 27.7 us, 256 -> 64 @56 13.7 -> 12.4.  (Not with staged outputs, where that warp moves the tiles:
// one producer warp for both was slower, 40.2 -> 45.1 us on 64 -> 256 @56 with a shortcut.)
// Returns true on a timeout.
template <int BK>
__device__ __forceinline__ bool mma_role(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base, uint32_t ring_addr,
                                         uint32_t planes_addr, uint32_t stage_bytes, uint32_t sub_bytes, uint32_t k_iters,
                                         uint32_t mine) {
  WaitCtl* wc = &ctl->wait;
  const bool leader = elect_one();
  const uint32_t full0 = smem_u32(p.flip ? &ctl->flipped[0] : &ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
  const uint32_t acc_full0 = smem_u32(&ctl->acc_full[0]), acc_empty0 = smem_u32(&ctl->acc_empty[0]);
  const uint32_t desc_hi = smem_desc_hi(BK);
  const bool whole = p.tail_ksteps == (uint32_t)(BK / 32);     // every K block is full of channels
  // resident digit planes: K blocks below planes_upto are known to have landed
  const uint32_t plane_part = (k_iters + kPlaneBars - 1) / kPlaneBars;
  uint32_t planes_ready = 0, planes_upto = p.resident ? 0u : 0xFFFFFFFFu;
  uint32_t s = 0, ph = 0, pass = 0;
  TileIter ti;
  for (ti.init(p); ti.valid(); ti.next()) {
    const uint32_t levels = tile_levels(p, ti.m_tile) & p.a.level_mask & 0x7Fu;
    if (!levels) continue;      // no sampled level: no pass from any role
    if (p.alternate && (pass & 1u) != mine) {      // the other warp's tile and stage
      ++pass;
      if (++s == p.stages) { s = 0; ph ^= 1u; }
      continue;
    }
    const uint32_t P = p.planes[(uint32_t)__ffs((int)levels) - 1u];
    const uint32_t buf = pass & 1u, aph = (pass >> 1) & 1u;
    ++pass;
    // instruction descriptor: s32 accumulators, s8 x s8, both K-major, M = 128, N = P * 64
    const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | (((P * kTileN) >> 3) << 17) | ((kTileM >> 4) << 24);
    const uint32_t d_tmem = tmem_base + buf * kTmemBufStride;
    const uint32_t blk = P * kTileN * BK;
    if (!warp_wait(acc_empty0 + 8u * buf, aph ^ 1u, wc)) return true;
    tc_fence_after();
    uint32_t b_res = planes_addr, acc = 0u, cb = 0u;
    for (uint32_t it = 0; it < k_iters;) {
      const uint32_t cnt = min(p.group, k_iters - it);
      if (!warp_wait(full0 + 8u * s, ph, wc)) return true;
      while (it + cnt > planes_upto) {
        if (!warp_wait(smem_u32(&ctl->planes_full[planes_ready]), 0u, wc)) return true;
        ++planes_ready;
        planes_upto = planes_ready == (uint32_t)kPlaneBars ? 0xFFFFFFFFu : planes_upto + plane_part;
      }
      tc_fence_after();
      // K blocks of the stage: activation tiles sub_bytes apart, planes beside them or resident; only the
      // low words of the descriptors move (by bytes / 16)
      uint32_t a_lo = smem_desc_lo(ring_addr + s * stage_bytes);
      uint32_t b_lo = p.resident ? smem_desc_lo(b_res) : a_lo + (p.stage_bytes_a >> 4);
      const uint32_t a_step = sub_bytes >> 4, b_step = p.resident ? blk >> 4 : sub_bytes >> 4;
      for (uint32_t j = 0; j < cnt; ++j, a_lo += a_step, b_lo += b_step) {
        // a tap's last channel block: only the K steps that hold channels
        const bool tail = ++cb == p.n_cb;
        if (tail) cb = 0u;
        if (whole || !tail) {
          if (leader) {
            tc_mma_i8(d_tmem, a_lo, b_lo, desc_hi, idesc, acc);
#pragma unroll
            for (int ks = 1; ks < BK / 32; ++ks) tc_mma_i8(d_tmem, a_lo + 2 * ks, b_lo + 2 * ks, desc_hi, idesc, 1u);
          }
        } else {
          for (uint32_t ks = 0; ks < p.tail_ksteps; ++ks)
            if (leader) tc_mma_i8(d_tmem, a_lo + 2 * ks, b_lo + 2 * ks, desc_hi, idesc, ks ? 1u : acc);
        }
        acc = 1u;
      }
      if (leader) tc_commit(empty0 + 8u * s);
      b_res += cnt * blk;
      it += cnt;
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
    if (leader) tc_commit(acc_full0 + 8u * buf);
    __syncwarp();
  }
  return false;
}

// The same role in band mode, where a ring stage holds the band of a whole tile: two warps work on every tile, the first
// on the first half of its taps, the second (mine = 1) on the rest, both into the one accumulator (the order of integer
// additions is immaterial), so that one's bookkeeping between tiles runs under the other's MMAs (3x3 64 -> 64 channels,
// 56x56, batch 64: 23.4 us with one warp).  The first one issues the overwriting MMA (`started`); both commit to the
// stage's and the accumulator's barriers (count 2 in this mode).
template <int BK>
__device__ __forceinline__ bool mma_role_band(const TensorParams& p, SharedCtl* ctl, uint32_t tmem_base,
                                              uint32_t ring_addr, uint32_t planes_addr, uint32_t stage_bytes, uint32_t mine) {
  WaitCtl* wc = &ctl->wait;
  const bool leader = elect_one();
  const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
  const uint32_t acc_full0 = smem_u32(&ctl->acc_full[0]), acc_empty0 = smem_u32(&ctl->acc_empty[0]);
  const uint32_t started0 = smem_u32(&ctl->started[0]);
  const uint32_t desc_hi = smem_desc_hi(BK);
  const uint32_t P = p.planes[p.a.uniform_log2k];
  const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | (((P * kTileN) >> 3) << 17) | ((kTileM >> 4) << 24);
  const uint32_t b_step = P * kTileN * BK / 16u, row_step = p.Wp * p.a.C / 16u;
  const uint32_t taps = p.a.KH * p.a.KW, half = (taps + 1u) / 2u;
  const uint32_t tap0 = mine ? half : 0u, tap1 = mine ? taps : half;
  const uint32_t kh0 = tap0 / p.a.KW, kw0 = tap0 - kh0 * p.a.KW;
  // resident digit planes arrive in kPlaneBars parts of `plane_part` K blocks (= taps)
  const uint32_t plane_part = (taps + kPlaneBars - 1) / kPlaneBars;
  const uint32_t parts_needed = tap1 > tap0 ? min((uint32_t)kPlaneBars, (tap1 - 1u) / plane_part + 1u) : 0u;
  uint32_t s = 0, ph = 0, pass = 0;
  TileIter ti;
  for (ti.init(p); ti.valid(); ti.next(), ++pass) {
    const uint32_t buf = pass & 1u, aph = (pass >> 1) & 1u;
    const uint32_t d_tmem = tmem_base + buf * kTmemBufStride;
    // byte offset of the tile's first position in its band
    const uint32_t t0 = (ti.m_tile - __umulhi(ti.m_tile, p.tpi_magic) * p.tpi) * kTileM;
    const uint32_t band_off = (t0 - __umulhi(t0, p.Wp_magic) * p.Wp) * (uint32_t)BK;
    if (!warp_wait(acc_empty0 + 8u * buf, aph ^ 1u, wc)) return true;
    if (!warp_wait(full0 + 8u * s, ph, wc)) return true;
    if (pass == 0u)
      for (uint32_t b = 0; b < parts_needed; ++b)
        if (!warp_wait(smem_u32(&ctl->planes_full[b]), 0u, wc)) return true;
    if (mine && !warp_wait(started0 + 8u * buf, aph, wc)) return true;
    tc_fence_after();
    uint32_t a_row = smem_desc_lo(ring_addr + s * stage_bytes + band_off) + kh0 * row_step, kw = kw0;
    uint32_t b_lo = smem_desc_lo(planes_addr) + tap0 * b_step;
    for (uint32_t tap = tap0; tap < tap1; ++tap, b_lo += b_step) {
      const uint32_t a_lo = a_row + kw * (BK / 16u);
      if (leader) {
        tc_mma_i8(d_tmem, a_lo, b_lo, desc_hi, idesc, tap ? 1u : 0u);
        if (tap == 0u) {
          tc_fence_before();
          mbar_arrive(started0 + 8u * buf);
        }
#pragma unroll
        for (int ks = 1; ks < BK / 32; ++ks) tc_mma_i8(d_tmem, a_lo + 2 * ks, b_lo + 2 * ks, desc_hi, idesc, 1u);
      }
      if (++kw == p.a.KW) { kw = 0; a_row += row_step; }
    }
    if (leader) {
      tc_commit(empty0 + 8u * s);
      tc_commit(acc_full0 + 8u * buf);
    }
    __syncwarp();
    if (++s == p.stages) { s = 0; ph ^= 1u; }
  }
  return false;
}

// Unsigned activations (p.flip): a warp of its own flips the top bit of every byte of the stages' activation tiles in
// shared memory, between the copy's arrival and the MMAs, makes the writes visible to the tensor core's proxy and
// hands the stage on (`flipped`).  A 16 KB tile is 32 steps of 16 bytes per lane, about the time of the four MMAs of its K
// block, under which it runs.  (A pass over the tensor in global memory cost a launch and a read and a write of all
// activations, and could not serve padded filters.)
__device__ __forceinline__ bool flip_role(const TensorParams& p, SharedCtl* ctl, uint32_t ring_addr, uint32_t stage_bytes,
                                          uint32_t sub_bytes, uint32_t k_iters) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t s = 0, ph = 0;
  TileIter ti;
  for (ti.init(p); ti.valid(); ti.next()) {
    if (!(tile_levels(p, ti.m_tile) & p.a.level_mask & 0x7Fu)) continue;
    for (uint32_t it = 0; it < k_iters;) {
      const uint32_t cnt = min(p.group, k_iters - it);
      if (!warp_wait(smem_u32(&ctl->full[s]), ph, &ctl->wait)) return true;
      for (uint32_t j = 0; j < cnt; ++j) {
        const uint32_t addr = ring_addr + s * stage_bytes + j * sub_bytes;
#pragma unroll 8
        for (uint32_t b = lane * 16u; b < p.stage_bytes_a; b += 512u) {
          uint32_t x, y, z, w;
          asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x), "=r"(y), "=r"(z), "=r"(w) : "r"(addr + b));
          asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr + b), "r"(x ^ 0x80808080u), "r"(y ^ 0x80808080u),
                       "r"(z ^ 0x80808080u), "r"(w ^ 0x80808080u) : "memory");
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->flipped[s]));
      it += cnt;
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
  }
  return false;
}

// kKind: which output stage the instance carries, the loops for the common case (uniform_epilogue), for one draw count or
// for rows sorted by level, those for real-valued outputs (with or without codes beside them), for one draw count or for sorted
// rows, or the general one; the host picks the instance, so that none drags the others' code and registers along (sorted rows
// in an instance of their own: ResNet-50 shape, batch 64, one draw count 1659 -> 1645 us; real-valued outputs out of the general
// instance: accumulators of 3x3 64 -> 64 on 81 locations 23.2 -> 19.9 us).
constexpr int kOneLevel = 0, kSortedRows = 1, kGeneralOutputs = 2, kRealOutputs = 3, kRealSorted = 4;
template <int BK, int kKind, int kRec>
__global__ void __launch_bounds__(kThreadsTensor, 1)
psb_mma_kernel(const __grid_constant__ TmapSet maps, const __grid_constant__ TensorParams p) {
  constexpr bool kSorted = kKind == kSortedRows, kReal = kKind == kRealOutputs || kKind == kRealSorted, kCodes = kKind == kOneLevel || kSorted;
  extern __shared__ uint8_t smem_raw[];
  // stage buffers need 1024-byte alignment for the 128-byte swizzle pattern
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023u) & ~(uintptr_t)1023u);
  // resident mode: [digit planes of all K blocks][ring of activation stages][control]
  // streaming mode: [ring of (activation, planes) stages][control]
  uint8_t* ring = smem + (p.resident ? p.resident_bytes : 0u);
  // a stage holds `group` K blocks, each an activation tile followed (streaming mode) by planes
  const uint32_t sub_bytes = p.stage_bytes_a + (p.resident ? 0u : p.stage_bytes_b_max);
  const uint32_t stage_bytes = p.band ? p.band_bytes : sub_bytes * p.group;
  // staged outputs: kIoSlots tiles between the ring and the control block
  const uint32_t slots_addr = smem_u32(ring) + p.stages * stage_bytes;
  SharedCtl* ctl = reinterpret_cast<SharedCtl*>(ring + (size_t)p.stages * stage_bytes + (p.staged | p.real_slots ? kIoSlots * kIoTileBytes : 0u));

  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const uint32_t k_iters = p.a.KH * p.a.KW * p.n_cb;

  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), p.band ? 2u : 1u);     // band mode: two warps use every stage
      mbar_init(smem_u32(&ctl->flipped[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctl->acc_full[b]), p.band ? 2u : 1u);
      mbar_init(smem_u32(&ctl->acc_empty[b]), p.staged ? kEpilogueWarps / 2 : kEpilogueWarps);   // staged: a group of warps per tile
    }
    {  // part b of the resident planes holds K blocks [b * part, (b + 1) * part): one arrival per block
      const uint32_t part = (k_iters + kPlaneBars - 1) / kPlaneBars;
      for (uint32_t b = 0; b < (uint32_t)kPlaneBars; ++b) {
        const uint32_t lo = b * part, hi = min(lo + part, k_iters);
        mbar_init(smem_u32(&ctl->planes_full[b]), hi > lo ? hi - lo : 1u);
      }
    }
    for (int b = 0; b < 2; ++b) mbar_init(smem_u32(&ctl->started[b]), 1);
    for (int l = 0; l < kMaxLevels; ++l) ctl->rowmax[l] = 0u;
    for (int b = 0; b < kIoSlots; ++b) {
      mbar_init(smem_u32(&ctl->slot_ready[b]), 1);
      mbar_init(smem_u32(&ctl->slot_done[b]), kEpilogueWarps / 2);
    }
    ctl->wait.abort = 0;
    ctl->wait.limit = p.wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    // descriptor fetches of the first copies would otherwise sit on the critical path of the first tile
    asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.a) : "memory");
  }
  if (warp == kMmaWarp1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&ctl->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  WaitCtl* abort = &ctl->wait;
  bool failed = false;
  // The kernel is launched with programmatic stream serialisation: a CTA may get here while the
  // kernel before it in the stream is still draining.  Nothing above touches global memory; from
  // here on everything does (activations, planes, constants, outputs), so every thread waits for
  // the earlier grids to complete and their writes to be visible.  The kernel after this one may
  // be scheduled as soon as SMs free up (it waits at the same point).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp < (uint32_t)kProducerWarps) {
    // ----------------------------------------------------------- producers
    // A copy instruction holds its thread for a few hundred clocks, whatever its size, while the
    // copy engine takes several at a time: the K blocks of a stage are therefore issued by as
    // many lanes of the warp in one go (lane j copies block j), after lane 0 has waited for the
    // stage and posted the byte count; and the producer warps take the stages in turns (all of
    // them walk the same sequence of stages, each issues every second one).
    uint32_t s = 0, ph = 0;   // ring position and phase of the current stage use
    uint32_t turn = 0;        // whose turn it is among the producer warps
    const uint32_t ring_addr = smem_u32(ring);
    TileIter ti;
    for (ti.init(p); ti.valid() && !failed; ti.next()) {
      const uint32_t m_tile = ti.m_tile, o_tile = ti.o_tile;
      const uint32_t m0 = m_tile * kTileM;
      const uint32_t levels = tile_levels(p, ti.m_tile) & p.a.level_mask;
      // image coordinates of the tile's first row: divisions, so only the warp that is about to
      // issue a copy of this tile computes them
      uint32_t n0 = 0;
      int h0 = 0, w0 = 0;
      bool have_coords = !p.im2col || p.band;
      for (uint32_t todo = levels & 0x7Fu; todo && !failed; todo &= todo - 1u) {
        const uint32_t l = (uint32_t)__ffs((int)todo) - 1u;
        const uint32_t P = p.planes[l];
        const uint32_t bytes = p.stage_bytes_a + (p.resident ? 0u : P * kTileN * BK);
        const uint32_t blk = P * kTileN * BK;
        const int8_t* b_tiles = p.planes_ptr[l] + (size_t)o_tile * k_iters * blk;   // this channel tile's K blocks
        for (uint32_t it = 0; it < k_iters;) {
          const uint32_t cnt = min(p.group, k_iters - it);
          if (turn == warp) {
            if (!have_coords) {
              const uint32_t ohow = p.a.OH * p.a.OW;
              n0 = m0 / ohow;
              const uint32_t rem = m0 - n0 * ohow, oy = rem / p.a.OW;
              h0 = (int)(oy * p.a.stride) - (int)p.a.pad;
              w0 = (int)((rem - oy * p.a.OW) * p.a.stride) - (int)p.a.pad;
              have_coords = true;
            }
            const uint32_t bar = smem_u32(&ctl->full[s]);
            bool ok = true;
            if (lane == 0) {
              ok = mbar_wait(smem_u32(&ctl->empty[s]), ph ^ 1u, abort);
              if (ok) mbar_expect_tx(bar, p.band ? p.band_rows * p.Wp * p.a.C : bytes * cnt);
            }
            if (!__shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0)) { failed = true; break; }
            if (p.band) {
              // one copy per tile: the band of padded input rows that holds every tap of the tile;
              // rows and columns outside the image read as zeros
              if (lane == 0) {
                const uint32_t n = __umulhi(m_tile, p.tpi_magic);
                const uint32_t r0 = __umulhi((m_tile - n * p.tpi) * kTileM, p.Wp_magic);
                tma_load_4d(ring_addr + s * stage_bytes, &maps.a, bar, 0, -(int)p.a.pad, (int)r0 - (int)p.a.pad, (int)n);
              }
            } else if (lane < cnt) {
              // K block it + lane: tap (kh, kw), channel block cb, column kcol of the plane matrix
              const uint32_t kb = it + lane;
              const uint32_t tap = kb / p.n_cb, cb = kb - tap * p.n_cb;
              const uint32_t kh = tap / p.a.KW, kw = tap - kh * p.a.KW;
              const uint32_t dst = ring_addr + s * stage_bytes + lane * sub_bytes;
              if (p.im2col)
                tma_load_im2col_4d(dst, &maps.a, bar, (int)(cb * BK), w0, h0, (int)n0, (uint16_t)kw, (uint16_t)kh);
              else
                tma_load_2d(dst, &maps.a, bar, (int)(cb * BK), (int)m0);
              if (!p.resident) bulk_load(dst + p.stage_bytes_a, b_tiles + (size_t)kb * blk, blk, bar);
            }
          }
          it += cnt;
          if (++s == p.stages) { s = 0; ph ^= 1u; }
          if (++turn == (uint32_t)kProducerWarps) turn = 0;
        }
      }
    }
  } else if (warp == (uint32_t)kMmaWarp0 || warp == (uint32_t)kMmaWarp1) {
    // ---------------------------------------------------------------- MMA
    if (!kSorted && p.band)
      failed = mma_role_band<BK>(p, ctl, tmem_base, smem_u32(ring), smem_u32(smem), stage_bytes, warp - (uint32_t)kMmaWarp0);
    else if (warp == (uint32_t)kMmaWarp0 || p.alternate)
      failed = mma_role<BK>(p, ctl, tmem_base, smem_u32(ring), smem_u32(smem), stage_bytes, sub_bytes, k_iters,
                            warp - (uint32_t)kMmaWarp0);
    else if (!kSorted && p.staged) {
      if (lane == 0) failed = io_role(p, maps, ctl, slots_addr);
      failed = __shfl_sync(0xFFFFFFFFu, failed ? 1 : 0, 0) != 0;
    } else if (p.flip)
      failed = flip_role(p, ctl, smem_u32(ring), stage_bytes, sub_bytes, k_iters);
  } else {
    // ----------------------------------------------------------- epilogue
    // 16 warps: warp & 3 selects the TMEM lane quarter (32 rows), ew >> 2 the 16 of the tile's 64
    // channels.
    const uint32_t ew = warp - (uint32_t)kFirstEpilogueWarp;   // 0..15
    const uint32_t quarter = ew & 3u;
    const uint32_t sub = ew >> 2;
    const uint32_t row = quarter * 32u + lane;
    const ConvArgs& a = p.a;
    const bool q_only = a.q_out && !a.f32_out && !a.acc_out && a.inv_step > 0.0f;
    EpiConst ec;
    ec.res_scale = a.residual_scale;
    // With inv_step > 0 (a condition of the fast paths) max(y, 0) * inv_step == max(y * inv_step, 0):
    // the relu is folded into the lower clamp bound.
    ec.inv_step = a.inv_step;
    ec.lo_f = (a.relu && a.qmin < 0) ? 0.0f : (float)a.qmin;
    ec.hi_f = (float)a.qmax;
    ec.out_signed = a.out_dtype == PSB_DT_S8 ? 1u : 0u;
    // unsigned codes from 0 up: the byte saturation of the packing instruction is the lower clamp
    const bool fast_u8 = a.out_dtype == PSB_DT_U8 && a.qmin == 0;
    const uint32_t res_kind = !a.residual ? 0u : (a.residual_dtype == PSB_DT_S8 ? 2u : 1u);
    uint32_t P0 = p.planes[a.uniform_log2k < (uint32_t)kMaxLevels ? a.uniform_log2k : 0u];
    if (a.kmap) P0 = p.planes[(uint32_t)__ffs((int)(a.level_mask & 0x7Fu)) - 1u];
    if (p.resident && lane == 0) {
      // the digit planes of this CTA's channel tile, all K blocks, once: the epilogue warps have
      // nothing else to do yet, and sixteen threads get the copies under way sooner than one
      const uint32_t o_tile = blockIdx.x / p.ctas_per_otile;
      const uint32_t blk = P0 * kTileN * BK;
      const uint32_t part = (k_iters + kPlaneBars - 1) / kPlaneBars;
      for (uint32_t it = ew; it < k_iters; it += (uint32_t)kEpilogueWarps) {
        const uint32_t bar = smem_u32(&ctl->planes_full[it / part]);
        mbar_expect_tx(bar, blk);
        bulk_load(smem_u32(smem) + it * blk, p.planes_ptr[a.uniform_log2k] + ((size_t)o_tile * k_iters + it) * blk, blk,
                  bar);
      }
    }
    // (accumulators are always recombined in 64 bits, real-valued outputs as the host knows beforehand (p.mid); no level instead
    // of a branch around the call, with which 3x3 100 -> 150 channels, codes only, took 49.3 us and not 48.4)
    const uint32_t bounded = a.kmap ? a.level_mask : 1u << a.uniform_log2k;
    if constexpr (!kReal) find_row_maxima(p, ctl, kCodes || q_only ? bounded : 0u);
    if constexpr (kCodes) {
      bool w32 = kRec != kPlainSums || p.corr[(uint32_t)__ffs((int)(a.level_mask & 0x7Fu)) - 1u] == nullptr;
      if (kSorted) {         // every level a tile may have must fit
        for (uint32_t lv = 0; lv < (uint32_t)kMaxLevels; ++lv)
          if ((a.level_mask >> lv) & 1u) w32 = fits_32_bits(p, ctl, lv) && w32;
      } else {
        w32 = fits_32_bits(p, ctl, a.uniform_log2k) && w32;
      }
      EpiChoice how;
      how.fast_u8 = fast_u8;
      how.res = res_kind;
      how.fits = w32;
      how.mid = p.mid != 0u;
      if constexpr (kRec != kPlainSums) failed = uniform_dispatch<3, kRec, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, ec, how);
      else if (P0 == 4u) failed = uniform_dispatch<4, kRec, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, ec, how);
      else if (P0 == 3u) failed = uniform_dispatch<3, kRec, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, ec, how);
      else failed = uniform_dispatch<2, kRec, kSorted>(p, ctl, tmem_base, slots_addr, ew, lane, ec, how);
    } else if constexpr (kKind == kRealOutputs) {
      if (P0 == 4u) failed = epilogue_real<4, kRec64>(p, ctl, tmem_base, slots_addr, ew, lane);
      else if (P0 == 3u && p.mid) failed = epilogue_real<3, kRecMidAdd>(p, ctl, tmem_base, slots_addr, ew, lane);
      else if (P0 == 3u) failed = epilogue_real<3, kRec64>(p, ctl, tmem_base, slots_addr, ew, lane);
      else if (P0 == 2u) failed = epilogue_real<2, kRec64>(p, ctl, tmem_base, slots_addr, ew, lane);
      else failed = epilogue_real<1, kRec64>(p, ctl, tmem_base, slots_addr, ew, lane);
    } else {
      // general loop: per-location draw counts, any outputs and layouts, ragged channel counts
      const float2* scb = ctl->scb[ew];
      const long long* corr = ctl->corr[ew];
      uint32_t pass = 0, cur_key = 0xFFFFFFFFu;
      uint32_t w32_levels = 0;      // levels whose accumulators are known to fit 32 bits
      if (!kReal && q_only)
        for (uint32_t l = 0; l < (uint32_t)kMaxLevels; ++l)
          if (((a.level_mask >> l) & 1u) && fits_32_bits(p, ctl, l)) w32_levels |= 1u << l;
      TileIter ti;
      for (ti.init(p); !failed && ti.valid(); ti.next()) {
        const uint32_t m0 = ti.m_tile * kTileM, o_tile = ti.o_tile;
        const uint32_t levels = tile_levels(p, ti.m_tile) & a.level_mask;
        uint32_t m = m0 + row;
        bool in_range = m < p.M;
        if (p.perm) {           // rows sorted by level: the location of this row
          m = p.perm[m0 + row];
          in_range = m != 0xFFFFFFFFu;
        }
        const uint32_t my_level = in_range ? (a.kmap ? (uint32_t)a.kmap[m] : a.uniform_log2k) : 0xFFu;
        if (in_range && (my_level >= (uint32_t)kMaxLevels || !((a.level_mask >> my_level) & 1u)))
          atomicOr(a.err, kDevErrBadLevel);
        const uint32_t o_base = o_tile * kTileN + sub * 16u;
        const size_t oidx = (size_t)m * a.O + o_base;
        const uint32_t unit = p.unit, count = o_base < a.O ? a.O - o_base : 0u;
        const bool fast = !kReal && q_only && !a.out_nchw && o_base < a.O;
        uint4 r4 = make_uint4(0, 0, 0, 0);
        if (fast && a.residual && in_range) r4 = unit < 8u ? load_narrow16((const uint8_t*)a.residual + oidx, unit, count)
                    : load_row16((const uint8_t*)a.residual + oidx, unit == 16u, count >= 16u);
        for (uint32_t todo = levels & 0x7Fu; todo && !failed; todo &= todo - 1u) {
          const uint32_t l = (uint32_t)__ffs((int)todo) - 1u;
          const uint32_t P = p.planes[l];
          const uint32_t buf = pass & 1u, aph = (pass >> 1) & 1u;
          const bool use_corr = p.corr[l] != nullptr;
          // per-channel constants of this (channel tile, level), refreshed only when the pair changes
          const uint32_t key = o_tile * 8u + l;
          if (key != cur_key) {
            __syncwarp();
            if (lane < 16u) {
              const uint32_t o = o_base + lane;
              float2 sb = make_float2(0.f, 0.f);
              long long cr = 0;
              if (o < a.O) {
                sb.x = ldexpf(a.scale[o], a.e_base[o] - (int)l);
                sb.y = a.bias[o];
                if (use_corr) cr = p.corr[l][o];
              }
              ctl->scb[ew][lane] = sb;
              ctl->corr[ew][lane] = kReal && p.mid && P == 3u ? addend_words<kRecMidAdd>(cr) : cr;
              ctl->corr32[ew][lane] = (int32_t)cr;
            }
            cur_key = key;
            __syncwarp();
          }
          const bool ok = mbar_wait(smem_u32(&ctl->acc_full[buf]), aph, abort, 32);
          failed = __any_sync(0xFFFFFFFFu, !ok) != 0;
          if (failed) break;
          tc_fence_after();
          const uint32_t taddr = tmem_base + buf * kTmemBufStride + ((quarter * 32u) << 16) + sub * 16u;
          const bool valid = in_range && my_level == l;
          if (o_base < a.O) {
            if constexpr (kReal) {
              const uint32_t slot = slots_addr + ew * 2048u;
              switch (P) {
                case 1: epilogue_chunk_real<1, kRec64>(p, taddr, slot, o_base, m, valid, scb, corr); break;
                case 2: epilogue_chunk_real<2, kRec64>(p, taddr, slot, o_base, m, valid, scb, corr); break;
                case 3:
                  if (p.mid) epilogue_chunk_real<3, kRecMidAdd>(p, taddr, slot, o_base, m, valid, scb, corr);
                  else epilogue_chunk_real<3, kRec64>(p, taddr, slot, o_base, m, valid, scb, corr);
                  break;
                default: epilogue_chunk_real<4, kRec64>(p, taddr, slot, o_base, m, valid, scb, corr); break;
              }
            } else if (fast) {
              const bool w32 = ((w32_levels >> l) & 1u) != 0u;
#define PSB_EPI(PV, WV, RV) epilogue_chunk_q<PV, WV, RV>(taddr, valid, (uint8_t*)a.q_out, oidx, r4, unit, count, scb, corr, \
                                                         use_corr ? ctl->corr32[ew] : nullptr, ec)
#define PSB_EPI_P(WV, RV)                                                                          \
  do {                                                                                             \
    if (P == 4) PSB_EPI(4, WV, RV); else if (P == 3) PSB_EPI(3, WV, RV);                           \
    else if (P == 2) PSB_EPI(2, WV, RV); else PSB_EPI(1, WV, RV);                                  \
  } while (0)
              if (w32) {
                if (res_kind == 0u) PSB_EPI_P(true, 0); else if (res_kind == 1u) PSB_EPI_P(true, 1); else PSB_EPI_P(true, 2);
              } else {
                if (res_kind == 0u) PSB_EPI_P(false, 0); else if (res_kind == 1u) PSB_EPI_P(false, 1); else PSB_EPI_P(false, 2);
              }
#undef PSB_EPI_P
#undef PSB_EPI
            } else {
              const uint32_t ohow = a.OH * a.OW;
              const uint32_t n = in_range ? m / ohow : 0u, pix = in_range ? m % ohow : 0u;
              switch (P) {
                case 1: epilogue_chunk<1>(p, taddr, o_base, m, valid, n, pix, scb, corr, use_corr); break;
                case 2: epilogue_chunk<2>(p, taddr, o_base, m, valid, n, pix, scb, corr, use_corr); break;
                case 3: epilogue_chunk<3>(p, taddr, o_base, m, valid, n, pix, scb, corr, use_corr); break;
                default: epilogue_chunk<4>(p, taddr, o_base, m, valid, n, pix, scb, corr, use_corr); break;
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[buf]));
          ++pass;
        }
      }
    }
  }

  // ------------------------------------------------------------- common exit
  if (failed) {
    if (lane == 0) {
      abort->abort = 1u;
      atomicOr(p.a.err, kDevErrTimeout);
    }
    // give copies and MMAs already in flight time to land before the CTA retires
    for (int i = 0; i < 64; ++i) __nanosleep(2000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kTmemCols)
                 : "memory");
  }
}

}  // namespace

// Launches the instance of the kernel with this K block (one translation unit per instance: psb_mma_bk*.cu).
template <int BK>
cudaError_t launch_mma_kernel(const cudaLaunchConfig_t& cfg, const TmapSet& maps, const TensorParams& p, int device, int kind, int rec);

}  // namespace psb
