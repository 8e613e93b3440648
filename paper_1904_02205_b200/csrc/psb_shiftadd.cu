// CUDA-core contraction ("shift-add" path) and the glue kernels.
//
// The paper's capacitor unit adds x << (e + B) over the draws (Eq. 9); summed over
// the k draws that is x * (k + c_k) << (e - e_base), an integer product with the
// sampled integer weight.  Depthwise and grouped filters hold that weight; dense
// ones hold its signed digit planes, whose byte products are summed plane by
// plane.  This path serves layers that are not dense matrix products for the
// tensor cores (depthwise filters) or too small for them (fully connected layers
// at small batch, filters on a few locations), and it honours per-location draw
// counts directly.
#include "psb_common.cuh"

#include <algorithm>

namespace psb {

namespace {

// True when one of the four bytes of `v` exceeds `limit` in magnitude (signed bytes: |b| > limit).
__device__ __forceinline__ bool bytes_beyond(uint32_t v, uint32_t is_signed, uint32_t limit) {
  const uint32_t mag = is_signed ? __vabs4(v) : v;        // |-128| = 128 as an unsigned byte
  return __vcmpgtu4(mag, limit * 0x01010101u) != 0u;
}

__device__ __forceinline__ int load_act(const void* x, uint32_t dtype, size_t idx) {
  return dtype == PSB_DT_U8 ? (int)((const uint8_t*)x)[idx] : (int)((const int8_t*)x)[idx];
}

__device__ __forceinline__ void store_outputs(const ConvArgs& a, size_t oidx, uint32_t o,
                                              uint32_t level, long long acc) {
  if (a.acc_out) a.acc_out[oidx] = acc;
  if (a.q_out || a.f32_out) {
    float sc = ldexpf(a.scale[o], a.e_base[o] - (int)level);
    int rq = a.residual ? load_act(a.residual, a.residual_dtype, oidx) : 0;
    float y = dequant(acc, sc, a.bias[o], a.residual != nullptr, rq, a.residual_scale, a.relu != 0);
    if (a.f32_out) a.f32_out[oidx] = y;
    if (a.q_out) {
      int q = requant(y, a.inv_step, a.qmin, a.qmax);
      if (a.out_dtype == PSB_DT_U8) ((uint8_t*)a.q_out)[oidx] = (uint8_t)q;
      else ((int8_t*)a.q_out)[oidx] = (int8_t)q;
    }
  }
}

// One thread per output element, output channel fastest.  For depthwise filters
// (one input channel per group) neighbouring threads read neighbouring bytes.
__global__ void __launch_bounds__(256) conv_direct_kernel(const ConvArgs a, const WintTable wt) {
  pdl_prologue();
  const size_t total = (size_t)a.N * a.OH * a.OW * a.O;
  const uint32_t Cg = a.C / a.groups, Og = a.O / a.groups;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const uint32_t o = (uint32_t)(idx % a.O);
    const size_t pix = idx / a.O;
    const uint32_t ox = (uint32_t)(pix % a.OW);
    const uint32_t oy = (uint32_t)((pix / a.OW) % a.OH);
    const uint32_t n = (uint32_t)(pix / ((size_t)a.OW * a.OH));
    const uint32_t level = a.kmap ? a.kmap[pix] : a.uniform_log2k;
    if (level >= (uint32_t)kMaxLevels || !((a.level_mask >> level) & 1u)) {
      atomicOr(a.err, kDevErrBadLevel);
      continue;
    }
    const int32_t* w = wt.w[level] + (size_t)o * a.KH * a.KW * Cg;
    const uint32_t cbase = (o / Og) * Cg;
    long long acc = 0;
    for (uint32_t kh = 0; kh < a.KH; ++kh) {
      const int iy = (int)(oy * a.stride + kh) - (int)a.pad;
      if (iy < 0 || iy >= (int)a.H) continue;
      for (uint32_t kw = 0; kw < a.KW; ++kw) {
        const int ix = (int)(ox * a.stride + kw) - (int)a.pad;
        if (ix < 0 || ix >= (int)a.W) continue;
        const size_t xoff = (((size_t)n * a.H + iy) * a.W + ix) * a.C + cbase;
        const int32_t* wr = w + (size_t)(kh * a.KW + kw) * Cg;
        for (uint32_t ci = 0; ci < Cg; ++ci) {
          int xv = load_act(a.x, a.in_dtype, xoff + ci);
          acc += (long long)xv * (long long)__ldca(wr + ci);
        }
      }
    }
    const size_t oidx = a.out_nchw ? (((size_t)n * a.O + o) * a.OH + oy) * a.OW + ox : idx;
    store_outputs(a, oidx, o, level, acc);
  }
}

// Four byte products of an unsigned / signed activation word with a signed digit word, accumulated.
template <bool kSignedIn>
__device__ __forceinline__ int dp4a_act(uint32_t x, uint32_t w, int acc) {
  int d;
  if (kSignedIn) asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(w), "r"(acc));
  else asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(w), "r"(acc));
  return d;
}

// Dense layers on CUDA cores (fully connected layers at small batch, filters with and without taps on a few locations),
// straight from the digit planes: a group of lanes per output channel, each lane 16 bytes of the K axis at a time (one
// 16-byte load per plane, four dp4a per plane and location), kNB output locations per pass over the weights; a plane's sum
// stays in 32 bits over one segment of the axis, the planes and segments meet in 64 bits and the lanes in a shuffle tree.
// The patches of the block's locations sit in shared memory in the order of the planes' K axis, kPlaneSegment bytes at a
// time, zero outside the image and beyond the channels.  Bound by the latency of its few loads; P bytes per weight are
// read instead of the 4 of an integer filter.  (One thread per output on an integer filter, which has to be put together
// from the planes first, took 698 us for 3x3 512 -> 512 on 9 locations, 44 us for 32 -> 32 on 49; this kernel 11.0 and 8.7,
// the latter in a stream of calls that the host bounds.)
constexpr int kPlaneLocations = 4;
constexpr uint32_t kPlaneSegment = 8192;      // kPlaneLocations patches of them take 32 KB
// Blocks per SM.  More registers than three or two of them leave (loads of four pieces in flight) help a single wave, which
// is what PSB_PATH_AUTO sends here: 3x3 512 -> 512 on 9 locations 11.0 us, with three blocks 15.2.
constexpr int kPlainBlocks = 3, kTapBlocks = 2;

// (Kept small: with 304 bytes of parameters instead of 280 a launch took 0.35 us longer on the host.)
struct DensePlanes {
  const int8_t* p[kMaxLevels];
  uint8_t count[kMaxLevels + 1];
  uint32_t bk, n_kb;
  uint32_t tap_pieces;     // 16-byte pieces of the K axis per tap (channels rounded up to whole K blocks); flat K axis: 0
  uint32_t run_pitch;      // flat K axis: bytes per filter row
  float per_tap, per_kw;   // 1 / tap_pieces, 1 / KW
};

// 16 bytes of the patch of one output location from K-axis byte k on; iy0, ix0: its first tap in image `img`.  kPlain:
// a filter of one tap without stride and padding, `img` is the location itself.
template <bool kPlain>
__device__ __forceinline__ uint4 patch_piece(const ConvArgs& a, const DensePlanes& w, const uint8_t* img, int iy0, int ix0,
                                             uint32_t k, uint32_t unit) {
  uint32_t b[4] = {0u, 0u, 0u, 0u};
  if (kPlain || w.tap_pieces) {
    uint32_t ci = k;
    const uint8_t* src = img + k;
    if (!kPlain) {
      // quotients of numbers below 2^22 (pieces) and 2^11 (taps) in fp32, the first one put right where it is one off
      const uint32_t piece = k / 16u;
      uint32_t tap = __float2uint_rz((float)piece * w.per_tap);
      if (tap * w.tap_pieces > piece) --tap;
      else if ((tap + 1u) * w.tap_pieces <= piece) ++tap;
      const uint32_t kh = __float2uint_rz(((float)tap + 0.5f) * w.per_kw);
      const int iy = iy0 + (int)kh, ix = ix0 + (int)(tap - kh * a.KW);
      if ((unsigned)iy >= a.H || (unsigned)ix >= a.W) return make_uint4(0u, 0u, 0u, 0u);
      ci = (piece - tap * w.tap_pieces) * 16u;
      src = img + ((size_t)iy * a.W + (uint32_t)ix) * a.C + ci;
    }
    if (ci >= a.C) return make_uint4(0u, 0u, 0u, 0u);
    if (unit == 16u) return __ldcg(reinterpret_cast<const uint4*>(src));
    if (unit == 4u) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (ci + 4u * j < a.C) b[j] = __ldcg(reinterpret_cast<const uint32_t*>(src + 4 * j));
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (ci + j < a.C) b[j >> 2] |= (uint32_t)src[j] << (8 * (j & 3));
    }
  } else {
    uint32_t kh = k / w.run_pitch, at = k - kh * w.run_pitch, kw = at / a.C, ci = at - kw * a.C;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int iy = iy0 + (int)kh, ix = ix0 + (int)kw;
      if (kh < a.KH && kw < a.KW && (unsigned)iy < a.H && (unsigned)ix < a.W)
        b[j >> 2] |= (uint32_t)img[((size_t)iy * a.W + (uint32_t)ix) * a.C + ci] << (8 * (j & 3));
      if (++ci == a.C) { ci = 0u; ++kw; }
      if (++at == w.run_pitch) { at = kw = ci = 0u; ++kh; }
    }
  }
  return make_uint4(b[0], b[1], b[2], b[3]);
}

template <int kNB, bool kSignedIn, bool kPlain>
__global__ void __launch_bounds__(256, kPlain ? kPlainBlocks : kTapBlocks) dense_planes_kernel(const __grid_constant__ ConvArgs a,
                                                           const __grid_constant__ DensePlanes w, uint32_t M,
                                                           uint32_t lanes_per_row) {
  pdl_prologue();
  extern __shared__ __align__(16) uint8_t patches[];     // [kNB][min(kp, kPlaneSegment)]
  const uint32_t bk = w.bk, kp = w.n_kb * bk, seg = min(kp, kPlaneSegment), ohow = a.OH * a.OW;
  const uint32_t align = a.C | (uint32_t)(uintptr_t)a.x;
  const uint32_t unit = (align & 15u) == 0u ? 16u : (align & 3u) == 0u ? 4u : 1u;
  const uint32_t sub = threadIdx.x & (lanes_per_row - 1u);
  const uint32_t o = blockIdx.x * (blockDim.x / lanes_per_row) + threadIdx.x / lanes_per_row;
  for (uint32_t n0 = blockIdx.y * (uint32_t)kNB; n0 < M; n0 += gridDim.y * (uint32_t)kNB) {
    const uint32_t nb = min((uint32_t)kNB, M - n0);
    const uint8_t* img[kNB];
    int iy0[kNB], ix0[kNB];
    if (!kPlain) {
#pragma unroll
      for (int r = 0; r < kNB; ++r) {
        const uint32_t m = n0 + min((uint32_t)r, nb - 1u), n = m / ohow, pix = m - n * ohow, oy = pix / a.OW;
        img[r] = (const uint8_t*)a.x + (size_t)n * a.H * a.W * a.C;
        iy0[r] = (int)(oy * a.stride) - (int)a.pad;
        ix0[r] = (int)((pix - oy * a.OW) * a.stride) - (int)a.pad;
      }
    }
    const uint32_t level = a.kmap ? a.kmap[n0] : a.uniform_log2k;      // with a map kNB is 1
    const bool level_ok = level < (uint32_t)kMaxLevels && ((a.level_mask >> level) & 1u);
    if (!level_ok && threadIdx.x == 0) atomicOr(a.err, kDevErrBadLevel);
    long long sum[kNB];
#pragma unroll
    for (int r = 0; r < kNB; ++r) sum[r] = 0;
    for (uint32_t k0 = 0; k0 < kp; k0 += seg) {
      const uint32_t len = min(seg, kp - k0), chunks = len / 16u;
      if (k0 || n0 != blockIdx.y * (uint32_t)kNB) __syncthreads();      // the patches of the step before have been read
      if (kPlain && kNB > 1) {
        // the pieces of all rows dealt out to the threads: one load per thread for up to 1024 features, and one copy of the
        // code (row by row: 64 -> 10 features, 17 rows 3.9 us on the device, 3.4 so; 1024 -> 1024, 12 rows 6.2 and 5.6)
        for (uint32_t i = threadIdx.x; i < nb * chunks; i += blockDim.x) {
          uint32_t r = 0;
#pragma unroll
          for (int q = 1; q < kNB; ++q) r += i >= (uint32_t)q * chunks ? 1u : 0u;
          const uint32_t k = (i - r * chunks) * 16u;
          *reinterpret_cast<uint4*>(patches + r * seg + k) =
              patch_piece<true>(a, w, (const uint8_t*)a.x + (size_t)(n0 + r) * a.C, 0, 0, k0 + k, unit);
        }
      } else {
#pragma unroll
        for (int r = 0; r < kNB; ++r) {
          const uint8_t* from = kPlain ? (const uint8_t*)a.x + (size_t)n0 * a.C : img[r];
          for (uint32_t i = threadIdx.x * 16u; i < len; i += blockDim.x * 16u)
            *reinterpret_cast<uint4*>(patches + r * seg + i) = patch_piece<kPlain>(a, w, from, iy0[r], ix0[r], k0 + i, unit);
        }
      }
      __syncthreads();
      if (!level_ok || o >= a.O) continue;
      const int P = w.count[level];
      const uint32_t shift = 31u - (uint32_t)__clz((int)bk), on = o % kTileN;
      const size_t tile_bytes = (size_t)P * kTileN * bk;
      const int8_t* base = w.p[level] + (size_t)(o / kTileN) * w.n_kb * tile_bytes;
      int acc[kMaxPlanes][kNB];
#pragma unroll
      for (int pl = 0; pl < kMaxPlanes; ++pl)
#pragma unroll
        for (int r = 0; r < kNB; ++r) acc[pl][r] = 0;
#pragma unroll 4
      for (uint32_t c = sub; c < chunks; c += lanes_per_row) {
        const uint32_t k = k0 + c * 16u, off = plane_offset(on, k & (bk - 1u), bk);
        const int8_t* tile = base + (size_t)(k >> shift) * tile_bytes + off;
        uint4 d[kMaxPlanes];
#pragma unroll
        for (int pl = 0; pl < kMaxPlanes; ++pl)
          if (pl < P) d[pl] = __ldcg(reinterpret_cast<const uint4*>(tile + (size_t)pl * kTileN * bk));
#pragma unroll
        for (int r = 0; r < kNB; ++r) {
          const uint4 v = *reinterpret_cast<const uint4*>(patches + (uint32_t)r * seg + c * 16u);
#pragma unroll
          for (int pl = 0; pl < kMaxPlanes; ++pl)
            if (pl < P) {
              acc[pl][r] = dp4a_act<kSignedIn>(v.x, d[pl].x, acc[pl][r]);
              acc[pl][r] = dp4a_act<kSignedIn>(v.y, d[pl].y, acc[pl][r]);
              acc[pl][r] = dp4a_act<kSignedIn>(v.z, d[pl].z, acc[pl][r]);
              acc[pl][r] = dp4a_act<kSignedIn>(v.w, d[pl].w, acc[pl][r]);
            }
        }
      }
      // a lane's sum over a segment is at most 8192 * 255 * 127 < 2^28
#pragma unroll
      for (int r = 0; r < kNB; ++r)
#pragma unroll
        for (int pl = 0; pl < kMaxPlanes; ++pl) sum[r] += (long long)acc[pl][r] * (1ll << (kDigitBits * pl));
    }
#pragma unroll
    for (int r = 0; r < kNB; ++r) {
      for (uint32_t d = lanes_per_row / 2u; d > 0; d >>= 1) sum[r] += __shfl_xor_sync(0xFFFFFFFFu, sum[r], d);
      if (!level_ok || o >= a.O || (uint32_t)r >= nb || sub != ((uint32_t)r & (lanes_per_row - 1u))) continue;
      const uint32_t m = n0 + (uint32_t)r, n = m / ohow;
      const size_t at = a.out_nchw ? ((size_t)n * a.O + o) * ohow + (m - n * ohow) : (size_t)m * a.O + o;
      store_outputs(a, at, o, level, sum[r]);
    }
  }
}

// Depthwise filters (one input channel per output channel), channels-last, one draw count for
// the layer: a thread owns 8 consecutive channels of one output location.  The block keeps the
// layer's integer filter in shared memory as [tap][channel]; activations come in 8-byte loads;
// the integer sum x * W_k over the taps is Eq. 9 summed over the draws.  Writes 8 codes at once.
__global__ void __launch_bounds__(256) dwconv_nhwc8_kernel(const ConvArgs a, const int32_t* wint) {
  pdl_prologue();
  extern __shared__ int32_t dw_w[];   // [KH*KW][C]
  const uint32_t taps = a.KH * a.KW, C = a.C;
  for (uint32_t i = threadIdx.x; i < taps * C; i += blockDim.x) dw_w[(i % taps) * C + i / taps] = wint[i];
  __syncthreads();
  const uint32_t level = a.uniform_log2k;
  const uint32_t groups = C / 8u;
  const size_t total = (size_t)a.N * a.OH * a.OW * groups;
  const bool has_res = a.residual != nullptr;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const uint32_t g = (uint32_t)(idx % groups);
    const size_t pix = idx / groups;
    const uint32_t ox = (uint32_t)(pix % a.OW), oy = (uint32_t)((pix / a.OW) % a.OH);
    const uint32_t n = (uint32_t)(pix / ((size_t)a.OW * a.OH));
    const uint32_t c0 = g * 8u;
    long long acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (uint32_t kh = 0; kh < a.KH; ++kh) {
      const int iy = (int)(oy * a.stride + kh) - (int)a.pad;
      if (iy < 0 || iy >= (int)a.H) continue;
      for (uint32_t kw = 0; kw < a.KW; ++kw) {
        const int ix = (int)(ox * a.stride + kw) - (int)a.pad;
        if (ix < 0 || ix >= (int)a.W) continue;
        const uint2 xv = __ldcg(reinterpret_cast<const uint2*>(
            (const uint8_t*)a.x + (((size_t)n * a.H + iy) * a.W + ix) * C + c0));
        const int32_t* wr = dw_w + (kh * a.KW + kw) * C + c0;
        const int4 w0 = *reinterpret_cast<const int4*>(wr), w1 = *reinterpret_cast<const int4*>(wr + 4);
        const int ws[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
        const uint32_t xw[2] = {xv.x, xv.y};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t b = (xw[j >> 2] >> (8 * (j & 3))) & 0xFFu;
          const int xi = a.in_dtype == PSB_DT_U8 ? (int)b : (int)(int8_t)b;
          acc[j] += (long long)xi * (long long)ws[j];
        }
      }
    }
    const size_t oidx = pix * C + c0;
    uint32_t rw[2] = {0, 0};
    if (has_res) {
      const uint2 rv = __ldcg(reinterpret_cast<const uint2*>((const uint8_t*)a.residual + oidx));
      rw[0] = rv.x; rw[1] = rv.y;
    }
    uint32_t qw[2] = {0, 0};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t o = c0 + j;
      const float sc = ldexpf(a.scale[o], a.e_base[o] - (int)level);
      int rb = (int)((rw[j >> 2] >> (8 * (j & 3))) & 0xFFu);
      if (a.residual_dtype == PSB_DT_S8) rb = (int)(int8_t)rb;
      const float y = dequant(acc[j], sc, a.bias[o], has_res, rb, a.residual_scale, a.relu != 0);
      const int q = requant(y, a.inv_step, a.qmin, a.qmax);
      qw[j >> 2] |= ((uint32_t)q & 0xFFu) << (8 * (j & 3));
    }
    *reinterpret_cast<uint2*>((uint8_t*)a.q_out + oidx) = make_uint2(qw[0], qw[1]);
  }
}

// Depthwise 3x3, channels-last, one draw count, only codes wanted: a thread owns 4 channels x kDwCols output columns and
// walks down the rows of an image with its 36 filter values in registers.  Every input row is read once per thread, its
// bytes are extracted once and serve up to three output rows, whose sums are open at the same time (unrolled by three
// so that no sum moves).  The integer sum x * W_k over the nine taps (Eq. 9 summed over the draws) fits 32 bits whenever
// (largest activation) x (sum of |W_k| of the channel) stays below 2^31; the sampler keeps those sums, and a thread with
// a channel where it does not computes its outputs one by one in 64 bits.  The output stage is dequant()/requant() with
// the relu folded into the lower clamp (inv_step > 0), rounded by adding 1.5 * 2^23.
// Bound by the nine 32-bit multiply-adds per output (2 clocks each): 15 us for 144 channels @56, batch 64.  That layer
// with its sampling: 78.6 -> 51.4 us (a thread with 8 outputs of one row spent 48 logic clocks per output and spilled).
constexpr int kDwCols = 2;

struct DwConst {
  float res_scale, inv_step, lo_f, hi_f;
};

template <int S>
struct DwIn { static constexpr int kCols = (kDwCols - 1) * S + 3; };

// One output in 64 bits, straight from global memory (channels whose sums may not fit 32).
template <bool kSignedIn>
__device__ __noinline__ void dw_output64(const ConvArgs& a, const int32_t* wch, uint32_t n, uint32_t oy, uint32_t ox, uint32_t o) {
  long long acc = 0;
  for (uint32_t kh = 0; kh < 3u; ++kh) {
    const int iy = (int)(oy * a.stride + kh) - (int)a.pad;
    if ((unsigned)iy >= a.H) continue;
    for (uint32_t kw = 0; kw < 3u; ++kw) {
      const int ix = (int)(ox * a.stride + kw) - (int)a.pad;
      if ((unsigned)ix >= a.W) continue;
      acc += (long long)load_act(a.x, kSignedIn ? PSB_DT_S8 : PSB_DT_U8, (((size_t)n * a.H + iy) * a.W + ix) * a.C + o) *
             (long long)__ldca(wch + kh * 3u + kw);
    }
  }
  store_outputs(a, (((size_t)n * a.OH + oy) * a.OW + ox) * a.C + o, o, a.uniform_log2k, acc);
}

// kVec: channel counts that are multiples of 4 at 4-byte aligned addresses; otherwise words are put together from bytes.
template <int S, bool kSignedIn, bool kVec>
__global__ void __launch_bounds__(128, 5) dwconv3x3_kernel(const ConvArgs a, const int32_t* wint, const uint32_t* rowsum256,
                                                           uint32_t amax, uint32_t rows_per_thread) {
  pdl_prologue();
  constexpr int NC = DwIn<S>::kCols;
  const uint32_t C = a.C, G = (C + 3u) / 4u;
  const uint32_t segs = (a.OW + kDwCols - 1) / kDwCols, strips = (a.OH + rows_per_thread - 1u) / rows_per_thread;
  const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= a.N * strips * segs * G) return;      // the launcher keeps this below 2^32
  uint32_t t = idx / G;
  const uint32_t c0 = (idx - t * G) * 4u, left = kVec ? 4u : min(4u, C - c0);
  const uint32_t seg = t % segs; t /= segs;
  const uint32_t strip = t % strips, n = t / strips;
  const uint32_t ox0 = seg * kDwCols, oy0 = strip * rows_per_thread, oy1 = min(oy0 + rows_per_thread, a.OH);
  const uint32_t level = a.uniform_log2k;
  bool fits = true;
  for (uint32_t j = 0; j < left; ++j)
    fits = fits && (unsigned long long)__ldca(rowsum256 + (size_t)level * a.O + c0 + j) * 256ull * amax < (1ull << 31);
  if (!fits) {
    for (uint32_t oy = oy0; oy < oy1; ++oy)
      for (uint32_t ox = ox0; ox < min(ox0 + (uint32_t)kDwCols, a.OW); ++ox)
        for (uint32_t j = 0; j < left; ++j) dw_output64<kSignedIn>(a, wint + (size_t)(c0 + j) * 9u, n, oy, ox, c0 + j);
    return;
  }
  int w[4][9];
  if (kVec) {
    const int4* wp = reinterpret_cast<const int4*>(wint + (size_t)c0 * 9u);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int4 v = __ldca(wp + i);
      const int e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) w[(4 * i + q) / 9][(4 * i + q) % 9] = e[q];
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 9; ++q) w[j][q] = (uint32_t)j < left ? __ldca(wint + (size_t)(c0 + j) * 9u + q) : 0;
  }
  float sc[4], bi[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t o = (uint32_t)j < left ? c0 + j : c0;
    sc[j] = ldexpf(a.scale[o], a.e_base[o] - (int)level);
    bi[j] = a.bias[o];
  }
  const float lo_f = a.relu && a.qmin < 0 ? 0.0f : (float)a.qmin, hi_f = (float)a.qmax;
  const bool has_res = a.residual != nullptr, res_signed = a.residual_dtype == PSB_DT_S8;
  const int ix0 = (int)(ox0 * S) - (int)a.pad;
  bool col_in[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) col_in[q] = (unsigned)(ix0 + q) < a.W;
  const size_t row_bytes = (size_t)a.W * C, out_row_bytes = (size_t)a.OW * C;
  const int iy0 = (int)(oy0 * S) - (int)a.pad;
  // the next input row to load (its number and address) and the next output row to write, both moved on row by row
  int iy = iy0;
  const uint8_t* in_row = (const uint8_t*)a.x + (((ptrdiff_t)n * a.H + iy0) * (ptrdiff_t)a.W + ix0) * (ptrdiff_t)C + c0;
  size_t out_at = (((size_t)n * a.OH + oy0) * a.OW + ox0) * C + c0;
  const bool second = ox0 + 1u < a.OW;
  static_assert(kDwCols == 2, "the last segment of a row has one or two columns");

  auto load_word = [&](const uint8_t* at) -> uint32_t {
    if (kVec) return __ldcg(reinterpret_cast<const uint32_t*>(at));
    uint32_t v = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((uint32_t)j < left) v |= (uint32_t)at[j] << (8 * j);
    return v;
  };
  auto load_row = [&](uint32_t (&raw)[NC]) {
    const bool in = (unsigned)iy < a.H;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      raw[q] = 0u;
      if (in && col_in[q]) raw[q] = load_word(in_row + (uint32_t)q * C);
    }
    ++iy;
    in_row += row_bytes;
  };
  auto extract = [&](const uint32_t (&raw)[NC], const int j, int (&x)[NC]) {
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const uint32_t b = (raw[q] >> (8 * j)) & 0xFFu;
      x[q] = kSignedIn ? (int)(signed char)b : (int)b;
    }
  };
  // adds row `kh` of the filter on one input row to the sums of channel j (kh == 0 starts them)
  auto add_row = [&](const int (&x)[NC], int (&sum)[kDwCols][4], const int j, const int kh) {
#pragma unroll
    for (int i = 0; i < kDwCols; ++i) {
      int v = kh == 0 ? 0 : sum[i][j];
      v += x[i * S] * w[j][kh * 3];
      v += x[i * S + 1] * w[j][kh * 3 + 1];
      v += x[i * S + 2] * w[j][kh * 3 + 2];
      sum[i][j] = v;
    }
  };
  int acc[3][kDwCols][4];
  auto emit = [&](const int (&sum)[kDwCols][4]) {
#pragma unroll
    for (int i = 0; i < kDwCols; ++i) {
      if (i && !second) break;
      const size_t at = out_at + (uint32_t)i * C;
      uint32_t rw = 0u;
      if (has_res) {
        const uint8_t* rp = (const uint8_t*)a.residual + at;
        rw = load_word(rp);
      }
      uint32_t q[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float y = __fmaf_rn(__int2float_rn(sum[i][j]), sc[j], bi[j]);
        if (has_res) {
          const uint32_t rb = (rw >> (8 * j)) & 0xFFu;
          y = __fmaf_rn(res_signed ? (float)(int)(signed char)rb : (float)rb, a.residual_scale, y);
        }
        q[j] = __float_as_uint(__fadd_rn(fminf(fmaxf(__fmul_rn(y, a.inv_step), lo_f), hi_f), 12582912.0f));
      }
      const uint32_t word = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
      if (kVec) {
        *reinterpret_cast<uint32_t*>((uint8_t*)a.q_out + at) = word;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((uint32_t)j < left) ((uint8_t*)a.q_out)[at + j] = (uint8_t)(word >> (8 * j));
      }
    }
    out_at += out_row_bytes;
  };
  const uint32_t rows = oy1 - oy0;
  uint32_t cur[NC], nxt[NC];
  load_row(cur);
  load_row(nxt);
  if (S == 1) {
    // input row r opens output r, adds to output r - 1 and closes output r - 2
    auto step = [&](uint32_t r, int (&open)[kDwCols][4], int (&mid)[kDwCols][4], int (&close)[kDwCols][4]) {
      uint32_t raw[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) { raw[q] = cur[q]; cur[q] = nxt[q]; }
      if (r < rows) load_row(nxt);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int x[NC];
        extract(raw, j, x);
        add_row(x, open, j, 0);
        add_row(x, mid, j, 1);
        add_row(x, close, j, 2);
      }
      if (r >= 2u && r - 2u < rows) emit(close);
    };
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < kDwCols; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][i][j] = 0;
    for (uint32_t r = 0; r < rows + 2u; r += 3u) {
      step(r, acc[0], acc[2], acc[1]);
      step(r + 1u, acc[1], acc[0], acc[2]);
      step(r + 2u, acc[2], acc[1], acc[0]);
    }
  } else {
    // two input rows per output row; the second one closes it and opens the next
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int x[NC];
      extract(cur, j, x);
      add_row(x, acc[0], j, 0);
    }
    load_row(cur);
    for (uint32_t r = 0; r < rows; ++r) {
      uint32_t mid[NC], end[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) { mid[q] = nxt[q]; end[q] = cur[q]; }
      if (r + 1u < rows) { load_row(nxt); load_row(cur); }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int x[NC];
        extract(mid, j, x);
        add_row(x, acc[0], j, 1);
        extract(end, j, x);
        add_row(x, acc[0], j, 2);
        add_row(x, acc[1], j, 0);
      }
      emit(acc[0]);
#pragma unroll
      for (int i = 0; i < kDwCols; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[0][i][j] = acc[1][i][j];
    }
  }
}

// [rows][C] -> [rows][pitch] (pitch a multiple of 16, zero beyond C): the copy engine wants rows that are 16-byte
// multiples at 16-byte addresses.  Bound by memory; a thread writes one 16-byte piece, put together from the aligned
// words it overlaps (byte loads at the tensor's two ends only).
__global__ void __launch_bounds__(256) repack_rows_kernel(const uint8_t* src, uint8_t* __restrict__ dst, size_t rows,
                                                         uint32_t C, uint32_t pitch, uint32_t is_signed, uint32_t limit,
                                                         uint32_t* __restrict__ err) {
  pdl_prologue();
  const uint32_t pieces = pitch / 16u;
  const size_t total = rows * pieces;
  const uint8_t* const end = src + rows * C;
  bool bad = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t row = i / pieces;
    const uint32_t c0 = (uint32_t)(i - row * pieces) * 16u;
    const uint32_t count = c0 < C ? min(16u, C - c0) : 0u;
    const uint8_t* from = src + row * C + c0;
    const uint32_t mis = (uint32_t)((uintptr_t)from & 3u);
    const uint8_t* word = from - mis;
    uint32_t w[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      w[j] = 0u;
      const uint8_t* q = word + 4 * j;
      if ((uint32_t)(4 * j) >= mis + count) continue;
      if (q >= src && q + 4 <= end) {
        w[j] = __ldca(reinterpret_cast<const uint32_t*>(q));
      } else {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (q + b >= src && q + b < end) w[j] |= (uint32_t)q[b] << (8 * b);
      }
    }
    uint32_t v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = __funnelshift_r(w[j], w[j + 1], 8u * mis);
      const uint32_t have = count > (uint32_t)(4 * j) ? count - 4 * j : 0u;      // bytes of this word that exist
      if (have < 4u) v[j] &= (1u << (8u * have)) - 1u;
      bad |= bytes_beyond(v[j], is_signed, limit);
    }
    *reinterpret_cast<uint4*>(dst + row * pitch + c0) = make_uint4(v[0], v[1], v[2], v[3]);
  }
  if (bad) atomicOr(err, kDevErrRange);
}

// Largest byte magnitude of a tensor against the bound the caller gave (PSB_CHECK_RANGE): 16 bytes per
// thread and iteration, the ragged tail byte by byte.
__global__ void range_check_kernel(const uint8_t* x, size_t bytes, uint32_t is_signed, uint32_t limit,
                                   uint32_t* __restrict__ err) {
  pdl_prologue();
  bool bad = false;
  const size_t head = min(bytes, (size_t)((16u - ((uintptr_t)x & 15u)) & 15u));   // bytes before 16-byte alignment
  const size_t n16 = (bytes - head) / 16u;
  const uint4* x16 = reinterpret_cast<const uint4*>(x + head);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x) {
    const uint4 v = __ldcg(x16 + i);
    bad |= bytes_beyond(v.x, is_signed, limit) | bytes_beyond(v.y, is_signed, limit) |
           bytes_beyond(v.z, is_signed, limit) | bytes_beyond(v.w, is_signed, limit);
  }
  if (blockIdx.x == 0) {
    const size_t tail0 = head + n16 * 16u;
    for (size_t i = threadIdx.x; i < head; i += blockDim.x) bad |= bytes_beyond((uint32_t)x[i], is_signed, limit);
    for (size_t i = tail0 + threadIdx.x; i < bytes; i += blockDim.x) bad |= bytes_beyond((uint32_t)x[i], is_signed, limit);
  }
  if (bad) atomicOr(err, kDevErrRange);
}

// Explicit gather of the activation matrix for filters with few input channels (e.g. a 7x7
// stem on 3 channels): row m = output location; filter row kh occupies bytes
// [kh * run_pitch, kh * run_pitch + KW * C) of it, which in a channels-last image is one
// contiguous run of the input row iy0 + kh; the rest of the matrix row is zero.  Values are
// stored minus `offset` (0 or 128) as signed bytes; a padded input position is the value 0, i.e.
// -offset.  A block handles a strip of up to kIm2colPix consecutive output locations of
// kIm2colRows consecutive output rows: the input-row spans they touch are staged in shared
// memory, each at the byte offset that keeps its 16-byte pieces aligned with global memory
// (whole-piece copies; single bytes only at the image's edges), then each thread copies whole
// runs: aligned shared-memory words, a funnel shift by the byte misalignment, 8-byte stores.
constexpr uint32_t kIm2colPix = 128;
constexpr uint32_t kIm2colRows = 2;

__host__ __device__ __forceinline__ uint32_t im2col_span_pitch(uint32_t stride, uint32_t C, uint32_t run_pitch) {
  // alignment shift (< 16) + the last pixel's run, read up to run_pitch + 7 bytes past its start in whole words
  return (15u + (kIm2colPix - 1u) * stride * C + run_pitch + 12u + 15u) & ~15u;
}

__global__ void __launch_bounds__(256) im2col_s8_kernel(const ConvArgs a, uint32_t kpad, uint32_t run_pitch,
                                                       uint32_t offset, uint32_t limit, int8_t* __restrict__ dst) {
  pdl_prologue();
  bool bad = false;
  extern __shared__ __align__(16) uint32_t im2col_smem[];     // [staged rows][span_pitch / 4] words
  __shared__ uint32_t row_adj[(kIm2colRows - 1u) * 8u + 128u];   // per staged row: byte offset of the span's start
  const uint32_t span_pitch = im2col_span_pitch(a.stride, a.C, run_pitch);
  const uint32_t strips = (a.OW + kIm2colPix - 1) / kIm2colPix;
  const uint32_t row_groups = (a.OH + kIm2colRows - 1) / kIm2colRows;
  const uint32_t strip = blockIdx.x % strips;
  const uint32_t oy0 = ((blockIdx.x / strips) % row_groups) * kIm2colRows;
  const uint32_t n = blockIdx.x / (strips * row_groups);
  const uint32_t nrows = min(kIm2colRows, a.OH - oy0);
  const uint32_t ox0 = strip * kIm2colPix;
  const uint32_t npix = min(kIm2colPix, a.OW - ox0);
  const int ix0 = (int)(ox0 * a.stride) - (int)a.pad;         // leftmost input column of the strip
  const int iy0 = (int)(oy0 * a.stride) - (int)a.pad;         // topmost input row
  const uint32_t staged = (nrows - 1u) * a.stride + a.KH;     // input rows the block touches
  const uint32_t span_bytes = ((npix - 1u) * a.stride + a.KW) * a.C;
  const uint8_t* x = (const uint8_t*)a.x;
  const uint32_t flip = offset ? 0x80808080u : 0u;            // v - 128 == v ^ 0x80 as a byte
  const uint32_t fill = (0u - offset) & 0xFFu;
  const uint32_t fill4 = fill * 0x01010101u;
  const uint32_t is_signed = a.in_dtype == PSB_DT_S8 ? 1u : 0u;
  // bytes [lo_b, hi_b) of a span lie inside the image row
  const int lo_b = ix0 < 0 ? -ix0 * (int)a.C : 0;
  const int hi_b = min((int)span_bytes, ((int)a.W - ix0) * (int)a.C);
  const uint32_t pieces = span_pitch / 16u;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  for (uint32_t sr = warp; sr < staged; sr += 8u) {
    const int iy = iy0 + (int)sr;
    const bool row_in = iy >= 0 && iy < (int)a.H;
    const uint8_t* src = x + (((size_t)n * a.H + (row_in ? iy : 0)) * a.W) * a.C + (ptrdiff_t)ix0 * (int)a.C;
    const uint32_t adj = (uint32_t)((uintptr_t)src & 15u);    // span byte b sits at shared byte adj + b
    if (lane == 0) row_adj[sr] = adj;
    const uint8_t* src16 = src - adj;                          // 16-byte aligned
    uint32_t* out_row = im2col_smem + sr * (span_pitch / 4u);
    for (uint32_t pc = lane; pc < pieces; pc += 32u) {
      const int b0 = (int)(pc * 16u) - (int)adj;               // span byte of the piece's first byte
      uint4 v;
      if (row_in && b0 >= lo_b && b0 + 16 <= hi_b) {
        v = __ldcg(reinterpret_cast<const uint4*>(src16 + pc * 16u));
        bad |= bytes_beyond(v.x, is_signed, limit) | bytes_beyond(v.y, is_signed, limit) |
               bytes_beyond(v.z, is_signed, limit) | bytes_beyond(v.w, is_signed, limit);
        v.x ^= flip; v.y ^= flip; v.z ^= flip; v.w ^= flip;
      } else {
        uint32_t wv[4] = {fill4, fill4, fill4, fill4};
        if (row_in && b0 + 16 > lo_b && b0 < hi_b) {
          for (int j = 0; j < 16; ++j) {
            const int b = b0 + j;
            if (b >= lo_b && b < hi_b) {
              const uint32_t raw = src[b];
              bad |= bytes_beyond(raw, is_signed, limit);
              wv[j >> 2] = (wv[j >> 2] & ~(0xFFu << (8 * (j & 3)))) | (((raw ^ offset) & 0xFFu) << (8 * (j & 3)));
            }
          }
        }
        v = make_uint4(wv[0], wv[1], wv[2], wv[3]);
      }
      *reinterpret_cast<uint4*>(out_row + pc * 4u) = v;
    }
  }
  if (bad) atomicOr(a.err, kDevErrRange);
  __syncthreads();
  const uint32_t run = a.KW * a.C;                            // bytes of one filter row
  const uint32_t words = run_pitch / 4u;
  const uint32_t tail0 = a.KH * run_pitch;                    // zero bytes [tail0, kpad)
  const uint32_t items = a.KH + (kpad > tail0 ? 1u : 0u);
  const uint32_t per_row = npix * items;
  for (uint32_t t = threadIdx.x; t < nrows * per_row; t += blockDim.x) {
    const uint32_t ry = t / per_row, t1 = t - ry * per_row;
    const uint32_t px = t1 / items, kh = t1 - px * items;
    const size_t m = ((size_t)n * a.OH + oy0 + ry) * a.OW + ox0 + px;
    int8_t* out = dst + m * kpad + kh * run_pitch;
    if (kh == a.KH) {
      for (uint32_t b = 0; b < kpad - tail0; b += 8u) *reinterpret_cast<uint2*>(out + b) = make_uint2(0u, 0u);
      continue;
    }
    const uint32_t sr = ry * a.stride + kh;
    const uint32_t o = row_adj[sr] + px * a.stride * a.C;     // byte offset of the run in the staged row
    const uint32_t* wsrc = im2col_smem + sr * (span_pitch / 4u) + (o >> 2);
    const uint32_t sh = (o & 3u) * 8u;
    uint32_t lo = wsrc[0];
    for (uint32_t w = 0; w < words; w += 2u) {
      const uint32_t mid = wsrc[w + 1], hi = wsrc[w + 2];
      uint32_t v0 = __funnelshift_r(lo, mid, sh), v1 = __funnelshift_r(mid, hi, sh);
      // bytes at or beyond the run are K padding: zero
      const uint32_t b0 = w * 4u;
      if (b0 + 4u > run) v0 = b0 >= run ? 0u : (v0 & (0xFFFFFFFFu >> (8u * (b0 + 4u - run))));
      if (b0 + 8u > run) v1 = b0 + 4u >= run ? 0u : (v1 & (0xFFFFFFFFu >> (8u * (b0 + 8u - run))));
      *reinterpret_cast<uint2*>(out + b0) = make_uint2(v0, v1);
      lo = hi;
    }
  }
}

// [N][C][HW] -> [N][HW][pitch], elements of 1 byte, zero beyond C, through a 32x33 tile.
__global__ void nchw_to_nhwc_u8_kernel(const uint8_t* src, uint8_t* dst, uint32_t C, uint32_t HW, uint32_t pitch,
                                       uint32_t is_signed, uint32_t limit, uint32_t* __restrict__ err) {
  pdl_prologue();
  __shared__ uint8_t tile[32][33];
  const size_t base = (size_t)blockIdx.z * C * HW, dbase = (size_t)blockIdx.z * pitch * HW;
  const uint32_t p0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  bool bad = false;
  for (uint32_t r = threadIdx.y; r < 32; r += blockDim.y) {
    uint32_t c = c0 + r, p = p0 + threadIdx.x;
    uint8_t v = 0;
    if (c < C && p < HW) {
      v = src[base + (size_t)c * HW + p];
      bad |= bytes_beyond((uint32_t)v, is_signed, limit);
    }
    tile[r][threadIdx.x] = v;
  }
  if (bad) atomicOr(err, kDevErrRange);
  __syncthreads();
  for (uint32_t r = threadIdx.y; r < 32; r += blockDim.y) {
    uint32_t p = p0 + r, c = c0 + threadIdx.x;
    if (c < pitch && p < HW) dst[dbase + (size_t)p * pitch + c] = tile[threadIdx.x][r];
  }
}

// The same for C and HW multiples of 4, four bytes at a time.  A block moves 32 channels x 128
// locations.  Warp i takes channels 4i..4i+3: each lane loads 4 locations of each of them (four
// 128-byte runs per warp), transposes the 4x4 bytes in registers and parks the four words (one
// per location, 4 channels each) in shared memory with one 16-byte store.  Then 8 consecutive
// lanes write the 32 channel bytes of one location: whole 32-byte sectors, no bank conflicts
// (row pitch 132 words: bank = 4 * quad + location).
__global__ void __launch_bounds__(256) nchw_to_nhwc_u8x4_kernel(const uint8_t* src,
                                                               uint8_t* __restrict__ dst, uint32_t C,
                                                               uint32_t HW, uint32_t pitch, uint32_t is_signed,
                                                               uint32_t limit, uint32_t* __restrict__ err) {
  pdl_prologue();
  __shared__ __align__(16) uint32_t tile[8][132];
  const size_t base = (size_t)blockIdx.z * C * HW, dbase = (size_t)blockIdx.z * pitch * HW;
  const uint32_t p0 = blockIdx.x * 128u, c0 = blockIdx.y * 32u;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  {
    const uint32_t c = c0 + 4u * warp, p = p0 + 4u * lane;
    uint32_t r[4] = {0u, 0u, 0u, 0u};
    if (c < C && p < HW) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        r[k] = __ldcg(reinterpret_cast<const uint32_t*>(src + base + (size_t)(c + k) * HW + p));
      if (bytes_beyond(r[0], is_signed, limit) | bytes_beyond(r[1], is_signed, limit) |
          bytes_beyond(r[2], is_signed, limit) | bytes_beyond(r[3], is_signed, limit))
        atomicOr(err, kDevErrRange);
    }
    const uint32_t a = __byte_perm(r[0], r[1], 0x5140), b = __byte_perm(r[2], r[3], 0x5140);
    const uint32_t cc = __byte_perm(r[0], r[1], 0x7362), d = __byte_perm(r[2], r[3], 0x7362);
    *reinterpret_cast<uint4*>(&tile[warp][4u * lane]) =
        make_uint4(__byte_perm(a, b, 0x5410), __byte_perm(a, b, 0x7632), __byte_perm(cc, d, 0x5410),
                   __byte_perm(cc, d, 0x7632));
  }
  __syncthreads();
  const uint32_t q = threadIdx.x & 7u;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint32_t pl = (threadIdx.x >> 3) + 32u * r;
    const uint32_t p = p0 + pl, c = c0 + 4u * q;
    if (p < HW && c < pitch) *reinterpret_cast<uint32_t*>(dst + dbase + (size_t)p * pitch + c) = tile[q][pl];
  }
}

__global__ void maxpool_kernel(const uint8_t* x, uint32_t nchw, uint32_t N, uint32_t C,
                               uint32_t H, uint32_t W, uint32_t k, uint32_t stride, uint32_t pad,
                               uint32_t OH, uint32_t OW, uint8_t* __restrict__ out) {
  pdl_prologue();
  const size_t total = (size_t)N * OH * OW * C;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    uint32_t c, ox, oy, n;
    if (nchw) {
      ox = idx % OW; oy = (idx / OW) % OH; c = (idx / ((size_t)OW * OH)) % C;
      n = idx / ((size_t)OW * OH * C);
    } else {
      c = idx % C; ox = (idx / C) % OW; oy = (idx / ((size_t)C * OW)) % OH;
      n = idx / ((size_t)C * OW * OH);
    }
    int best = 0;
    for (uint32_t kh = 0; kh < k; ++kh) {
      int iy = (int)(oy * stride + kh) - (int)pad;
      if (iy < 0 || iy >= (int)H) continue;
      for (uint32_t kw = 0; kw < k; ++kw) {
        int ix = (int)(ox * stride + kw) - (int)pad;
        if (ix < 0 || ix >= (int)W) continue;
        size_t xi = nchw ? (((size_t)n * C + c) * H + iy) * W + ix
                         : (((size_t)n * H + iy) * W + ix) * C + c;
        best = max(best, (int)x[xi]);
      }
    }
    out[idx] = (uint8_t)best;
  }
}

// Channels-last max-pooling, 16 channels per thread: 16-byte loads, byte-wise maxima.
__global__ void __launch_bounds__(256) maxpool_nhwc16_kernel(const uint8_t* x, uint32_t N, uint32_t C,
                                                            uint32_t H, uint32_t W, uint32_t k, uint32_t stride,
                                                            uint32_t pad, uint32_t OH, uint32_t OW,
                                                            uint8_t* __restrict__ out) {
  pdl_prologue();
  const uint32_t groups = C / 16u;
  const size_t total = (size_t)N * OH * OW * groups;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const uint32_t g = (uint32_t)(idx % groups);
    const size_t pix = idx / groups;
    const uint32_t ox = (uint32_t)(pix % OW), oy = (uint32_t)((pix / OW) % OH);
    const uint32_t n = (uint32_t)(pix / ((size_t)OW * OH));
    uint4 best = make_uint4(0, 0, 0, 0);
    for (uint32_t kh = 0; kh < k; ++kh) {
      const int iy = (int)(oy * stride + kh) - (int)pad;
      if (iy < 0 || iy >= (int)H) continue;
      for (uint32_t kw = 0; kw < k; ++kw) {
        const int ix = (int)(ox * stride + kw) - (int)pad;
        if (ix < 0 || ix >= (int)W) continue;
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(x + (((size_t)n * H + iy) * W + ix) * C + g * 16u));
        best.x = __vmaxu4(best.x, v.x); best.y = __vmaxu4(best.y, v.y);
        best.z = __vmaxu4(best.z, v.z); best.w = __vmaxu4(best.w, v.w);
      }
    }
    *reinterpret_cast<uint4*>(out + pix * C + g * 16u) = best;
  }
}

// One warp per (n, c): integer sum over H*W, then one re-quantisation.
// Channels-last, 16 channels per thread: every load is 16 bytes, neighbouring threads read neighbouring
// channel groups of the same position.
__global__ void __launch_bounds__(128) avgpool_nhwc16_kernel(const uint8_t* x, uint32_t N, uint32_t C, uint32_t HW,
                                                             float pool_mul, int qmin, int qmax, uint8_t* __restrict__ out) {
  pdl_prologue();
  const uint32_t groups = C / 16u;
  const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= N * groups) return;
  const uint32_t n = idx / groups, g = idx - n * groups;
  const uint8_t* src = x + (size_t)n * HW * C + g * 16u;
  int sum[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) sum[j] = 0;
#pragma unroll 4
  for (uint32_t p = 0; p < HW; ++p) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(src + (size_t)p * C));
    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 16; ++j) sum[j] += (int)((w4[j >> 2] >> (8 * (j & 3))) & 0xFFu);
  }
  uint32_t q[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 16; ++j)
    q[j >> 2] |= ((uint32_t)requant((float)sum[j], pool_mul, qmin, qmax) & 0xFFu) << (8 * (j & 3));
  *reinterpret_cast<uint4*>(out + (size_t)n * C + g * 16u) = make_uint4(q[0], q[1], q[2], q[3]);
}

__global__ void avgpool_kernel(const uint8_t* x, uint32_t nchw, uint32_t N, uint32_t C,
                               uint32_t HW, float pool_mul, int qmin, int qmax,
                               uint8_t* __restrict__ out) {
  pdl_prologue();
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= N * C) return;
  const uint32_t n = warp / C, c = warp % C;
  int sum = 0;
  for (uint32_t p = lane; p < HW; p += 32) {
    size_t xi = nchw ? ((size_t)n * C + c) * HW + p : ((size_t)n * HW + p) * C + c;
    sum += x[xi];
  }
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) out[warp] = (uint8_t)requant((float)sum, pool_mul, qmin, qmax);
}

uint32_t grid_for(size_t total, uint32_t threads) {
  size_t b = (total + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > kSms * 32u) b = kSms * 32u;
  return (uint32_t)b;
}

}  // namespace

cudaError_t launch_repack_rows(const void* src, void* dst, size_t rows, uint32_t C, uint32_t pitch, uint32_t is_signed,
                               uint32_t limit, uint32_t* err, cudaStream_t s) {
  launch_pdl(repack_rows_kernel, grid_for(rows * (pitch / 16u), 256), 256, 0, s, (const uint8_t*)src, (uint8_t*)dst, rows, C,
             pitch, is_signed, limit, err);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_range_check(const void* x, size_t bytes, uint32_t is_signed, uint32_t limit, uint32_t* err,
                               cudaStream_t s) {
  uint32_t blocks = grid_for(bytes / 16 + 1, 256);
  if (blocks > kSms * 8u) blocks = kSms * 8u;
  launch_pdl(range_check_kernel, blocks, 256, 0, s, (const uint8_t*)x, bytes, is_signed, limit, err);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_shift_add(const ConvArgs& a, const WintTable& wt, const uint32_t* rowsum256, uint32_t amax,
                             cudaStream_t s) {
  size_t total = (size_t)a.N * a.OH * a.OW * a.O;
  // depthwise 3x3, channels-last, one draw count, only codes wanted
  if (a.groups == a.C && a.O == a.C && a.KH == 3 && a.KW == 3 && a.stride <= 2u && !a.kmap && a.q_out && !a.f32_out && !a.acc_out &&
      !a.out_nchw && a.inv_step > 0.0f) {
    // Rows per thread: the machine holds five blocks of 128 threads per SM; among the strip lengths the one with the
    // least (waves of blocks) x (rows + what a thread spends before its first row, about four rows' worth)
    const uint64_t columns = (uint64_t)a.N * ((a.OW + kDwCols - 1) / kDwCols) * ((a.C + 3u) / 4u);
    uint32_t rows = a.OH;
    uint64_t best = ~0ull;
    for (uint32_t strips = 1; strips <= 32u && strips <= a.OH; ++strips) {
      const uint32_t r = (a.OH + strips - 1) / strips;
      const uint64_t waves = (columns * ((a.OH + r - 1) / r) + 5ull * kSms * 128 - 1) / (5ull * kSms * 128);
      const uint64_t cost = waves * (r + 4u);
      if (cost < best) { best = cost; rows = r; }
    }
    const uint64_t threads = columns * ((a.OH + rows - 1) / rows);
    if (threads < (1ull << 32) - 256u) {
      const uint32_t blocks = (uint32_t)((threads + 127u) / 128u);
      const int32_t* wl = wt.w[a.uniform_log2k];
      const bool vec = a.C % 4u == 0 && !(((uintptr_t)a.x | (uintptr_t)a.q_out | (uintptr_t)a.residual) & 3u);
#define PSB_DW(SV, SG, VC) launch_pdl(dwconv3x3_kernel<SV, SG, VC>, blocks, 128, 0, s, a, wl, rowsum256, amax, rows)
#define PSB_DW_V(SV, SG) do { if (vec) PSB_DW(SV, SG, true); else PSB_DW(SV, SG, false); } while (0)
      const bool sg = a.in_dtype == PSB_DT_S8;
      if (a.stride == 1) { if (sg) PSB_DW_V(1, true); else PSB_DW_V(1, false); }
      else { if (sg) PSB_DW_V(2, true); else PSB_DW_V(2, false); }
#undef PSB_DW_V
#undef PSB_DW
      note_launch();
      return cudaGetLastError();
    }
  }
  // other depthwise filters, channel counts that are multiples of 8: eight channels per thread
  const size_t dw_smem = (size_t)a.KH * a.KW * a.C * sizeof(int32_t);
  if (a.groups == a.C && a.O == a.C && a.C % 8u == 0 && !a.kmap && a.q_out && !a.f32_out && !a.acc_out &&
      !a.out_nchw && dw_smem <= 64 * 1024 &&
      !(((uintptr_t)a.x | (uintptr_t)a.q_out | (uintptr_t)a.residual) & 7u)) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
      cudaFuncSetAttribute(dwconv_nhwc8_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
      attr_set[dev] = true;
    }
    uint32_t blocks = grid_for(total / 8, 256);
    if (blocks > kSms * 4u) blocks = kSms * 4u;
    launch_pdl(dwconv_nhwc8_kernel, blocks, 256, dw_smem, s, a, wt.w[a.uniform_log2k]); note_launch();
    return cudaGetLastError();
  }
  launch_pdl(conv_direct_kernel, grid_for(total, 256), 256, 0, s, a, wt); note_launch();
  return cudaGetLastError();
}

namespace {
struct DenseGrid {
  uint32_t lanes;      // per output channel
  bool one;            // one location per block row, not kPlaneLocations
  bool plain;          // one tap, no stride, no padding
  uint32_t x, y;
};
DenseGrid dense_grid(const ConvArgs& a, const psb_weights* wt) {
  DenseGrid g;
  const uint32_t kp = wt->n_kb * wt->bk, M = a.N * a.OH * a.OW;
  g.lanes = 1;
  while (g.lanes < 32u && g.lanes * 16u < kp) g.lanes *= 2u;
  g.one = a.kmap || M == 1u;
  g.plain = !wt->packed_k && a.KH * a.KW == 1u && a.stride == 1u && a.pad == 0u;
  g.x = (a.O + 256u / g.lanes - 1u) / (256u / g.lanes);
  g.y = g.one ? M : (M + kPlaneLocations - 1u) / kPlaneLocations;
  return g;
}
}  // namespace

uint32_t dense_planes_rounds(const ConvArgs& a, const psb_weights* wt, int sm_count) {
  const DenseGrid g = dense_grid(a, wt);
  const uint64_t slots = (uint64_t)sm_count * (g.plain ? kPlainBlocks : kTapBlocks);
  return g.y == 1u ? 1u : (uint32_t)(((uint64_t)g.x * g.y + slots - 1u) / slots);
}

cudaError_t launch_dense_planes(const ConvArgs& a, const psb_weights* wt, cudaStream_t s) {
  DensePlanes w;
  for (int l = 0; l < kMaxLevels; ++l) {
    w.p[l] = wt->level[l].planes;
    w.count[l] = (uint8_t)wt->level[l].planes_count;
  }
  w.bk = wt->bk;
  w.n_kb = wt->n_kb;
  w.tap_pieces = wt->packed_k ? 0u : wt->n_cb * wt->bk / 16u;
  w.run_pitch = wt->run_pitch;
  w.per_tap = w.tap_pieces ? 1.0f / (float)w.tap_pieces : 0.0f;
  w.per_kw = 1.0f / (float)a.KW;
  const DenseGrid g = dense_grid(a, wt);
  const uint32_t kp = w.n_kb * w.bk, M = a.N * a.OH * a.OW;
  const dim3 grid(g.x, g.y < 65535u ? g.y : 65535u);
  const size_t smem = (size_t)(g.one ? 1 : kPlaneLocations) * (kp < kPlaneSegment ? kp : kPlaneSegment);
  const bool sg = a.in_dtype == PSB_DT_S8;
#define PSB_DP(NB, SG, PL) launch_pdl(dense_planes_kernel<NB, SG, PL>, grid, dim3(256), smem, s, a, w, M, g.lanes)
#define PSB_DP_SG(NB, PL) do { if (sg) PSB_DP(NB, true, PL); else PSB_DP(NB, false, PL); } while (0)
  if (g.one && g.plain) PSB_DP_SG(1, true);
  else if (g.one) PSB_DP_SG(1, false);
  else if (g.plain) PSB_DP_SG(kPlaneLocations, true);
  else PSB_DP_SG(kPlaneLocations, false);
#undef PSB_DP_SG
#undef PSB_DP
  note_launch();
  return cudaGetLastError();
}

size_t im2col_s8_smem(const ConvArgs& a, uint32_t run_pitch) {
  return (size_t)((kIm2colRows - 1u) * a.stride + a.KH) * im2col_span_pitch(a.stride, a.C, run_pitch);
}

cudaError_t launch_im2col_s8(const ConvArgs& a, uint32_t kpad, uint32_t run_pitch, uint32_t offset, int8_t* dst,
                             uint32_t limit, cudaStream_t s) {
  const uint32_t strips = (a.OW + kIm2colPix - 1) / kIm2colPix;
  const uint32_t row_groups = (a.OH + kIm2colRows - 1) / kIm2colRows;
  const size_t smem = im2col_s8_smem(a, run_pitch);
  if (smem > 48 * 1024 || (uint64_t)a.N * row_groups * strips >= (1ull << 31) || run_pitch % 8u || kpad % 16u ||
      (offset != 0u && offset != 128u) || a.KH * run_pitch > kpad || (kIm2colRows - 1u) * a.stride + a.KH > 128u)
    return cudaErrorInvalidValue;
  launch_pdl(im2col_s8_kernel, a.N * row_groups * strips, 256, smem, s, a, kpad, run_pitch, offset, limit, dst);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_nchw_to_nhwc(const void* src, void* dst, uint32_t N, uint32_t C, uint32_t HW, uint32_t pitch,
                                uint32_t is_signed, uint32_t limit, uint32_t* err, cudaStream_t s) {
  if (C % 4u == 0 && pitch % 4u == 0 && HW % 4u == 0 && !(((uintptr_t)src | (uintptr_t)dst) & 3u)) {
    dim3 grid4((HW + 127) / 128, (pitch + 31) / 32, N);
    launch_pdl(nchw_to_nhwc_u8x4_kernel, grid4, 256, 0, s, (const uint8_t*)src, (uint8_t*)dst, C, HW, pitch, is_signed,
               limit, err);
  } else {
    dim3 grid((HW + 31) / 32, (pitch + 31) / 32, N), block(32, 8);
    launch_pdl(nchw_to_nhwc_u8_kernel, grid, block, 0, s, (const uint8_t*)src, (uint8_t*)dst, C, HW, pitch, is_signed, limit,
               err);
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_maxpool(const uint8_t* x, uint32_t nchw, uint32_t N, uint32_t C, uint32_t H,
                           uint32_t W, uint32_t k, uint32_t stride, uint32_t pad, uint8_t* out,
                           cudaStream_t s) {
  uint32_t OH = (H + 2 * pad - k) / stride + 1, OW = (W + 2 * pad - k) / stride + 1;
  size_t total = (size_t)N * OH * OW * C;
  if (!nchw && C % 16u == 0 && !(((uintptr_t)x | (uintptr_t)out) & 15u))
    launch_pdl(maxpool_nhwc16_kernel, grid_for(total / 16, 256), 256, 0, s, x, N, C, H, W, k, stride, pad, OH, OW, out);
  else
    launch_pdl(maxpool_kernel, grid_for(total, 256), 256, 0, s, x, nchw, N, C, H, W, k, stride, pad, OH, OW, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_avgpool(const uint8_t* x, uint32_t nchw, uint32_t N, uint32_t C, uint32_t H,
                           uint32_t W, float pool_mul, int32_t qmin, int32_t qmax, uint8_t* out,
                           cudaStream_t s) {
  if (!nchw && C % 16u == 0 && !(((uintptr_t)x | (uintptr_t)out) & 15u) && (uint64_t)N * (C / 16u) < (1ull << 31)) {
    const uint32_t threads = N * (C / 16u);
    launch_pdl(avgpool_nhwc16_kernel, (threads + 127u) / 128u, 128, 0, s, x, N, C, H * W, pool_mul, qmin, qmax, out);
    note_launch();
    return cudaGetLastError();
  }
  size_t warps = (size_t)N * C;
  uint32_t blocks = (uint32_t)((warps * 32 + 255) / 256);
  launch_pdl(avgpool_kernel, blocks, 256, 0, s, x, nchw, N, C, H * W, pool_mul, qmin, qmax, out); note_launch();
  return cudaGetLastError();
}

}  // namespace psb
