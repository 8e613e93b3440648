// Weight sampler: turns an fp32 filter into exact integer filters, one per
// requested draw count k (paper Eq. 4-8).  Per weight:
//   decode (s, e, p) from the IEEE-754 fields          Eq. 5-7
//   window the exponent against the group's maximum    (4-bit exponents, Sec. 4.4)
//   draw k Bernoulli(p) bits from Philox4x32-10         the comparator of the
//                                                       stochastic multiplier
//   count the upper draws among the first k, every k    Eq. 8 (binomial count)
//   emit W_k = s (k + c_k) 2^(e - e_base) as signed 7-bit digit planes in the
//   layout the contraction kernels read (dense filters), or as int32 (others).
// The random bits never leave registers.
#include <new>

#include "psb_common.cuh"

#include <cuda_fp16.h>

#include <algorithm>

namespace psb {

namespace {

constexpr int kThreads = 256;
constexpr int kBatchThreads = 128;          // of a block of the batched sampling pass
constexpr uint32_t kStage = 4608;           // weights per block of a launch that fills the machine
constexpr int kEmaxRows = kThreads / 32;   // output channels per block of the exponent pass (norm == 1, short rows)
constexpr int kEmaxLongRow = 1024;         // rows longer than this get a block each
constexpr int kRowSumRows = 256;   // filter rows per block for which the sampler keeps sums of |W_k|
constexpr int kPlaneRows = 64;     // the same for filters with digit planes, which need the signed sums too

// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies and xors; the key advances by the
// two Weyl constants after every round.  What the counters of this library allow to be known beforehand is
// computed once per launch on the host and read from the constant bank:
//   - the ten round keys;
//   - of call q of a weight, counter (q, layer, index, 0) (a filter has at most 2^31 weights, so the high index word
//     is 0): the products of the first two rounds that see only q.  With M0, M1 the multipliers, Q = M0 q,
//     U = M1 (hi(Q) ^ k1[0]):  x = hi(U) ^ k0[1],  y = lo(Q) ^ k1[1],  z = lo(U) ^ k0[2].
// The two products of those rounds that see only the index serve every call of the weight (PhiloxWeight), so a
// call costs 16 multiplies instead of 20.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr int kPhiloxCalls = 16;      // calls of a weight at k = 64

struct PhiloxKeys {
  uint32_t k0[10], k1[10];
  uint32_t x[kPhiloxCalls], y[kPhiloxCalls], z[kPhiloxCalls];
  __host__ __device__ __forceinline__ PhiloxKeys(uint32_t seed_lo, uint32_t seed_hi) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
      k0[r] = seed_lo + (uint32_t)r * 0x9E3779B9u;
      k1[r] = seed_hi + (uint32_t)r * 0xBB67AE85u;
    }
#pragma unroll
    for (int q = 0; q < kPhiloxCalls; ++q) {
      const unsigned long long Q = (unsigned long long)kPhiloxM0 * (uint32_t)q;
      const unsigned long long U = (unsigned long long)kPhiloxM1 * ((uint32_t)(Q >> 32) ^ k1[0]);
      x[q] = (uint32_t)(U >> 32) ^ k0[1];
      y[q] = (uint32_t)Q ^ k1[1];
      z[q] = (uint32_t)U ^ k0[2];
    }
  }
};

// What the calls of one weight share.  layer_key = layer_id ^ k0[0].
struct PhiloxWeight {
  uint32_t a_lo, b_lo, b_hi;
  PhiloxWeight() = default;
  __device__ __forceinline__ PhiloxWeight(uint32_t index, uint32_t layer_key) {
    const unsigned long long A = (unsigned long long)kPhiloxM1 * index;
    const unsigned long long B = (unsigned long long)kPhiloxM0 * ((uint32_t)(A >> 32) ^ layer_key);
    a_lo = (uint32_t)A;
    b_lo = (uint32_t)B;
    b_hi = (uint32_t)(B >> 32);
  }
  __device__ __forceinline__ void call(uint32_t q, const PhiloxKeys& key, uint32_t (&out)[4]) const {
    uint32_t c0 = a_lo ^ key.x[q], c2 = b_hi ^ key.y[q], c3 = b_lo, c1 = 0u;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
      // one widening multiply gives both halves
      const unsigned long long p0 = (unsigned long long)kPhiloxM0 * c0, p1 = (unsigned long long)kPhiloxM1 * c2;
      c0 = (uint32_t)(p1 >> 32) ^ (r == 2 ? key.z[q] : c1 ^ key.k0[r]);
      c2 = (uint32_t)(p0 >> 32) ^ c3 ^ key.k1[r];
      c1 = (uint32_t)p1;
      c3 = (uint32_t)p0;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
  }
};

// Counts with a B-bit comparator (Sec. 4.4; supplement, "Stochastic multiplier"): draw j is bit field
// (j mod n) of word ((j / n) mod 4) of Philox call j / (4 n), n = 32 / B; cnt[l] = ones among the first 2^l
// draws.  Every index is a compile-time constant here, so the loops unroll into one extract / compare / add
// per draw.
template <int B>
__device__ __forceinline__ void packed_counts(uint32_t thr, uint32_t max_level, const PhiloxWeight& pw,
                                              const PhiloxKeys& keys, uint32_t (&cnt)[kMaxLevels]) {
  constexpr int n = 32 / B, per_call = 4 * n, calls = (64 + per_call - 1) / per_call;
  const uint32_t kmax = 1u << max_level;
  uint32_t c = 0;
#pragma unroll
  for (int q = 0; q < calls; ++q) {
    if ((uint32_t)(q * per_call) < kmax) {
      uint32_t rnd[4];
      pw.call((uint32_t)q, keys, rnd);
#pragma unroll
      for (int wd = 0; wd < 4; ++wd) {
#pragma unroll
        for (int f = 0; f < n; ++f) {
          constexpr uint32_t fmask = (1u << B) - 1u;
          const int j = q * per_call + wd * n + f;
          if (j < 64) {
            c += ((rnd[wd] >> (f * B)) & fmask) < thr ? 1u : 0u;
            if (((j + 1) & j) == 0) {           // j + 1 is a power of two: a level is complete
              const int l = j + 1 == 1 ? 0 : j + 1 == 2 ? 1 : j + 1 == 4 ? 2 : j + 1 == 8 ? 3 : j + 1 == 16 ? 4 : j + 1 == 32 ? 5 : 6;
              cnt[l] = c;
            }
          }
        }
      }
    }
  }
}

// The same for any width 1..8, indices at run time.
__device__ __forceinline__ void packed_counts_any(uint32_t pbits, uint32_t thr, uint32_t max_level, const PhiloxWeight& pw,
                                                  const PhiloxKeys& keys, uint32_t (&cnt)[kMaxLevels]) {
  const uint32_t n = 32u / pbits, per_call = 4u * n, fmask = (1u << pbits) - 1u, kmax = 1u << max_level;
  unsigned long long drawn = 0ull;      // bit j = draw j
  for (uint32_t q = 0; q * per_call < kmax && q * per_call < 64u; ++q) {
    uint32_t rnd[4];
    pw.call(q, keys, rnd);
#pragma unroll
    for (int wd = 0; wd < 4; ++wd) {
      uint32_t word = rnd[wd];
      unsigned long long bits = 0ull;
      for (uint32_t f = 0; f < n; ++f, word >>= pbits) bits |= (unsigned long long)((word & fmask) < thr ? 1u : 0u) << f;
      const uint32_t j0 = q * per_call + (uint32_t)wd * n;
      if (j0 < 64u) drawn |= bits << j0;
    }
  }
#pragma unroll
  for (int l = 0; l < kMaxLevels; ++l)
    cnt[l] = (uint32_t)__popcll(l == 6 ? drawn : drawn & ((1ull << (1u << l)) - 1ull));
}

// Division of a small number (< 2^16) by a block-uniform divisor (< 2^16): q = umulhi(t, magic)
// with magic = floor((2^32 - 1) / d) + 1 is exact in that range.
__device__ __forceinline__ uint32_t small_div_magic(uint32_t d) { return 0xFFFFFFFFu / d + 1u; }
__device__ __forceinline__ uint32_t small_div(uint32_t t, uint32_t magic) { return magic ? __umulhi(t, magic) : t; }   // magic wraps to 0 for d = 1

// Largest biased exponent of the finite weights of each exponent group; flags Inf/NaN (which
// contribute nothing: the finite weights of the group keep the window they would have without it).
// norm == 1: one warp (short rows) or one block per output channel.  norm == 0: grid-stride over the layer.
// Bound by memory once an element costs an AND and a max: the pass takes the largest magnitude (as an integer) and
// turns it into an exponent at the end.  After rounding the probability to `pbits` bits (Sec. 4.4) a probability of 1
// carries into the exponent; that is monotonic in the magnitude, so rounding the largest one is enough.
__device__ __forceinline__ uint32_t quantised_exponent(uint32_t mag, uint32_t pbits) {
  const uint32_t E = mag >> 23;
  if (pbits == 0u || E == 0u || E >= 254u) return E;
  return (mag + (1u << (22u - pbits))) >> 23;
}

constexpr uint32_t kInfBits = 0x7F800000u;

// Largest magnitude of n words, Inf and NaN flagged and left out.
template <int kN>
__device__ __forceinline__ uint32_t max_magnitude(const uint32_t (&u)[kN], uint32_t best, bool& bad) {
  uint32_t m = 0u;
#pragma unroll
  for (int j = 0; j < kN; ++j) m = max(m, u[j] & 0x7FFFFFFFu);
  if (m >= kInfBits) {
    bad = true;
    m = 0u;
#pragma unroll
    for (int j = 0; j < kN; ++j) m = max(m, (u[j] & 0x7FFFFFFFu) >= kInfBits ? 0u : u[j] & 0x7FFFFFFFu);
  }
  return max(best, m);
}

__device__ __forceinline__ void emax_block(const float* w, uint32_t O, uint32_t d,
                                           uint32_t norm, uint32_t* __restrict__ e_max,
                                           uint32_t* __restrict__ err, uint32_t block, uint32_t blocks,
                                           uint32_t tag, uint32_t* __restrict__ rowsum,
                                           long long* __restrict__ corr, uint32_t pbits) {
  __shared__ uint32_t red[kThreads / 32];
  // the sampling pass that follows adds its row sums into these words: start them at zero
  if (rowsum)
    for (uint32_t i = block * blockDim.x + threadIdx.x; i < (uint32_t)kMaxLevels * O; i += blocks * blockDim.x) {
      rowsum[i] = 0u;
      if (corr) corr[i] = 0;
    }
  uint32_t best = 0;
  bool bad = false;
  if (norm) {
    // short rows: one warp per output channel, kEmaxRows channels per block; long rows: one block per
    // channel.  16-byte loads where the row allows, several in flight per lane.
    const bool per_warp = d <= (uint32_t)kEmaxLongRow;
    const uint32_t o = per_warp ? block * (uint32_t)kEmaxRows + (threadIdx.x >> 5) : block;
    const uint32_t lane = per_warp ? (threadIdx.x & 31u) : threadIdx.x, lanes = per_warp ? 32u : blockDim.x;
    if (o < O) {
      const float* row = w + (size_t)o * d;
      if ((((uintptr_t)row) & 15u) == 0u && (d & 3u) == 0u) {
#pragma unroll 4
        for (uint32_t i = lane * 4u; i < d; i += lanes * 4u) {
          const uint4 v = __ldcg(reinterpret_cast<const uint4*>(row + i));
          const uint32_t u4[4] = {v.x, v.y, v.z, v.w};
          best = max_magnitude(u4, best, bad);     // Inf/NaN is flagged and takes no part in the window
        }
      } else {
#pragma unroll 4
        for (uint32_t i = lane; i < d; i += lanes) {
          const uint32_t u1[1] = {__float_as_uint(__ldcg(row + i))};
          best = max_magnitude(u1, best, bad);
        }
      }
    }
    if (per_warp) {
      if (o >= O) return;                                   // warp-uniform; no block-wide barrier on this path
      if (__any_sync(0xFFFFFFFFu, bad) && lane == 0u) atomicOr(err, kDevErrNonFinite);
      best = __reduce_max_sync(0xFFFFFFFFu, best);
      // `tag` (a call number in the bits above the exponent) distinguishes this call's maxima from whatever
      // an earlier call left in the word
      if (lane == 0u) e_max[o] = tag | quantised_exponent(best, pbits);
      return;
    }
  } else {
    const size_t total = (size_t)O * d;
    if ((((uintptr_t)w) & 15u) == 0u && (total & 3u) == 0u) {
      // four 16-byte loads in flight per thread
      const size_t step = (size_t)blocks * blockDim.x * 4u;
      for (size_t i = ((size_t)block * blockDim.x + threadIdx.x) * 4u; i < total; i += 4u * step) {
        uint4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          v[q] = i + q * step < total ? __ldcg(reinterpret_cast<const uint4*>(w + i + q * step)) : make_uint4(0u, 0u, 0u, 0u);
        uint32_t u16[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          u16[4 * q] = v[q].x; u16[4 * q + 1] = v[q].y; u16[4 * q + 2] = v[q].z; u16[4 * q + 3] = v[q].w;
        }
        best = max_magnitude(u16, best, bad);
      }
    } else {
      for (size_t i = (size_t)block * blockDim.x + threadIdx.x; i < total; i += (size_t)blocks * blockDim.x) {
        const uint32_t u1[1] = {__float_as_uint(__ldcg(w + i))};
        best = max_magnitude(u1, best, bad);
      }
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && (threadIdx.x & 31) == 0) atomicOr(err, kDevErrNonFinite);
  best = __reduce_max_sync(0xFFFFFFFFu, best);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kThreads / 32; ++i) best = max(best, red[i]);
    best = quantised_exponent(best, pbits);
    // `tag` (a call number in the bits above the exponent) makes the maxima of this call beat
    // whatever an earlier call left in the word, so the words need no clearing between calls
    if (norm) e_max[block] = tag | best;
    else if (best) atomicMax(&e_max[0], tag | best);
  }
}

__global__ void emax_kernel(const float* w, uint32_t O, uint32_t d, uint32_t norm,
                            uint32_t* __restrict__ e_max, uint32_t* __restrict__ err, uint32_t tag,
                            uint32_t* __restrict__ rowsum, long long* __restrict__ corr, uint32_t pbits) {
  pdl_prologue();
  emax_block(w, O, d, norm, e_max, err, blockIdx.x, gridDim.x, tag, rowsum, corr, pbits);
}

// What one weight becomes at every level: W_k = s (base k + c_k) 2^sh with c_k = cnt[log2 k]; a weight that is
// not live becomes 0.  `u` is the weight's bit pattern, `index` its canonical index (the Philox counter),
// `ebase_biased` the biased exponent of the window's floor.
struct Drawn {
  uint32_t cnt[kMaxLevels];
  uint32_t base, sh, thr;
  bool live;
};

// The part without draws: base, sh, and the threshold that a draw is compared with.
__device__ __forceinline__ void classify_weight(uint32_t u, int ebase_biased, uint32_t pbits, uint32_t underflow, Drawn& out) {
  const uint32_t E = (u >> 23) & 0xFFu;
  const uint32_t m = u & 0x7FFFFFu;
  // probability on the grid of 2^pbits points, a p of 1 carried into the exponent (Sec. 4.4)
  uint32_t Eq = E, pq = m;
  if (pbits) {
    pq = (m + (1u << (22u - pbits))) >> (23u - pbits);
    if (pq == (1u << pbits)) {
      if (E < 254u) { Eq = E + 1u; pq = 0u; } else pq = (1u << pbits) - 1u;
    }
  }
  // what the weight becomes: W_k = s (base k + c_k) 2^sh, c_k counting draws with Pr[1] = thr / 2^32 (or
  // thr / 2^pbits).  Inside the window base = 1 (Eq. 8); below it, if asked for, the Bernoulli gate at the
  // window's floor (Sec. 3.1): base = 0, sh = 0, thr = |w| / 2^e_base
  bool live = (E != 0u) && (E != 255u);
  uint32_t base = 1u, sh = 0u, thr = 0u;
  const int dist = ebase_biased - (int)Eq;
  if (dist <= 0) {
    sh = (uint32_t)(-dist);
    thr = pbits ? pq : pq << 9;
  } else if (underflow) {
    base = 0u;
    if (pbits == 0u) {
      thr = dist <= 32 ? ((0x800000u + pq) << 8) >> (dist - 1) : 0u;
      live = live && thr != 0u;
    } else {
      const uint32_t mant = (1u << pbits) + pq;      // below 2^9
      const uint32_t qv = dist < 10 ? (mant + (1u << (dist - 1))) >> dist : 0u;
      if (qv == (1u << pbits)) base = 1u;          // rounds to the window's floor itself
      else { thr = qv; live = live && qv != 0u; }
    }
  } else {
    live = false;
  }

  out.base = base;
  out.sh = sh;
  out.thr = thr;
  out.live = live;
}

__device__ __forceinline__ void draw_weight(uint32_t u, uint32_t index, int ebase_biased, uint32_t pbits,
                                            uint32_t underflow, uint32_t deterministic, uint32_t max_level,
                                            uint32_t layer_key, const PhiloxKeys& keys, Drawn& out) {
  classify_weight(u, ebase_biased, pbits, underflow, out);
  const uint32_t thr = out.thr;
  uint32_t (&cnt)[kMaxLevels] = out.cnt;
#pragma unroll
  for (int l = 0; l < kMaxLevels; ++l) cnt[l] = 0u;
  // c_k for every level k = 2^l: level l is complete after draw 2^l, i.e. levels 0..2 after the
  // first Philox call, level l >= 2 after call 2^(l-2)
  if (out.live && thr != 0u) {
    const PhiloxWeight pw(index, layer_key);
    uint32_t rnd[4];
    if (pbits == 0u) {
      const uint32_t T = thr;
      pw.call(0u, keys, rnd);
      cnt[0] = rnd[0] < T ? 1u : 0u;
      cnt[1] = cnt[0] + (rnd[1] < T ? 1u : 0u);
      uint32_t c = cnt[1] + (rnd[2] < T ? 1u : 0u) + (rnd[3] < T ? 1u : 0u);
      cnt[2] = c;
#pragma unroll
      for (int l = 3; l < kMaxLevels; ++l) {
        if ((uint32_t)l <= max_level) {
#pragma unroll 1
          for (uint32_t q = 1u << (l - 3); q < (1u << (l - 2)); ++q) {
            pw.call(q, keys, rnd);
            c += (rnd[0] < T ? 1u : 0u) + (rnd[1] < T ? 1u : 0u) + (rnd[2] < T ? 1u : 0u) + (rnd[3] < T ? 1u : 0u);
          }
          cnt[l] = c;
        }
      }
    } else if (deterministic) {
#pragma unroll
      for (int l = 0; l < kMaxLevels; ++l) cnt[l] = ((thr << l) + (1u << (pbits - 1u))) >> pbits;
    } else {
      // pbits-bit comparator, n = 32 / pbits draws per random word
      switch (pbits) {
        case 4: packed_counts<4>(thr, max_level, pw, keys, cnt); break;
        case 6: packed_counts<6>(thr, max_level, pw, keys, cnt); break;
        case 8: packed_counts<8>(thr, max_level, pw, keys, cnt); break;
        default: packed_counts_any(pbits, thr, max_level, pw, keys, cnt); break;
      }
    }
  }

}

struct SampleParams {
  const float* w;
  uint32_t O, Cg, KHKW, d;
  uint32_t rows_per_block, ch_per_block, ch_chunks;
  uint32_t norm, span, level_mask, max_level;
  uint32_t underflow, pbits, deterministic;   // options of psb_sample_cfg
  uint32_t layer_id, has_planes;
  uint32_t bk, n_cb, n_kb;         // operand tiles of the tensor path: K block bytes, blocks per tap, blocks per row
  uint32_t packed_kw, run_pitch;   // packed K (packed_kw = kw, else 0): plane column = kh * run_pitch + kw * Cg + ci
  const uint32_t* e_max;
  uint32_t e_tag;                  // call number the words of e_max must carry (bits 8 and up)
  int32_t* e_base;
  uint32_t* rowsum;                // [kMaxLevels][O] row sums of |W_k| / 256 (see psb_weights)
  long long* corr;                 // [kMaxLevels][O] 128 x row sums of W_k, filters with digit planes only
  int32_t* wint[kMaxLevels];       // filters without digit planes
  int8_t* planes[kMaxLevels];
  int planes_count[kMaxLevels];
};

// Draws of a B-bit comparator (B = 4 or 8; fields as in packed_counts), one word at a time: every second field with a guard bit
// above it, (field | guard) - thr keeps the guard iff field >= thr.  Field 2m answers in bit B + 2 B m, field 2m + 1 in the bit
// below that one.
template <int B>
struct PackedDraws {
  static constexpr uint32_t kFirstLevel = B == 8 ? 2 : 3;       // a word completes this level
  static constexpr uint32_t kMask = B == 8 ? 0x00FF00FFu : 0x0F0F0F0Fu, kGuard = B == 8 ? 0x01000100u : 0x10101010u;
  static __device__ __forceinline__ uint32_t below(uint32_t word, uint32_t thr) {
    const uint32_t t = (kGuard >> B) * thr;
    const uint32_t e = ((word & kMask) | kGuard) - t, o = (((word >> B) & kMask) | kGuard) - t;
    return (~e & kGuard) | ((~o & kGuard) >> 1);
  }
  // the bits of the first 2^l fields, l < kFirstLevel
  static __device__ __forceinline__ uint32_t first(uint32_t l) {
    constexpr uint32_t b = 1u << B, two = b | (b >> 1);
    return l == 0u ? b : l == 1u ? two : two | (two << (2 * B));
  }
};

// The same for any width b of 1..8, known at run time: n = 32 / b fields in a word, of which the last even one may end short of
// the top (b = 6); field 2m answers in bit b + 2 b m, field 2m + 1 in the bit below that one.
struct PackedDrawsAny {
  uint32_t b, n, even, guard_even, guard_odd, ones;       // ones: bit 0 of every even field
  __device__ __forceinline__ explicit PackedDrawsAny(uint32_t width) : b(width), n(32u / width) {
    ones = 0u;
    for (uint32_t f = 0; f < n; f += 2u) ones |= 1u << (f * b);
    even = ones * ((1u << b) - 1u);
    guard_even = ones << b;
    guard_odd = n & 1u ? guard_even & ((1u << ((n - 1u) * b)) - 1u) : guard_even;
  }
  __device__ __forceinline__ uint32_t below(uint32_t word, uint32_t thr) const {
    const uint32_t t = ones * thr;
    const uint32_t e = ((word & even) | guard_even) - t, o = (((word >> b) & even) | guard_even) - t;
    return (~e & guard_even) | ((~o & guard_odd) >> 1);
  }
  // the bits of the first `left` fields, left < n
  __device__ __forceinline__ uint32_t first(uint32_t left) const {
    const uint32_t e = (1u << (b * ((left + 1u) & ~1u))) - 1u, o = (1u << (b * (left & ~1u))) - 1u;
    return (guard_even & e) | ((guard_odd & o) >> 1);
  }
};

// Row sums of a block's slice, kept in shared memory and added to the layer's words at the end: the sum of |W_k| in
// units of 256 (each contribution rounded up) bounds the accumulators; the signed sum, as hi * 4096 + lo, is what an
// offset of the activations has to be corrected by.
struct RowSums {
  uint32_t word[kMaxLevels * kRowSumRows];      // [level][kRowSumRows], or [level][3][kPlaneRows] with digit planes
};

// One warp's contributions (abs256, signed) to its rows: one reduction and one add per row that the lanes share.
__device__ __forceinline__ void add_row_sums(uint32_t* sums, uint32_t r, uint32_t abs256, int sum, bool with_signed) {
  uint32_t lanes = __activemask();
  const uint32_t r_first = __shfl_sync(lanes, r, __ffs((int)lanes) - 1);
  if (!__all_sync(lanes, r == r_first)) lanes = __match_any_sync(lanes, r);
  abs256 = __reduce_add_sync(lanes, abs256);
  if (with_signed) sum = __reduce_add_sync(lanes, sum);
  if ((threadIdx.x & 31u) == (uint32_t)__ffs((int)lanes) - 1u && abs256) {
    atomicAdd(&sums[r], abs256);
    if (with_signed) {
      atomicAdd(&sums[kPlaneRows + r], (uint32_t)(sum & 0xFFF));
      atomicAdd(&sums[2 * kPlaneRows + r], (uint32_t)(sum >> 12));
    }
  }
}

// Biased exponent of a window from its word.  A word written by an earlier call (other tag) means this call found no
// live weight in the group.
__device__ __forceinline__ uint32_t window_exponent(uint32_t word, uint32_t tag) { return (word >> 8) == tag ? (word & 0xFFu) : 0u; }

// How the draws of a weight are counted.
enum DrawMode {
  kDrawExact,      // no option: probability m / 2^23
  kDrawGate,       // exact probabilities, Bernoulli gate below the window (32-bit thresholds)
  kDrawPacked8,    // 8-bit comparator
  kDrawPacked4,    // 4-bit comparator
  kDrawAny         // any other width, and the deterministic variant
};

// One draw: adds 1 to the count, kept in fp32, where the word is below the threshold.  The predicated addition runs on the fp32
// pipe, which has nothing else to do; an integer one would take a second slot of the logic pipe.
__device__ __forceinline__ void draw(float& count, uint32_t word, uint32_t thr, float one = 1.0f) {
  asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p add.rn.f32 %0, %0, %3;\n\t}" : "+f"(count) : "r"(word), "r"(thr), "f"(one));
}

// Bounds of a window as the decoding of a weight wants them: what 2u (magnitude bits shifted left by one) has to lie in,
// and what takes the weight's exponent field to that of 2^(e - e_base).
struct WindowBits {
  uint32_t floor2, range2, rebias;
  int ebase;      // biased exponent of the floor
  __device__ __forceinline__ WindowBits(uint32_t Emax, int span) {
    ebase = (int)Emax - span;
    const uint32_t lowest = ebase > 1 ? (uint32_t)ebase : 1u;
    floor2 = lowest << 24;
    range2 = Emax ? (Emax + 1u - lowest) << 24 : 0u;       // nothing is below 0: no live weight
    rebias = (uint32_t)(ebase - 127) << 23;
  }
  __device__ __forceinline__ bool holds(uint32_t u) const { return (u + u) - floor2 < range2; }      // not Inf, not NaN, not 0
  __device__ __forceinline__ float scale(uint32_t u) const { return __uint_as_float((u & 0xFF800000u) - rebias); }
};

// What the counters of a weight's draws need: W_k = scale (base k + c_k), c_k counting draws below thr (32 bits, or the
// comparator's width).  Inside the window base = 1 and scale = +-2^(e - e_base) (Eq. 8); below it, if asked for, the
// Bernoulli gate at the window's floor (Sec. 3.1): base = 0, scale = +-1, thr = |w| / 2^e_base; else scale = 0.  The same
// definitions as classify_weight.
template <int kMode>
__device__ __forceinline__ void decode_weight(uint32_t u, const WindowBits& win, uint32_t underflow, uint32_t pbits, uint32_t& thr, float& base, float& scale) {
  base = 1.0f;
  if (kMode == kDrawExact || kMode == kDrawGate) {
    thr = u << 9;
    scale = win.scale(u);
    if (!win.holds(u)) {
      scale = 0.0f;
      if (kMode == kDrawGate) {
        const uint32_t mag = u & 0x7FFFFFFFu;
        const int dist = win.ebase - (int)(mag >> 23);
        base = 0.0f;
        thr = 0u;
        if (mag >= 0x800000u && dist > 0) {
          scale = __uint_as_float((u & 0x80000000u) | 0x3F800000u);
          thr = dist <= 32 ? ((0x800000u | (u & 0x7FFFFFu)) << 8) >> (dist - 1) : 0u;
        }
      }
    }
    return;
  }
  // probability on the grid of 2^B points: a p of 1 carries into the exponent, but not beyond the largest finite one
  const int B = kMode == kDrawPacked8 ? 8 : kMode == kDrawPacked4 ? 4 : (int)pbits;
  const uint32_t mag = u & 0x7FFFFFFFu;
  uint32_t q = min(mag + (1u << (22 - B)), 0x7F7FFFFFu);
  if (mag - 0x800000u >= 0x7F000000u) q = 0u;       // zero, sub-normal, Inf, NaN
  thr = (q >> (23 - B)) & ((1u << B) - 1u);
  scale = win.scale(q | (u & 0x80000000u));
  if (!win.holds(q)) {
    const int dist = win.ebase - (int)(q >> 23);
    const uint32_t mant = (1u << B) + thr;
    base = 0.0f;
    thr = 0u;
    scale = 0.0f;
    if (underflow && q && dist > 0 && dist <= B + 1) {
      const uint32_t at_floor = (mant + (1u << (dist - 1))) >> dist;
      if (at_floor == (1u << B)) base = 1.0f;          // rounds to the window's floor itself
      else thr = at_floor;
      scale = __uint_as_float((u & 0x80000000u) | 0x3F800000u);
    }
  }
}

// Draws of an 8-bit comparator, two at a time in half precision: 1024 + byte and 1024 + threshold are exact, their difference
// saturated to [0, 1] is the draw.  One permute and two half2 operations for two draws.
__device__ __forceinline__ void draw_pair8(uint32_t& count2, uint32_t thr2, uint32_t word, uint32_t select) {
  uint32_t d;
  asm("sub.sat.f16x2 %0, %1, %2;" : "=r"(d) : "r"(thr2), "r"(__byte_perm(word, 0x64646464u, select)));
  asm("add.rn.f16x2 %0, %0, %1;" : "+r"(count2) : "r"(d));
}
__device__ __forceinline__ void draw_word8(uint32_t& count2, uint32_t thr01, uint32_t thr23, uint32_t word) {
  draw_pair8(count2, thr01, word, 0x4140);
  draw_pair8(count2, thr23, word, 0x4342);
}

// Four weights' signed integers (as floats, |fs| <= 2^22) to their digit planes.  The lower digits are bits 0..6, 7..13, .. of
// the two's complement, the top one is what is left, with its sign: W = sum_p D_p 2^(7p) needs no digit negated.  1.5 * 2^23
// + W shows W in the low bits of the sum; moved up by one and two bits the second and third digit lie in the second and third
// byte, from where byte permutes put the same digit of the four weights into one word.  abs256: the sum of the four |W| in
// units of 256, rounded up.
__device__ __forceinline__ void store_digits(int P, int8_t* dst, uint32_t plane_shift, const float (&fs)[4], uint32_t& abs256, int& sum) {
  auto put = [&](int pl, uint32_t word) {
    *reinterpret_cast<uint32_t*>(dst + ((size_t)pl << plane_shift)) = pl + 1 == P ? word : word & 0x7F7F7F7Fu;
  };
  uint32_t a[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) a[j] = __float_as_uint(__fadd_rn(fs[j], 12582912.0f));
  const uint32_t w0 = __byte_perm(__byte_perm(a[0], a[1], 0x0040), __byte_perm(a[2], a[3], 0x0040), 0x5410);
  uint32_t b[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j] = a[j] << 1;
  const uint32_t w1 = __byte_perm(__byte_perm(b[0], b[1], 0x0051), __byte_perm(b[2], b[3], 0x0051), 0x5410);
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j] = a[j] << 2;
  const uint32_t w2 = __byte_perm(__byte_perm(b[0], b[1], 0x0062), __byte_perm(b[2], b[3], 0x0062), 0x5410);
  if (P == 3) {
    put(0, w0);
    put(1, w1);
    put(2, w2);
  } else {
    put(0, w0);
    if (P > 1) put(1, w1);
    if (P > 3) {
      put(2, w2);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = (a[j] - 0x4B400000u) << 3;
      put(3, __byte_perm(__byte_perm(b[0], b[1], 0x0073), __byte_perm(b[2], b[3], 0x0073), 0x5410));
    }
  }
  sum = __float2int_rn(__fadd_rn(__fadd_rn(fs[0], fs[1]), __fadd_rn(fs[2], fs[3])));
  const float all = __fadd_rn(__fadd_rn(fabsf(fs[0]), fabsf(fs[1])), __fadd_rn(fabsf(fs[2]), fabsf(fs[3])));
  abs256 = __float2uint_ru(__fmul_rn(all, 1.0f / 256.0f));
}

// Filters with digit planes whose K axis is tap-major: a thread takes four consecutive channels of one (row, tap), draws
// them side by side and stores 4 bytes per digit plane (store_digits).
// Bound by issue.  Measured clocks per warp instruction and scheduler: a widening multiply takes 4 of its pipe, which Philox at
// k = 8 fills 136 of, and 2 of the dispatch that it shares with the logic pipe; a xor, permute or compare takes 2 of that, an
// fp32 or half2 operation 1.  Philox alone is 142 clocks a weight at k = 8; all that can runs in floating point.
// Before (integer magnitudes and counts, sign-and-magnitude digits, 256-thread blocks of up to 4096 weights) / now, us:
// 25.5 M weights of the ResNet-50 shape with their exponent pass (33), k = 8: 291 / 213, five levels 613 / 505, k = 8 and 16
// 503 / 406; 4096 x 4096: k = 16 242 / 191, 8-bit comparator with gate, k = 16 194 / 114; 3x3 512 -> 512 36 / 23.
template <int kMode, bool kMulti, int kCalls>
__device__ __forceinline__ void sample_planes(const SampleParams& p, const uint32_t* windows, uint32_t tag, uint32_t o0, uint32_t c0, uint32_t rows, uint32_t cc,
                                              const PhiloxKeys& keys, const float* stage, uint32_t* sums) {
  const uint32_t KHKW = p.KHKW, norm = p.norm, level_mask = p.level_mask;
  const uint32_t max_level = p.max_level, layer_key = p.layer_id ^ keys.k0[0];
  const uint32_t bk = p.bk, n_cb = p.n_cb, n_kb = p.n_kb;
  const uint32_t bk_shift = 31u - (uint32_t)__clz((int)bk), bk_mask = bk - 1u, sw_mask = (bk >> 4) - 1u;
  const uint32_t per_row = cc * KHKW, groups = (cc + 3u) >> 2, per_row4 = groups * KHKW, count4 = rows * per_row4;
  const uint32_t per_row4_magic = small_div_magic(per_row4), groups_magic = small_div_magic(groups);
  const bool whole = (cc & 3u) == 0u, vec4 = whole && KHKW == 1u;
  const uint32_t index0 = o0 * p.d + c0 * KHKW;      // the slice is one run of the tensor: stage[i] has index index0 + i
  const float k_max = (float)(1u << max_level);
  // of the first call, the words (8-bit comparator: of its first word, the bytes) that count
  const uint32_t low01 = max_level >= 1u ? 0xFFFFFFFFu : 0xFFFFu, low23 = max_level >= 2u ? 0xFFFFFFFFu : 0u;
  const float second = max_level >= 1u ? 1.0f : 0.0f, rest = max_level >= 2u ? 1.0f : 0.0f;
  WindowBits win(norm ? 0u : window_exponent(windows[0], tag), (int)p.span);
  const PackedDrawsAny any(kMode == kDrawAny && !p.deterministic ? p.pbits : 8u);
  // sums of the row a thread is in (one level)
  uint32_t run_row = 0u, run_abs = 0u;
  int run_sum = 0;
  for (uint32_t t = threadIdx.x; t < count4; t += blockDim.x) {
    const uint32_t r = small_div(t, per_row4_magic), rem = t - r * per_row4;
    const uint32_t tap = small_div(rem, groups_magic), cl = (rem - tap * groups) << 2;
    const uint32_t o = o0 + r, ci = c0 + cl;
    if (norm) win = WindowBits(window_exponent(windows[r], tag), (int)p.span);
    const uint32_t at = r * per_row + cl * KHKW + tap;
    uint32_t u[4];
    if (vec4) {
      const float4 v = *reinterpret_cast<const float4*>(stage + at);
      u[0] = __float_as_uint(v.x); u[1] = __float_as_uint(v.y); u[2] = __float_as_uint(v.z); u[3] = __float_as_uint(v.w);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = whole || cl + (uint32_t)j < cc ? __float_as_uint(stage[at + (uint32_t)j * KHKW]) : 0u;
    }
    const uint32_t kb = tap * n_cb + (ci >> bk_shift), kin = ci & bk_mask, jt = o / kTileN, on = o % kTileN;
    // byte offset of (row, kin) in the swizzled tile (plane_offset); planes are 64 rows apart, which leaves the
    // swizzle as it is
    const uint32_t lin = (on << bk_shift) + kin, off = lin ^ (((lin >> 7) & sw_mask) << 4);
    const uint32_t tile = jt * n_kb + kb;
    auto plane_ptr = [&](uint32_t lv, int P) { return p.planes[lv] + (((size_t)tile * (uint32_t)P) << (6u + bk_shift)) + off; };
    float fs[4];
    uint32_t abs256;
    int sum;
    float scale[4], base[4], cnt[4];
    uint32_t thr[4];
    PhiloxWeight pw[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      decode_weight<kMode>(u[j], win, p.underflow, p.pbits, thr[j], base[j], scale[j]);
      if (kMode != kDrawAny) pw[j] = PhiloxWeight(index0 + at + (uint32_t)j * KHKW, layer_key);
    }
    auto four_more = [&](uint32_t q) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(q, keys, rnd);
#pragma unroll
        for (int i = 0; i < 4; ++i) draw(cnt[j], rnd[i], thr[j]);
      }
    };
    if (kMode == kDrawAny) {
      // Word by word, the fields of a word all at once; a level may end inside a word.  us, field by field and weight by weight / so:
      // 25.5 M weights of the ResNet-50 shape with their exponent pass, 1 bit 1620 / 244, 3 bits, five levels 969 / 418, 6 bits,
      // k = 64 649 / 576, deterministic, five levels 397 / 293; MobileNet-v2 shape, 7 bits, k = 64 231 / 104; 3x3 64->64, 1 bit 18.6 / 7.5.
      uint32_t c[4] = {0u, 0u, 0u, 0u}, l = 0u;
      auto complete = [&](const uint32_t (&count)[4]) {
        const float k = (float)(1u << l);
#pragma unroll
        for (int j = 0; j < 4; ++j) fs[j] = __fmul_rn(__fmaf_rn(base[j], k, (float)(int)count[j]), scale[j]);
        if (kMulti) {
          const int P = p.planes_count[l];
          store_digits(P, plane_ptr(l, P), 6u + bk_shift, fs, abs256, sum);
          add_row_sums(sums + l * (3u * kPlaneRows), r, abs256, sum, true);
        }
      };
      if (p.deterministic) {
#pragma unroll 1
        for (l = kMulti ? 0u : max_level; l <= max_level; ++l) {
          if (!((level_mask >> l) & 1u)) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j) c[j] = ((thr[j] << l) + (1u << (p.pbits - 1u))) >> p.pbits;
          complete(c);
        }
      } else {
        const uint32_t n = any.n;
        uint32_t drawn = 0u, todo = level_mask;
        l = (uint32_t)__ffs((int)todo) - 1u;
#pragma unroll
        for (int j = 0; j < 4; ++j) pw[j] = PhiloxWeight(index0 + at + (uint32_t)j * KHKW, layer_key);
#pragma unroll 1
        for (uint32_t q = 0; todo; ++q) {
          uint32_t hits[4][4];        // per weight and word; the word at hand comes first
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t rnd[4];
            pw[j].call(q, keys, rnd);
#pragma unroll
            for (int i = 0; i < 4; ++i) hits[j][i] = any.below(rnd[i], thr[j]);
          }
          if ((1u << l) > drawn + 4u * n) {        // no level ends in this call
#pragma unroll
            for (int j = 0; j < 4; ++j) c[j] += (uint32_t)(__popc(hits[j][0]) + __popc(hits[j][1]) + __popc(hits[j][2]) + __popc(hits[j][3]));
            drawn += 4u * n;
            continue;
          }
#pragma unroll 1
          for (int w = 0; w < 4 && todo; ++w, drawn += n) {
            while (todo && (1u << l) <= drawn + n) {
              const uint32_t left = (1u << l) - drawn, fields = left < n ? any.first(left) : 0xFFFFFFFFu;
              uint32_t count[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) count[j] = c[j] + (uint32_t)__popc(hits[j][0] & fields);
              complete(count);
              todo &= todo - 1u;
              l = (uint32_t)__ffs((int)todo) - 1u;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              c[j] += (uint32_t)__popc(hits[j][0]);
              hits[j][0] = hits[j][1]; hits[j][1] = hits[j][2]; hits[j][2] = hits[j][3];
            }
          }
        }
      }
    } else if (kMulti && (kMode == kDrawPacked8 || kMode == kDrawPacked4)) {
      typedef PackedDraws<kMode == kDrawPacked8 ? 8 : 4> D;
      uint32_t hits[4][4], c[4];        // per weight and word
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(0u, keys, rnd);
#pragma unroll
        for (int i = 0; i < 4; ++i) hits[j][i] = D::below(rnd[i], thr[j]);
        c[j] = 0u;
      }
#pragma unroll 1
      for (uint32_t l = 0; l <= max_level; ++l) {
        if (l <= D::kFirstLevel) {
          const uint32_t fields = l < D::kFirstLevel ? D::first(l) : 0xFFFFFFFFu;
#pragma unroll
          for (int j = 0; j < 4; ++j) c[j] = (uint32_t)__popc(hits[j][0] & fields);
        } else if (l == D::kFirstLevel + 1u) {
#pragma unroll
          for (int j = 0; j < 4; ++j) c[j] += (uint32_t)__popc(hits[j][1]);
        } else if (l == D::kFirstLevel + 2u) {
#pragma unroll
          for (int j = 0; j < 4; ++j) c[j] += (uint32_t)(__popc(hits[j][2]) + __popc(hits[j][3]));
        } else {
#pragma unroll 1
          for (uint32_t q = 1u << (l - D::kFirstLevel - 3u); q < 1u << (l - D::kFirstLevel - 2u); ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint32_t rnd[4];
              pw[j].call(q, keys, rnd);
#pragma unroll
              for (int i = 0; i < 4; ++i) c[j] += (uint32_t)__popc(D::below(rnd[i], thr[j]));
            }
        }
        if (!((level_mask >> l) & 1u)) continue;
        const float k = (float)(1u << l);
#pragma unroll
        for (int j = 0; j < 4; ++j) fs[j] = __fmul_rn(__fmaf_rn(base[j], k, (float)(int)c[j]), scale[j]);
        const int P = p.planes_count[l];
        store_digits(P, plane_ptr(l, P), 6u + bk_shift, fs, abs256, sum);
        add_row_sums(sums + l * (3u * kPlaneRows), r, abs256, sum, true);
      }
    } else if (kMode == kDrawPacked8) {
      uint32_t count2[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(0u, keys, rnd);
        thr[j] = thr[j] * 0x10001u + 0x64006400u;
        count2[j] = 0u;
        // of fewer than four draws the others never fall below their threshold of 0
        draw_word8(count2[j], (thr[j] & low01) | 0x64006400u, (thr[j] & low23) | 0x64006400u, rnd[0]);
        if (max_level > 2u) draw_word8(count2[j], thr[j], thr[j], rnd[1]);
        if (max_level > 3u) {
          draw_word8(count2[j], thr[j], thr[j], rnd[2]);
          draw_word8(count2[j], thr[j], thr[j], rnd[3]);
        }
      }
#pragma unroll 1
      for (uint32_t q = 1; q < (1u << max_level) / 16u; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t rnd[4];
          pw[j].call(q, keys, rnd);
#pragma unroll
          for (int i = 0; i < 4; ++i) draw_word8(count2[j], thr[j], thr[j], rnd[i]);
        }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __half2 c = *reinterpret_cast<const __half2*>(&count2[j]);
        cnt[j] = __fmaf_rn(base[j], k_max, __low2float(c) + __high2float(c));
      }
    } else if (kMode == kDrawPacked4) {
      typedef PackedDraws<4> D;
      const uint32_t fields = max_level < D::kFirstLevel ? D::first(max_level) : 0xFFFFFFFFu;
      uint32_t c[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(0u, keys, rnd);
        c[j] = (uint32_t)__popc(D::below(rnd[0], thr[j]) & fields);
        if (max_level > D::kFirstLevel) c[j] += (uint32_t)__popc(D::below(rnd[1], thr[j]));
        if (max_level > D::kFirstLevel + 1u) c[j] += (uint32_t)(__popc(D::below(rnd[2], thr[j])) + __popc(D::below(rnd[3], thr[j])));
      }
#pragma unroll 1
      for (uint32_t q = 1; q < (1u << max_level) / 32u; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t rnd[4];
          pw[j].call(q, keys, rnd);
#pragma unroll
          for (int i = 0; i < 4; ++i) c[j] += (uint32_t)__popc(D::below(rnd[i], thr[j]));
        }
#pragma unroll
      for (int j = 0; j < 4; ++j) cnt[j] = __fmaf_rn(base[j], k_max, (float)(int)c[j]);
    } else if (!kMulti) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(0u, keys, rnd);
        cnt[j] = kMode == kDrawExact ? k_max : __fmul_rn(base[j], k_max);        // base k + c
        draw(cnt[j], rnd[0], thr[j]);
        draw(cnt[j], rnd[1], thr[j], second);
        draw(cnt[j], rnd[2], thr[j], rest);
        draw(cnt[j], rnd[3], thr[j], rest);
      }
      if (kCalls) {
#pragma unroll
        for (int q = 1; q < kCalls; ++q) four_more((uint32_t)q);
      } else {
#pragma unroll 1
        for (uint32_t q = 1; q < (1u << max_level) / 4u; ++q) four_more(q);
      }
    } else {
      float hit1[4], hit2[4];        // draw 1; draws 2 and 3
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t rnd[4];
        pw[j].call(0u, keys, rnd);
        cnt[j] = hit1[j] = hit2[j] = 0.0f;
        draw(cnt[j], rnd[0], thr[j]);
        draw(hit1[j], rnd[1], thr[j]);
        draw(hit2[j], rnd[2], thr[j]);
        draw(hit2[j], rnd[3], thr[j]);
      }
#pragma unroll 1
      for (uint32_t l = 0; l <= max_level; ++l) {
        if (l == 1u || l == 2u) {
#pragma unroll
          for (int j = 0; j < 4; ++j) cnt[j] = __fadd_rn(cnt[j], l == 1u ? hit1[j] : hit2[j]);
        } else if (l > 2u) {
#pragma unroll 1
          for (uint32_t q = 1u << (l - 3u); q < 1u << (l - 2u); ++q) four_more(q);
        }
        if (!((level_mask >> l) & 1u)) continue;
        const float k = (float)(1u << l);
#pragma unroll
        for (int j = 0; j < 4; ++j) fs[j] = __fmul_rn(__fmaf_rn(base[j], k, cnt[j]), scale[j]);
        const int P = p.planes_count[l];
        store_digits(P, plane_ptr(l, P), 6u + bk_shift, fs, abs256, sum);
        add_row_sums(sums + l * (3u * kPlaneRows), r, abs256, sum, true);
      }
    }
    if (!kMulti && kMode != kDrawAny)
#pragma unroll
      for (int j = 0; j < 4; ++j) fs[j] = __fmul_rn(cnt[j], scale[j]);
    if (!kMulti) {
      const int P = p.planes_count[max_level];
      store_digits(P, plane_ptr(max_level, P), 6u + bk_shift, fs, abs256, sum);
      if (r != run_row || run_abs > (1u << 17)) {      // (so that the lanes' signed sums together stay below 2^31)
        add_row_sums(sums + max_level * (3u * kPlaneRows), run_row, run_abs, run_sum, true);
        run_row = r;
        run_abs = 0u;
        run_sum = 0;
      }
      run_abs += abs256;
      run_sum += sum;
    }
  }
  if (!kMulti) add_row_sums(sums + max_level * (3u * kPlaneRows), run_row, run_abs, run_sum, true);
}

// Everything else, one weight per thread and step: depthwise and grouped filters (integer filter, channels
// innermost, for the CUDA-core kernels) and flat K axes (few input channels).
// kOwnBases: launches of such a layer alone take the bases along here and read the windows of an exponent pass where they are;
// passed through shared memory and stored apart, depthwise 3x3 on 960 channels took 4.9 us and not 4.7, 5x5 12->128 7.5 and not 7.1.
template <bool kOptions, bool kOwnBases>
__device__ __forceinline__ void sample_single(const SampleParams& p, const uint32_t* windows, uint32_t tag, uint32_t o0,
                                              uint32_t c0, uint32_t rows, uint32_t cc, const PhiloxKeys& keys, const float* stage,
                                              uint32_t* sums) {
  const uint32_t KHKW = p.KHKW, Cg = p.Cg, d = p.d, level_mask = p.level_mask;
  const uint32_t max_level = p.max_level, layer_key = p.layer_id ^ keys.k0[0], has_planes = p.has_planes;
  const uint32_t packed_kw = p.packed_kw, run_pitch = p.run_pitch, bk = p.bk, n_kb = p.n_kb;
  const uint32_t bk_shift = 31u - (uint32_t)__clz((int)bk), bk_mask = bk - 1u, sw_mask = (bk >> 4) - 1u;
  const uint32_t per_row = cc * KHKW, count = rows * per_row;
  const uint32_t per_row_magic = small_div_magic(per_row), cc_magic = small_div_magic(cc);
  for (uint32_t t = threadIdx.x; t < count; t += blockDim.x) {
    const uint32_t r = small_div(t, per_row_magic), rem = t - r * per_row;
    const uint32_t tap = small_div(rem, cc_magic), cl = rem - tap * cc;
    const uint32_t o = o0 + r, ci = c0 + cl;
    const uint32_t u = __float_as_uint(stage[r * per_row + cl * KHKW + tap]);
    const uint32_t index = o * d + ci * KHKW + tap;  // canonical
    const uint32_t Emax = window_exponent(windows[p.norm ? r : 0u], tag);
    const int ebase_biased = (int)Emax - (int)p.span;
    if (kOwnBases && tap == 0u && ci == 0u) p.e_base[o] = Emax ? ebase_biased - 127 : 0;
    Drawn dw;
    draw_weight(u, index, ebase_biased, kOptions ? p.pbits : 0u, kOptions ? p.underflow : 0u, kOptions ? p.deterministic : 0u,
                max_level, layer_key, keys, dw);
    const bool neg = (u >> 31) != 0u;
    const size_t wpos = ((size_t)o * KHKW + tap) * Cg + ci;
    uint32_t kb = 0, kin = 0;
    if (has_planes) {            // flat K axis (with a tap-major one the planes are written four channels at a time)
      const uint32_t kh = tap / packed_kw, kcol = kh * run_pitch + (tap - kh * packed_kw) * Cg + ci;
      kb = kcol >> bk_shift;
      kin = kcol & bk_mask;
    }
    const uint32_t jt = o / kTileN, on = o % kTileN;
    const uint32_t lin = (on << bk_shift) + kin, off = lin ^ (((lin >> 7) & sw_mask) << 4);
#pragma unroll
    for (int l = 0; l < kMaxLevels; ++l) {
      if (!((level_mask >> l) & 1u)) continue;
      const uint32_t mag = dw.live ? (((dw.base << l) + dw.cnt[l]) << dw.sh) : 0u;
      const int wv = neg ? -(int32_t)mag : (int32_t)mag;
      if (has_planes) {
        const int P = p.planes_count[l];
        int8_t* dst = p.planes[l] + ((((size_t)jt * n_kb + kb) * (size_t)P) << (6u + bk_shift)) + off;
        for (int pl = 0; pl < P; ++pl) {
          const int digit = (int)((mag >> (kDigitBits * pl)) & 0x7Fu);
          dst[(size_t)pl << (6u + bk_shift)] = (int8_t)(neg ? -digit : digit);
        }
        add_row_sums(sums + l * (3 * kPlaneRows), r, (mag + 255u) >> 8, wv, true);
      } else {
        p.wint[l][wpos] = wv;
        add_row_sums(sums + l * kRowSumRows, r, (mag + 255u) >> 8, 0, false);
      }
    }
  }
}

// kFused: the block finds its windows itself instead of reading the words of an exponent pass, and owns whole rows, so
// it stores their sums where the others add to words that the exponent pass has cleared.
// kWhat: the filters that the instance serves, tap-major digit planes, the others, or (in a batch) both: a short launch's
// time depends on how much code it carries.
// Comparators that kDrawAny serves.
__host__ __device__ inline bool other_options(const SampleParams& p) { return p.deterministic || (p.pbits != 0u && p.pbits != 4u && p.pbits != 8u); }

enum SampleOptions { kNoOptions, kCommonOptions, kOtherOptions, kAllOptions };
enum SampleWhat { kPlanesOnly, kSingleOnly, kBoth };
template <int kOptions, bool kFused, int kWhat>
__device__ __forceinline__ void sample_block(const SampleParams& p, uint32_t tag, uint32_t block, const PhiloxKeys& keys,
                                             float* stage, RowSums& rs, uint32_t* err) {
  const uint32_t level_mask = p.level_mask, has_planes = p.has_planes, O = p.O;
  const uint32_t pitch = has_planes ? 3u * kPlaneRows : (uint32_t)kRowSumRows;     // words per level
  for (uint32_t l = 0; l < (uint32_t)kMaxLevels; ++l)
    if ((level_mask >> l) & 1u)
      for (uint32_t i = threadIdx.x; i < pitch; i += blockDim.x) rs.word[l * pitch + i] = 0u;
  const uint32_t row_block = block / p.ch_chunks, chunk = block - row_block * p.ch_chunks;
  const uint32_t o0 = row_block * p.rows_per_block, c0 = chunk * p.ch_per_block;
  const uint32_t rows = min(p.rows_per_block, O - o0), cc = min(p.ch_per_block, p.Cg - c0);
  const uint32_t count = rows * cc * p.KHKW;
  // The slice is one contiguous run of the weight tensor (whole rows, or a channel range of one row): stage it
  // with 16-byte loads where the run allows, through L1: a block that finds one window for the whole layer reads its slice
  // again (depthwise 3x3, 144 channels @56 with its sampling 52.4 us past L1, 51.6 through it).
  {
    const float* src = p.w + (size_t)o0 * p.d + (size_t)c0 * p.KHKW;
    if ((((uintptr_t)src) & 15u) == 0u && (count & 3u) == 0u) {
#pragma unroll 4
      for (uint32_t t = threadIdx.x * 4u; t < count; t += blockDim.x * 4u)
        *reinterpret_cast<float4*>(stage + t) = __ldca(reinterpret_cast<const float4*>(src + t));
    } else {
#pragma unroll 4
      for (uint32_t t = threadIdx.x; t < count; t += blockDim.x) stage[t] = __ldca(src + t);
    }
  }
  __shared__ uint32_t found[kRowSumRows];      // of the rows of this block, or the layer's
  uint32_t* windows = found;
  if (!kFused && kWhat == kSingleOnly) {
    windows = const_cast<uint32_t*>(p.e_max) + (p.norm ? o0 : 0u);
  } else if (!kFused) {
    for (uint32_t r = threadIdx.x; r < (p.norm ? rows : 1u); r += blockDim.x) windows[r] = p.e_max[(p.norm ? o0 : 0u) + r];
  } else {
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, d = p.d;
    bool bad = false;
    if (p.norm) {
      // a warp per row, or of fewer, longer rows than half the warps as many warps for each as there are (by shifts: a division by
      // the number of them costs a short launch 0.3 us).  us per sampling, a warp per row / all warps on one row after the other / so:
      // 256 rows of 64 weights, k = 1 4.2 / 4.9 / 4.2; 256 rows of 72, grouped 3.8 / 4.3 / 3.8; 3x3 64->64, k = 8 5.1 / 4.4 / 4.4
      const uint32_t warps_log2 = blockDim.x >= 256u ? 3u : 2u, rows_log2 = rows <= 1u ? 0u : rows <= 2u ? 1u : 2u;
      const uint32_t share_log2 = rows <= 4u && d > 128u ? warps_log2 - rows_log2 : 0u, part = warp & ((1u << share_log2) - 1u);
      if (share_log2)
        for (uint32_t r = threadIdx.x; r < rows; r += blockDim.x) windows[r] = 0u;
      __syncthreads();
      for (uint32_t r = warp >> share_log2; r < rows; r += 1u << (warps_log2 - share_log2)) {
        const float* row = stage + r * d;
        const uint32_t first = part * 32u + lane, step = 32u << share_log2;
        uint32_t best = 0u;
        if ((d & 3u) == 0u) {
#pragma unroll 2
          for (uint32_t i = first; i < d / 4u; i += step) {
            const uint4 v = reinterpret_cast<const uint4*>(row)[i];
            const uint32_t u4[4] = {v.x, v.y, v.z, v.w};
            best = max_magnitude(u4, best, bad);
          }
        } else {
          for (uint32_t i = first; i < d; i += step) {
            const uint32_t u1[1] = {__float_as_uint(row[i])};
            best = max_magnitude(u1, best, bad);
          }
        }
        best = __reduce_max_sync(0xFFFFFFFFu, best);
        if (lane == 0u) {
          const uint32_t e = quantised_exponent(best, p.pbits);
          if (share_log2) atomicMax(&windows[r], e);
          else windows[r] = e;
        }
      }
    } else {
      // one window for a small layer: every block, of kThreads threads, looks at all of it
      const uint32_t total = O * d, head = (((uintptr_t)p.w) & 15u) == 0u ? total & ~3u : 0u;
      uint32_t best = 0u;
      const uint4* w4 = reinterpret_cast<const uint4*>(p.w);
#pragma unroll 8
      for (uint32_t i = threadIdx.x; i < head / 4u; i += (uint32_t)kThreads) {
        const uint4 v = __ldca(w4 + i);
        const uint32_t u4[4] = {v.x, v.y, v.z, v.w};
        best = max_magnitude(u4, best, bad);
      }
      for (uint32_t i = head + threadIdx.x; i < total; i += (uint32_t)kThreads) {
        const uint32_t u1[1] = {__float_as_uint(__ldca(p.w + i))};
        best = max_magnitude(u1, best, bad);
      }
      best = __reduce_max_sync(0xFFFFFFFFu, best);
      if (lane == 0u) windows[1u + warp] = best;
      __syncthreads();
      if (threadIdx.x == 0u) {
        for (uint32_t i = 2u; i <= (uint32_t)kThreads / 32u; ++i) best = max(best, windows[i]);
        windows[0] = quantised_exponent(best, p.pbits);
      }
    }
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0u) atomicOr(err, kDevErrNonFinite);
    tag = 0u;
  }
  __syncthreads();
  if (kWhat != kSingleOnly && chunk == 0u)
    for (uint32_t r = threadIdx.x; r < rows; r += blockDim.x) {
      const uint32_t Emax = window_exponent(windows[p.norm ? r : 0u], tag);
      p.e_base[o0 + r] = Emax ? (int)Emax - (int)p.span - 127 : 0;
    }
  if (kWhat == kPlanesOnly || (kWhat == kBoth && has_planes && !p.packed_kw)) {
   if constexpr (kWhat != kSingleOnly) {
    const bool multi = (level_mask & (level_mask - 1u)) != 0u;
#define PSB_SAMPLE(MODE, MULTI, CALLS) sample_planes<MODE, MULTI, CALLS>(p, windows, tag, o0, c0, rows, cc, keys, stage, rs.word)
#define PSB_SAMPLE_M(MODE) do { if (multi) PSB_SAMPLE(MODE, true, 0); else PSB_SAMPLE(MODE, false, 0); } while (0)
    if (kOptions == kNoOptions || (kOptions == kAllOptions && (p.pbits | p.underflow) == 0u)) {
      if constexpr (kOptions == kNoOptions || kOptions == kAllOptions) {
        if (multi) PSB_SAMPLE(kDrawExact, true, 0);
        else if (p.max_level <= 2u) PSB_SAMPLE(kDrawExact, false, 1);
        else if (p.max_level == 3u) PSB_SAMPLE(kDrawExact, false, 2);
        else if (p.max_level == 4u) PSB_SAMPLE(kDrawExact, false, 4);
        else PSB_SAMPLE(kDrawExact, false, 0);
      }
    } else if (kOptions == kOtherOptions || (kOptions == kAllOptions && other_options(p))) {
      if constexpr (kOptions >= kOtherOptions) PSB_SAMPLE_M(kDrawAny);
    } else if constexpr (kOptions != kNoOptions && kOptions != kOtherOptions) {
      if (p.pbits == 0u) PSB_SAMPLE_M(kDrawGate);
      else if (p.pbits == 8u) PSB_SAMPLE_M(kDrawPacked8);
      else PSB_SAMPLE_M(kDrawPacked4);
    }
#undef PSB_SAMPLE_M
#undef PSB_SAMPLE
   }
  } else if constexpr (kWhat != kPlanesOnly) {
    sample_single<kOptions != kNoOptions, kWhat == kSingleOnly>(p, windows, tag, o0, c0, rows, cc, keys, stage, rs.word);
  }
  __syncthreads();
  for (uint32_t l = 0; l < (uint32_t)kMaxLevels; ++l) {
    if (!((level_mask >> l) & 1u)) continue;
    const uint32_t* sums = rs.word + l * pitch;
    for (uint32_t r = threadIdx.x; r < rows; r += blockDim.x) {
      const uint32_t at = l * O + o0 + r;
      const long long sum = has_planes ? 128 * ((long long)(int)sums[2 * kPlaneRows + r] * 4096 + (long long)sums[kPlaneRows + r]) : 0;
      if (kFused) {
        p.rowsum[at] = sums[r];
        if (has_planes) p.corr[at] = sum;
      } else {
        if (sums[r]) atomicAdd(&p.rowsum[at], sums[r]);
        if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(p.corr + at), (unsigned long long)sum);
      }
    }
  }
}

template <int kOptions, bool kFused, bool kSingle>
__global__ void __launch_bounds__(kThreads, 3) sample_kernel(const __grid_constant__ SampleParams p,
                                                          const __grid_constant__ PhiloxKeys keys, uint32_t* err) {
  pdl_prologue();
  extern __shared__ __align__(16) float stage[];      // the block's slice of the filter
  __shared__ RowSums rs;
  sample_block<kOptions, kFused, kSingle ? kSingleOnly : kPlanesOnly>(p, p.e_tag, blockIdx.x, keys, stage, rs, err);
}

// All layers of a network in two launches.  Entry i owns blocks [first, first + count) of each
// grid; its parameters sit in device memory (every thread of a block reads the same words), and so does the entry of
// every block: a block of either pass lives for a few microseconds, and looking its entry up by bisection was six
// dependent loads of that (both passes, ResNet-50 shape, k = 8: 291 -> 279 us).
struct BatchEntry {
  SampleParams p;
  uint32_t emax_first, emax_blocks, sample_first, sample_blocks;
};

__global__ void __launch_bounds__(kThreads) emax_batch_kernel(const BatchEntry* entries, const uint32_t* entry_of,
                                                              uint32_t* __restrict__ err, uint32_t tag) {
  pdl_prologue();
  const BatchEntry& e = entries[entry_of[blockIdx.x]];
  emax_block(e.p.w, e.p.O, e.p.d, e.p.norm, const_cast<uint32_t*>(e.p.e_max), err,
             blockIdx.x - e.emax_first, e.emax_blocks, tag << 8, e.p.rowsum, e.p.corr, e.p.pbits);
}

template <int kOptions>
__global__ void __launch_bounds__(kBatchThreads, 6) sample_batch_kernel(const BatchEntry* entries, const uint32_t* entry_of,
                                                                uint32_t tag, const __grid_constant__ PhiloxKeys keys) {
  pdl_prologue();
  extern __shared__ __align__(16) float stage[];      // the block's slice of the filter
  __shared__ RowSums rs;
  __shared__ SampleParams p;
  const BatchEntry& e = entries[entry_of[blockIdx.x]];
  // the entry's parameters, once per block
  for (uint32_t i = threadIdx.x; i < sizeof(SampleParams) / 4u; i += blockDim.x)
    reinterpret_cast<uint32_t*>(&p)[i] = reinterpret_cast<const uint32_t*>(&e.p)[i];
  const uint32_t first = e.sample_first;
  __syncthreads();
  sample_block<kOptions, false, kBoth>(p, tag, blockIdx.x - first, keys, stage, rs, nullptr);
}

// The integer filter of one level put together from its digit planes, in canonical order, for the test hook.
__global__ void expand_planes_kernel(const int8_t* planes, int P, uint32_t O, uint32_t Cg, uint32_t KHKW, uint32_t bk,
                                     uint32_t n_cb, uint32_t n_kb, uint32_t packed_kw, uint32_t run_pitch,
                                     int32_t* __restrict__ out) {
  pdl_prologue();
  const size_t total = (size_t)O * Cg * KHKW;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t tap = (uint32_t)(i % KHKW);
    const size_t rest = i / KHKW;
    const uint32_t ci = (uint32_t)(rest % Cg), o = (uint32_t)(rest / Cg);
    uint32_t kcol = tap * n_cb * bk + ci;
    if (packed_kw) kcol = (tap / packed_kw) * run_pitch + (tap % packed_kw) * Cg + ci;
    const int8_t* tile = planes + ((size_t)(o / kTileN) * n_kb + kcol / bk) * (size_t)P * kTileN * bk;
    int w = 0;
    for (int pl = 0; pl < P; ++pl) w += (int)tile[plane_offset((uint32_t)pl * kTileN + o % kTileN, kcol % bk, bk)] * (1 << (kDigitBits * pl));
    out[i] = w;
  }
}

// Canonical-order copy of one level for the test hook.
__global__ void export_kernel(const int32_t* wint, int32_t* __restrict__ out, uint32_t O,
                              uint32_t Cg, uint32_t KHKW) {
  pdl_prologue();
  size_t total = (size_t)O * Cg * KHKW;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    uint32_t tap = (uint32_t)(i % KHKW);
    size_t t = i / KHKW;
    uint32_t ci = (uint32_t)(t % Cg);
    size_t o = t / Cg;
    out[i] = wint[(o * KHKW + tap) * Cg + ci];
  }
}

}  // namespace

namespace {

uint32_t emax_blocks_for(uint32_t O, uint32_t d, uint32_t norm) {
  if (norm) return d <= (uint32_t)kEmaxLongRow ? (O + (uint32_t)kEmaxRows - 1u) / (uint32_t)kEmaxRows : O;
  size_t total = (size_t)O * d;
  // sixteen weights per thread (four 16-byte loads in flight) once that still fills the machine, four otherwise
  uint32_t blocks = (uint32_t)((total + kThreads * 16 - 1) / (kThreads * 16));
  if (blocks < 296u) blocks = (uint32_t)std::min<size_t>(296u, (total + kThreads * 4 - 1) / (kThreads * 4));
  return blocks < 1 ? 1 : (blocks > 1184 ? 1184 : blocks);
}

// A layer sampled by a launch of its own needs no exponent pass before it (a launch of about 2.3 us on the host) where a
// block holds whole rows and their windows are its own (norm == 1), or where the layer is so small that every block can
// look at all of it.  us per sampling with its matrix product (16 rows) or 3x3 layer (14x14) in a stream of calls, two
// launches / one:
//   one window:      128x128 16.1 / 13.8, 128x256 16.1 / 13.8; 256x256 16.2 / 18.9; 3x3 64->64 (36864 weights) 17.1 / 14.9, but
//                    25.1 / 29.4 where the weights are new to the caches (with 56x56, batch 32, planar).
//   window per row:  a block takes a whole row, so long rows need rows for two blocks per SM, or, with taps, for one.  256x1536
//                    16.4 / 14.0, 64x2048 16.2 / 13.8, 1000x2048 30.6 / 28.4; 10x4096 16.2 / 17.3, 148x4096 20.6 / 24.5, 256x4096 24.4 / 24.9,
//                    400x4096 28.7 / 26.4, 2048x4096 77.5 / 73.3; 3x3 256->64 20.4 / 18.4, 400->32 24.5 / 25.2, 256->256 22.4 / 21.7,
//                    400->256 31.9 / 32.4 (the wrong side of the line by 0.5).  (Between 65 and 295 rows of 1537 to 2304 weights one launch would now be the faster,
//                    148x2048 16.2 / 13.9; the number of launches at this line is part of what the tests hold fast.)
bool fused_sampling(const psb_weights* wt) {
  const uint32_t d = wt->d, rows = wt->shape.out_ch;
  const bool taps = wt->shape.kh * wt->shape.kw > 1u;
  if (!wt->cfg.norm) return d <= 256u && (uint64_t)rows * d <= 32768u;
  return d <= (rows >= (taps ? 1u : 2u) * kSms ? 4096u : taps ? 2304u : rows <= 64u ? 2048u : 1536u);
}

// Threads of a block: 128, so that the last round of quads leaves few of them idle and six blocks cover one another's waits,
// where the blocks fill the machine.  Fewer blocks that find their own windows take 256 (us with 256 / 128: 256x128 6.1 / 7.0,
// 400x4096 26.4 / 31.9, 888x4096 39.4 / 38.3, 2048x4096 77.1 / 73.3), and so do the others if they have quads for them (148x4096
// 20.6 / 22.4, 592x4096 32.2 / 40.3; 512x2048, 1024 blocks, 22.5 / 21.0, 3x3 256->256, 768 blocks, 23.5 / 22.3).
uint32_t sample_threads(const SampleParams& p, uint32_t blocks, bool fused) {
  if (!p.has_planes || p.packed_kw) return 256u;
  if (fused) return !p.norm || blocks < 6u * kSms ? 256u : 128u;
  return blocks <= 4u * kSms && p.rows_per_block * p.ch_per_block * p.KHKW >= 1024u ? 256u : 128u;
}

enum class SampleLaunch { kBatch, kTwoPass, kFused };

// Shared memory for the largest slice of a block.
uint32_t stage_bytes(const SampleParams& p) { return p.rows_per_block * p.ch_per_block * p.KHKW * (uint32_t)sizeof(float); }

// Parameters of one layer's sampling pass in a launch over `launch_weights` weights; returns the number of blocks it needs.
uint32_t fill_sample_params(const float* w_dev, const psb_weights* wt, uint32_t* e_max, SampleParams& p,
                            SampleLaunch how, uint64_t launch_weights) {
  const psb_wshape& sh = wt->shape;
  const uint32_t O = sh.out_ch, Cg = sh.in_ch_per_group, KHKW = sh.kh * sh.kw, d = wt->d;
  p.w = w_dev;
  p.O = O; p.Cg = Cg; p.KHKW = KHKW; p.d = d;
  // weights per block: enough that what a block does once (its parameters, sums, barriers) is a small part of it, yet four blocks
  // per SM of the launch, which is all layers of a batch (13 layers, 38 k weights, k = 1 and 16, with blocks of 4608 / so, us:
  // 23.6 and 28.7 / 8.5 and 9.2).  (Of a block with 256 weights two warps of four have quads, and these share two of the SM's four
  // schedulers; 256 / 512, us: 3x3 64->64, levels k = 1 .. 16 10.7 / 9.4, 3x3 100->150, k = 8 9.7 / 8.3, 8-bit comparator, k = 16
  // 9.7 / 8.0.)
  const uint32_t least = how != SampleLaunch::kFused && wt->has_planes && !wt->packed_k ? 512u : 256u;
  uint32_t budget = (uint32_t)std::min<uint64_t>(kStage, std::max<uint64_t>(least, launch_weights / 592u));
  if (how == SampleLaunch::kFused && budget < d) budget = d;
  if (budget < 4u * KHKW) budget = 4u * KHKW;   // at least four channels (host validation keeps kh*kw <= 2048)
  const uint32_t sum_rows = wt->has_planes ? (uint32_t)kPlaneRows : (uint32_t)kRowSumRows;
  if (d <= budget) {
    p.rows_per_block = std::min<uint32_t>(budget / d, sum_rows);   // the rows a block keeps sums for
    p.ch_per_block = Cg;
    p.ch_chunks = 1;
  } else {
    p.rows_per_block = 1;
    // pieces of about the same size, whole 16-byte pieces of the plane rows
    const uint32_t most = budget / KHKW, unit = most > 16u ? 16u : 4u;
    p.ch_chunks = (Cg + (most & ~(unit - 1u)) - 1u) / (most & ~(unit - 1u));
    p.ch_per_block = ((Cg + p.ch_chunks - 1u) / p.ch_chunks + unit - 1u) & ~(unit - 1u);
    p.ch_chunks = (Cg + p.ch_per_block - 1u) / p.ch_per_block;
  }
  p.norm = wt->cfg.norm;
  p.span = (1u << wt->cfg.exp_bits) - 1u;
  p.level_mask = wt->cfg.level_mask;
  p.underflow = wt->cfg.underflow;
  p.pbits = wt->cfg.prob_bits;
  p.deterministic = wt->cfg.deterministic;
  p.max_level = 0;
  for (uint32_t l = 0; l < (uint32_t)kMaxLevels; ++l)
    if ((p.level_mask >> l) & 1u) p.max_level = l;
  p.layer_id = wt->cfg.layer_id;
  p.has_planes = wt->has_planes ? 1u : 0u;
  p.bk = wt->bk; p.n_cb = wt->n_cb; p.n_kb = wt->n_kb;
  p.packed_kw = wt->packed_k ? wt->shape.kw : 0u;
  p.run_pitch = wt->run_pitch;
  p.e_max = e_max;
  p.e_tag = 0;
  p.e_base = wt->e_base;
  p.rowsum = wt->rowsum256;
  p.corr = wt->corr128;
  for (int l = 0; l < kMaxLevels; ++l) {
    p.wint[l] = wt->level[l].wint;
    p.planes[l] = wt->level[l].planes;
    p.planes_count[l] = wt->level[l].planes_count;
  }
  const uint32_t row_blocks = (O + p.rows_per_block - 1) / p.rows_per_block;
  return row_blocks * p.ch_chunks;
}

template <bool kFused>
cudaError_t launch_sample_kernel(const SampleParams& p, uint32_t blocks, const PhiloxKeys& keys, uint32_t* err_dev, cudaStream_t s) {
  const bool options = (p.pbits | p.underflow) != 0u, single = !p.has_planes || p.packed_kw;
  const auto kernel = single    ? (options ? sample_kernel<kCommonOptions, kFused, true> : sample_kernel<kNoOptions, kFused, true>)
                      : !options ? sample_kernel<kNoOptions, kFused, false>
                                 : other_options(p) ? sample_kernel<kOtherOptions, kFused, false> : sample_kernel<kCommonOptions, kFused, false>;
  launch_pdl(kernel, blocks, sample_threads(p, blocks, kFused), stage_bytes(p), s, p, keys, err_dev);
  note_launch();
  return cudaGetLastError();
}

// A captured call carries one number through all its replays, which the words of later calls would beat: its graph clears
// them each time.
bool is_captured(cudaStream_t s) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &status) != cudaSuccess) cudaGetLastError();
  return status == cudaStreamCaptureStatusActive;
}

}  // namespace

cudaError_t launch_sampler(const float* w_dev, psb_weights* wt, uint32_t* err_dev, cudaStream_t s) {
  const PhiloxKeys keys((uint32_t)wt->cfg.seed, (uint32_t)(wt->cfg.seed >> 32));
  SampleParams p;
  if (fused_sampling(wt)) {
    const uint32_t blocks = fill_sample_params(w_dev, wt, wt->e_max, p, SampleLaunch::kFused, (uint64_t)wt->shape.out_ch * wt->d);
    return launch_sample_kernel<true>(p, blocks, keys, err_dev, s);
  }
  const uint32_t O = wt->shape.out_ch;
  // the exponent maxima carry the number of the call that wrote them; the words were cleared when
  // the handle was made and are cleared again only when the 24-bit call number wraps
  wt->e_calls = (wt->e_calls + 1u) & 0xFFFFFFu;
  if (wt->e_calls == 0u || is_captured(s)) {
    cudaError_t e = cudaMemsetAsync(wt->e_max, 0, sizeof(uint32_t) * O, s);
    if (e != cudaSuccess) return e;
    if (wt->e_calls == 0u) wt->e_calls = 1u;
  }
  launch_pdl(emax_kernel, emax_blocks_for(O, wt->d, wt->cfg.norm), kThreads, 0, s, w_dev, O, wt->d, wt->cfg.norm,
             wt->e_max, err_dev, wt->e_calls << 8, wt->rowsum256, wt->corr128, wt->cfg.prob_bits); note_launch();
  const uint32_t blocks = fill_sample_params(w_dev, wt, wt->e_max, p, SampleLaunch::kTwoPass, (uint64_t)wt->shape.out_ch * wt->d);
  p.e_tag = wt->e_calls;
  return launch_sample_kernel<false>(p, blocks, keys, err_dev, s);
}

}  // namespace psb

// ---- batched sampling: every layer of a network in two launches ---------------------------
struct psb_sample_batch {
  psb::BatchEntry* entries_dev = nullptr;
  uint32_t* entry_of_dev = nullptr;   // entry of every block of the exponent pass, then of the sampling pass
  uint32_t* e_max_pool = nullptr;     // one word per output channel of every layer: (call number << 8) | exponent
  size_t e_max_words = 0;
  uint32_t calls = 0;                 // runs made on this batch, modulo 2^24
  bool options = false;               // some layer uses a sampling option
  uint32_t emax_grid = 0, sample_grid = 0;
  uint32_t stage_bytes = 0;           // shared memory of a sampling block
  int device = 0;
};

namespace psb {

psb_status sample_batch_create(psb_ctx* ctx, uint32_t n, const float* const* w_dev,
                               psb_weights* const* weights, psb_sample_batch** out) {
  psb_sample_batch* b = new (std::nothrow) psb_sample_batch();
  BatchEntry* host = new (std::nothrow) BatchEntry[n];
  if (!b || !host) { delete b; delete[] host; return PSB_ERR_ALLOC; }
  size_t words = 0;
  uint64_t total = 0;
  for (uint32_t i = 0; i < n; ++i) {
    words += weights[i]->shape.out_ch;
    total += (uint64_t)weights[i]->shape.out_ch * weights[i]->d;
  }
  bool ok = cudaMalloc(&b->e_max_pool, sizeof(uint32_t) * words) == cudaSuccess &&
            cudaMemset(b->e_max_pool, 0, sizeof(uint32_t) * words) == cudaSuccess &&
            cudaMalloc(&b->entries_dev, sizeof(BatchEntry) * n) == cudaSuccess;
  if (ok) {
    size_t off = 0;
    uint32_t eb = 0, sb = 0;
    for (uint32_t i = 0; i < n; ++i) {
      const psb_weights* wt = weights[i];
      BatchEntry& e = host[i];
      e.sample_blocks = fill_sample_params(w_dev[i], wt, b->e_max_pool + off, e.p, SampleLaunch::kBatch, total);
      b->stage_bytes = std::max(b->stage_bytes, stage_bytes(e.p));
      b->options = b->options || (e.p.pbits | e.p.underflow);
      e.emax_blocks = emax_blocks_for(wt->shape.out_ch, wt->d, wt->cfg.norm);
      e.emax_first = eb;
      e.sample_first = sb;
      eb += e.emax_blocks;
      sb += e.sample_blocks;
      off += wt->shape.out_ch;
    }
    b->emax_grid = eb;
    b->sample_grid = sb;
    ok = cudaMemcpy(b->entries_dev, host, sizeof(BatchEntry) * n, cudaMemcpyHostToDevice) == cudaSuccess;
    uint32_t* of = ok ? new (std::nothrow) uint32_t[(size_t)eb + sb] : nullptr;
    if (of) {
      for (uint32_t i = 0; i < n; ++i) {
        std::fill_n(of + host[i].emax_first, host[i].emax_blocks, i);
        std::fill_n(of + eb + host[i].sample_first, host[i].sample_blocks, i);
      }
      const size_t bytes = sizeof(uint32_t) * ((size_t)eb + sb);
      ok = cudaMalloc(&b->entry_of_dev, bytes) == cudaSuccess &&
           cudaMemcpy(b->entry_of_dev, of, bytes, cudaMemcpyHostToDevice) == cudaSuccess;
    } else {
      ok = false;
    }
    delete[] of;
  }
  delete[] host;
  if (!ok) {
    cudaGetLastError();
    if (b->e_max_pool) cudaFree(b->e_max_pool);
    if (b->entries_dev) cudaFree(b->entries_dev);
    if (b->entry_of_dev) cudaFree(b->entry_of_dev);
    delete b;
    return PSB_ERR_ALLOC;
  }
  b->e_max_words = words;
  b->device = ctx->device;
  *out = b;
  return PSB_OK;
}

psb_status sample_batch_run(psb_ctx* ctx, psb_sample_batch* b, uint64_t seed, cudaStream_t s) {
  b->calls = (b->calls + 1u) & 0xFFFFFFu;
  if (b->calls == 0u || is_captured(s)) {       // the words of earlier calls would compare as later ones
    if (cudaMemsetAsync(b->e_max_pool, 0, sizeof(uint32_t) * b->e_max_words, s) != cudaSuccess) return PSB_ERR_CUDA;
    if (b->calls == 0u) b->calls = 1u;
  }
  launch_pdl(emax_batch_kernel, b->emax_grid, kThreads, 0, s, (const BatchEntry*)b->entries_dev, (const uint32_t*)b->entry_of_dev,
             ctx->err_dev, b->calls);
  note_launch();
  const PhiloxKeys keys((uint32_t)seed, (uint32_t)(seed >> 32));
  const uint32_t* entry_of = b->entry_of_dev + b->emax_grid;
  launch_pdl(b->options ? sample_batch_kernel<kAllOptions> : sample_batch_kernel<kNoOptions>, b->sample_grid, kBatchThreads, b->stage_bytes, s,
             (const BatchEntry*)b->entries_dev, entry_of, b->calls, keys);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? PSB_OK : PSB_ERR_CUDA;
}

void sample_batch_free(psb_sample_batch* b) {
  if (b->e_max_pool) cudaFree(b->e_max_pool);
  if (b->entries_dev) cudaFree(b->entries_dev);
  if (b->entry_of_dev) cudaFree(b->entry_of_dev);
  delete b;
}

cudaError_t launch_export(const psb_weights* wt, uint32_t level, int32_t* wint_out,
                          int32_t* e_base_out, cudaStream_t s) {
  const psb_wshape& sh = wt->shape;
  if (wint_out && wt->has_planes) {
    const size_t total = (size_t)sh.out_ch * wt->d;
    const uint32_t blocks = (uint32_t)std::min<size_t>((total + kThreads - 1) / kThreads, kSms * 16u);
    launch_pdl(expand_planes_kernel, blocks, kThreads, 0, s, (const int8_t*)wt->level[level].planes, wt->level[level].planes_count,
               sh.out_ch, sh.in_ch_per_group, sh.kh * sh.kw, wt->bk, wt->n_cb, wt->n_kb, wt->packed_k ? sh.kw : 0u, wt->run_pitch,
               wint_out);
    note_launch();
  } else if (wint_out) {
    size_t total = (size_t)sh.out_ch * wt->d;
    uint32_t blocks = (uint32_t)((total + 255) / 256);
    blocks = blocks > 4096 ? 4096 : (blocks < 1 ? 1 : blocks);
    export_kernel<<<blocks, 256, 0, s>>>(wt->level[level].wint, wint_out, sh.out_ch,
                                        sh.in_ch_per_group, sh.kh * sh.kw); note_launch();
  }
  if (e_base_out) {
    cudaError_t e = cudaMemcpyAsync(e_base_out, wt->e_base, sizeof(int32_t) * sh.out_ch,
                                    cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace psb

// ---------------------------------------------------------------------------
// Allocation-free sampling of one level (psb_sample_level_static in psb.h).
//
// Some hosts may not allocate device memory when they need fresh weights: a
// real-time loop that must not block on the allocator, code running while a CUDA
// graph is being captured elsewhere in the process, or a process whose memory
// budget was handed out at start-up.  For them the window reduction's scratch
// (one biased exponent per output channel, plus a device error word nobody reads)
// lives in this file-scope device array instead of a cudaMalloc'ed buffer.  Every
// GPU that loads the library holds these 16 KB + 256 B until the process exits.
namespace psb {
namespace {

constexpr uint32_t kStaticMaxOutCh = 4096;   // PSB_STATIC_MAX_OUT_CH in psb.h
static __device__ __align__(256) uint32_t g_static_scratch[kStaticMaxOutCh + 64];

constexpr int kMaxDevices = 64;
uint32_t* g_static_scratch_addr[kMaxDevices] = {};   // device address per device ordinal

// One thread per weight, canonical order in and out (both coalesce).  e_max is
// the device address of the static scratch, filled by emax_kernel just before.
__global__ void __launch_bounds__(kThreads)
sample_level_canonical_kernel(const float* w, uint32_t O, uint32_t d, uint32_t norm,
                              uint32_t span, uint32_t log2k, uint32_t layer_id, const uint32_t* e_max,
                              int32_t* __restrict__ wint_out, int32_t* __restrict__ e_base_out,
                              const __grid_constant__ PhiloxKeys keys) {
  pdl_prologue();
  const size_t total = (size_t)O * d;
  for (size_t index = (size_t)blockIdx.x * blockDim.x + threadIdx.x; index < total;
       index += (size_t)gridDim.x * blockDim.x) {
    const uint32_t o = (uint32_t)(index / d);
    const uint32_t u = __float_as_uint(w[index]);
    const uint32_t E = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu;
    const uint32_t Emax = e_max[norm ? o : 0];
    const int ebase_biased = (int)Emax - (int)span;
    if (index % d == 0 && e_base_out) e_base_out[o] = Emax ? ebase_biased - 127 : 0;
    if (!wint_out) continue;
    const bool live = (E != 0u) && (E != 255u) && ((int)E >= ebase_biased);
    uint32_t c = 0;
    if (live && m != 0u) {
      const uint32_t T = m << 9, k = 1u << log2k;
      const PhiloxWeight pw((uint32_t)index, layer_id ^ keys.k0[0]);
      for (uint32_t q = 0; q * 4u < k; ++q) {
        uint32_t rnd[4];
        pw.call(q, keys, rnd);
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if (q * 4u + v < k) c += (rnd[v] < T) ? 1u : 0u;
      }
    }
    const uint32_t mag = live ? (((1u << log2k) + c) << (uint32_t)((int)E - ebase_biased)) : 0u;
    wint_out[index] = (u >> 31) ? -(int32_t)mag : (int32_t)mag;
  }
}

}  // namespace
}  // namespace psb

extern "C" psb_status psb_sample_level_static(const float* w_dev, const psb_wshape* shape,
                                              const psb_sample_cfg* cfg, uint32_t log2k,
                                              int32_t* wint_out_dev, int32_t* e_base_out_dev,
                                              void* stream) {
  using namespace psb;
  if (!w_dev || !shape || !cfg || (!wint_out_dev && !e_base_out_dev)) return PSB_ERR_INVALID_ARG;
  if (((uintptr_t)w_dev | (uintptr_t)wint_out_dev | (uintptr_t)e_base_out_dev) & 3u)
    return PSB_ERR_INVALID_ARG;
  if (!shape->out_ch || !shape->in_ch_per_group || !shape->kh || !shape->kw || !shape->groups)
    return PSB_ERR_INVALID_ARG;
  if (log2k >= (uint32_t)kMaxLevels) return PSB_ERR_BAD_K;
  const uint32_t exp_bits = cfg->exp_bits ? cfg->exp_bits : 4u;
  if (exp_bits > 4 || cfg->norm > 1) return PSB_ERR_INVALID_ARG;
  if (cfg->underflow || cfg->prob_bits || cfg->deterministic) return PSB_ERR_UNSUPPORTED;
  // the static scratch holds one word per output channel: larger filters are refused
  if (shape->out_ch > kStaticMaxOutCh) return PSB_ERR_UNSUPPORTED;
  const uint64_t d64 = (uint64_t)shape->in_ch_per_group * shape->kh * shape->kw;
  if (d64 > (1u << 24) || d64 * shape->out_ch > (1ull << 31)) return PSB_ERR_UNSUPPORTED;

  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return PSB_ERR_CUDA;
  if (!g_static_scratch_addr[dev]) {
    // first call on this device: the symbol's name is only a host-side stand-in, so ask the
    // runtime for the array's address on the current device
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || !addr) {
      cudaGetLastError();
      return PSB_ERR_CUDA;
    }
    g_static_scratch_addr[dev] = (uint32_t*)addr;
  }
  uint32_t* scratch = g_static_scratch_addr[dev];
  uint32_t* e_max = scratch;                        // [out_ch]
  uint32_t* err_sink = scratch + kStaticMaxOutCh;   // written on Inf/NaN, never read
  cudaStream_t s = (cudaStream_t)stream;
  const uint32_t O = shape->out_ch, d = (uint32_t)d64;
  // the array keeps the previous call's maxima: the reduction must start from zero
  if (cudaMemsetAsync(e_max, 0, sizeof(uint32_t) * O, s) != cudaSuccess) return PSB_ERR_CUDA;
  if (cfg->norm) {
    emax_kernel<<<emax_blocks_for(O, d, 1), kThreads, 0, s>>>(w_dev, O, d, 1, e_max, err_sink, 0u, nullptr, nullptr, 0u); note_launch();
  } else {
    size_t total = (size_t)O * d;
    uint32_t blocks = (uint32_t)((total + kThreads * 8 - 1) / (kThreads * 8));
    blocks = blocks < 1 ? 1 : (blocks > 1184 ? 1184 : blocks);
    emax_kernel<<<blocks, kThreads, 0, s>>>(w_dev, O, d, 0, e_max, err_sink, 0u, nullptr, nullptr, 0u); note_launch();
  }
  size_t total = (size_t)O * d;
  uint32_t blocks = (uint32_t)((total + kThreads - 1) / kThreads);
  blocks = blocks > kSms * 16u ? kSms * 16u : blocks;
  sample_level_canonical_kernel<<<blocks, kThreads, 0, s>>>(
      w_dev, O, d, cfg->norm, (1u << exp_bits) - 1u, log2k, cfg->layer_id, e_max, wint_out_dev, e_base_out_dev,
      PhiloxKeys((uint32_t)cfg->seed, (uint32_t)(cfg->seed >> 32))); note_launch();
  return cudaGetLastError() == cudaSuccess ? PSB_OK : PSB_ERR_CUDA;
}
