// Host side of the dense contraction on the tensor cores (kernel: psb_mma.cuh): tensor maps, tile and ring geometry,
// choice of the mode, launch.
#include "psb_mma.cuh"

namespace psb {

namespace {

// Layers with a shortcut use the staged output stage from this many tiles per SM.  Below, the time to the first and the
// last tile counts, and half of the warps per tile lose it: 1x1 256 -> 1024 @14, batch 1 (32 tiles) 5.7 us directly, 6.5
// staged; batch 64 (1568 tiles) 18.4 and 15.7.  Without a shortcut both take the same, or the direct one less: 1x1
// 64 -> 256 @56 35.4 and 34.7, 256 -> 64 13.7 and 14.8, 3x3 128 -> 128 @28 24.3 and 25.3, 96 -> 16 @112 34.4 and 36.8.
constexpr uint64_t kStagedMinTiles = 3;

// One warp waits, with the given bound, on a barrier that has no other party: the wait runs out,
// the kernel raises the error word and returns.  Exercises mbar_wait's give-up path as the contraction
// kernel would take it, with nothing in flight.
__global__ void wait_selftest_kernel(unsigned long long limit, uint32_t* __restrict__ err) {
  __shared__ unsigned long long bar;
  __shared__ WaitCtl wc;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    wc.abort = 0;
    wc.limit = limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait(smem_u32(&bar), 0u, &wc);
  if (!ok) {
    wc.abort = 1u;
    atomicOr(err, kDevErrTimeout);
  }
  __syncthreads();
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const int*, const int*,
                                   cuuint32_t, cuuint32_t, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

CUtensorMapSwizzle swizzle_for(uint32_t bk) {
  return bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                   : (bk == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

bool is_plain_gemm(const ConvArgs& a) {
  return a.KH == 1 && a.KW == 1 && a.stride == 1 && a.pad == 0;
}

}  // namespace

cudaError_t launch_wait_selftest(psb_ctx* ctx, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(ctx->wait_limit_cycles, ctx->err_dev);
  note_launch();
  return cudaGetLastError();
}

psb_status tensor_supported(const psb_ctx* ctx, const psb_weights* wt, const ConvArgs& a) {
  if (!ctx->encode_tiled || !ctx->encode_im2col) return PSB_ERR_UNSUPPORTED;
  if (!wt->has_planes || a.groups != 1) return PSB_ERR_UNSUPPORTED;
  // each plane accumulates in 32 bits: |digit| <= 127, |x| <= 128
  if ((uint64_t)wt->d * 127ull * 128ull >= (1ull << 31)) return PSB_ERR_UNSUPPORTED;
  if (wt->packed_k) {
    // the gather kernel stages the input-row segments of a strip of output locations in 48 KB of shared memory
    return (a.KH > 120u || im2col_s8_smem(a, wt->run_pitch) > 48u * 1024u) ? PSB_ERR_UNSUPPORTED : PSB_OK;
  }
  if (a.stride > 8 || a.pad > 127 || a.KH > 128 || a.KW > 128) return PSB_ERR_UNSUPPORTED;
  return PSB_OK;
}

psb_status launch_tensor(psb_ctx* ctx, const psb_weights* wt, const ConvArgs& a, uint32_t amax, bool flip,
                         bool add_corr128, const SortedRows* sorted, cudaStream_t s) {
  TmapSet maps;
  TensorParams p;
  p.a = a;
  p.wait_limit = ctx->wait_limit_cycles;
  p.M = a.N * a.OH * a.OW;
  p.m_tiles = (p.M + kTileM - 1) / kTileM;
  p.o_tiles = wt->o_tiles;
  const uint32_t bk = wt->bk;
  p.n_cb = (a.C + bk - 1) / bk;
  p.tail_ksteps = (a.C - (p.n_cb - 1u) * bk + 31u) / 32u;
  p.im2col = is_plain_gemm(a) ? 0u : 1u;
  uint32_t pmax = 1;
  for (int l = 0; l < kMaxLevels; ++l) {
    p.planes[l] = (uint32_t)wt->level[l].planes_count;
    if (p.planes[l] > pmax) pmax = p.planes[l];
  }
  p.stage_bytes_a = kTileM * bk;
  p.stage_bytes_b_max = pmax * kTileN * bk;
  const size_t ctl_bytes = sizeof(SharedCtl) + 1024;
  const uint32_t k_iters = a.KH * a.KW * p.n_cb;
  // Resident mode: with one draw count for the whole layer, a CTA that owns a single tile of 64
  // output channels keeps that tile's digit planes in shared memory for all its row tiles.
  p.resident = 0;
  p.ctas_per_otile = 1;
  p.resident_bytes = 0;
  p.band = 0;
  p.Wp = p.tpi = p.band_rows = p.band_bytes = p.Wp_magic = p.tpi_magic = 0;
  const uintptr_t out_ptrs = (uintptr_t)a.q_out | (uintptr_t)a.residual | (uintptr_t)a.f32_out | (uintptr_t)a.acc_out;
  p.unit = 16u;
  while (p.unit > 1u && ((a.O | (uint32_t)(out_ptrs & 15u)) & (p.unit - 1u))) p.unit >>= 1;
  p.flip = flip ? 1u : 0u;
  p.perm = nullptr;
  if (a.kmap) {
    // the caller has sorted the rows by level and gathered the matrix in that order
    if (!sorted || p.im2col) return PSB_ERR_INVALID_ARG;
    p.perm = sorted->perm;
    p.m_tiles = sorted->tiles;
  }
  if (!a.kmap) {
    const uint32_t P = p.planes[a.uniform_log2k];
    const uint32_t need = k_iters * P * kTileN * bk;
    const uint32_t cpo = (uint32_t)ctx->sm_count / p.o_tiles;
    if (need <= kResidentMaxBytes && cpo >= 1 && p.o_tiles * cpo * 10u >= (uint32_t)ctx->sm_count * 9u) {
      p.resident = 1;
      p.resident_bytes = need;
      // band mode: see TensorParams; needs the specialised output stage (codes only)
      const bool codes_only = a.q_out && !a.f32_out && !a.acc_out && (p.unit >= 8u || a.out_nchw) && a.inv_step > 0.0f &&
                              P >= 2u && P <= 4u;
      const uint32_t Wp = a.W + 2u * a.pad;
      const uint32_t span = kTileM + (a.KH - 1u) * Wp + (a.KW - 1u);   // band pixels a tile touches
      const uint32_t rows = (Wp - 1u + span + Wp - 1u) / Wp;           // whatever the tile's offset in its first row
      const uint32_t bytes = round_up(rows * Wp * a.C, 1024u);
      // x / d == mulhi(x, ceil(2^32 / d)) while x * d < 2^32 (d >= 2): positions t < tpi * 128 against Wp,
      // tile numbers < N * tpi against tpi
      const uint64_t tpi = ((uint64_t)a.OH * Wp + kTileM - 1) / kTileM;
      const bool quotients_ok = Wp >= 2u && tpi >= 2u && tpi * kTileM * Wp < (1ull << 32) &&
                                (uint64_t)a.N * tpi * tpi < (1ull << 32);
      if (codes_only && !flip && p.im2col && a.stride == 1 && a.KH * a.KW > 1u && a.C == bk && (bk == 64u || bk == 128u) &&
          Wp <= 256u && rows <= 256u && (kSmemBudget - ctl_bytes - need) / bytes >= 2u && quotients_ok) {
        p.band = 1;
        p.Wp = Wp;
        p.tpi = (uint32_t)tpi;
        p.Wp_magic = (uint32_t)(((1ull << 32) + Wp - 1) / Wp);
        p.tpi_magic = (uint32_t)(((1ull << 32) + tpi - 1) / tpi);
        p.band_rows = rows;
        p.band_bytes = bytes;
        p.m_tiles = a.N * p.tpi;
      }
      p.ctas_per_otile = cpo < p.m_tiles ? cpo : p.m_tiles;
    }
  }
  // Staged outputs: channels-last codes in rows of whole 16-byte pieces.  Rows in tile order (epilogue_staged) only with a
  // shortcut: a whole row of 16 bytes per lane is written as fast directly.  Rows sorted by level (epilogue_sorted) always:
  // they lie anywhere, and no role but the output stage takes part, so flipped activations are served too.
  p.staged = (uniform_epilogue(p) && !p.band && !a.out_nchw && p.unit == 16u && (a.kmap || (a.residual && !flip)) &&
              (uint64_t)p.m_tiles * p.o_tiles >= kStagedMinTiles * (uint64_t)ctx->sm_count) ? 1u : 0u;
  const uint32_t sub_bytes = p.stage_bytes_a + (p.resident ? 0u : p.stage_bytes_b_max);
  // real-valued rows use the same region, 2 KB for each epilogue warp, where four stages still fit
  static_assert(kIoSlots * kIoTileBytes == kEpilogueWarps * 2048u, "one region serves both");
  p.real_slots = (a.f32_out && !a.acc_out && !a.out_nchw && (a.O & 3u) == 0u && !((uintptr_t)a.f32_out & 15u) &&
                  !(((uintptr_t)a.q_out | (uintptr_t)a.residual) & 3u) &&
                  (kSmemBudget - ctl_bytes - p.resident_bytes - kIoSlots * kIoTileBytes) / sub_bytes >= 4u) ? 1u : 0u;
  const size_t io_bytes = p.staged | p.real_slots ? (size_t)kIoSlots * kIoTileBytes : 0u;
  // K blocks are handed over in groups: every barrier round trip costs the issuing thread a
  // few hundred cycles, so a stage should carry about eight MMAs (M=128, N=P*64, K=32 each)
  const size_t avail = kSmemBudget - ctl_bytes - p.resident_bytes - io_bytes;
  uint32_t group = 8u / (bk / 32u);
  if (group < 1) group = 1;
  if (group > k_iters) group = k_iters;
  while (group > 1 && avail / ((size_t)group * sub_bytes) < 4) --group;
  {  // balance the groups of one tile: same number of groups, as even as possible
    const uint32_t n_groups = (k_iters + group - 1) / group;
    group = (k_iters + n_groups - 1) / n_groups;
  }
  if (p.band) group = k_iters;   // one stage = one band = every tap of a tile
  p.group = group;
  p.alternate = (!p.band && !(p.staged && !a.kmap) && !flip && group >= k_iters) ? 1u : 0u;
  uint32_t stages = (uint32_t)(p.band ? avail / p.band_bytes : avail / ((size_t)group * sub_bytes));
  if (stages > (uint32_t)kMaxStages) stages = kMaxStages;
  // An even number of stages: the two producer warps and the two MMA issuing threads each take
  // every second stage use, so with an even ring each of them keeps to its own slots and every
  // parity wait on a slot's barriers follows that same thread's previous use of the slot.  (With
  // an odd ring a thread could wait on a slot whose previous use, the other thread's, has not
  // happened yet, and a parity wait cannot tell two phases apart.)
  stages &= ~1u;
  if (stages < 2) return PSB_ERR_UNSUPPORTED;
  p.stages = stages;
  const size_t smem_bytes = (p.band ? (size_t)stages * p.band_bytes : (size_t)stages * group * sub_bytes) +
                            p.resident_bytes + io_bytes + ctl_bytes;
  for (int l = 0; l < kMaxLevels; ++l) p.corr[l] = add_corr128 && wt->level[l].planes ? wt->corr128 + (size_t)l * a.O : nullptr;
  p.rowsum256 = wt->rowsum256;
  p.amax = amax;
  // the lower two digits of a weight are at most 16383 together; the bytes fed are at most 128 where an offset is taken off
  p.mid = (uint64_t)wt->d * (add_corr128 ? 128u : amax) * 16383ull + 16383ull < (1ull << 31) ? 1u : 0u;
  const CUtensorMapSwizzle swz = swizzle_for(bk);
  EncodeTiledFn enc_tiled = (EncodeTiledFn)ctx->encode_tiled;
  EncodeIm2colFn enc_im2col = (EncodeIm2colFn)ctx->encode_im2col;
  if (p.band) {
    cuuint64_t dims[4] = {a.C, a.W, a.H, a.N};
    cuuint64_t strides[3] = {(cuuint64_t)a.C, (cuuint64_t)a.C * a.W, (cuuint64_t)a.C * a.W * a.H};
    cuuint32_t box[4] = {a.C, p.Wp, p.band_rows, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    if (enc_tiled(&maps.a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.x), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return PSB_ERR_CUDA;
  } else if (p.im2col) {
    cuuint64_t dims[4] = {a.C, a.W, a.H, a.N};
    cuuint64_t strides[3] = {(cuuint64_t)a.C, (cuuint64_t)a.C * a.W, (cuuint64_t)a.C * a.W * a.H};
    int lower[2] = {-(int)a.pad, -(int)a.pad};
    int upper[2] = {(int)a.pad - (int)(a.KW - 1), (int)a.pad - (int)(a.KH - 1)};
    cuuint32_t estr[4] = {1, a.stride, a.stride, 1};
    if (enc_im2col(&maps.a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.x), dims, strides,
                   lower, upper, bk, kTileM, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return PSB_ERR_CUDA;
  } else {
    cuuint64_t dims[2] = {a.C, a.kmap ? (cuuint64_t)p.m_tiles * kTileM : (cuuint64_t)p.M};
    cuuint64_t strides[1] = {(cuuint64_t)a.C};
    cuuint32_t box[2] = {bk, kTileM};
    cuuint32_t estr[2] = {1, 1};
    if (enc_tiled(&maps.a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(a.x), dims, strides, box,
                  estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return PSB_ERR_CUDA;
  }
  if (p.staged && !a.kmap) {
    cuuint64_t dims[2] = {a.O, p.M};
    cuuint64_t strides[1] = {(cuuint64_t)a.O};
    cuuint32_t box[2] = {(cuuint32_t)kTileN, kTileM};
    cuuint32_t estr[2] = {1, 1};
    for (int i = 0; i < 2; ++i)
      if (enc_tiled(i ? &maps.res : &maps.out, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, i ? const_cast<void*>(a.residual) : a.q_out, dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return PSB_ERR_CUDA;
  }
  for (int l = 0; l < kMaxLevels; ++l) p.planes_ptr[l] = wt->level[l].planes;

  p.tile_mask = a.kmap ? sorted->tile_mask : nullptr;
  const uint32_t n_tiles = p.m_tiles * p.o_tiles;
  const uint32_t grid = p.resident ? p.o_tiles * p.ctas_per_otile
                                   : (n_tiles < (uint32_t)ctx->sm_count ? n_tiles : (uint32_t)ctx->sm_count);
  cudaError_t e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreadsTensor);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int kind = uniform_epilogue(p) ? (a.kmap ? kSortedRows : kOneLevel)
                                       : !a.f32_out || a.acc_out ? kGeneralOutputs : a.kmap ? kRealSorted : kRealOutputs;
  // (the levels of sorted rows all have as many planes)
  const bool common = kind == kOneLevel || kind == kSortedRows;
  const uint32_t planes = p.planes[a.kmap ? (uint32_t)__builtin_ctz(a.level_mask & 0x7Fu) : a.uniform_log2k];
  const int rec = !common || planes != 3u ? kPlainSums : add_corr128 ? kAddSums : p.mid ? kMidSums : kPlainSums;
  const bool timed = ctx->time_contraction && ctx->t_begin[0] && ctx->timed_launches < psb_ctx::kTimedLaunches;
  if (timed) cudaEventRecord(ctx->t_begin[ctx->timed_launches], s);
  e = bk == 128 ? launch_mma_kernel<128>(cfg, maps, p, ctx->device, kind, rec)
      : bk == 64 ? launch_mma_kernel<64>(cfg, maps, p, ctx->device, kind, rec)
                 : launch_mma_kernel<32>(cfg, maps, p, ctx->device, kind, rec);
  note_launch();
  if (timed) {
    cudaEventRecord(ctx->t_end[ctx->timed_launches], s);
    ++ctx->timed_launches;
  }
  if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) return PSB_ERR_CUDA;
  return PSB_OK;
}

}  // namespace psb
