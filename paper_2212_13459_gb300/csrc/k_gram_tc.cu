// k_gram_tc.cu -- Gram statistics on the tensor cores: sum over owned pixels p of V_p V_p^T
// (Eq. 4, accumulated block by block as in Algorithm 1, Step 1).
//
// GEMM view: D[M x N] = A[M x K] B[K x N] with M = 128 channels of the I tile, N = channels of
// the J tile (64 / 128 / 256), K = pixels. Both operands are the same NHWC activation, so both
// are MN-major in shared memory (64 channels = 128 bytes contiguous per pixel row, 128-byte
// swizzle). One TMA box of 64 pixels feeds every operand slab of a K step. Each block gets its
// own tensor map whose bounds are its owned rectangle, so pixels outside it read as zero and
// never enter the sum. Every CTA accumulates one (I, J) tile over one run of boxes in TMEM
// (FP32) and writes it out; a fixed-order compensated reduction adds the runs (deterministic).
// When the I tile's channels are among the J tile's (C <= 128, and the diagonal tiles of
// larger C), the A operand is read from the B slabs already in shared memory instead of being
// loaded again; A channels past C (C = 64) read a slab of zeros written once per CTA.
#include <algorithm>

#include "nst_internal.cuh"
#include "nst_kernels.h"
#include "tc_ptx.cuh"

namespace nst {
namespace {

using namespace nst::tc;

constexpr int kThreads = 192;
constexpr uint32_t kSlab = 64 * 128;  // one 64-pixel x 64-channel BF16 slab
constexpr uint32_t kSmemMax = 227 * 1024;

// Stages of the box ring: ALOAD (some I tile's channels lie outside the J tile, C = 512) keeps
// room for two A slabs per stage; otherwise A is always read from the B slabs (or the zero slab)
// and a stage is the B slabs alone. Two CTAs per SM (96 KB of stages each) instead of one with
// twice the stages: one's setup and epilogue run under the other's loads. The four launches of
// 756 x 1008: 81 -> 74 us; 1512 x 2016: 172 -> 156 us.
template <int N, bool ALOAD>
struct GramCfg {
  static constexpr uint32_t A_BYTES = ALOAD ? 2 * kSlab : 0u;
  static constexpr uint32_t B_BYTES = (N / 64) * kSlab;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = (int)(96u * 1024u / STAGE_BYTES) > 8 ? 8 : (int)(96u * 1024u / STAGE_BYTES);
  static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + kSlab + 1024;
};
constexpr int kGramMaxStages = 8;
constexpr size_t kGramSmem = 96 * 1024 + kSlab + 1024;
static_assert(GramCfg<64, false>::SMEM <= kGramSmem && GramCfg<128, false>::SMEM <= kGramSmem &&
              GramCfg<256, false>::SMEM <= kGramSmem && GramCfg<256, true>::SMEM <= kGramSmem &&
              GramCfg<64, false>::STAGES <= kGramMaxStages, "Gram kernel shared memory");

// One CTA's work: tile `tile` over run `run` of layer a
template <int N, bool ALOAD>
__device__ __forceinline__ void gram_tc_body(const GramTcArgs &a, int run, int tile) {
  using Cfg = GramCfg<N, ALOAD>;
  constexpr int kStages = Cfg::STAGES;
  constexpr uint32_t A_BYTES = Cfg::A_BYTES;
  constexpr uint32_t B_BYTES = Cfg::B_BYTES;
  constexpr uint32_t STAGE_BYTES = Cfg::STAGE_BYTES;
  constexpr uint32_t ZERO_OFF = kStages * STAGE_BYTES;   // one slab of zeros after the stages
  constexpr uint32_t TMEM_COLS = N;
  // kind::f16, FP32 D, BF16 A/B, both MN-major, M = 128, N
  constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                             ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

  extern __shared__ uint8_t smem_raw[];
  // (shared by the kernel's variants: declared for the most stages)
  __shared__ __align__(8) uint64_t full_bar[kGramMaxStages], empty_bar[kGramMaxStages], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const GramTcChunk ch = a.chunks[run];
  const int I = tile / a.nJ, J = tile % a.nJ;
  const CUtensorMap *map = a.maps + ch.b;
  // A slab s (channels I*128 + 64 s ..) is B slab (I*128 + 64 s - J*N) / 64 when it lies inside
  // the J tile, zeros when it lies past C, else loaded
  int a_src[2];
  bool a_load = false;
#pragma unroll
  for (int sl = 0; sl < 2; sl++) {
    const int c0 = I * 128 + 64 * sl;
    if (c0 >= a.C) a_src[sl] = -2;                                   // zeros
    else if (c0 >= J * N && c0 + 64 <= J * N + N) a_src[sl] = (c0 - J * N) / 64;   // B slab
    else { a_src[sl] = -1; a_load = true; }                          // own A slab
  }
  // (without room for A slabs (ALOAD false) the host has checked that no tile needs them)
  const uint32_t tx_bytes = B_BYTES + (ALOAD && a_load ? A_BYTES : 0u);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; s++) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&done_bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (a_src[0] == -2 || a_src[1] == -2) {   // the zero slab (read by the MMAs only)
    uint8_t *z = smem_raw + (smem_base - smem_u32(smem_raw)) + ZERO_OFF;
    for (int i = threadIdx.x; i < (int)(kSlab / 16); i += kThreads)
      *reinterpret_cast<uint4 *>(z + (size_t)i * 16) = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(&tmem_base_sh), TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  pdl_begin();

  // (the whole warp runs the issue loops, one elected lane issues: see mbar_wait_warp)
  if (warp == 0) {
    int stage = 0;
    uint32_t phase = 1;
    int bx = ch.box0 % ch.nbx, by = ch.box0 / ch.nbx;
    for (int k = ch.box0; k < ch.box1; k++) {
      if (!mbar_wait_warp(smem_u32(&empty_bar[stage]), phase, &abort_flag, a.err)) break;
      if (elect_one()) {
        const uint32_t fb = smem_u32(&full_bar[stage]);
        const uint32_t sa = smem_base + stage * STAGE_BYTES, sb = sa + A_BYTES;
        const int x = bx * a.TW, y = by * a.TH;
        mbar_expect_tx(fb, tx_bytes);
        if (ALOAD && a_load) {
          tma_load_4d(sa, map, fb, I * 128, x, y, 0);
          tma_load_4d(sa + kSlab, map, fb, I * 128 + 64, x, y, 0);
        }
#pragma unroll
        for (int j = 0; j < N / 64; j++) tma_load_4d(sb + j * kSlab, map, fb, J * N + j * 64, x, y, 0);
      }
      __syncwarp();
      if (++bx == ch.nbx) { bx = 0; by++; }
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
  } else if (warp == 1) {
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int k = ch.box0; k < ch.box1; k++) {
      if (!mbar_wait_warp(smem_u32(&full_bar[stage]), phase, &abort_flag, a.err)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (elect_one()) {
        const uint32_t sa = smem_base + stage * STAGE_BYTES, sb = sa + A_BYTES;
        // A's two 64-channel atoms: its own slabs, B slabs, or the zero slab (after every stage,
        // so the atom distance, the descriptor's leading byte offset, stays positive)
        uint32_t a0 = sa, lbo = kSlab;
        if (!a_load) {
          a0 = a_src[0] >= 0 ? sb + (uint32_t)a_src[0] * kSlab : smem_base + ZERO_OFF;
          const uint32_t a1 =
              a_src[1] >= 0 ? sb + (uint32_t)a_src[1] * kSlab : smem_base + ZERO_OFF;
          lbo = a1 - a0;
        }
#pragma unroll
        for (int kk = 0; kk < 4; kk++)   // 16 pixels (two 8-row groups) per MMA
          mma_bf16(tmem_base, sw128_desc_mn(a0 + kk * 2048, lbo),
                   sw128_desc_mn(sb + kk * 2048, kSlab), IDESC,
                   (k > ch.box0 || kk > 0) ? 1u : 0u);
        mma_commit(smem_u32(&empty_bar[stage]));
      }
      __syncwarp();
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
    if (ok && elect_one()) mma_commit(smem_u32(&done_bar));
    __syncwarp();
  } else {
    const int q = warp & 3;
    const int row = q * 32 + lane;   // channel I * 128 + row
    // lane 0 waits (bounded); the warp then proceeds or leaves as one (tcgen05.ld is warp-wide)
    int ready = 0;
    if (lane == 0) ready = mbar_wait(smem_u32(&done_bar), 0, &abort_flag, a.err);
    if (__shfl_sync(0xffffffffu, ready, 0)) {
      tc_fence_after();
      float *out = a.part + (((size_t)run * a.nI * a.nJ + tile) * 128 + row) * N;
      const bool live = I * 128 + row < a.C;
#pragma unroll 1
      for (int c = 0; c < N; c += 32) {
        float v[32];
        tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
        if (live) {
#pragma unroll
          for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<float4 *>(out + c + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// whether tile I * nJ + J holds elements on or above the diagonal
__host__ __device__ inline bool gram_tile_needed(int tile, int nJ, int N) {
  return (tile / nJ) * 128 < (tile % nJ + 1) * N;
}

// The Grams of several layers in one launch (they are independent, and alone none fills the chip to
// its end: 756 x 1008, four launches 74 us, one 59; 64 x 64, 36 us, 10). CTA c of layer l
// takes run c / tiles, the (c % tiles)-th of the tiles that meet the diagonal or lie above it (for
// C = 512 six of the eight).
__global__ void __launch_bounds__(kThreads, 2) gram_tc_kernel(GramTcBatch g) {
  int l = 0;
  while (l + 1 < g.n && (int)blockIdx.x >= g.L[l + 1].cta0) l++;
  const GramTcArgs &a = g.L[l];
  const int c = (int)blockIdx.x - a.cta0, run = c / a.tiles;
  int left = c % a.tiles, tile = 0;
  while (!gram_tile_needed(tile, a.nJ, a.N) || left-- > 0) tile++;
  switch (a.N) {
    case 64: gram_tc_body<64, false>(a, run, tile); break;
    case 128: gram_tc_body<128, false>(a, run, tile); break;
    default:
      if (a.aload)
        gram_tc_body<256, true>(a, run, tile);
      else
        gram_tc_body<256, false>(a, run, tile);
  }
}

// Compensated FP32 addition (Knuth's TwoSum): s + c carries the sum of every added value with
// the rounding error of each addition kept in c, so the pair is as exact as an FP64 sum of the
// FP32 inputs up to O(n u^2) (u = 2^-24) and costs seven FP32 operations, where the FP64 unit of
// this GPU retires a few operations per SM and clock.
__device__ __forceinline__ void two_sum_add(float &s, float &c, float x) {
  const float t = s + x;
  const float z = t - s;
  c += (s - (t - z)) + (x - z);
  s = t;
}

// Gacc[i][j] (+)= sum over runs (fixed order, compensated FP32, then FP64) of the FP32 tile
// partials, all style layers in one launch. A warp takes 128 consecutive elements (a float4 per
// lane and run, coalesced; C^2 is a multiple of 4096 and four consecutive elements stay inside one
// N-wide tile row) and issues the loads of up to 8 of its runs before adding them in run order; a
// layer with many runs splits them over `split` warps of a CTA (warp s: runs s, s + split, ...),
// whose pairs are added in warp order (deterministic). Each element's pair becomes FP64 once.
// Bound: the read of the partials from L2. One launch per layer, with 64-bit index divisions and
// two barriers per 128 elements, took 58 us (64 x 64 pixels) to 83 us (756 x 1008) per evaluation;
// this takes 11 and 51 us (cold, under the profiler).
constexpr int kRedWarps = 16;
__global__ void __launch_bounds__(kRedWarps * 32) gram_tc_reduce_kernel(GramReduceArgs a) {
  __shared__ float2 red[kRedWarps][128];
  int l = 0;
  while (l + 1 < a.n && (int)blockIdx.x >= a.L[l + 1].cta0) l++;
  const GramReduceLayer L = a.L[l];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = warp % L.split, grp = warp / L.split;
  const int e = (((int)blockIdx.x - L.cta0) * (kRedWarps / L.split) + grp) * 128 + lane * 4;
  // G is symmetric, bit for bit (the same products in the same order), and the finaliser reads the
  // 32 x 32 tiles on and above the diagonal only
  const bool live = e < L.C * L.C && e % L.C >= (e / L.C & ~31);
  pdl_begin();
  float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
  if (live) {
    const int i = e / L.C, j = e % L.C;
    const size_t off = ((size_t)((i / 128) * L.nJ + j / L.N) * 128 + (i % 128)) * L.N + (j % L.N);
    const size_t stride = (size_t)L.nI * L.nJ * 128 * L.N;
    for (int r0 = sub; r0 < L.nruns; r0 += 8 * L.split) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; u++)
        if (r0 + L.split * u < L.nruns)
          v[u] = *reinterpret_cast<const float4 *>(L.part + (size_t)(r0 + L.split * u) * stride + off);
#pragma unroll
      for (int u = 0; u < 8; u++)
        if (r0 + L.split * u < L.nruns) {
          two_sum_add(s[0], c[0], v[u].x);
          two_sum_add(s[1], c[1], v[u].y);
          two_sum_add(s[2], c[2], v[u].z);
          two_sum_add(s[3], c[3], v[u].w);
        }
    }
  }
  if (L.split > 1) {
#pragma unroll
    for (int k = 0; k < 4; k++) red[warp][lane * 4 + k] = make_float2(s[k], c[k]);
    __syncthreads();
    if (sub) return;
    for (int w = 1; w < L.split; w++)
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const float2 p = red[warp + w][lane * 4 + k];
        two_sum_add(s[k], c[k], p.x);
        c[k] += p.y;
      }
  }
  if (!live) return;
  double *g = L.Gacc + e;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const double v = (double)s[k] + (double)c[k];
    g[k] = a.overwrite ? v : g[k] + v;
  }
}

// whether some (I, J) tile reads A slabs of its own: an I-tile slab below C that lies outside
// the J tile (the same test the kernel makes per tile)
bool gram_needs_aload(const GramTcArgs &a) {
  for (int I = 0; I < a.nI; I++)
    for (int J = 0; J < a.nJ; J++)
      for (int sl = 0; sl < 2; sl++) {
        const int c0 = I * 128 + 64 * sl;
        if (c0 < a.C && !(c0 >= J * a.N && c0 + 64 <= J * a.N + a.N)) return true;
      }
  return false;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

void gram_tc_shape(int C, int *N, int *nI, int *nJ) {
  *N = C >= 256 ? 256 : C;
  *nI = C <= 128 ? 1 : C / 128;
  *nJ = C / *N;
}

void gram_tc_patch(int own_h, int own_w, int *TH, int *TW) {
  static const int cand[5][2] = {{1, 64}, {2, 32}, {4, 16}, {8, 8}, {16, 4}};
  long long best = -1;
  for (auto &c : cand) {
    const long long area = (long long)((own_h + c[0] - 1) / c[0]) * c[0] *
                           ((own_w + c[1] - 1) / c[1]) * c[1];
    if (best < 0 || area < best) { best = area; *TH = c[0]; *TW = c[1]; }
  }
}

cudaError_t encode_gram_map(CUtensorMap *m, const void *base, int C, int own_w, int own_h,
                            long long row_stride_px, int TH, int TW) {
  EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(tc_encode_tiled_fn());
  if (!enc) return cudaErrorNotSupported;
  cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)std::max(own_w, 1),
                        (cuuint64_t)std::max(own_h, 1), 1};
  cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)row_stride_px * C * 2,
                           (cuuint64_t)row_stride_px * C * 2 * std::max(own_h, 1)};
  cuuint32_t box[4] = {64, (cuuint32_t)TW, (cuuint32_t)TH, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims,
                   strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_gram_tc(GramTcBatch g, cudaStream_t s) {
  int ctas = 0;
  for (int l = 0; l < g.n; l++) {
    GramTcArgs &a = g.L[l];
    if (a.N != 64 && a.N != 128 && a.N != 256) return cudaErrorInvalidValue;
    a.aload = gram_needs_aload(a) ? 1 : 0;
    if (a.aload && a.N != 256) return cudaErrorInvalidValue;
    a.cta0 = ctas;
    a.tiles = 0;
    for (int t = 0; t < a.nI * a.nJ; t++) a.tiles += gram_tile_needed(t, a.nJ, a.N) ? 1 : 0;
    ctas += a.nruns * a.tiles;
  }
  if (ctas <= 0) return cudaSuccess;
  constexpr size_t smem = kGramSmem;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(gram_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  return launch_pdl(true, gram_tc_kernel, ctas, kThreads, smem, s, g);
}

cudaError_t launch_gram_tc_reduce(GramReduceArgs a, cudaStream_t s) {
  int ctas = 0;
  for (int l = 0; l < a.n; l++) {
    GramReduceLayer &L = a.L[l];
    // about eight runs per warp: one batch of loads
    L.split = L.nruns <= 8 ? 1 : L.nruns <= 16 ? 2 : L.nruns <= 32 ? 4 : L.nruns <= 64 ? 8 : 16;
    L.cta0 = ctas;
    const int per = 128 * (kRedWarps / L.split);
    ctas += (L.C * L.C + per - 1) / per;
  }
  if (ctas <= 0) return cudaSuccess;
  return launch_pdl(true, gram_tc_reduce_kernel, ctas, kRedWarps * 32, 0, s, a);
}

}  // namespace nst
