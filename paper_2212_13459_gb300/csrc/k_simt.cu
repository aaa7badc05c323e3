// k_simt.cu -- CUDA-core kernels of the localized loss/gradient path:
//   * the plain FP32 convolution engine (implicit GEMM on CUDA cores, no TF32), used by the FP32
//     form of the path and as a cross-check of the tensor-core engine;
//   * conv1_1 forward straight from the caller's planar image (block gather fused) and conv1_1
//     input-gradient with the inner-part scatter into dE/dx fused (Algorithm 1, last step);
//   * 2x2 max pooling and its adjoint (argmax routing + ReLU gate);
//   * split Gram partial sums over owned pixels and their FP64 reduction (Eq. 4, Algorithm 1
//     Step 1), the style finalisation (Eq. 3 and Table 1 row 2), the content loss over owned
//     pixels (Algorithm 1 Step 2), the content-target crop, and a finiteness check.
#include <cfloat>

#include "nst_internal.cuh"
#include "nst_kernels.h"

namespace nst {

// ---- vector helpers ----------------------------------------------------------------------------
__device__ __forceinline__ void load4(const float *p, float v[4]) {
  float4 t = *reinterpret_cast<const float4 *>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16 *p, float v[4]) {
  uint2 t = *reinterpret_cast<const uint2 *>(p);
  __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&t.x);
  __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162 *>(&t.y);
  float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
  v[0] = fa.x; v[1] = fa.y; v[2] = fb.x; v[3] = fb.y;
}
__device__ __forceinline__ void store4(float *p, const float v[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(__nv_bfloat16 *p, const float v[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
  __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
  uint2 t;
  t.x = *reinterpret_cast<unsigned *>(&a);
  t.y = *reinterpret_cast<unsigned *>(&b);
  *reinterpret_cast<uint2 *>(p) = t;
}
__device__ __forceinline__ void load8(const float *p, float v[8]) { load4(p, v); load4(p + 4, v + 4); }
__device__ __forceinline__ void load8(const __nv_bfloat16 *p, float v[8]) {
  uint4 t = *reinterpret_cast<const uint4 *>(p);
  const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&t);
#pragma unroll
  for (int i = 0; i < 4; i++) {
    float2 f = __bfloat1622float2(h[i]);
    v[2 * i] = f.x;
    v[2 * i + 1] = f.y;
  }
}
__device__ __forceinline__ void store8(float *p, const float v[8]) { store4(p, v); store4(p + 4, v + 4); }
__device__ __forceinline__ void store8(__nv_bfloat16 *p, const float v[8]) {
  uint4 t;
  __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&t);
#pragma unroll
  for (int i = 0; i < 4; i++) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
  *reinterpret_cast<uint4 *>(p) = t;
}

// ---- shared epilogue (4 consecutive output channels of one pixel) ------------------------------
template <typename T>
__device__ __forceinline__ void conv_epilogue4(const ConvArgs &a, int b, int y, int x, int n,
                                               float v[4]) {
  const BlockGeom g = a.geom[b];
  const bool valid = y < (g.eh >> a.level) && x < (g.ew >> a.level);
  const size_t o = (((size_t)b * a.Hb + y) * a.Wb + x) * a.cout + n;
  if (a.mode == kEpiForward) {
#pragma unroll
    for (int j = 0; j < 4; j++) v[j] = valid ? fmaxf(v[j] + a.bias[n + j], 0.f) : 0.f;
  } else {
    if (a.cact && valid) {
      const int gy = (g.ey0 >> a.level) + y, gx = (g.ex0 >> a.level) + x;
      if (gy < a.Hc && gx < a.Wc) {
        float ca[4], ct[4];
        load4(reinterpret_cast<const T *>(a.cact) + o, ca);
        load4(reinterpret_cast<const T *>(a.ctgt) + ((size_t)gy * a.Wc + gx) * a.cout + n, ct);
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] += a.two_lambda * (ca[j] - ct[j]);
      }
    }
    if (a.addvec && valid) {
#pragma unroll
      for (int j = 0; j < 4; j++) v[j] += a.addvec[n + j];
    }
    if (a.mask) {
      float m[4];
      load4(reinterpret_cast<const T *>(a.mask) + o, m);
#pragma unroll
      for (int j = 0; j < 4; j++) v[j] = m[j] > 0.f ? v[j] : 0.f;
    }
    if (!valid) v[0] = v[1] = v[2] = v[3] = 0.f;
  }
  store4(reinterpret_cast<T *>(a.out) + o, v);
}

// ---- CUDA-core implicit-GEMM convolution ---------------------------------------------------------
// CTA tile: BM output pixels x BN output channels, TM x TN per thread; K slices of BK channels of
// one tap, double-buffered in shared memory, the next slice in flight to registers while one is
// multiplied (one barrier per slice). Every output is one chain of FP32 FMAs in tap, channel, then
// phase-2 order whatever the tile, so all tiles give the same bits.
//
// Bound: the FP32 FMA pipe (128 lanes per SM and clock) and, close behind, the shared-memory
// reads: a 16-byte read returns 512 bytes to a warp's registers at 128 bytes per clock, broadcast
// or not, so one K step of a warp costs TM + TN clocks of reads against TM TN / 4 of FMAs: 8 : 4 at
// 4 x 4 per thread, 16 : 16 at 8 x 8, 24 : 32 at 8 x 16. The FMAs are packed pairs (fma.rn.f32x2:
// two IEEE FMAs per lane, adjacent channels of one pixel), which frees the issue slots for the
// rest. Pixels are a run of a rectangle in row-major order (the launch's tile list, or the flat
// buffer), so only a rectangle's last tile is partly idle. Measured against the 8 x 8 pixel x 64
// channel tile with 4 x 4 per thread it replaced: 64 -> 64 channels at 16 x 368 x 368: 4,330 ->
// 3,040 us; 256 -> 256 with a phase 2 of 256 at 16 x 92 x 92: 5,150 -> 3,080 us (58 TFLOP/s);
// 512 -> 512 at 94 x 126: 1,675 -> 1,055 us; at 4 x 4 pixels: 199 -> 78 us.
//
// Slice layout: As[k][px ^ SW (k/4 % Q)], Bs[k][ch ^ SW (k/4 % Q)], Q = BK / 4 channel quads,
// SW = 32 / Q. 32 / Q pixels x Q quads make one warp's load instruction (4 BK contiguous bytes per
// pixel); the XOR puts the quads of the transposing stores on different banks, and leaves
// 4-element groups whole for the 16-byte reads. It moves elements within groups of 32, so BM and
// BN are multiples of 32.
__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a,
                                     unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}

template <typename T, int BM, int BN, int TM, int TN, int BK, int MINB>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), MINB) conv_simt_kernel(ConvArgs a) {
  constexpr int NT = (BM / TM) * (BN / TN);           // threads
  constexpr int Q = BK / 4, SW = 32 / Q;              // channel quads of a slice, swizzle step
  constexpr int LA = BM * Q / NT, LB = BN * Q / NT;   // quads each thread loads per slice
  // a warp covers (8 TM) pixels x (4 TN) channels; a thread's pixels and channels come in groups
  // of 4, 32 pixels / 16 channels apart
  constexpr int WN = BN / (4 * TN);                   // warps along the channels
  constexpr int PG = TM < 4 ? TM : 4;                 // pixels per group
  constexpr int GM = TM / PG, GN = TN / 4;
  static_assert(LA * NT == BM * Q && LB * NT == BN * Q && BM % (8 * TM) == 0 &&
                BN % (4 * TN) == 0 && BM % 32 == 0 && BN % 32 == 0 && 32 % Q == 0,
                "convolution tile");
  __shared__ __align__(16) float As[2][BK][BM];
  __shared__ __align__(16) float Bs[2][BK][BN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.y * BN;
  // this CTA's run of pixels: entry {block, first pixel, y0 << 16 | x0, height << 16 | width} of
  // the tile list, or pixels blockIdx.x BM .. of the whole buffer
  int rb = 0, q0 = blockIdx.x * BM, ry = 0, rx = 0, rh = a.B * a.Hb, rw = a.Wb;
  if (a.tiles) {
    const int4 e = a.tiles[blockIdx.x];
    rb = e.x;
    q0 = e.y;
    ry = (int)((unsigned)e.z >> 16);
    rx = e.z & 0xffff;
    rh = (int)((unsigned)e.w >> 16);
    rw = e.w & 0xffff;
  }
  const int rn = rh * rw;
  // pixel p of the run -> (block, y, x); false past the rectangle. (Without a list the rectangle
  // is all B blocks' rows, Hb per block.)
  auto pixel = [&](int p, int &b, int &y, int &x) -> bool {
    const int q = q0 + p;
    if (q >= rn) return false;
    y = q / rw;
    x = rx + q - y * rw;
    y += ry;
    b = rb;
    if (!a.tiles) {
      b = y / a.Hb;
      y -= b * a.Hb;
    }
    return true;
  };
  const int lc = (tid % Q) * 4;   // first channel of the quads this thread loads
  int ly[LA], lx[LA], lo[LA];     // their pixels
#pragma unroll
  for (int i = 0; i < LA; i++) {
    int b = 0, y = 0, x = 0;
    const bool in = pixel(tid / Q + i * (NT / Q), b, y, x);
    ly[i] = in ? y : -4;   // out of the buffer under every tap
    lx[i] = x;
    lo[i] = (b * a.Hb + y) * a.Wb + x;
  }
  const T *A = reinterpret_cast<const T *>(a.A), *A2 = reinterpret_cast<const T *>(a.A2);
  const T *Wt = reinterpret_cast<const T *>(a.Wt), *W2 = reinterpret_cast<const T *>(a.W2);
  const int n_main = a.taps * (a.cin / BK), n_slices = n_main + a.k2 / BK;

  float va[LA][4], vb[LB][4];   // the slice in flight
  // slices are loaded in order: the main phase tap by tap, channels ascending, then phase 2
  int ls = 0, tap = 0, c = lc, dy = -1, dx = -1;
  const T *wrow = Wt + (size_t)(n0 + tid / Q) * a.taps * a.cin;
  auto load = [&]() {
    if (ls < n_main) {
#pragma unroll
      for (int i = 0; i < LA; i++) {
        const int y = ly[i] + dy, x = lx[i] + dx;
        if (y >= 0 && y < a.Hb && x >= 0 && x < a.Wb)
          load4(A + (size_t)(lo[i] + dy * a.Wb + dx) * a.cin + c, va[i]);
        else
          va[i][0] = va[i][1] = va[i][2] = va[i][3] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < LB; i++)
        load4(wrow + (size_t)(i * (NT / Q) * a.taps + tap) * a.cin + c, vb[i]);
      c += BK;
      if (c >= a.cin) {
        c = lc;
        tap++;
        if (++dx == 2) { dx = -1; dy++; }
      }
    } else {
      const int c2 = (ls - n_main) * BK + lc;
#pragma unroll
      for (int i = 0; i < LA; i++) {
        if (ly[i] >= 0)
          load4(A2 + (size_t)lo[i] * a.k2 + c2, va[i]);
        else
          va[i][0] = va[i][1] = va[i][2] = va[i][3] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < LB; i++)
        load4(W2 + (size_t)(n0 + tid / Q + i * (NT / Q)) * a.k2 + c2, vb[i]);
    }
    ls++;
  };
  const int sw = (tid % Q) * SW;   // the swizzle of this thread's quads
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < LA; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) As[buf][lc + j][(tid / Q + i * (NT / Q)) ^ sw] = va[i][j];
#pragma unroll
    for (int i = 0; i < LB; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) Bs[buf][lc + j][(tid / Q + i * (NT / Q)) ^ sw] = vb[i][j];
  };

  const int p0 = (warp / WN) * 8 * TM + (lane >> 2) * PG;   // this thread's first pixel / channel
  const int c0 = (warp % WN) * 4 * TN + (lane & 3) * 4;
  unsigned long long acc[TM][TN / 2];   // [pixel][channel pair]
#pragma unroll
  for (int i = 0; i < TM; i++)
#pragma unroll
    for (int j = 0; j < TN / 2; j++) acc[i][j] = 0ull;

  load();
  store(0);
  if (n_slices > 1) load();
  __syncthreads();
  for (int s = 0; s < n_slices; s++) {
    const int buf = s & 1;
#pragma unroll
    for (int k = 0; k < BK; k++) {
      const int x = ((k >> 2) % Q) * SW;
      float ar[TM];
      ulonglong2 bv[GN];
#pragma unroll
      for (int g = 0; g < GM; g++) {
        const float *p = &As[buf][k][(p0 + 8 * PG * g) ^ x];
        if constexpr (PG == 4) {
          const float4 t = *reinterpret_cast<const float4 *>(p);
          ar[4 * g] = t.x; ar[4 * g + 1] = t.y; ar[4 * g + 2] = t.z; ar[4 * g + 3] = t.w;
        } else {
          const float2 t = *reinterpret_cast<const float2 *>(p);
          ar[2 * g] = t.x; ar[2 * g + 1] = t.y;
        }
      }
#pragma unroll
      for (int g = 0; g < GN; g++)
        bv[g] = *reinterpret_cast<const ulonglong2 *>(&Bs[buf][k][(c0 + 16 * g) ^ x]);
#pragma unroll
      for (int i = 0; i < TM; i++) {
        const unsigned long long ad = dup2(ar[i]);
#pragma unroll
        for (int j = 0; j < GN; j++) {
          fma2(acc[i][2 * j], ad, bv[j].x);
          fma2(acc[i][2 * j + 1], ad, bv[j].y);
        }
      }
    }
    if (s + 1 < n_slices) {
      store(buf ^ 1);
      if (s + 2 < n_slices) load();
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM; i++) {
    int b, y, x;
    if (!pixel(p0 + (i / PG) * 8 * PG + i % PG, b, y, x)) continue;
#pragma unroll
    for (int g = 0; g < GN; g++) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const unsigned long long t = acc[i][2 * g + (j >> 1)];
        v[j] = __uint_as_float((unsigned)((j & 1) ? t >> 32 : t));
      }
      conv_epilogue4<T>(a, b, y, x, n0 + c0 + 16 * g, v);
    }
  }
}

template <typename T, int BM, int BN, int TM, int TN, int BK, int MINB>
static void launch_simt_tile(const ConvArgs &a, cudaStream_t s) {
  const long long px = (long long)a.B * a.Hb * a.Wb;
  const int nt = a.tiles ? a.n_mtiles : (int)((px + BM - 1) / BM);
  if (nt <= 0) return;
  conv_simt_kernel<T, BM, BN, TM, TN, BK, MINB>
      <<<dim3(nt, a.cout / BN), (BM / TM) * (BN / TN), 0, s>>>(a);
}

// Tile of a launch over px pixels. Large launches take the tile with the fewest shared-memory
// reads per FMA; the smaller ones trade that for CTAs (152 SMs). Times in us, start of the line =
// the launch (pixels, channels in -> out):
//                          128x128  64x64   64x64   32x32   32x32
//                          8x16     8x8     4x8     4x4     2x4
//   33,856  512 -> 512     2,771    2,900   3,326   4,184   6,303
//    9,248  256 -> 256     266      246     273     343     512
//   18,786  128 -> 64      -        72      68      86      121
//    4,096  128 -> 128     124      68      41      45      64
//    3,960  64 -> 64       -        43      26      19      21
//      884  512 -> 256     464      242     148     101     125
//       16  512 -> 512     457      238     142     84      78
// Between the first two the number of waves decides (304 and 608 CTAs run at once; the second has
// a quarter of the first's work each, at 0.955 of its rate).
SimtTile conv_simt_tile(long long px, int cin, int cout, int k2) {
  if (cin % 32 || k2 % 32) return kSimt64x64k16;
  const long long n64 = (px + 63) / 64 * (cout / 64), n32 = (px + 31) / 32 * (cout / 32);
  if (n32 <= 152) return kSimt32x32t2;
  if (n64 < 100) return kSimt32x32;
  if (n64 <= 304) return kSimt64x64t4;
  if (cout % 128 == 0) {
    const double w128 = (double)((px + 127) / 128 * (cout / 128)) / 304, w64 = (double)n64 / 608;
    const double c128 = w128 <= 1 ? 1.0 : w128 + 0.3, c64 = w64 <= 1 ? 1.0 : w64 + 0.3;
    if (c128 <= 0.524 * c64) return kSimt128x128;
  }
  return kSimt64x64;
}
int conv_simt_tile_px(SimtTile t) {
  return t == kSimt128x128 ? 128 : t == kSimt32x32 || t == kSimt32x32t2 ? 32 : 64;
}

template <typename T>
void launch_conv_simt(const ConvArgs &a, cudaStream_t s) {
  const long long px = (long long)a.B * a.Hb * a.Wb;
  // (with a tile list: the tile it was cut for)
  switch (a.tiles ? (SimtTile)a.TW : conv_simt_tile(px, a.taps ? a.cin : 0, a.cout, a.k2)) {
    case kSimt128x128: launch_simt_tile<T, 128, 128, 8, 16, 16, 2>(a, s); break;
    case kSimt64x64: launch_simt_tile<T, 64, 64, 8, 8, 32, 4>(a, s); break;
    case kSimt64x64t4: launch_simt_tile<T, 64, 64, 4, 8, 32, 2>(a, s); break;
    case kSimt32x32: launch_simt_tile<T, 32, 32, 4, 4, 32, 4>(a, s); break;
    case kSimt32x32t2: launch_simt_tile<T, 32, 32, 2, 4, 32, 2>(a, s); break;
    case kSimt64x64k16: launch_simt_tile<T, 64, 64, 8, 8, 16, 6>(a, s); break;
  }
}
template void launch_conv_simt<float>(const ConvArgs &, cudaStream_t);
template void launch_conv_simt<__nv_bfloat16>(const ConvArgs &, cudaStream_t);

// ---- conv1_1 forward from the planar image (block extraction fused) ----------------------------
// out[b][y][x][c] = relu(b1[c] + sum W1[c][ci][ky][kx] * blk(ci, y+ky-1, x+kx-1)), where blk is the
// block's extended rectangle of x and reads zero outside it (the block is a standalone image).
// One thread computes all 64 channels of one pixel. The 27 x 64 weights travel as a
// __grid_constant__ kernel parameter: with the loops unrolled, every FMA takes its weight
// straight from the constant bank, so no load instruction competes with the FMAs. In the BF16 form
// each image value enters as hi + lo (hi = bf16(x), lo = bf16(x - hi)), the representation the
// tensor-core conv1_1 multiplies, so both engines see the same input.
template <typename T>
__global__ void __launch_bounds__(128) conv11_fwd_kernel(const float *__restrict__ img, int H,
                                                         int W, const __grid_constant__ Conv11W cw,
                                                         const BlockGeom *__restrict__ geom,
                                                         int B, int Hb, int Wb, T *__restrict__ out) {
  const long long npix = (long long)B * Hb * Wb;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < npix;
       p += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(p % Wb);
    const int y = (int)((p / Wb) % Hb);
    const int b = (int)(p / ((long long)Wb * Hb));
    const BlockGeom g = geom[b];
    float acc[64];
    if (y < g.eh && x < g.ew) {
      float in[27];
#pragma unroll
      for (int ci = 0; ci < 3; ci++)
#pragma unroll
        for (int ky = 0; ky < 3; ky++)
#pragma unroll
          for (int kx = 0; kx < 3; kx++) {
            const int yy = y + ky - 1, xx = x + kx - 1;
            const bool ok = yy >= 0 && yy < g.eh && xx >= 0 && xx < g.ew;
            float v = ok ? __ldg(img + ((size_t)ci * H + g.ey0 + yy) * W + g.ex0 + xx) : 0.f;
            if (sizeof(T) == 2) {   // the BF16 form reads the image as a BF16 pair hi + lo
              const float hi = __bfloat162float(__float2bfloat16_rn(v));
              v = hi + __bfloat162float(__float2bfloat16_rn(v - hi));
            }
            in[ci * 9 + ky * 3 + kx] = v;
          }
#pragma unroll
      for (int c = 0; c < 64; c++) acc[c] = cw.b[c];
#pragma unroll
      for (int k = 0; k < 27; k++) {
        const float v = in[k];
#pragma unroll
        for (int c = 0; c < 64; c++) acc[c] = fmaf(cw.w[k][c], v, acc[c]);
      }
#pragma unroll
      for (int c = 0; c < 64; c++) acc[c] = fmaxf(acc[c], 0.f);
    } else {
#pragma unroll
      for (int c = 0; c < 64; c++) acc[c] = 0.f;
    }
    T *o = out + (size_t)p * 64;
#pragma unroll
    for (int c8 = 0; c8 < 8; c8++) store8(o + c8 * 8, acc + c8 * 8);
  }
}

template <typename T>
void launch_conv11_fwd(const float *img, int H, int W, const Conv11W &cw, const BlockGeom *geom,
                       int B, int Hb, int Wb, T *out, cudaStream_t s) {
  long long npix = (long long)B * Hb * Wb;
  long long blocks = (npix + 127) / 128;
  int grid = (int)(blocks < 152 * 32 ? blocks : 152 * 32);
  conv11_fwd_kernel<T><<<grid, 128, 0, s>>>(img, H, W, cw, geom, B, Hb, Wb, out);
}
template void launch_conv11_fwd<float>(const float *, int, int, const Conv11W &,
                                       const BlockGeom *, int, int, int, float *, cudaStream_t);
template void launch_conv11_fwd<__nv_bfloat16>(const float *, int, int, const Conv11W &,
                                               const BlockGeom *, int, int, int,
                                               __nv_bfloat16 *, cudaStream_t);

// ---- conv1_1 input gradient + scatter of the inner part into dE/dx --------------------------------
// dx[ci](y,x) = sum_{co,ky,kx} W1[co][ci][ky][kx] * g[y-ky+1][x-kx+1][co] for the owned (inner)
// pixels of each block, written to grad at image coordinates (Algorithm 1, last line).
template <typename T>
__global__ void __launch_bounds__(256) conv11_dgrad_scatter_kernel(
    const T *__restrict__ g, const float *__restrict__ w11, const BlockGeom *__restrict__ geom,
    const OwnRect *__restrict__ inner, int B, int Hb, int Wb, float *__restrict__ grad, int H,
    int W) {
  // Eight lanes per pixel, lane group cg holding channels 8cg..8cg+7: a warp reads four pixels'
  // 128-byte channel vectors as 512 contiguous bytes. ws[k][cg][j] = {W1[co][0][k], W1[co][1][k],
  // W1[co][2][k], 0} with co = 8cg + j, rows padded to 9 float4 so the 8 groups hit distinct banks.
  __shared__ __align__(16) float4 ws[9][8][9];
  for (int i = threadIdx.x; i < 9 * 64; i += blockDim.x) {
    const int k = i / 64, co = i % 64;
    ws[k][co / 8][co % 8] =
        make_float4(w11[co * 27 + k], w11[co * 27 + 9 + k], w11[co * 27 + 18 + k], 0.f);
  }
  __syncthreads();
  const int b = blockIdx.y;
  if (b >= B) return;
  const OwnRect r = inner[b];
  const BlockGeom gm = geom[b];
  const int rw = r.x1 - r.x0, rh = r.y1 - r.y0;
  const long long n = (long long)rw * rh;
  const int cg = threadIdx.x & 7;
  const long long stride = (long long)gridDim.x * (blockDim.x >> 3);
  // every lane of a warp runs the same number of iterations (the bound is per 4-pixel group)
  for (long long q0 = (long long)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 5) * 4;
       q0 < n; q0 += stride) {
    const long long q = q0 + ((threadIdx.x & 31) >> 3);
    const bool live = q < n;
    const int y = live ? r.y0 + (int)(q / rw) : r.y0, x = live ? r.x0 + (int)(q % rw) : r.x0;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f;
#pragma unroll 3
    for (int k = 0; k < 9; k++) {
      const int yy = y - k / 3 + 1, xx = x - k % 3 + 1;
      if (live && yy >= 0 && yy < Hb && xx >= 0 && xx < Wb) {
        float gv[8];
        load8(g + (((size_t)b * Hb + yy) * Wb + xx) * 64 + cg * 8, gv);
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const float4 w = ws[k][cg][j];
          d0 = fmaf(w.x, gv[j], d0);
          d1 = fmaf(w.y, gv[j], d1);
          d2 = fmaf(w.z, gv[j], d2);
        }
      }
    }
#pragma unroll
    for (int m = 1; m < 8; m <<= 1) {
      d0 += __shfl_xor_sync(0xffffffffu, d0, m);
      d1 += __shfl_xor_sync(0xffffffffu, d1, m);
      d2 += __shfl_xor_sync(0xffffffffu, d2, m);
    }
    if (live && cg == 0) {
      const size_t o = (size_t)(gm.ey0 + y) * W + gm.ex0 + x;
      grad[o] = d0;
      grad[(size_t)H * W + o] = d1;
      grad[2 * (size_t)H * W + o] = d2;
    }
  }
}

template <typename T>
void launch_conv11_dgrad_scatter(const T *g, const float *w11, const BlockGeom *geom,
                                 const OwnRect *inner, int B, int Hb, int Wb, float *grad, int H,
                                 int W, int max_inner_px, cudaStream_t s) {
  int gx = (max_inner_px + 31) / 32;   // 32 pixels per 256-thread CTA pass
  if (gx > 2048) gx = 2048;
  if (gx < 1) gx = 1;
  dim3 grid(gx, B);
  conv11_dgrad_scatter_kernel<T><<<grid, 256, 0, s>>>(g, w11, geom, inner, B, Hb, Wb, grad, H, W);
}
template void launch_conv11_dgrad_scatter<float>(const float *, const float *, const BlockGeom *,
                                                 const OwnRect *, int, int, int, float *, int, int,
                                                 int, cudaStream_t);
template void launch_conv11_dgrad_scatter<__nv_bfloat16>(const __nv_bfloat16 *, const float *,
                                                         const BlockGeom *, const OwnRect *, int,
                                                         int, int, float *, int, int, int,
                                                         cudaStream_t);

// ---- 2x2 max pool (floor) and its adjoint ----------------------------------------------------------
// The window's first maximum in row-major order (strict '>') is the argmax, as in the oracle.
__device__ __forceinline__ int argmax4(float v0, float v1, float v2, float v3) {
  int k = 0;
  float m = v0;
  if (v1 > m) { m = v1; k = 1; }
  if (v2 > m) { m = v2; k = 2; }
  if (v3 > m) { k = 3; }
  return k;
}

// in: [B][2Hp][2Wp][C] at level l; out: [B][Hp][Wp][C] at level l+1; zero outside valid region
template <typename T>
__global__ void pool_kernel(const T *__restrict__ in, T *__restrict__ out, int B, int Hp, int Wp,
                            int C, const BlockGeom *__restrict__ geom, int level_out) {
  const int C8 = C / 8;
  const long long n = (long long)B * Hp * Wp * C8;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    long long p = i / C8;
    const int x = (int)(p % Wp);
    const int y = (int)((p / Wp) % Hp);
    const int b = (int)(p / ((long long)Wp * Hp));
    const BlockGeom g = geom[b];
    float o[8];
    if (y < (g.eh >> level_out) && x < (g.ew >> level_out)) {
      const int Wi = 2 * Wp;
      const T *base = in + (((size_t)b * 2 * Hp + 2 * y) * Wi + 2 * x) * C + c;
      float v0[8], v1[8], v2[8], v3[8];
      load8(base, v0);
      load8(base + C, v1);
      load8(base + (size_t)Wi * C, v2);
      load8(base + (size_t)Wi * C + C, v3);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int k = argmax4(v0[j], v1[j], v2[j], v3[j]);
        o[j] = k == 0 ? v0[j] : k == 1 ? v1[j] : k == 2 ? v2[j] : v3[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; j++) o[j] = 0.f;
    }
    store8(out + (size_t)p * C + c, o);
  }
}

// gp: [B][Hp][Wp][C] gradient w.r.t. the pooled map; act: [B][2Hp][2Wp][C] post-ReLU activation;
// g:  [B][2Hp][2Wp][C] gradient w.r.t. the pre-activation = routed gp gated by act > 0
template <typename T>
__global__ void unpool_kernel(const T *__restrict__ gp, const T *__restrict__ act,
                              T *__restrict__ g, int B, int Hp, int Wp, int C,
                              const BlockGeom *__restrict__ geom, int level_out) {
  const int C8 = C / 8;
  const long long n = (long long)B * Hp * Wp * C8;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    long long p = i / C8;
    const int x = (int)(p % Wp);
    const int y = (int)((p / Wp) % Hp);
    const int b = (int)(p / ((long long)Wp * Hp));
    const BlockGeom gm = geom[b];
    const int Wi = 2 * Wp;
    const size_t o0 = (((size_t)b * 2 * Hp + 2 * y) * Wi + 2 * x) * C + c;
    const size_t offs[4] = {o0, o0 + C, o0 + (size_t)Wi * C, o0 + (size_t)Wi * C + C};
    float r[4][8];
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int j = 0; j < 8; j++) r[k][j] = 0.f;
    if (y < (gm.eh >> level_out) && x < (gm.ew >> level_out)) {
      float gv[8], v[4][8];
      load8(gp + (size_t)p * C + c, gv);
#pragma unroll
      for (int k = 0; k < 4; k++) load8(act + offs[k], v[k]);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int k = argmax4(v[0][j], v[1][j], v[2][j], v[3][j]);
        const float av = k == 0 ? v[0][j] : k == 1 ? v[1][j] : k == 2 ? v[2][j] : v[3][j];
        const float val = av > 0.f ? gv[j] : 0.f;
        r[0][j] = k == 0 ? val : 0.f;
        r[1][j] = k == 1 ? val : 0.f;
        r[2][j] = k == 2 ? val : 0.f;
        r[3][j] = k == 3 ? val : 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) store8(g + offs[k], r[k]);
  }
}

// Tensor-core form of the same routing: the forward's fused pooling stored 4 bits per pooled
// value, bit q set where window pixel q (row-major) equals the window max and that max is
// positive; the gradient goes to the lowest set bit (the first maximum), none where no bit is
// set (the ReLU gate is shut). One 32-bit word per 8 channels c .. c+7 at byte (p C + c) / 2,
// channel c+k in the nibble at bit 8 (k & 3) + 4 (k >> 2). The backward reads half a byte per
// value instead of the four activations.
// rects (optional): per block, the pooled rectangle {y0, y1, x0, x1} to route (the rest of the
// block's full-resolution gradient is left as it is); grid (n, B), row b = block b. Without
// rects: every pooled position of the buffer, grid-stride over all blocks.
__global__ void unpool_idx_kernel(const __nv_bfloat16 *gp, const unsigned char *idx,
                                  __nv_bfloat16 *g, int B, int Hp, int Wp, int C,
                                  const BlockGeom *__restrict__ geom, int level_out,
                                  const int4 *__restrict__ rects) {
  pdl_begin();
  const int C8 = C / 8;
  int4 r = make_int4(0, Hp, 0, Wp);
  long long n = (long long)B * Hp * Wp * C8;
  long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (rects) {
    r = rects[blockIdx.y];
    n = (long long)max(0, r.y - r.x) * max(0, r.w - r.z) * C8;
  }
  const int rw = r.w - r.z;
  for (long long i = i0; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    const long long q = i / C8;
    int x, y, b;
    if (rects) {
      x = r.z + (int)(q % rw);
      y = r.x + (int)(q / rw);
      b = blockIdx.y;
    } else {
      x = (int)(q % Wp);
      y = (int)((q / Wp) % Hp);
      b = (int)(q / ((long long)Wp * Hp));
    }
    const long long p = ((long long)b * Hp + y) * Wp + x;
    const BlockGeom gm = geom[b];
    const int Wi = 2 * Wp;
    const size_t o0 = (((size_t)b * 2 * Hp + 2 * y) * Wi + 2 * x) * C + c;
    const size_t offs[4] = {o0, o0 + C, o0 + (size_t)Wi * C, o0 + (size_t)Wi * C + C};
    float rv[4][8];
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int j = 0; j < 8; j++) rv[k][j] = 0.f;
    if (y < (gm.eh >> level_out) && x < (gm.ew >> level_out)) {
      float gv[8];
      load8(gp + (size_t)p * C + c, gv);
      const uint32_t w = *reinterpret_cast<const uint32_t *>(idx + ((size_t)p * C + c) / 2);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const uint32_t nib = (w >> (8 * (j & 3) + 4 * (j >> 2))) & 0xfu;
        const uint32_t first = nib & (0u - nib);   // lowest set bit, 0 if none
#pragma unroll
        for (int qq = 0; qq < 4; qq++) rv[qq][j] = first == (1u << qq) ? gv[j] : 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) store8(g + offs[k], rv[k]);
  }
}

static int ew_grid(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

template <typename T>
void launch_pool(const T *in, T *out, int B, int Hp, int Wp, int C, const BlockGeom *geom,
                 int level_out, cudaStream_t s) {
  pool_kernel<T><<<ew_grid((long long)B * Hp * Wp * C / 8), 256, 0, s>>>(in, out, B, Hp, Wp, C,
                                                                          geom, level_out);
}
template <typename T>
void launch_unpool(const T *gp, const T *act, T *g, int B, int Hp, int Wp, int C,
                   const BlockGeom *geom, int level_out, cudaStream_t s) {
  unpool_kernel<T><<<ew_grid((long long)B * Hp * Wp * C / 8), 256, 0, s>>>(gp, act, g, B, Hp, Wp,
                                                                            C, geom, level_out);
}
void launch_unpool_idx(const __nv_bfloat16 *gp, const unsigned char *idx, __nv_bfloat16 *g,
                       int B, int Hp, int Wp, int C, const BlockGeom *geom, int level_out,
                       const int4 *rects, int max_rect_px, cudaStream_t s) {
  if (rects) {
    if (max_rect_px <= 0) return;
    const long long per = (long long)max_rect_px * C / 8;
    int nx = (int)std::min<long long>((per + 255) / 256, std::max(1, 152 * 32 / B));
    dim3 grid(nx, B);
    // (per 8 channels of a pooled pixel: 20 bytes in, 64 out)
    launch_pdl(traffic_us(84.0 * per * B) <= kEarlyUs, unpool_idx_kernel, grid, 256, 0, s, gp, idx,
               g, B, Hp, Wp, C, geom, level_out, rects);
    return;
  }
  launch_pdl(true, unpool_idx_kernel, ew_grid((long long)B * Hp * Wp * C / 8), 256, 0, s, gp, idx,
             g, B, Hp, Wp, C, geom, level_out, (const int4 *)nullptr);
}
template void launch_pool<float>(const float *, float *, int, int, int, int, const BlockGeom *,
                                 int, cudaStream_t);
template void launch_pool<__nv_bfloat16>(const __nv_bfloat16 *, __nv_bfloat16 *, int, int, int,
                                         int, const BlockGeom *, int, cudaStream_t);
template void launch_unpool<float>(const float *, const float *, float *, int, int, int, int,
                                   const BlockGeom *, int, cudaStream_t);
template void launch_unpool<__nv_bfloat16>(const __nv_bfloat16 *, const __nv_bfloat16 *,
                                           __nv_bfloat16 *, int, int, int, int, const BlockGeom *,
                                           int, cudaStream_t);

// ---- Gram partial sums over owned pixels (CUDA cores) --------------------------------------------
// chunk c covers pixels [p0, p1) of block b's owned rectangle (row-major inside the rectangle);
// CTA (c, pair) accumulates the 64x64 block (I, J), I <= J, of sum_p V_p V_p^T in FP32 (one chain
// of FMAs per element, in pixel order) and writes it to part[(c * npairs + pair) * 4096 + i * 64 + j].
// With chunks == null, V is one flat [n_flat][C] matrix and CTA c takes pixels
// [c * chunk_len, min((c + 1) * chunk_len, n_flat)).
//
// 64 threads; slices of 16 pixels, NBUF - 1 of them ahead on their way to shared memory (cp.async, in
// the features' own type); packed FMAs. BLK = 64: a CTA makes the whole 64 x 64 block, 8 x 8 elements per
// thread. BLK = 32: a quarter of it, 4 x 4 per thread. Times below: nst_gram, partials and reduction,
// against 256 threads with 4 x 4 elements each and loads straight into the slice.
// Many CTAs per SM: bound by FP32 FMAs and shared-memory reads, which take 16 clocks each per
// pixel and warp at 8 x 8 (8 : 4 at 4 x 4). Pixels x channels: 50,000 x 256 163 -> 89 us in FP32, 153
// -> 106 in BF16 (128 with BF16 staged in registers as FP32); 150,000 x 320 542 -> 357 and 534 -> 429.
// Two slices in FP32, three in BF16: the other way round 4 % and 1.5 % slower.
// Few CTAs: bound by a CTA's own 256 or more pixels, one after the other on the two schedulers its
// warps sit on; four quarters on four SMs take a quarter each, with more loads in flight. 300 to
// 5,000 x 64: 23 -> 15 us (whole blocks 25 in FP32, 27 in BF16).
constexpr int kGramPx = 16;
// 4 elements to shared memory (src is not read where live is false: zeros)
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(live ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async4(__nv_bfloat16 *dst, const __nv_bfloat16 *src, bool live) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(live ? 8 : 0)
               : "memory");
}
// 4 elements from shared memory as two pairs of floats
__device__ __forceinline__ void load4_pairs(const float *p, unsigned long long v[2]) {
  const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
  v[0] = t.x;
  v[1] = t.y;
}
__device__ __forceinline__ void load4_pairs(const __nv_bfloat16 *p, unsigned long long v[2]) {
  float f[4];
  load4(p, f);
  asm("mov.b64 %0, {%1, %2};" : "=l"(v[0]) : "f"(f[0]), "f"(f[1]));
  asm("mov.b64 %0, {%1, %2};" : "=l"(v[1]) : "f"(f[2]), "f"(f[3]));
}
template <typename T, int BLK, int NBUF>
__global__ void __launch_bounds__(64) gram_partial_kernel(const T *__restrict__ V, int Hb, int Wb,
                                                          int C, const OwnRect *__restrict__ own,
                                                          const GramChunk *__restrict__ chunks,
                                                          float *__restrict__ part,
                                                          long long chunk_len, long long n_flat) {
  constexpr int NQ = (64 / BLK) * (64 / BLK);   // CTAs per block pair
  constexpr int E = BLK / 8, GR = E / 4;        // elements per thread and side, in groups of 4
  __shared__ __align__(16) T Ai[NBUF][kGramPx][BLK];
  __shared__ __align__(16) T Aj[NBUF][kGramPx][BLK];
  const int nb = C / 64;
  const int npairs = nb * (nb + 1) / 2;
  const int pair = blockIdx.y / NQ, quarter = blockIdx.y % NQ;
  int I = 0, J = pair;
  while (J >= nb - I) { J -= nb - I; I++; }
  J += I;
  GramChunk ch;
  OwnRect r;
  if (chunks) {
    ch = chunks[blockIdx.x];
    r = own[ch.b];
  } else {
    const long long p0 = (long long)blockIdx.x * chunk_len;
    const long long p1 = p0 + chunk_len < n_flat ? p0 + chunk_len : n_flat;
    ch = {0, (int)p0, (int)p1};
    r = {0, 1, 0, (int)n_flat};
  }
  const int rw = r.x1 - r.x0, len = ch.p1 - ch.p0;
  const int tid = threadIdx.x;
  // the CTA's channels: ci .. ci + BLK - 1 against cj .. cj + BLK - 1
  const int ri = (NQ == 1 ? 0 : quarter / 2 * 32), rj = (NQ == 1 ? 0 : quarter % 2 * 32);
  const int ci = I * 64 + ri, cj = J * 64 + rj;
  const bool same = ci == cj;
  // this thread loads channels 4 lq .. of pixels lp, lp + 256 / BLK, ... of a slice
  constexpr int LP = 256 / BLK;
  const int lq = (tid % (BLK / 4)) * 4, lp = tid / (BLK / 4);
  auto fetch = [&](int buf, int k0) {   // pixels k0 .. of the chunk: one slice, one commit group
#pragma unroll
    for (int u = 0; u < kGramPx / LP; u++) {
      const int k = k0 + lp + LP * u, q = ch.p0 + (k < len ? k : 0);
      const int y = q / rw, x = q - y * rw;
      const T *row = V + (((size_t)ch.b * Hb + r.y0 + y) * Wb + r.x0 + x) * C;
      cp_async4(&Ai[buf][lp + LP * u][lq], row + ci + lq, k < len);
      if (!same) cp_async4(&Aj[buf][lp + LP * u][lq], row + cj + lq, k < len);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // elements (ti + 32 g .. + 3) x (tj + 32 h .. + 3): a warp covers BLK rows and 16 (+ 16) columns
  const int ti = ((tid & 31) >> 2) * 4, tj = (tid >> 5) * 16 + (tid & 3) * 4;
  unsigned long long acc[E][E / 2];
#pragma unroll
  for (int i = 0; i < E; i++)
#pragma unroll
    for (int j = 0; j < E / 2; j++) acc[i][j] = 0ull;
#pragma unroll
  for (int i = 0; i < NBUF - 1; i++) fetch(i, i * kGramPx);   // (past the end: zeros)
  int buf = 0;
  for (int k0 = 0; k0 < len; k0 += kGramPx) {
    // this slice has arrived in every thread's part, and every thread has left the slice before
    // it, whose buffer the next slice to fetch takes
    asm volatile("cp.async.wait_group %0;" ::"n"(NBUF - 2) : "memory");
    __syncthreads();
    fetch(buf == 0 ? NBUF - 1 : buf - 1, k0 + (NBUF - 1) * kGramPx);
    const T(*Bj)[BLK] = same ? Ai[buf] : Aj[buf];
#pragma unroll
    for (int p = 0; p < kGramPx; p++) {
      float ar[E];
      unsigned long long br[E / 2];
#pragma unroll
      for (int g = 0; g < GR; g++) {
        load4(&Ai[buf][p][ti + 32 * g], ar + 4 * g);
        load4_pairs(&Bj[p][tj + 32 * g], br + 2 * g);
      }
#pragma unroll
      for (int i = 0; i < E; i++) {
        const unsigned long long ad = dup2(ar[i]);
#pragma unroll
        for (int j = 0; j < E / 2; j++) fma2(acc[i][j], ad, br[j]);
      }
    }
    buf = buf == NBUF - 1 ? 0 : buf + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  float *o = part + ((size_t)blockIdx.x * npairs + pair) * 4096 + ri * 64 + rj;
#pragma unroll
  for (int i = 0; i < E; i++)
#pragma unroll
    for (int h = 0; h < GR; h++)
      *reinterpret_cast<ulonglong2 *>(o + (ti + (i >> 2) * 32 + (i & 3)) * 64 + tj + 32 * h) =
          make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
}

// Gacc[C][C] (+)= sum over chunks (fixed order) of the partial blocks, mirrored for I != J. 8 warps
// of a CTA take 128 consecutive elements and every 8th chunk each (a float4 per lane and chunk,
// eight chunks' loads in flight), in compensated FP32 (a pair per element, as exact as an FP64 sum
// of the FP32 partials to 2^-46; the FP64 unit retires two operations per SM and clock), and the
// warps' pairs are added in warp order and converted once. One thread per element adding all
// chunks in FP64: 186 us for 1,024 chunks of C = 64; this 21.
__global__ void __launch_bounds__(256) gram_reduce_kernel(const float *__restrict__ part, int nchunks,
                                                          int C, double *__restrict__ Gacc,
                                                          int overwrite) {
  __shared__ float2 red[8][128];
  const int nb = C / 64;
  const int npairs = nb * (nb + 1) / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t stride = (size_t)npairs * 4096;
  const float *p = part + (size_t)blockIdx.x * 128 + lane * 4;
  float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
  auto add = [](float &s1, float &c1, float x) {   // Knuth's TwoSum
    const float t = s1 + x, z = t - s1;
    c1 += (s1 - (t - z)) + (x - z);
    s1 = t;
  };
  for (int c0 = warp; c0 < nchunks; c0 += 64) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (c0 + 8 * u < nchunks)
        v[u] = __ldg(reinterpret_cast<const float4 *>(p + (size_t)(c0 + 8 * u) * stride));
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (c0 + 8 * u < nchunks) {
        add(s[0], c[0], v[u].x);
        add(s[1], c[1], v[u].y);
        add(s[2], c[2], v[u].z);
        add(s[3], c[3], v[u].w);
      }
  }
#pragma unroll
  for (int k = 0; k < 4; k++) red[warp][lane * 4 + k] = make_float2(s[k], c[k]);
  __syncthreads();
  if (threadIdx.x >= 128) return;
  float ts = 0.f, tc = 0.f;
#pragma unroll
  for (int w = 0; w < 8; w++) {
    const float2 q = red[w][threadIdx.x];
    add(ts, tc, q.x);
    tc += q.y;
  }
  const int e = blockIdx.x * 128 + threadIdx.x, k = e % 4096;
  double g = (double)ts + (double)tc;
  if (!(fabsf(ts) <= FLT_MAX)) {   // an infinite partial, or a sum that FP32 does not hold
    g = 0.0;
    for (int q = 0; q < nchunks; q++) g += (double)part[(size_t)q * stride + e];
  }
  int pair = e / 4096, I = 0;
  while (pair >= nb - I) { pair -= nb - I; I++; }
  const int J = I + pair;
  const int i = I * 64 + k / 64, j = J * 64 + k % 64;
  double *d = Gacc + (size_t)i * C + j;
  *d = overwrite ? g : *d + g;
  if (I != J) {
    d = Gacc + (size_t)j * C + i;
    *d = overwrite ? g : *d + g;
  }
}

// Up to one whole block per SM (152) runs as quarters: at 120 blocks (5,000 pixels x 192) 19.3
// against 25.4 us in FP32 and 21.3 against 29.5 in BF16; at 237 (20,000 x 128) 29.8 against 27.4 and
// 35.5 against 31.5.
constexpr int kGramQuarters = 152;
template <typename T>
static void launch_gram_blocks(const T *V, int Hb, int Wb, int C, const OwnRect *own,
                               const GramChunk *chunks, int nchunks, float *part,
                               long long chunk_len, long long n_flat, cudaStream_t s) {
  const int nb = C / 64, npairs = nb * (nb + 1) / 2;
  if ((long long)nchunks * npairs <= kGramQuarters)
    gram_partial_kernel<T, 32, 8><<<dim3(nchunks, 4 * npairs), 64, 0, s>>>(
        V, Hb, Wb, C, own, chunks, part, chunk_len, n_flat);
  else
    gram_partial_kernel<T, 64, sizeof(T) == 4 ? 2 : 3><<<dim3(nchunks, npairs), 64, 0, s>>>(
        V, Hb, Wb, C, own, chunks, part, chunk_len, n_flat);
}

template <typename T>
void launch_gram_partial(const T *V, int Hb, int Wb, int C, const OwnRect *own,
                         const GramChunk *chunks, int nchunks, float *part, cudaStream_t s) {
  launch_gram_blocks<T>(V, Hb, Wb, C, own, chunks, nchunks, part, 0, 0, s);
}

template <typename T>
void launch_gram_partial_flat(const T *V, long long npix, int C, long long chunk_len, int nchunks,
                              float *part, cudaStream_t s) {
  launch_gram_blocks<T>(V, 1, (int)npix, C, nullptr, nullptr, nchunks, part, chunk_len, npix, s);
}
template void launch_gram_partial_flat<float>(const float *, long long, int, long long, int,
                                              float *, cudaStream_t);
template void launch_gram_partial_flat<__nv_bfloat16>(const __nv_bfloat16 *, long long, int,
                                                      long long, int, float *, cudaStream_t);
template void launch_gram_partial<float>(const float *, int, int, int, const OwnRect *,
                                         const GramChunk *, int, float *, cudaStream_t);
template void launch_gram_partial<__nv_bfloat16>(const __nv_bfloat16 *, int, int, int,
                                                 const OwnRect *, const GramChunk *, int, float *,
                                                 cudaStream_t);
void launch_gram_reduce(const float *part, int nchunks, int C, double *Gacc, bool overwrite,
                        cudaStream_t s) {
  const int nb = C / 64;
  gram_reduce_kernel<<<nb * (nb + 1) / 2 * 32, 256, 0, s>>>(part, nchunks, C, Gacc,
                                                            overwrite ? 1 : 0);
}

// ---- style finalisation: G = Gacc / np, E_L = w ||G - Ghat||^2, R = (4 w / np)(G - Ghat) -------------
// One launch over the 32 x 32 tiles on and above the diagonals of all layers; G, Ghat and R are
// symmetric, and a tile above the diagonal also writes its mirror image (through shared memory).
// The thread of a diagonal element also forms the channel's mean / std terms of Eq. 5 from the
// channel sum and G_jj: beta_j (added to R_jj), alpha_j (epilogue offset), its share of the moment
// loss, and the moments themselves when requested. The CTAs' loss partials are added per layer, in
// CTA order, by the last CTA to finish.
// Bound: FP64 (about six operations per element at two per SM and clock) and latency; four
// elements per thread are loaded together. Three launches over all elements, 16 in turn per thread,
// with 64-bit divisions, took 36 us; one launch over all elements 16.5; this 15.
constexpr int kFinThreads = 256;
__host__ __device__ inline int fin_tiles(int C) { return C / 32 * (C / 32 + 1) / 2; }
__global__ void __launch_bounds__(kFinThreads) style_finalize_kernel(StyleFinalizeArgs a) {
  __shared__ double red[kFinThreads];
  __shared__ double tg[32][33];
  __shared__ float tr[32][33];
  __shared__ int last_sh;
  const int tid = threadIdx.x;
  int l = 0, b = blockIdx.x;
  while (b >= fin_tiles(a.L[l].C)) b -= fin_tiles(a.L[l++].C);
  const StyleLayerArgs L = a.L[l];
  int ti = 0;   // tile (ti, tj), ti <= tj
  for (int n = L.C / 32; b >= n - ti; ti++) b -= n - ti;
  const int tj = ti + b;
  const double inv = L.inv_np, rs = L.rs, we = ti == tj ? L.w : 2.0 * L.w;
  const int j = tj * 32 + (tid & 31), i0 = ti * 32 + (tid >> 5);   // rows i0, i0 + 8, ...
  pdl_begin();
  double s = 0.0, g[4], h[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int e = (i0 + 8 * k) * L.C + j;
    g[k] = L.Gacc[e];
    h[k] = L.Ghat ? L.Ghat[e] : 0.0;
  }
  auto put = [&](int e, double G, float r) {
    L.Gout[e] = G;
    if (a.r_is_bf16)
      reinterpret_cast<__nv_bfloat16 *>(L.R)[e] = __float2bfloat16_rn(r);
    else
      reinterpret_cast<float *>(L.R)[e] = r;
  };
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int i = i0 + 8 * k;
    const double G = g[k] * inv, d = G - h[k];
    s += we * d * d;
    double r = rs * d;
    if (i == j && L.S) {
      // rounded products (no contraction into an FMA), so the loss pass reproduces the target
      // pass's mean bit for bit when x = v
      const double m = __dmul_rn(L.S[j], inv);
      const double var = __dmul_rn(g[k], inv) - __dmul_rn(m, m);
      const double sd = var > 0.0 ? sqrt(var) : 0.0;
      if (L.mean_out) L.mean_out[j] = m;
      if (L.std_out) L.std_out[j] = sd;
      if (L.mu) {
        s += L.wm * (m - L.mu[j]) * (m - L.mu[j]) + L.ws * (sd - L.sigma[j]) * (sd - L.sigma[j]);
        const double beta = sd > 0.0 ? L.ws * 2.0 * inv * (sd - L.sigma[j]) / sd : 0.0;
        if (L.alpha) L.alpha[j] = (float)(L.wm * 2.0 * inv * (m - L.mu[j]) - beta * m);
        r += beta;
      }
    }
    put(i * L.C + j, G, (float)r);
    if (ti != tj) {
      tg[(tid >> 5) + 8 * k][tid & 31] = G;
      tr[(tid >> 5) + 8 * k][tid & 31] = (float)r;
    }
  }
  red[tid] = s;
  __syncthreads();
  if (ti != tj)
#pragma unroll
    for (int k = 0; k < 4; k++) {   // element (tj * 32 + row, ti * 32 + column)
      const int row = (tid >> 5) + 8 * k, col = tid & 31;
      put((tj * 32 + row) * L.C + ti * 32 + col, tg[col][row], tr[col][row]);
    }
  for (int k = kFinThreads / 2; k > 0; k >>= 1) {
    if (tid < k) red[tid] += red[tid + k];
    __syncthreads();
  }
  if (tid == 0) {
    a.partial[blockIdx.x] = red[0];
    __threadfence();
    last_sh = atomicAdd(a.arrived, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  if (tid < 32 * kNStyle) {   // a warp per layer: lane q the CTAs q, q + 32, ... in order, a tree
    const int wl = tid >> 5;
    int c0 = 0;
    for (int q = 0; q < wl; q++) c0 += fin_tiles(a.L[q].C);
    double t = 0.0;
    for (int q = tid & 31; q < fin_tiles(a.L[wl].C); q += 32) t += __ldcg(a.partial + c0 + q);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((tid & 31) == 0) a.Eparts[wl] = t;
  }
  if (tid == 0) *a.arrived = 0u;
}

void launch_style_finalize(const StyleFinalizeArgs &a, cudaStream_t s) {
  int n = 0;
  StyleFinalizeArgs b = a;
  for (int l = 0; l < kNStyle; l++) {
    n += fin_tiles(a.L[l].C);
    b.L[l].inv_np = 1.0 / a.L[l].np;   // (two FP64 divisions per thread are half the kernel)
    b.L[l].rs = 4.0 * a.L[l].w / a.L[l].np;
  }
  launch_pdl(true, style_finalize_kernel, n, kFinThreads, 0, s, b);
}

// ---- channel sums over owned pixels, all style layers in one launch -------------------------------
// FP32 sums of runs of 64 pixels (of each chunk, in pixel order), added in FP64. Bound: the read of
// the activations; a thread per channel took a pixel at a time (2 bytes a load, a division per
// pixel, 40 CTAs at the deep layers: 1,980 us for the five layers of 1512 x 2016). Here C / 8 lanes
// take a run, 16 bytes of a pixel each with eight pixels' loads in flight; a CTA holds 2048 / C
// runs at a time, and the runs of a chunk are dealt to as many CTAs as fill the chip:
// 174 us, 744 MB.
constexpr int kChansumThreads = 256, kChansumRun = 64;
template <typename T>
__global__ void __launch_bounds__(kChansumThreads) chansum_partial_kernel(ChansumArgs a) {
  __shared__ double red[kChansumThreads * 8];   // [lane group][C]
  pdl_begin();
  int l = 0;
  while (l + 1 < kNStyle && (int)blockIdx.x >= a.L[l + 1].cta0) l++;
  const ChansumLayer L = a.L[l];
  const int idx = blockIdx.x - L.cta0, chunk = idx / L.split, s = idx - chunk * L.split;
  const GramChunk ch = L.chunks[chunk];
  const OwnRect r = L.own[ch.b];
  const int rw = r.x1 - r.x0, C = L.C, G = C / 8, NG = kChansumThreads / G;
  const int grp = threadIdx.x / G, c0 = (threadIdx.x % G) * 8;
  const T *V = reinterpret_cast<const T *>(L.V);
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; j++) acc[j] = 0.0;
  // this CTA's runs: s, s + split, ...; this lane group's: every NG-th of those
  for (long long run = s + (long long)L.split * grp;; run += (long long)L.split * NG) {
    const long long qs = ch.p0 + run * kChansumRun;
    if (grp >= NG || qs >= ch.p1) break;
    int q = (int)qs;
    const int q1 = min(q + kChansumRun, ch.p1);
    int x = q % rw;
    const T *p = V + (((size_t)ch.b * L.Hb + r.y0 + q / rw) * L.Wb + r.x0 + x) * C + c0;
    auto next = [&]() {
      p += C;
      if (++x == rw) { x = 0; p += (size_t)(L.Wb - rw) * C; }
    };
    float f[8];
#pragma unroll
    for (int j = 0; j < 8; j++) f[j] = 0.f;
    for (; q + 8 <= q1; q += 8) {
      float v[8][8];
#pragma unroll
      for (int k = 0; k < 8; k++) {
        load8(p, v[k]);
        next();
      }
#pragma unroll
      for (int k = 0; k < 8; k++)
#pragma unroll
        for (int j = 0; j < 8; j++) f[j] += v[k][j];
    }
    for (; q < q1; q++) {
      float v[8];
      load8(p, v);
      next();
#pragma unroll
      for (int j = 0; j < 8; j++) f[j] += v[j];
    }
#pragma unroll
    for (int j = 0; j < 8; j++) acc[j] += (double)f[j];
  }
  if (grp < NG)
#pragma unroll
    for (int j = 0; j < 8; j++) red[grp * C + c0 + j] = acc[j];
  __syncthreads();
  for (int j = threadIdx.x; j < C; j += kChansumThreads) {   // the groups in index order
    double t = 0.0;
    for (int g = 0; g < NG; g++) t += red[g * C + j];
    L.partial[(size_t)idx * C + j] = t;
  }
}

// S[j] += sum of the layer's partials: a CTA takes 32 channels (lane = channel), its 16 warps
// split the partials (warp w: w, w + 16, ... in order), then the warps are added in order
constexpr int kChansumWarps = 16;
__global__ void __launch_bounds__(32 * kChansumWarps) chansum_reduce_kernel(ChansumArgs a) {
  __shared__ double red[kChansumWarps][32];
  pdl_begin();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int l = 0, b = blockIdx.x;
  while (b >= a.L[l].C / 32) b -= a.L[l++].C / 32;
  const ChansumLayer L = a.L[l];
  const int j = b * 32 + lane, n = L.nchunks * L.split;
  double s = 0.0;
  for (int c0 = warp; c0 < n; c0 += 8 * kChansumWarps) {   // eight loads in flight
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int c = c0 + k * kChansumWarps;
      v[k] = c < n ? L.partial[(size_t)c * L.C + j] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 8; k++) s += v[k];
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kChansumWarps; w++) t += red[w][lane];
    L.S[j] += t;
  }
}

int chansum_split(int nchunks, int max_chunk_px) {
  const int runs = (max_chunk_px + kChansumRun - 1) / kChansumRun;
  const int want = nchunks > 0 ? 1216 / nchunks : 1;   // eight CTAs per SM
  return want < 1 ? 1 : want > runs ? (runs > 0 ? runs : 1) : want;
}

template <typename T>
void launch_chansum(ChansumArgs a, cudaStream_t s) {
  int ctas = 0, rctas = 0;
  for (int l = 0; l < kNStyle; l++) {
    a.L[l].cta0 = ctas;
    ctas += a.L[l].nchunks * a.L[l].split;
    rctas += a.L[l].C / 32;
  }
  if (ctas <= 0) return;
  launch_pdl(true, chansum_partial_kernel<T>, ctas, kChansumThreads, 0, s, a);
  launch_pdl(true, chansum_reduce_kernel, rctas, 32 * kChansumWarps, 0, s, a);
}
template void launch_chansum<float>(ChansumArgs, cudaStream_t);
template void launch_chansum<__nv_bfloat16>(ChansumArgs, cudaStream_t);


// ---- content loss over owned pixels: parts[5] (+)= lambda sum (V - Vu)^2 ----------------------------
// partial[c] = chunk c's sum; the last CTA to finish adds the partials (thread t: t, t + 256, ... in
// order, then a fixed tree) and, for the evaluation's last batch, the six parts into the loss.
template <typename T>
__global__ void __launch_bounds__(256) content_loss_kernel(ContentLossArgs a) {
  __shared__ double red[256];
  __shared__ int last_sh;
  auto tree = [&]() {
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
      if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
      __syncthreads();
    }
  };
  double s = 0.0;
  pdl_begin();
  if ((int)blockIdx.x < a.nchunks) {
    const GramChunk ch = a.chunks[blockIdx.x];
    const OwnRect r = a.own[ch.b];
    const BlockGeom g = a.geom[ch.b];
    const int rw = r.x1 - r.x0;
    const int oy = g.ey0 >> kContentLevel, ox = g.ex0 >> kContentLevel;
    const T *V = reinterpret_cast<const T *>(a.V), *Vu = reinterpret_cast<const T *>(a.Vu);
    // 64 threads per pixel row of 512 channels (8 each)
    for (int q = ch.p0 + (threadIdx.x >> 6); q < ch.p1; q += 4) {
      const int y = r.y0 + q / rw, x = r.x0 + q % rw;
      const int c = (threadIdx.x & 63) * 8;
      float v[8], t[8];
      load8(V + (((size_t)ch.b * a.Hb + y) * a.Wb + x) * 512 + c, v);
      load8(Vu + ((size_t)(oy + y) * a.Wc + ox + x) * 512 + c, t);
      // differences of two stored values are exact in FP32 (BF16 inputs) or nearly so (FP32
      // inputs); 8 squares summed in FP32, then accumulated in FP64
      float f = 0.f;
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const float d = v[j] - t[j];
        f = fmaf(d, d, f);
      }
      s += (double)f;
    }
  }
  red[threadIdx.x] = s;
  tree();
  if (threadIdx.x == 0) {
    a.partial[blockIdx.x] = red[0];
    __threadfence();
    last_sh = atomicAdd(a.arrived, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  s = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) s += __ldcg(a.partial + i);
  red[threadIdx.x] = s;
  tree();
  if (threadIdx.x == 0) {
    const double c = a.lambda * red[0] + (a.first ? 0.0 : a.parts[kNStyle]);
    a.parts[kNStyle] = c;
    if (a.loss) {
      double t = 0.0;
      for (int i = 0; i < kNStyle; i++) t += a.parts[i];
      *a.loss = t + c;
    }
    *a.arrived = 0u;
  }
}

template <typename T>
void launch_content_loss(const ContentLossArgs &a, cudaStream_t s) {
  launch_pdl(true, content_loss_kernel<T>, a.nchunks > 0 ? a.nchunks : 1, 256, 0, s, a);
}
template void launch_content_loss<float>(const ContentLossArgs &, cudaStream_t);
template void launch_content_loss<__nv_bfloat16>(const ContentLossArgs &, cudaStream_t);

// ---- content target crop: owned ReLU4_2 features of each block into the global map ------------------
template <typename T>
__global__ void crop_content_kernel(const T *__restrict__ V, int B, int Hb, int Wb,
                                    const BlockGeom *__restrict__ geom,
                                    const OwnRect *__restrict__ own, T *__restrict__ Vu, int Hc,
                                    int Wc) {
  const int b = blockIdx.y;
  const OwnRect r = own[b];
  const BlockGeom g = geom[b];
  const int rw = r.x1 - r.x0;
  const long long n = (long long)(r.y1 - r.y0) * rw * 64;
  const int oy = g.ey0 >> kContentLevel, ox = g.ex0 >> kContentLevel;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % 64) * 8;
    const long long q = i / 64;
    const int y = r.y0 + (int)(q / rw), x = r.x0 + (int)(q % rw);
    float v[8];
    load8(V + (((size_t)b * Hb + y) * Wb + x) * 512 + c, v);
    store8(Vu + ((size_t)(oy + y) * Wc + ox + x) * 512 + c, v);
  }
  (void)B;
  (void)Hc;
}

template <typename T>
void launch_crop_content(const T *V, int B, int Hb, int Wb, const BlockGeom *geom,
                         const OwnRect *own, T *Vu, int Hc, int Wc, int max_own_px,
                         cudaStream_t s) {
  int gx = (int)(((long long)max_own_px * 64 + 255) / 256);
  if (gx > 2048) gx = 2048;
  if (gx < 1) gx = 1;
  crop_content_kernel<T><<<dim3(gx, B), 256, 0, s>>>(V, B, Hb, Wb, geom, own, Vu, Hc, Wc);
}
template void launch_crop_content<float>(const float *, int, int, int, const BlockGeom *,
                                         const OwnRect *, float *, int, int, int, cudaStream_t);
template void launch_crop_content<__nv_bfloat16>(const __nv_bfloat16 *, int, int, int,
                                                 const BlockGeom *, const OwnRect *,
                                                 __nv_bfloat16 *, int, int, int, cudaStream_t);

// ---- misc ---------------------------------------------------------------------------------------
__global__ void check_finite_kernel(const float *__restrict__ x, long long n,
                                    unsigned *__restrict__ err) {
  bool bad = false;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    bad |= !isfinite(x[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, kErrNonfinite);
}
void launch_check_finite(const float *x, long long n, unsigned *err, cudaStream_t s) {
  check_finite_kernel<<<ew_grid(n), 256, 0, s>>>(x, n, err);
}

}  // namespace nst
