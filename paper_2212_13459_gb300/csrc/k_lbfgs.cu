// k_lbfgs.cu -- HBM-bound vector kernels of the optimiser and of the multiscale initialisation:
//   * the L-BFGS step (Section 3.1, after Nocedal 1980) in the compact representation of the
//     inverse-BFGS matrix (Byrd, Nocedal and Schnabel 1994): with S, Y the stored pairs (oldest
//     first), R the upper triangle of S^T Y, D its diagonal and H0 = gamma I,
//         H g = gamma g + S p - gamma Y u,  u = R^-1 (S^T g),
//                                           p = R^-T ((D + gamma Y^T Y) u - gamma Y^T g),
//     the same matrix the two-loop recursion applies. A step reads every stored vector twice
//     (one fused pass for all dot products, one pass forming the step) instead of four times;
//     S^T Y and Y^T Y are kept up to date from the new pair's dot products. Dots are FP32 chunks
//     summed in compensated FP32 and FP64 with fixed-order reductions; the small solve runs in
//     FP64 in one CTA.
//     History slots are resolved on the device, so a step needs no host round trip.
//   * bicubic x2 upscaling used to initialise each scale after the first (Algorithm 2).
#include <cfloat>
#include <type_traits>

#include "nst_internal.cuh"
#include "nst_kernels.h"
#include "nst_lbfgs_dev.h"

namespace nst {

constexpr int kDotThreads = 256;
constexpr int kDotBlocksTotal = 1216;   // 8 CTAs per SM on 152 SMs, shared among the groups

static int dot_groups(int m) { return (m + 1 + kLbGroup - 1) / kLbGroup; }
static int dot_blocks(int m) {   // CTAs per group; fixed for a given m (reproducible reductions)
  const int b = kDotBlocksTotal / dot_groups(m);
  return b < 152 ? 152 : b;
}
int lbfgs_partials_count(int m) { return 4 * (m + 1) * dot_blocks(m); }

// Position p of the fused pass: p = 0 is the candidate pair (spare slot: last step s and the new
// y), p = 1 .. count the stored pairs order[p - 1]; c->dots[4 p + q], q = 0: s.g, 1: y.g,
// 2: s.y_new, 3: y.y_new. Elements go four at a time (float4) when every vector is 16-byte
// aligned, with all of an element group's loads issued before its FMAs.
//
// Bound: HBM (2 (count + 1) + 2 vectors read once). What kept it from there was the FP64 unit,
// which retires two operations per SM and clock on this GPU: a double add (and a conversion) per
// 16 elements and dot, and 80 double shuffle-adds per warp at the end. So a CTA's FP32 chunks are
// added in compensated FP32 (Sum, 48 bits): the error of the chunks themselves, about 2^-24 /
// sqrt(their number), stays orders above that of adding them (6,912 to 9.7 M elements, terms of one
// sign, of both, cancelling, heavy-tailed: chunks off by 3e-12 to 2e-8 of the terms' magnitudes, pairs and
// FP64 sums of the same chunks apart by 0 to 1e-15). The warp reduction is a reduce-scatter
// (16 exchanges for 16 dots, not 80), and the last CTA of a group to finish adds the CTAs'
// partials in FP64 in index order, in parallel over the groups, where the single CTA of the solve
// spent 15 us on it. CTAs of all groups that read the same elements are neighbours in launch
// order, so g and g_prev come from L2 for all but one of them. Measured with 100 stored pairs of
// 2.29 M elements: 594 -> 345 us (5.4 TB/s); 10 pairs of 36.6 M: 634 us (5.8 TB/s). The loads in
// flight are bounded by the registers: an FP64 sum of two of the dots beside the pairs, a test of
// every chunk's size, or a second pass over the elements after this one each cost 5 to 8 %.
// A dot that leaves FP32's range within a CTA comes out infinite or NaN, sets c->beyond, and is made
// again in FP64 by the solve (lbfgs_dots_again).
struct Sum {   // s + c: the sum with the rounding errors of its additions (Knuth's TwoSum)
  float s, c;
  __device__ __forceinline__ double value() const {   // (c says nothing beside an infinite s)
    return fabsf(s) <= FLT_MAX ? (double)s + (double)c : (double)s;
  }
  __device__ __forceinline__ void add(float x) {
    const float t = s + x, z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
  }
  __device__ __forceinline__ void merge(float xs, float xc) {
    add(xs);
    c += xc;
  }
};

template <int G>
struct DotAcc {
  Sum acc[4 * G];
  float part[4 * G];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int d = 0; d < 4 * G; d++) acc[d].s = acc[d].c = part[d] = 0.f;
  }
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int d = 0; d < 4 * G; d++) acc[d].add(part[d]), part[d] = 0.f;
  }
  __device__ __forceinline__ void add(int j, float sv, float wv, float gv, float yv) {
    part[4 * j] = fmaf(sv, gv, part[4 * j]);
    part[4 * j + 1] = fmaf(wv, gv, part[4 * j + 1]);
    part[4 * j + 2] = fmaf(sv, yv, part[4 * j + 2]);
    part[4 * j + 3] = fmaf(wv, yv, part[4 * j + 3]);
  }
};

__global__ void __launch_bounds__(kDotThreads) lbfgs_dots_kernel(
    const float *g, const float *g_prev, const float *S, float *Y, long long stride, long long n,
    LbfgsCtl *c, int first, int vec, double *partials) {
  constexpr int G = kLbGroup;
  static_assert(4 * G == 16, "the warp reduce-scatter below takes 16 dots");
  __shared__ long long off[G];
  __shared__ int nj_sh, last_sh;
  __shared__ long long sp_off;
  __shared__ Sum red[kDotThreads / 32][4 * G];
  const int grp = blockIdx.x, nb = gridDim.y, cta = blockIdx.y;
  pdl_begin();
  if (threadIdx.x == 0) {
    const int count = c->count;
    int nj = 0;
    for (int j = 0; j < G; j++) {
      const int p = grp * G + j;
      off[j] = 0;
      if (p <= count) {
        off[j] = (long long)(p == 0 ? c->spare : c->order[p - 1]) * stride;
        nj = j + 1;
      }
    }
    nj_sh = first ? (grp == 0 ? 1 : 0) : nj;
    sp_off = (long long)c->spare * stride;
  }
  __syncthreads();
  const int nj = nj_sh;
  if (nj == 0) return;
  float *ynew = Y + sp_off;
  const bool own_y = grp == 0;   // group 0 holds the candidate (position 0) and writes its y
  const long long tstride = (long long)nb * kDotThreads;
  const long long t0 = (long long)cta * kDotThreads + threadIdx.x;
  DotAcc<G> A;
  A.clear();
  int chunk = 0;
  const long long n4 = vec ? n / 4 : 0;
  for (long long v = t0; v < n4; v += tstride) {
    const float4 gv = reinterpret_cast<const float4 *>(g)[v];
    if (first) {
      A.part[0] += fabsf(gv.x) + fabsf(gv.y) + fabsf(gv.z) + fabsf(gv.w);
    } else {
      const float4 gp = reinterpret_cast<const float4 *>(g_prev)[v];
      const float4 yv = make_float4(gv.x - gp.x, gv.y - gp.y, gv.z - gp.z, gv.w - gp.w);
      float4 sv[G], wv[G];
#pragma unroll
      for (int j = 0; j < G; j++) {
        if (j < nj) {
          sv[j] = reinterpret_cast<const float4 *>(S + off[j])[v];
          wv[j] = (own_y && j == 0) ? yv : reinterpret_cast<const float4 *>(Y + off[j])[v];
        }
      }
      if (own_y) reinterpret_cast<float4 *>(ynew)[v] = yv;   // (after the loads are issued)
#pragma unroll
      for (int j = 0; j < G; j++) {
        if (j < nj) {
          A.add(j, sv[j].x, wv[j].x, gv.x, yv.x);
          A.add(j, sv[j].y, wv[j].y, gv.y, yv.y);
          A.add(j, sv[j].z, wv[j].z, gv.z, yv.z);
          A.add(j, sv[j].w, wv[j].w, gv.w, yv.w);
        }
      }
    }
    if (++chunk == 4) { chunk = 0; A.flush(); }   // plain FP32 over 16 elements at most
  }
  for (long long i = n4 * 4 + t0; i < n; i += tstride) {   // scalar path / tail
    const float gv = g[i];
    if (first) {
      A.part[0] += fabsf(gv);
    } else {
      const float yv = gv - g_prev[i];
      if (own_y) ynew[i] = yv;
#pragma unroll
      for (int j = 0; j < G; j++)
        if (j < nj) A.add(j, S[off[j] + i], (own_y && j == 0) ? yv : Y[off[j] + i], gv, yv);
    }
    if (++chunk == 16) { chunk = 0; A.flush(); }
  }
  A.flush();
  // fixed-order block reduction. Reduce-scatter over the warp: at distance 2^b (b = 4 .. 1) a lane
  // keeps the half of its dots whose index bit b - 1 equals its lane bit b and passes on the rest,
  // so lane l ends with dot l >> 1, which lanes 2d and 2d + 1 then add
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto level = [&](auto bit) {
    constexpr int b = decltype(bit)::value, h = 1 << (b - 1);
    const bool up = (lane >> b) & 1;
#pragma unroll
    for (int d = 0; d < h; d++) {
      const Sum lo = A.acc[d], hi = A.acc[d + h];
      A.acc[d].s = up ? hi.s : lo.s;
      A.acc[d].c = up ? hi.c : lo.c;
      A.acc[d].merge(__shfl_xor_sync(0xffffffffu, up ? lo.s : hi.s, 1 << b),
                     __shfl_xor_sync(0xffffffffu, up ? lo.c : hi.c, 1 << b));
    }
  };
  level(std::integral_constant<int, 4>{});
  level(std::integral_constant<int, 3>{});
  level(std::integral_constant<int, 2>{});
  level(std::integral_constant<int, 1>{});
  A.acc[0].merge(__shfl_xor_sync(0xffffffffu, A.acc[0].s, 1),
                 __shfl_xor_sync(0xffffffffu, A.acc[0].c, 1));
  if (!(lane & 1)) red[warp][lane >> 1] = A.acc[0];
  __syncthreads();
  if (threadIdx.x < 4 * nj) {   // the warps in index order
    Sum v = red[0][threadIdx.x];
    for (int w = 1; w < kDotThreads / 32; w++) v.merge(red[w][threadIdx.x].s, red[w][threadIdx.x].c);
    partials[(size_t)(grp * G * 4 + threadIdx.x) * nb + cta] = v.value();
    __threadfence();
  }
  __syncthreads();
  // the group's last CTA adds its partials: 16 lanes per dot, lane l the CTAs l, l + 16, ... in
  // order, then a fixed tree
  if (threadIdx.x == 0) last_sh = atomicAdd(&c->arrived[grp], 1u) == (unsigned)nb - 1;
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  const int d = threadIdx.x >> 4, l = threadIdx.x & 15;
  double v = 0.0;
  if (d < 4 * nj)
    for (int q = l; q < nb; q += 16) v += __ldcg(partials + (size_t)(grp * G * 4 + d) * nb + q);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (l == 0 && d < 4 * nj) {
    c->dots[grp * G * 4 + d] = v;
    if (!(fabs(v) <= DBL_MAX)) atomicOr(&c->beyond, 1u);
  }
  if (threadIdx.x == 0) c->arrived[grp] = 0u;
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

void launch_lbfgs_dots(const float *g, const float *g_prev, const float *S, float *Y,
                       long long stride, long long n, LbfgsCtl *c, int m, int first,
                       double *partials, cudaStream_t s) {
  const int vec = aligned16(g) && aligned16(g_prev) && aligned16(S) && aligned16(Y) &&
                  stride % 4 == 0;
  // no CTA without elements (a thread that has work has the same elements as with all CTAs)
  const long long need = ((vec ? n / 4 : n) + kDotThreads - 1) / kDotThreads;
  const int nb = (int)(need < 1 ? 1 : need < dot_blocks(m) ? need : dot_blocks(m));
  dim3 grid(first ? 1 : dot_groups(m), nb);
  launch_pdl(true, lbfgs_dots_kernel, grid, kDotThreads, 0, s, g, g_prev, S, Y, stride, n, c, first,
             vec, partials);
}

// The small solve: curvature test, bookkeeping, the two triangular systems and the coefficients
// of the step, one CTA. k = stored pairs, oldest first; R = D Rs with D = diag R, Rs unit upper:
//   u = Rs^-1 D^-1 (S^T g),  w = (D + gamma Y^T Y) u - gamma Y^T g,  p = D^-1 Rs^-T w.
// Bound: latency, and the FP64 unit (two operations per SM and clock). Rs is scaled and kept in
// shared memory; one warp runs both triangular systems column by column with the vector in
// registers (lane l: rows l, l + 32, ...), so a column costs one shuffle and one FMA of latency;
// Y^T Y is read into registers before the first system and used after it. One thread working from
// global memory took 1,496 us at k = 100 and 58 us at k = 10; this takes 47 and 17 us (all
// cold, under the profiler).
constexpr int kSolveThreads = 512;
// All but one only where the dots are made again; 16 take 0.5 us longer where they are not (1,000
// elements, 10 pairs: 32.0 -> 33.0 us a step, 31.9 with 4)
constexpr int kSolveCtas = 4;
constexpr int kSolveParts = kSolveThreads / kMaxHistory;          // threads per row of Y^T Y
constexpr int kSolveRow = kMaxHistory / kSolveParts;              // its elements each holds
static size_t solve_smem(int m) { return (size_t)m * (m | 1) * sizeof(double); }

// The dots of the fused pass once more, FP32 chunks of 16 elements added in FP64 throughout: for sums
// beyond FP32's range (gradients from about 1e17 on) and for NaN and infinity, which stay. CTA b of
// gridDim.x takes elements b kSolveThreads + thread, ...; true in the last CTA to finish, with c->dots
// set. Y holds y_new in the spare slot (the fused pass wrote it). No inlining: the solve's registers
// are its own.
__device__ __noinline__ bool lbfgs_dots_again(LbfgsCtl *c, const float *g, const float *S,
                                              const float *Y, long long stride, long long n, int first,
                                              double *partials) {
  __shared__ double red[kSolveThreads / 32][4];
  __shared__ int last_sh;
  const int tid = threadIdx.x, lane = tid & 31, nd = first ? 1 : 4 * (c->count + 1);
  const float *yn = Y + c->spare * stride;
  for (int p = 0; 4 * p < nd; p++) {
    const long long off = (p == 0 ? c->spare : c->order[p - 1]) * stride;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    float part[4] = {0.f, 0.f, 0.f, 0.f};
    int chunk = 0;
    auto flush = [&]() {
      chunk = 0;
#pragma unroll
      for (int q = 0; q < 4; q++) acc[q] += (double)part[q], part[q] = 0.f;
    };
    for (long long i = (long long)blockIdx.x * kSolveThreads + tid; i < n;
         i += (long long)gridDim.x * kSolveThreads) {
      if (first) {
        part[0] += fabsf(g[i]);
      } else {
        const float sv = S[off + i], yv = Y[off + i];
        part[0] = fmaf(sv, g[i], part[0]);
        part[1] = fmaf(yv, g[i], part[1]);
        part[2] = fmaf(sv, yn[i], part[2]);
        part[3] = fmaf(yv, yn[i], part[3]);
      }
      if (++chunk == 16) flush();
    }
    flush();
#pragma unroll
    for (int q = 0; q < 4; q++) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
      if (lane == 0) red[tid >> 5][q] = acc[q];
    }
    __syncthreads();
    if (tid < 4) {
      double v = 0.0;
      for (int w = 0; w < kSolveThreads / 32; w++) v += red[w][tid];
      partials[(size_t)(4 * p + tid) * gridDim.x + blockIdx.x] = v;
      __threadfence();
    }
    __syncthreads();
  }
  if (tid == 0) last_sh = atomicAdd(&c->arrived[0], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_sh) return false;
  __threadfence();
  for (int d = tid; d < nd; d += kSolveThreads) {   // the CTAs in index order
    double v = 0.0;
    for (unsigned b = 0; b < gridDim.x; b++) v += __ldcg(partials + (size_t)d * gridDim.x + b);
    c->dots[d] = v;
  }
  if (tid == 0) c->arrived[0] = c->beyond = 0u;
  __syncthreads();
  return true;
}

__global__ void __launch_bounds__(kSolveThreads)
    lbfgs_solve_kernel(LbfgsCtl *c, int m, int first, double eps, double *SY, double *YY,
                       const float *g, const float *S, const float *Y, long long stride, long long n,
                       double *partials) {
  extern __shared__ double Rs[];   // [k][m | 1]: odd row stride, columns without bank conflicts
  __shared__ double sg[kMaxHistory], yg[kMaxHistory], snew[kMaxHistory], ynew[kMaxHistory];
  __shared__ double diag[kMaxHistory], u[kMaxHistory], w[kMaxHistory];
  __shared__ double wpart[kSolveParts][kMaxHistory];
  __shared__ int sl[kMaxHistory], old[kMaxHistory];
  const int tid = threadIdx.x, lane = tid & 31;
  pdl_begin();
  // (one round of loads; c->beyond is unchanged until every CTA has read it, and the CTAs that leave
  // at once use nothing else of this)
  const unsigned beyond = c->beyond;
  const int count0 = c->count, sp = c->spare, ld = m + 1;
  const int slot = tid < kMaxHistory ? c->order[tid] : 0;   // newest first
  double ys = c->dots[2], yy = c->dots[3];
  if (beyond) {
    if (!lbfgs_dots_again(c, g, S, Y, stride, n, first, partials)) return;
    ys = c->dots[2];
    yy = c->dots[3];
  } else if (blockIdx.x) {
    return;
  }
  if (first) {
    if (tid == 0) {
      const double l1 = c->dots[0];
      c->k = 0;
      c->cg = (float)-(l1 > 1.0 ? 1.0 / l1 : 1.0);   // t = min(1, 1 / ||g||_1), d = -g
    }
    return;
  }
  // the candidate becomes the newest pair (dropping the oldest of m) or is left out
  const bool take = ys > eps;
  const int keep = take ? (count0 < m ? count0 : m - 1) : count0;   // older pairs kept
  const int k = keep + (take ? 1 : 0);
  const double gamma = take ? ys / yy : (k > 0 ? c->gamma : 1.0);
  if (tid < kMaxHistory) old[tid] = slot;
  __syncthreads();
  if (tid < k) {
    // pair tid (oldest first): its position in the fused pass, its slot, its four dots
    const int p = k - 1 - tid + (take ? 0 : 1);
    sl[tid] = p == 0 ? sp : old[p - 1];
    sg[tid] = c->dots[4 * p];
    yg[tid] = c->dots[4 * p + 1];
    snew[tid] = c->dots[4 * p + 2];
    ynew[tid] = c->dots[4 * p + 3];
  }
  __syncthreads();
  const int newest = take ? k - 1 : -1;   // its column and row come from the dots
  // this thread's part of row i of Y^T Y (symmetric: read down the column, coalesced over i)
  const int i = tid % kMaxHistory, part = tid / kMaxHistory;
  double yv[kSolveRow];
#pragma unroll
  for (int q = 0; q < kSolveRow; q++) {
    const int j = part * kSolveRow + q;
    yv[q] = 0.0;
    if (i < k && j < k)
      yv[q] = i == newest ? ynew[j] : j == newest ? ynew[i] : YY[(size_t)sl[j] * ld + sl[i]];
  }
  if (tid < k) {
    diag[tid] = tid == newest ? ys : SY[(size_t)sl[tid] * ld + sl[tid]];
    w[tid] = 1.0 / diag[tid];
  }
  __syncthreads();
  const int rs = m | 1;
  for (int r = tid >> 5; r < k; r += kSolveThreads / 32)   // a warp per row
    for (int j = r + 1 + lane; j < k; j += 32)
      Rs[r * rs + j] = w[r] * (j == newest ? snew[r] : SY[(size_t)sl[r] * ld + sl[j]]);
  if (tid < k) u[tid] = sg[tid] * w[tid];
  __syncthreads();
  constexpr int NR = kMaxHistory / 32;
  if (tid < 32) {   // Rs u = D^-1 (S^T g), from the last row up
    double v[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) v[r] = lane + 32 * r < k ? u[lane + 32 * r] : 0.0;
#pragma unroll
    for (int b = NR - 1; b >= 0; b--) {
      for (int q = 31; q >= 0; q--) {
        const int col = 32 * b + q;
        if (col >= k) continue;
        double a[NR];
#pragma unroll
        for (int r = 0; r <= b; r++) a[r] = lane + 32 * r < col ? Rs[(lane + 32 * r) * rs + col] : 0.0;
        const double x = __shfl_sync(0xffffffffu, v[b], q);
#pragma unroll
        for (int r = 0; r <= b; r++) v[r] -= a[r] * x;
      }
    }
#pragma unroll
    for (int r = 0; r < NR; r++)
      if (lane + 32 * r < k) u[lane + 32 * r] = v[r];
  }
  __syncthreads();
  {   // Y^T Y u, kSolveParts threads per row
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < kSolveRow; q++) {
      const int j = part * kSolveRow + q;
      if (j < k) v += yv[q] * u[j];
    }
    wpart[part][i] = v;
  }
  __syncthreads();
  if (tid < 32) {   // Rs^T z = w, from the first row down; p = D^-1 z
    double v[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) {
      const int j = lane + 32 * r;
      v[r] = 0.0;
      if (j < k) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kSolveParts; q++) t += wpart[q][j];
        v[r] = diag[j] * u[j] + gamma * (t - yg[j]);
      }
    }
#pragma unroll
    for (int b = 0; b < NR; b++) {
      for (int q = 0; q < 32; q++) {
        const int row = 32 * b + q;
        if (row >= k) break;
        double a[NR];
#pragma unroll
        for (int r = b; r < NR; r++) {
          const int j = lane + 32 * r;
          a[r] = j > row && j < k ? Rs[row * rs + j] : 0.0;
        }
        const double x = __shfl_sync(0xffffffffu, v[b], q);
#pragma unroll
        for (int r = b; r < NR; r++) v[r] -= a[r] * x;
      }
    }
    // d = -H g = -gamma g - S p + gamma Y u; step length 1
#pragma unroll
    for (int r = 0; r < NR; r++) {
      const int j = lane + 32 * r;
      if (j < k) {
        c->slot[j] = sl[j];
        c->cS[j] = (float)(-v[r] * w[j]);
        c->cY[j] = (float)(gamma * u[j]);
      }
    }
    if (lane == 0) {
      c->k = k;
      c->cg = (float)(-gamma);
    }
  } else if (take && tid < 64) {
    // the first slot not in use receives the next step
    int free_slot = -1;
    for (int s0 = 0; s0 <= m && free_slot < 0; s0 += 32) {
      bool used = s0 + lane > m;
      for (int q = 0; q < k; q++) used |= sl[q] == s0 + lane;
      const unsigned f = ~__ballot_sync(0xffffffffu, used);
      if (f) free_slot = s0 + __ffs(f) - 1;
    }
    if (lane == 0) {
      c->spare = free_slot;
      c->count = k;
      c->gamma = gamma;
    }
  } else if (take) {
    for (int q = tid - 64; q < k; q += kSolveThreads - 64) {
      c->order[q] = sl[k - 1 - q];
      // the candidate's column of S^T Y and row / column of Y^T Y
      SY[(size_t)sl[q] * ld + sp] = snew[q];
      YY[(size_t)sl[q] * ld + sp] = ynew[q];
      YY[(size_t)sp * ld + sl[q]] = ynew[q];
    }
  }
}

cudaError_t launch_lbfgs_solve(LbfgsCtl *c, int m, int first, double eps, double *SY, double *YY,
                               const float *g, const float *S, const float *Y, long long stride,
                               long long n, double *partials, cudaStream_t s) {
  const size_t smem = solve_smem(m);
  if (smem > 32 * 1024) {   // beyond what a launch may ask for without saying so
    const cudaError_t e =
        cudaFuncSetAttribute(lbfgs_solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)solve_smem(kMaxHistory));
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(true, lbfgs_solve_kernel, kSolveCtas, kSolveThreads, smem, s, c, m, first, eps, SY,
                    YY, g, S, Y, stride, n, partials);
}

__global__ void __launch_bounds__(256) lbfgs_combine_kernel(
    float *x, float *S, const float *Y, long long stride, float *g_prev, const float *g, long long n,
    const LbfgsCtl *c, int vec) {
  constexpr int U = 8;   // stored pairs whose loads are issued together
  pdl_begin();
  __shared__ float cS[kMaxHistory], cY[kMaxHistory];
  __shared__ long long off[kMaxHistory];
  __shared__ float cg_sh;
  __shared__ int k_sh;
  __shared__ long long sp_off;
  if (threadIdx.x == 0) {
    k_sh = c->k;
    cg_sh = c->cg;
    sp_off = (long long)c->spare * stride;
  }
  for (int i = threadIdx.x; i < kMaxHistory; i += blockDim.x) {
    cS[i] = c->cS[i];
    cY[i] = c->cY[i];
    off[i] = (long long)c->slot[i] * stride;
  }
  __syncthreads();
  const int k = k_sh;
  const float cg = cg_sh;
  float *snew = S + sp_off;
  const long long tstride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n4 = vec ? n / 4 : 0;
  for (long long v = t0; v < n4; v += tstride) {
    const float4 gv = reinterpret_cast<const float4 *>(g)[v];
    float4 xv = reinterpret_cast<float4 *>(x)[v];
    float4 d = make_float4(cg * gv.x, cg * gv.y, cg * gv.z, cg * gv.w);
    for (int j0 = 0; j0 < k; j0 += U) {
      float4 sv[U], yv[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (j0 + u < k) {
          sv[u] = reinterpret_cast<const float4 *>(S + off[j0 + u])[v];
          yv[u] = reinterpret_cast<const float4 *>(Y + off[j0 + u])[v];
        }
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (j0 + u < k) {
          const float a = cS[j0 + u], b = cY[j0 + u];
          d.x = fmaf(b, yv[u].x, fmaf(a, sv[u].x, d.x));
          d.y = fmaf(b, yv[u].y, fmaf(a, sv[u].y, d.y));
          d.z = fmaf(b, yv[u].z, fmaf(a, sv[u].z, d.z));
          d.w = fmaf(b, yv[u].w, fmaf(a, sv[u].w, d.w));
        }
      }
    }
    reinterpret_cast<float4 *>(snew)[v] = d;
    xv.x += d.x; xv.y += d.y; xv.z += d.z; xv.w += d.w;
    reinterpret_cast<float4 *>(x)[v] = xv;
    reinterpret_cast<float4 *>(g_prev)[v] = gv;
  }
  for (long long i = n4 * 4 + t0; i < n; i += tstride) {   // scalar path / tail
    const float gv = g[i];
    float d = cg * gv;
    for (int j = 0; j < k; j++) d = fmaf(cY[j], Y[off[j] + i], fmaf(cS[j], S[off[j] + i], d));
    snew[i] = d;
    x[i] += d;
    g_prev[i] = gv;
  }
}

void launch_lbfgs_combine(float *x, float *S, const float *Y, long long stride, float *g_prev,
                          const float *g, long long n, const LbfgsCtl *c, cudaStream_t s) {
  const int vec = aligned16(x) && aligned16(S) && aligned16(Y) && aligned16(g_prev) &&
                  aligned16(g) && stride % 4 == 0;
  long long b = (n / 4 + 255) / 256;
  const int grid = (int)(b < 152 * 8 ? (b > 0 ? b : 1) : 152 * 8);
  launch_pdl(true, lbfgs_combine_kernel, grid, 256, 0, s, x, S, Y, stride, g_prev, g, n, c, vec);
}

// ---- bicubic resampling ---------------------------------------------------------------------------
// Keys cubic convolution, a = -0.75, source coordinate (i + 0.5) * h / H - 0.5, clamped indices;
// rows are combined first, then columns.
__device__ __forceinline__ float keys_w(float t) {
  const float A = -0.75f;
  t = fabsf(t);
  if (t <= 1.f) return ((A + 2.f) * t - (A + 3.f)) * t * t + 1.f;
  if (t < 2.f) return ((A * t - 5.f * A) * t + 8.f * A) * t - 4.f * A;
  return 0.f;
}

// The weights of output coordinate i (s = source / output size): taps at source o - 1 .. o + 2
__device__ __forceinline__ int keys_taps(int i, float s, float *wt) {
  const float f = (i + 0.5f) * s - 0.5f;
  const int o = (int)floorf(f);
  const float t = f - o;
  wt[0] = keys_w(1.f + t);
  wt[1] = keys_w(t);
  wt[2] = keys_w(1.f - t);
  wt[3] = keys_w(2.f - t);
  return o;
}

// Enlarging (w <= W): a warp makes kBicX consecutive columns of up to R rows, all C channels. Bound:
// the store of the output; an output at a time (32 index divisions and weight evaluations, 16
// loads each) took 416 us for 1512 x 2016 -> 3024 x 4032, 3 channels, where the bytes take 27.
// Here a lane keeps the column weights of its four outputs for all rows and channels, the row
// weights serve three channels, and the rows are combined once per source column (not once per
// output and tap) into shared memory, from where every output takes its four columns:
// 64 us, with the L1 74 % busy. Lane l's outputs are columns l, l + 32, ... of the strip, so loads
// and stores are whole lines at any alignment. The same operations in the same order per output: the same bits.
// The rows are the CTA's (uniform base addresses, one 32-bit column offset per load).
constexpr int kBicX = 128, kBicSpan = 136;   // a strip reads at most kBicX + 1 + 3 source columns
constexpr int kBicWarps = 4;
__global__ void __launch_bounds__(32 * kBicWarps) bicubic_up_kernel(
    const float *__restrict__ x, int h, int w, float *__restrict__ out, int H, int W, int R) {
  constexpr int C = 3, NX = kBicX / 32, NS = (kBicSpan + 31) / 32;
  __shared__ float cols[kBicWarps][C][kBicSpan];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float sy = (float)h / (float)H, sx = (float)w / (float)W;
  const int X0 = (blockIdx.x * (blockDim.x >> 5) + warp) * kBicX;
  if (X0 >= W) return;
  float wx[NX][4];
  int slot[NX], xo[NS];
  float unused[4];
  const int first = keys_taps(X0, sx, unused) - 1;   // the strip's first source column
  const int span = min(keys_taps(min(X0 + kBicX, W) - 1, sx, unused) + 2 - first + 1, kBicSpan);
#pragma unroll
  for (int i = 0; i < NX; i++) slot[i] = keys_taps(X0 + lane + 32 * i, sx, wx[i]) - 1 - first;
#pragma unroll
  for (int q = 0; q < NS; q++) xo[q] = min(max(first + lane + 32 * q, 0), w - 1);
  const size_t plane = (size_t)h * w, oplane = (size_t)H * W;
  const int Y0 = blockIdx.y * R, Y1 = min(Y0 + R, H);
  for (int Y = Y0; Y < Y1; Y++) {
    float wy[4];
    const int iy = keys_taps(Y, sy, wy);
    const float *row[4];
#pragma unroll
    for (int k = 0; k < 4; k++) row[k] = x + (size_t)min(max(iy - 1 + k, 0), h - 1) * w;
    __syncwarp();   // the previous row's columns have been read
#pragma unroll
    for (int q = 0; q < NS; q++) {
      if (32 * q >= span) break;
      float v[C][4];
#pragma unroll
      for (int c = 0; c < C; c++)
#pragma unroll
        for (int k = 0; k < 4; k++) v[c][k] = __ldg(row[k] + c * plane + xo[q]);
#pragma unroll
      for (int c = 0; c < C; c++) {
        float col = 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) col = fmaf(wy[k], v[c][k], col);
        if (lane + 32 * q < kBicSpan) cols[warp][c][lane + 32 * q] = col;
      }
    }
    __syncwarp();
    float *o = out + (size_t)Y * W;
#pragma unroll
    for (int i = 0; i < NX; i++) {
      const int X = X0 + lane + 32 * i;
      if (X < W) {
#pragma unroll
        for (int c = 0; c < C; c++) {
          float acc = 0.f;
#pragma unroll
          for (int j = 0; j < 4; j++) acc = fmaf(wx[i][j], cols[warp][c][slot[i] + j], acc);
          o[c * oplane + X] = acc;
        }
      }
    }
  }
}

// Any ratio (reducing: w > W, where a strip's source columns have no useful bound)
__global__ void bicubic_kernel(const float *__restrict__ x, int C, int h, int w,
                               float *__restrict__ out, int H, int W) {
  const long long n = (long long)C * H * W;
  const float sy = (float)h / (float)H, sx = (float)w / (float)W;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int X = (int)(i % W);
    const int Y = (int)((i / W) % H);
    const int c = (int)(i / ((long long)W * H));
    float wy[4], wx[4];
    const int iy = keys_taps(Y, sy, wy), ix = keys_taps(X, sx, wx);
    const float *src = x + (size_t)c * h * w;
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int xx = min(max(ix - 1 + j, 0), w - 1);
      float col = 0.f;
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int yy = min(max(iy - 1 + k, 0), h - 1);
        col = fmaf(wy[k], src[(size_t)yy * w + xx], col);
      }
      acc = fmaf(wx[j], col, acc);
    }
    out[i] = acc;
  }
}

void launch_bicubic(const float *x, int C, int h, int w, float *out, int H, int W,
                    cudaStream_t s) {
  if (C == 3 && w <= W) {
    // rows per CTA: eight (the strips' setup is spread over them) while that leaves at least
    // four CTAs per SM
    const int strips = (W + kBicX - 1) / kBicX, warps = strips < kBicWarps ? strips : kBicWarps;
    const int gx = (strips + warps - 1) / warps;
    int R = 8;
    while (R > 1 && (long long)gx * ((H + R - 1) / R) < 4 * 152) R /= 2;
    const int gy = (H + R - 1) / R;
    if (gy <= 65535) {
      bicubic_up_kernel<<<dim3(gx, gy), 32 * warps, 0, s>>>(x, h, w, out, H, W, R);
      return;
    }
  }
  long long n = (long long)C * H * W;
  long long b = (n + 255) / 256;
  int grid = (int)(b < 152 * 32 ? b : 152 * 32);
  bicubic_kernel<<<grid > 0 ? grid : 1, 256, 0, s>>>(x, C, h, w, out, H, W);
}

// ---- area-average downscaling (adaptive average pooling) ---------------------------------------
// out[c][Y][X] = mean of x[c][y][x] over y in [floor(Y h / H), ceil((Y+1) h / H)) and
// x in [floor(X w / W), ceil((X+1) w / W)): the downscaling of (u, v) in Algorithm 2.
// Bound: the read of the source. With a double sum and a double division per output it was the
// FP64 unit (two operations per SM and clock: 146 us for 2113 x 2660 -> 1057 x 1330, 3 channels,
// whose bytes take 12), then 64-bit index divisions. A thread now keeps one column's bounds for R
// rows and all channels, the rows' bounds are made once per CTA, and the FP32 row sums are added
// in compensated FP32 and divided with a remainder step: the quotient is within 2^-46 of the
// exact one before it is rounded to FP32; with windows of at most 3 x 3 (a factor up to 2) or
// 5 x 5 their loads are issued together (area_kernel). 19 us with the source in L2.
__device__ __noinline__ float area_mean64(const float *src, int w, int y0, int y1, int x0, int x1) {
  double acc = 0.0;
  for (int y = y0; y < y1; y++) {
    float row = 0.f;
    for (int xx = x0; xx < x1; xx++) row += src[(size_t)y * w + xx];
    acc += (double)row;
  }
  return (float)(acc / ((double)(y1 - y0) * (double)(x1 - x0)));
}

// sum / cnt rounded once: q is within 2 ulp, its remainder exact (no contraction into q's product)
__device__ __forceinline__ float area_divide(const Sum &acc, float cnt, float inv) {
  const float q = __fmul_rn(acc.s, inv);
  return __fadd_rn(q, __fmul_rn(fmaf(-q, cnt, acc.s) + acc.c, inv));
}

constexpr int kAreaThreads = 128, kAreaRows = 8;
// Three channels, no window larger than NW x NW: the loads of an output's windows in all channels are
// issued together
template <int NW>
__global__ void __launch_bounds__(kAreaThreads) area_kernel(const float *__restrict__ x, int h,
                                                            int w, float *__restrict__ out, int H,
                                                            int W, int R) {
  __shared__ int ya[kAreaRows], yb[kAreaRows];
  const int X = blockIdx.x * kAreaThreads + threadIdx.x;
  for (long long Y0 = (long long)blockIdx.y * R; Y0 < H; Y0 += (long long)gridDim.y * R) {
    const int rows = (int)min((long long)R, H - Y0);
    __syncthreads();
    if (threadIdx.x < rows) {
      const long long Y = Y0 + threadIdx.x;
      ya[threadIdx.x] = (int)(Y * h / H);
      yb[threadIdx.x] = (int)(((Y + 1) * h + H - 1) / H);
    }
    __syncthreads();
    if (X >= W) continue;
    const int x0 = (int)((long long)X * w / W), x1 = (int)(((long long)(X + 1) * w + W - 1) / W);
    for (int r = 0; r < rows; r++) {
      const int y0 = ya[r], y1 = yb[r];
      const float cnt = (float)(y1 - y0) * (float)(x1 - x0), inv = 1.f / cnt;
      float *o = out + (size_t)(Y0 + r) * W + X;
      float v[3][NW][NW];
#pragma unroll
      for (int c = 0; c < 3; c++)
#pragma unroll
        for (int j = 0; j < NW; j++)
#pragma unroll
          for (int k = 0; k < NW; k++)
            v[c][j][k] = y0 + j < y1 && x0 + k < x1
                             ? __ldg(x + ((size_t)c * h + y0 + j) * w + x0 + k)
                             : 0.f;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        Sum acc{0.f, 0.f};
#pragma unroll
        for (int j = 0; j < NW; j++) {
          float row = 0.f;
#pragma unroll
          for (int k = 0; k < NW; k++) row += v[c][j][k];
          acc.add(row);
        }
        float m = area_divide(acc, cnt, inv);
        if (!(fabsf(acc.s) <= FLT_MAX))   // an infinite or overflowing sum
          m = area_mean64(x + (size_t)c * h * w, w, y0, y1, x0, x1);
        o[(size_t)c * H * W] = m;
      }
    }
  }
}

// Any window: a thread per output, consecutive outputs of a channel (grid y) in consecutive threads
// whatever the width. Bound: the chain of loads and adds of a window, so three CTAs of threads in four
// of what an SM holds (with all of them the registers spill); the rows' bounds are made once per CTA,
// the columns' without 64-bit divisions where W w fits 32 bits. A thread per output with FP64 sums
// took 45 us for 3024 x 4032 -> 378 x 504 and 139 for 6048 x 8064 -> 756 x 1008, a thread per three
// channels and up to eight rows 51 and 214; this 40 and 127.
constexpr int kAreaAnyThreads = 128;
__global__ void __launch_bounds__(kAreaAnyThreads, 12) area_any_kernel(const float *__restrict__ x,
                                                                      int h, int w,
                                                                      float *__restrict__ out,
                                                                      int H, int W, int narrow) {
  __shared__ int ya[kAreaAnyThreads + 1], yb[kAreaAnyThreads + 1];
  const long long i0 = (long long)blockIdx.x * kAreaAnyThreads, n = (long long)H * W;
  const int row0 = (int)(i0 / W);
  const unsigned at = (unsigned)(i0 - (long long)row0 * W) + threadIdx.x, r = at / (unsigned)W;
  // (rows row0 .. row0 + the last thread's r, at most kAreaAnyThreads + 1)
  const unsigned rows = (at - threadIdx.x + kAreaAnyThreads - 1) / (unsigned)W + 1;
  for (unsigned q = threadIdx.x; q < rows; q += kAreaAnyThreads) {
    const long long Y = row0 + (long long)q;
    ya[q] = (int)(Y * h / H);
    yb[q] = (int)(((Y + 1) * h + H - 1) / H);
  }
  __syncthreads();
  if (i0 + threadIdx.x >= n) return;
  const unsigned X = at - r * W;
  int x0, x1;
  if (narrow) {
    x0 = (int)(X * w / (unsigned)W);
    x1 = (int)(((X + 1) * w + W - 1) / (unsigned)W);
  } else {
    x0 = (int)((long long)X * w / W);
    x1 = (int)(((long long)(X + 1) * w + W - 1) / W);
  }
  const int ny = yb[r] - ya[r], nx = x1 - x0;
  const float *p = x + ((size_t)blockIdx.y * h + ya[r]) * w + x0;
  const float cnt = (float)ny * (float)nx;
  float m;
  if (cnt < 16777216.f) {
    Sum acc{0.f, 0.f};
    for (int y = 0; y < ny; y++, p += w) {
      float row = 0.f;
      for (int k = 0; k < nx; k++) row += __ldg(p + k);
      acc.add(row);
    }
    m = area_divide(acc, cnt, 1.f / cnt);
    if (!(fabsf(acc.s) <= FLT_MAX))   // (as above)
      m = area_mean64(p - (size_t)ny * w, w, 0, ny, 0, nx);
  } else {   // a count that FP32 does not hold
    m = area_mean64(p, w, 0, ny, 0, nx);
  }
  out[(size_t)blockIdx.y * n + i0 + threadIdx.x] = m;
}

void launch_area(const float *x, int C, int h, int w, float *out, int H, int W, cudaStream_t s) {
  // a window spans at most ceil(h / H) + 1 rows (ceil(h / H) when H divides h)
  const int ny = (h + H - 1) / H + (h % H ? 1 : 0), nx = (w + W - 1) / W + (w % W ? 1 : 0);
  if (C != 3 || ny > 5 || nx > 5) {
    const int narrow = (long long)(W + 1LL) * w + W < (1LL << 32);
    const unsigned ctas = (unsigned)(((long long)H * W + kAreaAnyThreads - 1) / kAreaAnyThreads);
    area_any_kernel<<<dim3(ctas, C), kAreaAnyThreads, 0, s>>>(x, h, w, out, H, W, narrow);
    return;
  }
  const int gx = (W + kAreaThreads - 1) / kAreaThreads;
  int R = kAreaRows;   // rows per CTA, fewer where that leaves less than eight CTAs per SM
  while (R > 1 && (long long)gx * ((H + R - 1) / R) < 8 * 152) R /= 2;
  const int gy = (H + R - 1) / R;
  const dim3 grid(gx, gy < 65535 ? gy : 65535);
  if (ny <= 3 && nx <= 3)
    area_kernel<3><<<grid, kAreaThreads, 0, s>>>(x, h, w, out, H, W, R);
  else
    area_kernel<5><<<grid, kAreaThreads, 0, s>>>(x, h, w, out, H, W, R);
}

}  // namespace nst
