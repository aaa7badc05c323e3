// nst_api_opt.cu -- C ABI of the optimiser step (L-BFGS, Section 3.1 / Section 5.1) and of the
// multiscale initialisation (Algorithm 2).
#include <cstring>
#include <string>

#include "../../include/nst.h"
#include "nst_kernels.h"
#include "nst_lbfgs_dev.h"

using namespace nst;

struct nst_lbfgs {
  long long n = 0;
  long long stride = 0;              // slot stride: n rounded up to 64 floats (256-byte slots)
  int m = 0;
  long long iters = 0;
  float *S = nullptr, *Y = nullptr;  // [m+1][n] history slots (device pointers)
  float *S_host = nullptr, *Y_host = nullptr;  // host allocations when the history lives there
  float *g_prev = nullptr;
  double *SY = nullptr, *YY = nullptr;   // [m+1][m+1] s_a . y_b and y_a . y_b by slot
  double *partials = nullptr;
  LbfgsCtl *ctl = nullptr;
  void *mem = nullptr;               // the one device allocation that holds all of the above
};

namespace {
constexpr double kCurvEps = 1e-10;
}

extern "C" {

nst_status nst_lbfgs_create(nst_lbfgs **out, long long n, int m) {
  return nst_lbfgs_create_ex(out, n, m, 0);
}

nst_status nst_lbfgs_create_ex(nst_lbfgs **out, long long n, int m, int flags) {
  if (!out || n <= 0 || m < 1 || m > kMaxHistory || (flags & ~NST_LBFGS_HOST_HISTORY))
    return NST_ERR_INVALID_ARG;
  *out = nullptr;
  nst_lbfgs *st = new nst_lbfgs();
  st->n = n;
  st->m = m;
  st->stride = (n + 63) / 64 * 64;
  const size_t slots = (size_t)(m + 1);
  const size_t hist = slots * st->stride * sizeof(float);
  // One device allocation (six took most of a small run's time). Nothing but the control block
  // needs a value: a slot, a kept gradient and an entry of S^T Y or Y^T Y are written before they
  // are read.
  const bool host = (flags & NST_LBFGS_HOST_HISTORY) != 0;
  size_t bytes = 0;
  auto take = [&](size_t n_bytes) {
    const size_t at = bytes;
    bytes += (n_bytes + 255) / 256 * 256;
    return at;
  };
  const size_t o_ctl = take(sizeof(LbfgsCtl)), o_sy = take(slots * slots * sizeof(double)),
               o_yy = take(slots * slots * sizeof(double)),
               o_part = take(lbfgs_partials_count(m) * sizeof(double)),
               o_g = take(n * sizeof(float)), o_s = take(host ? 0 : hist), o_y = take(host ? 0 : hist);
  bool ok = cudaMalloc(&st->mem, bytes) == cudaSuccess;
  if (ok) {
    char *p = static_cast<char *>(st->mem);
    st->ctl = reinterpret_cast<LbfgsCtl *>(p + o_ctl);
    st->SY = reinterpret_cast<double *>(p + o_sy);
    st->YY = reinterpret_cast<double *>(p + o_yy);
    st->partials = reinterpret_cast<double *>(p + o_part);
    st->g_prev = reinterpret_cast<float *>(p + o_g);
    st->S = reinterpret_cast<float *>(p + o_s);
    st->Y = reinterpret_cast<float *>(p + o_y);
  }
  if (ok && host)
    ok = cudaHostAlloc(&st->S_host, hist, cudaHostAllocMapped | cudaHostAllocPortable) ==
             cudaSuccess &&
         cudaHostAlloc(&st->Y_host, hist, cudaHostAllocMapped | cudaHostAllocPortable) ==
             cudaSuccess &&
         cudaHostGetDevicePointer(&st->S, st->S_host, 0) == cudaSuccess &&
         cudaHostGetDevicePointer(&st->Y, st->Y_host, 0) == cudaSuccess;
  if (!ok) {
    nst_lbfgs_destroy(st);
    return NST_ERR_OOM;
  }
  LbfgsCtl c;
  std::memset(&c, 0, sizeof(c));
  c.gamma = 1.0;
  c.count = 0;
  c.spare = 0;
  for (int i = 0; i < kMaxHistory; i++) c.order[i] = -1;
  cudaMemcpy(st->ctl, &c, sizeof(c), cudaMemcpyHostToDevice);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    nst_lbfgs_destroy(st);
    return NST_ERR_CUDA;
  }
  *out = st;
  return NST_OK;
}

nst_status nst_lbfgs_destroy(nst_lbfgs *st) {
  if (!st) return NST_OK;
  cudaDeviceSynchronize();
  if (st->S_host) cudaFreeHost(st->S_host);
  if (st->Y_host) cudaFreeHost(st->Y_host);
  cudaFree(st->mem);
  delete st;
  return NST_OK;
}

nst_status nst_lbfgs_step(nst_lbfgs *st, float *x, const float *g, void *stream) {
  if (!st || !x || !g) return NST_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int first = st->iters == 0 ? 1 : 0;
  // 1. one pass over g, g_prev and every stored vector: y = g - g_prev into the spare slot and
  //    all dot products of the compact representation (first call: ||g||_1)
  launch_lbfgs_dots(g, st->g_prev, st->S, st->Y, st->stride, st->n, st->ctl, st->m, first,
                    st->partials, s);
  // 2. curvature test, history update, S^T Y / Y^T Y update, small solve (one CTA)
  if (launch_lbfgs_solve(st->ctl, st->m, first, kCurvEps, st->SY, st->YY, g, st->S, st->Y,
                         st->stride, st->n, st->partials, s) != cudaSuccess)
    return NST_ERR_CUDA;
  // 3. one pass forming s = t d (into the spare slot), x += s, g_prev = g
  launch_lbfgs_combine(x, st->S, st->Y, st->stride, st->g_prev, g, st->n, st->ctl, s);
  if (cudaGetLastError() != cudaSuccess) return NST_ERR_CUDA;
  st->iters++;
  return NST_OK;
}

nst_status nst_lbfgs_info(nst_lbfgs *st, int *pairs, long long *iters, void *stream) {
  if (!st) return NST_ERR_INVALID_ARG;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return NST_ERR_CUDA;
  LbfgsCtl c;
  if (cudaMemcpy(&c, st->ctl, sizeof(c), cudaMemcpyDeviceToHost) != cudaSuccess)
    return NST_ERR_CUDA;
  if (pairs) *pairs = c.count;
  if (iters) *iters = st->iters;
  return NST_OK;
}

nst_status nst_upsample_init(const float *xs, int h, int w, float *x, int H, int W,
                             void *stream) {
  if (!xs || !x || h < 1 || w < 1 || H < 1 || W < 1) return NST_ERR_INVALID_ARG;
  launch_bicubic(xs, 3, h, w, x, H, W, (cudaStream_t)stream);
  return cudaGetLastError() == cudaSuccess ? NST_OK : NST_ERR_CUDA;
}

nst_status nst_downscale(const float *x, int h, int w, float *out, int H, int W, void *stream) {
  if (!x || !out || h < 1 || w < 1 || H < 1 || W < 1 || H > h || W > w) return NST_ERR_INVALID_ARG;
  launch_area(x, 3, h, w, out, H, W, (cudaStream_t)stream);
  return cudaGetLastError() == cudaSuccess ? NST_OK : NST_ERR_CUDA;
}

}  // extern "C"
