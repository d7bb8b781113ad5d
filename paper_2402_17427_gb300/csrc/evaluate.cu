// Evaluation with colour correction (paper Sec. 5.1, "Metrics"): a per-image least-squares
// affine colour map fitted in centred form (channel means, then centred second moments; FP32
// per thread, double-floats across threads and blocks, Cholesky in FP64), the corrected image clipped to
// [0, 1], then PSNR (peak 1) and the loss's SSIM on the corrected image.
//
// Five launches.  Each streaming pass leaves one row of partial sums a block; the blocks of the next
// pass add those rows up themselves (one 456-row column a warp, all loads independent), so that no
// one-block reduction stands between two passes.  One thread adding 1,024 rows serially, as a kernel
// of its own, took 59 to 77 us each (three of them: 206 of 372 us at 1920 x 1080).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "doublefloat.cuh"
#include "internal.h"
#include "vg_common.cuh"

namespace vg {
namespace {

// Blocks of a streaming pass: three an SM of the 152, so that a pass is one wave and the next one
// has few rows to add (1,024 blocks: 37 us for the first pass, mostly six serial block sums a block).
constexpr int kEvalBlocks = 456;
constexpr int kEvalThreads = 256;
constexpr int kMeans = 6;      // mean r, g, b of the rendering and of the target
constexpr int kMoments = 15;   // 6 of the symmetric 3x3 covariance of x, 9 of the cross-covariance x y^T

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A warp's sum of any values: where double-floats give no finite one (their error terms make a NaN of
// every infinity), what FP32 additions leave.
__device__ __forceinline__ dd warp_sum_any(dd v) {
  const dd t = warp_sum_dd(v);
  if (__all_sync(0xffffffffu, fabsf(t.h) < INFINITY)) return t;
  float s = v.h;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return dd(s);
}

// The block's sums of K per-thread values: one row of `part`.  In double-floats: an FP64 addition holds the
// SM's pipe for 16 clocks a warp, and 15 moments of 8 warps in FP64 took 20 us of the 44 us pass.
// Scaled by 2^-17, since fewer than 2^17 threads add up: no sum of finite values leaves FP32's range.
constexpr float kSumScale = 1.f / 131072.f;
static_assert(kEvalBlocks * kEvalThreads <= 131072, "the scale covers every thread");
template <int K>
__device__ __forceinline__ void write_row(const float (&m)[K], float2* __restrict__ part) {
  __shared__ float2 sm[kEvalThreads / 32][K];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const dd t = warp_sum_any(dd(m[k] * kSumScale));
    if (lane == 0) sm[w][k] = make_float2(t.h, t.l);
  }
  __syncthreads();
  if (threadIdx.x < K) {
    dd t(0.f);
#pragma unroll
    for (int j = 0; j < kEvalThreads / 32; ++j) t = t + dd(sm[j][threadIdx.x].x, sm[j][threadIdx.x].y);
    if (!(fabsf(t.h) < INFINITY)) {
      t = dd(0.f);
      for (int j = 0; j < kEvalThreads / 32; ++j) t.h += sm[j][threadIdx.x].x;
    }
    part[(size_t)blockIdx.x * K + threadIdx.x] = make_float2(t.h, t.l);
  }
}

// tot[k] = sum over the nb rows of `part`, by every block that needs it: a warp takes columns
// w, w + 8, ...  Ends with a block barrier.
template <int K>
__device__ __forceinline__ void sum_rows(const float2* __restrict__ part, int nb, double* tot /*shared [K]*/) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int k = w; k < K; k += kEvalThreads / 32) {
    dd t(0.f);
#pragma unroll 5
    for (int b = lane; b < nb; b += 32) {
      const float2 v = part[(size_t)b * K + k];
      t = t + dd(v.x, v.y);
    }
    if (!(fabsf(t.h) < INFINITY)) {
      t = dd(0.f);
      for (int b = lane; b < nb; b += 32) t.h += part[(size_t)b * K + k].x;
    }
    t = warp_sum_any(t);
    if (lane == 0) tot[k] = ((double)t.h + (double)t.l) / (double)kSumScale;
  }
  __syncthreads();
}

// body(x, y, p, n): the three channels of rendering and target at pixels p .. p + n - 1, n = 4 but
// at the image's end.  WIDE: 16-byte loads, where every plane starts on a 16-byte boundary and the
// pixel count is a multiple of 4; else the same four pixels by scalar loads (their lines stay in L1).
template <bool WIDE, typename Body>
__device__ __forceinline__ void each_quad(const float* __restrict__ img, const float* __restrict__ tgt, long long npx,
                                          Body body) {
  for (long long p = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x); p < npx;
       p += 4 * (long long)gridDim.x * blockDim.x) {
    float x[3][4], y[3][4];
    const int n = WIDE ? 4 : (int)(npx - p < 4 ? npx - p : 4);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if constexpr (WIDE) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(img + c * npx + p));
        const float4 b = __ldg(reinterpret_cast<const float4*>(tgt + c * npx + p));
        x[c][0] = a.x; x[c][1] = a.y; x[c][2] = a.z; x[c][3] = a.w;
        y[c][0] = b.x; y[c][1] = b.y; y[c][2] = b.z; y[c][3] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[c][j] = j < n ? __ldg(img + c * npx + p + j) : 0.f;
          y[c][j] = j < n ? __ldg(tgt + c * npx + p + j) : 0.f;
        }
      }
    }
    body(x, y, p, n);
  }
}

// pass 1: channel sums of the rendering and the target
template <bool WIDE>
__global__ void __launch_bounds__(kEvalThreads) cc_sums(const float* __restrict__ img, const float* __restrict__ tgt,
                                                        long long npx, float2* __restrict__ part) {
  pdl_enter();
  float m[kMeans] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  each_quad<WIDE>(img, tgt, npx, [&](const float (&x)[3][4], const float (&y)[3][4], long long, int) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {   // absent pixels are 0
      m[c] += (x[c][0] + x[c][1]) + (x[c][2] + x[c][3]);
      m[3 + c] += (y[c][0] + y[c][1]) + (y[c][2] + y[c][3]);
    }
  });
  write_row<kMeans>(m, part);
}

// pass 2: centred second moments (products of centred values are accurate in FP32).  Block 0 keeps
// the means for the fit.
template <bool WIDE>
__global__ void __launch_bounds__(kEvalThreads) cc_moments(const float* __restrict__ img, const float* __restrict__ tgt,
                                                           long long npx, const float2* __restrict__ sums, int nb,
                                                           double* __restrict__ mean, float2* __restrict__ part) {
  pdl_enter();
  __shared__ double tot[kMeans];
  sum_rows<kMeans>(sums, nb, tot);
  float mu[kMeans];
#pragma unroll
  for (int k = 0; k < kMeans; ++k) mu[k] = (float)(tot[k] / (double)npx);
  if (blockIdx.x == 0 && threadIdx.x < kMeans) mean[threadIdx.x] = tot[threadIdx.x] / (double)npx;
  float m[kMoments];
#pragma unroll
  for (int k = 0; k < kMoments; ++k) m[k] = 0.f;
  each_quad<WIDE>(img, tgt, npx, [&](const float (&xs)[3][4], const float (&ys)[3][4], long long, int n) {
    float t[kMoments];     // this quad's sums, added to the thread's once: a quarter of the additions in series
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (e >= n) break;
      const float x[3] = {xs[0][e] - mu[0], xs[1][e] - mu[1], xs[2][e] - mu[2]};
      const float y[3] = {ys[0][e] - mu[3], ys[1][e] - mu[4], ys[2][e] - mu[5]};
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          const int k = i * 3 - i * (i - 1) / 2 + (j - i);   // upper-triangle slot of (i, j)
          t[k] = e == 0 ? x[i] * x[j] : fmaf(x[i], x[j], t[k]);
        }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) t[6 + 3 * i + c] = e == 0 ? x[i] * y[c] : fmaf(x[i], y[c], t[6 + 3 * i + c]);
    }
#pragma unroll
    for (int k = 0; k < kMoments; ++k) m[k] += t[k];
  });
  write_row<kMoments>(m, part);
}

// Least squares in centred form: Cov(x) A^T = Cov(x, y), b = mean(y) - A mean(x), by a Cholesky
// factorisation that drops a colour direction whose pivot falls below 1e-10 of the trace (its
// coefficient is 0: the remaining columns span the same space, so the fitted values are those of
// every least-squares solution; a constant rendering gets A = 0, b = mean(y)).
// coef = (A row-major, b); one thread, from the totals and the means.
__device__ void cc_solve(const double* tot, const double* mean, double* coef) {
  double C[3][3], K[3][3], L[3][3] = {{0}};
  for (int i = 0, k = 0; i < 3; ++i)
    for (int j = i; j < 3; ++j, ++k) C[i][j] = C[j][i] = tot[k];
  for (int i = 0; i < 3; ++i)
    for (int c = 0; c < 3; ++c) K[i][c] = tot[6 + 3 * i + c];
  const double tol = 1e-10 * (C[0][0] + C[1][1] + C[2][2]);
  bool live[3];
  for (int j = 0; j < 3; ++j) {
    double d = C[j][j];
    for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
    live[j] = d > tol && d > 0.0;
    L[j][j] = live[j] ? sqrt(d) : 0.0;
    for (int i = j + 1; i < 3; ++i) {
      double v = C[i][j];
      for (int k = 0; k < j; ++k) v -= L[i][k] * L[j][k];
      L[i][j] = live[j] ? v / L[j][j] : 0.0;
    }
  }
  double At[3][3];   // At[i][c] = A[c][i]
  for (int c = 0; c < 3; ++c) {
    double z[3];
    for (int i = 0; i < 3; ++i) {
      double v = K[i][c];
      for (int k = 0; k < i; ++k) v -= L[i][k] * z[k];
      z[i] = live[i] ? v / L[i][i] : 0.0;
    }
    for (int i = 2; i >= 0; --i) {
      double v = z[i];
      for (int k = i + 1; k < 3; ++k) v -= L[k][i] * At[k][c];
      At[i][c] = live[i] ? v / L[i][i] : 0.0;
    }
  }
  for (int c = 0; c < 3; ++c) {
    double b = mean[3 + c];
    for (int i = 0; i < 3; ++i) {
      coef[3 * c + i] = At[i][c];
      b -= At[i][c] * mean[i];
    }
    coef[9 + c] = b;
  }
}

// pass 3: every block solves the 3 x 3 system for itself (block 0 writes the map out), then the
// corrected image and its squared error.
template <bool WIDE>
__global__ void __launch_bounds__(kEvalThreads) cc_apply(const float* __restrict__ img, const float* __restrict__ tgt,
                                                         long long npx, const float2* __restrict__ mom, int nb,
                                                         const double* __restrict__ mean, float* __restrict__ corr,
                                                         float2* __restrict__ part, float* __restrict__ out) {
  pdl_enter();
  __shared__ double tot[kMoments], coef[12];
  sum_rows<kMoments>(mom, nb, tot);
  if (threadIdx.x == 0) cc_solve(tot, mean, coef);
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x < 12) out[2 + threadIdx.x] = (float)coef[threadIdx.x];
  float A[9], b[3];
#pragma unroll
  for (int k = 0; k < 9; ++k) A[k] = (float)coef[k];
#pragma unroll
  for (int c = 0; c < 3; ++c) b[c] = (float)coef[9 + c];
  float se[1] = {0.f};
  each_quad<WIDE>(img, tgt, npx, [&](const float (&x)[3][4], const float (&y)[3][4], long long p, int n) {
    float t = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[e] = fminf(1.f, fmaxf(0.f, fmaf(A[3 * c], x[0][e], fmaf(A[3 * c + 1], x[1][e], fmaf(A[3 * c + 2], x[2][e], b[c])))));
        const float d = e < n ? v[e] - y[c][e] : 0.f;
        t = fmaf(d, d, t);
      }
      if constexpr (WIDE) {
        *reinterpret_cast<float4*>(corr + c * npx + p) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < n) corr[c * npx + p + e] = v[e];
      }
    }
    se[0] += t;
  });
  write_row<1>(se, part);
}

// PSNR from the squared-error rows, SSIM from the moment pass's partial sums (sum S, sum |x - y|).
__global__ void __launch_bounds__(1024) cc_finish(const float2* __restrict__ sq, int nb, const double* __restrict__ ssim,
                                                  int ns, long long n, float* __restrict__ out) {
  pdl_enter();
  __shared__ double sm[2][32];
  double e = 0.0, t = 0.0;
  for (int b = threadIdx.x; b < nb; b += 1024) e += (double)sq[b].x + (double)sq[b].y;
#pragma unroll 4
  for (int b = threadIdx.x; b < ns; b += 1024) t += ssim[2 * (size_t)b];
  e = warp_sum_d(e);
  t = warp_sum_d(t);
  if ((threadIdx.x & 31) == 0) {
    sm[0][threadIdx.x >> 5] = e;
    sm[1][threadIdx.x >> 5] = t;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  e = warp_sum_d(sm[0][threadIdx.x]);
  t = warp_sum_d(sm[1][threadIdx.x]);
  if (threadIdx.x != 0) return;
  const double mse = e / (double)kSumScale / (double)n;
  out[0] = mse > 0.0 ? (float)(-10.0 * log10(mse)) : INFINITY;
  out[1] = (float)(t / (double)n);
}

struct EvalLayout {
  size_t corr, sums, mean, mom, sq, ssim, total;
};

EvalLayout eval_layout(int W, int H) {
  EvalLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) { size_t at = o; o = align_up(o + b); return at; };
  const size_t px = (size_t)W * H;
  L.corr = take(3 * px * sizeof(float));
  L.sums = take((size_t)kEvalBlocks * kMeans * sizeof(float2));
  L.mean = take(kMeans * sizeof(double));
  L.mom = take((size_t)kEvalBlocks * kMoments * sizeof(float2));
  L.sq = take((size_t)kEvalBlocks * sizeof(float2));
  L.ssim = take((size_t)ssim_partials(W, H) * 2 * sizeof(double));
  L.total = o;
  return L;
}

template <bool WIDE>
cudaError_t launch_eval(const float* img, const float* target, int W, int H, const EvalLayout& L, char* ws, float* out,
                        cudaStream_t s) {
  const long long npx = (long long)W * H;
  const int nb = (int)std::min<long long>(kEvalBlocks, (npx + 4 * kEvalThreads - 1) / (4 * kEvalThreads));
  auto D = [&](size_t off) { return reinterpret_cast<double*>(ws + off); };
  auto P = [&](size_t off) { return reinterpret_cast<float2*>(ws + off); };
  float* corr = reinterpret_cast<float*>(ws + L.corr);
  note_launches(4);
  cc_sums<WIDE><<<nb, kEvalThreads, 0, s>>>(img, target, npx, P(L.sums));
  launch_pdl(cc_moments<WIDE>, nb, kEvalThreads, 0, s, img, target, npx, P(L.sums), nb, D(L.mean), P(L.mom));
  launch_pdl(cc_apply<WIDE>, nb, kEvalThreads, 0, s, img, target, npx, P(L.mom), nb, D(L.mean), corr, P(L.sq), out);
  const cudaError_t e = launch_ssim_value(corr, target, W, H, D(L.ssim), s);
  if (e != cudaSuccess) return e;
  launch_pdl(cc_finish, 1, 1024, 0, s, P(L.sq), nb, D(L.ssim), ssim_partials(W, H), 3 * npx, out);
  return cudaGetLastError();
}

}  // namespace
}  // namespace vg

using namespace vg;

extern "C" size_t vg_eval_workspace_bytes(int32_t width, int32_t height) {
  if (width <= 0 || height <= 0) return 0;
  return eval_layout(width, height).total;
}

extern "C" vg_status vg_eval_color_corrected(const float* img, const float* target, int32_t width, int32_t height,
                                             void* workspace, size_t workspace_bytes, float* out, vg_stream stream) {
  if (!img || !target || !workspace || !out || width <= 0 || height <= 0) return VG_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return VG_ERR_INVALID;
  const EvalLayout L = eval_layout(width, height);
  if (workspace_bytes < L.total) return VG_ERR_CAPACITY;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  // 16-byte loads need the images on 16-byte boundaries and planes of a multiple of 4 pixels
  const bool wide = ((reinterpret_cast<uintptr_t>(img) | reinterpret_cast<uintptr_t>(target)) & 15u) == 0 &&
                    ((long long)width * height) % 4 == 0;
  const cudaError_t e = wide ? launch_eval<true>(img, target, width, height, L, ws, out, s)
                             : launch_eval<false>(img, target, width, height, L, ws, out, s);
  return e == cudaSuccess ? VG_OK : VG_ERR_CUDA;
}
