// Per-Gaussian projection (EWA splatting + spherical-harmonic colour) and its adjoint.
//
// Paper Sec. 3: each 3D Gaussian (position, anisotropic covariance, opacity, SH colour) is
// projected to the image as a 2D Gaussian; R is differentiable.  One thread per Gaussian.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "vg_common.cuh"

namespace vg {
namespace {

// Real spherical harmonics with the Condon-Shortley phase, index l^2 + l + m, written as
// polynomials in the unit direction (x, y, z).  Constants: sqrt((2l+1)/(4 pi) (l-m)!/(l+m)!)
// times the Legendre-derivative factors, e.g. C1 = sqrt(3/(4 pi)), C2a = sqrt(15/pi)/2,
// C2b = sqrt(5/pi)/4, C2c = sqrt(15/pi)/4, C3a = sqrt(35/(32 pi)), C3b = sqrt(105/pi)/2,
// C3c = sqrt(21/(32 pi)), C3d = sqrt(7/pi)/4, C3e = sqrt(105/pi)/4.
constexpr float kC0 = 0.28209479177387814f;
constexpr float kC1 = 0.48860251190291992f;
constexpr float kC2a = 1.0925484305920792f;
constexpr float kC2b = 0.31539156525252005f;
constexpr float kC2c = 0.54627421529603959f;
constexpr float kC3a = 0.59004358992664352f;
constexpr float kC3b = 2.8906114426405538f;
constexpr float kC3c = 0.45704579946446577f;
constexpr float kC3d = 0.37317633259011540f;
constexpr float kC3e = 1.4453057213202769f;

template <int DEG>
__device__ __forceinline__ void sh_basis(float x, float y, float z, float* Y) {
  Y[0] = kC0;
  if (DEG >= 1) {
    Y[1] = -kC1 * y;
    Y[2] = kC1 * z;
    Y[3] = -kC1 * x;
  }
  if (DEG >= 2) {
    float xx = x * x, yy = y * y, zz = z * z;
    Y[4] = kC2a * x * y;
    Y[5] = -kC2a * y * z;
    Y[6] = kC2b * (2.f * zz - xx - yy);
    Y[7] = -kC2a * x * z;
    Y[8] = kC2c * (xx - yy);
    if (DEG >= 3) {
      Y[9] = -kC3a * y * (3.f * xx - yy);
      Y[10] = kC3b * x * y * z;
      Y[11] = -kC3c * y * (4.f * zz - xx - yy);
      Y[12] = kC3d * z * (2.f * zz - 3.f * xx - 3.f * yy);
      Y[13] = -kC3c * x * (4.f * zz - xx - yy);
      Y[14] = kC3e * z * (xx - yy);
      Y[15] = -kC3a * x * (xx - 3.f * yy);
    }
  }
}

// Gradient of each basis polynomial with respect to (x, y, z).
template <int DEG>
__device__ __forceinline__ void sh_basis_grad(float x, float y, float z, float (*G)[3]) {
  G[0][0] = G[0][1] = G[0][2] = 0.f;
  if (DEG >= 1) {
    G[1][0] = 0.f; G[1][1] = -kC1; G[1][2] = 0.f;
    G[2][0] = 0.f; G[2][1] = 0.f;  G[2][2] = kC1;
    G[3][0] = -kC1; G[3][1] = 0.f; G[3][2] = 0.f;
  }
  if (DEG >= 2) {
    float xx = x * x, yy = y * y, zz = z * z;
    G[4][0] = kC2a * y;        G[4][1] = kC2a * x;        G[4][2] = 0.f;
    G[5][0] = 0.f;             G[5][1] = -kC2a * z;       G[5][2] = -kC2a * y;
    G[6][0] = -2.f * kC2b * x; G[6][1] = -2.f * kC2b * y; G[6][2] = 4.f * kC2b * z;
    G[7][0] = -kC2a * z;       G[7][1] = 0.f;             G[7][2] = -kC2a * x;
    G[8][0] = 2.f * kC2c * x;  G[8][1] = -2.f * kC2c * y; G[8][2] = 0.f;
    if (DEG >= 3) {
      G[9][0] = -6.f * kC3a * x * y;  G[9][1] = -3.f * kC3a * (xx - yy); G[9][2] = 0.f;
      G[10][0] = kC3b * y * z;        G[10][1] = kC3b * x * z;           G[10][2] = kC3b * x * y;
      G[11][0] = 2.f * kC3c * x * y;  G[11][1] = -kC3c * (4.f * zz - xx - 3.f * yy); G[11][2] = -8.f * kC3c * y * z;
      G[12][0] = -6.f * kC3d * x * z; G[12][1] = -6.f * kC3d * y * z;    G[12][2] = kC3d * (6.f * zz - 3.f * xx - 3.f * yy);
      G[13][0] = -kC3c * (4.f * zz - 3.f * xx - yy); G[13][1] = 2.f * kC3c * x * y; G[13][2] = -8.f * kC3c * x * z;
      G[14][0] = 2.f * kC3e * x * z;  G[14][1] = -2.f * kC3e * y * z;    G[14][2] = kC3e * (xx - yy);
      G[15][0] = -3.f * kC3a * (xx - yy); G[15][1] = 6.f * kC3a * x * y; G[15][2] = 0.f;
    }
  }
}

// ---- double-float arithmetic (pairs hi + lo of FP32 numbers, error-free transformations) ----
// Used for the projected mean: R m + t cancels large terms at city scale, and FP32 alone loses
// ~1e-4 px there; the pair keeps ~1e-14 relative, at FP32 speed (FP64 is slow on this part).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}
// row . m + t as a double-float
__device__ __forceinline__ void df_dot3(const float* row, float t, const float* m, float& hi, float& lo) {
  float p0, e0, p1, e1, p2, e2, s, f0, f1, f2;
  two_prod(row[0], m[0], p0, e0);
  two_prod(row[1], m[1], p1, e1);
  two_prod(row[2], m[2], p2, e2);
  two_sum(t, p0, s, f0);
  two_sum(s, p1, s, f1);
  two_sum(s, p2, s, f2);
  const float l = __fadd_rn(__fadd_rn(__fadd_rn(e0, e1), e2), __fadd_rn(__fadd_rn(f0, f1), f2));
  fast_two_sum(s, l, hi, lo);
}
// f * (xh + xl) / (zh + zl) + c as a double-float
__device__ __forceinline__ void df_project(float xh, float xl, float zh, float zl, float f, float c, float& hi,
                                           float& lo) {
  const float q = __fdiv_rn(xh, zh);
  float ph, pl;
  two_prod(q, zh, ph, pl);
  // x - q z, where xh - ph is exact (the two are within a factor of two)
  const float r = __fadd_rn(__fsub_rn(__fsub_rn(xh, ph), pl), __fsub_rn(xl, __fmul_rn(q, zl)));
  const float ql = __fdiv_rn(r, zh);
  float ah, al, sh, se;
  two_prod(f, q, ah, al);
  two_sum(ah, c, sh, se);
  fast_two_sum(sh, __fadd_rn(__fadd_rn(se, al), __fmul_rn(f, ql)), hi, lo);
}

// Loads the K x 3 SH block of Gaussian i into registers (vector loads when 16-byte aligned).
template <int DEG>
__device__ __forceinline__ void load_sh(const float* __restrict__ sh, int i, float* c) {
  constexpr int K = (DEG + 1) * (DEG + 1);
  constexpr int F = 3 * K;
  const float* p = sh + (size_t)i * F;
  if constexpr (F % 4 == 0) {
    const float4* p4 = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int k = 0; k < F / 4; ++k) {
      float4 v = __ldg(p4 + k);
      c[4 * k] = v.x; c[4 * k + 1] = v.y; c[4 * k + 2] = v.z; c[4 * k + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < F; ++k) c[k] = __ldg(p + k);
  }
}

// Everything the projection computes that the adjoint needs again.
struct Proj {
  float m[3], p[3];
  float qn[4], qinv;      // normalised quaternion, 1/|q|
  float Rq[9], s[3];
  float Sig[6];           // 3D covariance, upper triangle: 00 01 02 11 12 22
  float T[6];             // J W, 2 x 3
  float A, B, C;          // 2D covariance (with dilation)
  float ca, cb, cc;       // conic (inverse 2D covariance)
  bool clx, cly;          // guard-band clamp active
  float xzc, yzc;         // clamped x/z, y/z
  float u, v, depth, r;
  bool valid;
};

// Projection of Gaussian i, whose mean the caller has put into P.m; log_scale(k) gives its k-th log-scale.
// The key-defining values (depth, u, v) follow the exact FP32 operation order stated for the sort keys;
// the rest is ordinary FP32.
template <typename LogScale>
__device__ __forceinline__ void project(const KGauss& g, const KCam& cm, const KOpts& op, int i, LogScale log_scale,
                                        Proj& P) {
  P.valid = false;
#pragma unroll
  for (int r = 0; r < 3; ++r)
    P.p[r] = __fmaf_rn(cm.R[3 * r], P.m[0], __fmaf_rn(cm.R[3 * r + 1], P.m[1], __fmaf_rn(cm.R[3 * r + 2], P.m[2], cm.t[r])));
  const float z = P.p[2];
  if (!(z > cm.near_plane)) return;
  const float xz = __fdiv_rn(P.p[0], z), yz = __fdiv_rn(P.p[1], z);
  P.depth = z;
  P.u = __fmaf_rn(cm.fx, xz, cm.cx);
  P.v = __fmaf_rn(cm.fy, yz, cm.cy);
  // rotation, scale, 3D covariance
  float4 q = __ldg(reinterpret_cast<const float4*>(g.quats) + i);
  float qq = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
  if (!(qq > 0.f)) return;
  P.qinv = rsqrtf(qq);
  P.qn[0] = q.x * P.qinv; P.qn[1] = q.y * P.qinv; P.qn[2] = q.z * P.qinv; P.qn[3] = q.w * P.qinv;
  const float w = P.qn[0], x = P.qn[1], y = P.qn[2], zq = P.qn[3];
  P.Rq[0] = 1.f - 2.f * (y * y + zq * zq); P.Rq[1] = 2.f * (x * y - w * zq);        P.Rq[2] = 2.f * (x * zq + w * y);
  P.Rq[3] = 2.f * (x * y + w * zq);        P.Rq[4] = 1.f - 2.f * (x * x + zq * zq); P.Rq[5] = 2.f * (y * zq - w * x);
  P.Rq[6] = 2.f * (x * zq - w * y);        P.Rq[7] = 2.f * (y * zq + w * x);        P.Rq[8] = 1.f - 2.f * (x * x + y * y);
#pragma unroll
  for (int k = 0; k < 3; ++k) P.s[k] = expf(log_scale(k));
  float M[9];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) M[3 * r + c] = P.Rq[3 * r + c] * P.s[c];
  P.Sig[0] = M[0] * M[0] + M[1] * M[1] + M[2] * M[2];
  P.Sig[1] = M[0] * M[3] + M[1] * M[4] + M[2] * M[5];
  P.Sig[2] = M[0] * M[6] + M[1] * M[7] + M[2] * M[8];
  P.Sig[3] = M[3] * M[3] + M[4] * M[4] + M[5] * M[5];
  P.Sig[4] = M[3] * M[6] + M[4] * M[7] + M[5] * M[8];
  P.Sig[5] = M[6] * M[6] + M[7] * M[7] + M[8] * M[8];
  // Jacobian of the pinhole map at the guard-band clamped point, T = J W
  P.xzc = fminf(cm.limx, fmaxf(-cm.limx, xz));
  P.yzc = fminf(cm.limy, fmaxf(-cm.limy, yz));
  P.clx = P.xzc != xz;
  P.cly = P.yzc != yz;
  const float iz = 1.f / z;
  const float j00 = cm.fx * iz, j02 = -cm.fx * P.xzc * iz, j11 = cm.fy * iz, j12 = -cm.fy * P.yzc * iz;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    P.T[c] = j00 * cm.R[c] + j02 * cm.R[6 + c];
    P.T[3 + c] = j11 * cm.R[3 + c] + j12 * cm.R[6 + c];
  }
  // 2D covariance T Sigma T^T + dilation I
  const float* S = P.Sig;
  float TS[2][3];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const float* t = P.T + 3 * a;
    TS[a][0] = t[0] * S[0] + t[1] * S[1] + t[2] * S[2];
    TS[a][1] = t[0] * S[1] + t[1] * S[3] + t[2] * S[4];
    TS[a][2] = t[0] * S[2] + t[1] * S[4] + t[2] * S[5];
  }
  P.A = TS[0][0] * P.T[0] + TS[0][1] * P.T[1] + TS[0][2] * P.T[2] + op.dilation;
  P.B = TS[0][0] * P.T[3] + TS[0][1] * P.T[4] + TS[0][2] * P.T[5];
  P.C = TS[1][0] * P.T[3] + TS[1][1] * P.T[4] + TS[1][2] * P.T[5] + op.dilation;
  // The fused form by name: visibility hangs on its sign, which must not depend on what else a kernel takes from
  // the determinant (where only the sign was used, the compiler compared the two rounded products, and needles
  // whose products round to the same value were culled).
  const float det = __fmaf_rn(P.A, P.C, -__fmul_rn(P.B, P.B));
  if (!(det > 0.f)) return;
  const float idet = 1.f / det;
  P.ca = P.C * idet;
  P.cb = -P.B * idet;
  P.cc = P.A * idet;
  // largest eigenvalue as mid + sqrt(((A - C) / 2)^2 + B^2): the same value as mid + sqrt(mid^2 -
  // det) without its cancellation for near-isotropic covariances (there mid^2 - det loses all
  // its bits in FP32 and r would err by ~1e-4 relative)
  const float mid = 0.5f * (P.A + P.C), hd = 0.5f * (P.A - P.C);
  const float lmax = mid + sqrtf(fmaf(hd, hd, P.B * P.B));
  P.r = 3.f * sqrtf(lmax);
  P.valid = true;
}

__device__ __forceinline__ void project(const KGauss& g, const KCam& cm, const KOpts& op, int i, Proj& P) {
#pragma unroll
  for (int k = 0; k < 3; ++k) P.m[k] = __ldg(g.means + 3 * i + k);
  project(g, cm, op, i, [&](int k) { return __ldg(g.log_scales + 3 * i + k); }, P);
}

// Whether a Gaussian may touch the image, from its mean and its log-scales alone: false only if
// project() and the rectangle rule would cull it.  lambda_max(T Sigma T^T) <= |T|_F^2 max(s)^2 bounds the
// radius; the margins (1e-3 relative, 0.01 px + 1e-6 (|u| + |cx|)) are far above the rounding of either side
// and above the errors of the approximate reciprocal, root and exponential (a few 1e-7; the exponential's
// grow with the exponent, to 1e-5 at scales of e^88).  Comparisons are written so that a NaN or an
// infinity passes on to project().
__device__ __forceinline__ bool may_touch(const KCam& cm, const KOpts& op, const float* m, const float* ls) {
  float p[3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
    p[r] = __fmaf_rn(cm.R[3 * r], m[0], __fmaf_rn(cm.R[3 * r + 1], m[1], __fmaf_rn(cm.R[3 * r + 2], m[2], cm.t[r])));
  const float z = p[2];
  if (!(z > cm.near_plane)) return false;
  const float smax = __expf(fmaxf(fmaxf(ls[0], ls[1]), ls[2]));
  const float iz = rcp_approx(z), xz = p[0] * iz, yz = p[1] * iz;
  const float u = fmaf(cm.fx, xz, cm.cx), v = fmaf(cm.fy, yz, cm.cy);
  const float xzc = fminf(cm.limx, fmaxf(-cm.limx, xz)), yzc = fminf(cm.limy, fmaxf(-cm.limy, yz));
  const float j00 = cm.fx * iz, j02 = -j00 * xzc, j11 = cm.fy * iz, j12 = -j11 * yzc;
  float f2 = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float a = j00 * cm.R[c] + j02 * cm.R[6 + c], b = j11 * cm.R[3 + c] + j12 * cm.R[6 + c];
    f2 = fmaf(a, a, fmaf(b, b, f2));
  }
  const float rb = 3.003f * sqrt_approx(fmaf(1.001f * f2, smax * smax, op.dilation)) + 0.01f;
  const float ru = fmaf(1e-6f, fabsf(u) + fabsf(cm.cx), rb), rv = fmaf(1e-6f, fabsf(v) + fabsf(cm.cy), rb);
  return !(u + ru < 0.f || u - ru > (float)(cm.W - 1) || v + rv < 0.f || v - rv > (float)(cm.H - 1));
}

// Projection, first part: the visible Gaussians of every run of 512, in index order, each as one
// entry (depth key, Gaussian, tile rectangle) in the run's own part of `entries`, and their number.
//
// Only ~1 in 5 Gaussians is visible (1 in 25 in the 20M-Gaussian city), in no order, so may_touch()
// first thins them out on 24 bytes a Gaussian; the candidates are packed densely in shared memory, and
// whole warps of them go through project().  No block waits for another: compact_kernel closes the gaps
// between the runs.  In one kernel with a look-back over the runs (and the spherical harmonics, which now
// follow in record_kernel) a block spent most of its ~19 us waiting: 963 us for the 20M Gaussians of the
// city and 58 us for 1M; with the harmonics moved out 550 and 44 us, without the look-back 283 and 22.
// What bounded it then was the latency of each block's loads (means, then scales, then the candidates'
// rows): the blocks are persistent now, and copy the next run's means and log-scales into shared memory
// (cp.async, 16 bytes where the run lies in one segment on a 16-byte boundary) while they work on this one.
constexpr int kCullThreads = 128, kCullItems = 4, kCullWarps = kCullThreads / 32, kCullBlocks = 8;
static_assert(kCullThreads * kCullItems == kCullRun, "a block takes one run");
__global__ void __launch_bounds__(kCullThreads, kCullBlocks) cull_kernel(const DevTables* __restrict__ tab,
                                                                         int total_n, int runs,
                                                                         uint4* __restrict__ entries,
                                                                         unsigned* __restrict__ counts,
                                                                         uint32_t* __restrict__ touched,
                                                                         float4* __restrict__ key_inputs) {
  pdl_enter();
  __shared__ __align__(16) float s_in[2][2][3 * kCullRun];   // [buffer][means, log-scales]
  __shared__ unsigned s_wc[2][kCullItems * kCullWarps];      // counts a warp (and item) leaves for the others
  __shared__ uint16_t s_cand[kCullRun];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // segment of a run's first Gaussian; complemented if the run reaches into the next one
  auto fetch = [&](int run, int buf) {
    const int base = run * kCullRun, last = min(total_n - 1, base + (kCullRun - 1));
    const int seg = find_seg(tab, base);
    const bool one = seg == tab->h.n_segs - 1 || tseg(tab, seg + 1).offset > last;
    const KSeg& sg = tseg(tab, seg);
    const float* m = sg.g.means + 3 * (size_t)(base - sg.offset);
    const float* ls = sg.g.log_scales + 3 * (size_t)(base - sg.offset);
    if (one && last - base == kCullRun - 1 &&
        ((reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(ls)) & 15u) == 0) {
#pragma unroll
      for (int k = 4 * tid; k < 3 * kCullRun; k += 4 * kCullThreads) {
        cp_async16(&s_in[buf][0][k], m + k);
        cp_async16(&s_in[buf][1][k], ls + k);
      }
    } else {
      for (int k = tid; k < 3 * (last - base + 1); k += kCullThreads) {
        const float *pm = m + k, *pl = ls + k;
        if (!one) {
          const int i = base + k / 3;
          const KSeg& si = tseg(tab, find_seg(tab, i));
          const size_t o = 3 * (size_t)(i - si.offset) + k % 3;
          pm = si.g.means + o;
          pl = si.g.log_scales + o;
        }
        cp_async4_zfill(&s_in[buf][0][k], pm, true);
        cp_async4_zfill(&s_in[buf][1][k], pl, true);
      }
    }
    return one ? seg : ~seg;
  };
  int seg_next = 0;
  if ((int)blockIdx.x < runs) seg_next = fetch(blockIdx.x, 0);
  cp_async_commit();
  int buf = 0;
  for (int run = blockIdx.x; run < runs; run += gridDim.x, buf ^= 1) {
    const int seg = seg_next;
    if (run + (int)gridDim.x < runs) seg_next = fetch(run + gridDim.x, buf ^ 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const float* const s_m = s_in[buf][0];
    const float* const s_ls = s_in[buf][1];
    const int base = run * kCullRun, last = min(total_n - 1, base + (kCullRun - 1));
    auto seg_of = [&](int i) -> const KSeg& { return tseg(tab, seg >= 0 ? seg : find_seg(tab, i)); };
    // 1. candidates
    unsigned votes[kCullItems];
#pragma unroll
    for (int j = 0; j < kCullItems; ++j) {
      const int k = j * kCullThreads + tid, i = base + k;
      bool c = false;
      if (i <= last) {
        const KView& vw = tview(tab, seg_of(i).view);
        c = key_inputs != nullptr || may_touch(vw.cam, vw.op, s_m + 3 * k, s_ls + 3 * k);
        if (!c) touched[i] = 0;
      }
      votes[j] = __ballot_sync(0xffffffffu, c);
      if (lane == 0) s_wc[0][j * kCullWarps + warp] = __popc(votes[j]);
    }
    __syncthreads();
    const uint32_t lt = lanemask_lt();
    int ncand = 0;
#pragma unroll
    for (int k = 0; k < kCullItems * kCullWarps; ++k) {      // counts in index order: item, then warp
      const int j = k / kCullWarps;
      if (k % kCullWarps == warp && (votes[j] >> lane & 1u))
        s_cand[ncand + __popc(votes[j] & lt)] = (uint16_t)(j * kCullThreads + tid);
      ncand += (int)s_wc[0][k];
    }
    __syncthreads();
    // 2. projection, tile rectangle and visibility of the candidates, the visible ones written in order
    unsigned tot = 0;
    for (int r = 0, odd = 1; r < ncand; r += kCullThreads, odd ^= 1) {
      bool vis = false;
      uint4 e = make_uint4(0u, 0u, 0u, 0u);
      if (r + tid < ncand) {
        const int k = s_cand[r + tid], i = base + k;
        const KSeg& sg = seg_of(i);
        const KView& vw = tview(tab, sg.view);
        Proj P;
#pragma unroll
        for (int a = 0; a < 3; ++a) P.m[a] = s_m[3 * k + a];
        project(sg.g, vw.cam, vw.op, i - sg.offset, [&](int a) { return s_ls[3 * k + a]; }, P);
        uint32_t cnt = 0;
        if (P.valid) {
          const int T = vw.op.tile;
          const int xlo = rect_lo(P.u, P.r, vw.cam.W), xhi = rect_hi(P.u, P.r, vw.cam.W);
          const int ylo = rect_lo(P.v, P.r, vw.cam.H), yhi = rect_hi(P.v, P.r, vw.cam.H);
          if (xlo <= xhi && ylo <= yhi) {
            const int tx0 = xlo / T, tx1 = xhi / T, ty0 = ylo / T, ty1 = yhi / T;
            cnt = (uint32_t)((tx1 - tx0 + 1) * (ty1 - ty0 + 1));
            vis = true;
            e = make_uint4(__float_as_uint(P.depth), (uint32_t)i, (uint32_t)tx0 | ((uint32_t)tx1 << 16),
                           (uint32_t)ty0 | ((uint32_t)ty1 << 16));
          }
        }
        touched[i] = cnt;
        if (key_inputs)
          key_inputs[i] = P.valid ? make_float4(P.u, P.v, P.r, P.depth) : make_float4(0.f, 0.f, -1.f, 0.f);
      }
      const unsigned vote = __ballot_sync(0xffffffffu, vis);
      if (lane == 0) s_wc[odd][warp] = __popc(vote);
      __syncthreads();                      // the other buffer is written in the next round
      unsigned at = tot + __popc(vote & lt);
#pragma unroll
      for (int w = 0; w < kCullWarps; ++w) {
        const unsigned c = s_wc[odd][w];
        if (w < warp) at += c;
        tot += c;
      }
      if (vis) entries[(size_t)base + at] = e;
    }
    if (tid == 0) counts[run] = tot;
    __syncthreads();                        // the buffers are free for the next run
  }
}

// Projection, second part: the runs' entries moved together in index order (slot = position among all
// visible Gaussians): depth keys and sort values (the slots), ids and rectangles, with the digit
// histograms and the range of the keys.  Each block owns consecutive runs and adds up the counts of
// the runs before it itself (L2 reads, a few us even for the 39K runs of 20M Gaussians), so there is
// neither a look-back nor a scan kernel.
constexpr int kCompactThreads = 256;
__global__ void __launch_bounds__(kCompactThreads) compact_kernel(const uint4* __restrict__ entries,
                                                                  const unsigned* __restrict__ counts, int runs,
                                                                  int per_block, uint2* __restrict__ rects,
                                                                  const Compact cp, WsHeader* __restrict__ hdr) {
  pdl_enter();
  __shared__ unsigned s_sm[8];
  __shared__ unsigned s_off[kCompactThreads];
  __shared__ unsigned s_h[kMaxPasses][kRadix];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int p = 0; p < kMaxPasses; ++p) s_h[p][tid] = 0;
  const int first = (int)blockIdx.x * per_block, end = min(runs, first + per_block);
  unsigned before = 0, all = 0;     // visible Gaussians before this block's runs, and in total
#pragma unroll 4
  for (int k = 4 * tid; k < runs; k += 4 * kCompactThreads) {
    const uint4 c = __ldg(reinterpret_cast<const uint4*>(counts + k));     // padded to 4
    const unsigned v[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (k + j < runs) all += v[j];
      if (k + j < first) before += v[j];
    }
  }
  unsigned total;
  block_exclusive_scan(all, &total, s_sm);
  unsigned base;
  block_exclusive_scan(before, &base, s_sm);
  if (blockIdx.x == 0 && tid == 0) hdr->visible = total;
  unsigned lo_key = 0xFFFFFFFFu, hi_key = 0u;
  for (int r0 = first; r0 < end; r0 += kCompactThreads) {
    unsigned sum;
    s_off[tid] = base + block_exclusive_scan(r0 + tid < end ? counts[r0 + tid] : 0u, &sum, s_sm);
    __syncthreads();
    base += sum;
    for (int r = r0 + warp; r < min(end, r0 + kCompactThreads); r += kCompactThreads / 32) {
      const unsigned o = s_off[r - r0];
      const unsigned n = (r + 1 - r0 < kCompactThreads ? s_off[r + 1 - r0] : base) - o;   // absent runs count 0
      for (unsigned k = lane; k < n; k += 32) {
        const uint4 e = __ldg(entries + (size_t)r * kCullRun + k);
        cp.vkeys[o + k] = e.x;
        cp.vvals[o + k] = o + k;
        cp.vis_ids[o + k] = e.y;
        rects[o + k] = make_uint2(e.z, e.w);
        lo_key = min(lo_key, e.x);
        hi_key = max(hi_key, e.x);
#pragma unroll
        for (int p = 0; p < kMaxPasses; ++p) atomicAdd(&s_h[p][(e.x >> (p * kRadixBits)) & (kRadix - 1)], 1u);
      }
    }
    __syncthreads();
  }
  // min / max depth key (they fix the bits the depth sort needs): one global atomic each a block
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo_key = min(lo_key, __shfl_xor_sync(0xffffffffu, lo_key, o));
    hi_key = max(hi_key, __shfl_xor_sync(0xffffffffu, hi_key, o));
  }
  __shared__ unsigned s_lo[kCompactThreads / 32], s_hi[kCompactThreads / 32];
  if (lane == 0) {
    s_lo[warp] = lo_key;
    s_hi[warp] = hi_key;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kCompactThreads / 32; ++w) {
      lo_key = min(lo_key, s_lo[w]);
      hi_key = max(hi_key, s_hi[w]);
    }
    if (lo_key <= hi_key) {
      atomicMin(&hdr->dmin, lo_key);
      atomicMax(&hdr->dmax, hi_key);
    }
  }
#pragma unroll
  for (int p = 0; p < kMaxPasses; ++p)
    if (s_h[p][tid]) atomicAdd(&cp.hist[p * kRadix + tid], s_h[p][tid]);
  // clear the look-back rows of the first depth-sort pass
  const size_t zero_words = (size_t)((total + kDepthTile - 1) / kDepthTile) * kRadix;
  for (size_t z = (size_t)blockIdx.x * kCompactThreads + tid; z < zero_words; z += (size_t)gridDim.x * kCompactThreads)
    cp.zero[z] = 0ull;
}

// Projection, third part: the splat record of every visible Gaussian, by slot: colour from
// spherical harmonics along the viewing direction, opacity, the accurate blending position and the
// alpha >= alpha_min box.  Bound by the latency of the scattered parameter rows, with no barrier and
// nothing to wait for; launched beside the depth sort, which needs only the keys.
template <int DEG>
__global__ void __launch_bounds__(128) record_kernel(const DevTables* __restrict__ tab,
                                                     const uint32_t* __restrict__ vis_ids,
                                                     const WsHeader* __restrict__ hdr, Splat* __restrict__ splats) {
  pdl_enter();
  const bool dead = render_dead(hdr);   // the depth sort beside this gave up: nobody reads the records
  const unsigned nv = hdr->visible;
  if (dead) return;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < nv; t += gridDim.x * blockDim.x) {
    const int i = (int)vis_ids[t];
    const KSeg* sg = &tseg(tab, find_seg(tab, i));
    const int li = i - sg->offset;
    const KView& vw = tview(tab, sg->view);
    const KCam& cm = vw.cam;
    constexpr int K = (DEG + 1) * (DEG + 1);
    float Y[16], c[3 * K];
    load_sh<DEG>(sg->g.sh, li, c);
    const float logit = __ldg(sg->g.logits + li);
    Proj P;
    project(sg->g, cm, vw.op, li, P);
    float d0 = P.m[0] - cm.cam_pos[0], d1 = P.m[1] - cm.cam_pos[1], d2 = P.m[2] - cm.cam_pos[2];
    const float il = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
    d0 *= il; d1 *= il; d2 *= il;
    sh_basis<DEG>(d0, d1, d2, Y);
    float rgb[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      float acc = 0.5f;
#pragma unroll
      for (int k = 0; k < K; ++k) acc = fmaf(c[3 * k + ch], Y[k], acc);
      rgb[ch] = fmaxf(0.f, acc);
    }
    const float o = 1.f / (1.f + expf(-logit));
    // the mean's projection for blending, as a double-float (see df_dot3)
    float xh, xl, yh, yl, zh, zl;
    df_dot3(cm.R, cm.t[0], P.m, xh, xl);
    df_dot3(cm.R + 3, cm.t[1], P.m, yh, yl);
    df_dot3(cm.R + 6, cm.t[2], P.m, zh, zl);
    float uh, ul, vh, vl;
    df_project(xh, xl, zh, zl, cm.fx, cm.cx, uh, ul);
    df_project(yh, yl, zh, zl, cm.fy, cm.cy, vh, vl);
    Splat sp;
    sp.u = uh;
    sp.v = vh;
    sp.uvlo = (uint32_t)__half_as_ushort(__float2half_rn(ul)) | ((uint32_t)__half_as_ushort(__float2half_rn(vl)) << 16);
    sp.ca = -0.5f * kLog2e * P.ca;
    sp.cb = -kLog2e * P.cb;
    sp.cc = -0.5f * kLog2e * P.cc;
    sp.lo = log2f(o);
    sp.r = rgb[0]; sp.g = rgb[1]; sp.b = rgb[2];
    sp.rank = 0;
    // alpha >= alpha_min  <=>  power2 >= tg = log2(alpha_min) - lo;  that region is the
    // ellipse d^T Sigma2^-1 d <= k2, k2 = 2 ln(opacity / alpha_min), whose bounding box has
    // half-extents k sqrt(A), k sqrt(C)
    const float tg = log2f(vw.op.alpha_min) - sp.lo;
    float hx = -65504.f, hy = -65504.f;
    if (tg <= 0.f) {
      const float k2 = -2.0f * 0.69314718f * tg;
      hx = sqrtf(k2 * P.A) * 1.001f + 0.01f;
      hy = sqrtf(k2 * P.C) * 1.001f + 0.01f;
    }
    sp.hxy = (uint32_t)__half_as_ushort(__float2half_ru(hx)) | ((uint32_t)__half_as_ushort(__float2half_ru(hy)) << 16);
    float4* dst = reinterpret_cast<float4*>(splats + t);
    const float4* src = reinterpret_cast<const float4*>(&sp);
    dst[0] = src[0]; dst[1] = src[1]; dst[2] = src[2];
  }
}

// Dense gradient outputs are zero for every Gaussian that touches no tile: 236 bytes a Gaussian, most of
// the bytes of a step (4.7 GB for 20M Gaussians, 0.79 ms alone).  The compositing adjoint before the
// projection's leaves HBM idle (2% of its bandwidth), so two warps an SM zero all rows, visible or not, beside
// it: bulk copies (cp.async.bulk) of a zeroed shared buffer, which take no issue slots.  The projection
// adjoint writes the visible rows afterwards.  20M step 2,800 -> 2,212 us, six-cell batch 2,010 -> 1,900.
//  * Launched in the caller's stream before the compositing adjoint, which follows as soon as every block here
//    has started: on a side stream the blocks came after the adjoint's and were packed on a few SMs.
//  * Nothing else zeroes: a kernel for the culled rows of what was left when the adjoint had taken its last
//    tile ran beside that one's last blocks and made them end 380 us later (20M).
//  * Two copies of 16 KB in flight a block: with 2 KB the adjoint was slowed and the zeroing too (20M 2,620 us),
//    with one block an SM the zeroing outlasts the adjoint (2,390).
// Evict-first, so that the adjoint's records and images stay in L2.
constexpr uint32_t kZeroBytes = 16384;
constexpr int kZeroPerSM = 2;
__device__ __forceinline__ void bulk_zero(float* dst, size_t bytes, uint32_t src, uint64_t policy) {
  char* p = reinterpret_cast<char*>(dst);
  char* const e = p + bytes;
  while (p < e && (reinterpret_cast<uintptr_t>(p) & 15u)) {     // to a 16-byte boundary by plain stores
    *reinterpret_cast<float*>(p) = 0.f;
    p += 4;
  }
  while (p + 16 <= e) {
    const uint32_t n = (uint32_t)min((size_t)kZeroBytes, (size_t)(e - p) & ~(size_t)15);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(p), "r"(src),
                 "r"(n), "l"(policy)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 1;" ::: "memory");
    p += n;
  }
  for (; p < e; p += 4) *reinterpret_cast<float*>(p) = 0.f;
}

// Zero gradients of the culled ones of Gaussians first .. last, by one warp.
__device__ __noinline__ void zero_culled(const DevTables* __restrict__ tab, const uint32_t* __restrict__ touched, int F,
                                         int first, int last) {
  for (int i = first + (int)(threadIdx.x & 31); i <= last; i += 32) {
    if (touched[i] != 0) continue;
    const KSeg& sg = tseg(tab, find_seg(tab, i));
    if (!sg.gm) continue;
    const size_t l = (size_t)(i - sg.offset);
    for (int k = 0; k < 3; ++k) { sg.gm[3 * l + k] = 0.f; sg.gs[3 * l + k] = 0.f; }
    for (int k = 0; k < 4; ++k) sg.gq[4 * l + k] = 0.f;
    sg.gl[l] = 0.f;
    for (int k = 0; k < F; ++k) sg.gsh[l * F + k] = 0.f;
  }
}

__global__ void __launch_bounds__(32) zero_grads(const DevTables* __restrict__ tab, int total_n, int F,
                                                 const uint32_t* __restrict__ touched, WsHeader* __restrict__ hdr) {
  __shared__ __align__(128) float4 s_zero[kZeroBytes / 16];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int k = threadIdx.x; k < (int)(kZeroBytes / 16); k += 32) s_zero[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  const int runs = (total_n - 1) / kCullRun + 1;
  if (render_dead(hdr)) {     // a wait of the forward gave up: no gradient of a visible Gaussian is written
    for (int run = blockIdx.x; run < runs; run += gridDim.x)
      zero_culled(tab, touched, F, run * kCullRun, min(total_n - 1, run * kCullRun + (kCullRun - 1)));
    return;
  }
  if (threadIdx.x != 0) return;
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  const uint32_t src = smem_u32(s_zero);
  for (;;) {
    const unsigned run = atomicAdd(&hdr->zero_next, 1u);
    if (run >= (unsigned)runs) break;
    const int first = (int)run * kCullRun, last = min(total_n - 1, first + (kCullRun - 1));
    for (int k = find_seg(tab, first); k < tab->h.n_segs && tseg(tab, k).offset <= last; ++k) {
      const KSeg& sg = tseg(tab, k);
      const int lo = max(first, sg.offset), hi = min(last + 1, sg.offset + sg.g.n);
      if (lo >= hi || !sg.gm) continue;
      const size_t l = (size_t)(lo - sg.offset), n = (size_t)(hi - lo) * 4;
      bulk_zero(sg.gsh + l * F, n * F, src, policy);
      bulk_zero(sg.gq + l * 4, n * 4, src, policy);
      bulk_zero(sg.gm + l * 3, n * 3, src, policy);
      bulk_zero(sg.gs + l * 3, n * 3, src, policy);
      bulk_zero(sg.gl + l, n, src, policy);
    }
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");        // written before the kernel ends
}

// Adjoint of the projection for visible Gaussian i: writes (or, accumulating, adds) the gradients
// of its mean, log-scale, quaternion, logit and SH coefficients.
template <int DEG>
__device__ __forceinline__ void project_adjoint(const DevTables* __restrict__ tab, const Splat& rec,
                                                const float* __restrict__ g2d, int accumulate, int i) {
  constexpr int K = (DEG + 1) * (DEG + 1);
  constexpr int F = 3 * K;
  const KSeg& sg = tseg(tab, find_seg(tab, i));
  if (!sg.gm) return;       // this segment asked for no gradients
  const size_t l = (size_t)(i - sg.offset);
  auto put = [&](float* dst, float v) { if (accumulate) *dst += v; else *dst = v; };
  auto put4 = [&](float* dst, float a, float b, float c, float d) {
    float4* p = reinterpret_cast<float4*>(dst);
    float4 v = make_float4(a, b, c, d);
    if (accumulate) {
      const float4 o = *p;
      v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
    }
    *p = v;
  };
  float* gsh = sg.gsh + l * F;
  const KGauss g = sg.g;
  const KCam cm = tview(tab, sg.view).cam;
  const KOpts op = tview(tab, sg.view).op;
  const int li = (int)l;
  const uint32_t rank = rec.rank;
  float d2[9];
  {
    // slots 0-5 hold the compositing adjoint's power moments; 6-8 d rgb
    float mom[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) mom[f] = g2d[(size_t)rank * 9 + f];
    grad2d_from_moments(mom, rec.ca, rec.cb, rec.cc, rec.lo, d2);
#pragma unroll
    for (int f = 6; f < 9; ++f) d2[f] = g2d[(size_t)rank * 9 + f];
  }
  Proj P;
  project(g, cm, op, li, P);
  float o_m[3], o_s[3], o_q[4];
  // opacity
  const float o = 1.f / (1.f + expf(-__ldg(g.logits + li)));
  put(sg.gl + l, d2[5] * o * (1.f - o));
  // colour: rgb = max(0, sum_k c_k Y_k(d) + 0.5), d = (m - cam_pos) / |m - cam_pos|
  float d0 = P.m[0] - cm.cam_pos[0], d1 = P.m[1] - cm.cam_pos[1], dz = P.m[2] - cm.cam_pos[2];
  const float il = rsqrtf(d0 * d0 + d1 * d1 + dz * dz);
  d0 *= il; d1 *= il; dz *= il;
  float Y[16];
  sh_basis<DEG>(d0, d1, dz, Y);
  const float* shp = g.sh + l * F;
  // one pass over the coefficients: pre_ch = 0.5 + sum_k c_k,ch Y_k and, per channel,
  // D_ch = sum_k c_k,ch grad Y_k (the direction gradient once the clamp mask is known)
  float pre[3] = {0.5f, 0.5f, 0.5f};
  float D[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  {
    float G[16][3];
    sh_basis_grad<DEG>(d0, d1, dz, G);
    auto term = [&](float c, int k, int ch) {
      pre[ch] = fmaf(c, Y[k], pre[ch]);
      D[ch][0] = fmaf(c, G[k][0], D[ch][0]);
      D[ch][1] = fmaf(c, G[k][1], D[ch][1]);
      D[ch][2] = fmaf(c, G[k][2], D[ch][2]);
    };
    if constexpr (F % 4 == 0) {   // 16-byte rows: one vector load per four coefficients, same order
      const float4* p4 = reinterpret_cast<const float4*>(shp);
#pragma unroll
      for (int q = 0; q < F / 4; ++q) {
        const float4 v = __ldg(p4 + q);
        term(v.x, (4 * q) / 3, (4 * q) % 3);
        term(v.y, (4 * q + 1) / 3, (4 * q + 1) % 3);
        term(v.z, (4 * q + 2) / 3, (4 * q + 2) % 3);
        term(v.w, (4 * q + 3) / 3, (4 * q + 3) % 3);
      }
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) term(__ldg(shp + 3 * k + ch), k, ch);
    }
  }
  float dpre[3];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) dpre[ch] = pre[ch] > 0.f ? d2[6 + ch] : 0.f;
  // d loss / d coefficient = dpre * Y, written as it is formed
  if constexpr (F % 4 == 0) {
#pragma unroll
    for (int f = 0; f < F; f += 4)
      put4(gsh + f, dpre[f % 3] * Y[f / 3], dpre[(f + 1) % 3] * Y[(f + 1) / 3], dpre[(f + 2) % 3] * Y[(f + 2) / 3],
           dpre[(f + 3) % 3] * Y[(f + 3) / 3]);
  } else {
#pragma unroll
    for (int f = 0; f < F; ++f) put(gsh + f, dpre[f % 3] * Y[f / 3]);
  }
  // d loss / d direction = sum_ch dpre_ch D_ch, projected on the tangent plane
  float dd[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) dd[c] = dpre[0] * D[0][c] + dpre[1] * D[1][c] + dpre[2] * D[2][c];
  const float dot = dd[0] * d0 + dd[1] * d1 + dd[2] * dz;
  o_m[0] = (dd[0] - d0 * dot) * il;
  o_m[1] = (dd[1] - d1 * dot) * il;
  o_m[2] = (dd[2] - dz * dot) * il;
  // conic -> 2D covariance: dS2 = -Q G Q, Q = [[a,b],[b,c]], G = [[da, db/2],[db/2, dc]]
  const float qa = P.ca, qb = P.cb, qc = P.cc;
  const float g0 = d2[2], g1 = 0.5f * d2[3], g2 = d2[4];
  const float m00 = qa * g0 + qb * g1, m01 = qa * g1 + qb * g2;
  const float m10 = qb * g0 + qc * g1, m11 = qb * g1 + qc * g2;
  const float s00 = -(m00 * qa + m01 * qb);
  const float s01 = -(m00 * qb + m01 * qc);
  const float s11 = -(m10 * qb + m11 * qc);
  // Sigma2 = T Sigma T^T: dSigma = T^T dS2 T, dT = 2 dS2 T Sigma
  const float* T = P.T;
  float U[2][3];   // dS2 T
#pragma unroll
  for (int c3 = 0; c3 < 3; ++c3) {
    U[0][c3] = s00 * T[c3] + s01 * T[3 + c3];
    U[1][c3] = s01 * T[c3] + s11 * T[3 + c3];
  }
  float dSig[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) dSig[a][b] = T[a] * U[0][b] + T[3 + a] * U[1][b];
  const float* S = P.Sig;
  const float Sf[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
  float dT[2][3];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int j = 0; j < 3; ++j) dT[a][j] = 2.f * (U[a][0] * Sf[0][j] + U[a][1] * Sf[1][j] + U[a][2] * Sf[2][j]);
  // dJ = dT W^T; only J00, J02, J11, J12 depend on p
  const float* W = cm.R;
  const float dJ00 = dT[0][0] * W[0] + dT[0][1] * W[1] + dT[0][2] * W[2];
  const float dJ02 = dT[0][0] * W[6] + dT[0][1] * W[7] + dT[0][2] * W[8];
  const float dJ11 = dT[1][0] * W[3] + dT[1][1] * W[4] + dT[1][2] * W[5];
  const float dJ12 = dT[1][0] * W[6] + dT[1][1] * W[7] + dT[1][2] * W[8];
  const float z = P.p[2], iz = 1.f / z, iz2 = iz * iz;
  float dp[3] = {0.f, 0.f, 0.f};
  dp[2] += -(dJ00 * cm.fx + dJ11 * cm.fy) * iz2;
  // J02 = -fx xzc / z with xzc = x / z unless clamped
  if (P.clx) {
    dp[2] += dJ02 * cm.fx * P.xzc * iz2;
  } else {
    dp[0] += -dJ02 * cm.fx * iz2;
    dp[2] += dJ02 * 2.f * cm.fx * P.p[0] * iz2 * iz;
  }
  if (P.cly) {
    dp[2] += dJ12 * cm.fy * P.yzc * iz2;
  } else {
    dp[1] += -dJ12 * cm.fy * iz2;
    dp[2] += dJ12 * 2.f * cm.fy * P.p[1] * iz2 * iz;
  }
  // u = fx x/z + cx, v = fy y/z + cy
  dp[0] += d2[0] * cm.fx * iz;
  dp[1] += d2[1] * cm.fy * iz;
  dp[2] += -(d2[0] * cm.fx * P.p[0] + d2[1] * cm.fy * P.p[1]) * iz2;
#pragma unroll
  for (int c3 = 0; c3 < 3; ++c3) o_m[c3] += W[c3] * dp[0] + W[3 + c3] * dp[1] + W[6 + c3] * dp[2];
  // Sigma = M M^T, M = Rq diag(s): dM = 2 dSigma M
  float M[9];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c3 = 0; c3 < 3; ++c3) M[3 * r + c3] = P.Rq[3 * r + c3] * P.s[c3];
  float dR[9];
#pragma unroll
  for (int c3 = 0; c3 < 3; ++c3) {
    float ds = 0.f;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const float dMrc = 2.f * (dSig[r][0] * M[c3] + dSig[r][1] * M[3 + c3] + dSig[r][2] * M[6 + c3]);
      ds += dMrc * P.Rq[3 * r + c3];
      dR[3 * r + c3] = dMrc * P.s[c3];
    }
    o_s[c3] = ds * P.s[c3];
  }
  // rotation matrix of the unit quaternion (w, x, y, z)
  const float w = P.qn[0], x = P.qn[1], y = P.qn[2], zq = P.qn[3];
  float dqn[4];
  dqn[0] = 2.f * (-zq * dR[1] + y * dR[2] + zq * dR[3] - x * dR[5] - y * dR[6] + x * dR[7]);
  dqn[1] = 2.f * (y * dR[1] + zq * dR[2] + y * dR[3] - 2.f * x * dR[4] - w * dR[5] + zq * dR[6] + w * dR[7] - 2.f * x * dR[8]);
  dqn[2] = 2.f * (-2.f * y * dR[0] + x * dR[1] + w * dR[2] + x * dR[3] + zq * dR[5] - w * dR[6] + zq * dR[7] - 2.f * y * dR[8]);
  dqn[3] = 2.f * (-2.f * zq * dR[0] - w * dR[1] + x * dR[2] + w * dR[3] - 2.f * zq * dR[4] + y * dR[5] + x * dR[6] + y * dR[7]);
  const float qd = P.qn[0] * dqn[0] + P.qn[1] * dqn[1] + P.qn[2] * dqn[2] + P.qn[3] * dqn[3];
#pragma unroll
  for (int k = 0; k < 4; ++k) o_q[k] = (dqn[k] - P.qn[k] * qd) * P.qinv;
#pragma unroll
  for (int k = 0; k < 3; ++k) { put(sg.gm + 3 * l + k, o_m[k]); put(sg.gs + 3 * l + k, o_s[k]); }
  put4(sg.gq + 4 * l, o_q[0], o_q[1], o_q[2], o_q[3]);
}

// Adjoint of the projection for the visible Gaussians, taken from the compact list of visible
// ids in index order (every lane of a warp has work, neighbouring lanes read nearby rows); the
// blocks stride over the list, so the grid is sized by the launcher, not by the visible count.
template <int DEG>
__global__ void __launch_bounds__(128, 4) preprocess_backward_kernel(
    const DevTables* __restrict__ tab, const uint32_t* __restrict__ vis_ids, const WsHeader* __restrict__ hdr,
    const Splat* __restrict__ splats, const float* __restrict__ g2d, int accumulate) {
  pdl_enter();
  const bool dead = render_dead(hdr);   // a sort gave up: ranks and accumulators are not this render's
  const int nv = (int)hdr->visible;
  if (dead) return;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nv; t += gridDim.x * blockDim.x)
    project_adjoint<DEG>(tab, splats[t], g2d, accumulate, (int)vis_ids[t]);
}

}  // namespace

cudaError_t launch_preprocess(const DevTables* tab, int total_n, uint2* rects, uint32_t* touched, const Compact& cp,
                              WsHeader* hdr, cudaStream_t s) {
  if (total_n == 0) return cudaSuccess;
  note_launches(2);
  const int runs = (total_n - 1) / kCullRun + 1;
  launch_pdl(cull_kernel, std::min(runs, kCullBlocks * sort_blocks() / 2), kCullThreads, 0, s, tab, total_n, runs, cp.entries,
             cp.counts, touched, cp.key_inputs);
  // a warp a run on small scenes, up to 4 blocks an SM (2 an SM left a block of a merged scene, whose
  // visible Gaussians sit in few runs, with a long tail: 41 us for four views; more add up more counts)
  const int blocks = std::max(1, std::min((runs + kCompactThreads / 32 - 1) / (kCompactThreads / 32), 2 * sort_blocks()));
  const int per = (runs + blocks - 1) / blocks;
  launch_pdl(compact_kernel, (runs + per - 1) / per, kCompactThreads, 0, s, cp.entries, cp.counts, runs, per, rects, cp, hdr);
  return cudaGetLastError();
}

cudaError_t launch_records(const DevTables* tab, int total_n, int degree, const uint32_t* vis_ids, const WsHeader* hdr,
                           Splat* splats, cudaStream_t s) {
  if (total_n == 0) return cudaSuccess;
  note_launches(1);
  const int rb = std::min((total_n - 1) / 128 + 1, 8 * sort_blocks());
  switch (degree) {
    case 0: record_kernel<0><<<rb, 128, 0, s>>>(tab, vis_ids, hdr, splats); break;
    case 1: record_kernel<1><<<rb, 128, 0, s>>>(tab, vis_ids, hdr, splats); break;
    case 2: record_kernel<2><<<rb, 128, 0, s>>>(tab, vis_ids, hdr, splats); break;
    default: record_kernel<3><<<rb, 128, 0, s>>>(tab, vis_ids, hdr, splats); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_zero_grads(const DevTables* tab, int total_n, int degree, const uint32_t* touched, WsHeader* hdr,
                              cudaStream_t s) {
  const int runs = (total_n - 1) / kCullRun + 1, F = 3 * (degree + 1) * (degree + 1);
  note_launches(1);
  // launched plainly: what precedes is complete before the adjoint may start (it does not wait for it itself), and the
  // blocks find the SMs empty and spread evenly (started early behind the accumulators' reset they took
  // the SMs that came free first: 20M 2,920 us)
  zero_grads<<<std::min(runs, kZeroPerSM * sort_blocks() / 2), 32, 0, s>>>(tab, total_n, F, touched, hdr);
  return cudaGetLastError();
}

cudaError_t launch_preprocess_backward(const DevTables* tab, int total_n, int degree, const Splat* splats,
                                       const uint32_t* vis_ids, const WsHeader* hdr, const float* g2d,
                                       bool accumulate, cudaStream_t s) {
  if (total_n == 0) return cudaSuccess;
  const int acc = accumulate ? 1 : 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // latency-bound at 128 registers a thread: 4 blocks an SM fill the register file
  const int blocks = std::max(1, std::min((total_n + 127) / 128, 4 * std::max(sms, 1)));
  note_launches(1);
  auto go = [&](auto kernel) { launch_pdl(kernel, blocks, 128, 0, s, tab, vis_ids, hdr, splats, g2d, acc); };
  switch (degree) {
    case 0: go(preprocess_backward_kernel<0>); break;
    case 1: go(preprocess_backward_kernel<1>); break;
    case 2: go(preprocess_backward_kernel<2>); break;
    default: go(preprocess_backward_kernel<3>); break;
  }
  return cudaGetLastError();
}

}  // namespace vg
