// Double-float arithmetic for the kernels that need more digits than FP32 holds.
#pragma once

#include <cuda_runtime.h>

namespace vg {

// Double-float: a value as an unevaluated sum of two FP32 numbers (48 bits), by the classical
// error-free transformations (Dekker, Knuth).  An operation is 6 to 20 FP32 instructions; FP64 issues at
// 1/64 of FP32's rate on this part, so this is the faster way to some 14 digits.
struct dd {
  float h, l;
  __device__ dd() {}
  __device__ dd(float a, float b = 0.f) : h(a), l(b) {}
};
__device__ __forceinline__ dd dd_norm(float h, float l) {        // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return dd(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ dd operator+(dd a, dd b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  return dd_norm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ dd operator-(dd a) { return dd(-a.h, -a.l); }
__device__ __forceinline__ dd operator-(dd a, dd b) { return a + (-b); }
__device__ __forceinline__ dd operator*(dd a, dd b) {
  const float p = __fmul_rn(a.h, b.h), e = __fmaf_rn(a.h, b.h, -p);
  return dd_norm(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e)));
}
__device__ __forceinline__ dd operator/(dd a, dd b) {
  const float q = __fdiv_rn(a.h, b.h);
  const float r = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));     // a - q b: the first term is exact
  return dd_norm(q, __fdividef(r, b.h));
}
__device__ __forceinline__ bool operator<(dd a, dd b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
__device__ __forceinline__ bool operator==(dd a, dd b) { return a.h == b.h && a.l == b.l; }

// Sum over a warp's lanes (every lane).
__device__ __forceinline__ dd warp_sum_dd(dd v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = v + dd(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
  return v;
}

}  // namespace vg
