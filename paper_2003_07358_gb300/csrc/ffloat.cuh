// Arithmetic on pairs of floats (hi + lo, about 2^-47 relative): what takes the place of
// FP64 inside kernels, which this GPU issues at one warp instruction per 64 clocks and
// sub-partition.
#pragma once

#include <cuda_runtime.h>

namespace fhs {

// Error-free transformation a + b = s + e (Knuth TwoSum), no contraction.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

struct ff {
  float h, l;
};

__device__ __forceinline__ ff ff_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double ff_val(ff a) { return (double)a.h + (double)a.l; }

// c a + s b.
__device__ __forceinline__ ff ff_lin(ff c, ff a, ff s, ff b) {
  const float p = __fmul_rn(c.h, a.h), q = __fmul_rn(s.h, b.h);
  float pe = __fmaf_rn(c.h, a.h, -p), qe = __fmaf_rn(s.h, b.h, -q);
  pe = __fmaf_rn(c.l, a.h, __fmaf_rn(c.h, a.l, pe));
  qe = __fmaf_rn(s.l, b.h, __fmaf_rn(s.h, b.l, qe));
  float t, e;
  two_sum(p, q, t, e);
  e = __fadd_rn(e, __fadd_rn(pe, qe));
  const float h = __fadd_rn(t, e);
  return {h, __fsub_rn(e, __fsub_rn(h, t))};
}

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
  const float h = __fadd_rn(p, e);
  return {h, __fsub_rn(e, __fsub_rn(h, p))};
}

// u^-1/2 (u > 0): one Newton step from the FP32 value with the residual 1 - u y^2 formed
// as a pair.
__device__ __forceinline__ ff ff_rsqrt(ff u) {
  const float y = rsqrtf(u.h);
  const float q = __fmul_rn(y, y), qe = __fmaf_rn(y, y, -q);
  const float w = __fmul_rn(u.h, q);
  const float we = __fmaf_rn(u.l, q, __fmaf_rn(u.h, qe, __fmaf_rn(u.h, q, -w)));
  const float r = __fsub_rn(__fsub_rn(1.f, w), we);
  const float cor = y * fmaf(0.375f * r, r, 0.5f * r);
  const float h = __fadd_rn(y, cor);
  return {h, __fsub_rn(cor, __fsub_rn(h, y))};
}

// a + b.
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}

// Sum over the lanes of a warp, in a fixed order; every lane gets it.
__device__ __forceinline__ ff ff_warp_sum(ff a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    a = ff_add(a, {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)});
  return a;
}

}  // namespace fhs
