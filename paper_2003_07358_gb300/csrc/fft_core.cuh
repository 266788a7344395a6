// Complex arithmetic and register-resident R-point DFTs shared by the transforms of
// nufft.cu and fft_mid.cu.
#pragma once

#include <cuda_runtime.h>

namespace fhs {

// ------------------------------------------------------------------ complex
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// ----------------------------------------------------------- R-point DFTs
// Forward sign exp(-2 pi i / R); `inv` flips the sign (unnormalised).
__device__ __forceinline__ void dft2(float2& a, float2& b) {
  float2 t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3, bool inv) {
  float2 a0 = cadd(x0, x2), a1 = csub(x0, x2), a2 = cadd(x1, x3), a3 = csub(x1, x3);
  // -i * a3 = (a3.y, -a3.x)
  float2 mia3 = inv ? make_float2(-a3.y, a3.x) : make_float2(a3.y, -a3.x);
  x0 = cadd(a0, a2);
  x2 = csub(a0, a2);
  x1 = cadd(a1, mia3);
  x3 = csub(a1, mia3);
}

__device__ __forceinline__ void dft8(float2* v, bool inv) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4(e0, e1, e2, e3, inv);
  dft4(o0, o1, o2, o3, inv);
  const float c = 0.70710678118654752440f;
  float sg = inv ? 1.f : -1.f;
  // w^1 = (c, sg c), w^2 = (0, sg), w^3 = (-c, sg c)
  float2 t1 = cmul(o1, make_float2(c, sg * c));
  float2 t2 = cmul(o2, make_float2(0.f, sg));
  float2 t3 = cmul(o3, make_float2(-c, sg * c));
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = cadd(e1, t1); v[5] = csub(e1, t1);
  v[2] = cadd(e2, t2); v[6] = csub(e2, t2);
  v[3] = cadd(e3, t3); v[7] = csub(e3, t3);
}

__device__ __forceinline__ void dft3(float2& x0, float2& x1, float2& x2, bool inv) {
  const float h = 0.866025403784438646764f;                  // sqrt(3) / 2
  const float2 t = cadd(x1, x2), d = csub(x1, x2);
  const float2 m = make_float2(fmaf(-0.5f, t.x, x0.x), fmaf(-0.5f, t.y, x0.y));
  const float2 ihd = make_float2(-h * d.y, h * d.x);         // i (sqrt(3) / 2) (x1 - x2)
  x0 = cadd(x0, t);
  // forward: y1 = m - i h d, y2 = m + i h d; the inverse flips the sign of i
  x1 = inv ? cadd(m, ihd) : csub(m, ihd);
  x2 = inv ? csub(m, ihd) : cadd(m, ihd);
}

// exp(-2 pi i j / 32), j < 16
static __constant__ float2 c_w32[16] = {
    {1.f, 0.f},                          {9.807852804e-01f, -1.950903220e-01f},
    {9.238795325e-01f, -3.826834324e-01f}, {8.314696123e-01f, -5.555702330e-01f},
    {7.071067812e-01f, -7.071067812e-01f}, {5.555702330e-01f, -8.314696123e-01f},
    {3.826834324e-01f, -9.238795325e-01f}, {1.950903220e-01f, -9.807852804e-01f},
    {0.f, -1.f},                           {-1.950903220e-01f, -9.807852804e-01f},
    {-3.826834324e-01f, -9.238795325e-01f}, {-5.555702330e-01f, -8.314696123e-01f},
    {-7.071067812e-01f, -7.071067812e-01f}, {-8.314696123e-01f, -5.555702330e-01f},
    {-9.238795325e-01f, -3.826834324e-01f}, {-9.807852804e-01f, -1.950903220e-01f},
};

// exp(-2 pi i j / 48), j < 24
static __constant__ float2 c_w48[24] = {
    {1.000000000e+00f, 0.000000000e+00f}, {9.914448614e-01f, -1.305261922e-01f}, {9.659258263e-01f, -2.588190451e-01f},
    {9.238795325e-01f, -3.826834324e-01f}, {8.660254038e-01f, -5.000000000e-01f}, {7.933533403e-01f, -6.087614290e-01f},
    {7.071067812e-01f, -7.071067812e-01f}, {6.087614290e-01f, -7.933533403e-01f}, {5.000000000e-01f, -8.660254038e-01f},
    {3.826834324e-01f, -9.238795325e-01f}, {2.588190451e-01f, -9.659258263e-01f}, {1.305261922e-01f, -9.914448614e-01f},
    {0.000000000e+00f, -1.000000000e+00f}, {-1.305261922e-01f, -9.914448614e-01f}, {-2.588190451e-01f, -9.659258263e-01f},
    {-3.826834324e-01f, -9.238795325e-01f}, {-5.000000000e-01f, -8.660254038e-01f}, {-6.087614290e-01f, -7.933533403e-01f},
    {-7.071067812e-01f, -7.071067812e-01f}, {-7.933533403e-01f, -6.087614290e-01f}, {-8.660254038e-01f, -5.000000000e-01f},
    {-9.238795325e-01f, -3.826834324e-01f}, {-9.659258263e-01f, -2.588190451e-01f}, {-9.914448614e-01f, -1.305261922e-01f},
};

// In-place R-point DFT of v (natural order in and out), R = 2^a or 3 2^a, radix-2
// decimation in time down to the 8-, 4-, 3- and 2-point kernels; sign exp(-2 pi i / R),
// INV flips it.
template <int R, bool INV>
__device__ __forceinline__ void rdft(float2* v) {
  if constexpr (R == 2) {
    dft2(v[0], v[1]);
  } else if constexpr (R == 3) {
    dft3(v[0], v[1], v[2], INV);
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3], INV);
  } else if constexpr (R == 8) {
    dft8(v, INV);
  } else {
    constexpr int H = R / 2;
    float2 e[H], o[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    rdft<H, INV>(e);
    rdft<H, INV>(o);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      float2 t;
      if (k == 0) {
        t = o[0];
      } else if (2 * k == H) {               // w = -i (forward), +i (inverse)
        t = INV ? make_float2(-o[k].y, o[k].x) : make_float2(o[k].y, -o[k].x);
      } else {
        float2 w = R % 3 ? c_w32[k * (32 / R)] : c_w48[k * (48 / R)];
        if (INV) w.y = -w.y;
        t = cmul(o[k], w);
      }
      v[k] = cadd(e[k], t);
      v[k + H] = csub(e[k], t);
    }
  }
}

}  // namespace fhs
