// Reweighted nuclear-norm duals of the apodised facets (Algorithm 2 P update,
// Table 2 row 2) on GB300.
//
// For facet q with Z_q = P_q + D_q S~_q Xcheck (N~_q x L):
//   (I - prox_{alpha ||.||_*,theta})(Z) = U diag(min(s_j, alpha_j)) V^T = Z V diag(m) V^T,
//   m_j = min(1, alpha_j / s_j), Z^T Z = V diag(s^2) V^T.
// Kernels:
//   k_gram   : partial Gram matrices Z^T Z of pixel chunks (float pairs, staged in smem;
//              k_gram_f64 for the weights, k_gram_small up to 8 channels);
//   k_eig    : FP64 sum of the partials in fixed order (k_gram_sum first where there are
//              many), cyclic Jacobi eigen-solve of the L x L Gram in float pairs, finished
//              in FP64, M_q = V diag(m) V^T (or weights);
//   k_apply  : pixel-driven: for each pixel and each facet covering it,
//              P_q <- Z_q M_q and A += zeta D_q P_q (every A pixel written once).
#include <cuda_runtime.h>

#include <algorithm>

#include "ffloat.cuh"
#include "fhs_internal.h"

namespace fhs {

constexpr int kGramChunk = 1024;   // pixels per Gram partial
constexpr int kGramSub = 64;       // pixels staged in shared memory at a time

__device__ __forceinline__ float facet_weight(const NucFacet& f, const float* __restrict__ win, int rr, int cc) {
  return win[f.wy_off + rr] * win[f.wx_off + cc];
}

// Partial Gram of chunk blockIdx.x of facet blockIdx.y, accumulated in
// float-float: each product a*b = p + e exactly (FMA), the running sum keeps a
// high part and a compensation term, so the partial equals the exact Gram of
// the FP32 matrix Z to ~1e-14 relative.  (A plain FP32 Gram has absolute
// errors ~eps * lambda_max, which wipes out singular values below
// sqrt(eps) s_max.)  Thread owns an LB x LB block of G; Lp = L rounded up to a
// multiple of LB.  Output: FP64 partials [Q][nchunk_max][L][L].
//
template <int LB>
__global__ void __launch_bounds__(256, LB == 4 ? 1 : 3) k_gram(const float* __restrict__ xc, const float* __restrict__ P,
                                              const NucFacet* __restrict__ facets, const float* __restrict__ win,
                                              int n1, int n2, int L, int use_P, double* __restrict__ part,
                                              int nchunk_max) {
  // the staged sub-chunk and, after the last one, the per-group partial sums
  __shared__ union {
    float z[kGramSub][kMaxL + 1];
    double red[256 * LB * LB];
  } sm;
  auto& z = sm.z;
  auto& red = sm.red;
  const int q = blockIdx.y;
  const NucFacet f = facets[q];
  const int h = f.r1 - f.r0, w = f.c1 - f.c0;
  const int Nq = h * w;
  const int p0 = blockIdx.x * kGramChunk;
  if (p0 >= Nq) return;
  const int p1 = min(Nq, p0 + kGramChunk);
  const int Lp = (L + LB - 1) / LB * LB;
  const int nb = Lp / LB;
  // thread -> (upper-triangle block pair, pixel group): npairs pairs, G groups share
  // the pixels of each staged sub-chunk; the groups are summed in a fixed order
  const int npairs = nb * (nb + 1) / 2;
  const int G = max(1, (int)blockDim.x / npairs);
  const int pair = threadIdx.x % npairs, g = threadIdx.x / npairs;
  const bool active = g < G;
  int ta = 0, rem = pair;
  while (rem >= nb - ta) { rem -= nb - ta; ++ta; }
  const int tb = ta + rem;
  float hi[LB][LB], lo[LB][LB];
#pragma unroll
  for (int i = 0; i < LB; ++i)
#pragma unroll
    for (int j = 0; j < LB; ++j) hi[i][j] = lo[i][j] = 0.f;
  const size_t N = (size_t)n1 * n2;
  // staging: thread -> pixel spix of the sub-chunk and channels sl0 + 4k; up to 16
  // channels the next sub-chunk's values are loaded into registers while the current
  // one is reduced
  constexpr int NPT = LB == 2 ? 4 : 1;      // channels per thread (Lp <= 4 NPT when prefetching)
  static_assert(kGramSub * 4 == 256, "256 threads stage 64 pixels x 4 channel lanes");
  const int spix = threadIdx.x % kGramSub, sl0 = threadIdx.x / kGramSub;
  float pre[NPT];
  auto fetch = [&](int s0) {
    const int p = s0 + spix;
    const bool okp = p < p1;
    int rr = 0, cc = 0;
    float d = 0.f;
    if (okp) {
      rr = p / w;
      cc = p - rr * w;
      d = facet_weight(f, win, rr, cc);
    }
    const size_t xo = (size_t)(f.r0 + rr) * n2 + (f.c0 + cc);
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int l = sl0 + 4 * k;
      float val = 0.f;
      if (okp && l < L) {
        val = d * xc[l * N + xo];
        if (use_P) val += P[f.p_off + (size_t)l * Nq + p];
      }
      pre[k] = val;
    }
  };
  constexpr bool PF = LB <= 2;                 // prefetch (registers permitting)
  if (PF) fetch(p0);
  for (int s0 = p0; s0 < p1; s0 += kGramSub) {
    if constexpr (PF) {
#pragma unroll
      for (int k = 0; k < NPT; ++k)
        if (sl0 + 4 * k < Lp) z[spix][sl0 + 4 * k] = pre[k];
    } else {
#pragma unroll 4
      for (int idx = threadIdx.x; idx < kGramSub * Lp; idx += blockDim.x) {
        const int pix = idx % kGramSub, l = idx / kGramSub;
        const int p = s0 + pix;
        float val = 0.f;
        if (p < p1 && l < L) {
          const int rr = p / w, cc = p - rr * w;
          const float d = facet_weight(f, win, rr, cc);
          val = d * xc[l * N + (size_t)(f.r0 + rr) * n2 + (f.c0 + cc)];
          if (use_P) val += P[f.p_off + (size_t)l * Nq + p];
        }
        z[pix][l] = val;
      }
    }
    __syncthreads();
    if (PF && s0 + kGramSub < p1) fetch(s0 + kGramSub);
    if (active) {
      for (int pix = g; pix < kGramSub; pix += G) {
        float a[LB], b[LB];
#pragma unroll
        for (int i = 0; i < LB; ++i) a[i] = z[pix][ta * LB + i];
#pragma unroll
        for (int j = 0; j < LB; ++j) b[j] = z[pix][tb * LB + j];
#pragma unroll
        for (int i = 0; i < LB; ++i)
#pragma unroll
          for (int j = 0; j < LB; ++j) {
            float pr = __fmul_rn(a[i], b[j]);
            float pe = __fmaf_rn(a[i], b[j], -pr);
            float s, e;
            two_sum(hi[i][j], pr, s, e);
            hi[i][j] = s;
            lo[i][j] = __fadd_rn(lo[i][j], __fadd_rn(e, pe));
          }
      }
    }
    __syncthreads();
  }
  if (active) {
#pragma unroll
    for (int i = 0; i < LB; ++i)
#pragma unroll
      for (int j = 0; j < LB; ++j) red[((size_t)g * npairs + pair) * LB * LB + i * LB + j] = (double)hi[i][j] + (double)lo[i][j];
  }
  __syncthreads();
  double* out = part + ((size_t)q * nchunk_max + blockIdx.x) * L * L;
  for (int k = threadIdx.x; k < npairs * LB * LB; k += blockDim.x) {
    const int pr = k / (LB * LB), ij = k - pr * LB * LB, i = ij / LB, j = ij - i * LB;
    double v = 0.0;
    for (int gg = 0; gg < G; ++gg) v += red[((size_t)gg * npairs + pr) * LB * LB + ij];
    int xa = 0, xr = pr;
    while (xr >= nb - xa) { xr -= nb - xa; ++xa; }
    const int a = xa * LB + i, b = (xa + xr) * LB + j;
    if (a < L && b < L) {
      out[a * L + b] = v;
      out[b * L + a] = v;
    }
  }
}

// Gram of D_q S~_q x in FP64 for the weights of Algorithm 1 (once per reweighting cycle):
// theta_bar = mu_bar / (s + mu_bar) depends on singular values far below s_max, and an error
// of the Gram enters them as its square root, so the windows, the products and the sums are
// FP64 (float pairs, whose low part rounds at about 2^-47 of the sum, were off by 4e-8 of s_max
// at 38 channels and 1.2e-7 at 64 where these are by 8e-9, and left FP32's range below 1e-18).
// Blocks of entries and pixel groups over the threads as in k_gram, so that every warp is
// full; blockIdx.z takes a share of the blocks (at most kGramShare), so that the CTAs of a facet
// balance over the SMs: bound by the FP64 pipe, 16 instructions of 64 clk per pixel, warp
// and 4 x 4 block.  0.69 ms at 36 facets of 85^2 pixels and 38 channels (1.68 ms in the earlier FP64
// kernel, whose warps were partly filled, 0.24 ms in float pairs).
constexpr int kGramShare = 28;     // blocks of entries per CTA of k_gram_f64

template <int LB>
__global__ void __launch_bounds__(256) k_gram_f64(const float* __restrict__ xc, const NucFacet* __restrict__ facets,
                                                  const double* __restrict__ win64, int n1, int n2, int L,
                                                  double* __restrict__ part, int nchunk_max) {
  __shared__ union {
    double z[kGramSub][kMaxL + 1];
    double red[256 * LB * LB];
  } sm;
  const int q = blockIdx.y;
  const NucFacet f = facets[q];
  const int h = f.r1 - f.r0, w = f.c1 - f.c0;
  const int Nq = h * w;
  const int p0 = blockIdx.x * kGramChunk;
  if (p0 >= Nq) return;
  const int p1 = min(Nq, p0 + kGramChunk);
  const int nb = (L + LB - 1) / LB, Lp = nb * LB;
  // this CTA's blocks first .. first + npairs - 1 of the upper triangle
  const int all = nb * (nb + 1) / 2, share = (all + gridDim.z - 1) / gridDim.z;
  const int first = blockIdx.z * share, npairs = min(share, all - first);
  const int G = max(1, (int)blockDim.x / npairs);
  const int pair = threadIdx.x % npairs, g = threadIdx.x / npairs;
  const bool active = g < G;
  int ta = 0, rem = first + pair;
  while (rem >= nb - ta) { rem -= nb - ta; ++ta; }
  const int tb = ta + rem;
  double acc[LB][LB];
#pragma unroll
  for (int i = 0; i < LB; ++i)
#pragma unroll
    for (int j = 0; j < LB; ++j) acc[i][j] = 0.0;
  const size_t N = (size_t)n1 * n2;
  const int spix = threadIdx.x % kGramSub, sl0 = threadIdx.x / kGramSub;      // pixel, first channel staged
  for (int s0 = p0; s0 < p1; s0 += kGramSub) {
    const int p = s0 + spix;
    const int rr = p < p1 ? p / w : 0, cc = p < p1 ? p - rr * w : 0;
    const double d = win64[f.wy_off + rr] * win64[f.wx_off + cc];
    const size_t xo = (size_t)(f.r0 + rr) * n2 + (f.c0 + cc);
#pragma unroll 4
    for (int l = sl0; l < Lp; l += 4) sm.z[spix][l] = p < p1 && l < L ? d * (double)xc[l * N + xo] : 0.0;
    __syncthreads();
    if (active) {
      for (int pix = g; pix < min(kGramSub, p1 - s0); pix += G) {
        double a[LB], b[LB];
#pragma unroll
        for (int i = 0; i < LB; ++i) a[i] = sm.z[pix][ta * LB + i];
#pragma unroll
        for (int j = 0; j < LB; ++j) b[j] = sm.z[pix][tb * LB + j];
#pragma unroll
        for (int i = 0; i < LB; ++i)
#pragma unroll
          for (int j = 0; j < LB; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
    }
    __syncthreads();
  }
  if (active) {
#pragma unroll
    for (int i = 0; i < LB; ++i)
#pragma unroll
      for (int j = 0; j < LB; ++j) sm.red[((size_t)g * npairs + pair) * LB * LB + i * LB + j] = acc[i][j];
  }
  __syncthreads();
  double* out = part + ((size_t)q * nchunk_max + blockIdx.x) * L * L;
  for (int k = threadIdx.x; k < npairs * LB * LB; k += blockDim.x) {
    const int pr = k / (LB * LB), ij = k - pr * LB * LB, i = ij / LB, j = ij - i * LB;
    double v = 0.0;
    for (int gg = 0; gg < G; ++gg) v += sm.red[((size_t)gg * npairs + pr) * LB * LB + ij];
    int xa = 0, xr = first + pr;
    while (xr >= nb - xa) { xr -= nb - xa; ++xa; }
    const int a = xa * LB + i, b = (xa + xr) * LB + j;
    if (a < L && b < L) {
      out[a * L + b] = v;
      out[b * L + a] = v;
    }
  }
}

// Partial Grams of up to LM <= 8 channels: a thread streams pixels (chunks blockIdx.x,
// blockIdx.x + parts, ... of the facet) and keeps every entry of the upper triangle as a
// float pair in registers (the products and sums of k_gram), so a pixel is read once and
// nothing is staged; the CTA adds its threads' pairs in a fixed order.  The pairs are normalised
// after each chunk (8 products a thread), as one facet of 4096^2 adds 2048 of them in a thread,
// over which a low part that grows would round at 2^-41 of the sum instead of 2^-44.  Output slot
// blockIdx.x, as k_gram_sum leaves it.  The tensor-core kernel pads such facets to 16
// channels and pays a chunk's slicing and epilogue all the same: 1.61 ms at 4 channels of
// 4096^2 (256 facets), here 0.25 ms.
//
// The pairs hold while the squares and their rounding errors stay in FP32's range: a CTA that
// meets a channel whose largest |z| is not zero and lies outside [1e-15, 1e15] goes over
// its pixels again in FP64.
template <int LM>
__global__ void __launch_bounds__(128) k_gram_small(const float* __restrict__ xc, const float* __restrict__ P,
                                                    const NucFacet* __restrict__ facets,
                                                    const float* __restrict__ win, int n1, int n2, int L, int use_P,
                                                    double* __restrict__ part, int nchunk_max, int parts) {
  constexpr int NP = LM * (LM + 1) / 2, LD = NP | 1, SH = 128 / NP;   // shares of the final sum
  __shared__ float2 red[128 * LD];
  __shared__ float2 red2[SH * NP];
  __shared__ unsigned s_nonzero, s_normal;          // channels with |z| > 0, |z| >= 1e-15
  const int q = blockIdx.y, tid = threadIdx.x;
  const NucFacet f = facets[q];
  const int w = f.c1 - f.c0, Nq = (f.r1 - f.r0) * w, nch = (Nq + kGramChunk - 1) / kGramChunk;
  if ((int)blockIdx.x >= nch) return;
  const size_t N = (size_t)n1 * n2;
  auto load = [&](int p, float (&z)[LM]) {          // z of pixel p (zero past the facet and from L on)
    const bool in = p < Nq;
    const int rr = in ? p / w : 0, cc = in ? p - rr * w : 0;
    const float d = facet_weight(f, win, rr, cc);
    const float* xp = xc + (size_t)(f.r0 + rr) * n2 + (f.c0 + cc);
    const float* pp = P + f.p_off + p;
    float u[LM];
#pragma unroll
    for (int l = 0; l < LM; ++l) {
      z[l] = in && l < L ? xp[(size_t)l * N] : 0.f;
      u[l] = in && use_P && l < L ? pp[(size_t)l * Nq] : 0.f;
    }
#pragma unroll
    for (int l = 0; l < LM; ++l) z[l] = fmaf(d, z[l], u[l]);
  };
  if (tid == 0) s_nonzero = s_normal = 0;
  float hi[NP], lo[NP], big[LM];
#pragma unroll
  for (int e = 0; e < NP; ++e) hi[e] = lo[e] = 0.f;
#pragma unroll
  for (int l = 0; l < LM; ++l) big[l] = 0.f;
  for (int c = blockIdx.x; c < nch; c += parts) {
#pragma unroll 2
    for (int k = 0; k < kGramChunk / 128; ++k) {
      float z[LM];
      load(c * kGramChunk + k * 128 + tid, z);
#pragma unroll
      for (int l = 0; l < LM; ++l) big[l] = fmaxf(big[l], fabsf(z[l]));
      int e = 0;
#pragma unroll
      for (int b = 0; b < LM; ++b)
#pragma unroll
        for (int a = 0; a <= b; ++a, ++e) {
          const float pr = __fmul_rn(z[a], z[b]), pe = __fmaf_rn(z[a], z[b], -pr);
          float t, er;
          two_sum(hi[e], pr, t, er);
          hi[e] = t;
          lo[e] = __fadd_rn(lo[e], __fadd_rn(er, pe));
        }
    }
#pragma unroll
    for (int e = 0; e < NP; ++e) {                  // the low part back below the high one's rounding
      const float h = __fadd_rn(hi[e], lo[e]);
      lo[e] = __fsub_rn(lo[e], __fsub_rn(h, hi[e]));
      hi[e] = h;
    }
  }
  unsigned nonzero = 0, normal = 0;
  bool large = false;
#pragma unroll
  for (int l = 0; l < LM; ++l) {
    nonzero |= big[l] > 0.f ? 1u << l : 0u;
    normal |= big[l] >= 1e-15f ? 1u << l : 0u;
    large = large || big[l] > 1e15f;
  }
  __syncthreads();
  if (nonzero & ~s_nonzero) atomicOr(&s_nonzero, nonzero);
  if (normal & ~s_normal) atomicOr(&s_normal, normal);
  const bool fp64 = __syncthreads_or(large) || s_nonzero != s_normal;
  const auto entry = [&](int e, double v) {         // entry e of the triangle into the output slot
    int b = 0;
    while ((b + 1) * (b + 2) / 2 <= e) ++b;
    const int a = e - b * (b + 1) / 2;
    if (b < L) {
      double* out = part + ((size_t)q * nchunk_max + blockIdx.x) * L * L;
      out[a * L + b] = out[b * L + a] = v;
    }
  };
  if (fp64) {
    double* red64 = reinterpret_cast<double*>(red);
    double acc[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) acc[e] = 0.0;
#pragma unroll 1
    for (int c = blockIdx.x; c < nch; c += parts) {
#pragma unroll 1
      for (int k = 0; k < kGramChunk / 128; ++k) {
        float z[LM];
        load(c * kGramChunk + k * 128 + tid, z);
        int e = 0;
#pragma unroll
        for (int b = 0; b < LM; ++b)
#pragma unroll
          for (int a = 0; a <= b; ++a, ++e) acc[e] = fma((double)z[a], (double)z[b], acc[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < NP; ++e) red64[tid * LD + e] = acc[e];
    __syncthreads();
    if (tid < NP) {
      double v = 0.0;
      for (int t = 0; t < 128; ++t) v += red64[t * LD + tid];
      entry(tid, v);
    }
    return;
  }
#pragma unroll
  for (int e = 0; e < NP; ++e) red[tid * LD + e] = make_float2(hi[e], lo[e]);
  __syncthreads();
  if (tid < SH * NP) {
    const int e = tid % NP;
    ff s = {0.f, 0.f};
    for (int t = tid / NP; t < 128; t += SH) s = ff_add(s, {red[t * LD + e].x, red[t * LD + e].y});
    red2[tid] = make_float2(s.h, s.l);
  }
  __syncthreads();
  if (tid < NP) {
    ff s = {0.f, 0.f};
    for (int t = 0; t < SH; ++t) s = ff_add(s, {red2[t * NP + tid].x, red2[t * NP + tid].y});
    entry(tid, ff_val(s));
  }
}

// ------------------------------------------------------------ eigen-solve
// A GB300 SM issues one FP64 warp instruction per 64 clocks and sub-partition, whatever
// the number of active lanes (measured: 64 clk per dependent or independent DFMA, 431 for
// 1/x or rsqrt, 1.7 lanes/clk per SM), 76 times below FP32.  The Jacobi sweeps therefore run
// on pairs of floats (hi + lo, about 2^-47 of the largest entry), and V^T G V is then formed in
// FP64: its diagonal has FP64's eigenvalues, the entries beside it correct M to first order, and
// where that would not do (entries below about 1e-7 of the largest) further sweeps run in FP64.

// Plane rotation (c, s) that annihilates g of [[gpp, g], [g, grr]], d = grr - gpp, up to the
// FP32 accuracy of its tangent (the remainder is annihilated in the next sweep); c and s are
// float pairs with c^2 + s^2 = 1 to about 2^-46 (a rotation scales its two rows alike, so the
// remainder moves an eigenvalue by that much of itself).
__device__ __forceinline__ void ff_rotation(float g, float d, ff& c, ff& s) {
  // tan = g / (|d|/2 + sqrt(d^2/4 + g^2)) with the sign of d, both scaled by a power of two so
  // that the squares stay in range; it may be off by a few ulp and is taken as exact from here on
  const float unit = __int_as_float((254 - (__float_as_int(fmaxf(0.5f * fabsf(d), fabsf(g))) >> 23)) << 23);
  const float h2 = 0.5f * fabsf(d) * unit, gs = g * unit;
  float root;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(fmaf(h2, h2, gs * gs)));
  const float t = __fdividef(copysignf(1.f, d) * gs, h2 + root);
  // c = (1 + t^2)^-1/2, s = t c
  const float p = __fmul_rn(t, t), pe = __fmaf_rn(t, t, -p);
  const float uh = __fadd_rn(1.f, p);
  c = ff_rsqrt({uh, __fadd_rn(__fsub_rn(p, __fsub_rn(uh, 1.f)), pe)});
  const float sp = __fmul_rn(t, c.h);
  const float se = __fmaf_rn(t, c.l, __fmaf_rn(t, c.h, -sp));
  s.h = __fadd_rn(sp, se);
  s.l = __fsub_rn(se, __fsub_rn(s.h, sp));
}

// Whether a pair of the float-pair matrix is rotated: g above the accuracy of the pairs
// relative to the geometric mean of the diagonal (false for NaN): the mean and not the larger
// entry, so that channels many decades fainter than the others keep their own singular
// vectors.  `more`: g lies above that accuracy of the larger entry as well, so a further sweep
// is due.
__device__ __forceinline__ bool pair_turns(float pp, float g, float rr, bool& more) {
  constexpr float kEps = 5.7e-14f;                                              // 2^-44
  const bool some = fabsf(g) > 1e-36f;
  more = some && fabsf(g) > kEps * fmaxf(fabsf(pp), fabsf(rr));
  return some && fabsf(g) > kEps * (sqrtf(fabsf(pp)) * sqrtf(fabsf(rr)));
}

// Whether a pair of the FP64 matrix is rotated: whether that would change a result.  The
// rotation by about theta = g / max(|d|, |g|) moves the diagonal entries by theta g and their
// vectors by theta.  tp, tr: (squared threshold, m) of the entries.
//  weights: an entry moves by more than 1e-11 of itself and of its threshold (1e-8 of mu_bar);
//  duals: not if both entries stay below their thresholds (m = 1 for any vectors); else if the
//  second-order change of M exceeds 1e-8 of the larger m (the first order is added to M), or
//  the smaller entry moves by more than 1e-9 of itself and its threshold.
template <bool W>
__device__ __forceinline__ bool pair_turns64(double gpp, double g64, double grr, float2 tp, float2 tr) {
  const float g = fabsf((float)g64), d = fabsf((float)(grr - gpp));
  const float p = fabsf((float)gpp), r = fabsf((float)grr);
  const float theta = __fdividef(g, fmaxf(d, g)), move = g * theta;
  const bool less = p < r;
  const float small = less ? p : r, ts = less ? tp.x : tr.x, large = less ? r : p, tl = less ? tr.x : tp.x;
  if (!(g > 1e-36f)) return false;
  if (W) return move > 1e-11f * fmaxf(small, ts);
  if (small + move < 0.99f * ts && large + move < 0.99f * tl) return false;
  return theta * theta * fabsf(tp.y - tr.y) > 1e-8f * fmaxf(tp.y, tr.y) ||
         move > 1e-9f * fmaxf(small, fminf(ts, large));
}

constexpr int kEigRows = 3;        // eigenvector-row items per worker thread, at most
constexpr int kEigParts = 32;      // partial Grams per facet after k_gram_sum
constexpr int kEigDirect = 64;     // up to this many partials k_eig adds them itself

// Adds the chunk partials of a facet in a fixed order down to kEigParts: CTA g sums the
// chunks g, g + kEigParts, ... into chunk g (facets of more than kEigDirect chunks, where
// one CTA of k_eig would read megabytes alone).
__global__ void __launch_bounds__(256) k_gram_sum(double* __restrict__ part, int nchunk_max,
                                                  const NucFacet* __restrict__ facets, int L) {
  __shared__ double acc[256];
  const int q = blockIdx.y, g = blockIdx.x;
  const NucFacet f = facets[q];
  const int nch = ((f.r1 - f.r0) * (f.c1 - f.c0) + kGramChunk - 1) / kGramChunk;
  if (nch <= kEigParts || g >= nch) return;
  double* pq = part + (size_t)q * nchunk_max * L * L;
  const int LL = L * L;
  // up to 128 entries: thread -> (entry, share of the chunks), shares added in order
  const int share = LL <= 128 ? 256 / LL : 1;
  const int per = share > 1 ? LL : 256;
  const int e0 = threadIdx.x % per, sh = threadIdx.x / per;
  for (int eb = 0; eb < LL; eb += per) {
    const int e = eb + e0;
    double s = 0.0;
    if (e < LL && sh < share) {
      int c = g + kEigParts * sh;
      for (; c + 3 * kEigParts * share < nch; c += 4 * kEigParts * share) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = pq[(size_t)(c + k * kEigParts * share) * LL + e];
#pragma unroll
        for (int k = 0; k < 4; ++k) s += v[k];
      }
      for (; c < nch; c += kEigParts * share) s += pq[(size_t)c * LL + e];
    }
    if (share == 1) {
      if (e < LL) pq[(size_t)g * LL + e] = s;
    } else {
      acc[threadIdx.x] = s;
      __syncthreads();
      if (sh == 0 && e < LL) {
        for (int k = 1; k < share; ++k) s += acc[k * per + e0];
        pq[(size_t)g * LL + e] = s;
      }
    }
  }
}

__device__ __forceinline__ ff ldp(const float2* m, int k) {
  const float2 x = m[k];
  return ff{x.x, x.y};
}

// Cyclic Jacobi sweeps by the whole CTA over the symmetric matrix [Le][Le + 1] in float pairs
// (G) or, F64, in FP64 (G64, with thr = (squared threshold, m)); the rotations also go to the
// rows of V.  A sweep is Le - 1 rounds of the round-robin tournament over Le indices; a round
// rotates H = Le/2 disjoint pairs at once.  rot, rot64, pr: [2][H], c and s in pairs, the same
// in FP64 and the index pairs of a round; s_more: 1 + the last sweep that left a pair for
// another one, zero before.  Starts and ends with the matrices settled (barriers inside).
template <bool F64, bool W>
__device__ __forceinline__ void eig_sweeps(float2* __restrict__ G, double* __restrict__ G64, float2* __restrict__ V,
                                           float4* __restrict__ rot, double2* __restrict__ rot64,
                                           int2* __restrict__ pr, volatile int* s_more, int L, int max_sweeps,
                                           const float2* __restrict__ thr) {
  const int Le = (L + 1) & ~1, H = Le / 2, Ls = Le + 1, tid = threadIdx.x, nt = blockDim.x;
  const int nB = H * (H - 1) / 2, wt = tid - 32, nw = nt - 32;     // worker threads: warps 1 and up
  int bi = 0, bj = 0;                            // the worker's block: (pair bi) x (pair bj), bi < bj;
  const bool has_block = wt >= 0 && wt < 2 * nB; // lane parity: the row of pair bi it writes
  const unsigned block_lanes = __ballot_sync(0xffffffffu, has_block);
  const int half = wt & 1;
  if (has_block) {
    const int t = wt >> 1;
    bj = (int)((sqrtf(8.f * t + 1.f) + 1.f) * 0.5f);
    while (bj * (bj - 1) / 2 > t) --bj;
    while ((bj + 1) * bj / 2 <= t) ++bj;
    bi = t - bj * (bj - 1) / 2;
  }
  int vi[kEigRows], vk[kEigRows];                // its eigenvector rows: (pair, component)
#pragma unroll
  for (int m = 0; m < kEigRows; ++m) {
    const int k = wt + m * nw;
    vi[m] = wt >= 0 && k < H * L ? k / L : -1;
    vk[m] = vi[m] >= 0 ? k - vi[m] * L : 0;
  }
  auto stg = [&](int a, int b, ff x) { G[a * Ls + b] = G[b * Ls + a] = make_float2(x.h, x.l); };
  auto stg64 = [&](int a, int b, double x) { G64[a * Ls + b] = G64[b * Ls + a] = x; };
  // eigenvector rows of the round in buffer `buf` (an identity rotation leaves its pairs as
  // they are)
  auto rotate_rows = [&](int buf) {
    int o[kEigRows], o2[kEigRows];
    ff vp[kEigRows], vr[kEigRows];
    float4 r[kEigRows];
#pragma unroll
    for (int m = 0; m < kEigRows; ++m) {
      const int i = max(vi[m], 0);
      const int2 pi = pr[buf * H + i];
      r[m] = rot[buf * H + i];
      o[m] = pi.x * Ls + vk[m];
      o2[m] = pi.y * Ls + vk[m];
      vp[m] = ldp(V, o[m]);
      vr[m] = ldp(V, o2[m]);
    }
    bool turn = false;
#pragma unroll
    for (int m = 0; m < kEigRows; ++m) turn = turn || r[m].z != 0.f;
    if (!turn) return;
#pragma unroll
    for (int m = 0; m < kEigRows; ++m) {
      const ff c = {r[m].x, r[m].y}, s = {r[m].z, r[m].w};
      const ff x = ff_lin(c, vp[m], {-s.h, -s.l}, vr[m]), y = ff_lin(s, vp[m], c, vr[m]);
      if (vi[m] >= 0) {
        V[o[m]] = make_float2(x.h, x.l);
        V[o2[m]] = make_float2(y.h, y.l);
      }
    }
  };
  int buf = 0, rows_due = 0;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    int rotated = 0;
    for (int rnd = 0; rnd < Le - 1; ++rnd) {
      int mine = 0, p = 0, r = 0;
      ff c = {1.f, 0.f}, s = {0.f, 0.f};
      if (tid < 32) {
        if (tid < H) {
          auto player = [&](int k) {
            int x = k - 1 + rnd;
            x = x >= Le - 1 ? x - (Le - 1) : x;
            return k == 0 ? 0 : x + 1;
          };
          p = player(tid);
          r = player(Le - 1 - tid);
          if (p > r) { const int x = p; p = r; r = x; }
          bool more;
          if constexpr (F64) {
            const double gpp = G64[p * Ls + p], gpr = G64[p * Ls + r], grr = G64[r * Ls + r];
            more = pair_turns64<W>(gpp, gpr, grr, thr[p], thr[r]);
            mine = more ? 1 : 0;
            if (mine) ff_rotation((float)gpr, (float)(grr - gpp), c, s);
            rot64[buf * H + tid] = mine ? make_double2(ff_val(c), ff_val(s)) : make_double2(1.0, 0.0);
            rot[buf * H + tid] = make_float4(c.h, c.l, s.h, s.l);
          } else {
            const ff gpp = ldp(G, p * Ls + p), gpr = ldp(G, p * Ls + r), grr = ldp(G, r * Ls + r);
            mine = pair_turns(gpp.h, gpr.h + gpr.l, grr.h, more) ? 1 : 0;
            if (mine)
              ff_rotation(gpr.h + gpr.l, __fadd_rn(__fsub_rn(grr.h, gpp.h), __fsub_rn(grr.l, gpp.l)), c, s);
            rot[buf * H + tid] = make_float4(c.h, c.l, s.h, s.l);
          }
          if (more) *s_more = sweep + 1;
          pr[buf * H + tid] = make_int2(p, r);
        }
      } else if (rows_due) {
        rotate_rows(buf ^ 1);
      }
      const int any = __syncthreads_or(mine);
      if (any) {
        rotated = 1;
        if (tid < 32) {
          if (mine) {                                        // diagonal block
            if constexpr (F64) {
              const double2 t = rot64[buf * H + tid];
              const double gpp = G64[p * Ls + p], gpr = G64[p * Ls + r], grr = G64[r * Ls + r];
              const double a1 = t.x * gpp - t.y * gpr, b1 = t.x * gpr - t.y * grr;
              const double c1 = t.y * gpp + t.x * gpr, d1 = t.y * gpr + t.x * grr;
              stg64(p, p, t.x * a1 - t.y * b1);
              stg64(p, r, t.y * a1 + t.x * b1);
              stg64(r, r, t.y * c1 + t.x * d1);
            } else {
              const ff gpp = ldp(G, p * Ls + p), gpr = ldp(G, p * Ls + r), grr = ldp(G, r * Ls + r);
              const ff ns = {-s.h, -s.l};
              const ff a1 = ff_lin(c, gpp, ns, gpr), b1 = ff_lin(c, gpr, ns, grr);
              const ff c1 = ff_lin(s, gpp, c, gpr), d1 = ff_lin(s, gpr, c, grr);
              stg(p, p, ff_lin(c, a1, ns, b1));
              stg(p, r, ff_lin(s, a1, c, b1));
              stg(r, r, ff_lin(s, c1, c, d1));
            }
          }
        } else if (has_block) {
          // the two threads of a block read all of it, then write a row each
          const int2 pi = pr[buf * H + bi], pj = pr[buf * H + bj];
          const int row = half ? pi.y : pi.x, other = half ? pi.x : pi.y;
          if constexpr (F64) {
            const double2 ri = rot64[buf * H + bi], rj = rot64[buf * H + bj];
            const bool turn = ri.y != 0.0 || rj.y != 0.0;    // (the same for both threads)
            double a2 = 0.0, b2 = 0.0;
            if (turn) {
              const double ci = ri.x, si = half ? ri.y : -ri.y;
              const double a = G64[row * Ls + pj.x], b = G64[row * Ls + pj.y];
              const double d = G64[other * Ls + pj.x], e = G64[other * Ls + pj.y];
              const double a1 = ci * a + si * d, b1 = ci * b + si * e;
              a2 = rj.x * a1 - rj.y * b1;
              b2 = rj.y * a1 + rj.x * b1;
            }
            __syncwarp(block_lanes);
            if (turn) {
              stg64(row, pj.x, a2);
              stg64(row, pj.y, b2);
            }
          } else {
            const float4 ri = rot[buf * H + bi], rj = rot[buf * H + bj];
            const ff ci = {ri.x, ri.y}, si = half ? ff{ri.z, ri.w} : ff{-ri.z, -ri.w};
            const ff cj = {rj.x, rj.y}, sj = {rj.z, rj.w};
            const ff a = ldp(G, row * Ls + pj.x), b = ldp(G, row * Ls + pj.y);
            const ff d = ldp(G, other * Ls + pj.x), e = ldp(G, other * Ls + pj.y);
            const ff a1 = ff_lin(ci, a, si, d), b1 = ff_lin(ci, b, si, e);
            const ff a2 = ff_lin(cj, a1, {-sj.h, -sj.l}, b1), b2 = ff_lin(sj, a1, cj, b1);
            __syncwarp(block_lanes);
            stg(row, pj.x, a2);
            stg(row, pj.y, b2);
          }
        }
        __syncthreads();
      }
      rows_due = any;
      buf ^= 1;
    }
    // (s_more only grows, so a thread that reads it late still sees that the sweep was not the last)
    if (!rotated || (sweep > 0 && *s_more <= sweep)) break;
  }
  if (rows_due && wt >= 0) rotate_rows(buf ^ 1);
  __syncthreads();
}

// Threads of k_eig: warp 0 (rotations, diagonal blocks) and two threads per 2 x 2 block of G
// above the diagonal blocks, which rotate the eigenvector rows as well.
static int eig_threads(int L) {
  const int H = (L + 1) / 2, nB = H * (H - 1) / 2;
  const int work = std::max(2 * nB, (H * L + kEigRows - 1) / kEigRows);
  return 32 + std::max(32, (work + 31) & ~31);
}
static size_t eig_smem(int L) {
  const size_t Le = (L + 1) & ~1, H = Le / 2;
  return 4 * Le * (Le + 1) * sizeof(float2) + 2 * H * (2 * sizeof(float4) + sizeof(int2)) +
         Le * (3 * sizeof(float2) + sizeof(float));
}

// One CTA per facet: G = sum of the partial Grams (FP64, chunk order), cyclic Jacobi
// eigen-decomposition G = V diag(lambda) V^T in float pairs, s = sqrt(max(lambda, 0))
// sorted descending, then either M = V diag(m) V^T with m_j = min(1, alpha_j / s_j),
// alpha_j = (mu_bar_q / zeta) theta_bar_q[rank j] (dual mode), or
// theta_bar_q[rank] = mu_bar_q / (s + mu_bar_q) (W, weights mode); lambda in FP64 as above.
//
// Bound by the latency of a round: the rotations of H = Le/2 disjoint index pairs (warp 0,
// about 500 clk), a barrier, every 2 x 2 block of G transformed in place from both
// sides by two threads, a barrier; the eigenvector rows of a round are rotated
// beside the next round's rotations.  One warp in FP64 took 1.09 ms at 20
// channels (16 facets), 3.74 ms at 32 (64 facets) and, for the weights, 6.48 ms at 38 (36
// facets); this kernel takes 0.125, 0.29 and 0.35 ms (device times of one launch; 0.098, 0.24
// and 0.33 without the FP64 stage).
template <bool W>
__global__ void __launch_bounds__(1024) k_eig(const double* __restrict__ part, int nchunk_max, int nparts_max,
                                             const NucFacet* __restrict__ facets, int L,
                                             const float* __restrict__ theta_bar, const float* __restrict__ mubar,
                                             float inv_zeta, float* __restrict__ Mout, float* __restrict__ tb_out,
                                             int max_sweeps) {
  extern __shared__ __align__(16) unsigned char eig_smem_raw[];
  __shared__ int s_emax;
  __shared__ volatile int s_more;
  const int Le = (L + 1) & ~1, H = Le / 2, Ls = Le + 1;
  float4* rot = reinterpret_cast<float4*>(eig_smem_raw);          // [2][H] (c, s) of a round
  double2* rot64 = reinterpret_cast<double2*>(rot + 2 * H);       // [2][H] the same in FP64
  int2* pr = reinterpret_cast<int2*>(rot64 + 2 * H);              // [2][H] index pairs of a round
  float2* G = reinterpret_cast<float2*>(pr + 2 * H);              // [Le][Ls] pairs, index L (odd L): zeros
  float2* V = G + Le * Ls;                                        // [Le][Ls], row j = eigenvector j
  double* G64 = reinterpret_cast<double*>(V + Le * Ls);           // [Le][Ls] G, then V^T G V
  double* V64 = reinterpret_cast<double*>(G);                     // [Le][Ls] V, once G is solved
  double* W64 = G64 + Le * Ls;                                    // [Le][Ls] V^T G
  float2* lam = reinterpret_cast<float2*>(W64 + Le * Ls);         // [Le]
  float2* tm = lam + Le;                                          // [Le] m_j
  float2* thr = tm + Le;                                          // [Le] squared threshold, m (duals)
  float* tbq = reinterpret_cast<float*>(thr + Le);                // [Le]
  const int q = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const NucFacet f = facets[q];
  const int Nq = (f.r1 - f.r0) * (f.c1 - f.c0);
  const int nch = min((Nq + kGramChunk - 1) / kGramChunk, nparts_max);
  const float mb = mubar[q];
  if (tid == 0) { s_emax = 0; s_more = 0; }
  for (int k = tid; k < Le * Ls; k += nt) {
    const int a = k / Ls, b = k - a * Ls;
    G[k] = make_float2(0.f, 0.f);
    V[k] = make_float2(a == b ? 1.f : 0.f, 0.f);
    G64[k] = 0.0;
  }
  if (!W)
    for (int j = tid; j < L; j += nt) tbq[j] = theta_bar[(size_t)q * L + j];
  __syncthreads();
  // ---- G (upper triangle; the partials are symmetric), kept in FP64 registers until the
  // scale 4^-k that takes the largest diagonal entry into [1, 4) is known
  const int nE = L * (L + 1) / 2;
  constexpr int kHold = 5;                       // nE <= kHold nt for every L <= 64
  double g64[kHold];
  const double* pq = part + (size_t)q * nchunk_max * L * L;
  auto entry = [](int e, int& a, int& b) {       // e -> (a, b), a <= b
    b = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
    while (b * (b + 1) / 2 > e) --b;
    while ((b + 1) * (b + 2) / 2 <= e) ++b;
    a = e - b * (b + 1) / 2;
  };
#pragma unroll
  for (int u = 0; u < kHold; ++u) {
    const int e = tid + u * nt;
    g64[u] = 0.0;
    if (e >= nE) continue;
    int a, b;
    entry(e, a, b);
    double s = 0.0;
    int c = 0;
    for (; c + 8 <= nch; c += 8) {
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = pq[(size_t)(c + k) * L * L + a * L + b];
#pragma unroll
      for (int k = 0; k < 8; ++k) s += v[k];
    }
    for (; c < nch; ++c) s += pq[(size_t)c * L * L + a * L + b];
    g64[u] = s;
    if (a == b) {
      const int ex = (__double2hiint(s) >> 20) & 0x7ff;
      if (ex != 0x7ff) atomicMax(&s_emax, ex);
    }
  }
  __syncthreads();
  // 4^k <= largest diagonal entry < 4^(k+1)
  const int k4 = s_emax == 0 ? 0 : (s_emax - 1023) >> 1;
  const double down = __hiloint2double((1023 - 2 * k4) << 20, 0);
#pragma unroll
  for (int u = 0; u < kHold; ++u) {
    const int e = tid + u * nt;
    if (e >= nE) continue;
    int a, b;
    entry(e, a, b);
    const double g = g64[u] * down;
    ff x = ff_of(g);
    if (!(fabsf(x.h) < 3e38f)) x = {__int_as_float(0x7fffffff), 0.f};
    G[a * Ls + b] = G[b * Ls + a] = make_float2(x.h, x.l);
    G64[a * Ls + b] = G64[b * Ls + a] = g;
  }
  __syncthreads();
  eig_sweeps<false, W>(G, nullptr, V, rot, rot64, pr, &s_more, L, max_sweeps, nullptr);
  // ---- V^T G V in FP64.  Terms of faint channels are as small as what they add up to, so
  // they keep their relative accuracy
  for (int k = tid; k < Le * Ls; k += nt) V64[k] = ff_val(ldp(V, k));
  if (tid == 0) s_more = 0;
  __syncthreads();
  for (int k = tid; k < L * L; k += nt) {
    const int j = k / L, b = k - j * L;
    double y = 0.0;
    for (int a = 0; a < L; ++a) y = fma(V64[j * Ls + a], G64[a * Ls + b], y);
    W64[j * Ls + b] = y;
  }
  __syncthreads();
  for (int e = tid; e < nE; e += nt) {
    int a, b;
    entry(e, a, b);
    double y = 0.0;
    for (int k = 0; k < L; ++k) y = fma(W64[a * Ls + k], V64[b * Ls + k], y);
    G64[a * Ls + b] = G64[b * Ls + a] = y;
  }
  __syncthreads();
  auto diagonal = [&]() {
    for (int j = tid; j < L; j += nt) {
      const ff x = ff_of(G64[j * Ls + j]);
      lam[j] = make_float2(x.h, x.l);
    }
    __syncthreads();
  };
  auto rank_of = [&](int j) {
    const float2 x = lam[j];
    int rk = 0;
#pragma unroll 4
    for (int k = 0; k < L; ++k) {
      const float2 y = lam[k];
      rk += (y.x > x.x) || (y.x == x.x && (y.y > x.y || (y.y == x.y && k < j)));
    }
    return rk;
  };
  // squared thresholds of the entries: duals, the smallest alpha from the entry's rank on;
  // weights, (3e-3 mu_bar)^2
  const double unit = __hiloint2double((1023 - k4) << 20, 0);
  diagonal();
  for (int j = tid; j < Le; j += nt) {
    float t = 3e-3f, m = 1.f;
    if (!W && j < L) {
      const int rk = rank_of(j);
      t = INFINITY;
      for (int k = rk; k < L; ++k) t = fminf(t, tbq[k]);
      const float al = (float)((double)mb * (double)inv_zeta * (double)tbq[rk] * unit);
      m = fminf(1.f, al * rsqrtf(fmaxf(lam[j].x, 1e-37f)));
    }
    t = (float)((double)mb * (W ? 1.0 : (double)inv_zeta) * (double)t * unit);
    thr[j] = make_float2(t * t, m);
  }
  __syncthreads();
  int due = 0;
  for (int e = tid; e < nE; e += nt) {
    int a, b;
    entry(e, a, b);
    if (a != b && pair_turns64<W>(G64[a * Ls + a], G64[a * Ls + b], G64[b * Ls + b], thr[a], thr[b])) due = 1;
  }
  if (__syncthreads_or(due)) {
    eig_sweeps<true, W>(nullptr, G64, V, rot, rot64, pr, &s_more, L, max_sweeps, thr);
    diagonal();
  }
  for (int j = tid; j < L; j += nt) {
    const int rk = rank_of(j);
    if constexpr (W) {
      const double sv = sqrt(fmax(G64[j * Ls + j], 0.0)) * __hiloint2double((1023 + k4) << 20, 0);
      tb_out[(size_t)q * L + rk] = (float)((double)mb / (sv + (double)mb));
    } else {
      // m = min(1, alpha lambda^-1/2) in the scaled units, 1 where lambda is not positive
      const ff al = ff_of((double)mb * (double)inv_zeta * (double)tbq[rk] * unit), x = ldp(lam, j);
      ff m = {1.f, 0.f};
      if (x.h > 0.f) {
        const ff t = ff_mul(al, ff_rsqrt(x));
        if (t.h < 1.f || (t.h == 1.f && t.l < 0.f)) m = t;
      }
      tm[j] = make_float2(m.h, m.l);
    }
  }
  if constexpr (!W) {
    __syncthreads();
    // first order of what the pairs left beside the diagonal: M = V (diag(m) + F) V^T with
    // F_ij = B_ij (m_i - m_j) / (lambda_i - lambda_j), B = V^T G V (F over V^T G, then
    // (diag(m) + F) V^T over G)
    float* F = reinterpret_cast<float*>(W64);
    for (int k = tid; k < L * L; k += nt) {
      const int i = k / L, j = k - i * L;
      const float dm = __fadd_rn(__fsub_rn(tm[i].x, tm[j].x), __fsub_rn(tm[i].y, tm[j].y));
      const float d = __fadd_rn(__fsub_rn(lam[i].x, lam[j].x), __fsub_rn(lam[i].y, lam[j].y));
      F[k] = dm != 0.f && d != 0.f ? (float)G64[i * Ls + j] / d * dm : 0.f;
    }
    __syncthreads();
    for (int k = tid; k < L * L; k += nt) {
      const int j = k / L, c = k - j * L, o = j * Ls + c;
      float first = 0.f;
#pragma unroll 4
      for (int i = 0; i < L; ++i) first = fmaf(F[j * L + i], V[i * Ls + c].x, first);
      const ff w = ff_add(ff_mul(ldp(tm, j), ldp(V, o)), {first, 0.f});
      G[o] = make_float2(w.h, w.l);
    }
    __syncthreads();
    // M_q^T, rows padded to Lp = L rounded up to 4 (zeros), so that a row is read as float4;
    // each entry (symmetric) is summed in float pairs and rounded once
    const int Lp = (L + 3) & ~3;
    float* Mq = Mout + (size_t)q * L * Lp;
    for (int e = tid; e < nE; e += nt) {
      int a, b;
      entry(e, a, b);
      ff m0 = {0.f, 0.f}, m1 = {0.f, 0.f};
      const ff one = {1.f, 0.f};
      int j = 0;
#pragma unroll 2
      for (; j + 2 <= L; j += 2) {
        m0 = ff_lin(ldp(G, j * Ls + b), ldp(V, j * Ls + a), one, m0);
        m1 = ff_lin(ldp(G, (j + 1) * Ls + b), ldp(V, (j + 1) * Ls + a), one, m1);
      }
      if (j < L) m0 = ff_lin(ldp(G, j * Ls + b), ldp(V, j * Ls + a), one, m0);
      m0 = ff_lin(one, m0, one, m1);
      Mq[b * Lp + a] = Mq[a * Lp + b] = m0.h + m0.l;
    }
    for (int k = tid; k < L * (Lp - L); k += nt) Mq[(k / (Lp - L)) * Lp + L + k % (Lp - L)] = 0.f;
  }
}

// Pixel-driven update: each thread owns one pixel; for every facet covering it,
// z = P_q + D_q x, P_q <- z M_q, A += zeta D_q P_q.  BB outputs at a time: their rows of
// M_q^T are read as float4 (the same address across the warp, L1) against 4 FMAs a row and
// load, and the BB accesses to A and to P are in flight together.  One output at a time, with
// A read and written between the outputs above 16 channels, took 0.744 ms at 1024^2 x 32 (64
// facets) and 1.50 ms at 4096^2 x 16 (256 facets); now 0.378 and 1.33 ms (4.4 TB/s).  BB (8 at
// 32 channels, else 4) and the register limits by measurement: at 16 channels BB = 8 spills (1.74 ms at 64
// registers) or loses occupancy (2.89 ms at 154), BB = 2 1.45 ms; at 32 channels BB = 4 0.419.
template <int LMAX>
__global__ void __launch_bounds__(256, LMAX == 16 ? 4 : (LMAX == 32 ? 3 : 2)) k_apply(const float* __restrict__ xc, float* __restrict__ P,
                                               const NucFacet* __restrict__ facets, const float* __restrict__ win,
                                               const float* __restrict__ Mt, int n1, int n2, int L, int Qy, int Qx,
                                               const int* __restrict__ ty_of, const int* __restrict__ tx_of,
                                               float zeta, float* __restrict__ A) {
  constexpr int BB = LMAX == 32 ? 8 : 4;
  const int c = blockIdx.x * 32 + (threadIdx.x & 31);
  const int r = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (r >= n1 || c >= n2) return;
  const size_t N = (size_t)n1 * n2;
  const size_t pix = (size_t)r * n2 + c;
  const int Lp = (L + 3) & ~3;
  const int ty = ty_of[r], tx = tx_of[c];
#pragma unroll 1
  for (int d4 = 0; d4 < 4; ++d4) {
    const int qy = ty + (d4 >> 1), qx = tx + (d4 & 1);
    if (qy >= Qy || qx >= Qx) continue;
    const NucFacet f = facets[qy * Qx + qx];
    if (r < f.r0 || r >= f.r1 || c < f.c0 || c >= f.c1) continue;
    const int w = f.c1 - f.c0;
    const int Nq = (f.r1 - f.r0) * w;
    const int p = (r - f.r0) * w + (c - f.c0);
    const float d = facet_weight(f, win, r - f.r0, c - f.c0);
    float* Pq = P + f.p_off + p;
    float z[LMAX];
#pragma unroll
    for (int l = 0; l < LMAX; ++l) z[l] = (l < L) ? fmaf(d, xc[l * N + pix], Pq[(size_t)l * Nq]) : 0.f;
    const float4* Mq = reinterpret_cast<const float4*>(Mt + (size_t)(qy * Qx + qx) * L * Lp);
    const float zd = zeta * d;
#pragma unroll 1
    for (int b0 = 0; b0 < L; b0 += BB) {
      float s[BB], a_old[BB];
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        a_old[b] = (b0 + b < L) ? A[(size_t)(b0 + b) * N + pix] : 0.f;
        s[b] = 0.f;
      }
#pragma unroll
      for (int a4 = 0; a4 < LMAX / 4; ++a4) {
        if (4 * a4 >= L) break;
#pragma unroll
        for (int b = 0; b < BB; ++b) {
          const float4 m = __ldg(Mq + (size_t)min(b0 + b, L - 1) * (Lp / 4) + a4);
          s[b] = fmaf(z[4 * a4], m.x, s[b]);
          s[b] = fmaf(z[4 * a4 + 1], m.y, s[b]);
          s[b] = fmaf(z[4 * a4 + 2], m.z, s[b]);
          s[b] = fmaf(z[4 * a4 + 3], m.w, s[b]);
        }
      }
#pragma unroll
      for (int b = 0; b < BB; ++b)
        if (b0 + b < L) {
          Pq[(size_t)(b0 + b) * Nq] = s[b];
          A[(size_t)(b0 + b) * N + pix] = fmaf(zd, s[b], a_old[b]);
        }
    }
  }
}

static int nchunk_max(const Cube& cb) { return (cb.max_facet_pix + kGramChunk - 1) / kGramChunk; }

void launch_nuclear(fhs_ctx* ctx, const Cube& cb, const float* xcheck, float* P, const float* theta_bar, float* A,
                    bool weights_mode, float* theta_bar_out, cudaStream_t st) {
  launch_nuclear_gram_eig(ctx, cb, xcheck, P, theta_bar, weights_mode, theta_bar_out, st);
  if (!weights_mode) launch_nuclear_apply(ctx, cb, xcheck, P, A, st);
}

static void gram_cuda_core(fhs_ctx* ctx, const Cube& cb, const float* xcheck, const float* P, cudaStream_t st) {
  const int L = cb.L, nch = nchunk_max(cb), use_P = P != nullptr ? 1 : 0;
  dim3 gg(nch, cb.Qy * cb.Qx);
  auto go = [&](auto kernel) {
    kernel<<<gg, 256, 0, st>>>(xcheck, P, cb.d_facets, cb.d_win, cb.n1, cb.n2, L, use_P, ctx->s.gram, nch);
  };
  if (L <= 4) go(k_gram<1>);
  else if (L <= 16) go(k_gram<2>);
  else go(k_gram<4>);
  note_launches(1);
}

static void gram_weights(fhs_ctx* ctx, const Cube& cb, const float* x, cudaStream_t st) {
  const int L = cb.L, nch = nchunk_max(cb);
  auto go = [&](auto kernel, int LB) {
    const int nb = (L + LB - 1) / LB, z = (nb * (nb + 1) / 2 + kGramShare - 1) / kGramShare;
    kernel<<<dim3(nch, cb.Qy * cb.Qx, z), 256, 0, st>>>(x, cb.d_facets, cb.d_win64, cb.n1, cb.n2, L, ctx->s.gram, nch);
  };
  if (L <= 4) go(k_gram_f64<1>, 1);
  else if (L <= 16) go(k_gram_f64<2>, 2);
  else go(k_gram_f64<4>, 4);
  note_launches(1);
}

// Per-chunk partial Grams of Z_q = D_q S~_q xcheck (+ P_q) into ctx->s.gram: the tcgen05
// kernel when tc and 8 < L <= 32, k_gram_small when tc and L <= 8, else the CUDA-core
// float-float kernel.  Returns the partials per facet (at most one per chunk).
int launch_gram(fhs_ctx* ctx, const Cube& cb, const float* xcheck, const float* P, bool tc, cudaStream_t st) {
  const int nch = nchunk_max(cb);
  if (tc && cb.L <= 8) {
    // a wave of eight CTAs per SM over the facets, each adding up its chunks; at most the
    // kEigDirect partials a facet that k_eig adds itself, so fewer CTAs below 19 facets (one
    // facet of 4096^2 x 4 still takes 2.1 ms with its update where the tensor-core kernel took 10.2)
    const int Q = cb.Qy * cb.Qx, parts = std::max(1, std::min({(8 * num_sms() + Q - 1) / Q, nch, kEigDirect}));
    const int use_P = P != nullptr ? 1 : 0;
    auto go = [&](auto kernel) {
      kernel<<<dim3(parts, Q), 128, 0, st>>>(xcheck, P, cb.d_facets, cb.d_win, cb.n1, cb.n2, cb.L, use_P, ctx->s.gram,
                                             nch, parts);
    };
    if (cb.L <= 4) go(k_gram_small<4>);
    else go(k_gram_small<8>);
    note_launches(1);
    return parts;
  }
  if (!tc || !launch_gram_tc(cb, xcheck, P, ctx->s.gram, nch, st))         // counts its launch
    gram_cuda_core(ctx, cb, xcheck, P, st);
  return nch;
}

void launch_nuclear_gram_eig(fhs_ctx* ctx, const Cube& cb, const float* xcheck, const float* P,
                             const float* theta_bar, bool weights_mode, float* theta_bar_out, cudaStream_t st) {
  const int L = cb.L;
  const int Q = cb.Qy * cb.Qx;
  const int nch = nchunk_max(cb);
  int parts = nch;
  if (weights_mode) gram_weights(ctx, cb, xcheck, st);
  else parts = launch_gram(ctx, cb, xcheck, P, ctx->path == FHS_PATH_FAST && cb.gram_tc, st);
  const bool sum = parts > kEigDirect;
  if (sum) {
    k_gram_sum<<<dim3(kEigParts, Q), 256, 0, st>>>(ctx->s.gram, nch, cb.d_facets, L);
    note_launches(1);
  }
  auto go = [&](auto kernel, bool& attr) {
    if (!attr) {
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eig_smem(kMaxL));
      attr = true;
    }
    kernel<<<Q, eig_threads(L), eig_smem(L), st>>>(
        ctx->s.gram, nch, sum ? kEigParts : parts, cb.d_facets, L, theta_bar, cb.d_mubar, (float)(1.0 / cb.zeta),
        ctx->s.nucM, theta_bar_out, 40);
  };
  static bool attr_w = false, attr_d = false;
  if (weights_mode) go(k_eig<true>, attr_w);
  else go(k_eig<false>, attr_d);
  note_launches(1);
}

void launch_nuclear_apply(fhs_ctx* ctx, const Cube& cb, const float* xcheck, float* P, float* A, cudaStream_t st) {
  const int L = cb.L;
  dim3 ga((cb.n2 + 31) / 32, (cb.n1 + 7) / 8);
  const int* tyo = cb.d_tile_of;
  const int* txo = cb.d_tile_of + cb.n1;
  float zeta = (float)cb.zeta;
  if (L <= 16) k_apply<16><<<ga, 256, 0, st>>>(xcheck, P, cb.d_facets, cb.d_win, ctx->s.nucM, cb.n1, cb.n2, L, cb.Qy, cb.Qx, tyo, txo, zeta, A);
  else if (L <= 32) k_apply<32><<<ga, 256, 0, st>>>(xcheck, P, cb.d_facets, cb.d_win, ctx->s.nucM, cb.n1, cb.n2, L, cb.Qy, cb.Qx, tyo, txo, zeta, A);
  else k_apply<64><<<ga, 256, 0, st>>>(xcheck, P, cb.d_facets, cb.d_win, ctx->s.nucM, cb.n1, cb.n2, L, cb.Qy, cb.Qx, tyo, txo, zeta, A);
  note_launches(1);
}

}  // namespace fhs
