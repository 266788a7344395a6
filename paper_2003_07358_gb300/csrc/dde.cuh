// DDE-extended de-gridding and gridding (Section 2.1, the paragraph after Eq. 1), for
// sm_103a.  Included at the end of nufft.cu (it uses that file's Kaiser-Bessel taps,
// grid layout and block reductions).
//
// Row m of G_l is the Kaiser-Bessel kernel convolved with the visibility's compact
// Fourier-domain DDE kernel K_m ((2R + 1)^2 complex, R <= 4):
//   g_m[k] = sum_j K_m[j] phi(t_r - (k_r - j_r)) phi(t_c - (k_c - j_c)),
// a footprint of F x F cells, F = 7 + 2R (15 x 15 for 9 x 9 kernels), from cell
// (k0_r - R, k0_c - R), k0 the first Kaiser-Bessel tap.  In footprint coordinates
// (row r, column c; kernel index j1, j2 in [0, 2R]; taps a = r - j1, b = c - j2):
//   de-gridding  u_m = sum_{j1,j2} K[j1][j2] sum_a w_r[a] sum_b w_c[b] x[j1 + a][j2 + b]
//   gridding     x[r][c] += sum_b w_c[b] sum_a w_r[a] conj(K[r - a][c - b]) v_m
// Both are separable passes of which each lane of a half-warp runs one row or column in
// registers (a polynomial product: F x 7 or SD x 7 complex FMAs with no shared-memory
// operand), with one transposition through shared memory in between; a warp works on two
// visibilities at a time.  De-gridding: lane c takes column c of the window (its loads
// coalesce along the row), then lane j1 row j1 of the intermediate and of the kernel.
// Gridding: lane j1 takes row j1 of the kernel, then lane c column c of the footprint, so a
// row's atomics fall on consecutive cells.  Lanes 0..13 of a half hold the polynomial of
// one Kaiser-Bessel tap each and exchange the 14 weights by shuffles.
// (One visibility per warp with every pass reading its operands from shared memory took
// 2.04 ms to de-grid and 4.03 to 4.13 ms to grid 2.1 M visibilities of 16 channels of 1024^2
// with 9 x 9 kernels, about 700 instructions a visibility; this form takes 0.83 and
// 1.64 ms, bound by issue: 126 FMAs a pass and lane, and for the gridder 30 conversions and
// atomics.)
//
// Gridding keeps the scheme of k_grid: one CTA per (grid tile, channel) owns the tile's
// cells in shared memory and adds, in 32-bit fixed point with integer atomics (order-
// independent, so bitwise deterministic), every footprint cell that falls in the tile.
// Visibilities are bucketed by the tile of their first tap, and a footprint (F <= 15 <
// tile side) reaches only the 3 x 3 neighbouring tiles, so a CTA scans those buckets,
// keeps (by warp ballot) the visibilities whose footprint meets its tile, and processes
// them two by two.  The scale S = 2^e of a tile satisfies C m S < 2^30 with C the largest sum
// over one of its cells of the extended weights covering it, sum_j (|Re K_j| + |Im K_j|)
// phi phi (summed once per kernel set, MODE 1), and m = max over the contributing
// visibilities of max(|Re v|, |Im v|).

namespace fhs {

constexpr int kDdeThreads = 256;
constexpr int kDdeWarps = kDdeThreads / 32;

constexpr int kDdeLd = 17;            // row pitch of the transposition (float2): odd, over 15 columns

// The polynomial of the lane's tap (row taps on lanes 0..6 of a half, column taps on 7..13).
struct DdeTap {
  float c[kPolyDeg + 1];
};
__device__ __forceinline__ DdeTap dde_tap_poly(int lane) {
  const int j = lane & 15, t = j < kTaps ? j : (j < 2 * kTaps ? j - kTaps : 0);
  DdeTap p;
#pragma unroll
  for (int d = 0; d <= kPolyDeg; ++d) p.c[d] = c_kb.c[t][d];
  return p;
}

// Row and column Kaiser-Bessel weights of the half-warp's visibility on each of its lanes.
__device__ __forceinline__ void dde_weights(const DdeTap& p, float xr, float xc, int lane, float* wr, float* wc) {
  const float x = (lane & 15) < kTaps ? xr : xc;
  float w = p.c[kPolyDeg];
#pragma unroll
  for (int d = kPolyDeg - 1; d >= 0; --d) w = fmaf(w, x, p.c[d]);
  const int h = lane & 16;
#pragma unroll
  for (int b = 0; b < kTaps; ++b) {
    wr[b] = __shfl_sync(0xffffffffu, w, h + b);
    wc[b] = __shfl_sync(0xffffffffu, w, h + kTaps + b);
  }
}

// u_m of the visibility of each half-warp (the value is returned on the half's lanes); tr:
// the half's [SD][kDdeLd] scratch.
template <int R>
__device__ __forceinline__ float2 dde_degrid_half(const float2* __restrict__ gl, float2 uvm,
                                                  const float2* __restrict__ Km, const VisGeom& vg, const DdeTap& tap,
                                                  float2* tr, int lane) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R;
  const int j = lane & 15;
  float xr, xc, wr[kTaps], wc[kTaps];
  const int kr = kb_first(uvm.y, vg.tc.hi_r, vg.tc.lo_r, xr);
  const int kc = kb_first(uvm.x, vg.tc.hi_c, vg.tc.lo_c, xc);
  // the lane's column of the window and its row of the kernel, all loads in flight
  const float2* col = gl + wrap2(kc - R + min(j, F - 1), vg);
  float2 x[F], K[SD];
#pragma unroll
  for (int r = 0; r < F; ++r) x[r] = __ldg(col + (size_t)phys_row2(wrap1(kr - R + r, vg), vg) * vg.K2);
  const float2* Kr = Km + min(j, SD - 1) * SD;
#pragma unroll
  for (int j2 = 0; j2 < SD; ++j2) K[j2] = __ldg(Kr + j2);
  dde_weights(tap, xr, xc, lane, wr, wc);
  // row pass: mid[j1][c] = sum_a w_r[a] x[j1 + a][c]
#pragma unroll
  for (int j1 = 0; j1 < SD; ++j1) {
    float2 m = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < kTaps; ++a) {
      m.x = fmaf(wr[a], x[j1 + a].x, m.x);
      m.y = fmaf(wr[a], x[j1 + a].y, m.y);
    }
    if (j < F) tr[j1 * kDdeLd + j] = m;
  }
  __syncwarp();
  // column pass and the kernel row: u = sum_j2 K[j1][j2] sum_b w_c[b] mid[j1][j2 + b]
  float2 u = make_float2(0.f, 0.f);
  if (j < SD) {
    float2 m[F];
#pragma unroll
    for (int c = 0; c < F; ++c) m[c] = tr[j * kDdeLd + c];
#pragma unroll
    for (int j2 = 0; j2 < SD; ++j2) {
      float2 I = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < kTaps; ++b) {
        I.x = fmaf(wc[b], m[j2 + b].x, I.x);
        I.y = fmaf(wc[b], m[j2 + b].y, I.y);
      }
      u.x = fmaf(K[j2].x, I.x, fmaf(-K[j2].y, I.y, u.x));
      u.y = fmaf(K[j2].x, I.y, fmaf(K[j2].y, I.x, u.y));
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
    u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
  }
  __syncwarp();                         // the scratch is reused by the next visibility
  return u;
}

// MODE 0: out[i] = u_i.  MODE 1: the PDFB data step of k_degrid_pdfb (z = v + 2u - u_prev,
// d = z - y, u_prev <- u, per-block FP64 partial sums).  CTA = 256 consecutive
// visibilities of channel blockIdx.y; half h of warp w computes those of lanes
// 32 w + 16 h .. + 15 one by one, and each lane keeps its own for the per-visibility epilogue.
template <int R, int MODE>
__global__ void __launch_bounds__(kDdeThreads) k_degrid_dde(const float2* __restrict__ grid,
                                                            const float2* __restrict__ uv,
                                                            const float2* __restrict__ kern,
                                                            const int32_t* __restrict__ kidx,
                                                            const int64_t* __restrict__ vis_off, VisGeom vg,
                                                            float2* __restrict__ out, const float2* __restrict__ y,
                                                            const float2* __restrict__ v, float2* __restrict__ u_prev,
                                                            const uint8_t* __restrict__ blk, int B,
                                                            double* __restrict__ partials, int nparts) {
  constexpr int SD = 2 * R + 1;
  __shared__ float2 scr[2 * kDdeWarps][SD * kDdeLd];
  __shared__ double sred[kDdeWarps * 2 * kMaxB];
  const int l = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t end = vis_off[l + 1];
  const int64_t wbase = vis_off[l] + (int64_t)blockIdx.x * kDdeThreads + wid * 32;
  const float2* gl = grid + (size_t)l * vg.K1 * vg.K2;
  float2 mine = make_float2(0.f, 0.f);
  const DdeTap tap = dde_tap_poly(lane);
#pragma unroll 1
  for (int t = 0; t < 16; ++t) {
    if (wbase + t >= end) break;                       // warp-uniform
    const int64_t i = min(wbase + (lane & 16) + t, end - 1);   // past the end: repeated, not kept
    const float2 u = dde_degrid_half<R>(gl, uv[i], kern + (size_t)kidx[i] * SD * SD, vg, tap,
                                        scr[2 * wid + (lane >> 4)], lane);
    if ((lane & 15) == t) mine = u;
  }
  const int64_t i = wbase + lane;
  const bool valid = i < end;
  if (MODE == 0) {
    if (valid) out[i] = mine;
    return;
  }
  float2 d = make_float2(0.f, 0.f), yy = d;
  int b = 0;
  if (valid) {
    const float2 vv = v[i], up = u_prev[i];
    yy = y[i];
    const float2 z = make_float2(vv.x + 2.f * mine.x - up.x, vv.y + 2.f * mine.y - up.y);
    d = make_float2(z.x - yy.x, z.y - yy.y);
    out[i] = d;
    u_prev[i] = mine;
    b = blk[i];
  }
  block_partials<kDdeWarps>(d, yy, mine, b, valid, B, sred, partials + ((size_t)l * nparts + blockIdx.x) * 2 * B);
}

// Local start (mod K) of a footprint that starts at absolute cell k, relative to tile
// start t0: cells (d + r) mod K < T of the footprint lie in the tile.
__device__ __forceinline__ int dde_local(int k, int t0, int K, int pw) {
  const int d = k - t0;
  return pw ? (d & (K - 1)) : ((d % K) + K) % K;
}

// Whether a footprint of F cells starting at local offset d (mod K) meets [0, T).
__device__ __forceinline__ bool dde_meets(int d, int F, int T, int K) { return d < T || d + F - 1 >= K; }

// Adds the footprint cells of each half-warp's visibility that lie in the tile: fixed-point
// values of conj(g) v S, with vS = v S (`on` false: nothing is added); tr: the half's
// [SD][kDdeLd] scratch.  MODE 1: the weights' bound (|Re K| + |Im K|) phi phi vS.x instead,
// rounded up.
template <int R, int MODE>
__device__ __forceinline__ void dde_grid_half(int* are, int* aim, int TP, int T, int dr, int dc, float xr, float xc,
                                              float2 vS, const float2* __restrict__ Km, bool on, const VisGeom& vg,
                                              const DdeTap& tap, float2* tr, int lane) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R;
  const int j = lane & 15;
  float wr[kTaps], wc[kTaps];
  const float2* Kr = Km + min(j, SD - 1) * SD;
  float2 Z[SD];
#pragma unroll
  for (int j2 = 0; j2 < SD; ++j2) {
    const float2 K = __ldg(Kr + j2);
    Z[j2] = MODE == 1 ? make_float2((fabsf(K.x) + fabsf(K.y)) * vS.x, 0.f)
                      : make_float2(fmaf(K.x, vS.x, K.y * vS.y), fmaf(K.x, vS.y, -K.y * vS.x));   // conj(K) v S
  }
  dde_weights(tap, xr, xc, lane, wr, wc);
  if (MODE == 1) {
#pragma unroll
    for (int b = 0; b < kTaps; ++b) {
      wr[b] = fabsf(wr[b]);
      wc[b] = fabsf(wc[b]);
    }
  }
  // column pass: H[j1][c] = sum_b w_c[b] Z[j1][c - b]
#pragma unroll
  for (int c = 0; c < F; ++c) {
    float2 h = make_float2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < kTaps; ++b) {
      const int j2 = c - b;
      if (j2 >= 0 && j2 < SD) {
        h.x = fmaf(wc[b], Z[j2].x, h.x);
        h.y = fmaf(wc[b], Z[j2].y, h.y);
      }
    }
    if (j < SD) tr[j * kDdeLd + c] = h;
  }
  __syncwarp();
  // row pass and the tile's cells of column c: x[r][c] = sum_a w_r[a] H[r - a][c]
  const int lc = wrap2(dc + j, vg);
  if (on && j < F && lc < T) {
    float2 H[SD];
#pragma unroll
    for (int j1 = 0; j1 < SD; ++j1) H[j1] = tr[j1 * kDdeLd + j];
#pragma unroll
    for (int r = 0; r < F; ++r) {
      float2 x = make_float2(0.f, 0.f);
#pragma unroll
      for (int a = 0; a < kTaps; ++a) {
        const int j1 = r - a;
        if (j1 >= 0 && j1 < SD) {
          x.x = fmaf(wr[a], H[j1].x, x.x);
          x.y = fmaf(wr[a], H[j1].y, x.y);
        }
      }
      const int lr = wrap1(dr + r, vg);
      if (lr < T) {
        if (MODE == 1) {
          atomicAdd(are + lr * TP + lc, __float2int_ru(x.x));
        } else {
          atomicAdd(are + lr * TP + lc, __float2int_rn(x.x));
          atomicAdd(aim + lr * TP + lc, __float2int_rn(x.y));
        }
      }
    }
  }
  __syncwarp();
}

// Source bucket s (0..8) of tile (tr, tc): the tile at offset (s / 3 - 1, s % 3 - 1),
// or -1 when it repeats an earlier one (fewer than 3 tiles along an axis).
__device__ __forceinline__ int dde_source(int s, int tr, int tc, int ntr, int ntc) {
  const int sr = (tr + s / 3 - 1 + ntr) % ntr, sc = (tc + s % 3 - 1 + ntc) % ntc;
  for (int e = 0; e < s; ++e) {
    const int er = (tr + e / 3 - 1 + ntr) % ntr, ec = (tc + e % 3 - 1 + ntc) % ntc;
    if (er == sr && ec == sc) return -1;
  }
  return sr * ntc + sc;
}

// MODE 0: grid the (block-scaled) values into tile blockIdx.x of channel blockIdx.y and
// store it (v_write, when set, receives the scaled values of the tile's own
// visibilities); MODE 1: store the tile's largest weight sum of a cell in cover[l][tile].
template <int R, int MODE>
__global__ void __launch_bounds__(kDdeThreads) k_grid_dde(const float2* __restrict__ vals,
                                                          const float* __restrict__ blk_scale,
                                                          float2* __restrict__ v_write, const float2* __restrict__ uv,
                                                          const uint8_t* __restrict__ blk,
                                                          const float2* __restrict__ kern,
                                                          const int32_t* __restrict__ kidx,
                                                          const float* __restrict__ kl1,
                                                          const int32_t* __restrict__ tile_off,
                                                          const int64_t* __restrict__ vis_off,
                                                          float2* __restrict__ grid, float* __restrict__ cover,
                                                          VisGeom vg, int T, int ntr, int ntc, int B) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R;
  extern __shared__ __align__(16) int dde_acc[];
  __shared__ float2 scr[2 * kDdeWarps][SD * kDdeLd];
  __shared__ float sred[kDdeWarps];
  __shared__ int sredi[kDdeWarps];
  const int TP = grid_row_stride(T);
  int* are = dde_acc;
  int* aim = are + T * TP;
  const int l = blockIdx.y, tau = blockIdx.x, tr = tau / ntc, tc = tau % ntc;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  {
    int4* z4 = reinterpret_cast<int4*>(dde_acc);
    const int n4 = (MODE == 1 ? T * TP : 2 * T * TP) / 4;
    for (int k = threadIdx.x; k < n4; k += kDdeThreads) z4[k] = make_int4(0, 0, 0, 0);
  }
  const int64_t vbase = vis_off[l];
  const int32_t* toff = tile_off + (size_t)l * (ntr * ntc * 4 + 1);
  const int t0r = tr * T, t0c = tc * T;
  float S = 1.f;
  // sweep 0: the largest |v| component of the visibilities meeting the tile (MODE 1: the sum
  // of their kernels' magnitudes); the tile's own visibilities also get their scaled value
  // written once
  float m = 0.f;
  for (int s = 0; s < 9; ++s) {
    const int src = dde_source(s, tr, tc, ntr, ntc);
    if (src < 0) continue;
    const bool own = src == tau;
    const int beg = toff[src * 4], end = toff[src * 4 + 4];
    for (int k = beg + (int)threadIdx.x; k < end; k += kDdeThreads) {
      const int64_t i = vbase + k;
      float2 val = make_float2(0.f, 0.f);
      if (MODE == 0) {
        val = vals[i];
        if (blk_scale) {
          const float sc = blk_scale[l * B + blk[i]];
          val.x *= sc;
          val.y *= sc;
        }
        if (own && v_write) v_write[i] = val;
      }
      const float2 w = uv[i];
      float xr, xc;
      const int kr = kb_first(w.y, vg.tc.hi_r, vg.tc.lo_r, xr);
      const int kc = kb_first(w.x, vg.tc.hi_c, vg.tc.lo_c, xc);
      if (dde_meets(dde_local(kr - R, t0r, vg.K1, vg.pw), F, T, vg.K1) &&
          dde_meets(dde_local(kc - R, t0c, vg.K2, vg.pw), F, T, vg.K2)) {
        if (MODE == 1) m += kl1[kidx[i]];
        else m = fmaxf(m, fmaxf(fabsf(val.x), fabsf(val.y)));
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float e = __shfl_xor_sync(0xffffffffu, m, o);
    m = MODE == 1 ? m + e : fmaxf(m, e);
  }
  if (lane == 0) sred[wid] = m;
  __syncthreads();
  m = 0.f;
#pragma unroll
  for (int w = 0; w < kDdeWarps; ++w) m = MODE == 1 ? m + sred[w] : fmaxf(m, sred[w]);
  if (MODE == 1) {
    S = cover_unit(m);
  } else {
    const float C = cover[l * ntr * ntc + tau];
    if (m > 1e-30f && C > 0.f) {
      const float t = 1073741824.f / (C * (m * 1.0009765625f));
      const int e = (int)((__float_as_uint(t) >> 23) & 0xffu) - 127;   // 2^e <= t
      S = pow2f(max(-120, min(e, 120)));
    }
  }
  // sweep 1: each warp takes 32 candidates at a time and processes the ones that meet
  // the tile, two by two (one per half-warp)
  const DdeTap tap = dde_tap_poly(lane);
  for (int s = 0; s < 9; ++s) {
    const int src = dde_source(s, tr, tc, ntr, ntc);
    if (src < 0) continue;
    const int beg = toff[src * 4], end = toff[src * 4 + 4];
    for (int k0 = beg + wid * 32; k0 < end; k0 += kDdeThreads) {
      const int k = k0 + lane;
      bool hit = false;
      int dr = 0, dc = 0;
      float xr = 0.f, xc = 0.f;
      if (k < end) {
        const float2 w = uv[vbase + k];
        const int kr = kb_first(w.y, vg.tc.hi_r, vg.tc.lo_r, xr);
        const int kc = kb_first(w.x, vg.tc.hi_c, vg.tc.lo_c, xc);
        dr = dde_local(kr - R, t0r, vg.K1, vg.pw);
        dc = dde_local(kc - R, t0c, vg.K2, vg.pw);
        hit = dde_meets(dr, F, T, vg.K1) && dde_meets(dc, F, T, vg.K2);
      }
      unsigned mask = __ballot_sync(0xffffffffu, hit);
      while (mask) {
        const int first = __ffs(mask) - 1;
        mask &= mask - 1;
        const int second = mask ? __ffs(mask) - 1 : -1;
        mask &= mask - 1;                                  // (0 stays 0)
        const bool on = lane < 16 || second >= 0;
        const int from = lane < 16 || second < 0 ? first : second;
        const int drs = __shfl_sync(0xffffffffu, dr, from), dcs = __shfl_sync(0xffffffffu, dc, from);
        const float xrs = __shfl_sync(0xffffffffu, xr, from), xcs = __shfl_sync(0xffffffffu, xc, from);
        const int64_t i = vbase + k0 + from;
        float2 vS = make_float2(S, 0.f);
        if (MODE == 0) {
          const float2 val = vals[i];
          const float sc = (blk_scale ? blk_scale[l * B + blk[i]] : 1.f) * S;
          vS = make_float2(val.x * sc, val.y * sc);
        }
        dde_grid_half<R, MODE>(are, aim, TP, T, drs, dcs, xrs, xcs, vS, kern + (size_t)kidx[i] * SD * SD, on,
                               vg, tap, scr[2 * wid + (lane >> 4)], lane);
      }
    }
  }
  __syncthreads();
  if (MODE == 1) {
    int mx = 0;
    for (int q = threadIdx.x; q < T * T; q += kDdeThreads) mx = max(mx, are[(q / T) * TP + q % T]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) sredi[wid] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 0; w < kDdeWarps; ++w) mx = max(mx, sredi[w]);
      cover[l * ntr * ntc + tau] = __int2float_ru(mx) / S;                 // S: a power of two
    }
    return;
  }
  const float inv = 1.f / S;                                   // power of two: exact
  float2* gl = grid + (size_t)l * vg.K1 * vg.K2;
  for (int q = threadIdx.x; q < T * T; q += kDdeThreads) {
    const int rr = q / T, cc = q % T, o = rr * TP + cc;
    const int row = phys_row2(t0r + rr, vg);
    gl[(size_t)row * vg.K2 + t0c + cc] = make_float2((float)are[o] * inv, (float)aim[o] * inv);
  }
}

// ------------------------------------------------------------- launchers
#define FHS_DDE_SWITCH(R, ...)                    \
  switch (R) {                                    \
    case 0: __VA_ARGS__(0); break;                \
    case 1: __VA_ARGS__(1); break;                \
    case 2: __VA_ARGS__(2); break;                \
    case 3: __VA_ARGS__(3); break;                \
    default: __VA_ARGS__(4); break;               \
  }

static size_t grid_dde_smem(const Cube& cb, int mode) {
  return (size_t)(mode == 1 ? 1 : 2) * cb.tile * grid_row_stride(cb.tile) * sizeof(int);
}

void launch_degrid_dde(const Cube& cb, const float2* grid, float2* out, cudaStream_t st) {
  dim3 grd(degrid_parts(cb), cb.L);
  const VisGeom vg = vis_geom(cb);
#define FHS_L(RR)                                                                                               \
  k_degrid_dde<RR, 0><<<grd, kDdeThreads, 0, st>>>(grid, cb.d_uv, cb.d_dde_kern, cb.d_dde_idx, cb.d_vis_off, vg, \
                                                   out, nullptr, nullptr, nullptr, nullptr, cb.B, nullptr, 0)
  FHS_DDE_SWITCH(cb.dde_R, FHS_L)
#undef FHS_L
  note_launches(1);
}

void launch_degrid_pdfb_dde(const Cube& cb, const float2* grid, const float2* y, const float2* v, float2* d_out,
                            float2* u_prev, double* partials, int nparts, cudaStream_t st) {
  dim3 grd(nparts, cb.L);
  const VisGeom vg = vis_geom(cb);
#define FHS_L(RR)                                                                                               \
  k_degrid_dde<RR, 1><<<grd, kDdeThreads, 0, st>>>(grid, cb.d_uv, cb.d_dde_kern, cb.d_dde_idx, cb.d_vis_off, vg, \
                                                   d_out, y, v, u_prev, cb.d_blk, cb.B, partials, nparts)
  FHS_DDE_SWITCH(cb.dde_R, FHS_L)
#undef FHS_L
  note_launches(1);
}

void launch_grid_dde(const Cube& cb, const float2* vals, const float* blk_scale, float2* v_write, float2* grid,
                     cudaStream_t st) {
  dim3 grd(cb.ntile_r * cb.ntile_c, cb.L);
  const VisGeom vg = vis_geom(cb);
  const size_t sm = grid_dde_smem(cb, 0);
  static bool attr[5] = {false, false, false, false, false};
#define FHS_L(RR)                                                                                                 \
  if (!attr[RR]) {                                                                                                \
    cudaFuncSetAttribute(k_grid_dde<RR, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);               \
    attr[RR] = true;                                                                                              \
  }                                                                                                               \
  k_grid_dde<RR, 0><<<grd, kDdeThreads, sm, st>>>(vals, blk_scale, v_write, cb.d_uv, cb.d_blk, cb.d_dde_kern,      \
                                                  cb.d_dde_idx, cb.d_dde_l1, cb.d_tile_off, cb.d_vis_off, grid,   \
                                                  cb.d_dde_cover, vg, cb.tile, cb.ntile_r, cb.ntile_c, cb.B)
  FHS_DDE_SWITCH(cb.dde_R, FHS_L)
#undef FHS_L
  note_launches(1);
}

void launch_grid_dde_count(const Cube& cb, cudaStream_t st) {
  dim3 grd(cb.ntile_r * cb.ntile_c, cb.L);
  const VisGeom vg = vis_geom(cb);
  const size_t sm = grid_dde_smem(cb, 1);
  static bool attr[5] = {false, false, false, false, false};
#define FHS_L(RR)                                                                                                 \
  if (!attr[RR]) {                                                                                                \
    cudaFuncSetAttribute(k_grid_dde<RR, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);               \
    attr[RR] = true;                                                                                              \
  }                                                                                                               \
  k_grid_dde<RR, 1><<<grd, kDdeThreads, sm, st>>>(nullptr, nullptr, nullptr, cb.d_uv, cb.d_blk, cb.d_dde_kern,     \
                                                  cb.d_dde_idx, cb.d_dde_l1, cb.d_tile_off, cb.d_vis_off, nullptr,         \
                                                  cb.d_dde_cover, vg, cb.tile, cb.ntile_r, cb.ntile_c, cb.B)
  FHS_DDE_SWITCH(cb.dde_R, FHS_L)
#undef FHS_L
  note_launches(1);
}

#undef FHS_DDE_SWITCH

}  // namespace fhs
