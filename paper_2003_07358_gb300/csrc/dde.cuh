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
// operand), with transpositions through shared memory in between; a warp works on two
// visibilities at a time.  De-gridding: lane c loads column c of the window (coalesced along
// the row), lane r runs the column pass of row r, lane j2 the row pass of column j2.
// Gridding: lane j2 takes column j2 of the kernel, then lane r row r of the footprint; the
// tile's row pitch is odd, so the rows' atomics fall on different banks.  Lanes 0..13 of a
// half hold the polynomial of one Kaiser-Bessel tap each and exchange the 14 weights by
// shuffles.  (One visibility per warp with every pass reading its operands from shared memory
// took 2.04 ms to de-grid and 4.03 to 4.13 ms to grid 2.1 M visibilities of 16 channels of
// 1024^2 with 9 x 9 kernels, about 700 instructions a visibility; this form takes 1.00 and
// 1.57 ms, bound by issue: 126 FMAs a pass and lane, and for the gridder 30 conversions and
// atomics.)
//
// Gridding keeps the scheme of k_grid: one CTA per (grid tile, channel) owns the tile's
// cells in shared memory and adds, in 32-bit fixed point with integer atomics (order-
// independent, so bitwise deterministic), every footprint cell that falls in the tile.
// Visibilities are bucketed by the tile of their first tap, and a footprint (F <= 15 <
// tile side) reaches only the 3 x 3 neighbouring tiles, so a CTA scans those buckets,
// keeps (by warp ballot) the visibilities whose footprint meets its tile, and processes
// them two by two.  The scale S = 2^e of a tile satisfies n_c m S < 2^30 with n_c the largest
// number of extended footprints covering one of its cells (counted once per kernel set,
// MODE 1) and m = max over the contributing visibilities of
// max(|Re v|, |Im v|) * sum_j (|Re K_j| + |Im K_j|), a bound of every tap value
// |Re|, |Im| of conj(g_m[k]) v_m (Kaiser-Bessel weights are at most 1).

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
// the half's scratch ([F][kDdeLd]: the window, the intermediate and the values that meet the
// kernel take turns in it).  The sums run in the order of the definition above (columns, rows, then
// the kernel coefficients 32 apart and a tree over their residues), whichever lane runs them.
template <int R>
__device__ __forceinline__ float2 dde_degrid_half(const float2* __restrict__ gl, float2 uvm,
                                                  const float2* __restrict__ Km, const VisGeom& vg, const DdeTap& tap,
                                                  float2* tr, int lane) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R, SD2 = SD * SD, NK = (SD2 + 31) / 32;
  const int j = lane & 15;
  float xr, xc, wr[kTaps], wc[kTaps];
  const int kr = kb_first(uvm.y, vg.tc.hi_r, vg.tc.lo_r, xr);
  const int kc = kb_first(uvm.x, vg.tc.hi_c, vg.tc.lo_c, xc);
  // the lane's column of the window and its kernel coefficients (k = 32 i + j and + 16), all
  // loads in flight
  const float2* col = gl + wrap2(kc - R + min(j, F - 1), vg);
  float2 x[F], K[2][NK];
#pragma unroll
  for (int r = 0; r < F; ++r) x[r] = __ldg(col + (size_t)phys_row2(wrap1(kr - R + r, vg), vg) * vg.K2);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int i = 0; i < NK; ++i) K[h][i] = __ldg(Km + min(32 * i + 16 * h + j, SD2 - 1));
  dde_weights(tap, xr, xc, lane, wr, wc);
#pragma unroll
  for (int r = 0; r < F; ++r)
    if (j < F) tr[r * kDdeLd + j] = x[r];
  __syncwarp();
  // column pass, lane = row: mid[r][j2] = sum_b w_c[b] x[r][j2 + b]
#pragma unroll
  for (int c = 0; c < F; ++c) x[c] = tr[min(j, F - 1) * kDdeLd + c];
  __syncwarp();
#pragma unroll
  for (int j2 = 0; j2 < SD; ++j2) {
    float2 m = make_float2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < kTaps; ++b) {
      m.x = fmaf(wc[b], x[j2 + b].x, m.x);
      m.y = fmaf(wc[b], x[j2 + b].y, m.y);
    }
    if (j < F) tr[j2 * kDdeLd + j] = m;
  }
  __syncwarp();
  // row pass, lane = j2: I[j1][j2] = sum_a w_r[a] mid[j1 + a][j2]
#pragma unroll
  for (int r = 0; r < F; ++r) x[r] = tr[min(j, SD - 1) * kDdeLd + r];
  __syncwarp();
#pragma unroll
  for (int j1 = 0; j1 < SD; ++j1) {
    float2 I = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < kTaps; ++a) {
      I.x = fmaf(wr[a], x[j1 + a].x, I.x);
      I.y = fmaf(wr[a], x[j1 + a].y, I.y);
    }
    if (j < SD) tr[j1 * SD + j] = I;
  }
  __syncwarp();
  // u = sum_k K[k] I[k]
  float2 u[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    u[h] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int k = 32 * i + 16 * h + j;
      if (k < SD2) {
        const float2 I = tr[k];
        u[h].x = fmaf(K[h][i].x, I.x, fmaf(-K[h][i].y, I.y, u[h].x));
        u[h].y = fmaf(K[h][i].x, I.y, fmaf(K[h][i].y, I.x, u[h].y));
      }
    }
  }
  float2 s = make_float2(u[0].x + u[1].x, u[0].y + u[1].y);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  __syncwarp();                         // the scratch is reused by the next visibility
  return s;
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
  __shared__ float2 scr[2 * kDdeWarps][(kTaps + 2 * R) * kDdeLd];
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

// Row pitch (ints) of the tile accumulators: odd, so that consecutive rows of a column lie
// on consecutive banks.
__host__ __device__ inline int dde_row_stride(int T) { return T + 1; }

// Counts one per footprint cell of a visibility that lies in the tile, by the whole warp.
template <int R>
__device__ __forceinline__ void dde_count_one(int* are, int TP, int T, int dr, int dc, const VisGeom& vg, int lane) {
  constexpr int F = kTaps + 2 * R;
  for (int k = lane; k < F * F; k += 32) {
    const int r = k / F, c = k - r * F;
    const int lr = wrap1(dr + r, vg), lc = wrap2(dc + c, vg);
    if (lr < T && lc < T) atomicAdd(are + lr * TP + lc, 1);
  }
}

// Adds the footprint cells of each half-warp's visibility that lie in the tile: fixed-point
// values of conj(g) v S, with vS = v S (`on` false: nothing is added); tr: the half's
// [SD][kDdeLd] scratch.
template <int R>
__device__ __forceinline__ void dde_grid_half(int* are, int* aim, int TP, int T, int dr, int dc, float xr, float xc,
                                              float2 vS, const float2* __restrict__ Km, bool on, const VisGeom& vg,
                                              const DdeTap& tap, float2* tr, int lane) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R;
  const int j = lane & 15;
  float wr[kTaps], wc[kTaps];
  const float2* Kc = Km + min(j, SD - 1);
  float2 Z[SD];
#pragma unroll
  for (int j1 = 0; j1 < SD; ++j1) {
    const float2 K = __ldg(Kc + j1 * SD);
    Z[j1] = make_float2(fmaf(K.x, vS.x, K.y * vS.y), fmaf(K.x, vS.y, -K.y * vS.x));   // conj(K) v S
  }
  dde_weights(tap, xr, xc, lane, wr, wc);
  // row pass: H[r][j2] = sum_a w_r[a] Z[r - a][j2]
#pragma unroll
  for (int r = 0; r < F; ++r) {
    float2 h = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < kTaps; ++a) {
      const int j1 = r - a;
      if (j1 >= 0 && j1 < SD) {
        h.x = fmaf(wr[a], Z[j1].x, h.x);
        h.y = fmaf(wr[a], Z[j1].y, h.y);
      }
    }
    if (j < SD) tr[j * kDdeLd + r] = h;
  }
  __syncwarp();
  // column pass and the tile's cells of row r: x[r][c] = sum_b w_c[b] H[r][c - b]
  const int lr = wrap1(dr + j, vg);
  if (on && j < F && lr < T) {
    float2 H[SD];
#pragma unroll
    for (int j2 = 0; j2 < SD; ++j2) H[j2] = tr[j2 * kDdeLd + j];
#pragma unroll
    for (int c = 0; c < F; ++c) {
      float2 x = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < kTaps; ++b) {
        const int j2 = c - b;
        if (j2 >= 0 && j2 < SD) {
          x.x = fmaf(wc[b], H[j2].x, x.x);
          x.y = fmaf(wc[b], H[j2].y, x.y);
        }
      }
      const int lc = wrap2(dc + c, vg);
      if (lc < T) {
        atomicAdd(are + lr * TP + lc, __float2int_rn(x.x));
        atomicAdd(aim + lr * TP + lc, __float2int_rn(x.y));
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
// visibilities); MODE 1: store the tile's largest footprint count of a cell in ncmax[l][tile].
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
                                                          float2* __restrict__ grid, int* __restrict__ ncmax,
                                                          VisGeom vg, int T, int ntr, int ntc, int B) {
  constexpr int SD = 2 * R + 1, F = kTaps + 2 * R;
  extern __shared__ __align__(16) int dde_acc[];
  __shared__ float2 scr[MODE == 0 ? 2 * kDdeWarps : 1][SD * kDdeLd];
  __shared__ float sred[kDdeWarps];
  __shared__ int sredi[kDdeWarps];
  const int TP = dde_row_stride(T);
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
  if (MODE == 0) {
    // sweep 0: bound m of the tap values of the visibilities meeting the tile; the
    // tile's own visibilities also get their scaled value written once
    float m = 0.f;
    for (int s = 0; s < 9; ++s) {
      const int src = dde_source(s, tr, tc, ntr, ntc);
      if (src < 0) continue;
      const bool own = src == tau;
      const int beg = toff[src * 4], end = toff[src * 4 + 4];
      for (int k = beg + (int)threadIdx.x; k < end; k += kDdeThreads) {
        const int64_t i = vbase + k;
        float2 val = vals[i];
        if (blk_scale) {
          const float sc = blk_scale[l * B + blk[i]];
          val.x *= sc;
          val.y *= sc;
        }
        if (own && v_write) v_write[i] = val;
        const float2 w = uv[i];
        float xr, xc;
        const int kr = kb_first(w.y, vg.tc.hi_r, vg.tc.lo_r, xr);
        const int kc = kb_first(w.x, vg.tc.hi_c, vg.tc.lo_c, xc);
        if (dde_meets(dde_local(kr - R, t0r, vg.K1, vg.pw), F, T, vg.K1) &&
            dde_meets(dde_local(kc - R, t0c, vg.K2, vg.pw), F, T, vg.K2))
          m = fmaxf(m, fmaxf(fabsf(val.x), fabsf(val.y)) * kl1[kidx[i]]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) sred[wid] = m;
    __syncthreads();
    m = 0.f;
#pragma unroll
    for (int w = 0; w < kDdeWarps; ++w) m = fmaxf(m, sred[w]);
    const int nc = ncmax[l * ntr * ntc + tau];
    if (m > 1e-30f && nc > 0) {
      const float t = 1073741824.f / ((float)nc * (m * 1.0009765625f));
      const int e = (int)((__float_as_uint(t) >> 23) & 0xffu) - 127;   // 2^e <= t
      S = pow2f(max(-120, min(e, 120)));
    }
  } else {
    __syncthreads();
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
        if (MODE == 1) {
          dde_count_one<R>(are, TP, T, __shfl_sync(0xffffffffu, dr, first), __shfl_sync(0xffffffffu, dc, first), vg,
                           lane);
          continue;
        }
        const int second = mask ? __ffs(mask) - 1 : -1;
        mask &= mask - 1;                                  // (0 stays 0)
        const bool on = lane < 16 || second >= 0;
        const int from = lane < 16 || second < 0 ? first : second;
        const int drs = __shfl_sync(0xffffffffu, dr, from), dcs = __shfl_sync(0xffffffffu, dc, from);
        const float xrs = __shfl_sync(0xffffffffu, xr, from), xcs = __shfl_sync(0xffffffffu, xc, from);
        const int64_t i = vbase + k0 + from;
        const float2 val = vals[i];
        const float sc = (blk_scale ? blk_scale[l * B + blk[i]] : 1.f) * S;
        const float2 vS = make_float2(val.x * sc, val.y * sc);
        dde_grid_half<R>(are, aim, TP, T, drs, dcs, xrs, xcs, vS, kern + (size_t)kidx[i] * SD * SD, on, vg,
                         tap, scr[2 * wid + (lane >> 4)], lane);
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
      ncmax[l * ntr * ntc + tau] = mx;
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
  return (size_t)(mode == 1 ? 1 : 2) * cb.tile * dde_row_stride(cb.tile) * sizeof(int);
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
                                                  cb.d_dde_ncmax, vg, cb.tile, cb.ntile_r, cb.ntile_c, cb.B)
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
  k_grid_dde<RR, 1><<<grd, kDdeThreads, sm, st>>>(nullptr, nullptr, nullptr, cb.d_uv, cb.d_blk, nullptr,           \
                                                  nullptr, nullptr, cb.d_tile_off, cb.d_vis_off, nullptr,         \
                                                  cb.d_dde_ncmax, vg, cb.tile, cb.ntile_r, cb.ntile_c, cb.B)
  FHS_DDE_SWITCH(cb.dde_R, FHS_L)
#undef FHS_L
  note_launches(1);
}

#undef FHS_DDE_SWITCH

}  // namespace fhs
