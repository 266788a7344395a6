// 2-D DFT of the zero-padded real image for grid sides K = 2^a (128 .. 2048) and 3 2^a (96 ..
// 3072) whose column transform takes one pass (grid rows in natural order): images of 64 to
// 512 on power-of-two sides, up to 1536 where a side is 3 2^m.
//
// Two-for-one: packed column j < n2/2 holds the image columns j + n2/2 (real part, grid
// column j) and j (imaginary part, grid column K2 - n2/2 + j), so n2/2 complex columns are
// transformed, and each pair of frequency rows (k, K1 - k) recovers both columns' spectra
// from Hermitian symmetry before its row DFTs (adjoint: the other way round).  Per channel
// and direction 4N + 8N + 8N + 32N bytes (N = n1 n2) against 4N + 3 x 32N of a row pass and
// a full column pass over the grid.
//
// A transform of length N = R1 R2 (R3) runs in two (three) register passes of R-point DFTs
// with one (two) exchanges through shared memory; R1 .. R3 are compile-time, at most 32, so
// a task keeps R loads in flight and indices are shifts and adds.  The mixed-radix kernels
// with run-time plans (radix 4, 2, 3 passes between two buffers, integer divisions per
// element, one CTA of 196 KB per SM) took 1651 us for the columns and 285 us for the rows
// of 23 channels of 1536^2; these take 70 and 122 us.  The shared-memory transforms of the
// power-of-two sides (radix-8 passes, unpacked) took 60 + 101 us forward and 101 + 79 us
// adjoint at 16 channels of 1024^2, these 32 + 41 and 43 + 25 us.  What bounds them now is
// DRAM for the columns and the rows' latency (two exchanges, 94 registers a thread).
#include <cuda_runtime.h>

#include "fft_core.cuh"
#include "fhs_internal.h"

namespace fhs {
namespace {

// Factors of a transform length (R3 = 1: two passes).
template <int N> struct MidCfg;
#define FHS_MID_CFG(N, A, B, C) \
  template <> struct MidCfg<N> { static constexpr int R1 = A, R2 = B, R3 = C; };
FHS_MID_CFG(96, 12, 8, 1)
FHS_MID_CFG(128, 16, 8, 1)
FHS_MID_CFG(192, 16, 12, 1)
FHS_MID_CFG(256, 16, 16, 1)
FHS_MID_CFG(384, 24, 16, 1)
FHS_MID_CFG(512, 32, 16, 1)
FHS_MID_CFG(768, 32, 24, 1)
FHS_MID_CFG(1024, 32, 32, 1)
FHS_MID_CFG(1536, 16, 12, 8)
FHS_MID_CFG(2048, 16, 16, 8)
FHS_MID_CFG(3072, 16, 16, 12)
#undef FHS_MID_CFG

#define FHS_MID_SWITCH(n, FN, ...)                   \
  switch (n) {                                       \
    case 96: FN<96>(__VA_ARGS__); break;             \
    case 128: FN<128>(__VA_ARGS__); break;           \
    case 192: FN<192>(__VA_ARGS__); break;           \
    case 256: FN<256>(__VA_ARGS__); break;           \
    case 384: FN<384>(__VA_ARGS__); break;           \
    case 512: FN<512>(__VA_ARGS__); break;           \
    case 768: FN<768>(__VA_ARGS__); break;           \
    case 1024: FN<1024>(__VA_ARGS__); break;         \
    case 1536: FN<1536>(__VA_ARGS__); break;         \
    case 2048: FN<2048>(__VA_ARGS__); break;         \
    case 3072: FN<3072>(__VA_ARGS__); break;         \
    default: break;                                  \
  }

bool mid_side(int K) {
  while (K % 2 == 0 && K > 128) K /= 2;
  return K == 128 || K == 96;
}

// v[k] *= w^k, w = exp(-+2 pi i b / len) (table step `step` per unit of b): the powers w^1 ..
// w^(S-1) and w^S, w^2S, ... come from the table and the others are one product of two of
// them.  (Products over the set bits of k, up to four, had a 1.1 times larger error; a load
// for every power took 1.6 to 1.8 times as long for the rows.)  Distance from 64 bits, beside
// the mixed-radix kernels that read one root per product: measuring 1.24e-7 (0.98e-7) at
// 384^2, 1.32e-7 (0.97e-7) at 1536^2; adjoint 2.8e-7 (2.5e-7) at 768^2, 2.4e-7 (2.0e-7) at 1536^2.
template <int R, bool INV>
__device__ __forceinline__ void mid_twiddle(float2* v, int b, int len, const float2* __restrict__ tw, int step) {
  constexpr int S = R >= 24 ? 8 : 4;
  float2 lo[S], hi[(R + S - 1) / S];
  int e = 0;
#pragma unroll
  for (int j = 1; j < S && j < R; ++j) {
    e = e + b >= len ? e + b - len : e + b;
    lo[j] = __ldg(&tw[(size_t)e * step]);
    if (INV) lo[j].y = -lo[j].y;
  }
  const int eS = (e + b) % len;
  e = 0;
#pragma unroll
  for (int j = 1; j < (R + S - 1) / S; ++j) {
    e = e + eS >= len ? e + eS - len : e + eS;
    hi[j] = __ldg(&tw[(size_t)e * step]);
    if (INV) hi[j].y = -hi[j].y;
  }
#pragma unroll
  for (int k = 1; k < R; ++k) {
    const int r = k % S, q = k / S;
    v[k] = cmul(v[k], r == 0 ? hi[q] : (q == 0 ? lo[r] : cmul(hi[q], lo[r])));
  }
}

// DFTs of W sequences of length N by the NT threads of the CTA: load(n, w) gives element n
// of sequence w, store(k, w, v) takes output k.  SEQ: tasks enumerated along a sequence
// (rows); otherwise across the sequences (columns).  With n = b + NB a, b = d + R3 c and
// k = ka + R1 (kc + R2 kd): pass 1 over a, pass 2 over c, pass 3 over d.  Shared memory
// mid_smem<N, W, SEQ>() bytes; rows of NB + 1 elements per (w, ka) keep the exchanges of a
// sequence free of bank conflicts.
template <int N, int W, bool SEQ>
__host__ __device__ constexpr int mid_smem() {
  constexpr int NB = N / MidCfg<N>::R1;
  return W * MidCfg<N>::R1 * (SEQ ? NB + 1 : NB) * (int)sizeof(float2);
}

template <int N, int W, bool SEQ, int NT, bool INV, class Load, class Store>
__device__ __forceinline__ void mid_fft(float2* sm, const float2* __restrict__ tw, int twstride, Load load,
                                        Store store) {
  constexpr int R1 = MidCfg<N>::R1, R2 = MidCfg<N>::R2, R3 = MidCfg<N>::R3;
  constexpr int NB = R2 * R3, LD = NB + 1;
  static_assert(R1 * NB == N, "factorisation");
  auto at = [](int w, int ka, int b) { return SEQ ? (w * R1 + ka) * LD + b : (ka * NB + b) * W + w; };
#pragma unroll 1
  for (int q = threadIdx.x; q < NB * W; q += NT) {
    const int b = SEQ ? q % NB : q / W, w = SEQ ? q / NB : q % W;
    float2 v[R1];
#pragma unroll
    for (int a = 0; a < R1; ++a) v[a] = load(b + NB * a, w);
    rdft<R1, INV>(v);
    mid_twiddle<R1, INV>(v, b, N, tw, twstride);
#pragma unroll
    for (int a = 0; a < R1; ++a) sm[at(w, a, b)] = v[a];
  }
  __syncthreads();
  if constexpr (R3 > 1) {
#pragma unroll 1
    for (int q = threadIdx.x; q < R1 * R3 * W; q += NT) {
      const int ka = SEQ ? q % R1 : q / W % R1, d = SEQ ? q / R1 % R3 : q / W / R1, w = SEQ ? q / (R1 * R3) : q % W;
      float2 u[R2];
#pragma unroll
      for (int c = 0; c < R2; ++c) u[c] = sm[at(w, ka, d + R3 * c)];
      rdft<R2, INV>(u);
      mid_twiddle<R2, INV>(u, d, NB, tw, twstride * R1);
#pragma unroll
      for (int c = 0; c < R2; ++c) sm[at(w, ka, d + R3 * c)] = u[c];
    }
    __syncthreads();
#pragma unroll 1
    for (int q = threadIdx.x; q < R1 * R2 * W; q += NT) {
      const int ka = SEQ ? q % R1 : q / W % R1, kc = SEQ ? q / R1 % R2 : q / W / R1, w = SEQ ? q / (R1 * R2) : q % W;
      float2 z[R3];
#pragma unroll
      for (int d = 0; d < R3; ++d) z[d] = sm[at(w, ka, d + R3 * kc)];
      rdft<R3, INV>(z);
#pragma unroll
      for (int d = 0; d < R3; ++d) store(ka + R1 * (kc + R2 * d), w, z[d]);
    }
  } else {
#pragma unroll 1
    for (int q = threadIdx.x; q < R1 * W; q += NT) {
      const int ka = SEQ ? q % R1 : q / W, w = SEQ ? q / R1 : q % W;
      float2 z[R2];
#pragma unroll
      for (int c = 0; c < R2; ++c) z[c] = sm[at(w, ka, c)];
      rdft<R2, INV>(z);
#pragma unroll
      for (int c = 0; c < R2; ++c) store(ka + R1 * c, w, z[c]);
    }
  }
}

constexpr int round32(int n) { return (n + 31) / 32 * 32; }
constexpr int min_c(int a, int b) { return a < b ? a : b; }

// Columns per CTA: 8 (64-byte row segments) keep several CTAs on an SM up to 1536 rows.
template <int N> struct MidCol {
  static constexpr int W = N <= 1536 ? 8 : 4;
  static constexpr int NT = min_c(256, round32(N / MidCfg<N>::R1 * W));
  static constexpr int SMEM = mid_smem<N, W, false>();
};

// Rows per CTA (pairs of frequencies): about 128 tasks.
template <int N> struct MidRow {
  static constexpr int NB = N / MidCfg<N>::R1;
  static constexpr int W = NB >= 64 ? 2 : (NB >= 24 ? 4 : (NB >= 12 ? 8 : 16));
  static constexpr int NT = min_c(384, round32(NB * W));
  static constexpr int SMEM = mid_smem<N, W, true>();
  static constexpr int SMEM_ADJ = SMEM + W * (N / 2) * (int)sizeof(float2);
};

// Z and column DFT of W packed columns of channel blockIdx.y -> P [L][K1][n2/2].
template <int N>
__global__ void __launch_bounds__(MidCol<N>::NT) k_mid_col_fwd(const float* __restrict__ x, float2* __restrict__ P,
                                                               const float* __restrict__ sr,
                                                               const float* __restrict__ sc, int n1, int n2,
                                                               const float2* __restrict__ tw, int twstride) {
  constexpr int W = MidCol<N>::W;
  extern __shared__ float2 sm[];
  const int hp = n2 / 2, h1 = n1 / 2, l = blockIdx.y, j0 = blockIdx.x * W;
  const float* xl = x + (size_t)l * n1 * n2;
  float2* pl = P + (size_t)l * N * hp;
  mid_fft<N, W, false, MidCol<N>::NT, false>(
      sm, tw, twstride,
      [&](int i, int w) {
        const int r = i < h1 ? i + h1 : (i >= N - h1 ? i - (N - h1) : -1), j = j0 + w;
        if (r < 0 || j >= hp) return make_float2(0.f, 0.f);
        const float s = sr[r];
        const float* xr = xl + (size_t)r * n2;
        return make_float2(xr[j + hp] * s * sc[j + hp], xr[j] * s * sc[j]);
      },
      [&](int k, int w, float2 v) {
        if (j0 + w < hp) pl[(size_t)k * hp + j0 + w] = v;
      });
}

// Inverse column DFT of W packed columns, crop, Z^T, real parts and eta:
// out[l][r][c] (+)= eta_l s_r s_c Re(...).
template <int N>
__global__ void __launch_bounds__(MidCol<N>::NT) k_mid_col_adj(const float2* __restrict__ P, float* __restrict__ out,
                                                               const float* __restrict__ sr,
                                                               const float* __restrict__ sc,
                                                               const float* __restrict__ eta, int accumulate, int n1,
                                                               int n2, const float2* __restrict__ tw, int twstride) {
  constexpr int W = MidCol<N>::W;
  extern __shared__ float2 sm[];
  const int hp = n2 / 2, h1 = n1 / 2, l = blockIdx.y, j0 = blockIdx.x * W;
  const float2* pl = P + (size_t)l * N * hp;
  const float el = eta ? eta[l] : 1.f;
  float* ol = out + (size_t)l * n1 * n2;
  mid_fft<N, W, false, MidCol<N>::NT, true>(
      sm, tw, twstride,
      [&](int i, int w) { return j0 + w < hp ? pl[(size_t)i * hp + j0 + w] : make_float2(0.f, 0.f); },
      [&](int k, int w, float2 v) {
        const int r = k < h1 ? k + h1 : (k >= N - h1 ? k - (N - h1) : -1), j = j0 + w;
        if (r < 0 || j >= hp) return;
        const float s = sr[r];
        float* o = ol + (size_t)r * n2 + j;
        const float va = el * sc[j + hp] * s * v.x, vb = el * sc[j] * s * v.y;
        o[hp] = accumulate ? o[hp] + va : va;
        o[0] = accumulate ? o[0] + vb : vb;
      });
}

// Row DFTs of the frequency pairs (k, K1 - k), k = blockIdx.x W/2 .., from the packed
// columns: sequence 2 m is row k of pair m, sequence 2 m + 1 row K1 - k.
template <int N>
__global__ void __launch_bounds__(MidRow<N>::NT) k_mid_row_fwd(float2* __restrict__ grid, const float2* __restrict__ P,
                                                               int K1, const float2* __restrict__ tw, int twstride) {
  constexpr int W = MidRow<N>::W, HP = N / 4;
  extern __shared__ float2 sm[];
  const int l = blockIdx.y, k0 = blockIdx.x * (W / 2);
  const float2* pl = P + (size_t)l * K1 * HP;
  float2* gl = grid + (size_t)l * K1 * N;
  auto row = [&](int w) {                              // frequency row of sequence w, or -1
    const int k = k0 + (w >> 1);
    if (k > K1 / 2) return -1;
    if (!(w & 1)) return k;
    return k == 0 || 2 * k == K1 ? -1 : K1 - k;
  };
  mid_fft<N, W, true, MidRow<N>::NT, false>(
      sm, tw, twstride,
      [&](int n, int w) {
        const int k = row(w);
        if (k < 0 || (n >= HP && n < N - HP)) return make_float2(0.f, 0.f);
        const int km = k == 0 ? 0 : K1 - k, j = n < HP ? n : n - (N - HP);
        const float2 A = pl[(size_t)k * HP + j], B = pl[(size_t)km * HP + j];
        return n < HP ? make_float2(0.5f * (A.x + B.x), 0.5f * (A.y - B.y))
                      : make_float2(0.5f * (A.y + B.y), -0.5f * (A.x - B.x));
      },
      [&](int k, int w, float2 v) {
        const int r = row(w);
        if (r >= 0) gl[(size_t)r * N + k] = v;
      });
}

// Inverse row DFTs of the frequency pairs, packed for the inverse column transform: with A
// the outputs of rows k and -k, c_j[k] = H_j + i H_{N-HP+j}, H_n = (A_n[k] + conj(A_n[-k])) / 2.
template <int N>
__global__ void __launch_bounds__(MidRow<N>::NT) k_mid_row_adj(const float2* __restrict__ grid, float2* __restrict__ P,
                                                               int K1, const float2* __restrict__ tw, int twstride) {
  constexpr int W = MidRow<N>::W, HP = N / 4;
  extern __shared__ float2 sm[];
  float2* keep = sm + MidRow<N>::SMEM / sizeof(float2);            // [W][2 HP]: columns j, then N - HP + j
  const int l = blockIdx.y, k0 = blockIdx.x * (W / 2);
  const float2* gl = grid + (size_t)l * K1 * N;
  float2* pl = P + (size_t)l * K1 * HP;
  mid_fft<N, W, true, MidRow<N>::NT, true>(
      sm, tw, twstride,
      [&](int n, int w) {
        const int k = k0 + (w >> 1);
        if (k > K1 / 2) return make_float2(0.f, 0.f);
        const int r = (w & 1) && k ? K1 - k : k;
        return gl[(size_t)r * N + n];
      },
      [&](int n, int w, float2 v) {
        if (n < HP) keep[w * 2 * HP + n] = v;
        else if (n >= N - HP) keep[w * 2 * HP + n - (N - 2 * HP)] = v;
      });
  __syncthreads();
  for (int idx = threadIdx.x; idx < (W / 2) * HP; idx += MidRow<N>::NT) {
    const int m = idx / HP, j = idx - m * HP, k = k0 + m;
    if (k > K1 / 2) break;
    const float2* q = keep + 4 * m * HP + j;
    const float2 ak = q[0], bk = q[HP], am = q[2 * HP], bm = q[3 * HP];
    const float2 ha = make_float2(0.5f * (ak.x + am.x), 0.5f * (ak.y - am.y));
    const float2 hb = make_float2(0.5f * (bk.x + bm.x), 0.5f * (bk.y - bm.y));
    pl[(size_t)k * HP + j] = make_float2(ha.x - hb.y, ha.y + hb.x);                       // ha + i hb
    if (k != 0 && 2 * k != K1) pl[(size_t)(K1 - k) * HP + j] = make_float2(ha.x + hb.y, hb.x - ha.y);
  }
}

template <int N>
void mid_col_fwd(const Cube& cb, const float* x, float2* P, const float2* tw, int Kmax, cudaStream_t st) {
  using C = MidCol<N>;
  static bool attr = false;
  if (!attr) { cudaFuncSetAttribute(k_mid_col_fwd<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM); attr = true; }
  k_mid_col_fwd<N><<<dim3((cb.n2 / 2 + C::W - 1) / C::W, cb.L), C::NT, C::SMEM, st>>>(
      x, P, cb.d_scale_r, cb.d_scale_c, cb.n1, cb.n2, tw, Kmax / N);
}

template <int N>
void mid_col_adj(const Cube& cb, const float2* P, float* out, const float* eta, bool acc, const float2* tw, int Kmax,
                 cudaStream_t st) {
  using C = MidCol<N>;
  static bool attr = false;
  if (!attr) { cudaFuncSetAttribute(k_mid_col_adj<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM); attr = true; }
  k_mid_col_adj<N><<<dim3((cb.n2 / 2 + C::W - 1) / C::W, cb.L), C::NT, C::SMEM, st>>>(
      P, out, cb.d_scale_r, cb.d_scale_c, eta, acc ? 1 : 0, cb.n1, cb.n2, tw, Kmax / N);
}

template <int N>
void mid_row_fwd(const Cube& cb, float2* grid, const float2* P, const float2* tw, int Kmax, cudaStream_t st) {
  using C = MidRow<N>;
  static bool attr = false;
  if (!attr) { cudaFuncSetAttribute(k_mid_row_fwd<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM); attr = true; }
  k_mid_row_fwd<N><<<dim3((cb.K1 / 2 + C::W / 2) / (C::W / 2), cb.L), C::NT, C::SMEM, st>>>(grid, P, cb.K1, tw,
                                                                                          Kmax / N);
}

template <int N>
void mid_row_adj(const Cube& cb, const float2* grid, float2* P, const float2* tw, int Kmax, cudaStream_t st) {
  using C = MidRow<N>;
  static bool attr = false;
  if (!attr) { cudaFuncSetAttribute(k_mid_row_adj<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_ADJ); attr = true; }
  k_mid_row_adj<N><<<dim3((cb.K1 / 2 + C::W / 2) / (C::W / 2), cb.L), C::NT, C::SMEM_ADJ, st>>>(grid, P, cb.K1, tw,
                                                                                              Kmax / N);
}

}  // namespace

// One-pass columns (natural row order) and both sides among the instantiated lengths.  Grids
// with a side of 32 or 64 cells (images of 16 and 32) keep the transforms they had: 2 to 13 us
// of a call, and the pairing of Phi with its adjoint over DDE kernels on 64 cells lies at the
// resolution of the fixed-point gridder, so its results there are left as they are.
bool fft_mid_supported(const Cube& cb) {
  return cb.N2c == 1 && cb.K1 >= 96 && cb.K2 >= 96 && mid_side(cb.K1) && mid_side(cb.K2) && cb.K1 <= 3072 && cb.K2 <= 3072;
}

void launch_fft_forward_mid(fhs_ctx* ctx, const Cube& cb, const float* x, float2* grid, cudaStream_t st) {
  FHS_MID_SWITCH(cb.K1, mid_col_fwd, cb, x, ctx->s.pack, ctx->d_tw, ctx->Kmax, st)
  FHS_MID_SWITCH(cb.K2, mid_row_fwd, cb, grid, ctx->s.pack, ctx->d_tw, ctx->Kmax, st)
  note_launches(2);
}

void launch_fft_adjoint_mid(fhs_ctx* ctx, const Cube& cb, const float2* grid, float* out, const float* eta,
                            bool accumulate, cudaStream_t st) {
  FHS_MID_SWITCH(cb.K2, mid_row_adj, cb, grid, ctx->s.pack, ctx->d_tw, ctx->Kmax, st)
  FHS_MID_SWITCH(cb.K1, mid_col_adj, cb, ctx->s.pack, out, eta, accumulate, ctx->d_tw, ctx->Kmax, st)
  note_launches(2);
}

}  // namespace fhs
