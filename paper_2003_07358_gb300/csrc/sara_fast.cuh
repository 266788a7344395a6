// Fast SARA l2,1 dual (Algorithm 2 W update, Table 2 row 3) on GB300, included
// at the end of sara.cu (it uses that file's c_filt filter table).
//
//   k_ana1_all  : level 1 of all eight bases for a 32x32 coefficient tile of one
//                 channel from one staged db8 input window.
//   k_ana2_all  : one level (2..4) of every basis in one launch (k_ana2_one: one
//                 basis, for levels whose every basis fills the GPU alone), a 32x32
//                 coefficient tile of one channel per CTA: the input tile with
//                 its filter halo is staged in shared memory, filtered along x
//                 then y with register blocking (each thread produces 4 outputs
//                 from one window of F + 6 loaded values); writes the LL band for
//                 the next level and the detail bands (/3) to the coefficient buffer.
//   k_prox2     : the l2,1 dual over every coefficient of the sub-cube in one
//                 streaming pass (Dirac block read straight from x):
//                 W <- z min(1, alpha_i / ||z_i||), z = W + Psi^dagger x
//                 (weights mode: theta_i = mu / (||Psi^dagger x||_i + mu)).
//   k_syn2_all  : one synthesis level (4 -> 3, 3 -> 2, 2 -> 1) of every basis in
//                 one launch (k_syn2_one: one basis, as above), a 64x64 or 32x32
//                 output tile of one channel per CTA,
//                 polyphase (even outputs take the odd taps and vice versa),
//                 register-blocked.
//   k_synfin    : level 1 of all eight bases and the Dirac block for a 64x64 or 32x32
//                 output tile, accumulated in registers; A += kappa * result.
// Same conventions as the plain kernels (zero-padded full convolution, odd
// phase, coefficients scaled by 1/3).

namespace fhs {

constexpr int kT2 = 32;                              // tile side (coefficients or outputs)
constexpr int kIn2 = 2 * kT2 + kMaxFilt - 2;         // 78: input rows/cols of an analysis tile

// Filter taps of basis F/2 - 1, read straight from the constant bank: with the tap
// index known at compile time (unrolled loops) every FMA takes the tap as a
// constant-bank operand, no register and no load.
template <int F>
struct FTaps {
  struct H { __device__ __forceinline__ float operator[](int t) const { return c_filt.h[F / 2 - 1][t]; } };
  struct G { __device__ __forceinline__ float operator[](int t) const { return c_filt.g[F / 2 - 1][t]; } };
  H h;
  G g;
  __device__ __forceinline__ void load() {}
};

// ------------------------------------------------------------- async copies
__device__ __forceinline__ void cp_async4(float* smem, const float* gmem, bool valid) {
  unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  int n = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(n));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// ------------------------------------------------------------- analysis
// x then y pass of one (basis, level) for the coefficient tile (k0, c0) of one channel.
// Staged input element (r, c) of this filter's window is tin[r + o][c + o] (o > 0 when
// the window sits inside a wider one staged for a longer filter).  Writes the three
// detail bands (/3) to cl + off_d and the LL band to llo (next level's input) or, when
// llo is null, to cl + off_ll (/3).  Starts with a barrier so that tlx / thx may be
// reused from a previous call.
template <int F>
__device__ __forceinline__ void ana_tile(const float (*tin)[kIn2 + 1], int o, float (*tlx)[kT2 + 1],
                                         float (*thx)[kT2 + 1], float* __restrict__ cl, float* __restrict__ llo,
                                         int64_t off0, int64_t off1, int64_t off2, int64_t off_ll, int k0, int c0,
                                         int mo1, int mo2) {
  constexpr int IN = 2 * kT2 + F - 2;
  constexpr int WIN = F + 6;                          // window of a 4-output block
  FTaps<F> f;
  __syncthreads();
  // x: lx[r][kc] = sum_t h[t] tin[r][2 kc + F - 1 - t], 4 consecutive kc per item
  for (int item = threadIdx.x; item < IN * 8; item += 256) {
    const int r = item >> 3, kc0 = (item & 7) * 4;
    float v[WIN];
#pragma unroll
    for (int u = 0; u < WIN; ++u) v[u] = tin[r + o][2 * kc0 + u + o];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float sl = 0.f, sh = 0.f;
#pragma unroll
      for (int t = 0; t < F; ++t) {
        sl = fmaf(f.h[t], v[2 * m + F - 1 - t], sl);
        sh = fmaf(f.g[t], v[2 * m + F - 1 - t], sh);
      }
      tlx[r][kc0 + m] = sl;
      thx[r][kc0 + m] = sh;
    }
  }
  __syncthreads();
  // y: 4 consecutive coefficient rows per thread, all four bands
  const int kc = threadIdx.x & 31, kr0 = (threadIdx.x >> 5) * 4;
  float a[WIN], b[WIN];
#pragma unroll
  for (int u = 0; u < WIN; ++u) {
    a[u] = tlx[2 * kr0 + u][kc];
    b[u] = thx[2 * kr0 + u][kc];
  }
  const float third = 1.f / 3.f;
  const int gc = c0 + kc;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    float ll = 0.f, d0 = 0.f, d1 = 0.f, d2 = 0.f;
#pragma unroll
    for (int t = 0; t < F; ++t) {
      const float va = a[2 * m + F - 1 - t], vb = b[2 * m + F - 1 - t];
      ll = fmaf(f.h[t], va, ll);
      d1 = fmaf(f.g[t], va, d1);
      d0 = fmaf(f.h[t], vb, d0);
      d2 = fmaf(f.g[t], vb, d2);
    }
    const int gk = k0 + kr0 + m;
    if (gk < mo1 && gc < mo2) {
      const int64_t pos = (int64_t)gk * mo2 + gc;
      cl[off0 + pos] = d0 * third;
      cl[off1 + pos] = d1 * third;
      cl[off2 + pos] = d2 * third;
      if (llo) llo[pos] = ll;
      else cl[off_ll + pos] = ll * third;
    }
  }
}

// Stage rows [r0, r0 + IN) x columns [c0, c0 + IN) of one channel image (zero outside)
// with asynchronous copies, so that all of a thread's loads are in flight at once:
// lane = column, warp = row.
template <int IN>
__device__ __forceinline__ void ana_stage(float (*tin)[kIn2 + 1], const float* __restrict__ inl, int r0, int c0,
                                          int m1, int m2) {
  const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5;
#pragma unroll
  for (int cj = 0; cj < (IN + 31) / 32; ++cj) {
    const int c = lane + 32 * cj, gc = c0 + c;
    if (c >= IN) continue;
    const bool vc = gc >= 0 && gc < m2;
#pragma unroll 4
    for (int r = wrp; r < IN; r += 8) {
      const int gr = r0 + r;
      const bool v = vc && gr >= 0 && gr < m1;
      cp_async4(&tin[r][c], v ? inl + (size_t)gr * m2 + gc : inl, v);
    }
  }
  cp_async_commit();
  cp_async_wait<0>();
}

// One level (2, 3 or 4) of every basis in one launch: blockIdx.x runs over the
// coefficient tiles of all bases (longest filters first), blockIdx.y over channels.
// The bases of a level are independent (each reads its own coarser LL band), so one
// launch per level replaces eight and the small levels fill the GPU together.
struct Ana2Basis {
  const float* in;     // LL band of the previous level [L][m1][m2]
  float* ll_out;       // LL band of this level [L][mo1][mo2], or null: LL4 into coef (/3)
  int64_t off[3];      // detail bands in the coefficient buffer
  int64_t off_ll;      // LL4 (last level only)
  int m1, m2, mo1, mo2;
  int tiles_x;         // coefficient tiles along a row of this basis
  int tile0;           // first linear tile of this basis
  int F;               // filter length
};
struct Ana2All {
  Ana2Basis b[8];
  int nb;
};

template <int F>
__device__ __forceinline__ void ana2_body(const Ana2Basis& B, int tile, int l, float* __restrict__ coef, int64_t I,
                                          float (*tin)[kIn2 + 1], float (*tlx)[kT2 + 1], float (*thx)[kT2 + 1]) {
  const int ty = tile / B.tiles_x, tx = tile - ty * B.tiles_x;
  const int k0 = ty * kT2, c0 = tx * kT2;
  ana_stage<2 * kT2 + F - 2>(tin, B.in + (size_t)l * B.m1 * B.m2, 2 * k0 + 2 - F, 2 * c0 + 2 - F, B.m1, B.m2);
  ana_tile<F>(tin, 0, tlx, thx, coef + (size_t)l * I, B.ll_out ? B.ll_out + (size_t)l * B.mo1 * B.mo2 : nullptr,
              B.off[0], B.off[1], B.off[2], B.off_ll, k0, c0, B.mo1, B.mo2);
}

__global__ void __launch_bounds__(256, 4) k_ana2_all(const Ana2All a, float* __restrict__ coef, int64_t I) {
  __shared__ float tin[kIn2][kIn2 + 1];
  __shared__ float tlx[kIn2][kT2 + 1];
  __shared__ float thx[kIn2][kT2 + 1];
  const int t = blockIdx.x, l = blockIdx.y;
  int bi = 0;
#pragma unroll 1
  for (int k = 1; k < a.nb; ++k)
    if (t >= a.b[k].tile0) bi = k;
  const Ana2Basis& B = a.b[bi];
  const int tile = t - B.tile0;
  switch (B.F) {
    case 2: ana2_body<2>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 4: ana2_body<4>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 6: ana2_body<6>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 8: ana2_body<8>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 10: ana2_body<10>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 12: ana2_body<12>(B, tile, l, coef, I, tin, tlx, thx); break;
    case 14: ana2_body<14>(B, tile, l, coef, I, tin, tlx, thx); break;
    default: ana2_body<16>(B, tile, l, coef, I, tin, tlx, thx); break;
  }
}

// One basis of a level on its own (tiles along blockIdx.x, channels along blockIdx.y):
// used when every basis's tiles fill the GPU by themselves, where the per-filter
// register allocation keeps more CTAs per SM than the merged kernel.
template <int F>
__global__ void __launch_bounds__(256) k_ana2_one(const Ana2Basis B, float* __restrict__ coef, int64_t I) {
  __shared__ float tin[kIn2][kIn2 + 1];
  __shared__ float tlx[kIn2][kT2 + 1];
  __shared__ float thx[kIn2][kT2 + 1];
  ana2_body<F>(B, blockIdx.x, blockIdx.y, coef, I, tin, tlx, thx);
}

// Level 1 of all eight bases for a 32x32 coefficient tile of one channel: the input
// window of the longest filter (db8, 78 x 78) is staged once and each basis reads its
// own window inside it (offset 16 - F), instead of one launch and one staging per
// basis.  The LL1 band of basis b goes to its slot in the LL1 buffer (the input of
// its level 2).
struct Ana1 {
  int64_t off[8][3];   // level-1 detail-band offsets of each basis
  int mo1[8], mo2[8];  // level-1 coefficient rows / columns of each basis
  int64_t ll_off[8];   // LL1 slot of each basis in the LL1 buffer (units of floats)
};

template <int F>
__device__ __forceinline__ void ana1_basis(const Ana1& a, const float (*tin)[kIn2 + 1], float (*tlx)[kT2 + 1],
                                           float (*thx)[kT2 + 1], float* cl, float* ll1, int l, int k0, int c0) {
  constexpr int b = F / 2 - 1;
  ana_tile<F>(tin, kMaxFilt - F, tlx, thx, cl, ll1 + a.ll_off[b] + (size_t)l * a.mo1[b] * a.mo2[b], a.off[b][0],
              a.off[b][1], a.off[b][2], 0, k0, c0, a.mo1[b], a.mo2[b]);
}

__global__ void __launch_bounds__(256) k_ana1_all(const float* __restrict__ x, float* __restrict__ coef,
                                                  float* __restrict__ ll1, Ana1 a, int64_t I, int n1, int n2) {
  __shared__ float tin[kIn2][kIn2 + 1];
  __shared__ float tlx[kIn2][kT2 + 1];
  __shared__ float thx[kIn2][kT2 + 1];
  const int l = blockIdx.z;
  const int k0 = blockIdx.y * kT2, c0 = blockIdx.x * kT2;
  ana_stage<kIn2>(tin, x + (size_t)l * n1 * n2, 2 * k0 + 2 - kMaxFilt, 2 * c0 + 2 - kMaxFilt, n1, n2);
  float* cl = coef + (size_t)l * I;
  ana1_basis<2>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<4>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<6>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<8>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<10>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<12>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<14>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
  ana1_basis<16>(a, tin, tlx, thx, cl, ll1, l, k0, c0);
}

// ---------------------------------------------------------- l2,1 dual
// K coefficients per thread; z of every channel is parked in shared memory (K x L x 256
// floats) instead of registers.  The channel loop runs in batches of 16/K with their loads in
// flight together, then in halves, quarters, ... of one for what is left of L: with a rolled
// remainder loop the kernel waited for each channel in turn (L = 12 128 us at 512^2, L = 4
// 3.07 ms at 4096^2; now 64 us and 1.47 ms).  K = 2 and 4 keep 16 loads in flight where L is
// below 16.
template <int CH, int K>
__device__ __forceinline__ void prox_load(float* zs, float (&n2)[K], const float* __restrict__ W,
                                          const float* __restrict__ coef, const float* __restrict__ x,
                                          const int64_t (&i)[K], int64_t I, int64_t dirac_off, int64_t N, int l0,
                                          int L, int weights) {
  float c[CH][K], w[CH][K];
#pragma unroll
  for (int u = 0; u < CH; ++u)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      c[u][k] = w[u][k] = 0.f;
      if (i[k] < 0) continue;
      const int l = l0 + u;
      c[u][k] = i[k] >= dirac_off ? x[(size_t)l * N + (i[k] - dirac_off)] * (1.f / 3.f) : coef[(size_t)l * I + i[k]];
      if (!weights) w[u][k] = W[(size_t)l * I + i[k]];
    }
#pragma unroll
  for (int u = 0; u < CH; ++u)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float v = weights ? c[u][k] : w[u][k] + c[u][k];
      if (!weights) zs[(k * L + l0 + u) * 256] = v;
      n2[k] = fmaf(v, v, n2[k]);
    }
}

template <int K>
__global__ void __launch_bounds__(256, 4) k_prox2(float* __restrict__ W, const float* __restrict__ coef,
                                               const float* __restrict__ x, const float* __restrict__ theta,
                                               float* __restrict__ theta_out, int64_t I, int64_t dirac_off, int64_t N,
                                               int L, float alpha_scale, float mu, int weights) {
  extern __shared__ float zs_all[];                     // [K][L][256]
  constexpr int CH = 16 / K;
  float* zs = zs_all + threadIdx.x;
  for (int64_t i0 = (int64_t)blockIdx.x * (256 * K) + threadIdx.x; i0 < I; i0 += (int64_t)gridDim.x * (256 * K)) {
    int64_t i[K];
    float n2[K], th[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      i[k] = i0 + 256 * k < I ? i0 + 256 * k : -1;
      n2[k] = 0.f;
      th[k] = weights || i[k] < 0 ? 0.f : theta[i[k]];
    }
    int l = 0;
    for (; l + CH <= L; l += CH) prox_load<CH, K>(zs, n2, W, coef, x, i, I, dirac_off, N, l, L, weights);
    if (CH > 8 && (L - l) & 8) { prox_load<8, K>(zs, n2, W, coef, x, i, I, dirac_off, N, l, L, weights); l += 8; }
    if (CH > 4 && (L - l) & 4) { prox_load<4, K>(zs, n2, W, coef, x, i, I, dirac_off, N, l, L, weights); l += 4; }
    if ((L - l) & 2) { prox_load<2, K>(zs, n2, W, coef, x, i, I, dirac_off, N, l, L, weights); l += 2; }
    if ((L - l) & 1) prox_load<1, K>(zs, n2, W, coef, x, i, I, dirac_off, N, l, L, weights);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (i[k] < 0) continue;
      const float nrm = sqrtf(n2[k]);
      if (weights) {
        theta_out[i[k]] = mu / (nrm + mu);
        continue;
      }
      const float alpha = alpha_scale * th[k];
      const float fct = nrm > alpha ? alpha / nrm : 1.f;
#pragma unroll 16 / K
      for (int m = 0; m < L; ++m) W[(size_t)m * I + i[k]] = zs[(k * L + m) * 256] * fct;
    }
  }
}

// ------------------------------------------------------------ synthesis
struct Syn2 {
  const float* ll;     // synthesised coarser band [L][mo1][mo2], or null: LL4 from W (/3)
  const float* W;
  int64_t I;
  int64_t off[4];      // d0, d1, d2, LL4
  int mo1, mo2, m1, m2;
};

// Synthesis of one (basis, level) tile of T x T outputs.  Pass y: a thread takes one
// coefficient column and STEPS coefficient rows of it (2 STEPS output rows), its
// STEPS + F/2 - 1 coefficients of two bands at a time straight from global memory into
// registers (coalesced along the row, all in flight), and leaves the low and high rows in
// shared memory; pass x: a thread takes OUT consecutive outputs of a row, its windows read
// as float4 (the row pitches spread a quarter-warp over all banks).  Per pixel and basis
// of length F this is about 2.3 F FMAs at T = 64 beside F/4 loads and stores; the form with
// 32 x 32 tiles that staged the bands in shared memory and read every operand of both passes
// from there spent 735 instructions a pixel at level 1 of all bases for 180 FMAs (6.70 ms at
// 16 channels of 4096^2; now 3.10 ms, 1.6 of them the bytes).
//
// 32 x 32 tiles (images too small for two waves of the others) are bound by latency: half the
// rows and outputs per thread, and all four bands' loads in flight at once.
template <int T> struct SynCfg {
  static constexpr int STEPS = T == 64 ? 4 : 2;      // coefficient rows per task of pass y
  static constexpr int OUT = T == 64 ? 16 : 8;       // outputs per thread of pass x
  static constexpr int KN = T / 2 + kMaxFilt / 2;    // coefficient columns, longest filter
  static constexpr int LD = T == 64 ? 44 : 28;       // pitch of the low / high rows
  static constexpr int SEGS = T / 2 / STEPS;
  static constexpr int NT = (KN * SEGS + 31) / 32 * 32;      // 320 or 192: one task of pass y each
  static constexpr int XT = T * T / OUT;                     // 256 or 128 threads of pass x
  static constexpr int BUF = 2 * T * LD;                     // floats: low rows, then high rows
  static_assert(LD >= KN && LD % 4 == 0 && XT <= NT, "synthesis tile");
};

template <int T, int F, bool INSIDE>
__device__ __forceinline__ void syn_pass_y(const Syn2& s, int l, int r0, int c0, float* lx, float ll_scale) {
  using C = SynCfg<T>;
  constexpr int KN = T / 2 + F / 2, ROWS = C::STEPS + F / 2 - 1;
  const int seg = threadIdx.x / KN, kc = threadIdx.x - seg * KN;
  if (seg >= C::SEGS) return;
  const int m0 = seg * C::STEPS, k = r0 / 2 + m0, gc = c0 / 2 + kc;
  const int nrow = INSIDE ? ROWS : (gc < s.mo2 ? s.mo1 - k : 0);       // rows of this column inside the band
  const float* Wl = s.W + (size_t)l * s.I;
  const int64_t start = (int64_t)k * s.mo2 + gc;
  const float third = 1.f / 3.f;
  FTaps<F> f;
  float* o = lx + 2 * m0 * C::LD + kc;
  // low rows (half 0) from LL and d1, high rows (half 1) from d0 and d2
  constexpr int NH = T == 64 ? 1 : 2;                // halves loaded together
  float va[NH][ROWS], vb[NH][ROWS];
  auto fetch = [&](int half, float* a, float* b) {
    const float* pa = half ? Wl + s.off[0] + start
                           : (s.ll ? s.ll + (size_t)l * s.mo1 * s.mo2 : Wl + s.off[3]) + start;
    const float* pb = Wl + s.off[half ? 2 : 1] + start;
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      a[u] = INSIDE || u < nrow ? pa[(size_t)u * s.mo2] : 0.f;
      b[u] = INSIDE || u < nrow ? pb[(size_t)u * s.mo2] : 0.f;
    }
  };
#pragma unroll
  for (int h = 0; h < NH; ++h) fetch(h, va[h], vb[h]);
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (half >= NH) fetch(half, va[0], vb[0]);
    const float* a = va[half < NH ? half : 0];
    const float* b = vb[half < NH ? half : 0];
#pragma unroll
    for (int m = 0; m < C::STEPS; ++m) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float sh = 0.f, sg = 0.f;
#pragma unroll
        for (int q = 0; q < F / 2; ++q) {
          sh = fmaf(f.h[2 * q + 1 - p], a[m + q], sh);
          sg = fmaf(f.g[2 * q + 1 - p], b[m + q], sg);
        }
        // the dictionary's 1/3 (ll_scale: 1 for a synthesised LL band) once per value
        o[(half * T + 2 * m + p) * C::LD] = half ? third * (sh + sg) : fmaf(ll_scale, sh, third * sg);
      }
    }
  }
}

// acc += outputs OUT (tid % (T/OUT)) .. of row tid / (T/OUT).
template <int T, int F>
__device__ __forceinline__ void syn_pass_x(const float* lx, float (&acc)[SynCfg<T>::OUT]) {
  using C = SynCfg<T>;
  constexpr int NW = SynCfg<T>::OUT / 2 + F / 2 - 1, N4 = (NW + 3) / 4;
  if ((int)threadIdx.x >= C::XT) return;
  const int il = threadIdx.x / (T / SynCfg<T>::OUT), mg = threadIdx.x % (T / SynCfg<T>::OUT) * (SynCfg<T>::OUT / 2);
  FTaps<F> f;
  float a[4 * N4], b[4 * N4];
#pragma unroll
  for (int u = 0; u < N4; ++u) {
    const float4 x = *reinterpret_cast<const float4*>(lx + il * C::LD + mg + 4 * u);
    const float4 y = *reinterpret_cast<const float4*>(lx + (T + il) * C::LD + mg + 4 * u);
    a[4 * u] = x.x; a[4 * u + 1] = x.y; a[4 * u + 2] = x.z; a[4 * u + 3] = x.w;
    b[4 * u] = y.x; b[4 * u + 1] = y.y; b[4 * u + 2] = y.z; b[4 * u + 3] = y.w;
  }
#pragma unroll
  for (int m = 0; m < SynCfg<T>::OUT / 2; ++m) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < F / 2; ++q)
        v = fmaf(f.h[2 * q + 1 - p], a[m + q], fmaf(f.g[2 * q + 1 - p], b[m + q], v));
      acc[2 * m + p] += v;
    }
  }
}

// Pass y, a barrier, pass x of filter length F on the buffer sh (2 T LD floats).
template <int T, int F>
__device__ __forceinline__ void syn_tile(const Syn2& s, int l, int r0, int c0, float* sh, float ll_scale,
                                         float (&acc)[SynCfg<T>::OUT]) {
  const bool inside = r0 / 2 + T / 2 + F / 2 <= s.mo1 && c0 / 2 + T / 2 + F / 2 <= s.mo2;
  if (inside) syn_pass_y<T, F, true>(s, l, r0, c0, sh, ll_scale);
  else syn_pass_y<T, F, false>(s, l, r0, c0, sh, ll_scale);
  __syncthreads();
  syn_pass_x<T, F>(sh, acc);
}

// The accumulators as a [T][T + 4] tile in sh (after a barrier), for coalesced stores.
template <int T>
__device__ __forceinline__ void syn_to_tile(float* sh, const float (&acc)[SynCfg<T>::OUT]) {
  __syncthreads();
  if ((int)threadIdx.x < SynCfg<T>::XT) {
    float* o = sh + threadIdx.x / (T / SynCfg<T>::OUT) * (T + 4) + threadIdx.x % (T / SynCfg<T>::OUT) * SynCfg<T>::OUT;
#pragma unroll
    for (int u = 0; u < SynCfg<T>::OUT / 4; ++u)
      *reinterpret_cast<float4*>(o + 4 * u) = make_float4(acc[4 * u], acc[4 * u + 1], acc[4 * u + 2], acc[4 * u + 3]);
  }
  __syncthreads();
}

// One synthesis level (4 -> 3, 3 -> 2 or 2 -> 1) of every basis in one launch, tiles of
// all bases along blockIdx.x (longest filters first), channels along blockIdx.y.
struct Syn2All {
  Syn2 s[8];
  float* out[8];       // synthesised LL band of the finer level [L][m1][m2]
  int tiles_x[8], tile0[8], F[8];
  int nb;
};

template <int T, int F>
__device__ __forceinline__ void syn2_body(const Syn2& s, float* __restrict__ out, int tiles_x, int tile, int l,
                                          float* sh) {
  const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
  const int r0 = ty * T, c0 = tx * T;
  float acc[SynCfg<T>::OUT];
#pragma unroll
  for (int u = 0; u < SynCfg<T>::OUT; ++u) acc[u] = 0.f;
  syn_tile<T, F>(s, l, r0, c0, sh, s.ll ? 1.f : 1.f / 3.f, acc);
  syn_to_tile<T>(sh, acc);
  float* ol = out + (size_t)l * s.m1 * s.m2;
  for (int k = threadIdx.x; k < T * T; k += SynCfg<T>::NT) {
    const int r = k / T, c = k % T;
    if (r0 + r < s.m1 && c0 + c < s.m2) ol[(size_t)(r0 + r) * s.m2 + c0 + c] = sh[r * (T + 4) + c];
  }
}

template <int T>
__global__ void __launch_bounds__(SynCfg<T>::NT) k_syn2_all(const Syn2All a) {
  __shared__ __align__(16) float sh[SynCfg<T>::BUF];
  const int t = blockIdx.x, l = blockIdx.y;
  int bi = 0;
#pragma unroll 1
  for (int k = 1; k < a.nb; ++k)
    if (t >= a.tile0[k]) bi = k;
  const int tile = t - a.tile0[bi];
  switch (a.F[bi]) {
    case 2: syn2_body<T, 2>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 4: syn2_body<T, 4>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 6: syn2_body<T, 6>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 8: syn2_body<T, 8>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 10: syn2_body<T, 10>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 12: syn2_body<T, 12>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    case 14: syn2_body<T, 14>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
    default: syn2_body<T, 16>(a.s[bi], a.out[bi], a.tiles_x[bi], tile, l, sh); break;
  }
}

template <int F>
__global__ void __launch_bounds__(SynCfg<64>::NT) k_syn2_one(const Syn2 s, float* __restrict__ out, int tiles_x) {
  __shared__ __align__(16) float sh[SynCfg<64>::BUF];
  syn2_body<64, F>(s, out, tiles_x, blockIdx.x, blockIdx.y, sh);
}

// A level runs as one launch per basis when the smallest basis alone has at least two
// waves of CTAs (four per SM), else as one merged launch over all bases.
static bool sara_level_per_basis(const int* tiles, int L) {
  int64_t mn = INT64_MAX;
  for (int k = 0; k < 8; ++k) mn = std::min<int64_t>(mn, (int64_t)tiles[k] * L);
  return mn >= 2LL * 4 * num_sms();
}

#define FHS_F_SWITCH(F, KERNEL, GRID, NT, ...)                           \
  switch (F) {                                                           \
    case 2: KERNEL<2><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;          \
    case 4: KERNEL<4><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;          \
    case 6: KERNEL<6><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;          \
    case 8: KERNEL<8><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;          \
    case 10: KERNEL<10><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;        \
    case 12: KERNEL<12><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;        \
    case 14: KERNEL<14><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;        \
    default: KERNEL<16><<<GRID, NT, 0, st>>>(__VA_ARGS__); break;        \
  }

struct SynFin2 {
  Syn2 lv[8];          // level-1 description of each basis (ll = its synthesised LL1)
  int64_t dirac_off;
  int n1, n2;
  float kappa;
  int vec4;            // A, W, the Dirac block and n2 allow 16-byte accesses
};

// Level 1 of all bases and the Dirac block for a T x T output tile, accumulated in
// registers; A += kappa * result.  The low / high rows of consecutive bases alternate between
// two buffers, so a basis costs one barrier.
template <int T>
__global__ void __launch_bounds__(SynCfg<T>::NT, T == 64 ? 3 : 2) k_synfin(const SynFin2 s, float* __restrict__ A) {
  extern __shared__ __align__(16) float synfin_sh[];             // 2 BUF floats
  constexpr int BUF = SynCfg<T>::BUF;
  const int l = blockIdx.z, r0 = blockIdx.y * T, c0 = blockIdx.x * T;
  float acc[SynCfg<T>::OUT];
#pragma unroll
  for (int u = 0; u < SynCfg<T>::OUT; ++u) acc[u] = 0.f;
  syn_tile<T, 2>(s.lv[0], l, r0, c0, synfin_sh, 1.f, acc);
  syn_tile<T, 4>(s.lv[1], l, r0, c0, synfin_sh + BUF, 1.f, acc);
  syn_tile<T, 6>(s.lv[2], l, r0, c0, synfin_sh, 1.f, acc);
  syn_tile<T, 8>(s.lv[3], l, r0, c0, synfin_sh + BUF, 1.f, acc);
  syn_tile<T, 10>(s.lv[4], l, r0, c0, synfin_sh, 1.f, acc);
  syn_tile<T, 12>(s.lv[5], l, r0, c0, synfin_sh + BUF, 1.f, acc);
  syn_tile<T, 14>(s.lv[6], l, r0, c0, synfin_sh, 1.f, acc);
  syn_tile<T, 16>(s.lv[7], l, r0, c0, synfin_sh + BUF, 1.f, acc);
  syn_to_tile<T>(synfin_sh, acc);
  const size_t N = (size_t)s.n1 * s.n2;
  const float* Wd = s.lv[0].W + (size_t)l * s.lv[0].I + s.dirac_off;
  float* Al = A + (size_t)l * N;
  // four consecutive outputs: one 16-byte read-modify-write of A where the rows and the
  // Dirac block allow it
  for (int k = threadIdx.x; k < T * T / 4; k += SynCfg<T>::NT) {
    const int rr = k / (T / 4), cc = k % (T / 4) * 4, r = r0 + rr, c = c0 + cc;
    if (r >= s.n1 || c >= s.n2) continue;
    const float4 v = *reinterpret_cast<const float4*>(synfin_sh + rr * (T + 4) + cc);
    const size_t o = (size_t)r * s.n2 + c;
    if (s.vec4 && c + 3 < s.n2) {
      const float4 wd = *reinterpret_cast<const float4*>(Wd + o);
      float4 a = *reinterpret_cast<const float4*>(Al + o);
      a.x = fmaf(s.kappa, v.x + wd.x * (1.f / 3.f), a.x);
      a.y = fmaf(s.kappa, v.y + wd.y * (1.f / 3.f), a.y);
      a.z = fmaf(s.kappa, v.z + wd.z * (1.f / 3.f), a.z);
      a.w = fmaf(s.kappa, v.w + wd.w * (1.f / 3.f), a.w);
      *reinterpret_cast<float4*>(Al + o) = a;
    } else {
      const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (c + q < s.n2) Al[o + q] = fmaf(s.kappa, e[q] + Wd[o + q] * (1.f / 3.f), Al[o + q]);
    }
  }
}

// Synthesis tiles: 64 x 64 where they make at least two waves of CTAs (three per SM; halo
// 1.56 coefficients per output pair against 2.25 at 32), else 32 x 32.
static bool syn_large_tiles(int64_t ctas64) { return ctas64 >= 2LL * 3 * num_sms(); }

// ------------------------------------------------------------- launchers
// launch_sara_dual: analysis of every basis and level into the coefficient buffer, the l2,1
// dual (or weights), then (dual mode) the synthesis down to the LL1 bands; launch_sara_fin:
// level 1 of the synthesis and the Dirac block, accumulated into A.
void launch_sara_fast(fhs_ctx* ctx, const Cube& cb, const float* x, float* W, const float* theta, float* A,
                      float* theta_out, bool weights, cudaStream_t st) {
  launch_sara_dual(ctx, cb, x, W, theta, theta_out, weights, st);
  if (!weights) launch_sara_fin(ctx, cb, W, A, st);
}

void launch_sara_dual(fhs_ctx* ctx, const Cube& cb, const float* x, float* W, const float* theta, float* theta_out,
                      bool weights, cudaStream_t st) {
  const SaraLayout& S = cb.sara;
  const int L = cb.L;
  float* coef = ctx->s.coef;
  // LL1, LL2 and LL3 slots of the eight bases (also used by the synthesis below)
  {
    int64_t o1 = 0, o2 = 0, o3 = 0;
    for (int b = 0; b < 8; ++b) {
      ctx->s.ll1_off[b] = o1;
      ctx->s.ll2_off[b] = o2;
      ctx->s.ll3_off[b] = o3;
      o1 += (int64_t)L * S.rows[b][1] * S.cols[b][1];
      o2 += (int64_t)L * S.rows[b][2] * S.cols[b][2];
      o3 += (int64_t)L * S.rows[b][3] * S.cols[b][3];
    }
  }
  // level 1 of every basis in one launch (grid over the longest filter's coefficients)
  {
    Ana1 a;
    for (int b = 0; b < 8; ++b) {
      for (int k = 0; k < 3; ++k) a.off[b][k] = S.off[b][1][k];
      a.mo1[b] = S.rows[b][1];
      a.mo2[b] = S.cols[b][1];
      a.ll_off[b] = ctx->s.ll1_off[b];
    }
    int r = 0, c = 0;
    for (int b = 0; b < 8; ++b) { r = std::max(r, S.rows[b][1]); c = std::max(c, S.cols[b][1]); }
    dim3 g((c + kT2 - 1) / kT2, (r + kT2 - 1) / kT2, L);
    k_ana1_all<<<g, 256, 0, st>>>(x, coef, ctx->s.ll1, a, S.I, cb.n1, cb.n2);
    note_launches(1);
  }
  // levels 2..4: one launch per level over the tiles of every basis (longest filters
  // first); LL2 and LL3 of each basis in its own slot of s.ll2 / s.ll3
  for (int j = 2; j <= kLevels; ++j) {
    Ana2All a;
    a.nb = 8;
    int t0 = 0;
    for (int k = 0; k < 8; ++k) {
      const int b = 7 - k;
      Ana2Basis& B = a.b[k];
      B.in = (j == 2) ? ctx->s.ll1 + ctx->s.ll1_off[b] : (j == 3) ? ctx->s.ll2 + ctx->s.ll2_off[b]
                                                                  : ctx->s.ll3 + ctx->s.ll3_off[b];
      B.ll_out = (j == 2) ? ctx->s.ll2 + ctx->s.ll2_off[b] : (j == 3) ? ctx->s.ll3 + ctx->s.ll3_off[b] : nullptr;
      for (int q = 0; q < 3; ++q) B.off[q] = S.off[b][j][q];
      B.off_ll = S.off[b][kLevels][3];
      B.m1 = S.rows[b][j - 1]; B.m2 = S.cols[b][j - 1];
      B.mo1 = S.rows[b][j]; B.mo2 = S.cols[b][j];
      B.tiles_x = (B.mo2 + kT2 - 1) / kT2;
      B.tile0 = t0;
      B.F = 2 * (b + 1);
      t0 += B.tiles_x * ((B.mo1 + kT2 - 1) / kT2);
    }
    int tiles[8];
    for (int k = 0; k < 8; ++k) tiles[k] = (k + 1 < 8 ? a.b[k + 1].tile0 : t0) - a.b[k].tile0;
    if (sara_level_per_basis(tiles, L)) {
      for (int k = 0; k < 8; ++k) {
        FHS_F_SWITCH(a.b[k].F, k_ana2_one, dim3(tiles[k], L), 256, a.b[k], coef, S.I);
      }
      note_launches(8);
    } else {
      k_ana2_all<<<dim3(t0, L), 256, 0, st>>>(a, coef, S.I);
      note_launches(1);
    }
  }
  {
    const int64_t N = (int64_t)cb.n1 * cb.n2;
    const float as = (float)(cb.mu / cb.kappa), mu = (float)cb.mu;
    const int wm = weights ? 1 : 0;
    auto go = [&](auto kernel, int K, bool& attr) {
      const unsigned g =
          (unsigned)std::min<int64_t>((S.I + 256 * K - 1) / (256 * K), (int64_t)num_sms() * cb.prox_cps);
      const size_t smem = weights ? 0 : (size_t)K * L * 256 * sizeof(float);
      if (!attr) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxL * 256 * (int)sizeof(float));
        attr = true;
      }
      kernel<<<g, 256, smem, st>>>(W, coef, x, theta, theta_out, S.I, S.dirac_off, N, L, as, mu, wm);
    };
    static bool attr1 = false, attr2 = false, attr4 = false;
    if (L <= 4) go(k_prox2<4>, 4, attr4);
    else if (L <= 8) go(k_prox2<2>, 2, attr2);
    else go(k_prox2<1>, 1, attr1);
    note_launches(1);
  }
  if (weights) return;
  float* slots = ctx->s.ll1;
  // levels 4 -> 2: one launch per level over the tiles of every basis; the synthesised
  // LL3, LL2 and LL1 bands reuse the analysis slots (s.ll3, s.ll2, s.ll1)
  for (int j = kLevels; j >= 2; --j) {
    Syn2All a;
    a.nb = 8;
    auto tiles_of = [&](int b, int T) {
      return ((S.cols[b][j - 1] + T - 1) / T) * ((S.rows[b][j - 1] + T - 1) / T);
    };
    int64_t n64 = 0;
    for (int b = 0; b < 8; ++b) n64 += tiles_of(b, 64);
    const int T = syn_large_tiles(n64 * L) ? 64 : 32;
    int t0 = 0, tiles[8];
    for (int k = 0; k < 8; ++k) {
      const int b = 7 - k;
      Syn2& s = a.s[k];
      s.ll = (j == kLevels) ? nullptr : (j == 3) ? ctx->s.ll3 + ctx->s.ll3_off[b] : ctx->s.ll2 + ctx->s.ll2_off[b];
      s.W = W;
      s.I = S.I;
      s.off[0] = S.off[b][j][0]; s.off[1] = S.off[b][j][1]; s.off[2] = S.off[b][j][2];
      s.off[3] = S.off[b][kLevels][3];
      s.mo1 = S.rows[b][j]; s.mo2 = S.cols[b][j];
      s.m1 = S.rows[b][j - 1]; s.m2 = S.cols[b][j - 1];
      a.out[k] = (j == 2) ? slots + ctx->s.ll1_off[b] : (j == 3) ? ctx->s.ll2 + ctx->s.ll2_off[b]
                                                                 : ctx->s.ll3 + ctx->s.ll3_off[b];
      a.tiles_x[k] = (s.m2 + T - 1) / T;
      a.tile0[k] = t0;
      a.F[k] = 2 * (b + 1);
      tiles[k] = tiles_of(b, T);
      t0 += tiles[k];
    }
    if (T == 64 && sara_level_per_basis(tiles, L)) {
      for (int k = 0; k < 8; ++k) {
        FHS_F_SWITCH(a.F[k], k_syn2_one, dim3(tiles[k], L), SynCfg<64>::NT, a.s[k], a.out[k], a.tiles_x[k]);
      }
      note_launches(8);
    } else {
      if (T == 64) k_syn2_all<64><<<dim3(t0, L), SynCfg<64>::NT, 0, st>>>(a);
      else k_syn2_all<32><<<dim3(t0, L), SynCfg<32>::NT, 0, st>>>(a);
      note_launches(1);
    }
  }
}

void launch_sara_fin(fhs_ctx* ctx, const Cube& cb, const float* W, float* A, cudaStream_t st) {
  const SaraLayout& S = cb.sara;
  const int L = cb.L;
  SynFin2 fin;
  int64_t o1 = 0;                                    // the LL1 slots of launch_sara_dual
  for (int b = 0; b < 8; ++b) {
    Syn2& f = fin.lv[b];
    f.ll = ctx->s.ll1 + o1;
    o1 += (int64_t)L * S.rows[b][1] * S.cols[b][1];
    f.W = W;
    f.I = S.I;
    f.off[0] = S.off[b][1][0]; f.off[1] = S.off[b][1][1]; f.off[2] = S.off[b][1][2];
    f.off[3] = S.off[b][kLevels][3];
    f.mo1 = S.rows[b][1]; f.mo2 = S.cols[b][1];
    f.m1 = cb.n1; f.m2 = cb.n2;
  }
  fin.dirac_off = S.dirac_off;
  fin.n1 = cb.n1;
  fin.n2 = cb.n2;
  fin.kappa = (float)cb.kappa;
  fin.vec4 = (cb.n2 % 4 == 0 && S.dirac_off % 4 == 0 && S.I % 4 == 0 && ((uintptr_t)A % 16) == 0 &&
              ((uintptr_t)W % 16) == 0) ? 1 : 0;
  auto launch_fin = [&](auto kernel, int T, int nt, int buf) {
    const size_t sm = 2 * (size_t)buf * sizeof(float);
    kernel<<<dim3((cb.n2 + T - 1) / T, (cb.n1 + T - 1) / T, L), nt, sm, st>>>(fin, A);
  };
  const int64_t n64 = (int64_t)((cb.n2 + 63) / 64) * ((cb.n1 + 63) / 64) * L;
  if (syn_large_tiles(n64)) launch_fin(k_synfin<64>, 64, SynCfg<64>::NT, SynCfg<64>::BUF);
  else launch_fin(k_synfin<32>, 32, SynCfg<32>::NT, SynCfg<32>::BUF);
  note_launches(1);
}

bool sara_fast_supported(const Cube&) { return true; }

}  // namespace fhs
