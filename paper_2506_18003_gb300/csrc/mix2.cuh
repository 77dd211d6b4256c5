// Mixed-radix transforms on the packed lanes: the SSCA strips of a length that splits into two factors with
// such a plan (17 .. 4096 each), and the FAM pair transform for a P of at most 4096 that is not a
// power of two but a product of up to four radices out of 2 .. 10, 12, 15 and 16 (P = 2^a 3^b 5^c 7^d; lengths
// with a larger prime factor, 11 x 11 or 11 x 13 for instance, have no plan),
// FP32 form.  One transform of size P per pair, where Bluestein's identity (bluestein2.cuh) takes two of
// size >= 2 P - 1.
//
// Gentleman-Sande passes in place (W. M. Gentleman, G. Sande, 1966): with L_0 = P, L_{s+1} = L_s / r_s,
// pass s transforms the r_s values L_{s+1} apart of each block of L_s and multiplies output k at offset m by
// W_{L_s}^{k m}; after the last pass the value of digits (k_0, k_1, ..) is bin k_0 + r_0 k_1 + r_0 r_1 k_2 + ..
// The first pass reads the products X conj(Y) from global memory, the last one writes the bins there, so n
// passes cost n - 1 shared-memory round trips and n barriers.  A pass hands its butterflies, over all pairs of
// the tile, to the block's threads in turn; its radix is a uniform switch.  Inside a butterfly: powers of
// two as fft2.cuh, 3, 5 and 7 over sums and differences of conjugate inputs, products of coprime factors
// without twiddle factors by the prime-factor mapping (I. J. Good, 1958), 9 as 3 x 3.
// Blocks of first digit k_0 lie at an odd stride: the last pass, whose threads run over k_0 first so that
// its stores are contiguous, then reads 16-byte values from 8 different banks per quarter-warp.
// Bound by latency: at Np = 256, P = 1000 (radices 10, 10, 10) the 524 MB of results leave at 3.7 TB/s (L2 takes
// 6.3) with 0.35 of the issue slots used; 16 warps per SM wait on the row reads (a first-pass butterfly
// of radix 10 issues 40 of 8 bytes) and at the barriers between the passes.
// Microseconds per estimate, Bluestein one-pair / packed Bluestein / this:
//   (Np, P) = (64, 20) 10.8 / 5.7 / 6.1, (32, 45) 12.7 / 6.5 / 6.0, (64, 100) 10.6 / 7.6 / 6.2,
//   (128, 200, cross) 60 / 35 / 21, (256, 500) 213 / 146 / 82, (256, 1000) 357 / 313 / 142,
//   (128, 1000, cross) 180 / 153 / 66, (64, 1500) 56 / - / 20, (64, 3000) 132 / - / 45, (64, 4050) 144 / - / 56.
#pragma once
#include "fft2.cuh"
#include "pdl.cuh"
#include "tiles.cuh"

namespace scd {

// cos and sin of 2 pi j / R
template <int R>
__host__ __device__ constexpr float odd_cos(int j) {
  if (j == 0) return 1.f;
  if (2 * j > R) j = R - j;
  if (R == 3) return -0.5f;
  if (R == 5) return j == 1 ? 0.30901699437494742f : -0.80901699437494742f;
  if (R == 7) return j == 1 ? 0.62348980185873353f : (j == 2 ? -0.22252093395631440f : -0.90096886790241913f);
  // 9
  return j == 1 ? 0.76604444311897804f : (j == 2 ? 0.17364817766693035f : (j == 3 ? -0.5f : -0.93969262078590838f));
}
template <int R>
__host__ __device__ constexpr float odd_sin(int j) {
  if (j == 0) return 0.f;
  if (2 * j > R) return -odd_sin<R>(R - j);
  if (R == 3) return 0.86602540378443865f;
  if (R == 5) return j == 1 ? 0.95105651629515357f : 0.58778525229247313f;
  if (R == 7) return j == 1 ? 0.78183148246802981f : (j == 2 ? 0.97492791218182361f : 0.43388373911755812f);
  return j == 1 ? 0.64278760968653933f : (j == 2 ? 0.98480775301220806f : (j == 3 ? 0.86602540378443865f : 0.34202014332566873f));
}

// (constants as template-evaluated: computed in unrolled loops they stayed in registers, 119 instead of 54 for
// R = 10 and 40% on the kernel)
// R = 3, 5, 7: X_k, X_{R-k} = A_k -+ i B_k, A_k = v_0 + sum_j cos(2 pi j k / R) (v_j + v_{R-j}),
// B_k = sum_j sin(2 pi j k / R) (v_j - v_{R-j})
template <int R, int K, int J>
__host__ __device__ __forceinline__ void odd_sums(const C2* a, const C2* b, C2& A, C2& B) {
  if constexpr (J <= R / 2) {
    constexpr float c = odd_cos<R>(J * K % R), s = odd_sin<R>(J * K % R);
    A = C2{fma2(a[J].re, dup2(c), A.re), fma2(a[J].im, dup2(c), A.im)};
    if constexpr (J == 1) B = C2{mul2(b[J].re, dup2(s)), mul2(b[J].im, dup2(s))};
    else B = C2{fma2(b[J].re, dup2(s), B.re), fma2(b[J].im, dup2(s), B.im)};
    odd_sums<R, K, J + 1>(a, b, A, B);
  }
}
template <int R, int K>
__host__ __device__ __forceinline__ void odd_outputs(const C2* a, const C2* b, const C2& v0, C2* v) {
  if constexpr (K <= R / 2) {
    C2 A = v0, B;
    odd_sums<R, K, 1>(a, b, A, B);
    v[K] = C2{add2(A.re, B.im), sub2(A.im, B.re)};
    v[R - K] = C2{sub2(A.re, B.im), add2(A.im, B.re)};
    odd_outputs<R, K + 1>(a, b, v0, v);
  }
}
template <int R>
__host__ __device__ __forceinline__ void dft_odd(C2* v) {
  constexpr int H = R / 2;
  C2 a[H + 1], b[H + 1];
  const C2 v0 = v[0];
#pragma unroll
  for (int j = 1; j <= H; ++j) {
    a[j] = cadd(v[j], v[R - j]);
    b[j] = csub(v[j], v[R - j]);
    v[0] = cadd(v[0], a[j]);
  }
  odd_outputs<R, 1>(a, b, v0, v);
}

__host__ __device__ constexpr int inverse_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if (a * i % m == 1) return i;
  return 1;
}

template <int R>
__host__ __device__ __forceinline__ void dft_any(C2* v) {
  if constexpr ((R & (R - 1)) == 0) {
    dft2<R>(v);
  } else if constexpr (R == 3 || R == 5 || R == 7) {
    dft_odd<R>(v);
  } else if constexpr (R == 9) {                               // n = 3 n1 + n2, k = k1 + 3 k2
    C2 u[3][3];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
      C2 w[3] = {v[n2], v[3 + n2], v[6 + n2]};
      dft_odd<3>(w);
#pragma unroll
      for (int k1 = 0; k1 < 3; ++k1)
        u[k1][n2] = n2 * k1 == 0 ? w[k1] : cmul(w[k1], make_float2(odd_cos<9>(n2 * k1), -odd_sin<9>(n2 * k1)));
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      dft_odd<3>(u[k1]);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = u[k1][k2];
    }
  } else {                                                     // n = B n1 + A n2, k = k1 mod A, k2 mod B
    constexpr int B = R % 7 == 0 ? 7 : (R % 5 == 0 ? 5 : 3), A = R / B;
    constexpr int ka = B * inverse_mod(B % A, A), kb = A * inverse_mod(A % B, B);
    C2 u[A][B];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) u[n1][n2] = v[(B * n1 + A * n2) % R];
      dft_odd<B>(u[n1]);
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
      C2 w[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) w[n1] = u[n1][k2];
      dft_any<A>(w);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) v[(k1 * ka + k2 * kb) % R] = w[k1];
    }
  }
}

// d -> x / d for x < 65536, d < 65536: the high word of x times ceil(2^32 / d)
struct Div16 {
  unsigned d, magic;
  __host__ __device__ void set(unsigned v) { d = v; magic = v > 1 ? (unsigned)(((uint64_t(1) << 32) + v - 1) / v) : 0; }
  __host__ __device__ unsigned quot(unsigned x) const {
    return d > 1 ? (unsigned)(((uint64_t)x * magic) >> 32) : x;
  }
};

// The passes of one size: radices, block lengths, table offsets; `stride` float4 per first digit, `unit` per
// transform.
struct MixPlan {
  int P, n;
  int r[4], len[5], off[4];                                    // len[s] = L_s
  int stride, unit, tw_len;
  Div16 per[4], m[4], r0, r1;                                  // P / r_s, L_{s+1}, r_0, r_1
};

// The plan of any length 17 .. 4096 that is such a product (powers of two too); false: none.
bool mix_factor(int P, MixPlan* plan);
// The plan of a FAM length P (only its n, radices, lengths and table sizes depend on P); false: no plan.
bool mix_plan(int P, MixPlan* plan);
// SSCA strips of length N (FP32): the split N1 N2 and the tile widths; false: no split.
struct StripPlan {
  MixPlan a, b;                                                // the column pass (N1), the row pass (N2)
  int N1, N2, lca, lcb;
};
bool strip_plan(int64_t N, StripPlan* plan);
cudaError_t strip_cols(const StripPlan& plan, int64_t N, int rows, const float2* in, int64_t ld, float2* out, int64_t ldo,
                       cudaStream_t st);
cudaError_t strip_rows(const StripPlan& plan, int64_t N, int rows, const float2* in, int64_t ld, float2* out, int64_t ldo,
                       cudaStream_t st);
cudaError_t fam_mix_pairs(const float2* X, const float2* Y, int Np, const MixPlan& plan, float2* out, cudaStream_t st);

constexpr int kMixThreads = 256, kMixCtas = 2, kMixMaxUnits = 16;
inline int mix_smem(const MixPlan& p, int C) { return C * p.unit * 16 + (p.tw_len + 1) / 2 * 16 + 2 * C * 32; }

template <int R> struct Radix { static constexpr int r = R; };
template <class F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
  switch (r) {
    case 2: f(Radix<2>{}); break;
    case 3: f(Radix<3>{}); break;
    case 4: f(Radix<4>{}); break;
    case 5: f(Radix<5>{}); break;
    case 6: f(Radix<6>{}); break;
    case 7: f(Radix<7>{}); break;
    case 8: f(Radix<8>{}); break;
    case 9: f(Radix<9>{}); break;
    case 10: f(Radix<10>{}); break;
    case 12: f(Radix<12>{}); break;
    case 15: f(Radix<15>{}); break;
    case 16: f(Radix<16>{}); break;
  }
}

// The passes of one tile, cv transforms (of C, a power of two when CF) in the exchange area sm.  CF: neighbouring
// threads take the same butterfly of neighbouring transforms (interleaved data), else neighbouring butterflies.
// src(radix, c, m, step, v) gives v[j] = input m + j step of transform c; dst(radix, c, i, step, v) takes bins
// i + j step.
template <bool CF>
__device__ __forceinline__ bool mix_split(int b, const Div16& per, int lc, int cv, int* c, int* i) {
  if constexpr (CF) {
    *c = b & ((1 << lc) - 1);
    *i = b >> lc;
    return *c < cv;
  } else {
    *c = (int)per.quot(b);
    *i = b - *c * (int)per.d;
    return true;
  }
}
template <bool CF>
__device__ __forceinline__ int mix_total(const Div16& per, int lc, int cv) {
  return CF ? (int)per.d << lc : cv * (int)per.d;
}

template <bool CF, class Src>
__device__ __forceinline__ void mix_first(float4* sm, const float2* tws, const MixPlan& pl, int lc, int cv, Src&& src) {
  with_radix(pl.r[0], [&](auto rr) {
    constexpr int R = decltype(rr)::r;
    const int L1 = pl.len[1], total = mix_total<CF>(pl.per[0], lc, cv);
    for (int b = threadIdx.x; b < total; b += kMixThreads) {
      int c, m;
      if (!mix_split<CF>(b, pl.per[0], lc, cv, &c, &m)) continue;
      C2 v[R];
      src(rr, c, m, L1, v);
      dft_any<R>(v);
      float4* d = sm + c * pl.unit + m;
      d[0] = c2_f4(v[0]);
#pragma unroll
      for (int k = 1; k < R; ++k) d[k * pl.stride] = c2_f4(cmul(v[k], tws[k * L1 + m]));
    }
  });
}

template <bool CF>
__device__ __forceinline__ void mix_middle(float4* sm, const float2* tws, const MixPlan& pl, int lc, int cv) {
  for (int s = 1; s + 1 < pl.n; ++s) {
    with_radix(pl.r[s], [&](auto rr) {
      constexpr int R = decltype(rr)::r;
      const int Ln = pl.len[s + 1], total = mix_total<CF>(pl.per[s], lc, cv);
      const float2* w = tws + pl.off[s];
      for (int b = threadIdx.x; b < total; b += kMixThreads) {
        int c, i;
        if (!mix_split<CF>(b, pl.per[s], lc, cv, &c, &i)) continue;
        const int blk = (int)pl.m[s].quot(i), m = i - blk * Ln;
        const int k0 = s == 1 ? blk : (int)pl.r1.quot(blk), rest = s == 1 ? 0 : (blk - k0 * pl.r[1]) * pl.len[2];
        float4* d = sm + c * pl.unit + k0 * pl.stride + rest + m;
        C2 v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = take2(d + j * Ln);
        dft_any<R>(v);
        d[0] = c2_f4(v[0]);
#pragma unroll
        for (int k = 1; k < R; ++k) d[k * Ln] = c2_f4(cmul(v[k], w[k * Ln + m]));
      }
    });
    __syncthreads();
  }
}

template <bool CF, class Dst>
__device__ __forceinline__ void mix_last(const float4* sm, const MixPlan& pl, int lc, int cv, Dst&& dst) {
  with_radix(pl.r[pl.n - 1], [&](auto rr) {
    constexpr int R = decltype(rr)::r;
    const Div16& per = pl.per[pl.n - 1];
    const int total = mix_total<CF>(per, lc, cv);
    for (int b = threadIdx.x; b < total; b += kMixThreads) {
      int c, i;
      if (!mix_split<CF>(b, per, lc, cv, &c, &i)) continue;
      const int i1 = (int)pl.r0.quot(i), k0 = i - i1 * pl.r[0];
      int at = k0 * pl.stride;
      if (pl.n == 3) at += i1 * pl.len[2];
      if (pl.n == 4) {
        const int k2 = (int)pl.r1.quot(i1);
        at += (i1 - k2 * pl.r[1]) * pl.len[2] + k2 * pl.len[3];
      }
      const float4* d = sm + c * pl.unit + at;
      C2 v[R];
#pragma unroll
      for (int j = 0; j < R; ++j) v[j] = take2(d + j);
      dft_any<R>(v);
      dst(rr, c, i, (int)per.d, v);
    }
  });
}

// FAM pairs two by two, persistent over tiles of C units (one unit = two pairs; their number is even).
template <bool SYM>
__device__ __forceinline__ void fam_mix_cta(unsigned char* smem, const MixPlan& pl, int C, const float2* __restrict__ X,
                                            const float2* __restrict__ Y, int Np, float2* __restrict__ out,
                                            const float2* __restrict__ tw) {
  const int P = pl.P, half = P / 2, tid = (int)threadIdx.x;
  float4* sm = reinterpret_cast<float4*>(smem);
  float2* tws = reinterpret_cast<float2*>(sm + C * pl.unit);
  int4* info = reinterpret_cast<int4*>(tws + (pl.tw_len + 1) / 2 * 2);       // per parity and unit: rows, outputs
  for (int e = tid; e < pl.tw_len; e += kMixThreads) tws[e] = __ldg(tw + e);
  const int units = (int)(fam_pair_count<0>(Np, SYM) / 2), tiles = (units + C - 1) / C;
  wait_for_previous();
  int par = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, par ^= 1) {
    if (tile + (int)gridDim.x >= tiles) let_next_start();
    const int cv = min(C, units - tile * C);
    int4* my = info + par * 2 * C;
    if (tid < cv) {
      int k0, l0, k1, l1;
      fam_pair_of<SYM>(2 * (tile * C + tid), Np, &k0, &l0);
      fam_pair_of<SYM>(2 * (tile * C + tid) + 1, Np, &k1, &l1);
      my[2 * tid] = make_int4(k0 * P, l0 * P, k1 * P, l1 * P);
      my[2 * tid + 1] = make_int4((k0 * Np + l0) * P, (k1 * Np + l1) * P, SYM && k0 != l0 ? (l0 * Np + k0) * P : -1,
                                  SYM && k1 != l1 ? (l1 * Np + k1) * P : -1);
    }
    __syncthreads();                                           // and every read of the last tile's values is done
    mix_first<false>(sm, tws, pl, 0, cv, [&](auto rr, int c, int m, int L1, C2* v) {
      constexpr int R = decltype(rr)::r;
      const int4 row = my[2 * c];
      const float2 *a0 = X + row.x + m, *b0 = Y + row.y + m, *a1 = X + row.z + m, *b1 = Y + row.w + m;
#pragma unroll
      for (int j = 0; j < R; ++j)
        v[j] = c2_pack(cmulc(load_written(a0 + j * L1), load_written(b0 + j * L1)),
                       cmulc(load_written(a1 + j * L1), load_written(b1 + j * L1)));
    });
    __syncthreads();
    mix_middle<false>(sm, tws, pl, 0, cv);
    mix_last<false>(sm, pl, 0, cv, [&](auto rr, int c, int i, int nb, const C2* v) {
      constexpr int R = decltype(rr)::r;
      const int4 o = my[2 * c + 1];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int f = i + nb * j;
        const float2 s0 = c2_lane0(v[j]), s1 = c2_lane1(v[j]);
        const int q = f + half < P ? f + half : f + half - P;
        out[o.x + q] = s0;
        out[o.y + q] = s1;
        if constexpr (SYM) {
          const int fm = f == 0 ? 0 : P - f, qm = fm + half < P ? fm + half : fm + half - P;
          if (o.z >= 0) out[o.z + qm] = cconj(s0);
          if (o.w >= 0) out[o.w + qm] = cconj(s1);
        }
      }
    });
  }
}

// ---------------------------------------------------------------- SSCA strips of length N = N1 N2
// Two passes over Np N values, where Bluestein's identity takes three over Np M, M >= 2 N - 1, with twice the
// transforms: N = 100,000 (250 x 400), Np = 128 takes 171 us instead of 407 (28 of them the channeliser in both).
// Bound by latency: 16 warps per SM at 0.3 of the issue slots, waiting on the tile's loads and at the barriers
// between its phases (76 and 65 us cold, 2 TB/s of DRAM traffic).  16 columns or row pairs per tile where they
// fit half an SM's shared memory, so that both passes read or write runs of 256 bytes.
// Column pass: n = n1 N2 + n2, transforms over n1 of the columns n2, two columns per lane pair:
//   out[k1 N2 + n2] = W_N^{n2 k1} sum_{n1} W_N1^{k1 n1} in[n1 N2 + n2],
// in rows of stride ld, out rows of stride ldo (both even, 16-byte aligned).  The rotation is W_N^{n0 k1}
// (table of roots) times W_N^{d k1} (`cols`, [k1][d], d < 2 C) for column n0 + d of a tile.
struct StripArgs {
  int64_t ld, ldo;
  int N1, N2, N, rows, lc;                                     // rows: strips; C = 2^lc lane pairs per tile
};

__device__ __forceinline__ void mix_cols_cta(unsigned char* smem, const MixPlan& pl, const StripArgs& A,
                                             const float2* __restrict__ in, float2* __restrict__ out,
                                             const float2* __restrict__ tw, const float2* __restrict__ wN,
                                             const float2* __restrict__ cols) {
  const int C = 1 << A.lc, N2 = A.N2, tid = (int)threadIdx.x;
  float4* sm = reinterpret_cast<float4*>(smem);
  float2* tws = reinterpret_cast<float2*>(sm + C * pl.unit);
  for (int e = tid; e < pl.tw_len; e += kMixThreads) tws[e] = __ldg(tw + e);
  const int per_row = ((N2 + 1) / 2 + C - 1) / C, tiles = per_row * A.rows;
  const bool even = N2 % 2 == 0;
  wait_for_previous();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (tile + (int)gridDim.x >= tiles) let_next_start();
    const int row = tile / per_row, n0 = (tile - row * per_row) * 2 * C, cv = min(C, (N2 - n0 + 1) / 2);
    const float2* src = in + row * A.ld + n0;
    float2* dst = out + row * A.ldo + n0;
    __syncthreads();
    mix_first<true>(sm, tws, pl, A.lc, cv, [&](auto rr, int c, int m, int L1, C2* v) {
      constexpr int R = decltype(rr)::r;
      const float2* p = src + m * N2 + 2 * c;
      const bool both = n0 + 2 * c + 1 < N2;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        if (even) {
          const float4 q = load_written(reinterpret_cast<const float4*>(p + j * L1 * N2));
          v[j] = c2_pack(make_float2(q.x, q.y), make_float2(q.z, q.w));
        } else {
          v[j] = c2_pack(load_written(p + j * L1 * N2), both ? load_written(p + j * L1 * N2 + 1) : make_float2(0.f, 0.f));
        }
      }
    });
    __syncthreads();
    mix_middle<true>(sm, tws, pl, A.lc, cv);
    mix_last<true>(sm, pl, A.lc, cv, [&](auto rr, int c, int i, int nb, const C2* v) {
      constexpr int R = decltype(rr)::r;
      const bool both = n0 + 2 * c + 1 < N2;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int k1 = i + nb * j;
        const float4 w = __ldg(reinterpret_cast<const float4*>(cols + 2 * (k1 * C + c)));
        const C2 g = cmul(cmul(v[j], C2{make_float2(w.x, w.z), make_float2(w.y, w.w)}), __ldg(wN + n0 * k1));
        float2* p = dst + (int64_t)k1 * N2 + 2 * c;
        if (even) {
          *reinterpret_cast<float4*>(p) = make_float4(g.re.x, g.im.x, g.re.y, g.im.y);
        } else {
          p[0] = c2_lane0(g);
          if (both) p[1] = c2_lane1(g);
        }
      }
    });
  }
}

// Row pass: transforms over n2 of the rows k1, two rows per lane pair; bin q = k1 + N1 k2 goes to
// out[(q + N / 2) mod N] of its strip.
__device__ __forceinline__ void mix_rows_cta(unsigned char* smem, const MixPlan& pl, const StripArgs& A,
                                             const float2* __restrict__ in, float2* __restrict__ out,
                                             const float2* __restrict__ tw) {
  const int C = 1 << A.lc, N1 = A.N1, N2 = A.N2, N = A.N, half = N / 2, tid = (int)threadIdx.x;
  float4* sm = reinterpret_cast<float4*>(smem);
  float2* tws = reinterpret_cast<float2*>(sm + C * pl.unit);
  for (int e = tid; e < pl.tw_len; e += kMixThreads) tws[e] = __ldg(tw + e);
  const int per_row = ((N1 + 1) / 2 + C - 1) / C, tiles = per_row * A.rows;
  const bool even = N1 % 2 == 0 && N % 4 == 0;                 // two bins then are one aligned 16-byte store
  wait_for_previous();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (tile + (int)gridDim.x >= tiles) let_next_start();
    const int row = tile / per_row, r0 = (tile - row * per_row) * 2 * C, cv = min(C, (N1 - r0 + 1) / 2);
    const float2* src = in + row * A.ld + (int64_t)r0 * N2;
    float2* dst = out + row * A.ldo;
    __syncthreads();
    mix_first<false>(sm, tws, pl, 0, cv, [&](auto rr, int c, int m, int L1, C2* v) {
      constexpr int R = decltype(rr)::r;
      const float2* p0 = src + 2 * c * N2 + m;
      const float2* p1 = r0 + 2 * c + 1 < N1 ? p0 + N2 : p0;
#pragma unroll
      for (int j = 0; j < R; ++j) v[j] = c2_pack(load_written(p0 + j * L1), load_written(p1 + j * L1));
    });
    __syncthreads();
    mix_middle<false>(sm, tws, pl, 0, cv);
    mix_last<true>(sm, pl, A.lc, cv, [&](auto rr, int c, int i, int nb, const C2* v) {
      constexpr int R = decltype(rr)::r;
      const int k1 = r0 + 2 * c;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int q = k1 + N1 * (i + nb * j), at = q + half < N ? q + half : q + half - N;
        if (even) {
          *reinterpret_cast<float4*>(dst + at) = make_float4(v[j].re.x, v[j].im.x, v[j].re.y, v[j].im.y);
        } else {
          dst[at] = c2_lane0(v[j]);
          if (k1 + 1 < N1) dst[at + 1 < N ? at + 1 : 0] = c2_lane1(v[j]);
        }
      }
    });
  }
}

}  // namespace scd
