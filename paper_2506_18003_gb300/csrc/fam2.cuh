// FAM pair transform (K2, Eq. II.B-SCD_function_FAM), FP32 form, on the packed lanes, for the P of
// fam2_supported:
//     out[kh][lh][qh] = sum_p X[kh][p] conj(Y[lh][p]) W_P^{(q p) mod P}
// as one radix-2 split in time, P = 2 M, z(p) = X(p, k) conj(Y(p, l)):
//     E(f) = sum_n z(2 n) W_M^{n f},  O(f) = sum_n z(2 n + 1) W_M^{n f},
//     S(f) = E(f) + W_P^f O(f),       S(f + M) = E(f) - W_P^f O(f),
// the two M-point transforms in the two lanes of the packed instructions (fft2.cuh): they share every
// twiddle factor, a thread's loads are 16 bytes of each row, and the lanes meet only in the last
// step.  The pairs, the mirrored rows of the auto estimate (SYM) and the alpha-profile form (PROF) are
// fam_pairs_tile's (tiles.cuh).
//
// Bound: a transform reads two rows of X (L2) and writes two rows of S (8 P bytes each); GB300's L2 takes
// 6.3 TB/s of writes alone and 5.1-5.7 TB/s of each with as many reads.  So the kernel is persistent with
// its twiddle factors in shared memory, and issues 40% fewer instructions than the scalar transform.
// P = 1024, Np = 256: 104 us for 537 MB of estimates (5.2 TB/s), from 142; what bounds it now is the
// shared-memory pipe (77% of its cycles) with 16 warps per SM.
#pragma once
#include "fft2.cuh"
#include "pdl.cuh"
#include "tiles.cuh"

namespace scd {

struct FamSig {
  int64_t x, out;                                           // X (and Y) and S of a signal, elements of the arenas
};
struct FamArgs {
  const FamSig* sig;                                        // nullptr: one signal at offset 0
  const float2* X;
  const float2* Y;
  float2* out;
  float* prof;
  const float2* tw;                                         // pass table of the M-point pair transform
  const float2* wP;                                         // W_P^j
  int Np, nsig, PL, Q, power;                               // PL = P L, Q = P L / Np (profiles)
};

template <int PP>
struct FamPair {
  static constexpr int M = PP / 2, NT = 256;
  using PI = Plan2Info<M>;
  static constexpr int C = NT / PI::T;
  using F = PairFft<M, C, kConsecutive>;
  static constexpr int tw_off = F::smem_f4 * 16;
  static constexpr int smem = tw_off + PI::tw_len() * 8;
  // CTAs per SM: two at E = 16 (128 registers; three of 80 spill: P = 1024, Np = 256 111 -> 153 us)
  static constexpr int minb = PI::E >= 16 ? 2 : 4;
};

// v W_{2 RL}^j for a j that unrolling makes a constant
template <int RL>
__device__ __forceinline__ float2 turn_by(float2 v, int j) {
  switch (j) {
#define SCD_T(J) case J: return twc<2 * RL, (J < RL ? J : 0)>(v);
    SCD_T(1) SCD_T(2) SCD_T(3) SCD_T(4) SCD_T(5) SCD_T(6) SCD_T(7) SCD_T(8)
    SCD_T(9) SCD_T(10) SCD_T(11) SCD_T(12) SCD_T(13) SCD_T(14) SCD_T(15)
#undef SCD_T
    default: return v;
  }
}

template <int PP, bool SYM, bool PROF>
__device__ __forceinline__ void fam_pairs2_cta(unsigned char* sm, const FamArgs& A) {
  using K = FamPair<PP>;
  using PI = typename K::PI;
  constexpr int M = K::M, C = K::C, E = PI::E, T = PI::T, RL = PI::rl, B = E / RL;
  float2* tws = reinterpret_cast<float2*>(sm + K::tw_off);
  for (int e = threadIdx.x; e < PI::tw_len(); e += K::NT) tws[e] = __ldg(A.tw + e);
  const int c = K::F::in_c(), t = K::F::in_t(), Np = A.Np;
  float2 wb[B];                                             // W_P^{t + b T}
#pragma unroll
  for (int b = 0; b < B; ++b) wb[b] = __ldg(A.wP + t + b * T);
  const int npairs = (int)fam_pair_count<0>(Np, SYM), per = (npairs + C - 1) / C, tiles = per * A.nsig;
  wait_for_previous();
  __syncthreads();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (tile + (int)gridDim.x >= tiles) let_next_start();   // this CTA's last tile
    const int s = tile / per, pair = (tile - s * per) * C + c;
    const FamSig g = A.sig ? A.sig[s] : FamSig{0, 0};
    const bool valid = pair < npairs;
    int kh = 0, lh = 0;
    if (valid) {
      if constexpr (SYM) {
        const int r = pair / (Np + 1), k = pair - r * (Np + 1);
        if (k < Np - r) { kh = r; lh = r + k; }
        else { kh = Np - 1 - r; lh = k - 1; }
      } else {
        kh = pair / Np;
        lh = pair - kh * Np;
      }
    }
    const bool mirror = SYM && kh != lh;
    const float4* xk = reinterpret_cast<const float4*>(A.X + g.x + (int64_t)kh * PP) + t;
    const float4* yl = reinterpret_cast<const float4*>(A.Y + g.x + (int64_t)lh * PP) + t;
    C2 v[E];
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const float4 a = load_written(xk + r * (M / E)), b = load_written(yl + r * (M / E));
      v[r] = c2_pack(cmulc(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                     cmulc(make_float2(a.z, a.w), make_float2(b.z, b.w)));
    }
    auto free = [] { team_sync<T, false>(); };              // the next tile's first stores follow these reads
    if constexpr (PROF) {
      unsigned* pr = reinterpret_cast<unsigned*>(A.prof + g.out);
      auto put = [&](int f, float2 z) {
        const int q = ((f + M) & (PP - 1)) - M;
        const float m2 = fmaf(z.x, z.x, z.y * z.y);
        const unsigned val = __float_as_uint(A.power == 2 ? m2 : sqrtf(m2));
        if (valid && q >= -A.Q && q < A.Q) profile_max(pr + ((kh - lh) * A.Q + q + A.PL), val);
        if (mirror && -q >= -A.Q && -q < A.Q) profile_max(pr + ((lh - kh) * A.Q - q + A.PL), val);
      };
      auto dst = [&](int b, int j, int f, const C2& val) {
        const float2 e = c2_lane0(val), o = turn_by<RL>(cmul(c2_lane1(val), wb[b]), j);
        put(f, cadd(e, o));
        put(f + M, csub(e, o));
      };
      K::F::run(reinterpret_cast<float4*>(sm), tws, v, free, dst);
    } else {
      float2* o = A.out + g.out + ((int64_t)kh * Np + lh) * PP;
      float2* om = A.out + g.out + ((int64_t)lh * Np + kh) * PP;
      // bin f at (f + M) mod P, its mirror image at (M - f) mod P
      auto dst = [&](int b, int j, int f, const C2& val) {
        const float2 e = c2_lane0(val), w = turn_by<RL>(cmul(c2_lane1(val), wb[b]), j);
        const float2 z0 = cadd(e, w), z1 = csub(e, w);
        if (valid) {
          o[f + M] = z0;
          o[f] = z1;
        }
        if (mirror) {
          om[M - f] = cconj(z0);
          om[(PP - f) & (PP - 1)] = cconj(z1);
        }
      };
      K::F::run(reinterpret_cast<float4*>(sm), tws, v, free, dst);
    }
  }
}

// The sizes where it is the faster form (Np = 256 pair stage with its channeliser, scalar / this one): P = 32
// 24.7 / 14.4 us (a scalar transform of 32 points is one thread's), 512 cross 88 / 78 us (Np = 128 auto
// 33 / 24), 1024 auto 142 / 110, cross 164 / 171; at 64 18.5 / 20.6, 128 24.7 / 24.7, 256 34.9 / 50.6
// (its rows leave in runs of 64 bytes); at 2048 .. 8192 (Np = 128) 65 / 71, 128 / 132, 263 / 285 us:
// three passes of exchanges, as many as the scalar radix-32 plans, with half the threads per SM.
inline bool fam2_supported(int P, bool sym) { return P == 32 || P == 512 || (P == 1024 && sym); }
cudaError_t fam2_prepare(int P);
cudaError_t fam2_pairs(const FamArgs& A, int P, bool sym, bool prof, cudaStream_t st);   // X == Y if sym

}  // namespace scd
