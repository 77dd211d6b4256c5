// SSCA auto estimate in the lag domain (FP32 form, N a power of two).
//
// With x zero outside [0, N) the definition (Sec. II-C, Eq. Xg and Eq. II.B-SSCA_auto)
//     S(k, q) = sum_n conj(x[n]) W_N^{q n} sum_r a[r] x[n + r - Np/2] W_Np^{k (n + r - Np/2)}
// is a two-dimensional transform of the lag products p_m(n) = x[n + m] conj(x[n]), m = r - Np/2:
//     S(k, q) = sum_m a[m + Np/2] W_Np^{k m} R_m(q + k N/Np),     R_m(c) = sum_n p_m(n) W_N^{c n}
// (W_Np^{k n} = W_N^{(k N/Np) n}; c mod N).  Taking the long transforms first lets the conjugate
// symmetry of the lag products halve them: p_{-m}(n) = conj(p_m(n - m)), so
//     R_{-m}(c) = W_N^{c m} conj(R_m(-c)),
// and only the Np/2 + 1 lags m >= 0 are transformed (the channeliser order runs Np transforms of N
// points after N transforms of Np points).  The arithmetic falls by a third (N = 2^17, Np = 128: 24
// butterfly levels per output value to 15.5), the intermediate to half the size of the output.
// Rounding: the same number of butterfly levels in sequence as the channeliser order; the measured
// distance from the FP64 value (2-norm) is the same within 10% on every size.
//
// Three kernels, all on pairs of transforms in the packed lanes (fft2.cuh):
//   cols  the M1-point transforms over n = m1 M2 + m2 (m1 summed) of two neighbouring lags, lag
//         products formed on load, times the rotate factor W_N^{q1 m2}: Y[pair][q1][m2], 16 bytes per
//         lag pair;
//   rows  the M2-point transforms over m2, in place on each block of CB rows: R_m(c), c = q1 + M1 q2,
//         lag 2 p + s at [p][q1 / CB][s][q2][q1 mod CB] (8-byte values), so that the next pass reads
//         whole lines along q1;
//   chan  per frequency c the window and the Np-point transform over the lags, two frequencies to a lane
//         pair, written to S[kh][(c - k N/Np + N/2) mod N] in runs of CB values; or (alpha profiles) the
//         maxima over the channels of the two alpha columns c and c + N that frequency c feeds.
// Traffic: the intermediate (4 Np N bytes) out, back in place and in again, and S out: 2.5 x 8 Np N
// bytes, of which only S must reach HBM while the intermediate fits L2.
#pragma once
#include "fft2.cuh"
#include "tiles.cuh"

namespace scd {

// N = M1 M2 with M1 <= M2, both in 64..1024.
struct LagSplit {
  int M1, M2;
};
inline bool lag_split(int64_t N, LagSplit* s) {
  if (N < 4096 || N > (int64_t(1) << 20) || (N & (N - 1))) return false;
  int e = 0;
  while ((int64_t(1) << e) < N) ++e;
  s->M1 = 1 << (e / 2);
  s->M2 = 1 << ((e + 1) / 2);
  return true;
}
// lag pairs (2 p, 2 p + 1), p <= Np/4: the last one's second lag, Np/2 + 1, is not used
__host__ __device__ constexpr int lag_pairs(int Np) { return Np / 4 + 1; }

// T = M / E threads of a size-M transform pair; threads and pairs of a CTA.  128 threads where a
// tile of that size still has 8 neighbouring columns or rows: four independent CTAs per SM hide each
// other's load, exchange and store phases better than two of 256 (N = 2^16, Np = 256: 100 -> 93 us; three
// of 256 at 80 registers ran slower, 111 us: their exchange areas leave L1 too small for the loads in
// flight).
__host__ __device__ constexpr int lag_t(int M) { return M <= 32 ? 4 : (M <= 128 ? 8 : M / 16); }
__host__ __device__ constexpr int lag_strip_threads(int M) { return M >= 1024 ? 512 : (M >= 512 ? 256 : 128); }
__host__ __device__ constexpr int lag_strip_c(int M) { return lag_strip_threads(M) / lag_t(M); }
__host__ __device__ constexpr int lag_chan_threads(int Np) { return Np >= 256 ? 256 : 128; }
__host__ __device__ constexpr int lag_chan_c(int Np) { return lag_chan_threads(Np) / lag_t(Np); }
// CTAs per SM that the kernels' registers are held for
__host__ __device__ constexpr int lag_strip_minb(int M) { return M >= 1024 ? 1 : (M >= 512 ? 2 : (M >= 128 ? 4 : 8)); }
__host__ __device__ constexpr int lag_chan_minb(int Np) { return Np >= 256 ? 2 : (Np >= 128 ? 4 : 8); }
// log2 of CB, the rows of one block of R
constexpr int kLagLcb = 3;
inline int64_t lag_cols_tiles(int Np, int M1, int M2) { return (int64_t)lag_pairs(Np) * (M2 / lag_strip_c(M1)); }
inline int64_t lag_rows_tiles(int Np, int M1, int M2) { return (int64_t)lag_pairs(Np) * M1 / lag_strip_c(M2); }
inline int64_t lag_chan_tiles(int Np, int M1, int M2) { return (int64_t)M1 * M2 / (2 * lag_chan_c(Np)); }

template <int M1>
struct LagCols {
  using PI = Plan2Info<M1>;
  static constexpr int NT = lag_strip_threads(M1), C = lag_strip_c(M1);
  using F = PairFft<M1, C, kInterleaved>;
  static_assert(C * PI::T == NT, "tile shape");
  static constexpr int stage_off = F::smem_f4 * 16;         // rotate factors of the last radix, [j][c]
  static constexpr int smem = stage_off + PI::rl * C * 8;
};
template <int M2>
struct LagRows {
  using PI = Plan2Info<M2>;
  static constexpr int NT = lag_strip_threads(M2), C = lag_strip_c(M2);
  using F = PairFft<M2, C, kRowsToCols>;
  static_assert(C * PI::T == NT, "tile shape");
  static constexpr int smem = F::smem_f4 * 16;
};
template <int NP>
struct LagChan {
  using PI = Plan2Info<NP>;
  static constexpr int NT = lag_chan_threads(NP), C = lag_chan_c(NP);
  using F = PairFft<NP, C, kInterleaved>;
  static_assert(C * PI::T == NT, "tile shape");
  static constexpr int step_off = F::smem_f4 * 16;          // W_N^{-c S0 i}, [i][c]
  static constexpr int smem = step_off + PI::r0 / 2 * C * 16;
};

// base + off bytes: a base that is the same for the whole CTA and a 32-bit offset per thread address
// with one add (the intermediate and S of one estimate stay below 4 GB).
template <class T>
__device__ __forceinline__ T* at_bytes(T* base, uint32_t off) {
  return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(base) + off);
}

// Tile `tile` of the column pass: lag pair tile / (M2 / C), columns m20 .. m20 + C - 1.
template <int M1>
__device__ __forceinline__ void lag_cols_tile(unsigned char* sm, const float2* __restrict__ x, int N, int M2,
                                              const float2* __restrict__ tw, const float2* __restrict__ wN,
                                              float4* __restrict__ Y, int tile) {
  using K = LagCols<M1>;
  using PI = typename K::PI;
  constexpr int C = K::C, E = PI::E, T = PI::T, p = M1 / PI::rl, B = E / PI::rl;
  const int per = M2 / C;
  const int pair = tile / per, m20 = (tile % per) * C;
  const int c = (int)threadIdx.x % C, t = (int)threadIdx.x / C;
  const int m2 = m20 + c, m = 2 * pair;
  float2* stage = reinterpret_cast<float2*>(sm + K::stage_off);
  // rotate factor of bin f = i + p j: W_N^{m2 i} W_N^{m2 p j}, the second shared by the butterflies
  for (int e = threadIdx.x; e < PI::rl * C; e += K::NT) stage[e] = __ldg(wN + (m20 + e % C) * p * (e / C));
  float2 rot[B];
#pragma unroll
  for (int b = 0; b < B; ++b) rot[b] = __ldg(wN + m2 * (t + b * T));
  C2 v[E];
  const float2* xp = x + (t * M2 + m2);
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int n = r * (M1 / E) * M2;
    const float2 a = __ldg(xp + n);
    float2 b0, b1;
    if (r < E - 1) {                                        // n + m + 1 < N: the lags are far below N / E
      b0 = __ldg(xp + n + m);
      b1 = __ldg(xp + n + m + 1);
    } else {
      const int nn = n + t * M2 + m2 + m;
      b0 = nn < N ? __ldg(xp + n + m) : make_float2(0.f, 0.f);
      b1 = nn + 1 < N ? __ldg(xp + n + m + 1) : make_float2(0.f, 0.f);
    }
    v[r] = c2_pack(cmulc(b0, a), cmulc(b1, a));
  }
  float4* yo = Y + (int64_t)pair * N + m2;
  auto dst = [&](int b, int j, int f, const C2& val) {
    yo[(int64_t)f * M2] = c2_f4(cmul(val, cmul(rot[b], stage[j * C + c])));
  };
  K::F::run(reinterpret_cast<float4*>(sm), tw, v, dst);
}

// Tile `tile` of the row pass: rows (pair, q1) tile C .. tile C + C - 1, blocks of CB rows in place.
template <int M2>
__device__ __forceinline__ void lag_rows_tile(unsigned char* sm, float4* __restrict__ Y, const float2* __restrict__ tw,
                                              int tile) {
  using K = LagRows<M2>;
  constexpr int E = K::PI::E, CB = 1 << kLagLcb;
  const float4* row = Y + ((int64_t)tile * K::C + K::F::in_c()) * M2 + K::F::in_t();
  C2 v[E];
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = c2_from(row[r * (M2 / E)]);
  const int c = K::F::out_c();
  float2* ro = reinterpret_cast<float2*>(Y + ((int64_t)tile * K::C + (c & ~(CB - 1))) * M2) + (c & (CB - 1));
  // every row of the tile is in registers once the CTA barrier before the last pass is passed
  auto dst = [&](int, int, int f, const C2& val) {
    ro[f * CB] = c2_lane0(val);
    ro[(M2 + f) * CB] = c2_lane1(val);
  };
  K::F::run(reinterpret_cast<float4*>(sm), tw, v, dst);
}

// Tile `tile` of the channel pass: one block of CB rows q1 and 2 QP neighbouring q2 (QP = C / CB): C pairs
// of frequencies.  R: the row pass's output.  PROF: instead of storing S, frequency c's largest
// |S|^power over the channels is reduced into prof[c] and prof[c + N].
template <int NP, bool PROF>
__device__ __forceinline__ void lag_chan_tile(unsigned char* sm, const float2* __restrict__ R, int N, int M1, int M2,
                                              const float* __restrict__ a, const float2* __restrict__ tw,
                                              const float2* __restrict__ wN, float2* __restrict__ out, int tile,
                                              float* prof = nullptr, int power = 1) {
  using K = LagChan<NP>;
  using PI = typename K::PI;
  constexpr int C = K::C, E = PI::E, H = NP / 2, S0 = NP / PI::r0;
  static_assert(S0 % 2 == 0, "a thread's lags share their parity");
  const int c = (int)threadIdx.x % C, t = (int)threadIdx.x / C;
  constexpr int lcb = kLagLcb, CB = 1 << lcb, QP = C >> lcb;
  const int nq = M1 >> lcb;
  const int qb = tile % nq, q2b = (tile / nq) * 2 * QP;
  const int q1 = (qb << lcb) + (c & (CB - 1)), q2 = q2b + (c >> lcb);
  const int f0 = q1 + M1 * q2, df = M1 * QP;                // this thread's frequencies: f0 and f0 + df
  float4* step = reinterpret_cast<float4*>(sm + K::step_off);
  for (int e = threadIdx.x; e < E / 2 * C; e += K::NT) {
    const int ec = e % C, ei = e / C;
    const int ef = (qb << lcb) + (ec & (CB - 1)) + M1 * (q2b + (ec >> lcb));
    const float2 s0 = __ldg(wN + ((-ef * S0 * ei) & (N - 1))), s1 = __ldg(wN + ((-(ef + df) * S0 * ei) & (N - 1)));
    step[e] = make_float4(s0.x, s1.x, s0.y, s1.y);
  }
  C2 v[E];
  // lags m = t + i S0 >= 0: inputs i < E / 2
  {
    const uint32_t off = 8u * (uint32_t)((t >> 1) * 2 * N + ((2 * qb + (t & 1)) * M2 + q2) * CB + (c & (CB - 1)));
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const float2* ri = at_bytes(R + i * S0 * N, off);
      const float2 r0 = __ldg(ri), r1 = __ldg(ri + C);
      const float w = __ldg(a + H + t + i * S0);
      v[i] = c2_pack(cscale(r0, w), cscale(r1, w));
    }
  }
  __syncthreads();                                          // the steps are staged
  // lags m = t + i S0 - H < 0, i < E / 2: R_m(c) = W_N^{c |m|} conj(R_|m|(-c)), |m| = (H - t) - i S0
  {
    const int mh = H - t;
    const int qm = (M1 - q1) & (M1 - 1), z = q1 ? 1 : 0;
    // offsets from lag |m| - (E/2 - 1) S0, the smallest of the thread's
    const int base = (mh >> 1) * 2 * N - (E / 2 - 1) * S0 * N + (2 * (qm >> lcb) + (mh & 1)) * M2 * CB + (qm & (CB - 1));
    const uint32_t o0 = 8u * (uint32_t)(base + ((M2 - q2 - z) & (M2 - 1)) * CB);
    const uint32_t o1 = 8u * (uint32_t)(base + ((M2 - q2 - QP - z) & (M2 - 1)) * CB);
    const float2 u0 = __ldg(wN + ((f0 * mh) & (N - 1))), u1 = __ldg(wN + (((f0 + df) * mh) & (N - 1)));
    const C2 u = c2_pack(u0, u1);
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const float2* ri = R + (E / 2 - 1 - i) * S0 * N;
      const float2 r0 = __ldg(at_bytes(ri, o0)), r1 = __ldg(at_bytes(ri, o1));
      const float w = __ldg(a + t + i * S0);
      C2 f = i ? cmul(u, K::F::take(step + i * C + c)) : u;
      f.re = mul2(f.re, dup2(w));
      f.im = mul2(f.im, dup2(w));
      v[E / 2 + i] = c2_pack(cmulc(c2_lane0(f), r0), cmulc(c2_lane1(f), r1));
    }
  }
  if constexpr (PROF) {
    // S(k, q) with k D + q = c mod N (D = N / Np, q in [-N/2, N/2)) lies on alpha column c + N if
    // k D + q = c, on column c if it is c - N
    const int D = N / NP;
    float best[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    auto dst = [&](int, int, int f, const C2& val) {
      const int k = ((f + H) & (NP - 1)) - H;
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const float2 s = l ? c2_lane1(val) : c2_lane0(val);
        const float m2 = fmaf(s.x, s.x, s.y * s.y);
        const int q = f0 + l * df - k * D;                  // in [-N/2, 3N/2): q + N/2 - N if that is >= N/2
        float* b = best[l];
        if (q < N / 2) b[1] = fmaxf(b[1], m2);
        else b[0] = fmaxf(b[0], m2);
      }
    };
    K::F::run(reinterpret_cast<float4*>(sm), tw, v, dst);
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        profile_max(reinterpret_cast<unsigned*>(prof) + f0 + l * df + h * N,
                    __float_as_uint(power == 2 ? best[l][h] : sqrtf(best[l][h])));
  } else {
    // thread t's bin f = i + p j goes to channel kh = i + p ((j + RL / 2) mod RL), position
    // (f0 + N/2 - f D) mod N of its row
    constexpr int RL = PI::rl, p = NP / RL;
    const int D = N / NP, s0 = f0 + N / 2;
    const uint32_t mask = 8u * (uint32_t)N - 8u;
    auto dst = [&](int b, int j, int f, const C2& val) {
      float2* o = out + (int64_t)(p * ((j + RL / 2) % RL)) * N;
      const int i = t + b * PI::T;
      const uint32_t row = 8u * (uint32_t)(i * N), pos = 8u * (uint32_t)(s0 - i * D) - 8u * (uint32_t)(j * p * D);
      *at_bytes(o, row + (pos & mask)) = c2_lane0(val);
      *at_bytes(o, row + ((pos + 8u * (uint32_t)df) & mask)) = c2_lane1(val);
    };
    K::F::run(reinterpret_cast<float4*>(sm), tw, v, dst);
  }
}

}  // namespace scd
