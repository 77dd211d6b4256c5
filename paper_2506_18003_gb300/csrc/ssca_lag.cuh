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
//   rows  the M2-point transforms over m2 of each row of Y: R[m][c] = R_m(c), c = q1 + M1 q2;
//   chan  per frequency c the window and the Np-point transform over the lags, two neighbouring
//         frequencies to a lane pair, written to S[kh][(c - k N/Np + N/2) mod N]; or (alpha profiles)
//         the maxima over the channels of the two alpha columns c and c + N that frequency c feeds.
// rows and chan are persistent: a tile's inputs arrive by TMA in the area that the transform then uses
// for its exchanges, and the next tile's loads start as soon as this tile's last exchange is read, under
// the last radix pass and the stores.  Loads through registers instead need L1 lines for every load
// in flight, which the exchange areas of enough CTAs leave too few of (fft2.cuh's 16 bytes per value
// and thread: 64 KB per CTA of 256 threads).
// Y lies in the output's own memory (S is written last) or, for alpha profiles, in the workspace: beside R, or
// behind it in two groups of lag pairs.  Traffic: the intermediate (4 Np N bytes) out, in, out and in again,
// and S out: 3 x 8 Np N bytes, of which only S must reach HBM while the intermediate fits L2.
#pragma once
#include "fft2.cuh"
#include "pdl.cuh"
#include "tma.cuh"

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

// T = M / E threads of a size-M transform pair; threads and pairs of a CTA.
__host__ __device__ constexpr int lag_t(int M) { return M <= 32 ? 4 : (M <= 128 ? 8 : M / 16); }
__host__ __device__ constexpr int lag_strip_threads(int M) { return M >= 1024 ? 512 : 256; }
__host__ __device__ constexpr int lag_strip_c(int M) { return lag_strip_threads(M) / lag_t(M); }
__host__ __device__ constexpr int lag_up128(int v) { return (v + 127) / 128 * 128; }
__host__ __device__ constexpr int lag_max(int a, int b) { return a > b ? a : b; }
// CTAs of `smem` bytes that share an SM (227 KB, 1 KB of it the system's per CTA), at most by_regs
__host__ __device__ constexpr int lag_resident(int smem, int by_regs) {
  const int by_smem = 227 * 1024 / (smem + 1024);
  return by_smem < by_regs ? by_smem : by_regs;
}
// Large launches go out the ordinary way with at most 512 threads per SM, at Np = 256 in tiles of 256 threads:
// fewer tiles in flight leave the lines that several of them share in L2, and longer runs of S go to memory.
// Smaller ones gain more from early launch and full SMs.  Microseconds in the two forms, capped / full:
// estimates, line at 256 MB of S: 2^15 x 64, 8 signals (128 MB) 93 / 76, 17 (272 MB) 178 / 164; between 256 MB and
// 1 GB the short N favour the full form and the long ones the capped one, by up to 7% either way (2^15 x 64, 24
// signals 244 / 229; 2^18 x 256 360 / 369; 2^19 x 128 352 / 362); above, 2^18 x 128, 8 (2 GB) 1322 / 1460, 2^20 x 256
// (2 GB) 1443 / 1717.  Alpha profiles, which write the intermediate alone, half of S, line at 1 GB of it:
// 2^15 x 64, 17 windows (136 MB) 168 / 151; 2^16 x 256, 8 (512 MB) 576 / 549; 2^18 x 128, 8 (1 GB) 1237 / 1229; 512
// signals of 2^12 .. 2^18, Np = 128 (classes of up to 5 GB) 11.5 / 12.0 ms.
inline bool lag_large(int64_t N, int Np, int nsig, bool prof) {
  return prof ? 4 * N * Np * nsig > (int64_t(1) << 30) : 8 * N * Np * nsig > (int64_t(256) << 20);
}

// What the three passes of one launch share: nsig signals of one size N, signal s at the given offsets
// of the arenas (one signal: sig = nullptr, every offset 0).
struct LagSig {
  int64_t x, y, r, out;                                     // samples; Y, R, S complex64 (out: float in profiles)
};
struct LagArgs {
  const LagSig* sig;
  const float2* x;
  float2* Y;
  float2* R;
  float2* out;
  float* prof;
  const float* window;
  const float* gain;                                        // factor of the lag products, or nullptr (cols)
  const float2* tw;                                         // pass table of the pass's transform
  const float2* wN;
  unsigned* err;
  int N, M1, M2, nsig, Np, power, clear;                    // clear: the column pass zeroes the profiles
  int p0, np;                                               // lag pairs [p0, p0 + np) (cols, rows)
};
__device__ __forceinline__ LagSig lag_sig(const LagArgs& A, int s) {
  return A.sig ? A.sig[s] : LagSig{0, 0, 0, 0};
}

template <int M1>
struct LagCols {
  using PI = Plan2Info<M1>;
  static constexpr int NT = lag_strip_threads(M1), C = lag_strip_c(M1);
  using F = PairFft<M1, C, kInterleaved>;
  static_assert(C * PI::T == NT, "tile shape");
  static constexpr int stage_off = F::smem_f4 * 16;         // rotate factors of the last radix, [j][c]
  static constexpr int tw_off = stage_off + PI::rl * C * 8;
  static constexpr int smem = tw_off + PI::tw_len() * 8;
  static constexpr int minb = M1 >= 1024 ? 1 : (M1 >= 128 ? 2 : 4);
};
template <int M2>
struct LagRows {
  using PI = Plan2Info<M2>;
  static constexpr int NT = lag_strip_threads(M2), C = lag_strip_c(M2);
  using F = PairFft<M2, C, kRowsToCols>;
  static_assert(C * PI::T == NT, "tile shape");
  static constexpr int bytes = C * M2 * 16;                 // a tile's rows, contiguous in Y
  static constexpr int tw_off = lag_up128(lag_max(bytes, F::smem_f4 * 16));
  static constexpr int mbar_off = tw_off + PI::tw_len() * 8;
  static constexpr int smem = mbar_off + 16;
  // three of 256 threads (80 registers, at M2 = 512 44 bytes of spills: strip 50 -> 47 us at N = 2^16, Np = 256)
  static constexpr int minb = lag_resident(smem, NT > 256 ? 1 : (PI::E >= 16 ? 3 : 4));
};
// NTHR threads: 128, or 256 for the Np = 256 tiles of large outputs, whose runs of S then take 256 bytes
// rather than 128 (GB300 writes 2 GB in runs of 64 bytes at 2.5 TB/s, of 128 at 4.9, of 256 at 6.5).
template <int NP, int NTHR>
struct LagChan {
  using PI = Plan2Info<NP>;
  static constexpr int NT = NTHR, C = NTHR / lag_t(NP);
  using F = PairFft<NP, C, kInterleaved>;
  static_assert(C * PI::T == NT, "tile shape");
  // blocks of CB lane pairs with a per-tile factor each (`turn`): as many lane pairs as a 128-thread tile has, so
  // that a frequency's factors, and with them the estimate's bits, do not depend on the tile's width
  static constexpr int BLOCKS = NTHR / 128, CB = C / BLOCKS;
  static_assert(BLOCKS == 1 || BLOCKS * (NP / 2) == NT, "one thread per block and lag");
  // landing area: R_m of the tile's 2 C frequencies for the lags m < Np/2, and of the 2 C + 2 frequencies
  // from -(c0 + 2 C) for the lags 1 .. Np/2
  static constexpr int pos_row = 2 * C, neg_row = 2 * C + 2;
  static constexpr int neg_off = lag_up128(NP / 2 * pos_row * 8);
  static constexpr int bytes = NP / 2 * (pos_row + neg_row) * 8;
  static constexpr int step_off = lag_up128(lag_max(neg_off + NP / 2 * neg_row * 8, F::smem_f4 * 16));
  // W_N^{-d S0 i} of a lane pair's offsets d = 2 (c mod CB) and d + 1 at [i][c] (i < r0 / 2); a[Np/2 - l] W_N^{f l}
  // of each block's first frequency f, l = 1 .. Np/2; a[Np/2 ..]; the pass table
  static constexpr int turn_off = step_off + PI::r0 / 2 * C * 16;
  static constexpr int win_off = turn_off + BLOCKS * NP / 2 * 8;
  static constexpr int tw_off = win_off + NP / 2 * 4;
  static constexpr int mbar_off = tw_off + PI::tw_len() * 8;
  static constexpr int smem = mbar_off + 16;
  // registers without spills in the large launches (three of 256 threads spill 92 bytes: N = 2^20, Np = 256
  // 614 -> 795 us)
  static constexpr int minb = lag_resident(smem, PI::E >= 16 ? (NT > 128 ? 2 : 5) : 1024 / NT);
};

inline int lag_cols_tiles(int np, int M1, int M2) { return np * (M2 / lag_strip_c(M1)); }      // of one signal
inline int lag_rows_tiles(int np, int M1, int M2) { return np * (M1 / lag_strip_c(M2)); }

// base + off bytes: a base that is the same for the whole CTA and a 32-bit offset per thread address
// with one add (the intermediate and S of one signal stay below 4 GB).
template <class T>
__device__ __forceinline__ T* at_bytes(T* base, uint32_t off) {
  return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(base) + off);
}

// One CTA's tile of the column pass: lag pair p0 + tile / (M2 / C), columns m20 .. m20 + C - 1.
template <int M1>
__device__ __forceinline__ void lag_cols_tile(unsigned char* sm, const LagArgs& A, int tile) {
  using K = LagCols<M1>;
  using PI = typename K::PI;
  constexpr int C = K::C, E = PI::E, T = PI::T, p = M1 / PI::rl, B = E / PI::rl;
  const int N = A.N, M2 = A.M2, per = M2 / C, sig_tiles = A.np * per;
  const LagSig g = lag_sig(A, tile / sig_tiles);
  tile %= sig_tiles;
  const int pair = tile / per, m20 = (tile % per) * C;
  const int c = (int)threadIdx.x % C, t = (int)threadIdx.x / C;
  const int m2 = m20 + c, m = 2 * (A.p0 + pair);
  float2* stage = reinterpret_cast<float2*>(sm + K::stage_off);
  float2* tws = reinterpret_cast<float2*>(sm + K::tw_off);
  // rotate factor of bin f = i + p j: W_N^{m2 i} W_N^{m2 p j}, the second shared by the butterflies
  for (int e = threadIdx.x; e < PI::rl * C; e += K::NT) stage[e] = __ldg(A.wN + (m20 + e % C) * p * (e / C));
  for (int e = threadIdx.x; e < PI::tw_len(); e += K::NT) tws[e] = __ldg(A.tw + e);
  float2 rot[B];
#pragma unroll
  for (int b = 0; b < B; ++b) rot[b] = __ldg(A.wN + m2 * (t + b * T));
  wait_for_previous();
  const float gain = A.gain ? load_written(A.gain) : 1.f;   // (exact: a power of two)
  C2 v[E];
  const float2* xp = A.x + g.x + (t * M2 + m2);
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int n = r * (M1 / E) * M2;
    const float2 a = cscale(load_written(xp + n), gain);
    float2 b0, b1;
    if (r < E - 1) {                                        // n + m + 1 < N: the lags are far below N / E
      b0 = load_written(xp + n + m);
      b1 = load_written(xp + n + m + 1);
    } else {
      const int nn = n + t * M2 + m2 + m;
      b0 = nn < N ? load_written(xp + n + m) : make_float2(0.f, 0.f);
      b1 = nn + 1 < N ? load_written(xp + n + m + 1) : make_float2(0.f, 0.f);
    }
    v[r] = c2_pack(cmulc(b0, a), cmulc(b1, a));
  }
  float4* yo = reinterpret_cast<float4*>(A.Y + g.y) + (int64_t)pair * N;
  auto dst = [&](int b, int j, int f, const C2& val) {
    *at_bytes(yo, 16u * (uint32_t)(f * M2 + m2)) = c2_f4(cmul(val, cmul(rot[b], stage[j * C + c])));
  };
  K::F::run(reinterpret_cast<float4*>(sm), tws, v, [] { let_next_start(); }, dst);
  if (A.clear) {                                            // (here, where the values have left the registers)
    float* pr = A.prof + lag_sig(A, (int)blockIdx.x / sig_tiles).out;
    for (int i = tile * K::NT + (int)threadIdx.x; i < 2 * N; i += sig_tiles * K::NT) pr[i] = 0.f;
  }
}

// Row pass: persistent over the tiles of C rows (pair, q1).
template <int M2>
__device__ __forceinline__ void lag_rows_cta(unsigned char* sm, const LagArgs& A) {
  using K = LagRows<M2>;
  constexpr int E = K::PI::E, C = K::C;
  const int N = A.N, M1 = A.M1, per = M1 / C, sig_tiles = A.np * per, tiles = sig_tiles * A.nsig;
  float2* tws = reinterpret_cast<float2*>(sm + K::tw_off);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + K::mbar_off);
  auto issue = [&](int tile) {                              // thread 0
    const LagSig g = lag_sig(A, tile / sig_tiles);
    mbar_expect_tx(mbar, K::bytes);
    tma_load_bulk(sm, reinterpret_cast<const float4*>(A.Y + g.y) + (int64_t)(tile % sig_tiles) * (C * M2), K::bytes, mbar);
  };
  if (threadIdx.x == 0) {
    umma::mbar_init(mbar, 1);
    fence_mbar_init();
  }
  for (int e = threadIdx.x; e < K::PI::tw_len(); e += K::NT) tws[e] = __ldg(A.tw + e);
  wait_for_previous();
  __syncthreads();
  if (threadIdx.x == 0 && (int)blockIdx.x < tiles) issue(blockIdx.x);
  uint32_t phase = 0u;
  bool ok = true;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const bool got = umma::mbar_wait_bounded(mbar, phase, kMbarPollLimit);
    if (__syncthreads_or(!got)) { ok = false; break; }      // one decision for the whole CTA
    // this CTA's last tile (not before the wait: the channel pass reads the window before its own)
    if (tile + (int)gridDim.x >= tiles) let_next_start();
    phase ^= 1u;
    C2 v[E];
    {
      const float4* row = reinterpret_cast<const float4*>(sm) + K::F::in_c() * M2 + K::F::in_t();
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = take2(row + r * (M2 / E));
    }
    __syncthreads();                                        // the landing area becomes the exchange area
    const LagSig g = lag_sig(A, tile / sig_tiles);
    const int local = tile % sig_tiles, pair = A.p0 + local / per;
    float2* ro = A.R + g.r + (int64_t)(2 * pair) * N + (local % per) * C;
    const bool both = 2 * pair < A.Np / 2;                  // the last pair's second lag is not used
    const uint32_t co = 8u * (uint32_t)K::F::out_c();
    auto free = [&] {
      fence_before_tma();
      __syncthreads();                                      // every read of the area is done
      if (threadIdx.x == 0 && tile + (int)gridDim.x < tiles) issue(tile + gridDim.x);
    };
    auto dst = [&](int, int, int f, const C2& val) {
      const uint32_t off = 8u * (uint32_t)(f * M1) + co;
      *at_bytes(ro, off) = c2_lane0(val);
      if (both) *at_bytes(ro + N, off) = c2_lane1(val);
    };
    K::F::run(reinterpret_cast<float4*>(sm), tws, v, free, dst);
  }
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(A.err, 4u);
    umma::mbar_wait_bounded(mbar, phase, kMbarPollLimit);   // the copy in flight, if any
  }
  __syncthreads();
  if (threadIdx.x == 0) umma::mbar_inval(mbar);
}

// Channel pass: persistent over the tiles of 2 C frequencies c0 .. c0 + 2 C - 1; thread (c, t) holds the
// frequencies f0 = c0 + 2 c and f0 + 1.  tp / tn: R as [signal][lag][c], boxes of pos_row and neg_row
// frequencies by Np/2 lags.
template <int NP, int NTHR, bool PROF>
__device__ __forceinline__ void lag_chan_cta(unsigned char* sm, const LagArgs& A, const CUtensorMap* tp,
                                             const CUtensorMap* tn) {
  using K = LagChan<NP, NTHR>;
  using PI = typename K::PI;
  constexpr int C = K::C, E = PI::E, H = NP / 2, S0 = NP / PI::r0, RL = PI::rl, p = NP / RL;
  const int N = A.N, sig_tiles = N / (2 * C), tiles = sig_tiles * A.nsig;
  const int c = K::F::in_c(), t = K::F::in_t();
  float4* step = reinterpret_cast<float4*>(sm + K::step_off);
  float2* turn = reinterpret_cast<float2*>(sm + K::turn_off);
  float* win = reinterpret_cast<float*>(sm + K::win_off);
  float2* tws = reinterpret_cast<float2*>(sm + K::tw_off);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + K::mbar_off);
  // The factor of lag -l at frequency f + d, f the first of its block, is a[Np/2 - l] W_N^{f l} W_N^{d l}: the
  // first two are one value per lag and block (a thread of its own fetches the next tile's root under this
  // tile's last pass), the last is the same for every block, u W_N^{-d S0 i} for the thread's l = mh - i S0.  (One root gathered
  // per lag and frequency instead costs 24 scattered reads per lane pair: N = 2^20, Np = 256 1012 us.)
  constexpr int CB = K::CB;
  const int blk = K::BLOCKS > 1 ? (int)threadIdx.x / H : 0, lag = (int)threadIdx.x - blk * H + 1;
  const float alag = lag <= H ? __ldg(A.window + H - lag) : 0.f;
  // tiles from both ends in turn: tile b's mirrored frequencies are tile sig_tiles - 1 - b's, read while
  // they are still in L2
  auto c0_of = [&](int tile) {
    const int b = tile % sig_tiles;
    return (b & 1 ? sig_tiles - 1 - (b >> 1) : b >> 1) * (2 * C);
  };
  auto root = [&](int tile) { return __ldg(A.wN + (((c0_of(tile) + 2 * CB * blk) * lag) & (N - 1))); };
  const int mh = H - t;
  const int cb = K::BLOCKS > 1 ? c % CB : c;
  const C2 u = c2_pack(__ldg(A.wN + 2 * cb * mh), __ldg(A.wN + (2 * cb + 1) * mh));
  auto issue = [&](int tile) {                              // thread 0
    const int s = tile / sig_tiles, c0 = c0_of(tile);
    mbar_expect_tx(mbar, K::bytes);
    tma_load_3d(sm, tp, c0, 0, s, mbar);
    tma_load_3d(sm + K::neg_off, tn, N - c0 - 2 * C, 1, s, mbar);
  };
  if (threadIdx.x == 0) {
    umma::mbar_init(mbar, 1);
    fence_mbar_init();
  }
  for (int e = threadIdx.x; e < PI::tw_len(); e += K::NT) tws[e] = __ldg(A.tw + e);
  for (int e = threadIdx.x; e < H; e += K::NT) win[e] = __ldg(A.window + H + e);
  for (int e = threadIdx.x; e < E / 2 * C; e += K::NT) {
    const int d = 2 * (e % CB), l = S0 * (e / C);            // (C is a multiple of CB)
    const float2 s0 = __ldg(A.wN + ((-d * l) & (N - 1))), s1 = __ldg(A.wN + ((-(d + 1) * l) & (N - 1)));
    step[e] = make_float4(s0.x, s1.x, s0.y, s1.y);
  }
  wait_for_previous();
  __syncthreads();
  if (threadIdx.x == 0 && (int)blockIdx.x < tiles) issue(blockIdx.x);
  float2 next = lag <= H && (int)blockIdx.x < tiles ? root(blockIdx.x) : make_float2(0.f, 0.f);
  uint32_t phase = 0u;
  bool ok = true;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int c0 = c0_of(tile), f0 = c0 + 2 * c;
    const LagSig g = lag_sig(A, tile / sig_tiles);
    if (lag <= H) turn[blk * H + lag - 1] = cscale(next, alag);
    const bool got = umma::mbar_wait_bounded(mbar, phase, kMbarPollLimit);
    if (__syncthreads_or(!got)) { ok = false; break; }      // one decision for the whole CTA
    if (tile + (int)gridDim.x >= tiles) let_next_start();   // this CTA's last tile
    phase ^= 1u;
    C2 v[E];
    {                                                       // lags m = t + i S0 >= 0
      const float4* pos = reinterpret_cast<const float4*>(sm) + t * C + c;
#pragma unroll
      for (int i = 0; i < E / 2; ++i) {
        const C2 r = take2(pos + i * S0 * C);          // (re, im) of f0, of f0 + 1
        const float w = win[t + i * S0];
        v[i] = c2_pack(cscale(r.re, w), cscale(r.im, w));
      }
    }
    {                                                       // lags m - Np/2 < 0: W_N^{c |m|} conj(R_|m|(-c))
      const float2* neg = reinterpret_cast<const float2*>(sm + K::neg_off) + (mh - 1) * K::neg_row + 2 * (C - c);
      const bool wrap = f0 == 0;                            // -0 is frequency 0, not N
      const float2* r0p = A.R + g.r + (int64_t)mh * N;
      const float2* mine = turn + (K::BLOCKS > 1 ? c / CB * H : 0) + mh - 1;
#pragma unroll
      for (int i = 0; i < E / 2; ++i) {
        float2 r0 = neg[-i * S0 * K::neg_row];
        const float2 r1 = neg[-i * S0 * K::neg_row - 1];
        if (wrap) r0 = load_written(r0p - i * S0 * N);
        const C2 f = cmul(i ? cmul(u, take2(step + i * C + c)) : u, mine[-i * S0]);
        v[E / 2 + i] = c2_pack(cmulc(c2_lane0(f), r0), cmulc(c2_lane1(f), r1));
      }
    }
    __syncthreads();                                        // the landing area becomes the exchange area
    auto free = [&] {
      fence_before_tma();
      __syncthreads();                                      // every read of the area is done
      if (tile + (int)gridDim.x < tiles) {
        if (lag <= H) next = root(tile + gridDim.x);
        if (threadIdx.x == 0) issue(tile + gridDim.x);
      }
    };
    const int D = N / NP;
    if constexpr (PROF) {
      // S(k, q) with k D + q = c mod N (q in [-N/2, N/2)) lies on alpha column c + N if k D + q = c, on
      // column c if it is c - N
      // (maxima of the bits, as profile_max takes them: a NaN bin makes its column NaN, where fmaxf drops it)
      unsigned best[2][2] = {{0u, 0u}, {0u, 0u}};
      auto dst = [&](int, int, int f, const C2& val) {
        const int k = ((f + H) & (NP - 1)) - H;
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const float2 s = l ? c2_lane1(val) : c2_lane0(val);
          const unsigned m2 = __float_as_uint(fmaf(s.x, s.x, s.y * s.y));
          unsigned* b = best[l];                               // q = f0 + l - k D, less N if that is >= N/2
          if (f0 + l - k * D < N / 2) b[1] = max(b[1], m2);
          else b[0] = max(b[0], m2);
        }
      };
      K::F::run(reinterpret_cast<float4*>(sm), tws, v, free, dst);
      unsigned* pr = reinterpret_cast<unsigned*>(A.prof + g.out) + f0;
#pragma unroll
      for (int l = 0; l < 2; ++l)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          profile_max(pr + l + h * N, A.power == 2 ? best[l][h] : __float_as_uint(sqrtf(__uint_as_float(best[l][h]))));
    } else {
      // thread t's bin f = i + p j goes to channel kh = i + p ((j + RL / 2) mod RL), position
      // (f0 + N/2 - f D) mod N of its row (even, as are f0, N/2 and D)
      const uint32_t mask = 8u * (uint32_t)N - 8u;
      float2* o = A.out + g.out;
      auto dst = [&](int b, int j, int f, const C2& val) {
        const int i = t + b * PI::T;
        const uint32_t row = 8u * (uint32_t)(i * N), pos = 8u * (uint32_t)(f0 + N / 2 - i * D) - 8u * (uint32_t)(j * p * D);
        *reinterpret_cast<float4*>(at_bytes(o + (int64_t)(p * ((j + RL / 2) % RL)) * N, row + (pos & mask))) =
            make_float4(val.re.x, val.im.x, val.re.y, val.im.y);
      };
      K::F::run(reinterpret_cast<float4*>(sm), tws, v, free, dst);
    }
  }
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(A.err, 4u);
    umma::mbar_wait_bounded(mbar, phase, kMbarPollLimit);   // the copies in flight, if any
  }
  __syncthreads();
  if (threadIdx.x == 0) umma::mbar_inval(mbar);
}

// Host side (ssca_lag.cu): sets the kernels' attributes; enqueues one pass over A.nsig signals.
cudaError_t lag_prepare(int M1, int M2, int Np);
cudaError_t lag_cols(const LagArgs& A, cudaStream_t st);
cudaError_t lag_rows(const LagArgs& A, cudaStream_t st);
// R of signal s at A.R + r0 + s Np N
cudaError_t lag_chan(const LagArgs& A, int64_t r0, bool prof, cudaStream_t st);

}  // namespace scd
