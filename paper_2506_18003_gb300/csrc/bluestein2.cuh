// FAM pair transform for a P that is not a power of two (Bluestein's identity, bluestein.cuh), FP32 form,
// two pairs at a time in the lanes of the packed instructions (fft2.cuh), cyclic lengths M = 64 .. 4096:
//     z(p) c[p] -> FFT_M -> times Bh, conjugated -> FFT_M -> c[q] conj(.)
// Both transforms take the plan PlanSym<M>, whose last pass leaves a thread exactly the values that the
// second transform's first pass wants from it: the product with Bh happens in registers, and the
// shared-memory round trip between the transforms (two of eight with three passes each) is gone.  The
// chirp, Bh and every twiddle factor serve both lanes.  P <= M / 2, so the first pass of the first
// transform reads half of its inputs and skips the butterflies with the zero half, and the last bins
// from M / 2 on are not formed at all.
// Bound by instruction issue and the loads of chirp, Bh and the channel rows: at Np = 256, P = 1000
// (M = 2048) 178 M warp instructions at 0.46 of the issue slots, 16 warps per SM (128 registers; the
// one-pair form issued 296 M).  Microseconds per estimate, one-pair form / this one:
//   (Np, P) = (64, 20) 10.7 / 5.7, (64, 100) 10.7 / 7.6, (128, 200, cross) 60 / 35, (64, 333) 21.7 / 15.0,
//   (256, 500) 213 / 146, (256, 1000) 357 / 313, (32, 1999) 24.7 / 20.2, (128, 1999) 205 / 196.
// At M = 4096 the one-pair form stays where few pairs leave the packed form's last round short (bluestein.cu).
// M < 64 (P <= 16) and M > 4096 stay with the one-pair form: the first has too few values for a two-pass
// plan with equal ends, the second exceeds the 16 x 16 x 16 plan.
#pragma once
#include "fft2.cuh"
#include "pdl.cuh"
#include "tiles.cuh"

namespace scd {

template <int M>
struct FamAny2 {
  using PI = Plan2Info<M, PlanSym>;
  // 256 threads: within 2% of 128 at every M (the transforms synchronise by team, not by block)
  static constexpr int NT = PI::T > 256 ? PI::T : 256, C = NT / PI::T;
  using F = PairFft<M, C, kConsecutive, PlanSym>;
  static_assert(PI::rl == PI::r0 && PI::E == PI::rl, "the last pass's bins are the first pass's inputs");
  static constexpr int tw_off = F::smem_f4 * 16;
  static constexpr int smem = tw_off + PI::tw_len() * 8;
  static constexpr int minb = PI::E >= 16 ? 512 / NT : 1024 / NT;
};

// Persistent over the pairs two by two (their number is even).
template <int M, bool SYM>
__device__ __forceinline__ void fam_any2_cta(unsigned char* smem, const float2* __restrict__ X,
                                             const float2* __restrict__ Y, int Np, int P, float2* __restrict__ out,
                                             const float2* __restrict__ tw, const float2* __restrict__ chirp,
                                             const float2* __restrict__ bh) {
  using K = FamAny2<M>;
  using PI = typename K::PI;
  constexpr int C = K::C, E = PI::E, T = PI::T;
  float4* sm = reinterpret_cast<float4*>(smem);
  float2* tws = reinterpret_cast<float2*>(smem + K::tw_off);
  for (int e = threadIdx.x; e < PI::tw_len(); e += K::NT) tws[e] = __ldg(tw + e);
  const int c = K::F::in_c(), t = K::F::in_t(), half = P / 2;
  const int units = (int)(fam_pair_count<0>(Np, SYM) / 2), tiles = (units + C - 1) / C;
  wait_for_previous();
  __syncthreads();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (tile + (int)gridDim.x >= tiles) let_next_start();
    const int unit = tile * C + c;
    const bool valid = unit < units;
    int k0 = 0, l0 = 0, k1 = 0, l1 = 0;
    if (valid) {
      fam_pair_of<SYM>(2 * unit, Np, &k0, &l0);
      fam_pair_of<SYM>(2 * unit + 1, Np, &k1, &l1);
    }
    C2 v[E];
    {
      const float2 *a0 = X + (int64_t)k0 * P, *b0 = Y + (int64_t)l0 * P;
      const float2 *a1 = X + (int64_t)k1 * P, *b1 = Y + (int64_t)l1 * P;
      // P <= M / 2: the second half of the inputs is zero
#pragma unroll
      for (int r = 0; r < E / 2; ++r) {
        const int p = t + r * T;
        if (p < P)
          v[r] = cmul(c2_pack(cmulc(load_written(a0 + p), load_written(b0 + p)), cmulc(load_written(a1 + p), load_written(b1 + p))),
                      __ldg(chirp + p));
        else
          v[r] = C2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      }
    }
    auto free = [] { team_sync<T, false>(); };              // the next first pass's stores follow these reads
    K::F::template transform<true>(sm, tws, v, free);
#pragma unroll
    for (int j = 0; j < E; ++j) {                           // bin t + j T, input t + j T of the second transform
      v[j] = cmul(v[j], __ldg(bh + t + j * T));
      v[j].im = neg2(v[j].im);
    }
    float2 *o0 = out + ((int64_t)k0 * Np + l0) * P, *o1 = out + ((int64_t)k1 * Np + l1) * P;
    float2 *m0 = out + ((int64_t)l0 * Np + k0) * P, *m1 = out + ((int64_t)l1 * Np + k1) * P;
    const bool mirror0 = SYM && k0 != l0, mirror1 = SYM && k1 != l1;
    K::F::transform(sm, tws, v, free);
#pragma unroll
    for (int j = 0; j < E / 2; ++j) {                       // the bins f < P <= M / 2
      const int f = t + j * T;
      const C2 g = v[j];
      if (f < P && valid) {
        const float2 w = __ldg(chirp + f);                  // w conj(g), both lanes
        const C2 s{fma2(dup2(w.x), g.re, mul2(dup2(w.y), g.im)), fma2(dup2(w.y), g.re, neg2(mul2(dup2(w.x), g.im)))};
        const float2 s0 = c2_lane0(s), s1 = c2_lane1(s);
        const int q = f + half < P ? f + half : f + half - P;
        o0[q] = s0;
        o1[q] = s1;
        const int fm = f == 0 ? 0 : P - f, qm = fm + half < P ? fm + half : fm + half - P;
        if (mirror0) m0[qm] = cconj(s0);
        if (mirror1) m1[qm] = cconj(s1);
      }
    }
  }
}

}  // namespace scd
