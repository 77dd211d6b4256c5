// Launch of the mixed-radix FAM pair transforms (mix2.cuh).
#include <algorithm>

#include "internal.h"
#include "mix2.cuh"

namespace scd {

namespace {

constexpr int kRadices[] = {16, 15, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};

template <bool SYM>
__global__ void __launch_bounds__(kMixThreads, kMixCtas)
k_fam_mix(const __grid_constant__ MixPlan plan, int C, const float2* __restrict__ X, const float2* __restrict__ Y, int Np,
          float2* __restrict__ out, const float2* __restrict__ tw) {
  extern __shared__ __align__(128) unsigned char mix_sm[];
  fam_mix_cta<SYM>(mix_sm, plan, C, X, Y, Np, out, tw);
}

// (Radices of at most 12 for three blocks per SM at 80 registers: within 3% at Np = 256, P = 500 and 1000,
// slower where a further pass is needed: Np = 64, P = 1500 20.6 -> 26.6 us.)
// The non-increasing radices with the smallest sum whose product is P, n of them (0: none).
int best_radices(int P, int n, int from, int* r) {
  if (n == 0) return P == 1 ? 0 : -1;
  int best = -1, cand[4];
  for (int i = from; i < (int)(sizeof(kRadices) / sizeof(*kRadices)); ++i) {
    const int R = kRadices[i];
    if (P % R) continue;
    const int sum = best_radices(P / R, n - 1, i, cand + 1);
    if (sum < 0 || (best >= 0 && sum + R >= best)) continue;
    best = sum + R;
    cand[0] = R;
    for (int j = 0; j < n; ++j) r[j] = cand[j];
  }
  return best;
}

}  // namespace

bool mix_plan(int P, MixPlan* p) {
  if (P <= 16 || P > 4096 || is_pow2(P)) return false;         // 4096: one unit's values and twiddles in 113 KB
  p->n = 0;
  for (int n = 2; n <= 4 && !p->n; ++n)                        // as few passes as the radices allow
    if (best_radices(P, n, 0, p->r) > 0) p->n = n;
  if (!p->n) return false;
  p->P = P;
  p->len[0] = P;
  p->tw_len = 0;
  for (int s = 0; s < p->n; ++s) {
    p->len[s + 1] = p->len[s] / p->r[s];
    p->off[s] = p->tw_len;
    if (s + 1 < p->n) p->tw_len += p->len[s];
    p->per[s].set(P / p->r[s]);
    p->m[s].set(p->len[s + 1]);
  }
  p->r0.set(p->r[0]);
  p->r1.set(p->r[1]);
  p->stride = p->len[1] | 1;
  p->unit = p->r[0] * p->stride;
  return true;
}

bool prepare_mix(int P, cudaError_t* err) {
  MixPlan plan;
  return !mix_plan(P, &plan) || table_mix(plan, err);
}

// Units per tile: as many as keep the block's threads busy in every pass, but not so many that the last
// wave of tiles is short of work.  The estimate of a tile's time is the rounds of butterflies per thread,
// weighted by the radix, and a constant for barriers and set-up.  The limit is half an SM's shared memory (two
// blocks): at 84 and 60 KB, with more L1 left, Np = 256, P = 1000 takes 151 and 166 us instead of 146.
static int mix_units(const MixPlan& p, int64_t units, int slots) {
  int best = 1;
  double cost = 1e30;
  for (int C = 1; C <= kMixMaxUnits && mix_smem(p, C) <= 112 * 1024; ++C) {
    double t = 20;
    for (int s = 0; s < p.n; ++s) t += (double)((C * (p.P / p.r[s]) + kMixThreads - 1) / kMixThreads) * (p.r[s] + 6);
    const double total = t * (double)(((units + C - 1) / C + slots - 1) / slots);
    if (total < cost) { cost = total; best = C; }
  }
  return best;
}

cudaError_t fam_mix_pairs(const float2* X, const float2* Y, int Np, const MixPlan& plan, float2* out, cudaStream_t st) {
  cudaError_t err;
  const float2* tw = table_mix(plan, &err);
  if (!tw) return err;
  const int sms = sm_count(&err);
  if (!sms) return err;
  constexpr int kMost = 113 * 1024;
  if ((err = allow_smem<k_fam_mix<true>>(kMost)) != cudaSuccess || (err = allow_smem<k_fam_mix<false>>(kMost)) != cudaSuccess)
    return err;
  const bool sym = X == Y;                                     // the auto estimate: pairs kh <= lh
  const int64_t units = fam_pair_count<0>(Np, sym) / 2;
  const int C = mix_units(plan, units, kMixCtas * sms);
  const int64_t tiles = (units + C - 1) / C;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, kMixCtas * sms);
  count_launches(1);
  return launch_dependent(true, sym ? k_fam_mix<true> : k_fam_mix<false>, grid, kMixThreads, mix_smem(plan, C), st, plan, C,
                          X, Y, Np, out, tw);
}

}  // namespace scd
