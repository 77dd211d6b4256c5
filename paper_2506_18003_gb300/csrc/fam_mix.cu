// Plans and launches of the mixed-radix FAM pair transforms and SSCA strips (mix2.cuh).
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

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
__global__ void __launch_bounds__(kMixThreads, kMixCtas)
k_mix_cols(const __grid_constant__ MixPlan plan, const __grid_constant__ StripArgs A, const float2* __restrict__ in,
           float2* __restrict__ out, const float2* __restrict__ tw, const float2* __restrict__ wN,
           const float2* __restrict__ cols) {
  extern __shared__ __align__(128) unsigned char mix_sm[];
  mix_cols_cta(mix_sm, plan, A, in, out, tw, wN, cols);
}
__global__ void __launch_bounds__(kMixThreads, kMixCtas)
k_mix_rows(const __grid_constant__ MixPlan plan, const __grid_constant__ StripArgs A, const float2* __restrict__ in,
           float2* __restrict__ out, const float2* __restrict__ tw) {
  extern __shared__ __align__(128) unsigned char mix_sm[];
  mix_rows_cta(mix_sm, plan, A, in, out, tw);
}

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

bool mix_plan(int P, MixPlan* p) { return !is_pow2(P) && mix_factor(P, p); }

bool mix_factor(int P, MixPlan* p) {
  if (P <= 16 || P > 4096) return false;                       // 4096: one unit's values and twiddles in 113 KB
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
  p->unit = (p->r[0] * p->stride) | 1;                         // odd too, for interleaved transforms
  return true;
}

bool prepare_mix(int P, cudaError_t* err) {
  MixPlan plan;
  return !mix_plan(P, &plan) || table_mix(plan, err);
}

// Units per tile: as many as keep the block's threads busy in every pass, but not so many that the last
// wave of tiles is short of work.  The estimate of a tile's time is the rounds of butterflies per thread,
// weighted by the radix, and a constant for barriers and set-up.  The limit is half an SM's shared memory (two
// blocks): at 84 and 60 KB, with more L1 left, Np = 256, P = 1000 took 151 and 166 us instead of 146.
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

// ---------------------------------------------------------------- SSCA strips
// Lane pairs per tile: up to 16, so that a tile's rows are contiguous runs of 256 bytes.
static int strip_width(const MixPlan& p) {
  int lc = 4;
  while (lc > 0 && mix_smem(p, 1 << lc) > 112 * 1024) --lc;
  return lc;
}

// Both factors with a plan; the widest tiles, then the fewest passes, then the smallest radix sum.
static bool find_strip_plan(int64_t N, StripPlan* best) {
  int64_t score = -1;
  if (N > (int64_t)4096 * 4096 || N > INT32_MAX / 2) return false;
  for (int64_t d = 17; d <= 4096 && d <= N / 17; ++d) {
    StripPlan p;
    if (N % d || N / d > 4096 || !mix_factor((int)d, &p.a) || !mix_factor((int)(N / d), &p.b)) continue;
    p.N1 = (int)d;
    p.N2 = (int)(N / d);
    p.lca = strip_width(p.a);
    p.lcb = strip_width(p.b);
    int sum = 0;
    for (int s = 0; s < p.a.n; ++s) sum += p.a.r[s];
    for (int s = 0; s < p.b.n; ++s) sum += p.b.r[s];
    const int odd = N % 4 == 0 && (p.N1 % 2 || p.N2 % 2);      // 16-byte accesses in both passes if N allows them
    const int64_t v = ((int64_t)(p.lca < p.lcb ? p.lca : p.lcb) << 32) - ((int64_t)odd << 24) - ((p.a.n + p.b.n) << 16) - sum;
    if (score < 0 || v > score) { score = v; *best = p; }
  }
  return score >= 0;
}

// The splits of up to 64 lengths, also of those without one: the search takes 20 to 40 us, as long as a small
// estimate's launches, and a program may take several lengths in turn.  (A call asks three times: the
// thread's last answer first.)
bool strip_plan(int64_t N, StripPlan* plan) {
  constexpr size_t kMost = 64;
  static std::mutex mu;
  static std::map<int64_t, std::pair<bool, StripPlan>> kept;
  thread_local int64_t last = 0;
  thread_local std::pair<bool, StripPlan> mine;
  if (last != N) {
    bool known = false;
    {
      std::lock_guard<std::mutex> lock(mu);
      const auto it = kept.find(N);
      if ((known = it != kept.end())) mine = it->second;
    }
    if (!known) {
      mine.first = find_strip_plan(N, &mine.second);
      std::lock_guard<std::mutex> lock(mu);
      if (kept.size() >= kMost) kept.clear();
      kept[N] = mine;
    }
    last = N;
  }
  if (mine.first) *plan = mine.second;
  return mine.first;
}

bool prepare_strip(int64_t N, cudaError_t* err) {
  StripPlan plan;
  return !strip_plan(N, &plan) || (table_mix(plan.a, err) && table_mix(plan.b, err) && table_roots((int)N, err) &&
                                   table_cols((int)N, plan.N1, 2 << plan.lca, err));
}

cudaError_t strip_cols(const StripPlan& plan, int64_t N, int rows, const float2* in, int64_t ld, float2* out, int64_t ldo,
                       cudaStream_t st) {
  cudaError_t err;
  const int C = 1 << plan.lca;
  const float2* tw = table_mix(plan.a, &err);
  if (!tw) return err;
  const float2* wN = table_roots((int)N, &err);
  if (!wN) return err;
  const float2* cols = table_cols((int)N, plan.N1, 2 * C, &err);
  if (!cols) return err;
  const int sms = sm_count(&err);
  if (!sms) return err;
  if ((err = allow_smem<k_mix_cols>(113 * 1024)) != cudaSuccess) return err;
  StripArgs A{ld, ldo, plan.N1, plan.N2, (int)N, rows, plan.lca};
  const int64_t tiles = (int64_t)(((plan.N2 + 1) / 2 + C - 1) / C) * rows;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, kMixCtas * sms);
  return launch_dependent(true, k_mix_cols, grid, kMixThreads, mix_smem(plan.a, C), st, plan.a, A, in, out, tw, wN, cols);
}

cudaError_t strip_rows(const StripPlan& plan, int64_t N, int rows, const float2* in, int64_t ld, float2* out, int64_t ldo,
                       cudaStream_t st) {
  cudaError_t err;
  const int C = 1 << plan.lcb;
  const float2* tw = table_mix(plan.b, &err);
  if (!tw) return err;
  const int sms = sm_count(&err);
  if (!sms) return err;
  if ((err = allow_smem<k_mix_rows>(113 * 1024)) != cudaSuccess) return err;
  StripArgs A{ld, ldo, plan.N1, plan.N2, (int)N, rows, plan.lcb};
  const int64_t tiles = (int64_t)(((plan.N1 + 1) / 2 + C - 1) / C) * rows;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, kMixCtas * sms);
  return launch_dependent(true, k_mix_rows, grid, kMixThreads, mix_smem(plan.b, C), st, plan.b, A, in, out, tw);
}

}  // namespace scd
