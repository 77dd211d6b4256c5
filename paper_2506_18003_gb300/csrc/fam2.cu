// FAM pair transforms of fam2.cuh, for one signal or for the signals of one size of a batch plan.
#include "fam2.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace scd {
namespace {

template <int PP, bool SYM, bool PROF>
__global__ void __launch_bounds__(FamPair<PP>::NT, FamPair<PP>::minb) k_fam_pairs2(const FamArgs A) {
  extern __shared__ __align__(128) unsigned char fam_sm[];
  fam_pairs2_cta<PP, SYM, PROF>(fam_sm, A);
}

template <int PP>
cudaError_t prepare_t() {
  cudaError_t e = allow_smem<k_fam_pairs2<PP, true, false>>(FamPair<PP>::smem);
  if (e == cudaSuccess) e = allow_smem<k_fam_pairs2<PP, true, true>>(FamPair<PP>::smem);
  if (e == cudaSuccess) e = allow_smem<k_fam_pairs2<PP, false, false>>(FamPair<PP>::smem);
  return e;
}

template <int PP>
cudaError_t launch_t(const FamArgs& A, bool sym, bool prof, cudaStream_t st) {
  using K = FamPair<PP>;
  cudaError_t e;
  const int sms = sm_count(&e);
  if (!sms) return e;
  const int64_t tiles = (fam_pair_count<0>(A.Np, sym) + K::C - 1) / K::C * A.nsig;
  if (tiles >= (int64_t)0x7FFFFFFF) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)(tiles < (int64_t)K::minb * sms ? tiles : (int64_t)K::minb * sms);
  return launch_dependent(true, prof ? k_fam_pairs2<PP, true, true> : (sym ? k_fam_pairs2<PP, true, false> : k_fam_pairs2<PP, false, false>),
                          grid, K::NT, K::smem, st, A);
}

}  // namespace

#define SCD_FAM2(X) X(32) X(512) X(1024)
cudaError_t fam2_prepare(int P) {
  switch (P) {
#define SCD_X(PP) case PP: return prepare_t<PP>();
    SCD_FAM2(SCD_X)
#undef SCD_X
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t fam2_pairs(const FamArgs& A, int P, bool sym, bool prof, cudaStream_t st) {
  switch (P) {
#define SCD_X(PP) case PP: return launch_t<PP>(A, sym, prof, st);
    SCD_FAM2(SCD_X)
#undef SCD_X
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace scd
