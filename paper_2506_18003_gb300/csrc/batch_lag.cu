// Lag-domain SSCA (ssca_lag.cuh) over the signals of a batch plan, one launch per pass and group of
// signals of one size (staged schedule, batch_staged.cu): kinds 7 (cols, M = M1), 8 (rows, M = M2)
// and 9 (chan, M = Np; with an alpha-profile output the kernel that reduces into the profiles).
// One CTA runs one tile; task i covers the tiles [first_i, first_i + subtiles_i).
#include "batch_kernel.cuh"
#include "ssca_lag.cuh"

namespace scd {
namespace bk {
namespace {

template <int M1>
__global__ void __launch_bounds__(LagCols<M1>::NT, lag_strip_minb(M1))
k_st_lag_cols(BatchArgs A, const Task* __restrict__ tl, int nt) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  const int64_t tile = blockIdx.x;
  const Task& t = tl[find_task(tl, nt, tile)];
  lag_cols_tile<M1>(lag_sm, A.x + t.x_off, t.N, t.M2, t.tw, t.wN, reinterpret_cast<float4*>(A.ws + t.ws_off),
                    (int)(tile - t.first));
}

template <int M2>
__global__ void __launch_bounds__(LagRows<M2>::NT, lag_strip_minb(M2))
k_st_lag_rows(BatchArgs A, const Task* __restrict__ tl, int nt) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  const int64_t tile = blockIdx.x;
  const Task& t = tl[find_task(tl, nt, tile)];
  lag_rows_tile<M2>(lag_sm, reinterpret_cast<float4*>(A.ws + t.ws_off), t.tw, (int)(tile - t.first));
}

template <int NP, bool PROF>
__global__ void __launch_bounds__(LagChan<NP>::NT, lag_chan_minb(NP))
k_st_lag_chan(BatchArgs A, const Task* __restrict__ tl, int nt) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  const int64_t tile = blockIdx.x;
  const Task& t = tl[find_task(tl, nt, tile)];
  if constexpr (PROF)
    lag_chan_tile<NP, true>(lag_sm, A.ws + t.ws_off, t.N, t.M1, t.M2, A.window, t.tw, t.wN, nullptr,
                            (int)(tile - t.first), reinterpret_cast<float*>(A.out) + t.out_off, A.prof_power);
  else
    lag_chan_tile<NP, false>(lag_sm, A.ws + t.ws_off, t.N, t.M1, t.M2, A.window, t.tw, t.wN, A.out + t.out_off,
                             (int)(tile - t.first));
}

template <class K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <int M>
cudaError_t prep(int kind, int* smem) {
  if constexpr (M >= 64) {
    if (kind == 7) return set_smem(k_st_lag_cols<M>, *smem = LagCols<M>::smem);
    if (kind == 8) return set_smem(k_st_lag_rows<M>, *smem = LagRows<M>::smem);
  }
  if constexpr (M <= 256) {
    if (kind == 9) {
      const cudaError_t e = set_smem(k_st_lag_chan<M, true>, *smem = LagChan<M>::smem);
      return e != cudaSuccess ? e : set_smem(k_st_lag_chan<M, false>, *smem);
    }
  }
  return cudaErrorInvalidValue;
}

template <int M>
cudaError_t launch(int kind, int grid, int smem, const BatchArgs& A, const Task* tl, int nt, cudaStream_t st) {
  if constexpr (M >= 64) {
    if (kind == 7) {
      k_st_lag_cols<M><<<grid, LagCols<M>::NT, smem, st>>>(A, tl, nt);
      return cudaGetLastError();
    }
    if (kind == 8) {
      k_st_lag_rows<M><<<grid, LagRows<M>::NT, smem, st>>>(A, tl, nt);
      return cudaGetLastError();
    }
  }
  if constexpr (M <= 256) {
    if (kind == 9) {
      if (A.prof_power) k_st_lag_chan<M, true><<<grid, LagChan<M>::NT, smem, st>>>(A, tl, nt);
      else k_st_lag_chan<M, false><<<grid, LagChan<M>::NT, smem, st>>>(A, tl, nt);
      return cudaGetLastError();
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t lag_prepare(int kind, int M, int* smem) {
  switch (M) {
#define SCD_LP(MV) case MV: return prep<MV>(kind, smem);
    SCD_LP(16) SCD_LP(32) SCD_LP(64) SCD_LP(128) SCD_LP(256) SCD_LP(512) SCD_LP(1024)
#undef SCD_LP
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t lag_launch(int kind, int M, int grid, int smem, const BatchArgs& A, const Task* tl, int nt,
                       cudaStream_t st) {
  switch (M) {
#define SCD_LL(MV) case MV: return launch<MV>(kind, grid, smem, A, tl, nt, st);
    SCD_LL(16) SCD_LL(32) SCD_LL(64) SCD_LL(128) SCD_LL(256) SCD_LL(512) SCD_LL(1024)
#undef SCD_LL
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bk
}  // namespace scd
