// SSCA auto estimates in the lag domain, single estimates: the three passes of ssca_lag.cuh, one
// kernel each.
#include "internal.h"
#include "ssca_lag.cuh"

namespace scd {
namespace {

template <int M1>
__global__ void __launch_bounds__(LagCols<M1>::NT, lag_strip_minb(M1))
k_lag_cols(const float2* __restrict__ x, int N, int M2, const float2* __restrict__ tw, const float2* __restrict__ wN,
           float4* __restrict__ Y) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_cols_tile<M1>(lag_sm, x, N, M2, tw, wN, Y, (int)blockIdx.x);
}

template <int M2>
__global__ void __launch_bounds__(LagRows<M2>::NT, lag_strip_minb(M2))
k_lag_rows(float4* __restrict__ Y, const float2* __restrict__ tw) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_rows_tile<M2>(lag_sm, Y, tw, (int)blockIdx.x);
}

template <int NP>
__global__ void __launch_bounds__(LagChan<NP>::NT, lag_chan_minb(NP))
k_lag_chan(const float2* __restrict__ R, int N, int M1, int M2, const float* __restrict__ a,
           const float2* __restrict__ tw, const float2* __restrict__ wN, float2* __restrict__ out) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_chan_tile<NP, false>(lag_sm, R, N, M1, M2, a, tw, wN, out, (int)blockIdx.x);
}

template <class K>
cudaError_t set_smem(K kernel, int bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <int M1>
cudaError_t launch_cols(const float2* x, int N, int Np, int M2, const float2* wN, float4* Y, cudaStream_t st) {
  cudaError_t e;
  const float2* tw = table_pass2(M1, &e);
  if (!tw || (e = set_smem(k_lag_cols<M1>, LagCols<M1>::smem)) != cudaSuccess) return e;
  k_lag_cols<M1><<<(unsigned)lag_cols_tiles(Np, M1, M2), LagCols<M1>::NT, LagCols<M1>::smem, st>>>(x, N, M2, tw, wN, Y);
  return cudaGetLastError();
}

template <int M2>
cudaError_t launch_rows(int Np, int M1, float4* Y, cudaStream_t st) {
  cudaError_t e;
  const float2* tw = table_pass2(M2, &e);
  if (!tw || (e = set_smem(k_lag_rows<M2>, LagRows<M2>::smem)) != cudaSuccess) return e;
  k_lag_rows<M2><<<(unsigned)lag_rows_tiles(Np, M1, M2), LagRows<M2>::NT, LagRows<M2>::smem, st>>>(Y, tw);
  return cudaGetLastError();
}

template <int NP>
cudaError_t launch_chan(const float2* R, int N, int M1, int M2, const float* a, const float2* wN, float2* out,
                        cudaStream_t st) {
  cudaError_t e;
  const float2* tw = table_pass2(NP, &e);
  if (!tw || (e = set_smem(k_lag_chan<NP>, LagChan<NP>::smem)) != cudaSuccess) return e;
  k_lag_chan<NP><<<(unsigned)lag_chan_tiles(NP, M1, M2), LagChan<NP>::NT, LagChan<NP>::smem, st>>>(R, N, M1, M2, a, tw,
                                                                                                 wN, out);
  return cudaGetLastError();
}

}  // namespace

bool ssca_lag_tables(int64_t N, int Np, cudaError_t* err) {
  LagSplit s;
  if (!lag_split(N, &s)) { *err = cudaErrorInvalidValue; return false; }
  return table_pass2(s.M1, err) && table_pass2(s.M2, err) && table_pass2(Np, err) && table_roots((int)N, err);
}

cudaError_t ssca_lag_cols(const float2* x, int64_t N, int Np, float2* ws, cudaStream_t st) {
  LagSplit s;
  if (!lag_split(N, &s)) return cudaErrorInvalidValue;
  cudaError_t e;
  const float2* wN = table_roots((int)N, &e);
  if (!wN) return e;
  count_launches(1);
  switch (s.M1) {
#define SCD_LC(M) case M: return launch_cols<M>(x, (int)N, Np, s.M2, wN, (float4*)ws, st);
    SCD_LC(64) SCD_LC(128) SCD_LC(256) SCD_LC(512) SCD_LC(1024)
#undef SCD_LC
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t ssca_lag_rows(int64_t N, int Np, float2* ws, cudaStream_t st) {
  LagSplit s;
  if (!lag_split(N, &s)) return cudaErrorInvalidValue;
  count_launches(1);
  switch (s.M2) {
#define SCD_LR(M) case M: return launch_rows<M>(Np, s.M1, (float4*)ws, st);
    SCD_LR(64) SCD_LR(128) SCD_LR(256) SCD_LR(512) SCD_LR(1024)
#undef SCD_LR
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t ssca_lag_chan(const float2* ws, int64_t N, int Np, const float* window, float2* out, cudaStream_t st) {
  LagSplit s;
  if (!lag_split(N, &s)) return cudaErrorInvalidValue;
  cudaError_t e;
  const float2* wN = table_roots((int)N, &e);
  if (!wN) return e;
  count_launches(1);
  switch (Np) {
#define SCD_LN(M) case M: return launch_chan<M>(ws, (int)N, s.M1, s.M2, window, wN, out, st);
    SCD_LN(16) SCD_LN(32) SCD_LN(64) SCD_LN(128) SCD_LN(256)
#undef SCD_LN
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace scd
