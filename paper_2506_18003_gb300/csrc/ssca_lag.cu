// SSCA auto estimates in the lag domain: the kernels of ssca_lag.cuh's three passes, for one signal or
// for the signals of one size of a batch plan.
#include "internal.h"
#include "pdl.cuh"
#include "ssca_lag.cuh"

namespace scd {
namespace {

template <int M1>
__global__ void __launch_bounds__(LagCols<M1>::NT, LagCols<M1>::minb) k_lag_cols(const LagArgs A) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_cols_tile<M1>(lag_sm, A, (int)blockIdx.x);
}
template <int M2>
__global__ void __launch_bounds__(LagRows<M2>::NT, LagRows<M2>::minb) k_lag_rows(const LagArgs A) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_rows_cta<M2>(lag_sm, A);
}
template <int NP, int NTHR, bool PROF>
__global__ void __launch_bounds__(NTHR, LagChan<NP, NTHR>::minb)
k_lag_chan(const LagArgs A, const __grid_constant__ CUtensorMap tp, const __grid_constant__ CUtensorMap tn) {
  extern __shared__ __align__(128) unsigned char lag_sm[];
  lag_chan_cta<NP, NTHR, PROF>(lag_sm, A, &tp, &tn);
}

bool large(const LagArgs& A) { return lag_large(A.N, A.Np, A.nsig, A.power != 0); }

// persistent CTAs of a launch over `tiles` tiles: per_sm of nt threads on every SM, of a large launch at
// most 512 threads
cudaError_t grid_of(const LagArgs& A, int64_t tiles, int per_sm, int nt, unsigned* grid) {
  if (large(A) && per_sm * nt > 512) per_sm = 512 / nt;
  cudaError_t e;
  const int sms = sm_count(&e);
  if (!sms) return e;
  *grid = (unsigned)(tiles < (int64_t)per_sm * sms ? tiles : (int64_t)per_sm * sms);
  return cudaSuccess;
}

#define SCD_LAG_STRIP(X) X(64) X(128) X(256) X(512) X(1024)

template <int M1>
cudaError_t launch_cols(const LagArgs& A, cudaStream_t st) {
  const int64_t tiles = (int64_t)lag_cols_tiles(A.np, M1, A.M2) * A.nsig;
  if (tiles >= (int64_t)0x7FFFFFFF) return cudaErrorInvalidValue;
  return launch_dependent(!large(A), k_lag_cols<M1>, (unsigned)tiles, LagCols<M1>::NT, LagCols<M1>::smem, st, A);
}

template <int M2>
cudaError_t launch_rows(const LagArgs& A, cudaStream_t st) {
  using K = LagRows<M2>;
  const int64_t tiles = (int64_t)lag_rows_tiles(A.np, A.M1, M2) * A.nsig;
  if (tiles >= (int64_t)0x7FFFFFFF) return cudaErrorInvalidValue;
  unsigned grid;
  cudaError_t e = grid_of(A, tiles, K::minb, K::NT, &grid);
  if (e != cudaSuccess) return e;
  return launch_dependent(!large(A), k_lag_rows<M2>, grid, K::NT, K::smem, st, A);
}

template <int NP, int NTHR>
cudaError_t launch_chan(const LagArgs& A, int64_t r0, bool prof, cudaStream_t st) {
  using K = LagChan<NP, NTHR>;
  const int64_t tiles = (int64_t)(A.N / (2 * K::C)) * A.nsig;
  if (tiles >= (int64_t)0x7FFFFFFF) return cudaErrorInvalidValue;
  unsigned grid;
  cudaError_t e = grid_of(A, tiles, K::minb, K::NT, &grid);
  if (e != cudaSuccess) return e;
  CUtensorMap tp, tn;                                       // R as [signal][lag][c]
  const cuuint64_t dims[3] = {(cuuint64_t)A.N, NP / 2 + 1, (cuuint64_t)A.nsig};
  const cuuint64_t strides[2] = {(cuuint64_t)A.N * 8, (cuuint64_t)A.N * NP * 8};
  const cuuint32_t bp[3] = {K::pos_row, NP / 2, 1}, bn[3] = {K::neg_row, NP / 2, 1};
  if ((e = encode_map_c64(&tp, A.R + r0, 3, dims, strides, bp)) != cudaSuccess) return e;
  if ((e = encode_map_c64(&tn, A.R + r0, 3, dims, strides, bn)) != cudaSuccess) return e;
  return prof ? launch_dependent(!large(A), k_lag_chan<NP, NTHR, true>, grid, K::NT, K::smem, st, A, tp, tn)
              : launch_dependent(!large(A), k_lag_chan<NP, NTHR, false>, grid, K::NT, K::smem, st, A, tp, tn);
}

}  // namespace

cudaError_t lag_prepare(int M1, int M2, int Np) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (M1) {
#define SCD_X(M) case M: e = allow_smem<k_lag_cols<M>>(LagCols<M>::smem); break;
    SCD_LAG_STRIP(SCD_X)
#undef SCD_X
  }
  if (e != cudaSuccess) return e;
  e = cudaErrorInvalidValue;
  switch (M2) {
#define SCD_X(M) case M: e = allow_smem<k_lag_rows<M>>(LagRows<M>::smem); break;
    SCD_LAG_STRIP(SCD_X)
#undef SCD_X
  }
  if (e != cudaSuccess) return e;
  e = cudaErrorInvalidValue;
  switch (Np) {
#define SCD_X(M, T)                                                                                \
  if (e == cudaSuccess) e = allow_smem<k_lag_chan<M, T, false>>(LagChan<M, T>::smem);               \
  if (e == cudaSuccess) e = allow_smem<k_lag_chan<M, T, true>>(LagChan<M, T>::smem);
    case 16: e = cudaSuccess; SCD_X(16, 128) break;
    case 32: e = cudaSuccess; SCD_X(32, 128) break;
    case 64: e = cudaSuccess; SCD_X(64, 128) break;
    case 128: e = cudaSuccess; SCD_X(128, 128) break;
    case 256: e = cudaSuccess; SCD_X(256, 128) SCD_X(256, 256) break;
#undef SCD_X
  }
  return e;
}

cudaError_t lag_cols(const LagArgs& A, cudaStream_t st) {
  switch (A.M1) {
#define SCD_X(M) case M: return launch_cols<M>(A, st);
    SCD_LAG_STRIP(SCD_X)
#undef SCD_X
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t lag_rows(const LagArgs& A, cudaStream_t st) {
  switch (A.M2) {
#define SCD_X(M) case M: return launch_rows<M>(A, st);
    SCD_LAG_STRIP(SCD_X)
#undef SCD_X
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t lag_chan(const LagArgs& A, int64_t r0, bool prof, cudaStream_t st) {
  switch (A.Np) {
    case 16: return launch_chan<16, 128>(A, r0, prof, st);
    case 32: return launch_chan<32, 128>(A, r0, prof, st);
    case 64: return launch_chan<64, 128>(A, r0, prof, st);
    case 128: return launch_chan<128, 128>(A, r0, prof, st);
    case 256:
      return large(A) ? launch_chan<256, 256>(A, r0, prof, st) : launch_chan<256, 128>(A, r0, prof, st);
    default: return cudaErrorInvalidValue;
  }
}

bool ssca_lag_tables(int64_t N, int Np, cudaError_t* err) {
  LagSplit s;
  if (!lag_split(N, &s)) { *err = cudaErrorInvalidValue; return false; }
  return table_pass2(s.M1, err) && table_pass2(s.M2, err) && table_pass2(Np, err) && table_roots((int)N, err) &&
         device_error_word(err);
}

// One signal: Y in the output's memory, R in the workspace.
cudaError_t ssca_lag(const float2* x, const float* gain, int64_t N, int Np, const float* window, float2* ws, float2* out,
                     cudaStream_t st, cudaError_t (*between)(void*, int), void* ctx) {
  LagSplit s;
  if (!lag_split(N, &s)) return cudaErrorInvalidValue;
  LagArgs A{};
  A.x = x; A.gain = gain; A.Y = out; A.R = ws; A.out = out; A.window = window;
  A.N = (int)N; A.M1 = s.M1; A.M2 = s.M2; A.nsig = 1; A.Np = Np; A.np = lag_pairs(Np);
  cudaError_t e;
  const float2 *tw1, *tw2, *twc;
  if (!(A.wN = table_roots((int)N, &e)) || !(A.err = device_error_word(&e)) || !(tw1 = table_pass2(s.M1, &e)) ||
      !(tw2 = table_pass2(s.M2, &e)) || !(twc = table_pass2(Np, &e)) || (e = lag_prepare(s.M1, s.M2, Np)) != cudaSuccess)
    return e;
  count_launches(3);
  A.tw = tw1;
  if ((e = lag_cols(A, st)) != cudaSuccess || (e = between(ctx, 0)) != cudaSuccess) return e;
  A.tw = tw2;
  if ((e = lag_rows(A, st)) != cudaSuccess || (e = between(ctx, 1)) != cudaSuccess) return e;
  A.tw = twc;
  return lag_chan(A, 0, false, st);
}

}  // namespace scd
