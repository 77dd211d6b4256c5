// Paired power-of-two FFT building blocks: two independent transforms per thread team, carried in
// the two lanes of the packed FP32 instructions (add / sub / mul / fma .rn.f32x2).
//
// A C2 holds one element of both transforms: (re of lane x, re of lane y), (im of lane x, im of
// lane y).  Every butterfly then is a sequence of packed instructions with no lane crossing, and a
// twiddle factor that both transforms share is a broadcast operand, so one issued instruction does
// the work of two: on GB300 a packed instruction takes the FP32 pipe for two cycles but one issue
// slot (measured: 64 lane pairs per SM and clock for add, mul and fma .f32x2, as many as scalar
// pairs, with an independent integer instruction issued beside each for free; negations, broadcasts
// and constants fold into the operands, only exchanging lanes costs moves).  The scalar transforms
// of fft.cuh issue about 150 instructions per SSCA output point at 45-60% of the issue slots; these
// kernels are bound by their issue slots and latencies, not by the FP32 pipe.  Shared-memory
// exchanges move 16 bytes per access.  Each lane's arithmetic is the scalar one of fft.cuh,
// rounding by rounding.
#pragma once
#include "fft.cuh"

namespace scd {

struct C2 {
  float2 re, im;
};

#if defined(__CUDA_ARCH__)
#define SCD_F32X2_BINOP(NAME, OP)                                                                      \
  __device__ __forceinline__ float2 NAME(float2 a, float2 b) {                                         \
    unsigned long long r;                                                                              \
    asm(OP ".rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));                      \
    return f2_from(r);                                                                                 \
  }
SCD_F32X2_BINOP(add2, "add")
SCD_F32X2_BINOP(sub2, "sub")
SCD_F32X2_BINOP(mul2, "mul")
#undef SCD_F32X2_BINOP
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return f2_from(r);
}
#else
__host__ __device__ inline float2 add2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ inline float2 sub2(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__host__ __device__ inline float2 mul2(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
__host__ __device__ inline float2 fma2(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
#endif
__host__ __device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__host__ __device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

__host__ __device__ __forceinline__ C2 cadd(C2 a, C2 b) { return C2{add2(a.re, b.re), add2(a.im, b.im)}; }
__host__ __device__ __forceinline__ C2 csub(C2 a, C2 b) { return C2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// both lanes times the same factor w
__host__ __device__ __forceinline__ C2 cmul(C2 a, float2 w) {
  return C2{fma2(a.re, dup2(w.x), neg2(mul2(a.im, dup2(w.y)))), fma2(a.re, dup2(w.y), mul2(a.im, dup2(w.x)))};
}
// lane by lane
__host__ __device__ __forceinline__ C2 cmul(C2 a, C2 w) {
  return C2{fma2(a.re, w.re, neg2(mul2(a.im, w.im))), fma2(a.re, w.im, mul2(a.im, w.re))};
}
__host__ __device__ __forceinline__ C2 c2_pack(float2 a, float2 b) {
  return C2{make_float2(a.x, b.x), make_float2(a.y, b.y)};
}
__host__ __device__ __forceinline__ float2 c2_lane0(const C2& v) { return make_float2(v.re.x, v.im.x); }
__host__ __device__ __forceinline__ float2 c2_lane1(const C2& v) { return make_float2(v.re.y, v.im.y); }
__host__ __device__ __forceinline__ float4 c2_f4(const C2& v) { return make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }
__host__ __device__ __forceinline__ C2 c2_from(float4 q) {
  return C2{make_float2(q.x, q.y), make_float2(q.z, q.w)};
}

// One 16-byte load: from plain C++ the compiler makes two 8-byte ones, each of which then walks the
// 16-byte elements at half the bank bandwidth.
__device__ __forceinline__ C2 take2(const float4* p) {
#if defined(__CUDA_ARCH__)
  unsigned long long re, im;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(re), "=l"(im) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
  return C2{f2_from(re), f2_from(im)};
#else
  return c2_from(*p);
#endif
}

// ----------------------------------------------------------------------------- radix plans
// As Plan (fft.cuh) with radices of at most 16: a thread holds E = r0 element pairs, 4 E registers.
template <int M> struct Plan2;
#define SCD_PLAN2(M, N, R0, R1, R2) \
  template <> struct Plan2<M> { static constexpr int n = N; static constexpr int r[3] = {R0, R1, R2}; };
SCD_PLAN2(16, 2, 4, 4, 0)
SCD_PLAN2(32, 2, 8, 4, 0)
SCD_PLAN2(64, 2, 8, 8, 0)
SCD_PLAN2(128, 2, 16, 8, 0)
SCD_PLAN2(256, 2, 16, 16, 0)
SCD_PLAN2(512, 3, 16, 8, 4)
SCD_PLAN2(1024, 3, 16, 8, 8)
#undef SCD_PLAN2
// Plans whose last radix is the first: the bins that a thread gets from the last pass are the inputs that
// the first pass of another transform of the size takes from it (any-length transforms, bluestein2.cuh).
template <int M> struct PlanSym;
#define SCD_PLAN_SYM(M, N, R0, R1, R2) \
  template <> struct PlanSym<M> { static constexpr int n = N; static constexpr int r[3] = {R0, R1, R2}; };
SCD_PLAN_SYM(64, 2, 8, 8, 0)
SCD_PLAN_SYM(128, 3, 8, 2, 8)
SCD_PLAN_SYM(256, 2, 16, 16, 0)
SCD_PLAN_SYM(512, 3, 16, 2, 16)
SCD_PLAN_SYM(1024, 3, 16, 4, 16)
SCD_PLAN_SYM(2048, 3, 16, 8, 16)
SCD_PLAN_SYM(4096, 3, 16, 16, 16)
#undef SCD_PLAN_SYM

template <int M, template <int> class PlanT = Plan2> struct Plan2Info {
  using PL = PlanT<M>;
  static constexpr int n = PL::n, r0 = PL::r[0], rl = PL::r[PL::n - 1];
  static constexpr int E = r0, T = M / E;
  static constexpr int R(int s) { return PL::r[s]; }
  static constexpr int p(int s) { return s == 0 ? 1 : p(s - 1) * PL::r[s - 1]; }       // before pass s
  // the pass table: entry (r, k) of pass s >= 1 at off(s) + r p(s) + k, W_{p R}^{k r}
  static constexpr int off(int s) { return s <= 1 ? 0 : off(s - 1) + p(s - 1) * PL::r[s - 1]; }
  static constexpr int tw_len() { return off(n); }
  // consecutive exchange position: one pad element after every r0, so that the 8 threads of a
  // quarter-warp (the unit of a 16-byte shared-memory access) storing their pass-0 outputs at
  // stride r0 hit 8 different 16-byte banks
  static constexpr int lr0 = r0 >= 16 ? 4 : (r0 >= 8 ? 3 : 2);
  __host__ __device__ static constexpr int pad(int i) { return i + (i >> lr0); }
};

// ----------------------------------------------------------------------------- radix-R DFT
template <int L, int J>
__host__ __device__ __forceinline__ C2 twc2(C2 d) {
  constexpr int q = J * (32 / L);
  if constexpr (q == 0) {
    return d;
  } else if constexpr (q == 8) {
    return C2{d.im, neg2(d.re)};
  } else if constexpr (q == 4) {
    constexpr float h = 0.70710678118654752f;
    return C2{mul2(add2(d.re, d.im), dup2(h)), mul2(sub2(d.im, d.re), dup2(h))};
  } else if constexpr (q == 12) {
    constexpr float h = 0.70710678118654752f;
    return C2{mul2(sub2(d.im, d.re), dup2(h)), neg2(mul2(add2(d.re, d.im), dup2(h)))};
  } else {
    constexpr float c = W32::c[q], s = W32::s[q];
    return C2{fma2(d.re, dup2(c), neg2(mul2(d.im, dup2(s)))), fma2(d.re, dup2(s), mul2(d.im, dup2(c)))};
  }
}
template <int SPAN, int START, int J>
__host__ __device__ __forceinline__ void dif2_bfly(C2* v) {
  if constexpr (J < SPAN) {
    const C2 a = v[START + J], b = v[START + J + SPAN];
    v[START + J] = cadd(a, b);
    v[START + J + SPAN] = twc2<2 * SPAN, J>(csub(a, b));
    dif2_bfly<SPAN, START, J + 1>(v);
  }
}
template <int R, int SPAN, int START>
__host__ __device__ __forceinline__ void dif2_stage(C2* v) {
  if constexpr (START < R) {
    dif2_bfly<SPAN, START, 0>(v);
    dif2_stage<R, SPAN, START + 2 * SPAN>(v);
  }
}
template <int R, int SPAN>
__host__ __device__ __forceinline__ void dif2_all(C2* v) {
  if constexpr (SPAN >= 1) {
    dif2_stage<R, SPAN, 0>(v);
    dif2_all<R, SPAN / 2>(v);
  }
}
template <int R, int I>
__host__ __device__ __forceinline__ void unscramble2(C2* v) {
  if constexpr (I < R) {
    constexpr int J = bitrev(I, R);
    if constexpr (J > I) { const C2 t = v[I]; v[I] = v[J]; v[J] = t; }
    unscramble2<R, I + 1>(v);
  }
}
template <int R, int J>
__host__ __device__ __forceinline__ void spread2(C2* v) {       // the first stage on v[R / 2 ..] = 0
  if constexpr (J < R / 2) {
    v[J + R / 2] = twc2<R, J>(v[J]);
    spread2<R, J + 1>(v);
  }
}
// R-point DFT whose inputs from R / 2 on are zero (v[R / 2 ..] not read).
template <int R>
__host__ __device__ __forceinline__ void dft2_half(C2* v) {
  spread2<R, 0>(v);
  dif2_all<R, R / 4>(v);
  unscramble2<R, 0>(v);
}
template <int R>
__host__ __device__ __forceinline__ void dft2(C2* v) {
  dif2_all<R, R / 2>(v);
  unscramble2<R, 0>(v);
}

// ----------------------------------------------------------------------------- batched pairs
// Mapping of a CTA's threads to its C transform pairs: interleaved (a pair's threads C apart: good
// where neighbouring pairs touch neighbouring addresses), consecutive (a pair's T threads side by
// side: good along a pair's own data), or consecutive up to the last exchange and interleaved from
// there on (rows in, columns out: a transposition at no cost but a CTA barrier in place of a team
// one).
enum PairMap { kInterleaved, kConsecutive, kRowsToCols };

// C transform pairs of size M per CTA.  Exchange position pos of pair c: interleaved at pos C + c, free
// of bank conflicts for C >= 8; otherwise padded regions of tstride elements, odd, so that both the
// consecutive and the interleaved accesses of a quarter-warp fill 8 different 16-byte banks.
// v holds the pass-0 inputs t + r (M / r0) of this thread's pair; dst(b, j, f, value) receives bin f
// = i + p j, i = t + b T, p = M / rl, b < E / rl, j < rl of the last pass's thread (c, t) = out_c(),
// out_t().  Callers that run several batches put a barrier between them.
template <int M, int C, int MAP, template <int> class PlanT = Plan2>
struct PairFft {
  using PI = Plan2Info<M, PlanT>;
  static constexpr int E = PI::E, T = PI::T;
  static constexpr int tstride = (M + M / PI::r0) | 1;
  static constexpr int smem_f4 = MAP == kInterleaved ? M * C : tstride * C;

  __device__ __forceinline__ static int in_c() { return MAP == kInterleaved ? (int)threadIdx.x % C : (int)threadIdx.x / T; }
  __device__ __forceinline__ static int in_t() { return MAP == kInterleaved ? (int)threadIdx.x / C : (int)threadIdx.x % T; }
  __device__ __forceinline__ static int out_c() { return MAP == kConsecutive ? (int)threadIdx.x / T : (int)threadIdx.x % C; }
  __device__ __forceinline__ static int out_t() { return MAP == kConsecutive ? (int)threadIdx.x % T : (int)threadIdx.x / C; }
  __device__ __forceinline__ static int at(int c, int pos) {
    return MAP == kInterleaved ? pos * C + c : c * tstride + PI::pad(pos);
  }
  // LAST: the exchange before the last pass
  template <bool LAST>
  __device__ __forceinline__ static void sync() {
    team_sync<T, MAP == kInterleaved || (LAST && MAP == kRowsToCols)>();
  }

  // Twiddled inputs of pass S (tw: the pass table, in shared memory) and its radix transforms.
  template <int S>
  __device__ __forceinline__ static void load(const float4* sm, const float2* tw, int c, int t, C2* v) {
    constexpr int R = PI::R(S), p = PI::p(S), B = E / R;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int i = t + b * T, k = i & (p - 1);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        C2 x = take2(sm + at(c, i + r * (M / R)));
        if (r > 0) x = cmul(x, tw[PI::off(S) + r * p + k]);
        v[b * R + r] = x;
      }
    }
  }
  template <int S>
  __device__ __forceinline__ static void dfts(C2* v) {
    constexpr int R = PI::R(S), B = E / R;
#pragma unroll
    for (int b = 0; b < B; ++b) dft2<R>(v + b * R);
  }
  // passes S .. n - 2: inputs from and outputs to the exchange area
  template <int S>
  __device__ __forceinline__ static void middle(float4* sm, const float2* tw, int c, int t, C2* v) {
    if constexpr (S < PI::n - 1) {
      sync<false>();
      load<S>(sm, tw, c, t, v);
      dfts<S>(v);
      sync<false>();                                       // every read of the pass precedes its writes
      constexpr int R = PI::R(S), p = PI::p(S);
#pragma unroll
      for (int b = 0; b < E / R; ++b) {
        const int i = t + b * T, k = i & (p - 1);
#pragma unroll
        for (int j = 0; j < R; ++j) sm[at(c, (i - k) * R + k + p * j)] = c2_f4(v[b * R + j]);
      }
      middle<S + 1>(sm, tw, c, t, v);
    }
  }
  // The transform up to its last pass's results in v[b rl + j]; free(): called when this thread has read
  // the last of the exchange area.
  // HALF: the inputs M / 2 .. M - 1 (v[r0 / 2 ..]) are zero and not read.
  template <bool HALF = false, class Free>
  __device__ __forceinline__ static void transform(float4* sm, const float2* tw, C2* v, Free&& free) {
    const int c = in_c(), t = in_t();
    if constexpr (HALF) dft2_half<PI::r0>(v);
    else dft2<PI::r0>(v);
#pragma unroll
    for (int j = 0; j < PI::r0; ++j) sm[at(c, t * PI::r0 + j)] = c2_f4(v[j]);
    middle<1>(sm, tw, c, t, v);
    sync<true>();
    load<PI::n - 1>(sm, tw, out_c(), out_t(), v);
    free();
    dfts<PI::n - 1>(v);
  }
  template <class Free, class Dst>
  __device__ __forceinline__ static void run(float4* sm, const float2* tw, C2* v, Free&& free, Dst& dst) {
    constexpr int RL = PI::rl;
    transform(sm, tw, v, free);
#pragma unroll
    for (int b = 0; b < E / RL; ++b)
#pragma unroll
      for (int j = 0; j < RL; ++j) dst(b, j, out_t() + b * T + (M / RL) * j, v[b * RL + j]);
  }
};

}  // namespace scd
