// One output line of a separable contraction, made by one thread: the tree
// passes (upward.cu, downward.cu).
#pragma once

#include "fmm_internal.cuh"

// `return call<order> args;` for the plan's order 1..8.
#define FMM_BY_ORDER(p, call, args)              \
  switch (p) {                                   \
    case 1: return call<1> args;                 \
    case 2: return call<2> args;                 \
    case 3: return call<3> args;                 \
    case 4: return call<4> args;                 \
    case 5: return call<5> args;                 \
    case 6: return call<6> args;                 \
    case 7: return call<7> args;                 \
    case 8: return call<8> args;                 \
    default: return cudaErrorInvalidValue;       \
  }

namespace fmm {
namespace lines {

// a[o] = sum_{k < K} W(o, k) in[k stride], o < NO, weight (hi, lo) at
// W[o wo + k wk]; values (hi, lo), the terms summed in double-float as in
// contract_mid_df, normalised at the end.
template <int NO>
__device__ __forceinline__ void expand_line(const float2* in, int stride, int K, const float2* W, int wo, int wk,
                                            float2 (&a)[NO]) {
#pragma unroll
  for (int o = 0; o < NO; ++o) a[o] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const float2 x = in[k * stride];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const float2 w = W[o * wo + k * wk];
      const float pr = __fmul_rn(w.x, x.x);
      const float pe = fmaf(w.x, x.x, -pr);            // exact product error
      const float2 t = df_two_sum(a[o].x, pr);
      a[o].x = t.x;
      a[o].y = fmaf(w.x, x.y, fmaf(w.y, x.x, __fadd_rn(a[o].y, __fadd_rn(pe, t.y))));
    }
  }
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    const float s = __fadd_rn(a[o].x, a[o].y);
    a[o] = make_float2(s, __fsub_rn(a[o].y, __fsub_rn(s, a[o].x)));
  }
}
// The same in FP32, the low halves of the weights summed apart, as in contract_mid.
template <int NO>
__device__ __forceinline__ void expand_line_f(const float* in, int stride, int K, const float2* W, int wo, int wk,
                                              float (&a)[NO]) {
  float lo[NO];
#pragma unroll
  for (int o = 0; o < NO; ++o) a[o] = lo[o] = 0.f;
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const float x = in[k * stride];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const float2 w = W[o * wo + k * wk];
      a[o] = fmaf(w.x, x, a[o]);
      lo[o] = fmaf(w.y, x, lo[o]);
    }
  }
#pragma unroll
  for (int o = 0; o < NO; ++o) a[o] += lo[o];
}

}  // namespace lines
}  // namespace fmm
