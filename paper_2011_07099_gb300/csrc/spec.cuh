// Shared parts of the spectral kernels (m2l_spec.cu: M2L, near_spec.cu: near
// zone): FP32 and double-float lane arithmetic, the line DFT, the shape of a
// zero-padded transform of P^3 real points.
//
// Two blocks of P points per axis interact through lags in [-(P-1), P-1], so
// NM = 2P - 1 points per axis hold the linear convolution without wrap; the
// half spectrum of real input is kx in [0, P - 1], NK = NM^2 P frequencies,
// k = (kz NM + ky) P + kx.
#pragma once

#include "fmm_internal.cuh"

namespace fmm {
namespace spec {

template <int P>
struct Shape {
  static constexpr int NM = 2 * P - 1;
  static constexpr int LINES = NM * P;
  // blocks per CTA of the transforms: about 128 lines of the widest pass
  static constexpr int NB = LINES <= 16 ? 8 : (LINES <= 32 ? 4 : (LINES <= 72 ? 2 : 1));
};

// ------------------------------------------------------------- arithmetic
// Lane value of one complex frequency and its accumulation, FP32 or double-float.
template <bool DF>
struct Num;
template <>
struct Num<false> {
  using real = float;
  using cplx = float2;                    // (re, im)
  static constexpr int LANES = 16;        // frequencies per chunk
  static __device__ __forceinline__ real zero() { return 0.f; }
  static __device__ __forceinline__ void mac(real& a, float wh, float, real x) { a = fmaf(wh, x, a); }
  static __device__ __forceinline__ real done(real a) { return a; }
  static __device__ __forceinline__ real twice(real a) { return 2.f * a; }
  static __device__ __forceinline__ real add(real a, real b) { return a + b; }
  static __device__ __forceinline__ cplx pack(real re, real im) { return make_float2(re, im); }
  static __device__ __forceinline__ real re(cplx c) { return c.x; }
  static __device__ __forceinline__ real im(cplx c) { return c.y; }
};
template <>
struct Num<true> {
  using real = float2;                    // (hi, lo)
  using cplx = float4;                    // (re hi, re lo, im hi, im lo)
  static constexpr int LANES = 8;
  static __device__ __forceinline__ real zero() { return make_float2(0.f, 0.f); }
  // a += w x in double-float (TwoProd by FMA, TwoSum; the error terms in a.y)
  static __device__ __forceinline__ void mac(real& a, float wh, float wl, real x) {
    const float pr = __fmul_rn(wh, x.x);
    const float pe = fmaf(wh, x.x, -pr);
    const float2 t = df_two_sum(a.x, pr);
    a.x = t.x;
    a.y = fmaf(wh, x.y, fmaf(wl, x.x, __fadd_rn(a.y, __fadd_rn(pe, t.y))));
  }
  static __device__ __forceinline__ real done(real a) {
    const float s = __fadd_rn(a.x, a.y);
    return make_float2(s, __fsub_rn(a.y, __fsub_rn(s, a.x)));
  }
  static __device__ __forceinline__ real twice(real a) { return make_float2(2.f * a.x, 2.f * a.y); }
  static __device__ __forceinline__ real add(real a, real b) {
    const float2 t = df_two_sum(a.x, b.x);
    return done(make_float2(t.x, __fadd_rn(t.y, __fadd_rn(a.y, b.y))));
  }
  static __device__ __forceinline__ cplx pack(real re, real im) { return make_float4(re.x, re.y, im.x, im.y); }
  static __device__ __forceinline__ real re(cplx c) { return make_float2(c.x, c.y); }
  static __device__ __forceinline__ real im(cplx c) { return make_float2(c.z, c.w); }
};

// One line's DFT value at frequency (or point) k: sum_{s < NIN} x_s e^{-+ 2 pi i k s / NM};
// `inv` takes the conjugate twiddles.  tw in shared memory.
template <bool DF, int NM, int NIN, bool REAL_IN, bool INV>
__device__ __forceinline__ void dft_at(const typename Num<DF>::real* xr, const typename Num<DF>::real* xi, int k,
                                       const float4* tw, typename Num<DF>::real& re, typename Num<DF>::real& im) {
  using T = Num<DF>;
  re = T::zero();
  im = T::zero();
  int j = 0;
#pragma unroll
  for (int s = 0; s < NIN; ++s) {
    const float4 w = tw[j];
    const float sh = INV ? w.z : -w.z, sl = INV ? w.w : -w.w;   // e^{i a} = c + i s (inverse), c - i s (forward)
    T::mac(re, w.x, w.y, xr[s]);
    T::mac(im, sh, sl, xr[s]);
    if (!REAL_IN) {
      T::mac(re, -sh, -sl, xi[s]);
      T::mac(im, w.x, w.y, xi[s]);
    }
    j += k;
    j -= j >= NM ? NM : 0;
  }
  re = T::done(re);
  im = T::done(im);
}


// A stored value (FP32 or double-float) as the arithmetic's.
template <bool DFA>
__device__ __forceinline__ typename Num<DFA>::real widen(float v) {
  if constexpr (DFA) return make_float2(v, 0.f);
  else return v;
}
template <bool DFA>
__device__ __forceinline__ typename Num<DFA>::real widen(float2 v) {
  static_assert(DFA, "double-float storage needs double-float arithmetic");
  return v;
}
// The arithmetic's value rounded to the storage.
template <bool DFS, bool DFA>
__device__ __forceinline__ typename Num<DFS>::real narrow(typename Num<DFA>::real v) {
  if constexpr (DFA && !DFS) return v.x + v.y;
  else return v;
}

inline int lanes(bool df) { return df ? Num<true>::LANES : Num<false>::LANES; }
inline int chunks_of(int p, bool df) {
  const int nk = (2 * p - 1) * (2 * p - 1) * p;
  return (nk + lanes(df) - 1) / lanes(df);
}

}  // namespace spec
}  // namespace fmm
