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
  static constexpr int threads(int blocks) { return (blocks * P * P + 31) / 32 * 32; }
  static constexpr int NM = 2 * P - 1;
  // row stride of the shared arrays whose x lines a thread walks: odd, so that
  // a warp's rows start on different banks (P = 16 has no room for it)
  static constexpr int PS = P >= 16 ? P : (P | 1);
  // blocks per CTA of the forward transforms, and the threads: one round of the
  // x and y lines (P^2 per block), just under two of the z lines (NM P)
  static constexpr int NB = P >= 16 ? 1 : (P >= 7 ? 2 : (P >= 5 ? 4 : (P >= 3 ? 8 : 16)));
  static constexpr int THR = threads(NB);
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
  static __device__ __forceinline__ real neg(real a) { return -a; }
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
  static __device__ __forceinline__ real neg(real a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ real add(real a, real b) {
    const float2 t = df_two_sum(a.x, b.x);
    return done(make_float2(t.x, __fadd_rn(t.y, __fadd_rn(a.y, b.y))));
  }
  static __device__ __forceinline__ cplx pack(real re, real im) { return make_float4(re.x, re.y, im.x, im.y); }
  static __device__ __forceinline__ real re(cplx c) { return make_float2(c.x, c.y); }
  static __device__ __forceinline__ real im(cplx c) { return make_float2(c.z, c.w); }
};

// Line transforms of NM = 2P - 1 points.  cos is even and sin odd about half
// the line, so the forward transform of P nonzero inputs makes the outputs k
// and NM - k from the same four sums, and the inverse, which keeps P outputs,
// folds the inputs s and NM - s into their sum and difference first: half the
// multiply-adds of the plain sums.
// Twiddles: FP32 has cos and sin of 2 pi j / NM as constants of the unrolled
// code (read from shared memory, one load per four multiply-adds, the loads
// bounded the transforms); double-float reads (cos hi, lo,
// sin hi, lo) from shared memory.
template <bool DF, int P>
struct Twiddle;
// cos x for |x| <= pi, by its Taylor series, at compile time.
constexpr double series_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 40; ++k) {
    term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    sum += term;
  }
  return sum;
}
template <int P>
struct TwiddleTable {
  float c[P] = {}, s[P] = {};
  constexpr TwiddleTable() {
    constexpr double pi = 3.14159265358979323846;
    for (int j = 0; j < P; ++j) {
      const double a = 2.0 * pi * j / (2 * P - 1);
      c[j] = (float)series_cos(a);
      s[j] = j ? (float)series_cos(a - 0.5 * pi) : 0.f;     // sin a
    }
  }
};
template <int P>
struct Twiddle<false, P> {
  static constexpr int NM = 2 * P - 1;
  __device__ __forceinline__ Twiddle(const float4* __restrict__, const float4*) {}
  // j in [0, NM)
  __device__ __forceinline__ float4 at(int j) const {
    constexpr TwiddleTable<P> t{};
    return j < P ? make_float4(t.c[j], 0.f, t.s[j], 0.f) : make_float4(t.c[NM - j], 0.f, -t.s[NM - j], 0.f);
  }
};
template <int P>
struct Twiddle<true, P> {
  const float4* tw;
  __device__ __forceinline__ Twiddle(const float4* __restrict__, const float4* shared) : tw(shared) {}
  __device__ __forceinline__ float4 at(int j) const { return tw[j]; }
};

// X_k = sum_{s < P} x_s e^{-2 pi i k s / NM}; emit(k, re, im) for k < NM, or for
// real input (xi unused) k < P only.
template <bool DF, int P, bool REAL, typename Emit>
__device__ __forceinline__ void forward_line(const typename Num<DF>::real (&xr)[P],
                                             const typename Num<DF>::real (&xi)[P], const Twiddle<DF, P>& tw,
                                             Emit emit) {
  using T = Num<DF>;
  using real = typename T::real;
  constexpr int NM = 2 * P - 1;
  {
    real re = xr[0], im = REAL ? T::zero() : xi[0];
#pragma unroll
    for (int s = 1; s < P; ++s) {
      re = T::add(re, xr[s]);
      if (!REAL) im = T::add(im, xi[s]);
    }
    emit(0, re, im);
  }
#pragma unroll(DF ? 1 : P)
  for (int k = 1; k < P; ++k) {
    real cr = T::zero(), ci = T::zero(), sr = T::zero(), si = T::zero();
    T::mac(cr, 1.f, 0.f, xr[0]);
    if (!REAL) T::mac(ci, 1.f, 0.f, xi[0]);
    int j = 0;
#pragma unroll
    for (int s = 1; s < P; ++s) {
      j += k;
      j -= j >= NM ? NM : 0;
      const float4 w = tw.at(j);
      T::mac(cr, w.x, w.y, xr[s]);
      T::mac(sr, w.z, w.w, xr[s]);
      if (!REAL) {
        T::mac(ci, w.x, w.y, xi[s]);
        T::mac(si, w.z, w.w, xi[s]);
      }
    }
    cr = T::done(cr);
    sr = T::done(sr);
    if (REAL) {
      emit(k, cr, T::neg(sr));
    } else {
      ci = T::done(ci);
      si = T::done(si);
      emit(k, T::add(cr, si), T::add(ci, T::neg(sr)));
      emit(NM - k, T::add(cr, T::neg(si)), T::add(ci, sr));
    }
  }
}

// y_z = sum_{s < NM} x_s e^{+2 pi i z s / NM}; emit(z, re, im) for z < P (ALL:
// every z < NM).  xr, xi are used up.
// RISING: the sums run from the highest frequency down to 0.  The spectrum of a
// near field falls off, so the terms then grow along the sum and most of its
// FP32 roundings are of a small running value; the constant term last costs one
// addition per output (FMM_NEAR_FFT: near_spec.cu).
template <bool DF, int P, bool ALL = false, bool RISING = false, typename Emit>
__device__ __forceinline__ void inverse_line(typename Num<DF>::real (&xr)[2 * P - 1],
                                             typename Num<DF>::real (&xi)[2 * P - 1], const Twiddle<DF, P>& tw,
                                             Emit emit) {
  using T = Num<DF>;
  using real = typename T::real;
  constexpr int NM = 2 * P - 1;
#pragma unroll
  for (int s = 1; s < P; ++s) {                  // [s]: sum, [NM - s]: difference
    const real ar = xr[s], ai = xi[s], br = xr[NM - s], bi = xi[NM - s];
    xr[s] = T::add(ar, br);
    xi[s] = T::add(ai, bi);
    xr[NM - s] = T::add(ar, T::neg(br));
    xi[NM - s] = T::add(ai, T::neg(bi));
  }
  {
    real re = xr[RISING ? P - 1 : 0], im = xi[RISING ? P - 1 : 0];
#pragma unroll
    for (int i = 1; i < P; ++i) {
      const int s = RISING ? P - 1 - i : i;
      re = T::add(re, xr[s]);
      im = T::add(im, xi[s]);
    }
    emit(0, re, im);
  }
#pragma unroll(DF ? 1 : P)
  for (int z = 1; z < P; ++z) {
    real cr = T::zero(), ci = T::zero(), sr = T::zero(), si = T::zero();
    if (!RISING) {
      T::mac(cr, 1.f, 0.f, xr[0]);
      T::mac(ci, 1.f, 0.f, xi[0]);
    }
    int j = RISING ? P * z % NM : 0;
#pragma unroll
    for (int i = 1; i < P; ++i) {
      const int s = RISING ? P - i : i;
      j += RISING ? NM - z : z;
      j -= j >= NM ? NM : 0;
      const float4 w = tw.at(j);
      if (ALL) {
        T::mac(cr, w.x, w.y, xr[s]);
        T::mac(ci, w.x, w.y, xi[s]);
        T::mac(si, w.z, w.w, xi[NM - s]);
        T::mac(sr, w.z, w.w, xr[NM - s]);
      } else {
        T::mac(cr, w.x, w.y, xr[s]);
        T::mac(ci, w.x, w.y, xi[s]);
        T::mac(cr, -w.z, -w.w, xi[NM - s]);
        T::mac(ci, w.z, w.w, xr[NM - s]);
      }
    }
    if (RISING) {
      T::mac(cr, 1.f, 0.f, xr[0]);
      T::mac(ci, 1.f, 0.f, xi[0]);
    }
    cr = T::done(cr);
    ci = T::done(ci);
    if (ALL) {
      sr = T::done(sr);
      si = T::done(si);
      emit(z, T::add(cr, T::neg(si)), T::add(ci, sr));
      emit(NM - z, T::add(cr, si), T::add(ci, T::neg(sr)));
    } else {
      emit(z, cr, ci);
    }
  }
}

// The real points x < P of a half spectrum v[0..P-1]: Re v_0 + 2 sum Re(v_s e^{+2 pi i x s / NM}).
template <bool DF, int P, bool RISING = false, typename Emit>
__device__ __forceinline__ void inverse_real_line(const typename Num<DF>::real (&xr)[P],
                                                  const typename Num<DF>::real (&xi)[P], const Twiddle<DF, P>& tw,
                                                  Emit emit) {
  using T = Num<DF>;
  using real = typename T::real;
  constexpr int NM = 2 * P - 1;
#pragma unroll(DF ? 1 : P)
  for (int x = 0; x < P; ++x) {
    real a = T::zero();
    int j = RISING ? P * x % NM : 0;
#pragma unroll
    for (int i = 1; i < P; ++i) {
      const int s = RISING ? P - i : i;
      j += RISING ? NM - x : x;
      j -= j >= NM ? NM : 0;
      const float4 w = tw.at(j);
      T::mac(a, w.x, w.y, xr[s]);
      T::mac(a, -w.z, -w.w, xi[s]);
    }
    emit(x, T::add(T::twice(T::done(a)), xr[0]));
  }
}

// X_k = sum_{s < NM} x_s e^{-2 pi i k s / NM} of NM real values, k < P; xr is used up.
template <bool DF, int P, typename Emit>
__device__ __forceinline__ void forward_real_full_line(typename Num<DF>::real (&xr)[2 * P - 1], const Twiddle<DF, P>& tw,
                                                       Emit emit) {
  using T = Num<DF>;
  using real = typename T::real;
  constexpr int NM = 2 * P - 1;
#pragma unroll
  for (int s = 1; s < P; ++s) {
    const real a = xr[s], b = xr[NM - s];
    xr[s] = T::add(a, b);
    xr[NM - s] = T::add(a, T::neg(b));
  }
#pragma unroll 1
  for (int k = 0; k < P; ++k) {
    real c = T::zero(), d = T::zero();
    T::mac(c, 1.f, 0.f, xr[0]);
    int j = 0;
#pragma unroll
    for (int s = 1; s < P; ++s) {
      j += k;
      j -= j >= NM ? NM : 0;
      const float4 w = tw.at(j);
      T::mac(c, w.x, w.y, xr[s]);
      T::mac(d, -w.z, -w.w, xr[NM - s]);
    }
    emit(k, T::done(c), T::done(d));
  }
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
