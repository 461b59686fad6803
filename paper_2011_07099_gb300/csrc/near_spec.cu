// Leaf stage by spectral products: the near-zone sum over the 27 neighbour
// leaves as zero-padded convolutions, and the leaf's L2P far field.
//
// Sec. 3 computes the near zone of a regular grid with an FFT under
// non-periodic boundary conditions, obtained by doubling the grid.  Here that
// is done per pair of leaves: for a target leaf T of S cells per side and a
// neighbour T + o, o in {-1, 0, 1}^3, the field at cell r is the linear
// convolution
//   Phi_T(r) += sum_{r'} K(r - r' - S o) m_{T+o}(r'),   r, r' in [0, S)^3,
// with lags in [-(S-1), S-1]^3: circular without wrap on NM = 2S - 1 points
// per axis (spec.cuh), so on the spectra Phi^_T(k) = sum_o K^_o(k) m^_{T+o}(k).
// K = (G, -grad G) at the cell offsets is the plan's near table, the FP32
// values the direct kernels use.  Per leaf and offset that is NK = NM^2 S
// complex multiply-adds and field instead of S^6 real ones: 27 x 4 x 1800
// against 27 x 4 x 262 144 at S = 8.
//
// Kernels
//   k_ns_planes, k_ns_lines  plan time: the kernel spectra, double-float rounded once
//   k_ns_fwd     per leaf: the spectrum of its masses
//   k_ns_mac     per (tile of 4^3 target leaves, chunk of frequencies): the
//                27-term sums of the 4 fields
//   k_ns_inv     per (leaf, field): inverse transform, only the S^3 cells, plus
//                the L2P far field (eq. fmm3 at the leaves), written once
// Arithmetic: FP32 spectra and sums; the transforms in FP32 (FMM_NEAR_FFT) or,
// where the plan asks for the direct sum's accuracy (FMM_NEAR_DIRECT), in
// double-float with one rounding on store.  That accuracy is of the mesh's
// norm: the rounding of a pair of leaves is spread over both, so a cell beside
// a heavy one errs by ~1e-7 of the heavy one's peak field, and a lone cell's
// force on itself, exactly 0 by pairs, reads 4e-10 of its peak field (1e-8 with
// FP32 transforms).  With 16-cell leaves the L2P reads
// the FP64 local field (fmm_internal.cuh, kWideLeaf) in double-float.
// Measured (direct kernels of p2p.cu before -> here): 128^3 isolated with
// 16-cell leaves 177 -> 1.6 ms; 256^3, S = 8 30.6 -> 6.1 ms at direct accuracy
// (sums 0.91, inverse with L2P 4.3); 96^3, S = 6 1.04 -> 0.31 ms; 128^3, S = 4
// 0.87 -> 0.47 ms.  FMM_NEAR_FFT at 256^3: 2.23 ms for radix-2 transforms of 16
// points and a separate L2P -> 1.74 ms (sums 1.08 -> 0.91: 22 % fewer
// frequencies; inverse and L2P 0.92 -> 0.69).  The error of the plain 256^3
// solve against FP64 went from 3.7e-7 to 2.9e-7 with the direct form, and with
// FP32 transforms in its place to 3.1e-7 there but from 1.2e-7 to 1.8e-7 at
// 48^3, S = 6, so the direct form keeps double-float ones.
// FP32 inverse transforms sum from the highest frequency down (spec.cuh,
// RISING).  FMM_NEAR_FFT against FP64, 64^3, S = 8, p = 6, potential: radix-2 of
// 16 points 1.96e-7 (lognormal), 1.62e-7 (clumps); 15-term lines from frequency
// 0 up 2.28e-7, 1.93e-7; rising 1.86e-7, 1.35e-7, at 256^3 for 0.2 % of a solve.
#include "fmm_internal.cuh"
#include "spec.cuh"
#include "tc_ptx.cuh"

namespace fmm {
namespace {

using spec::chunks_of;
using spec::forward_line;
using spec::inverse_line;
using spec::inverse_real_line;
using spec::narrow;
using spec::Num;
using spec::Shape;
using spec::Twiddle;
using spec::widen;

constexpr int kKernels = 14;                // offsets 0..13 of 27: the others' kernels are their conjugates
constexpr int kTile = 4;                    // target leaves per tile side
constexpr int kHaloN = kTile + 2;
constexpr int kSlots = kHaloN * kHaloN * kHaloN;

// Leaves whose L2P reads the FP64 local field.
template <int S>
constexpr bool kWideField = S >= kWideLeaf;

// (leaf, field) items per inverse CTA: one wave of lines over its threads, and
// two CTAs' shared memory within an SM.
template <int S, bool DFA>
constexpr int kItems = S >= 16 ? 1 : (S <= 4 ? 8 : (S >= 8 && DFA ? 2 : 4));

// ------------------------------------------------------------- plan time
// Kernel spectra of the offsets 0..13 (kKernels) only: Phi's kernel is even and
// g's odd, so the opposite offsets' are their conjugates up to sign (k_ns_mac).
// Line transforms in double-float, rounded once on store.  With all 27 offsets
// in FP64, at 1/64 of the FP32 rate, the plan of the isolated 128^3 solve (16-
// cell leaves) took 4.7 ms to create; 1.4 with these.
//
// The kernel's value for field f at lag d (cells), from the folded near table
// (|d_i| in [0, 2S-1]); the gradient fields take the sign of their own
// component as the direct sum does, and vanish where that component is 0.
__device__ __forceinline__ float near_value(const float4* __restrict__ tab, int S, int f, int dx, int dy, int dz) {
  const int TD = 2 * S;
  const int ax = dx < 0 ? -dx : dx, ay = dy < 0 ? -dy : dy, az = dz < 0 ? -dz : dz;
  const float v = __ldg(reinterpret_cast<const float*>(tab + (az * TD + ay) * TD + ax) + f);
  const int own = f == 1 ? dx : (f == 2 ? dy : dz);
  return f == 0 || own > 0 ? v : (own < 0 ? -v : 0.f);
}

// CTA (z lag, offset x field): the x and y transforms of one lag plane, a line
// per thread.  out [offset x field][z lag][ky][kx].
constexpr int kPlaneThr = 32;
template <int S>
__global__ void __launch_bounds__(kPlaneThr) k_ns_planes(const float4* __restrict__ tab, const float4* __restrict__ twg,
                                                         float4* __restrict__ out) {
  using T = Num<true>;
  constexpr int NM = Shape<S>::NM;
  static_assert(NM <= kPlaneThr, "a thread per x line");
  __shared__ float4 tw[NM];
  __shared__ float4 t1[NM * S];           // [y][kx]
  const int vz = blockIdx.x, of = blockIdx.y, o = of / 4, f = of % 4, tid = threadIdx.x;
  const int ox = o % 3 - 1, oy = (o / 3) % 3 - 1, oz = o / 9 - 1;
  if (tid < NM) tw[tid] = __ldg(twg + tid);
  __syncthreads();
  const Twiddle<true, S> wt(twg, tw);
  auto lag = [](int v) { return v < S ? v : v - NM; };
  if (tid < NM) {                         // x: line y lag = tid
    float2 x[NM];
#pragma unroll
    for (int vx = 0; vx < NM; ++vx)
      x[vx] = widen<true>(near_value(tab, S, f, lag(vx) - S * ox, lag(tid) - S * oy, lag(vz) - S * oz));
    spec::forward_real_full_line<true, S>(x, wt,
                                          [&](int k, float2 re, float2 im) { t1[tid * S + k] = T::pack(re, im); });
  }
  __syncthreads();
  if (tid < S) {                          // y: line kx = tid
    float2 xr[NM], xi[NM];
#pragma unroll
    for (int v = 0; v < NM; ++v) {
      const float4 c = t1[v * S + tid];
      xr[v] = T::re(c);
      xi[v] = T::im(c);
    }
    // the forward transform at k is the inverse one at NM - k
    inverse_line<true, S, true>(xr, xi, wt, [&](int y, float2 re, float2 im) {
      out[(((size_t)of * NM + vz) * NM + (y ? NM - y : 0)) * S + tid] = T::pack(re, im);
    });
  }
}

// The z transform, 1/NM^3, and the store K^[chunk][offset][2 field pairs][16]
// float4 (re, im of two fields); a line (ky, kx) per thread.
template <int S>
__global__ void __launch_bounds__(128) k_ns_lines(const float4* __restrict__ in, const float4* __restrict__ twg,
                                                  float* __restrict__ K) {
  using T = Num<true>;
  constexpr int NM = Shape<S>::NM, LANES = Num<false>::LANES;
  __shared__ float4 tw[NM];
  const int o = blockIdx.y / 4, f = blockIdx.y % 4;
  if (threadIdx.x < NM) tw[threadIdx.x] = __ldg(twg + threadIdx.x);
  __syncthreads();
  const Twiddle<true, S> wt(twg, tw);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= NM * S) return;
  float2 xr[NM], xi[NM];
#pragma unroll
  for (int v = 0; v < NM; ++v) {
    const float4 c = __ldg(in + ((size_t)blockIdx.y * NM + v) * NM * S + q);
    xr[v] = T::re(c);
    xi[v] = T::im(c);
  }
  const float2 scale = df_from_double(1.0 / ((double)NM * NM * NM));
  inverse_line<true, S, true>(xr, xi, wt, [&](int z, float2 re, float2 im) {
    const int k = (z ? NM - z : 0) * NM * S + q, l = k % LANES;
    float2 a = T::zero(), b = T::zero();
    T::mac(a, scale.x, scale.y, re);
    T::mac(b, scale.x, scale.y, im);
    const size_t base = ((size_t)(k / LANES) * kKernels + o) * 128;   // floats
    reinterpret_cast<float2*>(K + base)[((f / 2) * LANES + l) * 2 + (f & 1)] = make_float2(a.x + a.y, b.x + b.y);
  });
}

// ------------------------------------------------------------- transforms
// Spectra of the leaves' masses m = (rho - mean) / N^3, NB leaves per CTA.
template <int S, bool DFA>
__global__ void __launch_bounds__(Shape<S>::THR) k_ns_fwd(const float* __restrict__ rho,
                                                                  const double* __restrict__ mean, int N, int L,
                                                                  const float4* __restrict__ twg,
                                                                  void* __restrict__ Mout) {
  using T = Num<DFA>;
  using store = Num<false>;
  using real = typename T::real;
  using cplx = typename T::cplx;
  constexpr int NM = Shape<S>::NM, NB = Shape<S>::NB, S3 = S * S * S, PS = Shape<S>::PS,
                LANES = store::LANES;
  extern __shared__ float4 sm4[];
  __shared__ float4 tw[NM];
  cplx* t1 = reinterpret_cast<cplx*>(sm4);                 // [NB][z][y][kx]
  cplx* t2 = t1 + NB * S * S * PS;                         // [NB][z][ky][kx]
  real* in = reinterpret_cast<real*>(t2);                  // [NB][z][y][x], consumed before t2 is written
  const int tid = threadIdx.x, nthr = blockDim.x;
  const size_t leaf0 = (size_t)blockIdx.x * NB, leaves = (size_t)1 << (3 * L);
  if (DFA && tid < NM) tw[tid] = __ldg(twg + tid);
  const Twiddle<DFA, S> wt(twg, tw);
  const double mu = *mean;
  const float mu_hi = (float)mu, mu_lo = (float)(mu - (double)mu_hi);
  const double ivd = 1.0 / ((double)N * N * N);
  const float iv = (float)ivd, iv_lo = (float)(ivd - (double)iv);
  for (int i = tid; i < NB * S3; i += nthr) {
    const int x = i % S, y = (i / S) % S, z = (i / (S * S)) % S;
    uint32_t lx, ly, lz;
    unmorton((uint32_t)(leaf0 + i / S3), lx, ly, lz);
    const float r = __ldg(rho + ((size_t)(lz * S + z) * N + (ly * S + y)) * N + lx * S + x);
    if constexpr (DFA) {                                   // exactly, as P2M forms them
      const float2 d = df_two_sum(r, -mu_hi);
      const float dlo = __fsub_rn(d.y, mu_lo);
      const float ph = __fmul_rn(d.x, iv);
      const float lo = fmaf(d.x, iv_lo, fmaf(dlo, iv, fmaf(d.x, iv, -ph)));
      in[(i / S) * PS + x] = T::done(make_float2(ph, lo));
    } else {
      in[(i / S) * PS + x] = ((r - mu_hi) - mu_lo) * iv;
    }
  }
  __syncthreads();
  for (int l = tid; l < NB * S * S; l += nthr) {           // x: S reals -> S frequencies
    real x[S];
#pragma unroll
    for (int s = 0; s < S; ++s) x[s] = in[l * PS + s];
    forward_line<DFA, S, true>(x, x, wt, [&](int k, real re, real im) { t1[l * PS + k] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < NB * S * S; l += nthr) {           // y: line (leaf, z, kx)
    const int kx = l % S, nz = l / S;
    real xr[S], xi[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const cplx c = t1[(nz * S + s) * PS + kx];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    forward_line<DFA, S, false>(xr, xi, wt, [&](int k, real re, real im) { t2[(nz * NM + k) * S + kx] = T::pack(re, im); });
  }
  __syncthreads();
  typename store::cplx* Mh = reinterpret_cast<typename store::cplx*>(Mout);
  for (int l = tid; l < NB * NM * S; l += nthr) {          // z: line (leaf, ky, kx)
    const int q = l % (NM * S), nb = l / (NM * S);
    real xr[S], xi[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const cplx c = t2[(nb * S + s) * NM * S + q];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    forward_line<DFA, S, false>(xr, xi, wt, [&](int kz, real re, real im) {
      const int k = kz * NM * S + q;
      Mh[((size_t)(k / LANES) * (leaves + 1) + leaf0 + nb) * LANES + k % LANES] =
          store::pack(narrow<false, DFA>(re), narrow<false, DFA>(im));
    });
  }
}

// One separable L2P pass: out[a][c][b] = sum_k W[k][c] in[a][k][b], b < B, a < A;
// weights (hi, lo).  A thread makes the S outputs of a line (a, b).  OS: row
// stride of `out`'s innermost S values.
template <bool DFA, int S, int B, int OS>
__device__ __forceinline__ void l2p_pass(const typename Num<DFA>::real* in, typename Num<DFA>::real* out, int A, int p,
                                         const float2* W, int tid, int nthr) {
  using T = Num<DFA>;
  for (int l = tid; l < A * B; l += nthr) {
    const int b = l % B, a = l / B;
    const typename T::real* src = in + (size_t)a * p * B + b;
    float hi[S], lo[S];
#pragma unroll
    for (int c = 0; c < S; ++c) hi[c] = lo[c] = 0.f;
#pragma unroll 1
    for (int k = 0; k < p; ++k) {
      const typename T::real x = src[k * B];
#pragma unroll
      for (int c = 0; c < S; ++c) {
        const float2 w = W[k * S + c];
        if constexpr (DFA) {
          float2 t = make_float2(hi[c], lo[c]);
          T::mac(t, w.x, w.y, x);
          hi[c] = t.x;
          lo[c] = t.y;
        } else {
          hi[c] = fmaf(w.x, x, hi[c]);
          lo[c] = fmaf(w.y, x, lo[c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < S; ++c) {
      const int o = (a * S + c) * B + b;
      typename T::real& dst = out[OS == S ? o : (o / S) * OS + o % S];
      if constexpr (DFA) dst = T::done(make_float2(hi[c], lo[c]));
      else dst = hi[c] + lo[c];
    }
  }
  __syncthreads();
}

// Outputs.  CTA: IB (leaf, field) items.
template <int S, bool DFA>
__global__ void __launch_bounds__(Shape<S>::threads(kItems<S, DFA>)) k_ns_inv(const void* __restrict__ Pin, int nkp, int far_at, int N, int p,
                                                                  const float* __restrict__ F,
                                                                  const double* __restrict__ F64,
                                                                  const float2* __restrict__ wp2m,
                                                                  const float4* __restrict__ twg,
                                                                  float* __restrict__ phi, float* __restrict__ acc) {
  using T = Num<DFA>;
  using store = Num<false>;
  using real = typename T::real;
  using cplx = typename T::cplx;
  constexpr int NM = Shape<S>::NM, IB = kItems<S, DFA>, PS = Shape<S>::PS;
  extern __shared__ float4 sm4[];
  __shared__ float4 tw[NM];
  __shared__ float2 W[kMaxOrder * S];
  cplx* t2 = reinterpret_cast<cplx*>(sm4);                 // [IB][z][y][kx]
  cplx* t1 = t2 + IB * S * S * PS;                         // [IB][z][ky][kx]
  real* far = reinterpret_cast<real*>(reinterpret_cast<char*>(sm4) + far_at);   // [IB][z][y][x], behind t1 and the L2P scratch
  const int tid = threadIdx.x, nthr = blockDim.x;
  const size_t item0 = (size_t)blockIdx.x * IB;
  const int p3 = p * p * p;
  if (DFA && tid < NM) tw[tid] = __ldg(twg + tid);
  const Twiddle<DFA, S> wt(twg, tw);
  for (int i = tid; i < p * S; i += nthr) W[i] = __ldg(wp2m + i);
  {                                                        // L2P, scratch in t2's and t1's space
    real* a = reinterpret_cast<real*>(sm4);                // [IB][p^3]
    real* b = a + IB * p3;                                 // [IB][p][p][S]
    real* c = b + IB * p * p * S;                          // [IB][p][S][S]
    for (int i = tid; i < IB * p3; i += nthr) {
      if constexpr (kWideField<S>) a[i] = df_from_double(__ldg(F64 + item0 * p3 + i));
      else a[i] = widen<DFA>(__ldg(F + item0 * p3 + i));
    }
    __syncthreads();
    l2p_pass<DFA, S, 1, S>(a, b, IB * p * p, p, W, tid, nthr);
    l2p_pass<DFA, S, S, S>(b, c, IB * p, p, W, tid, nthr);
    l2p_pass<DFA, S, S * S, PS>(c, far, IB, p, W, tid, nthr);
  }
  const typename store::cplx* Ph = reinterpret_cast<const typename store::cplx*>(Pin) + item0 * nkp;
  for (int l = tid; l < IB * NM * S; l += nthr) {          // z: line (item, ky, kx), NM -> S
    const int q = l % (NM * S), it = l / (NM * S);
    real xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const typename store::cplx v = __ldg(Ph + (size_t)it * nkp + s * NM * S + q);
      xr[s] = widen<DFA>(store::re(v));
      xi[s] = widen<DFA>(store::im(v));
    }
    inverse_line<DFA, S, false, !DFA>(xr, xi, wt, [&](int z, real re, real im) { t1[(it * S + z) * NM * S + q] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < IB * S * S; l += nthr) {           // y: line (item, z, kx), NM -> S
    const int kx = l % S, iz = l / S;
    real xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const cplx v = t1[(iz * NM + s) * S + kx];
      xr[s] = T::re(v);
      xi[s] = T::im(v);
    }
    inverse_line<DFA, S, false, !DFA>(xr, xi, wt, [&](int y, real re, real im) { t2[(iz * S + y) * PS + kx] = T::pack(re, im); });
  }
  __syncthreads();
  const size_t N3 = (size_t)N * N * N;
  for (int l = tid; l < IB * S * S; l += nthr) {           // x: line (item, z, y), half spectrum -> S cells
    real xr[S], xi[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const cplx v = t2[l * PS + s];
      xr[s] = T::re(v);
      xi[s] = T::im(v);
    }
    const size_t item = item0 + l / (S * S);
    const int y = l % S, z = (l / S) % S, f = (int)(item & 3);
    uint32_t lx, ly, lz;
    unmorton((uint32_t)(item >> 2), lx, ly, lz);
    float* dst = (f == 0 ? phi : acc + (size_t)(f - 1) * N3) +
                 ((size_t)(lz * S + z) * N + (ly * S + y)) * N + lx * S;
    const real* fr = far + l * PS;
    if constexpr (!DFA && S % 4 == 0) {
      float o[S];
      inverse_real_line<DFA, S, !DFA>(xr, xi, wt, [&](int x, float v) { o[x] = v + fr[x]; });
#pragma unroll
      for (int q = 0; q < S; q += 4) *reinterpret_cast<float4*>(dst + q) = make_float4(o[q], o[q + 1], o[q + 2], o[q + 3]);
    } else {
      inverse_real_line<DFA, S, !DFA>(xr, xi, wt, [&](int x, real v) { dst[x] = narrow<false, DFA>(T::add(v, fr[x])); });
    }
  }
}

// ---------------------------------------------------------- spectral sums
// Rows of 4 target leaves along x per thread, as k_spec_mac; the chunk's 14
// kernel spectra and the tile's 6^3 source spectra in shared memory (35 KB),
// the next chunk's copied (cp.async) during the current sums: a CTA takes
// `per` consecutive chunks of one tile, up to 8, fewer where that leaves fewer
// than 4 CTAs per SM.
constexpr int kChunks = 8;
constexpr int kStage = kKernels * 32 + kSlots * 8;   // float4 per stage
__global__ void __launch_bounds__(256) k_ns_mac(const float4* __restrict__ K, const void* __restrict__ Mh,
                                                          void* __restrict__ Ph, int L, int nkp, int iso, int per) {
  constexpr int LANES = Num<false>::LANES, NTHR = 256;
  extern __shared__ float4 sm4[];
  const int tid = threadIdx.x, n = 1 << L, nt = n / kTile;
  const int tile = blockIdx.x;
  const int TX = tile % nt, TY = (tile / nt) % nt, TZ = tile / (nt * nt);
  const size_t leaves = (size_t)1 << (3 * L);
  unsigned* slot_leaf = reinterpret_cast<unsigned*>(sm4 + 2 * kStage);   // [216]
  for (int slot = tid; slot < kSlots; slot += NTHR) {
    const int ux = TX * kTile - 1 + slot % kHaloN, uy = TY * kTile - 1 + (slot / kHaloN) % kHaloN,
              uz = TZ * kTile - 1 + slot / (kHaloN * kHaloN);
    const bool inbox = (unsigned)ux < (unsigned)n && (unsigned)uy < (unsigned)n && (unsigned)uz < (unsigned)n;
    slot_leaf[slot] = inbox || !iso ? morton(ux & (n - 1), uy & (n - 1), uz & (n - 1)) : (unsigned)leaves;
  }
  __syncthreads();
  auto load = [&](int chunk, int st) {
    float4* to = sm4 + st * kStage;
    const float4* Kc = K + (size_t)chunk * kKernels * 32;
    for (int i = tid; i < kKernels * 32; i += NTHR) tc::cp_async16_full(tc::smem_u32(to + i), Kc + i);
    const char* src = reinterpret_cast<const char*>(Mh) + (size_t)chunk * (leaves + 1) * 128;
    for (int i = tid; i < kSlots * 8; i += NTHR)
      tc::cp_async16_full(tc::smem_u32(to + kKernels * 32 + i), src + (size_t)slot_leaf[i >> 3] * 128 + (i & 7) * 16);
    tc::cp_async_commit();
  };
  const int chunks = nkp / LANES, c_end = min(chunks, ((int)blockIdx.y + 1) * per);
  int chunk = blockIdx.y * per;
  load(chunk, 0);
#pragma unroll 1
  for (int st = 0; chunk < c_end; ++chunk, st ^= 1) {
  if (chunk + 1 < c_end) {
    load(chunk + 1, st ^ 1);
    tc::cp_async_wait<1>();
  } else {
    tc::cp_async_wait<0>();
  }
  __syncthreads();
  const float4* sK = sm4 + st * kStage;     // [14][32]
  const float4* sM = sK + kKernels * 32;    // [216][8]
    const int fr = tid & 15, ty = (tid >> 4) & 3, tz = tid >> 6;
    const float2* halo = reinterpret_cast<const float2*>(sM) + fr;
    float2 tot[4][4];
    auto kernel = [&](int o, float2 (&k)[4]) {
      const float4 ka = sK[o * 32 + fr], kb = sK[o * 32 + 16 + fr];
      k[0] = make_float2(ka.x, ka.y);
      k[1] = make_float2(ka.z, ka.w);
      k[2] = make_float2(kb.x, kb.y);
      k[3] = make_float2(kb.z, kb.w);
    };
    auto row = [&](int oy, int oz, float2 (&m)[kHaloN]) {
      const float2* m0 = halo + ((tz + 1 + oz) * kHaloN + ty + 1 + oy) * kHaloN * LANES;
#pragma unroll
      for (int h = 0; h < kHaloN; ++h) m[h] = m0[h * LANES];
    };
    float2 mp[kHaloN], mm[kHaloN], k[4];
    row(0, 0, mp);
    kernel(13, k);                                             // the leaf itself
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int f = 0; f < 4; ++f)
        tot[j][f] = make_float2(fmaf(-k[f].y, mp[j + 1].y, k[f].x * mp[j + 1].x),
                                fmaf(k[f].y, mp[j + 1].x, k[f].x * mp[j + 1].y));
    // Phi's kernel is even and g's odd, so K^_{-o} = s conj(K^_o) (s = 1, -1)
    // and with M+ = m^_{T+o}, M- = m^_{T-o}, K^_o = a + ib the pair's terms are
    // a (M+ + s M-) + i b (M+ - s M-): 20 instructions for the 4 fields
    // instead of 32
    auto pairs = [&](int oy, int oz, int oxs) {                 // x offsets -1 .. oxs of rows (oy, oz), -(oy, oz)
#pragma unroll
      for (int ox = -1; ox <= 1; ++ox) {
        if (ox > oxs) continue;
        kernel((oz + 1) * 9 + (oy + 1) * 3 + ox + 1, k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 p = mp[j + 1 + ox], q = mm[j + 1 - ox];
          const float2 su = make_float2(p.x + q.x, p.y + q.y), di = make_float2(p.x - q.x, p.y - q.y);
          tot[j][0].x = fmaf(k[0].x, su.x, tot[j][0].x);
          tot[j][0].y = fmaf(k[0].x, su.y, tot[j][0].y);
          tot[j][0].x = fmaf(-k[0].y, di.y, tot[j][0].x);
          tot[j][0].y = fmaf(k[0].y, di.x, tot[j][0].y);
#pragma unroll
          for (int f = 1; f < 4; ++f) {
            tot[j][f].x = fmaf(k[f].x, di.x, tot[j][f].x);
            tot[j][f].y = fmaf(k[f].x, di.y, tot[j][f].y);
            tot[j][f].x = fmaf(-k[f].y, su.y, tot[j][f].x);
            tot[j][f].y = fmaf(k[f].y, su.x, tot[j][f].y);
          }
        }
      }
    };
#pragma unroll
    for (int h = 0; h < kHaloN; ++h) mm[h] = mp[h];
    pairs(0, 0, -1);
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {                               // rows (-1, -1), (0, -1), (1, -1), (-1, 0)
      const int oz = r < 3 ? -1 : 0, oy = r < 3 ? r - 1 : -1;
      row(oy, oz, mp);
      row(-oy, -oz, mm);
      pairs(oy, oz, 1);
    }
    float2* out = reinterpret_cast<float2*>(Ph);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t leaf = morton(TX * kTile + j, TY * kTile + ty, TZ * kTile + tz);
#pragma unroll
      for (int f = 0; f < 4; ++f) out[(leaf * 4 + f) * nkp + (size_t)chunk * LANES + fr] = tot[j][f];
    }
  __syncthreads();                          // this stage is refilled next
  }
}
constexpr size_t kMacSmem = sizeof(float4) * 2 * kStage + sizeof(unsigned) * kSlots;

template <int S, bool DFA>
size_t fwd_smem() {
  constexpr int NB = Shape<S>::NB, NM = Shape<S>::NM;
  return sizeof(typename Num<DFA>::cplx) * NB * (S * S * Shape<S>::PS + S * NM * S);
}
template <int S, bool DFA>
size_t inv_smem(int p) {
  constexpr int IB = kItems<S, DFA>, NM = Shape<S>::NM, X3 = S * S * Shape<S>::PS;
  const size_t real = sizeof(typename Num<DFA>::real), cplx = sizeof(typename Num<DFA>::cplx);
  const size_t t = cplx * IB * (X3 + S * NM * S), l2p = real * IB * (p * p * p + p * p * S + p * S * S);
  return (t > l2p ? t : l2p) + real * IB * X3;
}

template <int S, bool DFA>
cudaError_t fwd_as(Plan& P, const float* rho, cudaStream_t s) {
  const unsigned leaves = 1u << (3 * P.L);
  k_ns_fwd<S, DFA><<<leaves / Shape<S>::NB, Shape<S>::THR, fwd_smem<S, DFA>(), s>>>(rho, P.d_mean, P.N, P.L,
                                                                                            P.ns_tw, P.ns_M);
  return cudaGetLastError();
}
// The sums: like the source spectra they need the density only.
template <int S>
cudaError_t sums_as(Plan& P, cudaStream_t s) {
  const int nt = (1 << P.L) / kTile, ch = chunks_of(S, false), nkp = ch * Num<false>::LANES;
  const int tiles = nt * nt * nt, fit = (int)((long)tiles * ch / (4 * P.num_sms));
  const int per = fit < 1 ? 1 : (fit < kChunks ? fit : kChunks);
  k_ns_mac<<<dim3(tiles, (ch + per - 1) / per), 256, kMacSmem, s>>>(static_cast<const float4*>(P.ns_K), P.ns_M, P.ns_P,
                                                                   P.L, nkp, P.iso, per);
  return cudaGetLastError();
}
template <int S, bool DFA>
cudaError_t rest_as(Plan& P, float* phi, float* acc, cudaStream_t s) {
  const unsigned leaves = 1u << (3 * P.L);
  const int nkp = chunks_of(S, false) * Num<false>::LANES;
  k_ns_inv<S, DFA><<<leaves * 4 / kItems<S, DFA>, Shape<S>::threads(kItems<S, DFA>), inv_smem<S, DFA>(P.p), s>>>(
      P.ns_P, nkp, (int)(inv_smem<S, DFA>(P.p) - sizeof(typename Num<DFA>::real) * kItems<S, DFA> * S * S * Shape<S>::PS), P.N,
      P.p, P.F[P.L], P.F64[P.L], P.w_p2m, P.ns_tw, phi, acc);
  return cudaGetLastError();
}

template <int S>
cudaError_t kernels_s(Plan& P, cudaStream_t s) {
  constexpr int NM = Shape<S>::NM;
  // the target spectra's space holds the half-transformed kernels meanwhile
  float4* scratch = static_cast<float4*>(P.ns_P);
  k_ns_planes<S><<<dim3(NM, kKernels * 4), kPlaneThr, 0, s>>>(P.near_tab, P.ns_tw, scratch);
  k_ns_lines<S><<<dim3((NM * S + 127) / 128, kKernels * 4), 128, 0, s>>>(scratch, P.ns_tw, static_cast<float*>(P.ns_K));
  return cudaGetLastError();
}

template <typename F>
cudaError_t opt_in(F* f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int S>
cudaError_t setup_s() {
  cudaError_t e;
  if constexpr (!kWideField<S>) {
    if ((e = opt_in(k_ns_fwd<S, false>, fwd_smem<S, false>())) != cudaSuccess) return e;
    if ((e = opt_in(k_ns_inv<S, false>, inv_smem<S, false>(kMaxOrder))) != cudaSuccess) return e;
  }
  if ((e = opt_in(k_ns_fwd<S, true>, fwd_smem<S, true>())) != cudaSuccess) return e;
  if ((e = opt_in(k_ns_inv<S, true>, inv_smem<S, true>(kMaxOrder))) != cudaSuccess) return e;
  return opt_in(k_ns_mac, kMacSmem);
}

}  // namespace

bool near_spec_shape(const Plan& P) { return P.S == 4 || P.S == 6 || P.S == 8 || P.S == 16; }

void near_spec_bytes(const Plan& P, size_t& nK, size_t& nM, size_t& nP) {
  const size_t leaves = (size_t)1 << (3 * P.L), ch = chunks_of(P.S, false);
  nK = ch * kKernels * 512;
  nM = ch * (leaves + 1) * 128;
  nP = leaves * 4 * ch * 128;
}

cudaError_t setup_near_spec(const Plan& P) {
  switch (P.S) {
    case 4: return setup_s<4>();
    case 6: return setup_s<6>();
    case 8: return setup_s<8>();
    case 16: return setup_s<16>();
    default: return cudaSuccess;
  }
}

cudaError_t launch_near_spec_kernels(Plan& P, cudaStream_t s) {
  switch (P.S) {
    case 4: return kernels_s<4>(P, s);
    case 6: return kernels_s<6>(P, s);
    case 8: return kernels_s<8>(P, s);
    case 16: return kernels_s<16>(P, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_near_spec_sums(Plan& P, const float* rho, cudaStream_t s) {
  cudaError_t e;
  switch (P.S) {
    case 4: e = fwd_as<4, true>(P, rho, s); return e != cudaSuccess ? e : sums_as<4>(P, s);
    case 6: e = fwd_as<6, true>(P, rho, s); return e != cudaSuccess ? e : sums_as<6>(P, s);
    case 8:
      e = P.near_fft ? fwd_as<8, false>(P, rho, s) : fwd_as<8, true>(P, rho, s);
      return e != cudaSuccess ? e : sums_as<8>(P, s);
    case 16: e = fwd_as<16, true>(P, rho, s); return e != cudaSuccess ? e : sums_as<16>(P, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_near_spec(Plan& P, float* phi, float* acc, cudaStream_t s) {
  switch (P.S) {
    case 4: return rest_as<4, true>(P, phi, acc, s);
    case 6: return rest_as<6, true>(P, phi, acc, s);
    case 8: return P.near_fft ? rest_as<8, false>(P, phi, acc, s) : rest_as<8, true>(P, phi, acc, s);
    case 16: return rest_as<16, true>(P, phi, acc, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fmm
