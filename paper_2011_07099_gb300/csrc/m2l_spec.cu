// M2L by spectral products (CUDA cores, FP32 or double-float).
//
// Eq. fmm2 (Sec. 3) for one target node T and one interaction offset o is the
// linear convolution of the source gridlet with the level table,
//   F_T[r] += sum_s Tab[o p + r - s] M_{T-o}[s],   r, s in [0, p)^3,
// whose lags r - s lie in [-(p-1), p-1]^3.  On a zero-padded grid of
// NM = 2p - 1 points per axis that is a circular convolution with no lag
// wrapped onto another, so with M^ the NM^3 transform of a node's gridlet and
// K^_o that of the offset's table window,
//   F^_T(k) = sum_o K^_o(k) M^_{T-o}(k):
// one complex multiply-add per frequency, offset and field where the dense
// contraction takes p^3 x p^3 terms (p = 6: 11 616 FP32 multiply-adds per
// offset and node against 186 624).  Real input: kx in [0, p - 1] only,
// NK = NM^2 p frequencies.  (The paper's HPM uses the same idea over a whole
// parent block, Sec. 2.)
//
// Kernels (each launch takes all levels of one arithmetic together, so a
// small tree costs three launches and not three per level):
//   k_spec_kernel  plan time: K^_o of every offset and field
//   k_spec_fwd     per node: M^ of its gridlet, separable line DFTs
//   k_spec_mac     per (tile of 4^3 target nodes, chunk of frequencies): the
//                  189-offset sums of the 4 fields
//   k_spec_inv     per node: the 4 fields' p^3 values
// Arithmetic: FP32 at the fine levels; at the wide levels (FP64 local fields)
// values, twiddles and sums are double-float, and products too but for level 3
// of orders < kWideOrder: there a row's products run in FP32 chains of at most
// 12 terms on the high halves of the source spectra (mac_df, ROWS).
// Measured (dense kernels of m2l_fp32.cu before -> here, with transforms):
// 256^3 p = 6, levels 4 + 5 FP32 87.1 -> 6.6 ms (plain form; 4.5 ms with FP32
// transforms, sums 4.1 ms), levels 2 + 3 1.95 -> 0.35 ms; 512^3 p = 8, levels
// 2 - 4 in double-float 344 -> 11 ms, level 6 against the tensor cores 281 ->
// 77 ms; 128^3 p = 6 isolated with 16-cell leaves 10.2 -> 0.76 ms; 32^3 p = 4
// 251 -> 75 us.
#include "fmm_internal.cuh"
#include "spec.cuh"
#include "tc_ptx.cuh"

namespace fmm {
namespace {

using spec::chunks_of;
using spec::forward_line;
using spec::inverse_line;
using spec::inverse_real_line;
using spec::lanes;
using spec::narrow;
using spec::Num;
using spec::Shape;
using spec::Twiddle;
using spec::widen;

constexpr int kTile = 4;                  // target nodes per tile side
constexpr int kHaloN = 8;                 // source nodes per halo side: T - 2 .. T + 5 of the tile's first node
constexpr int kSlots = kHaloN * kHaloN * kHaloN;
constexpr int kOff3 = 343;                // offsets o in [-3, 3]^3
constexpr int kHalfN = 6;                 // source planes of half a tile

// One level of a launch.
struct SpecLevel {
  const float* M;          // gridlet masses
  const double* M64;       // their FP64 copy (wide levels of the high orders) or null
  void* Mh;                // spectra [chunk][node (+ 1 all-zero slot)][lanes]
  void* Ph;                // target spectra [node][4][NKP]
  const void* K;           // kernel spectra [chunk][343][...]
  float* F;
  double* F64;             // FP64 local field (wide levels) or null
  int level;
  int first;               // first block of this level
  size_t nodes;            // gridlets of the level
};
struct SpecArgs {
  SpecLevel lev[kMaxLevel + 1];
  int n;                   // levels in the launch
  int chunks;              // frequency chunks
  int nkp;                 // padded frequencies
  int iso;
  int rows;                // level 3 from FP32 masses: row chains (mac_df)
  const float4* tw;        // (cos hi, cos lo, sin hi, sin lo) of 2 pi j / NM
};

__device__ __forceinline__ const SpecLevel& level_of(const SpecArgs& A, int block) {
  int i = 0;
  while (i + 1 < A.n && block >= A.lev[i + 1].first) ++i;
  return A.lev[i];
}

// ------------------------------------------------------------ plan time
// K^[chunk][o][...]: FP32 as [2 field pairs][16] float4 (re, im of two
// fields), double-float as [4 fields][8] float4 (re hi, re lo, im hi, im lo).
// CTA (o, field): window values from the level table (hi + lo), three
// separable passes in double-float (the spectra are stored as FP32 or as
// double-float pairs; in FP64, at 1/64 of the FP32 rate, a level of order 6
// took 0.37 ms); the inverse transform's 1/NM^3 is folded in.
template <int P, bool DF>
__global__ void __launch_bounds__(128) k_spec_kernel(const float4* __restrict__ tab, const float4* __restrict__ tab_lo,
                                                     const float4* __restrict__ twg, float* __restrict__ K) {
  using T = Num<true>;
  constexpr int NM = Shape<P>::NM, HW = 4 * P - 1, E = 8 * P - 1, LANES = Num<DF>::LANES;
  const int o = blockIdx.x, f = blockIdx.y, tid = threadIdx.x;
  const int ox = o % 7 - 3, oy = (o / 7) % 7 - 3, oz = o / 49 - 3;
  if (abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1) return;    // near nodes: never used
  __shared__ float4 tw[NM];
  extern __shared__ float4 sm4[];
  float4* T1 = sm4;                       // [z][y][kx]
  float4* T2 = sm4 + NM * NM * P;         // [z][ky][kx]
  if (tid < NM) tw[tid] = __ldg(twg + tid);
  const Twiddle<true, P> wt(twg, tw);
  __syncthreads();
  auto lag = [](int v) { return v < P ? v : v - NM; };
  for (int l = tid; l < NM * NM; l += blockDim.x) {            // x: line (vz, vy)
    const int vy = l % NM, vz = l / NM;
    const size_t row = ((size_t)(oz * P + lag(vz) + HW) * E + (oy * P + lag(vy) + HW)) * E + ox * P + HW;
    float2 x[NM];
#pragma unroll
    for (int vx = 0; vx < NM; ++vx)
      x[vx] = make_float2(__ldg(reinterpret_cast<const float*>(tab + row + lag(vx)) + f),
                          __ldg(reinterpret_cast<const float*>(tab_lo + row + lag(vx)) + f));
    spec::forward_real_full_line<true, P>(x, wt,
                                          [&](int k, float2 re, float2 im) { T1[l * P + k] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < NM * P; l += blockDim.x) {             // y: line (vz, kx)
    const int kx = l % P, vz = l / P;
    float2 xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float4 c = T1[(vz * NM + s) * P + kx];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    // the forward transform at k is the inverse one at NM - k
    inverse_line<true, P, true>(xr, xi, wt, [&](int z, float2 re, float2 im) {
      T2[(vz * NM + (z ? NM - z : 0)) * P + kx] = T::pack(re, im);
    });
  }
  __syncthreads();
  const float2 scale = df_from_double(1.0 / ((double)NM * NM * NM));
  for (int q = tid; q < NM * P; q += blockDim.x) {             // z: line (ky, kx)
    float2 xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float4 c = T2[s * NM * P + q];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    inverse_line<true, P, true>(xr, xi, wt, [&](int z, float2 re, float2 im) {
      const int k = (z ? NM - z : 0) * NM * P + q;
      float2 a = T::zero(), b = T::zero();
      T::mac(a, scale.x, scale.y, re);
      T::mac(b, scale.x, scale.y, im);
      a = T::done(a);
      b = T::done(b);
      const size_t base = ((size_t)(k / LANES) * kOff3 + o) * (DF ? 16 : 8) * LANES;   // floats
      const int l = k % LANES;
      if (DF)
        reinterpret_cast<float4*>(K + base)[f * LANES + l] = T::pack(a, b);
      else
        reinterpret_cast<float2*>(K + base)[((f / 2) * LANES + l) * 2 + (f & 1)] = make_float2(a.x, b.x);
    });
  }
}

// ------------------------------------------------------------- transforms
// Nodes per CTA of the inverse transforms (4 fields each).
template <int P>
constexpr int kInvNodes = P >= 5 ? 1 : (P == 4 ? 2 : (P == 3 ? 4 : 8));

// DFS: double-float storage (the wide levels); DFA: double-float arithmetic
// (always with DFS; with FP32 storage in the plain form, whose transforms then
// round once, on store; the mixed forms transform in FP32).
// Source spectra.  CTA: NB nodes; passes x, y, z through shared memory.
template <int P, bool DFS, bool DFA>
__global__ void __launch_bounds__(Shape<P>::THR) k_spec_fwd(const __grid_constant__ SpecArgs A) {
  using T = Num<DFA>;
  using store = Num<DFS>;
  using real = typename T::real;
  using cplx = typename T::cplx;
  constexpr int NM = Shape<P>::NM, NB = Shape<P>::NB, P3 = P * P * P, PS = Shape<P>::PS,
                LANES = store::LANES;
  extern __shared__ float4 sm4[];
  __shared__ float4 tw[NM];
  cplx* t1 = reinterpret_cast<cplx*>(sm4);                 // [NB][z][y][kx]
  cplx* t2 = t1 + NB * P * P * PS;                         // [NB][z][ky][kx]
  real* in = reinterpret_cast<real*>(t2 + NB * P * NM * P);   // [NB][z][y][x]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const SpecLevel& V = level_of(A, blockIdx.x);
  const size_t node0 = (size_t)(blockIdx.x - V.first) * NB, nodes = V.nodes;
  if (DFA && tid < NM) tw[tid] = __ldg(A.tw + tid);
  const Twiddle<DFA, P> wt(A.tw, tw);
  for (int i = tid; i < NB * P3; i += nthr) {
    real& v = in[(i / P) * PS + i % P];
    if constexpr (DFS)
      v = V.M64 ? df_from_double(__ldg(V.M64 + node0 * P3 + i)) : make_float2(__ldg(V.M + node0 * P3 + i), 0.f);
    else
      v = widen<DFA>(__ldg(V.M + node0 * P3 + i));
  }
  __syncthreads();
  for (int l = tid; l < NB * P * P; l += nthr) {           // x: P reals -> P frequencies
    real x[P];
#pragma unroll
    for (int s = 0; s < P; ++s) x[s] = in[l * PS + s];
    forward_line<DFA, P, true>(x, x, wt, [&](int k, real re, real im) { t1[l * PS + k] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < NB * P * P; l += nthr) {           // y: line (node, z, kx)
    const int kx = l % P, nz = l / P;
    real xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const cplx c = t1[(nz * P + s) * PS + kx];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    forward_line<DFA, P, false>(xr, xi, wt, [&](int k, real re, real im) { t2[(nz * NM + k) * P + kx] = T::pack(re, im); });
  }
  __syncthreads();
  typename store::cplx* Mh = reinterpret_cast<typename store::cplx*>(V.Mh);
  for (int l = tid; l < NB * NM * P; l += nthr) {          // z: line (node, ky, kx)
    const int q = l % (NM * P), nb = l / (NM * P);
    real xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const cplx c = t2[(nb * P + s) * NM * P + q];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    forward_line<DFA, P, false>(xr, xi, wt, [&](int kz, real re, real im) {
      const int k = kz * NM * P + q;
      Mh[((size_t)(k / LANES) * (nodes + 1) + node0 + nb) * LANES + k % LANES] =
          store::pack(narrow<DFS, DFA>(re), narrow<DFS, DFA>(im));
    });
  }
}

// Local fields from the target spectra.  CTA: NB nodes, 4 fields each.
template <int P, bool DFS, bool DFA>
__global__ void __launch_bounds__(Shape<P>::threads(4 * kInvNodes<P>)) k_spec_inv(const __grid_constant__ SpecArgs A) {
  using T = Num<DFA>;
  using store = Num<DFS>;
  using real = typename T::real;
  using cplx = typename T::cplx;
  constexpr int NM = Shape<P>::NM, NB = kInvNodes<P>, P3 = P * P * P, PS = Shape<P>::PS;
  extern __shared__ float4 sm4[];
  __shared__ float4 tw[NM];
  cplx* t1 = reinterpret_cast<cplx*>(sm4);                 // [NB][4][z][ky][kx]
  cplx* t2 = t1 + NB * 4 * P * NM * P;                     // [NB][4][z][y][kx]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const SpecLevel& V = level_of(A, blockIdx.x);
  const size_t node0 = (size_t)(blockIdx.x - V.first) * NB;
  if (DFA && tid < NM) tw[tid] = __ldg(A.tw + tid);
  const Twiddle<DFA, P> wt(A.tw, tw);
  __syncthreads();
  const typename store::cplx* Ph = reinterpret_cast<const typename store::cplx*>(V.Ph) + node0 * 4 * A.nkp;
  for (int l = tid; l < NB * 4 * NM * P; l += nthr) {      // z: line (node, f, ky, kx), NM -> P
    const int q = l % (NM * P), nf = l / (NM * P);
    real xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const typename store::cplx c = __ldg(Ph + (size_t)nf * A.nkp + s * NM * P + q);
      xr[s] = widen<DFA>(store::re(c));
      xi[s] = widen<DFA>(store::im(c));
    }
    inverse_line<DFA, P>(xr, xi, wt, [&](int z, real re, real im) { t1[(nf * P + z) * NM * P + q] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < NB * 4 * P * P; l += nthr) {       // y: line (node, f, z, kx), NM -> P
    const int kx = l % P, nfz = l / P;
    real xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const cplx c = t1[(nfz * NM + s) * P + kx];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    inverse_line<DFA, P>(xr, xi, wt, [&](int y, real re, real im) { t2[(nfz * P + y) * PS + kx] = T::pack(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < NB * 4 * P * P; l += nthr) {       // x: line (node, f, z, y), half spectrum -> P reals
    real xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const cplx c = t2[l * PS + s];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    inverse_real_line<DFA, P>(xr, xi, wt, [&](int x, real v) {
      const size_t g = node0 * 4 * P3 + (size_t)l * P + x;
      if constexpr (DFS) {
        const double d = df_to_double(v);
        V.F64[g] = d;
        V.F[g] = (float)d;
      } else {
        V.F[g] = narrow<DFS, DFA>(v);
      }
    });
  }
}

// ---------------------------------------------------------- spectral sums
// CTA: a tile of 4^3 target nodes (2 parents per axis) x one chunk of
// frequencies.  The sources of the tile's interaction zones are the 8^3 nodes
// T0 - 2 .. T0 + 5 (parents' neighbours' children), staged in shared memory.
// A thread holds one frequency of a row of 4 targets along x (4 fields each);
// the lanes of a warp are the chunk's frequencies times rows of the same
// child type (cy, cz), so the warp's kernel spectra loads are shared by its
// rows.  Per (oy, oz) a thread loads its 8 source spectra once and runs the
// 7 x offsets over them: 8 shared-memory loads and 14 (FP32) kernel loads
// feed 384 multiply-adds, so the FP32 pipe is the bound.
// MODE 0: levels >= 3 (child c takes o in [-3, 2] or [-2, 3] per axis);
// 1: level 2, periodic (o in [-1, 2]); 2: level 2, isolated (o in [-3, 3]).
template <int MODE>
__device__ __forceinline__ constexpr bool allowed(int c, int o) {
  return MODE == 0 ? (c ? o >= -2 : o <= 2) : (MODE == 1 ? o >= -1 && o <= 2 : true);
}

template <int MODE>
__device__ __forceinline__ void mac_fp32(const float2* __restrict__ halo, const float4* __restrict__ K, int ty, int tz,
                                         float2 (&tot)[4][4]) {
  const int cy = ty & 1, cz = tz & 1;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int f = 0; f < 4; ++f) tot[j][f] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int oz = -3; oz <= 3; ++oz) {
    const int hz = tz + 2 - oz;
    if (!allowed<MODE>(cz, oz) || hz < 0 || hz >= kHaloN) continue;
    // a plane's sums stay apart from the total: the running FP32 sums are no
    // longer than one plane's terms.  (A stage per row as well took 10 % off the
    // error of 32^3, p = 2 .. 4 and 7 % more time of this kernel.)
    float2 acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int f = 0; f < 4; ++f) acc[j][f] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int oy = -3; oy <= 3; ++oy) {
      const int hy = ty + 2 - oy;
      if (!allowed<MODE>(cy, oy) || hy < 0 || hy >= kHaloN) continue;
      const bool near = oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1;
      const float2* row = halo + (hz * kHaloN + hy) * kHaloN * 16;
      float2 m[kHaloN];
#pragma unroll
      for (int h = 0; h < kHaloN; ++h) m[h] = row[h * 16];
      const float4* Kr = K + ((oz + 3) * 49 + (oy + 3) * 7) * 32;
      auto terms = [&](int ox) {                       // ox is a constant after unrolling
        const float4 ka = __ldg(Kr + (ox + 3) * 32), kb = __ldg(Kr + (ox + 3) * 32 + 16);
        const float2 k[4] = {make_float2(ka.x, ka.y), make_float2(ka.z, ka.w), make_float2(kb.x, kb.y),
                             make_float2(kb.z, kb.w)};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int h = j + 2 - ox;
          if (!allowed<MODE>(j & 1, ox) || h < 0 || h >= kHaloN) continue;
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            acc[j][f].x = fmaf(k[f].x, m[h].x, acc[j][f].x);
            acc[j][f].y = fmaf(k[f].x, m[h].y, acc[j][f].y);
            acc[j][f].x = fmaf(-k[f].y, m[h].y, acc[j][f].x);
            acc[j][f].y = fmaf(k[f].y, m[h].x, acc[j][f].y);
          }
        }
      };
      terms(-3);
      terms(-2);
      if (!near) {
        terms(-1);
        terms(0);
        terms(1);
      }
      terms(2);
      terms(3);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        tot[j][f].x += acc[j][f].x;
        tot[j][f].y += acc[j][f].y;
      }
  }
}

// Double-float, one field of a row of 4 targets per thread: (re hi, re lo, im
// hi, im lo) sums.  The kernel values of the row's 7 x offsets stay in
// registers while the 8 source spectra pass by, and one field per thread keeps
// the unrolled row within the instruction cache (4 fields per thread waited for
// instruction fetch most of the time).
// ROWS: the sums of one (oy, oz) row run as FP32 multiply-add chains (at most
// 12 terms) and are then added to the double-float total, the low halves of
// the kernel values gathered beside them: 2 instructions per product instead
// of 12, for the level whose masses are FP32 (level 3 of orders < kWideOrder).
template <int MODE, bool ROWS>
__device__ __forceinline__ void mac_df(const float4* __restrict__ halo, const float4* __restrict__ K, int ty, int cz,
                                       float4 (&tot)[4]) {
  const int cy = ty & 1;
#pragma unroll
  for (int j = 0; j < 4; ++j) tot[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int oz = -3; oz <= 3; ++oz) {
    const int hz = cz + 2 - oz;                   // of the 6 source planes of this half tile
    if (!allowed<MODE>(cz, oz) || hz < 0 || hz >= kHalfN) continue;
#pragma unroll 1
    for (int oy = -3; oy <= 3; ++oy) {
      const int hy = ty + 2 - oy;
      if (!allowed<MODE>(cy, oy) || hy < 0 || hy >= kHaloN) continue;
      const bool near = oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1;
      const float4* row = halo + (hz * kHaloN + hy) * kHaloN * 8;
      const float4* Kr = K + ((oz + 3) * 49 + (oy + 3) * 7) * 32;
      float4 k[7];
#pragma unroll
      for (int i = 0; i < 7; ++i)
        k[i] = near && i >= 2 && i <= 4 ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(Kr + i * 32);
      float2 part[4];
      if (ROWS) {
#pragma unroll
        for (int j = 0; j < 4; ++j) part[j] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int h = 0; h < kHaloN; ++h) {
        const float4 m = row[h * 8];
        const float2 mr = make_float2(m.x, m.y), mi = make_float2(m.z, m.w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int ox = j + 2 - h;
          if (ox < -3 || ox > 3 || !allowed<MODE>(j & 1, ox)) continue;
          if (ox >= -1 && ox <= 1 && near) continue;
          const float4 q = k[ox + 3];
          if (ROWS) {
            part[j].x = fmaf(-q.z, m.z, fmaf(q.x, m.x, part[j].x));
            part[j].y = fmaf(q.z, m.x, fmaf(q.x, m.z, part[j].y));
            tot[j].y = fmaf(-q.w, m.z, fmaf(q.y, m.x, tot[j].y));
            tot[j].w = fmaf(q.w, m.x, fmaf(q.y, m.z, tot[j].w));
          } else {
            float2 re = make_float2(tot[j].x, tot[j].y), im = make_float2(tot[j].z, tot[j].w);
            Num<true>::mac(re, q.x, q.y, mr);
            Num<true>::mac(im, q.x, q.y, mi);
            Num<true>::mac(re, -q.z, -q.w, mi);
            Num<true>::mac(im, q.z, q.w, mr);
            tot[j] = make_float4(re.x, re.y, im.x, im.y);
          }
        }
      }
      if (ROWS) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 a = df_two_sum(tot[j].x, part[j].x), b = df_two_sum(tot[j].z, part[j].y);
          tot[j] = make_float4(a.x, __fadd_rn(tot[j].y, a.y), b.x, __fadd_rn(tot[j].w, b.y));
        }
      }
    }
  }
}

constexpr int kMacThr = 256;        // FP32: 16 frequencies x 16 rows
constexpr int kMacThrDf = 256;      // double-float: 8 frequencies x 8 rows x 4 fields

// The tile's source spectra (z planes z0 .. z0 + nz - 1 of the halo), 128 bytes
// per slot, into shared memory.
__device__ __forceinline__ void load_halo(const SpecLevel& V, int iso, int tile, int z0, int nz, int chunk, float4* sm,
                                          int tid, int nthr) {
  const int n = 1 << V.level, nt = n / kTile;
  const int TX = tile % nt, TY = (tile / nt) % nt, TZ = tile / (nt * nt);
  const size_t nodes = (size_t)1 << (3 * V.level);
  const char* src = reinterpret_cast<const char*>(V.Mh) + (size_t)chunk * (nodes + 1) * 128;
  for (int i = tid; i < nz * kHaloN * kHaloN * 8; i += nthr) {
    const int slot = i >> 3, part = i & 7;
    const int ux = TX * kTile - 2 + (slot & 7), uy = TY * kTile - 2 + ((slot >> 3) & 7),
              uz = TZ * kTile - 2 + z0 + (slot >> 6);
    const bool inbox = (unsigned)ux < (unsigned)n && (unsigned)uy < (unsigned)n && (unsigned)uz < (unsigned)n;
    const size_t node = inbox || !iso ? morton(ux & (n - 1), uy & (n - 1), uz & (n - 1)) : nodes;
    tc::cp_async16_full(tc::smem_u32(sm + i), src + node * 128 + part * 16);
  }
  tc::cp_async_commit();
  tc::cp_async_wait<0>();
  __syncthreads();
}

__global__ void __launch_bounds__(kMacThr, 2) k_spec_mac(const __grid_constant__ SpecArgs A) {
  extern __shared__ float4 sm4[];
  const int tid = threadIdx.x;
  const SpecLevel& V = level_of(A, blockIdx.x);
  const int nt = (1 << V.level) / kTile, tiles = nt * nt * nt;
  const int local = blockIdx.x - V.first, tile = local % tiles, chunk = local / tiles;
  const int TX = tile % nt, TY = (tile / nt) % nt, TZ = tile / (nt * nt);
  load_halo(V, A.iso, tile, 0, kHaloN, chunk, sm4, tid, kMacThr);
  // lane: frequency and the y half of the row; warp: child type (cy, cz) and the z half
  const int lane = tid & 31, warp = tid >> 5, fr = lane & 15;
  const int ty = (warp & 1) + 2 * (lane >> 4), tz = ((warp >> 1) & 1) + 2 * (warp >> 2);
  const float4* K = reinterpret_cast<const float4*>(V.K) + (size_t)chunk * kOff3 * 32 + fr;
  float2 tot[4][4];
  mac_fp32<0>(reinterpret_cast<const float2*>(sm4) + fr, K, ty, tz, tot);   // level 2 is always wide
  float2* Ph = reinterpret_cast<float2*>(V.Ph);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const size_t node = morton(TX * kTile + j, TY * kTile + ty, TZ * kTile + tz);
#pragma unroll
    for (int f = 0; f < 4; ++f) Ph[(node * 4 + f) * A.nkp + (size_t)chunk * 16 + fr] = tot[j][f];
  }
}

// CTA: half a tile (2 target planes, 6 source planes), so that the few tiles
// of levels 2 and 3 make CTAs enough to load the SMs evenly (32^3, p = 4: 225
// whole tiles x chunks left one or two CTAs per SM).
__global__ void __launch_bounds__(kMacThrDf, 4) k_spec_mac_df(const __grid_constant__ SpecArgs A) {
  extern __shared__ float4 sm4[];
  const int tid = threadIdx.x;
  const SpecLevel& V = level_of(A, blockIdx.x);
  const int nt = (1 << V.level) / kTile, tiles = nt * nt * nt;
  const int local = blockIdx.x - V.first, zh = local & 1, tile = (local >> 1) % tiles, chunk = (local >> 1) / tiles;
  const int TX = tile % nt, TY = (tile / nt) % nt, TZ = tile / (nt * nt);
  load_halo(V, A.iso, tile, 2 * zh, kHalfN, chunk, sm4, tid, kMacThrDf);
  // lane: frequency, y half of the row, low bit of the field; warp: child type (cy, cz), high bit of the field
  const int lane = tid & 31, warp = tid >> 5, fr = lane & 7;
  const int ty = (warp & 1) + 2 * ((lane >> 3) & 1), cz = (warp >> 1) & 1, f = 2 * (warp >> 2) + (lane >> 4);
  const int tz = 2 * zh + cz;
  const float4* K = reinterpret_cast<const float4*>(V.K) + (size_t)chunk * kOff3 * 32 + f * 8 + fr;
  float4 tot[4];
  if (V.level > 2) {
    if (A.rows)
      mac_df<0, true>(sm4 + fr, K, ty, cz, tot);
    else
      mac_df<0, false>(sm4 + fr, K, ty, cz, tot);
  } else if (!A.iso) {
    mac_df<1, false>(sm4 + fr, K, ty, cz, tot);
  } else {
    mac_df<2, false>(sm4 + fr, K, ty, cz, tot);
  }
  float4* Ph = reinterpret_cast<float4*>(V.Ph);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const size_t node = morton(TX * kTile + j, TY * kTile + ty, TZ * kTile + tz);
    const float2 re = Num<true>::done(make_float2(tot[j].x, tot[j].y));
    const float2 im = Num<true>::done(make_float2(tot[j].z, tot[j].w));
    Ph[(node * 4 + f) * A.nkp + (size_t)chunk * 8 + fr] = make_float4(re.x, re.y, im.x, im.y);
  }
}

// Zeros in units of 16 bytes: ka at a, kb at b, and 8 at c, c + stride, ... (n
// times).  (Filling all of the spectra of 512^3, order 8 took 2 ms of a plan.)
__global__ void k_clear(float4* __restrict__ a, size_t ka, float4* __restrict__ b, size_t kb, char* __restrict__ c,
                        size_t stride, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < ka + kb + 8 * n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t j = i - ka - kb;                    // (used from there on)
    float4* to = i < ka ? a + i : (i < ka + kb ? b + (i - ka) : reinterpret_cast<float4*>(c + j / 8 * stride) + j % 8);
    *to = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

template <int P, bool DFA>
size_t fwd_smem() {
  constexpr int NB = Shape<P>::NB, NM = Shape<P>::NM;
  constexpr int X3 = P * P * Shape<P>::PS;
  return sizeof(typename Num<DFA>::cplx) * NB * (X3 + P * NM * P) + sizeof(typename Num<DFA>::real) * NB * X3;
}
template <int P, bool DFA>
size_t inv_smem() {
  constexpr int NB = kInvNodes<P>, NM = Shape<P>::NM;
  return sizeof(typename Num<DFA>::cplx) * NB * 4 * (P * NM * P + P * P * Shape<P>::PS);
}
constexpr size_t kMacSmem = (size_t)kSlots * 128;

// All spectral levels l0..l1 of one arithmetic, block ranges filled by `per`
// (blocks of a level); larger levels first.
template <typename PerLevel>
int fill(const Plan& Pl, bool df, int l0, int l1, SpecArgs& A, PerLevel per) {
  A.n = 0;
  A.chunks = chunks_of(Pl.p, df);
  A.nkp = A.chunks * lanes(df);
  A.iso = Pl.iso;
  A.rows = Pl.p < kWideOrder && Pl.S < kWideLeaf;
  A.tw = Pl.spec_tw;
  int blocks = 0;
  for (int l = l1; l >= l0; --l) {
    if (!Pl.spec_K[l] || wide_level(Pl, l) != df) continue;
    SpecLevel& V = A.lev[A.n++];
    V = {Pl.M[l], df ? Pl.M64[l] : nullptr, Pl.spec_M[l], Pl.spec_P[l], Pl.spec_K[l], Pl.F[l], Pl.F64[l], l, blocks,
         (size_t)1 << (3 * l)};
    blocks += per(l);
  }
  return blocks;
}

template <int P, bool DFS, bool DFA>
cudaError_t launch_as(Plan& Pl, int l0, int l1, cudaStream_t s) {
  SpecArgs A;
  int b = fill(Pl, DFS, l0, l1, A, [](int l) { return (1 << (3 * l)) / Shape<P>::NB; });
  if (!b) return cudaSuccess;
  k_spec_fwd<P, DFS, DFA><<<b, Shape<P>::THR, fwd_smem<P, DFA>(), s>>>(A);
  b = fill(Pl, DFS, l0, l1, A, [](int l) { return (1 << (3 * (l - 2))) * chunks_of(P, DFS) * (DFS ? 2 : 1); });
  if (DFS)
    k_spec_mac_df<<<b, kMacThrDf, kMacSmem * kHalfN / kHaloN, s>>>(A);
  else
    k_spec_mac<<<b, kMacThr, kMacSmem, s>>>(A);
  b = fill(Pl, DFS, l0, l1, A, [](int l) { return (1 << (3 * l)) / kInvNodes<P>; });
  k_spec_inv<P, DFS, DFA><<<b, Shape<P>::threads(4 * kInvNodes<P>), inv_smem<P, DFA>(), s>>>(A);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_p(Plan& Pl, bool df, int l0, int l1, cudaStream_t s) {
  if (df) return launch_as<P, true, true>(Pl, l0, l1, s);
  return Pl.prec == FMM_PREC_FP32 ? launch_as<P, false, true>(Pl, l0, l1, s) : launch_as<P, false, false>(Pl, l0, l1, s);
}

template <int P>
cudaError_t fwd_p(Plan& Pl, const float* src, void* dst, size_t blocks, cudaStream_t s) {
  SpecArgs A;
  fill(Pl, false, 1, 0, A, [](int) { return 0; });
  A.n = 1;
  A.lev[0] = {src, nullptr, dst, nullptr, nullptr, nullptr, nullptr, 0, 0, blocks};
  k_spec_fwd<P, false, true><<<(unsigned)(blocks / Shape<P>::NB), Shape<P>::THR, fwd_smem<P, true>(), s>>>(A);
  return cudaGetLastError();
}

template <int P>
cudaError_t kernels_p(Plan& Pl, int l, cudaStream_t s) {
  constexpr int NM = Shape<P>::NM;
  const size_t smem = 2 * sizeof(double2) * NM * NM * P;
  const dim3 grid(kOff3, 4);
  if (wide_level(Pl, l))
    k_spec_kernel<P, true><<<grid, 128, smem, s>>>(Pl.tab[l], Pl.tab_lo[l], Pl.spec_tw, static_cast<float*>(Pl.spec_K[l]));
  else
    k_spec_kernel<P, false><<<grid, 128, smem, s>>>(Pl.tab[l], Pl.tab_lo[l], Pl.spec_tw, static_cast<float*>(Pl.spec_K[l]));
  return cudaGetLastError();
}

template <typename F>
cudaError_t opt_in(F* f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int P>
cudaError_t setup_p() {
  const size_t ks = 2 * sizeof(double2) * Shape<P>::NM * Shape<P>::NM * P;
  cudaError_t e;
  if ((e = opt_in(k_spec_kernel<P, true>, ks)) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_kernel<P, false>, ks)) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_fwd<P, true, true>, fwd_smem<P, true>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_fwd<P, false, true>, fwd_smem<P, true>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_fwd<P, false, false>, fwd_smem<P, false>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_inv<P, true, true>, inv_smem<P, true>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_inv<P, false, true>, inv_smem<P, true>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_inv<P, false, false>, inv_smem<P, false>())) != cudaSuccess) return e;
  if ((e = opt_in(k_spec_mac_df, kMacSmem)) != cudaSuccess) return e;
  return opt_in(k_spec_mac, kMacSmem);
}

}  // namespace

cudaError_t launch_clear_spectra(void* K, size_t nK, void* M, size_t nM, size_t blocks, cudaStream_t s) {
  const size_t chunk = (blocks + 1) * 128, chunks = nM / chunk, kc = nK / chunks;
  char *k = static_cast<char*>(K), *m = static_cast<char*>(M);
  const size_t units = kc / 16 + chunk / 16 + 8 * chunks, grid = (units + 255) / 256;
  k_clear<<<(unsigned)(grid < 2048 ? grid : 2048), 256, 0, s>>>(
      reinterpret_cast<float4*>(k + nK - kc), kc / 16, reinterpret_cast<float4*>(m + nM - chunk), chunk / 16,
      m + blocks * 128, chunk, chunks);
  return cudaGetLastError();
}

size_t spec_kernel_bytes(const Plan& P, int l) {
  const bool df = wide_level(P, l);
  return (size_t)chunks_of(P.p, df) * kOff3 * 512;
}
size_t spec_source_bytes(const Plan& P, int l) {
  const bool df = wide_level(P, l);
  return (size_t)chunks_of(P.p, df) * (((size_t)1 << (3 * l)) + 1) * 128;
}
size_t spec_target_bytes(const Plan& P, int l) {
  const bool df = wide_level(P, l);
  return ((size_t)1 << (3 * l)) * 4 * chunks_of(P.p, df) * 128;
}

cudaError_t setup_m2l_spec(const Plan& P) {
  switch (P.p) {
    case 2: return setup_p<2>();
    case 3: return setup_p<3>();
    case 4: return setup_p<4>();
    case 5: return setup_p<5>();
    case 6: return setup_p<6>();
    case 7: return setup_p<7>();
    case 8: return setup_p<8>();
    default: return cudaSuccess;
  }
}

cudaError_t launch_spec_kernels(Plan& P, int l, cudaStream_t s) {
  switch (P.p) {
    case 2: return kernels_p<2>(P, l, s);
    case 3: return kernels_p<3>(P, l, s);
    case 4: return kernels_p<4>(P, l, s);
    case 5: return kernels_p<5>(P, l, s);
    case 6: return kernels_p<6>(P, l, s);
    case 7: return kernels_p<7>(P, l, s);
    case 8: return kernels_p<8>(P, l, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_spec_fwd(Plan& P, const float* src, void* dst, size_t blocks, cudaStream_t s) {
  switch (P.p) {
    case 2: return fwd_p<2>(P, src, dst, blocks, s);
    case 3: return fwd_p<3>(P, src, dst, blocks, s);
    case 4: return fwd_p<4>(P, src, dst, blocks, s);
    case 5: return fwd_p<5>(P, src, dst, blocks, s);
    case 6: return fwd_p<6>(P, src, dst, blocks, s);
    case 7: return fwd_p<7>(P, src, dst, blocks, s);
    case 8: return fwd_p<8>(P, src, dst, blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_m2l_spec(Plan& P, bool df, int l0, int l1, cudaStream_t s) {
  switch (P.p) {
    case 2: return launch_p<2>(P, df, l0, l1, s);
    case 3: return launch_p<3>(P, df, l0, l1, s);
    case 4: return launch_p<4>(P, df, l0, l1, s);
    case 5: return launch_p<5>(P, df, l0, l1, s);
    case 6: return launch_p<6>(P, df, l0, l1, s);
    case 7: return launch_p<7>(P, df, l0, l1, s);
    case 8: return launch_p<8>(P, df, l0, l1, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fmm
