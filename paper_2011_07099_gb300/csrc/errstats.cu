// Sampled error of a solution against the PM solution with the same Green's
// function.  Sec. 3 defines the optimal G_* as the function with which PM and
// FMM give the same potential, and measures the FMM against that PM: the
// periodic convolution of the cell masses with G sampled at the mesh offsets
// d/N (eq. pmconv), with the cell self term at d = 0.  That convolution is
// evaluated here exactly, by a direct sum over every source cell, at a set of
// sampled target cells; the relative L2 error of the given potential and
// acceleration over those cells is the result.
//
// Arithmetic: per-axis xi(d/N), xi'(d/N) in FP64 (green_s1.cuh) rounded to
// FP32; each pair's (G, -grad G) in FP32, its root and quotients rounded once;
// masses, in a unit that follows the density, their products with the pair
// values and the sums in double-float (fmm_internal.cuh).  The error of these
// sums against FP64 (1024 cells, N = 24 .. 192, sigma = 0.3 and 1.5) is that of
// the same pair values summed in FP64 within 0.2 % for the potential, and 3 %
// above (N = 24) to 19 % below it for the acceleration.
#include <cuda_runtime.h>

#include "fmm_internal.cuh"
#include "green_s1.cuh"

namespace fmm {
namespace {

constexpr int kEsThreads = 256;   // one target cell per thread
constexpr int kEsChunk = 512;     // source cells staged in shared memory per step (128^3: 6.7 steps per CTA)

// amax = max |rho| as the bits of a non-negative float (a NaN lies above all).
__global__ void __launch_bounds__(256) k_es_amax(const float4* __restrict__ rho4, size_t n4, float* __restrict__ amax) {
  float m = 0.f;
  auto take = [&](float v) { m = fabsf(v) > m || v != v ? fabsf(v) : m; };
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 v = __ldg(rho4 + i);
    take(v.x);
    take(v.y);
    take(v.z);
    take(v.w);
  }
  const int b = __reduce_max_sync(0xffffffffu, __float_as_int(m));
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int*>(amax), b);
}

// The power of two that takes amax to [1, 2): the double-float masses, whose
// product errors reach 2^-48 below them, then stay clear of FP32's ends
// whatever the density's unit (1 where amax is 0 or not finite).
__device__ __forceinline__ double es_scale(float amax) {
  return amax > 0.f && amax <= 3.4e38f ? ldexp(1.0, -ilogbf(amax)) : 1.0;
}

// (s, c) += (mh + ml) g: exact product by FMA, TwoSum, the errors in c
__device__ __forceinline__ void es_mac(float2& a, float mh, float ml, float g) {
  const float pr = __fmul_rn(mh, g);
  const float pe = fmaf(mh, g, -pr);
  const float2 t = df_two_sum(a.x, pr);
  a.x = t.x;
  a.y = fmaf(ml, g, __fadd_rn(a.y, __fadd_rn(pe, t.y)));
}

// partials[(blockIdx.x * T + t) * 4 + f]: block blockIdx.x's share of the
// direct sum (Phi, g_x, g_y, g_z) at target t, over the source chunks
// blockIdx.x, blockIdx.x + gridDim.x, ...  Bound by FP32 issue, ~60
// instructions per pair: G = -1/(4 pi |xhat|) and c = G / |xhat|^2 come from
// one rsqrtf, each corrected by its FMA residual (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000", 1990): one Newton step
// and plain products, 4 % faster, had left up to 40 % more error at N = 24.
// Along a row g_y and g_z differ from the sum of c m by row constants only, so
// one double-float sum serves both.  256 targets of a 128^3 mesh: 1.19 ms, with
// FP64 sums, at 1/64 of the FP32 rate, 8.97 ms.
__global__ void __launch_bounds__(kEsThreads) k_es_direct(const float* __restrict__ rho,
                                                          const double* __restrict__ mean,
                                                          const float* __restrict__ amax, int N,
                                                          const unsigned long long* __restrict__ targets, int T,
                                                          double* __restrict__ partials) {
  extern __shared__ __align__(16) unsigned char es_smem[];
  float2* sm = reinterpret_cast<float2*>(es_smem);                 // kEsChunk masses (hi, lo)
  float2* sx = reinterpret_cast<float2*>(sm + kEsChunk);           // N pairs (xi, xi')(d/N)
  for (int d = threadIdx.x; d < N; d += blockDim.x)
    sx[d] = make_float2((float)green::xi_s1((double)d / N), (float)green::dxi_s1((double)d / N));
  const size_t n3 = (size_t)N * N * N;
  const double mu = *mean;
  const double sc = es_scale(*amax);
  const int ti = blockIdx.y * kEsThreads + threadIdx.x;
  const bool valid = ti < T;
  int tx = 0, ty = 0, tz = 0;
  if (valid) {
    const unsigned long long t = targets[ti];
    tx = (int)(t % N);
    ty = (int)((t / N) % N);
    tz = (int)(t / ((unsigned long long)N * N));
  }
  const float inv4pi = (float)(1.0 / (4.0 * green::kPi));
  const float self = (float)(-green::cube_mean_inv_r() * N / (4.0 * green::kPi));
  float2 a[4] = {};
  for (size_t c0 = (size_t)blockIdx.x * kEsChunk; c0 < n3; c0 += (size_t)gridDim.x * kEsChunk) {
    const int cnt = (int)((n3 - c0) < (size_t)kEsChunk ? (n3 - c0) : (size_t)kEsChunk);
    __syncthreads();
    for (int k = threadIdx.x; k < cnt; k += blockDim.x) sm[k] = df_from_double(((double)rho[c0 + k] - mu) * sc);
    __syncthreads();
    if (!valid) continue;
    // offsets d = (t - j) mod N per axis, stepped along the chunk (x fastest)
    int jx = (int)(c0 % N), jy = (int)((c0 / N) % N);
    const int jz = (int)(c0 / ((size_t)N * N));
    int dx = tx - jx, dy = ty - jy, dz = tz - jz;
    dx += dx < 0 ? N : 0;
    dy += dy < 0 ? N : 0;
    dz += dz < 0 ? N : 0;
    for (int k = 0; k < cnt;) {
      // the sources of one row
      const int run = N - jx < cnt - k ? N - jx : cnt - k;
      const float2 vy = sx[dy], vz = sx[dz];
      const float ryz2 = fmaf(vz.x, vz.x, vy.x * vy.x);
      const bool on_row = (dy | dz) == 0;
      float2 sc = make_float2(0.f, 0.f);
      for (int q = 0; q < run; ++q) {
        const float2 mj = sm[k + q];
        const float2 vx = sx[dx];
        const float r2 = fmaf(vx.x, vx.x, ryz2);
        const bool at0 = on_row && dx == 0;             // self term; grad G(0) = 0
        // r = sqrt(r2), G = -1/(4 pi r), c = G / r2
        const float ir = rsqrtf(at0 ? 1.f : r2), i2 = ir * ir;
        float r = r2 * ir;
        r = fmaf(fmaf(-r, r, r2), 0.5f * ir, r);
        float G = -inv4pi * ir;
        G = fmaf(fmaf(-G, r, -inv4pi), ir, G);
        float c = G * i2;                               // -1 / (4 pi |xhat|^3)
        c = fmaf(fmaf(-c, r2, G), i2, c);
        if (at0) {
          G = self;
          c = 0.f;
        }
        es_mac(a[0], mj.x, mj.y, G);
        es_mac(a[1], mj.x, mj.y, c * vx.x * vx.y);
        es_mac(sc, mj.x, mj.y, c);
        dx = dx == 0 ? N - 1 : dx - 1;
      }
      es_mac(a[2], sc.x, sc.y, vy.x * vy.y);
      es_mac(a[3], sc.x, sc.y, vz.x * vz.y);
      k += run;
      jx += run;
      if (jx == N) {                      // next row: x restarts, y advances
        jx = 0;
        dx = tx;
        dy = dy == 0 ? N - 1 : dy - 1;
        if (++jy == N) {                  // next plane
          jy = 0;
          dy = ty;
          dz = dz == 0 ? N - 1 : dz - 1;
        }
      }
    }
  }
  if (valid) {
    double* o = partials + ((size_t)blockIdx.x * T + ti) * 4;
    const double unit = 1.0 / (sc * (double)n3);        // masses are (rho - mean) / N^3
    for (int f = 0; f < 4; ++f) o[f] = df_to_double(a[f]) * unit;
  }
}

// One warp per target: the sum of its partials over the blocks, compared with
// the given solution there: terms[t] = (dPhi^2, Phi_ref^2, |dg|^2, |g_ref|^2).
__global__ void __launch_bounds__(256) k_es_reduce(const double* __restrict__ partials, int nblocks, int T,
                                                  const unsigned long long* __restrict__ targets, size_t n3,
                                                  const float* __restrict__ phi, const float* __restrict__ acc,
                                                  double* __restrict__ terms) {
  const int lane = threadIdx.x & 31, t = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (t >= T) return;
  double ref[4] = {0.0, 0.0, 0.0, 0.0};
  for (int b = lane; b < nblocks; b += 32)
    for (int f = 0; f < 4; ++f) ref[f] += partials[((size_t)b * T + t) * 4 + f];
  for (int o = 16; o > 0; o >>= 1)
    for (int f = 0; f < 4; ++f) ref[f] += __shfl_down_sync(0xffffffffu, ref[f], o);
  if (lane) return;
  const size_t i = targets[t];
  const double dp = (double)phi[i] - ref[0];
  double e[4] = {dp * dp, ref[0] * ref[0], 0.0, 0.0};
  for (int c = 0; c < 3; ++c) {
    const double dg = (double)acc[(size_t)c * n3 + i] - ref[1 + c];
    e[2] += dg * dg;
    e[3] += ref[1 + c] * ref[1 + c];
  }
  for (int f = 0; f < 4; ++f) terms[4 * (size_t)t + f] = e[f];
}

// sums[f] = sum over the targets of terms[t][f], one block.
constexpr int kEsMaxSamples = 1024;
__global__ void __launch_bounds__(256) k_es_finish(const double* __restrict__ terms, int T, double* __restrict__ sums) {
  __shared__ double red[256];
  const int f = threadIdx.x & 3;
  double a = 0.0;
  for (int t = threadIdx.x >> 2; t < T; t += 64) a += terms[4 * t + f];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int h = 128; h >= 4; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x < 4) sums[threadIdx.x] = red[threadIdx.x];
}

}  // namespace

int error_stats_max_samples() { return kEsMaxSamples; }

int error_stats_grid_x(const Plan& P, int T) {
  const int gy = (T + kEsThreads - 1) / kEsThreads;
  const int gx = (4 * P.num_sms + gy - 1) / gy;
  return gx < 1 ? 1 : gx;
}

cudaError_t launch_error_stats(Plan& P, const float* rho, const float* phi, const float* acc,
                               const unsigned long long* targets, int T, double* partials, double* sums,
                               double* mean_scratch, cudaStream_t s) {
  double* mean = mean_scratch + P.n_partials;
  float* amax = reinterpret_cast<float*>(mean + 1);
  cudaError_t e = launch_mean_into(P, rho, mean_scratch, mean, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(amax, 0, sizeof(float), s);
  if (e != cudaSuccess) return e;
  k_es_amax<<<4 * P.num_sms, 256, 0, s>>>(reinterpret_cast<const float4*>(rho), (size_t)P.N * P.N * P.N / 4, amax);
  const int gx = error_stats_grid_x(P, T);
  const dim3 grid(gx, (T + kEsThreads - 1) / kEsThreads);
  const size_t smem = sizeof(float2) * (size_t)kEsChunk + sizeof(float2) * (size_t)P.N;
  k_es_direct<<<grid, kEsThreads, smem, s>>>(rho, mean, amax, P.N, targets, T, partials);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t n3 = (size_t)P.N * P.N * P.N;
  k_es_reduce<<<(T + 7) / 8, 256, 0, s>>>(partials, gx, T, targets, n3, phi, acc, sums + 4);
  k_es_finish<<<1, 256, 0, s>>>(sums + 4, T, sums);
  return cudaGetLastError();
}

}  // namespace fmm
