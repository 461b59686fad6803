// Upward pass: mean removal, P2M at the leaves and M2M up to level 2
// (double-float arithmetic, see fmm_internal.cuh).
//
// Gridlet masses (Sec. 2): a node's order^3 effective masses on its
// cell-centred mini-mesh must reproduce every Cartesian multipole Q_n,
// n_i < order, of the mass they stand for.  The unique solution of that
// Vandermonde system is separable: M_s = sum_c l_s(x_c) m_c with l_s the 1-D
// Lagrange basis on the gridlet points, one factor per axis.  M2M (eq. fmm1)
// is the same map with the children's gridlet points as sources: the 8 child
// gridlets form a uniform (2 order)^3 cell-centred mesh over the parent.
#include "fmm_internal.cuh"
#include "lines.cuh"

namespace fmm {
namespace {

using lines::expand_line;

// a0: block partial sums of the density in FP64.
__global__ void k_partial_sum(const float4* __restrict__ rho4, size_t n4, double* __restrict__ partials) {
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 v = __ldg(rho4 + i);
    acc += ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double red[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (warp == 0) {
    acc = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) partials[blockIdx.x] = acc;
  }
}

__global__ void k_final_mean(const double* __restrict__ partials, int n, double inv_cells, double* __restrict__ mean) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partials[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double red[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (warp == 0) {
    acc = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) *mean = acc * inv_cells;
  }
}

// a3: nb leaves per CTA (consecutive Morton keys).  Cell masses
// m = (rho - mean) / N^3 are formed exactly as double-float pairs from the
// FP32 density and the mean split into hi + lo, and contracted in
// double-float with (hi, lo) Lagrange weights; the gridlet masses are rounded
// once to FP32 (and kept as FP64 at high order).  FP32 arithmetic here fails
// the point-source test: every node of the uniform background rounds the
// same way, so the errors add up coherently across the mesh.
// Bound by FP32 issue (12 instructions per double-float term).  A thread makes
// the P outputs of a line from registers, so a term costs its 12 instructions
// and 1/P of an operand load; 1/N^3 comes from the host (an FP64 division per
// thread took half the time of a 1-cell leaf); small leaves share a CTA.
template <int P>
__global__ void __launch_bounds__(128) k_p2m(const float* __restrict__ rho, const double* __restrict__ mean, int N,
                                            int S, int nb, float iv, float iv_lo, const float2* __restrict__ w,
                                            float* __restrict__ Mout, double* __restrict__ Mout64) {
  extern __shared__ float2 smdf[];
  __shared__ float s_mu[2];
  const int S2 = S * S, S3 = S2 * S, SR = S | 1;   // odd row stride: a thread walks its own row
  float2* W = smdf;                      // [P][S]
  float2* in = W + P * S;                // [nb][z][y][x]
  float2* t1 = in + nb * S2 * SR;             // [nb][z][y][sx]
  float2* t2 = t1 + nb * S2 * P;         // [nb][z][sy][sx]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const uint32_t leaf0 = blockIdx.x * (uint32_t)nb;
  if (tid == 0) {
    const double mu = *mean;
    s_mu[0] = (float)mu;
    s_mu[1] = (float)(mu - (double)s_mu[0]);
  }
  for (int i = tid; i < P * S; i += nthr) W[i] = __ldg(w + i);
  __syncthreads();
  const float mu_hi = s_mu[0], mu_lo = s_mu[1];
  for (int i = tid; i < nb * S3; i += nthr) {
    const int leaf = i / S3, c = i - leaf * S3, cz = c / S2, cy = (c - cz * S2) / S, cx = c - cz * S2 - cy * S;
    uint32_t lx, ly, lz;
    unmorton(leaf0 + leaf, lx, ly, lz);
    const size_t g = ((size_t)(lz * S + cz) * N + (ly * S + cy)) * N + (lx * S + cx);
    const float2 d = df_two_sum(__ldg(rho + g), -mu_hi);      // rho - mu_hi exactly
    const float dlo = __fsub_rn(d.y, mu_lo);
    const float ph = __fmul_rn(d.x, iv);                        // (d.x + dlo) (iv + iv_lo)
    const float pe = fmaf(d.x, iv, -ph);
    const float lo = fmaf(d.x, iv_lo, fmaf(dlo, iv, pe));
    const float sum = __fadd_rn(ph, lo);
    in[(leaf * S2 + cz * S + cy) * SR + cx] = make_float2(sum, __fsub_rn(lo, __fsub_rn(sum, ph)));
  }
  __syncthreads();
  float2 a[P];
  for (int l = tid; l < nb * S2; l += nthr) {                 // x: line (leaf, z, y)
    expand_line<P>(in + l * SR, 1, S, W, S, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) t1[l * P + s] = a[s];
  }
  __syncthreads();
  for (int l = tid; l < nb * S * P; l += nthr) {              // y: line (leaf, z, sx)
    const int sx = l % P, lz = l / P;
    expand_line<P>(t1 + lz * S * P + sx, P, S, W, S, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) t2[(lz * P + s) * P + sx] = a[s];
  }
  __syncthreads();
  for (int l = tid; l < nb * P * P; l += nthr) {              // z: line (leaf, sy, sx)
    const int q = l % (P * P), leaf = l / (P * P);
    expand_line<P>(t2 + leaf * S * P * P + q, P * P, S, W, S, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const size_t o = (size_t)(leaf0 + leaf) * P * P * P + s * P * P + q;
      Mout[o] = a[s].x;
      if (Mout64) Mout64[o] = df_to_double(a[s]);
    }
  }
}

// a4: one CTA per parent; the 8 children (keys 8P + c) are gathered into a
// (2p)^3 mesh and contracted with the [p][2p] (hi, lo) Lagrange matrix on each
// axis in double-float, line by line as in k_p2m.  At high order the FP64
// copies are read (Mc64, when the children keep one) and written (Mp64).
template <int P>
__global__ void __launch_bounds__(4 * P * P <= 64 ? 64 : (4 * P * P <= 160 ? 160 : 256))
k_m2m(const float* __restrict__ Mc, const double* __restrict__ Mc64, const float2* __restrict__ w,
      float* __restrict__ Mp, double* __restrict__ Mp64) {
  constexpr int K = 2 * P, P3 = P * P * P, KS = K + 1;
  extern __shared__ float2 smdf[];
  float2* W = smdf;              // [P][K]
  float2* in = W + P * K;        // [z][y][x], rows padded to an odd stride
  float2* t1 = in + K * K * KS;  // [z][y][sx]
  float2* t2 = t1 + K * K * P;   // [z][sy][sx]
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int i = tid; i < P * K; i += nthr) W[i] = __ldg(w + i);
  const size_t base = (size_t)blockIdx.x * 8 * P3;
  for (int i = tid; i < 8 * P3; i += nthr) {
    const int c = i / P3, q = i % P3;
    const int qx = q % P, qy = (q / P) % P, qz = q / (P * P);
    const int ux = (c & 1) * P + qx, uy = ((c >> 1) & 1) * P + qy, uz = (c >> 2) * P + qz;
    in[(uz * K + uy) * KS + ux] = Mc64 ? df_from_double(__ldg(Mc64 + base + i)) : make_float2(__ldg(Mc + base + i), 0.f);
  }
  __syncthreads();
  float2 a[P];
  for (int l = tid; l < K * K; l += nthr) {                   // x
    expand_line<P>(in + l * KS, 1, K, W, K, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) t1[l * P + s] = a[s];
  }
  __syncthreads();
  for (int l = tid; l < K * P; l += nthr) {                   // y
    const int sx = l % P, z = l / P;
    expand_line<P>(t1 + z * K * P + sx, P, K, W, K, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) t2[(z * P + s) * P + sx] = a[s];
  }
  __syncthreads();
  for (int l = tid; l < P * P; l += nthr) {                   // z
    expand_line<P>(t2 + l, P * P, K, W, K, 1, a);
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const size_t o = (size_t)blockIdx.x * P3 + s * P * P + l;
      Mp[o] = a[s].x;
      if (Mp64) Mp64[o] = df_to_double(a[s]);
    }
  }
}

// Leaves per P2M CTA: about 128 lines of its widest pass, a power of two.
int p2m_leaves(const Plan& P) {
  const int lines = P.S * (P.S > P.p ? P.S : P.p);
  int nb = 1;
  while (nb * 2 * lines <= 128 && nb < 64) nb *= 2;
  return nb;
}

template <int P>
cudaError_t p2m_p(Plan& Pl, const float* rho, cudaStream_t s) {
  const int S = Pl.S, nb = p2m_leaves(Pl);
  const size_t smem = sizeof(float2) * (P * S + (size_t)nb * (S * S * (S | 1) + S * S * P + S * P * P));
  const double ivd = 1.0 / ((double)Pl.N * Pl.N * Pl.N);
  const float iv = (float)ivd;
  k_p2m<P><<<(1u << (3 * Pl.L)) / nb, 128, smem, s>>>(rho, Pl.d_mean, Pl.N, S, nb, iv, (float)(ivd - (double)iv),
                                                     Pl.w_p2m, Pl.M[Pl.L], Pl.M64[Pl.L]);
  return cudaGetLastError();
}

template <int P>
cudaError_t m2m_p(Plan& Pl, int level, cudaStream_t s) {
  constexpr int K = 2 * P, T = 4 * P * P <= 64 ? 64 : (4 * P * P <= 160 ? 160 : 256);
  const size_t smem = sizeof(float2) * (P * K + K * K * (K + 1) + K * K * P + K * P * P);
  k_m2m<P><<<1u << (3 * level), T, smem, s>>>(Pl.M[level + 1], Pl.M64[level + 1], Pl.w_m2m, Pl.M[level], Pl.M64[level]);
  return cudaGetLastError();
}

template <int P>
cudaError_t setup_p() {
  const cudaError_t e = cudaFuncSetAttribute(k_p2m<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_m2m<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

}  // namespace

cudaError_t setup_upward(const Plan& P) { FMM_BY_ORDER(P.p, setup_p, ()); }

cudaError_t launch_mean_into(const Plan& P, const float* rho, double* partials, double* mean, cudaStream_t s) {
  const size_t n4 = (size_t)P.N * P.N * P.N / 4;
  k_partial_sum<<<P.n_partials, 256, 0, s>>>(reinterpret_cast<const float4*>(rho), n4, partials);
  k_final_mean<<<1, 1024, 0, s>>>(partials, P.n_partials, 1.0 / ((double)P.N * P.N * P.N), mean);
  return cudaGetLastError();
}

cudaError_t launch_mean(Plan& P, const float* rho, cudaStream_t s) {
  return launch_mean_into(P, rho, P.d_partials, P.d_mean, s);
}

cudaError_t launch_p2m(Plan& P, const float* rho, cudaStream_t s) { FMM_BY_ORDER(P.p, p2m_p, (P, rho, s)); }

cudaError_t launch_m2m(Plan& P, int level, cudaStream_t s) { FMM_BY_ORDER(P.p, m2m_p, (P, level, s)); }

}  // namespace fmm
