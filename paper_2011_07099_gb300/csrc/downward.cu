// Downward pass: L2L (eq. fmm3).
//
// The local field of a child is the parent's local field projected with the
// transpose of the child's M2M matrix: Phi_child[q] = sum_r T_{r q} Phi_parent[r]
// (Sec. 3 eq. fmm3).  With T the separable Lagrange matrix, that is the parent
// field interpolated at the child's gridlet points.  The 8 children's points
// form one uniform (2p)^3 mesh over the parent, so a CTA expands a parent's
// field onto that mesh, line by line, and adds it to the children's fields
// (which already hold their own M2L result).
#include "fmm_internal.cuh"
#include "lines.cuh"

namespace fmm {
namespace {

using lines::expand_line;
using lines::expand_line_f;

// Mesh index of child value i = (child c, q) of one field.
template <int P>
__device__ __forceinline__ int mesh_index(int i) {
  constexpr int K = 2 * P, P3 = P * P * P;
  const int c = i / P3, q = i % P3;
  const int qx = q % P, qy = (q / P) % P, qz = q / (P * P);
  return (((c >> 2) * P + qz) * K + ((c >> 1) & 1) * P + qy) * K + (c & 1) * P + qx;
}

// FP32: CTA per parent, all four fields (one field's passes have p^2, 2p^2 and
// 4p^2 lines and would leave most threads idle).  A thread makes the 2p outputs
// of a line from registers; the last pass goes through shared memory so that
// the children's values are read and written along memory.  Measured at 256^3,
// p = 6 (level 4 -> 5): 0.30 ms when each output was its own loop with two
// divisions, 0.15 with a CTA per field.
template <int P>
constexpr int kL2lThr = (8 * P * P + 31) / 32 * 32 > 512 ? 512 : (8 * P * P + 31) / 32 * 32;

template <int P>
__global__ void __launch_bounds__(kL2lThr<P>) k_l2l(const float* __restrict__ Fp, const float2* __restrict__ w,
                                                   float* __restrict__ Fc) {
  constexpr int K = 2 * P, P3 = P * P * P, KS = K + 1, PR = P | 1;
  extern __shared__ float2 smdf[];
  float2* W = smdf;                                  // [P][2P], used transposed
  float* in = reinterpret_cast<float*>(W + P * K);   // [f][z][y][x]
  float* t1 = in + 4 * P * P * PR;                   // [f][z][y][ux]
  float* t2 = t1 + 4 * P * P * KS;                   // [f][z][uy][ux]
  float* out = t2 + 4 * P * K * K;                   // [f][uz][uy][ux]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const size_t parent = blockIdx.x;
  for (int i = tid; i < P * K; i += nthr) W[i] = __ldg(w + i);
  for (int i = tid; i < 4 * P3; i += nthr) in[(i / P) * PR + i % P] = __ldg(Fp + parent * 4 * P3 + i);
  __syncthreads();
  float a[K];
  for (int l = tid; l < 4 * P * P; l += nthr) {             // x: line (f, z, y)
    expand_line_f<K>(in + l * PR, 1, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) t1[l * KS + u] = a[u];
  }
  __syncthreads();
  for (int l = tid; l < 4 * P * K; l += nthr) {             // y: line (f, z, ux)
    const int ux = l % K, fz = l / K;
    expand_line_f<K>(t1 + fz * P * KS + ux, KS, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) t2[(fz * K + u) * K + ux] = a[u];
  }
  __syncthreads();
  for (int l = tid; l < 4 * K * K; l += nthr) {             // z: line (f, uy, ux)
    const int q = l % (K * K), f = l / (K * K);
    expand_line_f<K>(t2 + f * P * K * K + q, K * K, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) out[(f * K + u) * K * K + q] = a[u];
  }
  __syncthreads();
  float* dst = Fc + parent * 32 * P3;
  for (int i = tid; i < 32 * P3; i += nthr) {               // (child, f, q)
    const int c = i / (4 * P3), fq = i % (4 * P3), f = fq / P3;
    dst[i] += out[f * K * K * K + mesh_index<P>(c * P3 + fq % P3)];
  }
}

// Variant for parents at the wide levels (the coarse levels 2 and 3; at
// order >= 7 every level above the leaves): FP64 local fields, interpolated
// in double-float (fmm_internal.cuh).  The child field is F64 (a coarse child,
// whose FP32 copy is refreshed too) or the FP32 field of the first fine level,
// to which the contribution is added in double-float before a single rounding
// (in FP64, at 1/64 of the FP32 rate, these adds alone took 2.5 ms of the
// 512^3 order-8 solve).
template <int P>
__global__ void __launch_bounds__(128) k_l2l64(const double* __restrict__ Fp, const float2* __restrict__ w,
                                              double* __restrict__ Fc64, float* __restrict__ Fc) {
  constexpr int K = 2 * P, P3 = P * P * P, KS = K + 1, PR = P | 1;
  extern __shared__ float2 smdf[];
  float2* W = smdf;                  // [P][2P], used transposed
  float2* t1 = W + P * K;            // [z][y][ux], odd row stride
  float2* t2 = t1 + P * P * KS;       // [z][uy][ux]
  float2* out = t2 + P * K * K;      // [uz][uy][ux]
  float2* in = out;                  // [z][y][x], consumed before `out` is written
  const int tid = threadIdx.x, nthr = blockDim.x;
  const size_t parent = blockIdx.x >> 2;
  const int f = blockIdx.x & 3;
  for (int i = tid; i < P * K; i += nthr) W[i] = __ldg(w + i);
  for (int i = tid; i < P3; i += nthr) in[(i / P) * PR + i % P] = df_from_double(__ldg(Fp + (parent * 4 + f) * P3 + i));
  __syncthreads();
  float2 a[K];
  for (int l = tid; l < P * P; l += nthr) {                 // x
    expand_line<K>(in + l * PR, 1, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) t1[l * KS + u] = a[u];
  }
  __syncthreads();
  for (int l = tid; l < P * K; l += nthr) {                 // y
    const int ux = l % K, z = l / K;
    expand_line<K>(t1 + z * P * KS + ux, KS, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) t2[(z * K + u) * K + ux] = a[u];
  }
  __syncthreads();
  for (int l = tid; l < K * K; l += nthr) {                 // z
    expand_line<K>(t2 + l, K * K, P, W, 1, K, a);
#pragma unroll
    for (int u = 0; u < K; ++u) out[u * K * K + l] = a[u];
  }
  __syncthreads();
  for (int i = tid; i < 8 * P3; i += nthr) {
    const size_t d = ((parent * 8 + i / P3) * 4 + f) * P3 + i % P3;
    const float2 v = out[mesh_index<P>(i)];
    if (Fc64) {
      const double t = Fc64[d] + df_to_double(v);
      Fc64[d] = t;
      Fc[d] = (float)t;
    } else {
      const float2 t = df_two_sum(Fc[d], v.x);
      Fc[d] = __fadd_rn(t.x, __fadd_rn(t.y, v.y));
    }
  }
}

template <int P>
size_t smem64() {
  constexpr int K = 2 * P;
  return sizeof(float2) * (P * K + P * P * (K + 1) + P * K * K + K * K * K);
}

template <int P>
size_t smem32() {
  constexpr int K = 2 * P;
  return sizeof(float2) * P * K + sizeof(float) * 4 * (P * P * (P | 1) + P * P * (K + 1) + P * K * K + K * K * K);
}

template <int P>
cudaError_t setup_p() {
  const cudaError_t e = cudaFuncSetAttribute(k_l2l<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem32<P>());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_l2l64<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64<P>());
}

template <int P>
cudaError_t l2l_p(Plan& Pl, int level, cudaStream_t s) {
  const unsigned parents = 1u << (3 * level);
  if (wide_level(Pl, level))
    k_l2l64<P><<<4 * parents, 128, smem64<P>(), s>>>(Pl.F64[level], Pl.w_m2m,
                                               wide_level(Pl, level + 1) ? Pl.F64[level + 1] : nullptr, Pl.F[level + 1]);
  else
    k_l2l<P><<<parents, kL2lThr<P>, smem32<P>(), s>>>(Pl.F[level], Pl.w_m2m, Pl.F[level + 1]);
  return cudaGetLastError();
}

}  // namespace

cudaError_t setup_downward(const Plan& P) { FMM_BY_ORDER(P.p, setup_p, ()); }

cudaError_t launch_l2l(Plan& P, int level, cudaStream_t s) { FMM_BY_ORDER(P.p, l2l_p, (P, level, s)); }

}  // namespace fmm
