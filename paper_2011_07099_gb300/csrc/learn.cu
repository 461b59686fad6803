// Training kernels of the learned table correction (FP32).
//
// The FMM output is linear in the M2L tables.  For a loss
//   J = w_phi |Phi - Phi*|^2 + w_g |g - g*|^2
// against a target solution (PM with G_S1, Sec. 3: the optimal G_* is the one
// for which FMM and PM agree), the gradient with respect to a table entry is
//   dJ/dT_l[f][n] = sum_T sum_{o in IL(T)} sum_{r - s = n - o p} lam_l[T][f][r] M_l[T - o][s],
// where lam_l is the adjoint of the level-l local field: lam_L = L2P^T of the
// cell residual, lam_l = L2L^T(lam_{l+1}) (eq. fmm3 transposed is eq. fmm1's
// map, so the adjoint sweep reuses the upward contractions).  The table
// gradient then flows through the MLP (mlp.cuh) by its own backward kernel.
#include <cuda_runtime.h>

#include "fmm_internal.cuh"
#include "green_s1.cuh"
#include "mlp.cuh"

namespace fmm {
namespace {

// ------------------------------------------------------------ residual, loss
// lam[f][i] = 2 w_f (out_f - target_f), f = Phi, g_x, g_y, g_z (SoA, N^3 each);
// partials[block] = the block's share of sum w_f (out_f - target_f)^2, added to
// the loss in block order by k_loss_add: one rounding per field, where an
// FP32 atomic per warp (4864 of them) drifted by 1e-6 from run to run.
__global__ void __launch_bounds__(256) k_residual(const float* __restrict__ phi, const float* __restrict__ acc, const float* __restrict__ tphi,
                           const float* __restrict__ tacc, size_t n3, float w_phi, float w_g, float* __restrict__ lam,
                           double* __restrict__ partials) {
  __shared__ double warps[8];
  double part = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < 4 * n3; i += (size_t)gridDim.x * blockDim.x) {
    const bool isphi = i < n3;
    const float d = isphi ? phi[i] - tphi[i] : acc[i - n3] - tacc[i - n3];
    const float w = isphi ? w_phi : w_g;
    lam[i] = 2.f * w * d;
    part += (double)w * d * d;
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) warps[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) part += warps[w];
    partials[blockIdx.x] = part;
  }
}

// *loss += sum of the n partials (one warp).
__global__ void k_loss_add(const double* __restrict__ partials, int n, float* __restrict__ loss) {
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) a += partials[i];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if (threadIdx.x == 0) atomicAdd(loss, (float)a);
}

// --------------------------------------------------------- adjoint of L2P
// lam_L[leaf][f][s] = sum_c w_p2m(s, c) lam_cell[f][c]: the transpose of L2P is
// the P2M contraction, applied to the four residual fields.
__global__ void k_adj_l2p(const float* __restrict__ lam, int N, int S, int p, const float2* __restrict__ w,
                          float* __restrict__ lamL) {
  extern __shared__ float smf[];
  const int p3 = p * p * p, S3 = S * S * S;
  float2* W = reinterpret_cast<float2*>(smf);      // p*S
  float* in = reinterpret_cast<float*>(W + p * S); // 4*S^3
  float* t1 = in + 4 * S3;                         // 4*S*S*p
  float* t2 = t1 + 4 * S * S * p;                  // 4*S*p*p
  float* out = t2 + 4 * S * p * p;                 // 4*p^3
  const int tid = threadIdx.x, nthr = blockDim.x;
  uint32_t lx, ly, lz;
  unmorton(blockIdx.x, lx, ly, lz);
  const size_t n3 = (size_t)N * N * N;
  for (int i = tid; i < p * S; i += nthr) W[i] = w[i];
  for (int i = tid; i < 4 * S3; i += nthr) {
    const int f = i / S3, c = i % S3;
    const int cx = c % S, cy = (c / S) % S, cz = c / (S * S);
    in[i] = lam[f * n3 + ((size_t)(lz * S + cz) * N + (ly * S + cy)) * N + (lx * S + cx)];
  }
  __syncthreads();
  contract3(in, t1, t2, out, 4, S, p, W, S, false, tid, nthr);
  for (int i = tid; i < 4 * p3; i += nthr) lamL[(size_t)blockIdx.x * 4 * p3 + i] = out[i];
}

// --------------------------------------------------------- adjoint of L2L
// lam_l[P] = sum_children T^c lam_{l+1}[8P + c] (the M2M contraction, 4 fields).
__global__ void k_adj_l2l(const float* __restrict__ lamc, int p, const float2* __restrict__ w, float* __restrict__ lamp) {
  extern __shared__ float smf[];
  const int K = 2 * p, p3 = p * p * p, K3 = K * K * K;
  float2* W = reinterpret_cast<float2*>(smf);      // p*K
  float* in = reinterpret_cast<float*>(W + p * K); // 4*K^3
  float* t1 = in + 4 * K3;                         // 4*K*K*p
  float* t2 = t1 + 4 * K * K * p;                  // 4*K*p*p
  float* out = t2 + 4 * K * p * p;                 // 4*p^3
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int i = tid; i < p * K; i += nthr) W[i] = w[i];
  const float* src = lamc + (size_t)blockIdx.x * 8 * 4 * p3;
  for (int i = tid; i < 8 * 4 * p3; i += nthr) {
    const int c = i / (4 * p3), rem = i % (4 * p3);
    const int f = rem / p3, q = rem % p3;
    const int qx = q % p, qy = (q / p) % p, qz = q / (p * p);
    const int ux = (c & 1) * p + qx, uy = ((c >> 1) & 1) * p + qy, uz = (c >> 2) * p + qz;
    in[((f * K + uz) * K + uy) * K + ux] = src[i];
  }
  __syncthreads();
  contract3(in, t1, t2, out, 4, K, p, W, K, false, tid, nthr);
  for (int i = tid; i < 4 * p3; i += nthr) lamp[(size_t)blockIdx.x * 4 * p3 + i] = out[i];
}

// ------------------------------------------------------ table gradient
// Direct sums: isolated plans, order 1, and levels whose spectra have no
// buffers (the others: learn_spec.cu).
// CTA (offset index io, child type c, field f): for every d in [-(p-1), p-1]^3,
//   g[d] = sum over targets T of type c, sum_r lam[T][f][r] M[T - o][r - d],
// added to dT[o p + d][f].  Targets are staged 32 at a time in shared memory.
constexpr int kTgChunk = 32;

__global__ void k_table_grad(const float* __restrict__ lam, const float* __restrict__ M, const int8_t* __restrict__ offs,
                             int n_off, int level, int p, float* __restrict__ dT) {
  extern __shared__ float smf[];
  const int p3 = p * p * p, D = 2 * p - 1, D3 = D * D * D, E = 8 * p - 1, HW = 4 * p - 1;
  float* sl = smf;                      // kTgChunk * p3
  float* sm = sl + kTgChunk * p3;       // kTgChunk * p3
  const int io = blockIdx.x, ctype = blockIdx.y, f = blockIdx.z;
  const int8_t* o3 = offs + ((size_t)ctype * n_off + io) * 3;
  const int ox = o3[0], oy = o3[1], oz = o3[2];
  const int n = 1 << level;
  const uint32_t n_par = 1u << (3 * (level - 1));
  constexpr int KMAX = 8;      // (2p-1)^3 <= 8 x 512 for p <= 8
  float acc[KMAX];
#pragma unroll
  for (int k = 0; k < KMAX; ++k) acc[k] = 0.f;
  for (uint32_t t0 = 0; t0 < n_par; t0 += kTgChunk) {
    __syncthreads();
    for (int i = threadIdx.x; i < kTgChunk * p3; i += blockDim.x) {
      const uint32_t t = t0 + i / p3;
      const int r = i % p3;
      float lv = 0.f, mv = 0.f;
      if (t < n_par) {
        const uint32_t T = 8u * t + ctype;
        uint32_t x, y, z;
        unmorton(T, x, y, z);
        const uint32_t S = morton((x - ox) & (n - 1), (y - oy) & (n - 1), (z - oz) & (n - 1));
        lv = lam[((size_t)T * 4 + f) * p3 + r];
        mv = M[(size_t)S * p3 + r];
      }
      sl[i] = lv;
      sm[i] = mv;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
      const int dd = threadIdx.x + k * blockDim.x;
      if (dd >= D3) break;
      const int dx = dd % D - (p - 1), dy = (dd / D) % D - (p - 1), dz = dd / (D * D) - (p - 1);
      const int x0 = dx > 0 ? dx : 0, x1 = dx < 0 ? p + dx : p;
      const int y0 = dy > 0 ? dy : 0, y1 = dy < 0 ? p + dy : p;
      const int z0 = dz > 0 ? dz : 0, z1 = dz < 0 ? p + dz : p;
      const int shift = (dz * p + dy) * p + dx;     // s = r - shift
      float a = 0.f;
      for (int t = 0; t < kTgChunk; ++t) {
        const float* lt = sl + t * p3;
        const float* mt = sm + t * p3;
        for (int rz = z0; rz < z1; ++rz)
          for (int ry = y0; ry < y1; ++ry) {
            const int rb = (rz * p + ry) * p;
            for (int rx = x0; rx < x1; ++rx) a = fmaf(lt[rb + rx], mt[rb + rx - shift], a);
          }
      }
      acc[k] += a;
    }
  }
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int dd = threadIdx.x + k * blockDim.x;
    if (dd >= D3) break;
    const int dx = dd % D - (p - 1), dy = (dd / D) % D - (p - 1), dz = dd / (D * D) - (p - 1);
    const int nx = ox * p + dx + HW, ny = oy * p + dy + HW, nz = oz * p + dz + HW;
    atomicAdd(&dT[(((size_t)nz * E + ny) * E + nx) * 4 + f], acc[k]);
  }
}

// ----------------------------------------------------------- MLP backward
// Samples are the distinct network inputs of every level (learn_spec.cu) with
// their folded upstream gradients.  A block of 256 threads takes tiles of 64
// samples: in the layer passes a thread holds 16 neurons of one sample (the
// weights, four at a time, are broadcasts), in the weight gradients a 4 x 4
// block of a layer's matrix summed over the tile's samples; activation rows are
// padded to 65 floats, so that a warp's 32 rows start on different banks.
// Per-block partials are summed by k_grad_reduce.  Measured at p = 6, L = 3,
// one field: 16.4 ms for the 830 600 table entries one by one, 0.27 ms for
// their distinct inputs with one thread per sample.
constexpr int kBwdTile = 64;
constexpr int kBwdThr = 256;
constexpr int kRow = mlp::kH + 1;

// acc[ii] = sum over j of W[(16 q + ii)][j] in[j], added in order of j.
__device__ __forceinline__ void layer16(const float* __restrict__ W, const float* __restrict__ in, int q, float (&acc)[16]) {
  for (int j = 0; j < mlp::kH; j += 4) {
    const float h0 = in[j], h1 = in[j + 1], h2 = in[j + 2], h3 = in[j + 3];
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) {
      const float4 w = *reinterpret_cast<const float4*>(W + (16 * q + ii) * mlp::kH + j);
      acc[ii] = fmaf(w.w, h3, fmaf(w.z, h2, fmaf(w.y, h1, fmaf(w.x, h0, acc[ii]))));
    }
  }
}
// acc[jj] = sum over i of W[i][16 q + jj] in[i].
__device__ __forceinline__ void layer16_t(const float* __restrict__ W, const float* __restrict__ in, int q,
                                          float (&acc)[16]) {
  for (int i = 0; i < mlp::kH; ++i) {
    const float g = in[i];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 w = *reinterpret_cast<const float4*>(W + i * mlp::kH + 16 * q + 4 * c);
      acc[4 * c] = fmaf(w.x, g, acc[4 * c]);
      acc[4 * c + 1] = fmaf(w.y, g, acc[4 * c + 1]);
      acc[4 * c + 2] = fmaf(w.z, g, acc[4 * c + 2]);
      acc[4 * c + 3] = fmaf(w.w, g, acc[4 * c + 3]);
    }
  }
}
// dW[4 a + x][4 b + y] += sum_s G[s][4 a + x] H[s][4 b + y], (a, b) = (tid / 16, tid % 16).
__device__ __forceinline__ void outer16(const float* __restrict__ G, const float* __restrict__ H, int tid, float (&dW)[16]) {
  const float *g0 = G + 4 * (tid >> 4), *h0 = H + 4 * (tid & 15);
  for (int s = 0; s < kBwdTile; ++s) {
    float g[4], h[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      g[x] = g0[s * kRow + x];
      h[x] = h0[s * kRow + x];
    }
#pragma unroll
    for (int x = 0; x < 16; ++x) dW[x] = fmaf(g[x / 4], h[x % 4], dW[x]);
  }
}

__global__ void __launch_bounds__(kBwdThr) k_mlp_backward(const float* __restrict__ w, const float* __restrict__ up,
                                                         const uint32_t* __restrict__ samples, int ns, int lmax, int p,
                                                         float* __restrict__ partials) {
  using namespace mlp;
  static_assert(kOffW2 % 4 == 0 && kOffW3 % 4 == 0, "float4 weight rows");
  extern __shared__ float4 smf4[];
  float* sw = reinterpret_cast<float*>(smf4);    // kParams (+ padding)
  float* X = sw + (kParams + 3) / 4 * 4;         // tile x kIn
  float* Z1 = X + kBwdTile * kIn;                // tile x kRow (pre-activations; Z3 then holds dz2)
  float* Z2 = Z1 + kBwdTile * kRow;
  float* Z3 = Z2 + kBwdTile * kRow;
  float* H1 = Z3 + kBwdTile * kRow;              // post-activations
  float* H2 = H1 + kBwdTile * kRow;
  float* H3 = H2 + kBwdTile * kRow;
  float* G = H3 + kBwdTile * kRow;               // dz3, then dz1
  float* GO = G + kBwdTile * kRow;               // tile (upstream gradient)
  const int tid = threadIdx.x, s = tid & 63, q = tid >> 6;
  for (int i = tid; i < kParams; i += kBwdThr) sw[i] = w[i];
  const int total = (lmax - 1) * ns;
  float d3[16] = {}, d2[16] = {}, dv = 0.f, dw1[2] = {0.f, 0.f}, db4 = 0.f;
  for (int base = blockIdx.x * kBwdTile; base < total; base += gridDim.x * kBwdTile) {
    __syncthreads();
    if (tid < kBwdTile) {
      const int sidx = base + tid;
      float x[kIn] = {0.f, 0.f, 0.f, 0.f, 0.f};
      float go = 0.f;
      if (sidx < total) {
        const uint32_t v = samples[sidx % ns];
        const float inv = 1.f / (4.f * p);
        x[0] = (int)((v >> 16) & 255) * inv;
        x[1] = (int)((v >> 8) & 255) * inv;
        x[2] = (int)(v & 255) * inv;
        x[3] = (2 + sidx / ns) * 0.125f;
        x[4] = (float)(v >> 24);
        go = up[sidx];
      }
      GO[tid] = go;
      for (int j = 0; j < kIn; ++j) X[tid * kIn + j] = x[j];
    }
    __syncthreads();
    float a[16];
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) {
      const int i = 16 * q + ii;
      float z = sw[kOffB1 + i];
      for (int j = 0; j < kIn; ++j) z = fmaf(sw[kOffW1 + i * kIn + j], X[s * kIn + j], z);
      Z1[s * kRow + i] = z;
      H1[s * kRow + i] = gelu(z);
    }
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) a[ii] = sw[kOffB2 + 16 * q + ii];
    layer16(sw + kOffW2, H1 + s * kRow, q, a);
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) {
      Z2[s * kRow + 16 * q + ii] = a[ii];
      H2[s * kRow + 16 * q + ii] = gelu(a[ii]);
    }
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) a[ii] = sw[kOffB3 + 16 * q + ii];
    layer16(sw + kOffW3, H2 + s * kRow, q, a);
    const float go = GO[s];
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) {
      const int i = 16 * q + ii;
      H3[s * kRow + i] = gelu(a[ii]);
      G[s * kRow + i] = go * sw[kOffW4 + i] * gelu_grad(a[ii]);   // dz3 = go W4 gelu'(z3)
    }
    __syncthreads();
    outer16(G, H2, tid, d3);
    if (q == 0)                                    // b3
      for (int t = 0; t < kBwdTile; ++t) dv += G[t * kRow + s];
    else if (q == 1)                               // W4
      for (int t = 0; t < kBwdTile; ++t) dv = fmaf(GO[t], H3[t * kRow + s], dv);
    if (tid == 0)
      for (int t = 0; t < kBwdTile; ++t) db4 += GO[t];
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) a[jj] = 0.f;   // dz2 = (W3^T dz3) gelu'(z2)
    layer16_t(sw + kOffW3, G + s * kRow, q, a);
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) Z3[s * kRow + 16 * q + jj] = a[jj] * gelu_grad(Z2[s * kRow + 16 * q + jj]);
    __syncthreads();
    outer16(Z3, H1, tid, d2);
    if (q == 2)                                    // b2
      for (int t = 0; t < kBwdTile; ++t) dv += Z3[t * kRow + s];
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) a[jj] = 0.f;   // dz1 = (W2^T dz2) gelu'(z1)
    layer16_t(sw + kOffW2, Z3 + s * kRow, q, a);
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) G[s * kRow + 16 * q + jj] = a[jj] * gelu_grad(Z1[s * kRow + 16 * q + jj]);
    __syncthreads();
    if (q == 3)                                    // b1
      for (int t = 0; t < kBwdTile; ++t) dv += G[t * kRow + s];
#pragma unroll
    for (int k = 0; k < 2; ++k) {                  // W1
      const int e = tid + k * kBwdThr;
      if (e < kH * kIn)
        for (int t = 0; t < kBwdTile; ++t) dw1[k] = fmaf(G[t * kRow + e / kIn], X[t * kIn + e % kIn], dw1[k]);
    }
  }
  float* out = partials + (size_t)blockIdx.x * kParams;
#pragma unroll
  for (int x = 0; x < 16; ++x) {
    const int e = (4 * (tid >> 4) + x / 4) * kH + 4 * (tid & 15) + x % 4;
    out[kOffW3 + e] = d3[x];
    out[kOffW2 + e] = d2[x];
  }
  out[(q == 0 ? kOffB3 : (q == 1 ? kOffW4 : (q == 2 ? kOffB2 : kOffB1))) + s] = dv;
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (tid + k * kBwdThr < kH * kIn) out[kOffW1 + tid + k * kBwdThr] = dw1[k];
  if (tid == 0) out[kOffB4] = db4;
}

// grad += sum over the blocks of their partials (FP64): 32 parameters per
// block, the partials dealt to 8 rows of threads.
__global__ void __launch_bounds__(256) k_grad_reduce(const float* __restrict__ partials, int nblocks,
                                                    float* __restrict__ grad) {
  __shared__ double red[8][32];
  const int q = blockIdx.x * 32 + threadIdx.x;
  double a = 0.0;
  if (q < mlp::kParams)
    for (int b = threadIdx.y; b < nblocks; b += 8) a += partials[(size_t)b * mlp::kParams + q];
  red[threadIdx.y][threadIdx.x] = a;
  __syncthreads();
  if (threadIdx.y || q >= mlp::kParams) return;
  for (int r = 1; r < 8; ++r) a += red[r][threadIdx.x];
  grad[q] += (float)a;
}

// ------------------------------------------------------------------ Adam
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       size_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ------------------------------------------------- mesh Green's function
// G_S1 and -grad G_S1 at the periodic mesh offsets d/N, d in [0, N)^3, with
// the cell self term at d = 0 (for the PM target, Sec. 3 eq. pmconv).
__global__ void k_mesh_green(int N, float* __restrict__ out) {
  const size_t n3 = (size_t)N * N * N;
  const double inv4pi = 1.0 / (4.0 * green::kPi);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n3; i += (size_t)gridDim.x * blockDim.x) {
    const int ix = (int)(i % N), iy = (int)((i / N) % N), iz = (int)(i / ((size_t)N * N));
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (ix | iy | iz)
      green::gs1((double)ix / N, (double)iy / N, (double)iz / N, v);
    else
      v[0] = -green::cube_mean_inv_r() * N * inv4pi;
    for (int f = 0; f < 4; ++f) out[f * n3 + i] = (float)v[f];
  }
}

// The plan's Green's function on a mesh, for the PM references of Sec. 3:
// periodic (M = N): offsets d/N, d in [0, N)^3, the function the plan
// tabulates; isolated (M = 2N, the zero-padded Hockney mesh): G_0 at signed
// offsets k/N, k in [-N, N) in FFT order.  Self term at d = 0.
__global__ void k_mesh_green_plan(int N, int M, green::Spec gs, double* __restrict__ out) {
  const size_t m3 = (size_t)M * M * M;
  const double inv4pi = 1.0 / (4.0 * green::kPi);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < m3; i += (size_t)gridDim.x * blockDim.x) {
    int k[3] = {(int)(i % M), (int)((i / M) % M), (int)(i / ((size_t)M * M))};
    if (M != N)
      for (int c = 0; c < 3; ++c)
        if (k[c] >= N) k[c] -= M;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (k[0] | k[1] | k[2])
      green::eval(gs, (double)k[0] / N, (double)k[1] / N, (double)k[2] / N, v);
    else
      v[0] = -green::cube_mean_inv_r() * N * inv4pi;
    for (int f = 0; f < 4; ++f) out[f * m3 + i] = v[f];
  }
}

}  // namespace

cudaError_t launch_mesh_green_plan(const Plan& P, double* out, cudaStream_t s) {
  if (!P.iso && P.gspec.kind == 4)   // the function is the mesh itself
    return cudaMemcpyAsync(out, P.gmesh, sizeof(double) * 4 * (size_t)P.N * P.N * P.N, cudaMemcpyDeviceToDevice, s);
  green::Spec g = P.gspec;
  if (P.iso) {
    g = green::Spec();
    g.kind = 2;
  }
  k_mesh_green_plan<<<4 * P.num_sms, 256, 0, s>>>(P.N, P.iso ? 2 * P.N : P.N, g, out);
  return cudaGetLastError();
}

// --------------------------------------------------------------- launchers
cudaError_t launch_residual(const float* phi, const float* acc, const float* tphi, const float* tacc, size_t n3,
                            float w_phi, float w_g, float* lam, double* partials, float* loss, int sms,
                            cudaStream_t s) {
  k_residual<<<4 * sms, 256, 0, s>>>(phi, acc, tphi, tacc, n3, w_phi, w_g, lam, partials);
  k_loss_add<<<1, 32, 0, s>>>(partials, 4 * sms, loss);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_and_table_grad(Plan& P, const float* lam_cells, cudaStream_t s) {
  const int p = P.p, S = P.S, p3 = p * p * p, K = 2 * p;
  // leaf adjoint
  {
    const size_t smem = sizeof(float2) * p * S + sizeof(float) * (4 * S * S * S + 4 * S * S * p + 4 * S * p * p + 4 * p3);
    k_adj_l2p<<<1u << (3 * P.L), 128, smem, s>>>(lam_cells, P.N, S, p, P.w_p2m, P.lam[P.L]);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  for (int l = P.L - 1; l >= 2; --l) {
    const size_t smem = sizeof(float2) * p * K + sizeof(float) * (4 * K * K * K + 4 * K * K * p + 4 * K * p * p + 4 * p3);
    k_adj_l2l<<<1u << (3 * l), 256, smem, s>>>(P.lam[l + 1], p, P.w_m2m, P.lam[l]);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const size_t E = 8 * p - 1;
  for (int l = 2; l <= P.L; ++l) {
    if (P.tg_la && !P.iso) {
      const cudaError_t e = launch_table_grad_spec(P, l, s);
      if (e != cudaSuccess) return e;
      continue;
    }
    cudaError_t e = cudaMemsetAsync(P.dT[l], 0, sizeof(float) * E * E * E * 4, s);
    if (e != cudaSuccess) return e;
    const size_t smem = sizeof(float) * 2 * kTgChunk * p3;
    dim3 grid(P.n_off[l], 8, 4);
    k_table_grad<<<grid, 512, smem, s>>>(P.lam[l], P.M[l], P.offsets[l], P.n_off[l], l, p, P.dT[l]);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t mlp_backward_smem() {
  return sizeof(float) * ((mlp::kParams + 3) / 4 * 4 + kBwdTile * mlp::kIn + 7 * kBwdTile * kRow + kBwdTile);
}

int mlp_backward_blocks(const Plan& P) { return 2 * P.num_sms; }

cudaError_t setup_learn() {
  cudaError_t e = cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mlp_backward_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_table_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_adj_l2l, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_adj_l2p, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

cudaError_t launch_mlp_backward(Plan& P, const float* w, float* grad, cudaStream_t s) {
  cudaError_t e = launch_corr_fold(P, s);
  if (e != cudaSuccess) return e;
  const int tiles = ((P.L - 1) * P.n_corr + kBwdTile - 1) / kBwdTile;
  const int nb = tiles < mlp_backward_blocks(P) ? tiles : mlp_backward_blocks(P);
  k_mlp_backward<<<nb, kBwdThr, mlp_backward_smem(), s>>>(w, P.corr_up, P.corr_samples, P.n_corr, P.L, P.p,
                                                         P.grad_partials);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_grad_reduce<<<(mlp::kParams + 31) / 32, dim3(32, 8), 0, s>>>(P.grad_partials, nb, grad);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* w, const float* g, float* m, float* v, size_t n, int step, float lr, float b1, float b2,
                        float eps, cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<64, 256, 0, s>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_mesh_green(int N, float* out, int sms, cudaStream_t s) {
  k_mesh_green<<<4 * sms, 256, 0, s>>>(N, out);
  return cudaGetLastError();
}

}  // namespace fmm
