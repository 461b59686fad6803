// M2L by spectral products on the tcgen05 tensor cores: the FP32-field levels
// of the mixed forms.
//
// The spectral form of eq. fmm2 (m2l_spec.cu) couples, at one frequency k, the
// 8 children of a target parent P with the 8 children of its 27 neighbour
// parents P + d: with o = c - (2 d + q) for target child c and source child q,
//   F^_{P,c,f}(k) = sum_{d, q} K^_{o,f}(k) M^_{P+d,q}(k)
// (near offsets hold 0).  Written in real and imaginary parts that is one
// dense product per frequency,
//   D[row, P] = sum_{d, e} W_k[row, (d, e)] B_k[(d, e), P],
// rows (c, f, re|im) = 64, e = (q, re|im) = 16, d over 27: the contraction the
// tensor cores take, at 27 x 16 x 64 multiply-adds per frequency and parent
// against 189 x 4 p^3 x p^3 per node of the dense form (p = 6: 11x fewer).
//
// Precision.  Operands are split in two FP16 parts (22 significant bits)
// scaled by powers of two: W per frequency and field, B per level (from the
// largest gridlet mass sum, k_stc_amax), which keeps every value in range; the
// split of BF16 pairs keeps 16 bits.  The 128 rows of an MMA hold W_hi and
// W_lo, and both multiply B_hi and B_lo, so all four products are taken; FP32
// accumulation in TMEM over 27 x 2 MMAs, the two row halves added in FP32.
//
// Kernels
//   k_stc_weights  plan time: the split W_k tiles, in the MMA's K-major core-
//                  matrix layout, and the scales
//   k_stc_amax     per level: the largest sum of |gridlet masses| of a node
//   k_stc_fwd      per parents: FP32 transforms of their children, split to
//                  FP16, [k][split][half of e][z][y][x][8] with a one-parent
//                  halo (periodic copies, or zeros for the isolated problem)
//   k_stc_mac      persistent over the frequencies: W_k (108 KB) stays in
//                  shared memory while the boxes of 8 x 8 x 4 parents pass;
//                  D in two TMEM buffers, drained beside the next box
//   k_stc_inv      per nodes: the inverse transforms
// B operand.  For one (dy, dz) the three dx are windows of one box of 10 x 8 x
// 4 parents, loaded by one TMA copy per (dy, dz) (20 KB: both splits, both
// halves of e): in the no-swizzle K-major layout a row is 16 bytes, so a
// window starts 16 bytes further along x, its 8-row groups are the (y, z) rows
// 160 bytes apart, and 9 copies feed 54 MMAs of 128 x 256 x 16.  Loading the 27
// windows one by one would move 442 KB per box and frequency from L2, 64 bytes
// per clock and SM; this moves 184 KB.
// Measured at 256^3, p = 6 (levels 4 + 5): amax 0.03, forward 0.34, products
// 0.51, inverse 0.25 ms; the same products on the CUDA cores (m2l_spec.cu) 4.2
// ms, the dense bf16x3 contraction 4.78 ms.  512^3, p = 8, level 6: 18.9 ms
// (products 8.3) against 281 ms.  128^3, p = 4, levels 4 + 5: 0.37 against 0.83.
// Error against FP64 there 9.9e-7 (bf16x3: 6.0e-6).
// Every wait is bounded as in m2l_tc.cu: a timeout sets the plan's error word,
// nothing stays in flight, TMEM is freed.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <new>

#include "fmm_internal.cuh"
#include "spec.cuh"
#include "tc_ptx.cuh"

namespace fmm {
namespace {

using spec::forward_line;
using spec::inverse_line;
using spec::inverse_real_line;
using spec::Shape;
using spec::Twiddle;

constexpr int kShifts = 27;
constexpr int kRows = 128;                       // W_hi | W_lo
constexpr int kWTile = kRows * 16 * 2;           // bytes of one shift's W tile: [half 2][128 rows][8]
constexpr int kWBytes = kShifts * kWTile;        // 110 592
constexpr int kBX = 8, kBY = 8, kBZ = 4, kN = kBX * kBY * kBZ;
constexpr int kHalfBytes = (kBX + 2) * kBY * kBZ * 16;   // one (split, half) of a box: 5120
constexpr int kBoxBytes = 4 * kHalfBytes;        // 20 480
constexpr int kStages = 4;
constexpr int kXPad = 2;                         // x origin of the source array (pairs of parents on 32 bytes)
constexpr int kThr = 64 + 128;                   // MMA warp, copy warp, 4 drain warps
constexpr int kExch = 2 * 32 * 64 * 4;           // drain exchange: 2 x [32 columns][64 rows]
constexpr int kSmem = kWBytes + kStages * kBoxBytes + kExch + 1024;
static_assert(kSmem <= 225 * 1024, "shared memory");

// Power-of-two scale that takes values up to `amax` to at most 2^14 (0, NaN and
// infinities keep 1).
__host__ __device__ inline float scale_for(float amax) {
  if (!(amax > 0.f) || amax > 3e38f) return 1.f;
  int e;
  frexpf(amax, &e);                              // amax < 2^e
  e = 14 - e;
  return ldexpf(1.f, e > 120 ? 120 : (e < -120 ? -120 : e));
}

// --------------------------------------------------------------- plan time
// CTA: frequency k.  K^ as k_spec_kernel<P, false> wrote it
// ([chunk of 16][343][2 field pairs][16] float4).
__global__ void __launch_bounds__(256) k_stc_weights(const float* __restrict__ K, uint8_t* __restrict__ W,
                                                    float* __restrict__ inv_scale) {
  const int k = blockIdx.x, tid = threadIdx.x;
  __shared__ float amax[4], sc[4];
  if (tid < 4) amax[tid] = 0.f;
  __syncthreads();
  const float2* Kk = reinterpret_cast<const float2*>(K) + (size_t)(k / 16) * 343 * 64;
  auto value = [&](int o, int f) { return Kk[(size_t)o * 64 + ((f / 2) * 16 + k % 16) * 2 + (f & 1)]; };
  for (int i = tid; i < 343 * 4; i += blockDim.x) {
    const int o = i / 4, ox = o % 7 - 3, oy = (o / 7) % 7 - 3, oz = o / 49 - 3;
    if (abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1) continue;
    const float2 v = value(o, i & 3);
    atomicMax(reinterpret_cast<int*>(&amax[i & 3]), __float_as_int(fmaxf(fabsf(v.x), fabsf(v.y))));
  }
  __syncthreads();
  if (tid < 4) {
    sc[tid] = scale_for(amax[tid]);
    inv_scale[(size_t)k * 4 + tid] = 1.f / sc[tid];
  }
  __syncthreads();
  __half* out = reinterpret_cast<__half*>(W + (size_t)k * kWBytes);
  for (int i = tid; i < kShifts * 64 * 16; i += blockDim.x) {
    const int e = i % 16, row = (i / 16) % 64, s = i / 1024;
    const int c = row >> 3, f = (row >> 1) & 3, ri = row & 1, q = e >> 1, si = e & 1;
    const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    const int ox = (c & 1) - 2 * dx - (q & 1), oy = ((c >> 1) & 1) - 2 * dy - ((q >> 1) & 1),
              oz = (c >> 2) - 2 * dz - (q >> 2);
    float v = 0.f;
    if (!(abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1)) {
      const float2 z = value(((oz + 3) * 7 + oy + 3) * 7 + ox + 3, f);
      v = (ri == si ? z.x : (ri ? z.y : -z.y)) * sc[f];     // (re, im) = (a re' - b im', b re' + a im')
    }
    const __half h = __float2half_rn(v);
    const size_t at = (size_t)s * (kWTile / 2) + (size_t)(e / 8) * kRows * 8 + e % 8;
    out[at + (size_t)row * 8] = h;
    out[at + (size_t)(row + 64) * 8] = __float2half_rn(v - __half2float(h));
  }
}

// ------------------------------------------------------------------ scale
// amax = max over nodes of sum |M_s|, an upper bound of |M^(k)|: one warp per node.
__global__ void __launch_bounds__(256) k_stc_amax(const float* __restrict__ M, int p3, int nodes, float* __restrict__ amax) {
  const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x >> 5);
  float best = 0.f;
  for (int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); n < nodes; n += warps) {
    float a = 0.f;
    for (int i = lane; i < p3; i += 32) a += fabsf(__ldg(M + (size_t)n * p3 + i));
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    best = a > best || a != a ? a : best;
  }
  // non-negative floats (and NaN above them) order as integers
  if (lane == 0) atomicMax(reinterpret_cast<int*>(amax), __float_as_int(best));
}

// -------------------------------------------------------------- transforms
template <int P>
struct StcShape {
  static constexpr int NM = Shape<P>::NM;
  static constexpr int NK = NM * NM * P;
  static constexpr int PB = P >= 7 ? 1 : 2;                 // parents (along x) per forward CTA
  static constexpr int NF = 8 * PB;                         // their children
  static constexpr int NI = P >= 7 ? 2 : (P >= 5 ? 4 : 8);  // nodes per inverse CTA
};

// Children fastest in every shared array, so that a warp's stores of one
// frequency are the adjacent children of adjacent parents.
template <int P>
__global__ void __launch_bounds__(256) k_stc_fwd(const float* __restrict__ M, int level, int iso,
                                                const float* __restrict__ amax, __half2* __restrict__ out) {
  constexpr int NM = StcShape<P>::NM, P3 = P * P * P, NF = StcShape<P>::NF, PB = StcShape<P>::PB;
  extern __shared__ float2 sf[];
  const Twiddle<false, P> wt(nullptr, nullptr);
  float2* t1 = sf;                                          // [z][y][kx][NF]
  float2* t2 = t1 + P3 * NF;                                // [z][ky][kx][NF]
  float* in = reinterpret_cast<float*>(t2);                 // [z][y][x][NF], consumed before t2 is written
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int nh = 1 << (level - 1), bx = nh / PB;
  const int px0 = (int)(blockIdx.x % bx) * PB, py = (int)(blockIdx.x / bx) % nh, pz = (int)blockIdx.x / (bx * nh);
  const float sm = scale_for(*amax);
  for (int i = tid; i < P3 * NF; i += nthr) {
    const int s = i % P3, ch = i / P3;
    const size_t node = 8 * (size_t)morton(px0 + ch / 8, py, pz) + ch % 8;
    in[s * NF + ch] = __ldg(M + node * P3 + s);
  }
  __syncthreads();
  for (int l = tid; l < P * P * NF; l += nthr) {            // x
    const int ch = l % NF, zy = l / NF;
    float x[P];
#pragma unroll
    for (int s = 0; s < P; ++s) x[s] = in[(zy * P + s) * NF + ch];
    forward_line<false, P, true>(
        x, x, wt, [&](int k, float re, float im) { t1[(zy * P + k) * NF + ch] = make_float2(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < P * P * NF; l += nthr) {            // y
    const int ch = l % NF, kx = (l / NF) % P, z = l / (NF * P);
    float xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const float2 c = t1[((z * P + s) * P + kx) * NF + ch];
      xr[s] = c.x;
      xi[s] = c.y;
    }
    forward_line<false, P, false>(
        xr, xi, wt, [&](int k, float re, float im) { t2[((z * NM + k) * P + kx) * NF + ch] = make_float2(re, im); });
  }
  __syncthreads();
  const int WY = nh + 2, WX = nh + 2 * kXPad;
  const size_t plane = (size_t)WX * WY * WY * 4;            // half2 units of one (split, half)
  for (int l = tid; l < NM * P * NF; l += nthr) {           // z
    const int ch = l % NF, q = l / NF;
    float xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const float2 c = t2[(s * NM * P + q) * NF + ch];
      xr[s] = c.x;
      xi[s] = c.y;
    }
    const int px = px0 + ch / 8, child = ch % 8;
    __half2* dst = out + (child >> 2) * plane + (child & 3);
    const size_t at = (((size_t)(pz + 1) * WY + py + 1) * WX + px + kXPad) * 4;
    // the face parents' periodic copies in the halo, as distances along each axis
    const ptrdiff_t ex = iso || (px > 0 && px < nh - 1) ? 0 : (px == 0 ? nh : -nh) * (ptrdiff_t)4;
    const ptrdiff_t ey = iso || (py > 0 && py < nh - 1) ? 0 : (py == 0 ? nh : -nh) * (ptrdiff_t)(4 * WX);
    const ptrdiff_t ez = iso || (pz > 0 && pz < nh - 1) ? 0 : (pz == 0 ? nh : -nh) * (ptrdiff_t)(4 * WX * WY);
    const bool face = ex != 0 || ey != 0 || ez != 0;
    forward_line<false, P, false>(xr, xi, wt, [&](int kz, float re, float im) {
      re *= sm;
      im *= sm;
      const __half2 hi = __floats2half2_rn(re, im);
      const float2 back = __half22float2(hi);
      const __half2 lo = __floats2half2_rn(re - back.x, im - back.y);
      __half2* d = dst + (size_t)(kz * NM * P + q) * 4 * plane + at;
      d[0] = hi;
      d[2 * plane] = lo;
      if (face) {
#pragma unroll 1
        for (int m = 1; m < 8; ++m) {
          if (((m & 1) && !ex) || ((m & 2) && !ey) || ((m & 4) && !ez)) continue;
          const ptrdiff_t o = (m & 1 ? ex : 0) + (m & 2 ? ey : 0) + (m & 4 ? ez : 0);
          d[o] = hi;
          d[o + 2 * (ptrdiff_t)plane] = lo;
        }
      }
    });
  }
}

// Inverse: NI nodes of one parent per CTA, (node, field) fastest everywhere.
template <int P>
__global__ void __launch_bounds__(256) k_stc_inv(const float2* __restrict__ Ph, size_t parents,
                                                float* __restrict__ F) {
  constexpr int NM = StcShape<P>::NM, NI = StcShape<P>::NI, NF = NI * 4, P3 = P * P * P;
  extern __shared__ float2 sf[];
  const Twiddle<false, P> wt(nullptr, nullptr);
  float2* t1 = sf;                                          // [z][ky][kx][NF]
  float2* t2 = t1 + P * NM * P * NF;                        // [z][y][kx][NF]
  const int tid = threadIdx.x, nthr = blockDim.x;
  const size_t node0 = (size_t)blockIdx.x * NI;
  const float2* src = Ph + (node0 >> 3) * 32 + (node0 & 7) * 4;
  for (int l = tid; l < NM * P * NF; l += nthr) {           // z
    const int nf = l % NF, q = l / NF;
    float xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float2 c = __ldg(src + (size_t)(s * NM * P + q) * parents * 32 + nf);
      xr[s] = c.x;
      xi[s] = c.y;
    }
    inverse_line<false, P>(
        xr, xi, wt, [&](int z, float re, float im) { t1[(z * NM * P + q) * NF + nf] = make_float2(re, im); });
  }
  __syncthreads();
  for (int l = tid; l < P * P * NF; l += nthr) {            // y
    const int nf = l % NF, kx = (l / NF) % P, z = l / (NF * P);
    float xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float2 c = t1[((z * NM + s) * P + kx) * NF + nf];
      xr[s] = c.x;
      xi[s] = c.y;
    }
    inverse_line<false, P>(
        xr, xi, wt, [&](int y, float re, float im) { t2[((z * P + y) * P + kx) * NF + nf] = make_float2(re, im); });
  }
  __syncthreads();
  float* out = F + node0 * 4 * P3;
  for (int l = tid; l < P * P * NF; l += nthr) {            // x
    const int nf = l % NF, zy = l / NF;
    float xr[P], xi[P];
#pragma unroll
    for (int s = 0; s < P; ++s) {
      const float2 c = t2[(zy * P + s) * NF + nf];
      xr[s] = c.x;
      xi[s] = c.y;
    }
    // values parked in t1's space, so that the store runs along memory
    inverse_real_line<false, P>(
        xr, xi, wt, [&](int x, float v) { reinterpret_cast<float*>(t1)[nf * (P3 | 1) + zy * P + x] = v; });
  }
  __syncthreads();
  for (int i = tid; i < NF * P3; i += nthr) out[i] = reinterpret_cast<float*>(t1)[(i / P3) * (P3 | 1) + i % P3];
}

// ---------------------------------------------------------------- products
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  tc::mma_bf16(d, a, b, idesc, acc);             // kind::f16; the operand type is in the descriptor
}

__global__ void __launch_bounds__(kThr, 1)
k_stc_mac(const __grid_constant__ CUtensorMap mapB, const uint8_t* __restrict__ W, const float* __restrict__ inv_w,
          const float* __restrict__ amax, int nk, int parts, int level, float* __restrict__ Ph, int* __restrict__ err,
          uint64_t wait_ns, int stall) {
  // D FP32, A and B FP16 (format 0), both K-major, M = 128, N = 256
  constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(kN >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
  extern __shared__ uint8_t smem[];
  __shared__ uint64_t wfull, wfree, full[kStages], empty[kStages], pfull[2], pfree[2], mdone;
  __shared__ uint32_t tmem_holder;
  __shared__ int s_err, d_err;                    // any role gave up; a drain wait gave up
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nh = 1 << (level - 1), tx = nh / kBX, ty = nh / kBY, tiles = tx * ty * (nh / kBZ);
  const size_t parents = (size_t)1 << (3 * (level - 1));
  const uint32_t base = (tc::smem_u32(smem) + 1023u) & ~1023u;
  const uint32_t sW = base, sB = base + kWBytes;
  float* exch = reinterpret_cast<float*>(smem + (base - tc::smem_u32(smem)) + kWBytes + kStages * kBoxBytes);
  if (tid == 0) {
    s_err = d_err = 0;
    tc::mbar_init(&wfull, 1);
    tc::mbar_init(&wfree, 1);
    for (int i = 0; i < kStages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&pfull[i], 1);
      tc::mbar_init(&pfree[i], 128);
    }
    tc::mbar_init(&mdone, 1);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(&tmem_holder, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_holder;
  // this CTA's units: unit v = (frequency v / parts, part v % parts of the boxes)
  const int units = nk * parts, tpp = tiles / parts;
  const int nmine = (int)blockIdx.x < units ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp == 0) {
    // -------------------------------------------------------- MMA issuer
    if (lane == 0) {
      bool ok = true;
      int it = 0, u = 0;                          // stages, boxes
      for (int m = 0; m < nmine && ok && !stall; ++m) {
        if (!tc::mbar_wait_bounded(&wfull, (uint32_t)m & 1u, wait_ns)) {
          ok = false;
          break;
        }
        for (int t = 0; t < tpp && ok; ++t, ++u) {
          const uint32_t part = tmem + (uint32_t)((u & 1) * kN);
          if (u >= 2 && !tc::mbar_wait_bounded(&pfree[u & 1], (uint32_t)(u / 2 - 1) & 1u, wait_ns)) {
            ok = false;
            break;
          }
          for (int g = 0; g < 9; ++g, ++it) {
            const int st = it % kStages;
            if (!tc::mbar_wait_bounded(&full[st], (uint32_t)(it / kStages) & 1u, wait_ns)) {
              ok = false;
              break;
            }
            tc::fence_after_sync();
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              const uint64_t ad = tc::smem_desc(sW + (g * 3 + dx) * kWTile, kRows * 16, 128);
#pragma unroll
              for (int sp = 0; sp < 2; ++sp) {
                const uint64_t bd =
                    tc::smem_desc(sB + st * kBoxBytes + sp * 2 * kHalfBytes + dx * 16, kHalfBytes, (kBX + 2) * 16);
                mma_f16(part, ad, bd, IDESC, (g | dx | sp) ? 1u : 0u);
              }
            }
            tc::mma_commit(&empty[st]);
          }
          if (ok) tc::mma_commit(&pfull[u & 1]);
        }
        if (ok) tc::mma_commit(&wfree);
      }
      tc::mma_commit(&mdone);
      if (!tc::mbar_wait_bounded(&mdone, 0u, wait_ns)) ok = false;
      if (!ok || stall) atomicExch(&s_err, 1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------- copy thread
    if (lane == 0) {
      bool ok = true;
      int it = 0, wloads = 0;
      for (int m = 0; m < nmine && ok; ++m) {
        const int v = (int)blockIdx.x + m * (int)gridDim.x, k = v / parts, t0 = v % parts * tpp;
        if (m > 0 && !tc::mbar_wait_bounded(&wfree, (uint32_t)(m - 1) & 1u, wait_ns)) {
          ok = false;
          break;
        }
        tc::mbar_arrive_expect_tx(&wfull, kWBytes);
        for (int s = 0; s < kShifts; ++s)
          tc::bulk_g2s(sW + s * kWTile, W + (size_t)k * kWBytes + (size_t)s * kWTile, kWTile, &wfull);
        ++wloads;
        for (int t = t0; t < t0 + tpp && ok; ++t) {
          const int bx = (t % tx) * kBX, by = ((t / tx) % ty) * kBY, bz = t / (tx * ty) * kBZ;
          for (int g = 0; g < 9; ++g) {
            const int st = it % kStages, dy = g % 3, dz = g / 3;       // 0..2: the shift + the halo of 1
            if (!tc::mbar_wait_bounded(&empty[st], ((uint32_t)(it / kStages) & 1u) ^ 1u, wait_ns)) {
              ok = false;
              break;
            }
            tc::mbar_arrive_expect_tx(&full[st], kBoxBytes);
            tc::tma_load_4d(sB + st * kBoxBytes, &mapB, (bx + kXPad - 1) * 8, by + dy, bz + dz, k * 4, &full[st]);
            ++it;
          }
        }
      }
      // the copies issued last may not have been consumed (after a timeout):
      // wait (bounded) until each has landed
      for (int i = it - kStages > 0 ? it - kStages : 0; i < it; ++i)
        if (!tc::mbar_wait_bounded(&full[i % kStages], (uint32_t)(i / kStages) & 1u, wait_ns)) ok = false;
      if (wloads && !tc::mbar_wait_bounded(&wfull, (uint32_t)(wloads - 1) & 1u, wait_ns)) ok = false;
      if (!ok) atomicExch(&s_err, 1);
    }
    __syncwarp();
  } else {
    // -------------------------------------------------------- drain warps
    // TMEM lanes (rows): quadrants 0, 1 hold the W_hi rows, 2, 3 the W_lo rows
    // of the same 64; the latter pass through shared memory.
    const int q = warp & 3;
    const uint32_t lanebase = (uint32_t)(q * 32) << 16;
    const int row = (q & 1) * 32 + lane;           // 0..63
    const bool lo = q >= 2;
    const float inv_m = 1.f / scale_for(*amax);
    bool ok = true;
    int u = 0, turn = 0;
    for (int m = 0; m < nmine && ok; ++m) {
      const int v = (int)blockIdx.x + m * (int)gridDim.x, k = v / parts, t0 = v % parts * tpp;
      const float sc = inv_m * __ldg(inv_w + (size_t)k * 4 + ((row >> 1) & 3));
      for (int t = t0; t < t0 + tpp && ok; ++t, ++u) {
        const int bx = (t % tx) * kBX, by = ((t / tx) % ty) * kBY, bz = t / (tx * ty) * kBZ;
        // the wait's outcome must be common to the 128 drain threads (they meet at a named barrier)
        const bool got = tc::mbar_wait_bounded(&pfull[u & 1], (uint32_t)(u / 2) & 1u, wait_ns);
        if (!got) atomicExch(&d_err, 1);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        ok = atomicAdd(&d_err, 0) == 0;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (!ok) break;
        tc::fence_after_sync();
        const uint32_t part = tmem + (uint32_t)((u & 1) * kN) + lanebase;
        for (int c0 = 0; c0 < kN; c0 += 32, turn ^= 1) {
          uint32_t r[32];
          tc::tmem_ld32_nowait(part + c0, r);
          tc::tmem_wait_ld();
          float* ex = exch + turn * 32 * 64;
          if (lo) {
#pragma unroll
            for (int c = 0; c < 32; ++c) ex[c * 64 + row] = __uint_as_float(r[c]);
          }
          // one barrier per chunk: the two exchange buffers alternate, so the
          // buffer written next was read before the barrier just passed
          asm volatile("bar.sync 1, 128;" ::: "memory");
          if (!lo) {
#pragma unroll
            for (int c = 0; c < 32; ++c) {
              const int col = c0 + c;
              const uint32_t par = morton(bx + (col & 7), by + ((col >> 3) & 7), bz + (col >> 6));
              Ph[((size_t)k * parents + par) * 64 + row] = (__uint_as_float(r[c]) + ex[c * 64 + row]) * sc;
            }
          }
        }
        tc::fence_before_sync();
        tc::mbar_arrive(&pfree[u & 1]);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
  if (tid == 0 && (s_err | d_err)) atomicExch(err, 1);
}

template <int P>
size_t stc_fwd_smem() {
  constexpr int NF = StcShape<P>::NF, NM = StcShape<P>::NM;
  return sizeof(float2) * NF * (P * P * P + P * NM * P);
}
template <int P>
size_t stc_inv_smem() {
  constexpr int NF = StcShape<P>::NI * 4, NM = StcShape<P>::NM;
  return sizeof(float2) * NF * (P * NM * P + P * P * P);
}

template <typename F>
cudaError_t opt_in(F* f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int P>
cudaError_t setup_p() {
  cudaError_t e;
  if ((e = opt_in(k_stc_fwd<P>, stc_fwd_smem<P>())) != cudaSuccess) return e;
  if ((e = opt_in(k_stc_inv<P>, stc_inv_smem<P>())) != cudaSuccess) return e;
  return opt_in(k_stc_mac, kSmem);
}

template <int P>
cudaError_t launch_p(Plan& Pl, int level, cudaStream_t s) {
  constexpr int NK = StcShape<P>::NK;
  const size_t nodes = (size_t)1 << (3 * level), parents = nodes / 8;
  float* amax = static_cast<float*>(Pl.stc_amax[level]);
  cudaError_t e = cudaMemsetAsync(amax, 0, sizeof(float), s);
  if (e != cudaSuccess) return e;
  const size_t want = (nodes + 63) / 64;            // 8 nodes per warp at least
  const unsigned blocks = (unsigned)(want < (size_t)(4 * Pl.num_sms) ? want : (size_t)(4 * Pl.num_sms));
  k_stc_amax<<<blocks, 256, 0, s>>>(Pl.M[level], P * P * P, (int)nodes, amax);
  k_stc_fwd<P><<<(unsigned)(parents / StcShape<P>::PB), 256, stc_fwd_smem<P>(), s>>>(
      Pl.M[level], level, Pl.iso, amax, static_cast<__half2*>(Pl.stc_B[level]));
  // few frequencies: halves of the boxes (196 frequencies of p = 4 are 1.3
  // waves, rounded up to 2; 392 halves 2.6, to 1.5 frequencies' time); nh >= 8, so the tiles are even in number
  const int parts = NK < 3 * Pl.num_sms ? 2 : 1;
  const unsigned grid = NK * parts < Pl.num_sms ? NK * parts : Pl.num_sms;
  k_stc_mac<<<grid, kThr, kSmem, s>>>(*static_cast<const CUtensorMap*>(Pl.stc_map[level]),
                                     static_cast<const uint8_t*>(Pl.stc_W[level]),
                                     static_cast<const float*>(Pl.stc_scale[level]), amax, NK, parts, level,
                                     static_cast<float*>(Pl.spec_P[level]), Pl.d_err, Pl.wait_ns, Pl.inject_stall);
  k_stc_inv<P><<<(unsigned)(nodes / StcShape<P>::NI), 256, stc_inv_smem<P>(), s>>>(
      static_cast<const float2*>(Pl.spec_P[level]), parents, Pl.F[level]);
  return cudaGetLastError();
}

int nk_of(int p) { return (2 * p - 1) * (2 * p - 1) * p; }

}  // namespace

void stc_bytes(const Plan& P, int level, size_t& nW, size_t& nB, size_t& nS) {
  const size_t nh = (size_t)1 << (level - 1);
  nW = (size_t)nk_of(P.p) * kWBytes;
  nB = (size_t)nk_of(P.p) * 4 * (nh + 2 * kXPad) * (nh + 2) * (nh + 2) * 16;
  nS = (size_t)nk_of(P.p) * 4 * sizeof(float);
}

// The 4-D map of a level's split spectra: dims (x units of 8 halves, y, z,
// frequency x split x half), box (10 units, 8, 4, 4).
int make_stc_map(Plan& P, int level) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return FMM_ERR_CUDA;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  CUtensorMap* map = new (std::nothrow) CUtensorMap;
  if (!map) return FMM_ERR_ALLOC;
  const cuuint64_t nh = (cuuint64_t)1 << (level - 1), WX = nh + 2 * kXPad, WY = nh + 2;
  const cuuint64_t dims[4] = {WX * 8, WY, WY, (cuuint64_t)nk_of(P.p) * 4};
  const cuuint64_t strides[3] = {WX * 16, WX * 16 * WY, WX * 16 * WY * WY};
  const cuuint32_t box[4] = {(kBX + 2) * 8, kBY, kBZ, 4};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, P.stc_B[level], dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {      // a level with a map counts as prepared: keep none that failed
    delete map;
    return FMM_ERR_CUDA;
  }
  P.stc_map[level] = map;
  return FMM_OK;
}

cudaError_t setup_spec_tc(const Plan& P) {
  switch (P.p) {
    case 4: return setup_p<4>();
    case 5: return setup_p<5>();
    case 6: return setup_p<6>();
    case 7: return setup_p<7>();
    case 8: return setup_p<8>();
    default: return cudaSuccess;
  }
}

cudaError_t launch_stc_weights(Plan& P, int level, cudaStream_t s) {
  k_stc_weights<<<nk_of(P.p), 256, 0, s>>>(static_cast<const float*>(P.spec_K[level]),
                                          static_cast<uint8_t*>(P.stc_W[level]), static_cast<float*>(P.stc_scale[level]));
  return cudaGetLastError();
}

cudaError_t launch_m2l_spec_tc(Plan& P, int level, cudaStream_t s) {
  switch (P.p) {
    case 4: return launch_p<4>(P, level, s);
    case 5: return launch_p<5>(P, level, s);
    case 6: return launch_p<6>(P, level, s);
    case 7: return launch_p<7>(P, level, s);
    case 8: return launch_p<8>(P, level, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fmm
