// Table gradient of the training step by spectral products, and the learned
// correction evaluated and differentiated on the distinct table entries only.
//
// Table gradient.  For one interaction offset o, lag d in [-(p-1), p-1]^3 and
// field f, dJ/dT[o p + d][f] gathers
//   g_o(d) = sum_T sum_r lam_T[f][r] M_{T-o}[r - d]
// over the targets T whose interaction zone holds T - o: a correlation, which
// on the zero-padded NM = 2p - 1 grid of m2l_spec.cu is
//   g^_o(k) = sum_T lam^_T(k) conj(M^_{T-o}(k)),
// one complex multiply-add per frequency and field where the direct sum over
// (r, d) takes p^6 / NK times as many.  Measured at 64^3, p = 6 (levels 2 + 3,
// 8 fields): 224 ms for the direct sums, 2.3 ms here.
//
// Correction.  The network sees a table entry only through the sorted absolute
// components of its (nearest-image) offset, so the (8p-1)^3 x 4 entries of a
// level hold about 1/40 as many distinct inputs.  The network runs once per
// distinct input (k_corr_eval); the table gradient is folded onto them before
// the backward pass (k_corr_fold), which is linear in the upstream gradient.
#include <vector>

#include "fmm_internal.cuh"
#include "mlp.cuh"
#include "spec.cuh"

namespace fmm {
namespace {

using spec::chunks_of;
using spec::inverse_line;
using spec::Num;
using spec::Shape;
using spec::Twiddle;
using spec::widen;

constexpr int kOff3 = 343;
constexpr int kLn = 16;                 // frequencies per chunk (FP32)
constexpr int kTgGroups = 8;            // target rows in flight per CTA
constexpr int kTgChain = 32;            // steps (of two targets) per FP32 chain

// Offsets a child at position c of its parent takes, per axis.
template <int MODE>   // 0: levels >= 3; 1: level 2, periodic
__device__ __forceinline__ constexpr bool allowed(int c, int o) {
  return MODE == 0 ? (c ? o >= -2 : o <= 2) : (o >= -1 && o <= 2);
}

// CTA: one row of offsets (oy, oz; the 7 ox) x one chunk of 16 frequencies.
// Lane: a frequency; the 8 groups of 16 lanes walk the (z, y) rows of targets,
// two targets (one parent's x pair) per step, whose 6 sources along x serve
// both.  56 sums per thread; every kTgChain steps they are added to the group's
// totals in shared memory, so that the FP32 chains do not grow with the level;
// the groups are added at the end.  Bound by the FP32 pipe (192 multiply-adds
// per 14 eight-byte loads from L1/L2).
// Error of the table gradient against FP64, relative, at the leaf level: direct
// sums 7.0e-8 to 7.9e-8 (128^3, L = 5, p = 4), 6.6e-8 to 7.8e-8 (192^3, L = 6,
// p = 3); with one chain per group and FP32 transforms 1.4e-7 to 1.7e-7, 3.3e-7
// to 3.6e-7; with these chains and double-float transforms, rounded on store,
// 6.2e-8 to 7.9e-8, 6.6e-8 to 7.7e-8.  The training step of 8 fields at 64^3,
// p = 6 takes 7.4 ms with them, 6.6 without.
template <int MODE>
__device__ __forceinline__ void tg_rows(const float2* __restrict__ La, const float2* __restrict__ Mh, int level, int oy,
                                        int oz, int grp, float2 (*tot)[kLn]) {
  const int n = 1 << level;
  float2 acc[7][4];
  auto flush = [&](bool first) {
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        float2& t = tot[i * 4 + f][0];
        t = first ? make_float2(0.f, 0.f) : make_float2(t.x + acc[i][f].x, t.y + acc[i][f].y);
        acc[i][f] = make_float2(0.f, 0.f);
      }
  };
  flush(true);
  int steps = 0;
  const bool near = oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1;
  for (int r = grp; r < n * n; r += kTgGroups) {
    const int y = r % n, z = r / n;
    if (!allowed<MODE>(y & 1, oy) || !allowed<MODE>(z & 1, oz)) continue;
    const uint32_t ts = (spread3(y) << 1) | (spread3(z) << 2);
    const uint32_t ss = (spread3((y - oy) & (n - 1)) << 1) | (spread3((z - oz) & (n - 1)) << 2);
    for (int x = 0; x < n; x += 2) {
      float2 m[6], l[2][4];
#pragma unroll
      for (int h = 0; h < 6; ++h) m[h] = __ldg(Mh + (size_t)(spread3((x - 2 + h) & (n - 1)) | ss) * kLn);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int f = 0; f < 4; ++f) l[j][f] = __ldg(La + ((size_t)(spread3(x + j) | ts) * 4 + f) * kLn);
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        const int ox = i - 3;
        if (ox >= -1 && ox <= 1 && near) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int h = j + 2 - ox;
          if (!allowed<MODE>(j, ox) || h < 0 || h >= 6) continue;
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            acc[i][f].x = fmaf(l[j][f].x, m[h].x, acc[i][f].x);
            acc[i][f].y = fmaf(l[j][f].y, m[h].x, acc[i][f].y);
            acc[i][f].x = fmaf(l[j][f].y, m[h].y, acc[i][f].x);
            acc[i][f].y = fmaf(-l[j][f].x, m[h].y, acc[i][f].y);
          }
        }
      }
      if (++steps == kTgChain) {
        flush(false);
        steps = 0;
      }
    }
  }
  flush(false);
}

__global__ void __launch_bounds__(kLn* kTgGroups) k_tg_mac(const float2* __restrict__ La, const float2* __restrict__ Mh,
                                                          int level, int nkp, float2* __restrict__ out) {
  const int tid = threadIdx.x, fr = tid % kLn, grp = tid / kLn;
  const int row = blockIdx.x, chunk = blockIdx.y, oy = row % 7 - 3, oz = row / 7 - 3;
  const size_t nodes = (size_t)1 << (3 * level);
  La += (size_t)chunk * (4 * nodes + 1) * kLn + fr;
  Mh += (size_t)chunk * (nodes + 1) * kLn + fr;
  __shared__ float2 red[kTgGroups][28][kLn];
  float2(*tot)[kLn] = reinterpret_cast<float2(*)[kLn]>(&red[grp][0][fr]);   // this thread's column
  if (level > 2)
    tg_rows<0>(La, Mh, level, oy, oz, grp, tot);
  else
    tg_rows<1>(La, Mh, level, oy, oz, grp, tot);
  __syncthreads();
  for (int q = grp; q < 28; q += kTgGroups) {
    float2 v = red[0][q][fr];
#pragma unroll
    for (int g = 1; g < kTgGroups; ++g) {
      v.x += red[g][q][fr].x;
      v.y += red[g][q][fr].y;
    }
    out[((size_t)row * 28 + q) * nkp + chunk * kLn + fr] = v;   // [o][f][nkp]
  }
}

// Lags g_o(d) of one (offset, field): CTA, three separable inverse passes over
// all NM points of each axis, in double-float with one rounding at the end.
// out [o][f][dz][dy][dx], index d mod NM.
template <int P>
size_t inv_smem() {
  return 2 * sizeof(float4) * Shape<P>::NM * Shape<P>::NM * P;
}
template <int P>
__global__ void __launch_bounds__(128) k_tg_inv(const float2* __restrict__ G, int nkp, const float4* __restrict__ twg,
                                               float* __restrict__ out) {
  using T = Num<true>;
  constexpr int NM = Shape<P>::NM;
  extern __shared__ float4 sg[];
  __shared__ float4 tw[NM];
  float4* t1 = sg;                        // [z][ky][kx]
  float4* t2 = sg + NM * NM * P;          // [z][y][kx]
  const int tid = threadIdx.x, o = blockIdx.x / 4;
  const int ox = o % 7 - 3, oy = (o / 7) % 7 - 3, oz = o / 49 - 3;
  if (abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1) return;   // near nodes: never gathered
  if (tid < NM) tw[tid] = __ldg(twg + tid);
  __syncthreads();
  const float2* src = G + (size_t)blockIdx.x * nkp;
  const Twiddle<true, P> wt(twg, tw);
  for (int q = tid; q < NM * P; q += blockDim.x) {
    float2 xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float2 c = __ldg(src + s * NM * P + q);
      xr[s] = widen<true>(c.x);
      xi[s] = widen<true>(c.y);
    }
    inverse_line<true, P, true>(xr, xi, wt, [&](int z, float2 re, float2 im) { t1[z * NM * P + q] = T::pack(re, im); });
  }
  __syncthreads();
  for (int q = tid; q < NM * P; q += blockDim.x) {            // line (z, kx)
    const int kx = q % P, z = q / P;
    float2 xr[NM], xi[NM];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
      const float4 c = t1[(z * NM + s) * P + kx];
      xr[s] = T::re(c);
      xi[s] = T::im(c);
    }
    inverse_line<true, P, true>(xr, xi, wt,
                                [&](int y, float2 re, float2 im) { t2[(z * NM + y) * P + kx] = T::pack(re, im); });
  }
  __syncthreads();
  const float2 scale = df_from_double(1.0 / ((double)NM * NM * NM));
  for (int i = tid; i < NM * NM * NM; i += blockDim.x) {
    const int x = i % NM;
    const float4* v = t2 + (i / NM) * P;
    float2 a = T::zero(), g = T::zero();
    int j = x;
#pragma unroll
    for (int s = 1; s < P; ++s) {
      const float4 w = tw[j];
      T::mac(a, w.x, w.y, T::re(v[s]));
      T::mac(a, -w.z, -w.w, T::im(v[s]));
      j += x;
      j -= j >= NM ? NM : 0;
    }
    T::mac(g, scale.x, scale.y, T::add(T::twice(T::done(a)), T::re(v[0])));
    out[(size_t)blockIdx.x * NM * NM * NM + i] = g.x + g.y;
  }
}

// dT[n][f] = sum of g_o(n - o p) over the (at most 2 per axis) offsets o whose
// window holds n and that the level's interaction lists contain.
__global__ void k_tg_gather(const float* __restrict__ g, int p, int level, float* __restrict__ dT) {
  const int E = 8 * p - 1, HW = 4 * p - 1, NM = 2 * p - 1, NM3 = NM * NM * NM;
  const int lo = level == 2 ? -1 : -3, hi = level == 2 ? 2 : 3;
  const long total = (long)E * E * E * 4;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int f = (int)(i % 4);
    const long e = i / 4;
    const int n[3] = {(int)(e % E) - HW, (int)((e / E) % E) - HW, (int)(e / ((long)E * E)) - HW};
    int o0[3], cnt[3];
    for (int a = 0; a < 3; ++a) {
      const int q = (n[a] + 4 * p) / p - 4;                   // floor(n / p)
      o0[a] = q;
      cnt[a] = n[a] == q * p ? 1 : 2;                         // lag 0, or the windows of q and q + 1
    }
    float v = 0.f;
    for (int cz = 0; cz < cnt[2]; ++cz)
      for (int cy = 0; cy < cnt[1]; ++cy)
        for (int cx = 0; cx < cnt[0]; ++cx) {
          const int ox = o0[0] + cx, oy = o0[1] + cy, oz = o0[2] + cz;
          if (ox < lo || ox > hi || oy < lo || oy > hi || oz < lo || oz > hi) continue;
          if (ox >= -1 && ox <= 1 && oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1) continue;
          const int dx = (n[0] - ox * p + NM) % NM, dy = (n[1] - oy * p + NM) % NM, dz = (n[2] - oz * p + NM) % NM;
          const int o = ((oz + 3) * 7 + (oy + 3)) * 7 + ox + 3;
          v += __ldg(g + ((size_t)o * 4 + f) * NM3 + (dz * NM + dy) * NM + dx);
        }
    dT[i] = v;
  }
}

template <int P>
cudaError_t inv_p(const float2* G, int nkp, const float4* tw, float* out, cudaStream_t s) {
  k_tg_inv<P><<<kOff3 * 4, 128, inv_smem<P>(), s>>>(G, nkp, tw, out);
  return cudaGetLastError();
}

// ------------------------------------------------------ distinct network inputs
// A sample packs (class, a, b, c): class 0 with a <= b <= c for G, class 1 with
// a the own component and b <= c for -dG/dx_i.  Its value sits at
// corr[level - 2][class][a][b][c], 4p per axis.
__host__ __device__ inline uint32_t pack_sample(int cls, int a, int b, int c) {
  return (uint32_t)cls << 24 | (uint32_t)a << 16 | (uint32_t)b << 8 | (uint32_t)c;
}

// Upstream gradient of a sample: the table gradients of every entry that folds
// onto it, each times the sign it is applied with, summed in FP64.  Eight lanes
// per sample share its up to 6 x 64 entries.
constexpr int kFoldLanes = 8;
__global__ void k_corr_fold(const float* __restrict__ dT_all, const uint32_t* __restrict__ samples, int ns, int p,
                            int lmax, float* __restrict__ up) {
  const int E = 8 * p - 1, HW = 4 * p - 1;
  const int total = (lmax - 1) * ns;
  const int sub = threadIdx.x % kFoldLanes, i = (blockIdx.x * blockDim.x + threadIdx.x) / kFoldLanes;
  double sum = 0.0;
  const bool valid = i < total;
  if (valid) {
    const int level = 2 + i / ns;
    const uint32_t s = samples[i % ns];
    const int cls = s >> 24, v[3] = {(int)(s >> 16) & 255, (int)(s >> 8) & 255, (int)s & 255};
    const int period = (1 << level) * p;
    const float* dT = dT_all + (size_t)(level - 2) * E * E * E * 4;
    // half the box: sign 0
    if (!(cls && 2 * v[0] == period))
    for (int f = cls ? 1 : 0; f < (cls ? 4 : 1); ++f) {
      // arrangements of (a, b, c) on the axes: all distinct ones (G), or own on
      // axis f - 1 and the two distinct orders of (b, c)
      for (int perm = 0; perm < 6; ++perm) {
        const int P3[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
        int w[3];
        for (int a = 0; a < 3; ++a) w[a] = v[P3[perm][a]];
        if (cls) {
          if (P3[perm][f - 1] != 0) continue;
          if (v[1] == v[2]) {
            bool first = true;                                // b = c: one order only
            for (int q = 0; q < perm; ++q)
              if (P3[q][f - 1] == 0) first = false;
            if (!first) continue;
          }
        } else {
          bool seen = false;                                  // equal components: skip repeats
          for (int q = 0; q < perm && !seen; ++q)
            seen = v[P3[q][0]] == w[0] && v[P3[q][1]] == w[1] && v[P3[q][2]] == w[2];
          if (seen) continue;
        }
        // preimages per axis: +-w, and, where the box is no larger than the
        // table, +-(period - w)
        int pre[3][4], np[3];
        for (int a = 0; a < 3; ++a) {
          np[a] = 0;
          const int cand[4] = {w[a], -w[a], period - w[a], w[a] - period};
          for (int q = 0; q < 4; ++q) {
            const int wr = mlp::wrap_offset(cand[q], period);
            bool ok = cand[q] >= -HW && cand[q] <= HW && (wr < 0 ? -wr : wr) == w[a];
            for (int r = 0; r < q && ok; ++r) ok = cand[r] != cand[q];
            if (ok) pre[a][np[a]++] = cand[q];
          }
        }
        for (int e = sub; e < np[0] * np[1] * np[2]; e += kFoldLanes) {
          const int n[3] = {pre[0][e % np[0]], pre[1][(e / np[0]) % np[1]], pre[2][e / (np[0] * np[1])]};
          if (!(n[0] | n[1] | n[2])) continue;
          double sg = 1.0;
          if (cls) sg = mlp::wrap_offset(n[f - 1], period) > 0 ? 1.0 : -1.0;
          sum += sg * (double)__ldg(dT + (((size_t)(n[2] + HW) * E + n[1] + HW) * E + n[0] + HW) * 4 + f);
        }
      }
    }
    const double base = (double)(1 << level) * p;
    sum *= mlp::kKappa * (cls ? base * base : base) / (4.0 * 3.14159265358979323846);
  }
  for (int o = kFoldLanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (valid && sub == 0) up[i] = (float)sum;
}

// The network at every distinct input of every level: one warp per sample, two
// neurons per lane, weights in shared memory (rows padded to 65 floats).
constexpr int kEvalWarps = 8;
constexpr int kWPad = mlp::kH + 1;
template <bool BF16>
__global__ void __launch_bounds__(32 * kEvalWarps) k_corr_eval(const float* __restrict__ w,
                                                              const uint32_t* __restrict__ samples, int ns, int p,
                                                              int lmax, float* __restrict__ corr) {
  using namespace mlp;
  extern __shared__ float se[];
  float* W2 = se;                          // [64][65]
  float* W3 = W2 + kH * kWPad;             // [64][65]
  float* W1 = W3 + kH * kWPad;             // [64][5]
  float* bias = W1 + kH * kIn;             // b1 | b2 | b3 | W4 | b4
  float* hs = bias + 4 * kH + 1;           // [warp][64]
  auto rd = [&](float v) { return BF16 ? round_bf16(v) : v; };
  for (int i = threadIdx.x; i < kH * kH; i += blockDim.x) {
    W2[(i / kH) * kWPad + i % kH] = rd(w[kOffW2 + i]);
    W3[(i / kH) * kWPad + i % kH] = rd(w[kOffW3 + i]);
  }
  for (int i = threadIdx.x; i < kH * kIn; i += blockDim.x) W1[i] = rd(w[kOffW1 + i]);
  for (int i = threadIdx.x; i < kH; i += blockDim.x) {
    bias[i] = w[kOffB1 + i];
    bias[kH + i] = w[kOffB2 + i];
    bias[2 * kH + i] = w[kOffB3 + i];
    bias[3 * kH + i] = rd(w[kOffW4 + i]);
  }
  if (threadIdx.x == 0) bias[4 * kH] = w[kOffB4];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = 4 * p, total = (lmax - 1) * ns;
  float* h = hs + warp * kH;
  const float inv = 1.f / (4.f * p);
  for (int i = blockIdx.x * kEvalWarps + warp; i < total; i += gridDim.x * kEvalWarps) {
    const int level = 2 + i / ns;
    const uint32_t s = samples[i % ns];
    const int cls = s >> 24, a = (s >> 16) & 255, b = (s >> 8) & 255, c = s & 255;
    const float x[kIn] = {rd(a * inv), rd(b * inv), rd(c * inv), rd(level * 0.125f), (float)cls};
    float z[2];
    for (int k = 0; k < 2; ++k) {
      const int q = lane + 32 * k;
      z[k] = bias[q];
      for (int j = 0; j < kIn; ++j) z[k] = fmaf(W1[q * kIn + j], x[j], z[k]);
    }
    for (int layer = 0; layer < 2; ++layer) {
      __syncwarp();
      for (int k = 0; k < 2; ++k) h[lane + 32 * k] = rd(gelu(z[k]));
      __syncwarp();
      const float* W = layer ? W3 : W2;
      for (int k = 0; k < 2; ++k) z[k] = bias[(layer + 1) * kH + lane + 32 * k];
#pragma unroll 8
      for (int j = 0; j < kH; ++j) {
        z[0] = fmaf(W[lane * kWPad + j], h[j], z[0]);
        z[1] = fmaf(W[(lane + 32) * kWPad + j], h[j], z[1]);
      }
    }
    float o = fmaf(bias[3 * kH + lane], rd(gelu(z[0])), bias[3 * kH + lane + 32] * rd(gelu(z[1])));
    for (int d = 16; d > 0; d >>= 1) o += __shfl_xor_sync(0xffffffffu, o, d);
    if (lane == 0) corr[((((size_t)(level - 2) * 2 + cls) * G + a) * G + b) * G + c] = o + bias[4 * kH];
  }
}
size_t eval_smem() {
  return sizeof(float) * (2 * mlp::kH * kWPad + mlp::kH * mlp::kIn + 4 * mlp::kH + 1 + kEvalWarps * mlp::kH);
}

}  // namespace

// The distinct inputs of order p.  Components run over [0, 4p); own = 0 carries
// sign 0 and is left out (half the box, which also does, depends on the level
// and is dropped where it is used).
std::vector<uint32_t> corr_samples(int p) {
  const int G = 4 * p;
  std::vector<uint32_t> v;
  for (int a = 0; a < G; ++a)
    for (int b = a; b < G; ++b)
      for (int c = b; c < G; ++c)
        if (a | b | c) v.push_back(pack_sample(0, a, b, c));
  for (int a = 1; a < G; ++a)
    for (int b = 0; b < G; ++b)
      for (int c = b; c < G; ++c) v.push_back(pack_sample(1, a, b, c));
  return v;
}

size_t corr_values(const Plan& P) {
  const size_t G = 4 * (size_t)P.p;
  return (size_t)(P.L - 1) * 2 * G * G * G;
}

cudaError_t launch_corr_eval(Plan& P, cudaStream_t s) {
  const unsigned blocks = (unsigned)P.num_sms * 2;
  if (P.corr_fp32)
    k_corr_eval<false><<<blocks, 32 * kEvalWarps, eval_smem(), s>>>(P.corr_w, P.corr_samples, P.n_corr, P.p, P.L, P.corr_val);
  else
    k_corr_eval<true><<<blocks, 32 * kEvalWarps, eval_smem(), s>>>(P.corr_w, P.corr_samples, P.n_corr, P.p, P.L, P.corr_val);
  return cudaGetLastError();
}

cudaError_t launch_corr_fold(Plan& P, cudaStream_t s) {
  const int total = (P.L - 1) * P.n_corr;
  k_corr_fold<<<(total * kFoldLanes + 127) / 128, 128, 0, s>>>(P.dT_all, P.corr_samples, P.n_corr, P.p, P.L, P.corr_up);
  return cudaGetLastError();
}

cudaError_t setup_learn_spec(const Plan& P) {
  cudaError_t e = cudaFuncSetAttribute(k_corr_eval<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eval_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_corr_eval<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eval_smem());
  if (e != cudaSuccess) return e;
  switch (P.p) {                          // above 48 KB
    case 8: return cudaFuncSetAttribute(k_tg_inv<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)inv_smem<8>());
    default: return cudaSuccess;
  }
}

// Scratch of the spectral table gradient, shared by the levels (bytes):
// spectra of lam and M, offset spectra, offset lags.
void tg_bytes(const Plan& P, size_t& la, size_t& mh, size_t& gh, size_t& gl) {
  const size_t nodes = (size_t)1 << (3 * P.L), ch = (size_t)chunks_of(P.p, false), nm = 2 * (size_t)P.p - 1;
  la = ch * (4 * nodes + 1) * 128;
  mh = ch * (nodes + 1) * 128;
  gh = (size_t)kOff3 * 4 * ch * 128;
  gl = (size_t)kOff3 * 4 * nm * nm * nm * sizeof(float);
}

cudaError_t launch_table_grad_spec(Plan& P, int level, cudaStream_t s) {
  const int ch = chunks_of(P.p, false), nkp = ch * kLn;
  const size_t nodes = (size_t)1 << (3 * level);
  float2 *La = static_cast<float2*>(P.tg_la), *Mh = static_cast<float2*>(P.tg_mh), *Gh = static_cast<float2*>(P.tg_gh);
  float* Gl = static_cast<float*>(P.tg_gl);
  cudaError_t e = launch_spec_fwd(P, P.lam[level], La, 4 * nodes, s);
  if (e == cudaSuccess) e = launch_spec_fwd(P, P.M[level], Mh, nodes, s);
  if (e != cudaSuccess) return e;
  k_tg_mac<<<dim3(49, ch), kLn * kTgGroups, 0, s>>>(La, Mh, level, nkp, Gh);
  switch (P.p) {
    case 2: e = inv_p<2>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 3: e = inv_p<3>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 4: e = inv_p<4>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 5: e = inv_p<5>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 6: e = inv_p<6>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 7: e = inv_p<7>(Gh, nkp, P.spec_tw, Gl, s); break;
    case 8: e = inv_p<8>(Gh, nkp, P.spec_tw, Gl, s); break;
    default: e = cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  k_tg_gather<<<4 * P.num_sms, 256, 0, s>>>(Gl, P.p, level, P.dT[level]);
  return cudaGetLastError();
}

}  // namespace fmm
