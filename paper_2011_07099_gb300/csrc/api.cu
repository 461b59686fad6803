// The C-ABI of libfmm: plan lifecycle, solve orchestration and errors.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <initializer_list>
#include <new>
#include <set>
#include <tuple>
#include <vector>

#include <cuda.h>

#include "fmm_internal.cuh"
#include "mlp.cuh"

using fmm::Plan;

namespace {

thread_local int g_last_error = FMM_OK;

int set_err(int code) {
  g_last_error = code;
  return code;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

#define FMM_CUDA_TRY(expr)                  \
  do {                                      \
    cudaError_t _e = (expr);                \
    if (_e != cudaSuccess) {                \
      return set_err(FMM_ERR_CUDA);         \
    }                                       \
  } while (0)

// 1-D Lagrange basis on the gridlet points X_j = (j + 1/2)/p (node-size units)
// evaluated at the K cell-centred points y_k = (k + 1/2)/K: w[s][k] = l_s(y_k).
// This is the separable solution of the Sec. 2 Vandermonde system (the
// gridlet masses that keep every multipole Q_n, n_i < p).  Computed in double.
std::vector<double> lagrange_weights(int p, int K) {
  std::vector<double> w((size_t)p * K);
  for (int s = 0; s < p; ++s) {
    const double xs = (s + 0.5) / p;
    for (int k = 0; k < K; ++k) {
      const double y = (k + 0.5) / K;
      double v = 1.0;
      for (int j = 0; j < p; ++j) {
        if (j == s) continue;
        const double xj = (j + 0.5) / p;
        v *= (y - xj) / (xs - xj);
      }
      w[(size_t)s * K + k] = v;
    }
  }
  return w;
}

// Interaction-zone offsets o = T - S (node units, nearest periodic image) for
// the node whose position in its parent is c = cx | cy << 1 | cz << 2: the
// children of the parent's periodic neighbours minus the node's own periodic
// neighbours (Sec. 2, Fig. fmm).  Under periodic wrap every node with the same
// position in its parent has the translated list, so one list per child type.
std::vector<int8_t> interaction_offsets(int level, int c) {
  const int n = 1 << level, np = n >> 1;
  auto wrapn = [](int v, int m) { return ((v % m) + m) % m; };
  const int tx = c & 1, ty = (c >> 1) & 1, tz = (c >> 2) & 1;   // parent is (0,0,0)
  std::set<std::tuple<int, int, int>> kids, near;
  for (int a = -1; a <= 1; ++a)
    for (int b = -1; b <= 1; ++b)
      for (int d = -1; d <= 1; ++d) {
        const int qx = wrapn(a, np), qy = wrapn(b, np), qz = wrapn(d, np);
        for (int i = 0; i < 8; ++i)
          kids.insert(std::make_tuple(2 * qx + (i & 1), 2 * qy + ((i >> 1) & 1), 2 * qz + (i >> 2)));
        near.insert(std::make_tuple(wrapn(tx + a, n), wrapn(ty + b, n), wrapn(tz + d, n)));
      }
  std::vector<int8_t> out;
  for (const auto& k : kids) {
    if (near.count(k)) continue;
    int o[3] = {tx - std::get<0>(k), ty - std::get<1>(k), tz - std::get<2>(k)};
    for (int& v : o) {
      v = wrapn(v, n);
      if (v > n / 2) v -= n;          // nearest image; +n/2 kept (G_S1 is 1-periodic)
    }
    out.push_back((int8_t)o[0]);
    out.push_back((int8_t)o[1]);
    out.push_back((int8_t)o[2]);
  }
  return out;
}

// Offsets of the isolated problem's interaction zones at level 2 (Sec. 3's
// non-periodic reference, Sec. 2 zones without the wrap): the parent level 1
// has 2 nodes per dimension, all neighbours of each other, so a level-2
// node's zone is every in-box node that is not its neighbour; as offsets
// o = T - S, every o in [-3, 3]^3 with max |o_i| >= 2 (316), the in-box test
// being done by the kernels.  Levels >= 3 use the periodic lists: a periodic
// list restricted to in-box sources is the isolated list there.
std::vector<int8_t> isolated_level2_offsets() {
  std::vector<int8_t> out;
  for (int z = -3; z <= 3; ++z)
    for (int y = -3; y <= 3; ++y)
      for (int x = -3; x <= 3; ++x) {
        const int m = std::max(std::abs(x), std::max(std::abs(y), std::abs(z)));
        if (m < 2) continue;
        out.push_back((int8_t)x);
        out.push_back((int8_t)y);
        out.push_back((int8_t)z);
      }
  return out;
}

// Frees a set of buffers that set_alloc made: the first owns the memory.
void free_set(std::initializer_list<void**> parts) {
  cudaFree(**parts.begin());
  for (void** p : parts) *p = nullptr;
}

// Training buffers (alloc_train).
void free_train(Plan& P) {
  free_set({&P.tg_la, &P.tg_mh, &P.tg_gh, &P.tg_gl});
  for (float** b : {&P.train_out, &P.lam_cells, &P.dT_all, &P.grad_partials}) {
    cudaFree(*b);
    *b = nullptr;
  }
  for (int l = 0; l <= fmm::kMaxLevel; ++l) {
    cudaFree(P.lam[l]);
    P.lam[l] = P.dT[l] = nullptr;
  }
}

void free_near_spec(Plan& P) { free_set({&P.ns_K, &P.ns_M, &P.ns_P}); }

// A level's spectra: of the CUDA cores and, without them or alone, of the tensor cores.
void free_stc(Plan& P, int l) {
  free_set({&P.stc_W[l], &P.stc_B[l], &P.stc_scale[l], &P.stc_amax[l]});
  delete static_cast<CUtensorMap*>(P.stc_map[l]);
  P.stc_map[l] = nullptr;
}
void free_spec(Plan& P, int l) {
  free_stc(P, l);
  free_set({&P.spec_K[l], &P.spec_M[l], &P.spec_P[l]});
}

void free_plan(Plan* P) {
  if (!P) return;
  cudaFree(P->d_partials);
  cudaFree(P->m2l_part);
  cudaFree(P->d_mean);
  for (int l = 0; l <= fmm::kMaxLevel; ++l) {
    cudaFree(P->M[l]);
    cudaFree(P->F[l]);
    cudaFree(P->tab[l]);
    cudaFree(P->tab_lo[l]);
    cudaFree(P->F64[l]);
    cudaFree(P->M64[l]);
    cudaFree(P->offsets[l]);
    free_spec(*P, l);
  }
  cudaFree(P->spec_tw);
  cudaFree(P->near_tab);
  free_near_spec(*P);
  cudaFree(P->d_err);
  cudaFree(P->corr_w);
  cudaFree(P->corr_samples);
  cudaFree(P->corr_val);
  cudaFree(P->corr_up);
  free_train(*P);
  cudaFree(P->grid);
  cudaFree(P->gmesh);
  fmm::free_fft(*P);
  for (int l = 0; l <= fmm::kMaxLevel; ++l) {
    cudaFree(P->tab_bf[l]);
    cudaFree(P->Mbf_hi[l]);
    cudaFree(P->Apre[l]);
    delete static_cast<CUtensorMap*>(P->tmapB[l]);
  }
  cudaFree(P->es_scratch);
  cudaFree(P->w_p2m);
  cudaFree(P->w_m2m);
  cudaFree(P->stage_in);
  cudaFree(P->stage_out);
  for (auto& e : P->ev)
    if (e) cudaEventDestroy(e);
  for (auto& e : P->fev)
    if (e) cudaEventDestroy(e);
  for (auto& a : P->aux)
    if (a) cudaStreamDestroy(a);
  delete P;
}

// Device memory.  An allocation that fails is the caller's to report: CUDA's
// record of it is cleared, so that no later launch reads it as its own error.
bool dev_alloc_bytes(void** ptr, size_t bytes) {
  if (cudaMalloc(ptr, bytes) == cudaSuccess) return true;
  (void)cudaGetLastError();
  *ptr = nullptr;
  return false;
}
template <typename T>
bool dev_alloc(T** ptr, size_t count) {
  return dev_alloc_bytes(reinterpret_cast<void**>(ptr), sizeof(T) * count);
}
// The same for a plan in use, whose allocation FMM_FAULT_ALLOC names asks for
// more than any device holds.
template <typename T>
bool plan_alloc(Plan& P, T** ptr, size_t count) {
  const bool fail = P.fail_alloc >= 0 && P.fail_alloc-- == 0;
  return dev_alloc(ptr, fail ? ((size_t)1 << 60) / sizeof(T) : count);
}
bool plan_alloc(Plan& P, void** ptr, size_t bytes) { return plan_alloc(P, reinterpret_cast<char**>(ptr), bytes); }

// A set of buffers in one allocation (free_set), all of them or none: an
// allocation takes 30 to 60 us and a plan has up to 11 sets.
struct Part {
  void** at;
  size_t bytes;
};
bool set_alloc(Plan& P, std::initializer_list<Part> parts) {
  auto rounded = [](size_t n) { return (n + 255) / 256 * 256; };
  size_t total = 0;
  for (const Part& p : parts) total += rounded(p.bytes);
  char* base = nullptr;
  if (!plan_alloc(P, &base, total)) return false;
  for (const Part& p : parts) {
    *p.at = base;
    base += rounded(p.bytes);
  }
  return true;
}

// Spectra are optional: the dense kernels need ~20 times less memory.  A plan
// holds at most what its caller allows (fmm_plan_set_spectra_limit) or, by
// default, kSpecMaxBytes and no more than the memory that stays free beside
// them, counted over all its sets of buffers: the M2L levels (m2l_spec.cu,
// m2l_spec_tc.cu), the near zone (near_spec.cu), the training step
// (learn_spec.cu).  A set that has no room, or whose allocation fails, is left
// out and its dense kernels run.
constexpr size_t kSpecMaxBytes = (size_t)96 << 30;

size_t spectra_bytes(const Plan& P) {
  size_t sum = 0, a, b, c, d;
  for (int l = 2; l <= P.L; ++l) {
    if (P.spec_K[l]) sum += fmm::spec_kernel_bytes(P, l) + fmm::spec_source_bytes(P, l) + fmm::spec_target_bytes(P, l);
    if (P.stc_map[l]) {
      fmm::stc_bytes(P, l, a, b, c);
      sum += a + b + c;
    }
  }
  if (P.ns_K) {
    fmm::near_spec_bytes(P, a, b, c);
    sum += a + b + c;
  }
  if (P.tg_la) {
    fmm::tg_bytes(P, a, b, c, d);
    sum += a + b + c + d;
  }
  return sum;
}

// The most bytes of spectra the plan may hold now; held and free memory change
// by the same amount while its sets are made, so one look serves them all.
size_t spectra_room(const Plan& P) {
  if (P.spec_limit != SIZE_MAX) return P.spec_limit;
  size_t free_b = 0, total = 0;
  if (cudaMemGetInfo(&free_b, &total) != cudaSuccess) {
    (void)cudaGetLastError();
    return kSpecMaxBytes;
  }
  return std::min(kSpecMaxBytes, (free_b + spectra_bytes(P)) / 2);
}
bool spectra_fit(const Plan& P, size_t room, size_t bytes) { return spectra_bytes(P) + bytes <= room; }

// (cos, sin) of 2 pi j / (2 points - 1) as (hi, lo) FP32 pairs, for gridlets
// (points = order) and for leaves (points = S).
int make_twiddles(Plan& P) {
  std::vector<float4> tw;
  for (int points : {P.p, P.S}) {
    const int nm = 2 * points - 1;
    for (int j = 0; j < nm; ++j) {
      const double a = 2.0 * 3.14159265358979323846 * j / nm, c = std::cos(a), s = std::sin(a);
      tw.push_back(make_float4((float)c, (float)(c - (double)(float)c), (float)s, (float)(s - (double)(float)s)));
    }
  }
  if (!dev_alloc(&P.spec_tw, tw.size())) return FMM_ERR_ALLOC;
  P.ns_tw = P.spec_tw + 2 * P.p - 1;
  return cudaMemcpy(P.spec_tw, tw.data(), tw.size() * sizeof(float4), cudaMemcpyHostToDevice) == cudaSuccess
             ? FMM_OK
             : FMM_ERR_CUDA;
}

// Buffers of the near zone's spectral products (near_spec.cu) for the leaf
// sizes it is built for.
int alloc_near_spec(Plan& P, size_t room) {
  if (P.ns_K || !fmm::near_spec_shape(P)) return FMM_OK;
  size_t nK, nM, nP;
  fmm::near_spec_bytes(P, nK, nM, nP);
  if (!spectra_fit(P, room, nK + nM + nP) || !set_alloc(P, {{&P.ns_K, nK}, {&P.ns_M, nM}, {&P.ns_P, nP}}))
    return FMM_OK;
  return fmm::launch_clear_spectra(P.ns_K, nK, P.ns_M, nM, (size_t)1 << (3 * P.L), 0) == cudaSuccess ? FMM_OK
                                                                                                     : FMM_ERR_CUDA;
}

// Buffers of the spectral M2L for every level of orders >= 2, the coarse first.
int alloc_spec(Plan& P, size_t room) {
  if (P.p < 2) return FMM_OK;
  for (int l = 2; l <= P.L; ++l) {
    const size_t nk = fmm::spec_kernel_bytes(P, l), ns = fmm::spec_source_bytes(P, l),
                 nt = fmm::spec_target_bytes(P, l);
    if (!spectra_fit(P, room, nk + ns + nt) ||
        !set_alloc(P, {{&P.spec_K[l], nk}, {&P.spec_M[l], ns}, {&P.spec_P[l], nt}}))
      continue;
    if (fmm::launch_clear_spectra(P.spec_K[l], nk, P.spec_M[l], ns, (size_t)1 << (3 * l), 0) != cudaSuccess)
      return FMM_ERR_CUDA;
  }
  return FMM_OK;
}

// Scratch for the offset-range partials of the dense wide levels, which
// follows the length of their interaction lists; the old one is given up only
// once there is a new one.
int alloc_m2l_part(Plan& P) {
  size_t part = 0;
  const size_t p3 = (size_t)P.p * P.p * P.p;
  for (int l = 2; l <= P.L; ++l) {
    if (!fmm::wide_level(P, l) || P.spec_K[l]) continue;
    const size_t need = 2 * (size_t)fmm::m2l_fp32_splits(P, l) * ((size_t)1 << (3 * l)) * 4 * p3;
    if (need > part) part = need;
  }
  float* fresh = nullptr;
  if (part && !plan_alloc(P, &fresh, part)) return FMM_ERR_ALLOC;
  cudaFree(P.m2l_part);
  P.m2l_part = fresh;
  return FMM_OK;
}

// How the M2L of level l runs in the plan's present settings (FMM_FORM_*).
int m2l_form(const Plan& P, int l) {
  if (fmm::fft_level(P, l)) return FMM_FORM_FFT;
  if (P.prec != FMM_PREC_FP32 && P.tc_ready) {
    if (fmm::spec_tc_level(P, l)) return FMM_FORM_SPECTRAL_TC;
    if (fmm::tc_level(P, l)) return FMM_FORM_DENSE_TC;
  }
  return P.spec_K[l] ? FMM_FORM_SPECTRAL : FMM_FORM_DENSE;
}

// Re-tabulate every table form from G_S1 plus the plan's corrections (MLP,
// grid), synchronously.  Returns an FMM_* code.
// near = false: a correction of the M2L tables only (the near zone keeps its table).
int retabulate(Plan& P, bool near = true) {
  if (fmm::launch_tables(P, near, 0) != cudaSuccess) return FMM_ERR_CUDA;
  if (P.fft) {   // the FFT form keeps the tables' spectra: rebuild them
    fmm::free_fft(P);
    if (P.m2l_fft) {
      if (cudaDeviceSynchronize() != cudaSuccess) return FMM_ERR_CUDA;
      const int rc = fmm::prepare_fft(P);
      if (rc != FMM_OK) return rc;
    }
  }
  if (near && P.ns_K && fmm::launch_near_spec_kernels(P, 0) != cudaSuccess) return FMM_ERR_CUDA;
  for (int l = 2; l <= P.L; ++l) {
    if (P.spec_K[l] && fmm::launch_spec_kernels(P, l, 0) != cudaSuccess) return FMM_ERR_CUDA;
    if (P.stc_map[l] && fmm::launch_stc_weights(P, l, 0) != cudaSuccess) return FMM_ERR_CUDA;
  }
  if (P.tc_ready) {
    for (int l = fmm::kTcMinLevel; l <= P.L; ++l) {
      if (!P.tmapB[l]) continue;
      if ((!fmm::tc_wide(P, l) && fmm::launch_tab_bf16(P, l, 0) != cudaSuccess) ||
          fmm::launch_build_a(P, l, 0) != cudaSuccess)
        return FMM_ERR_CUDA;
    }
  }
  return cudaDeviceSynchronize() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

// Training buffers, all of them or none (FMM_* code); the scratch of the
// spectral table gradient where it has room.
int alloc_train(Plan& P) {
  const size_t n3 = (size_t)P.N * P.N * P.N, p3 = (size_t)P.p * P.p * P.p, E = 8 * P.p - 1;
  bool ok = plan_alloc(P, &P.train_out, 4 * n3) && plan_alloc(P, &P.lam_cells, 4 * n3) &&
            plan_alloc(P, &P.dT_all, (size_t)(P.L - 1) * E * E * E * 4) &&
            plan_alloc(P, &P.grad_partials, (size_t)fmm::mlp_backward_blocks(P) * fmm::mlp::kParams);
  for (int l = 2; l <= P.L && ok; ++l) ok = plan_alloc(P, &P.lam[l], ((size_t)1 << (3 * l)) * 4 * p3);
  if (!ok) {
    free_train(P);
    return FMM_ERR_ALLOC;
  }
  size_t la, mh, gh, gl;
  fmm::tg_bytes(P, la, mh, gh, gl);
  if (P.p >= 2 && spectra_fit(P, spectra_room(P), la + mh + gh + gl))   // else the direct sums
    (void)set_alloc(P, {{&P.tg_la, la}, {&P.tg_mh, mh}, {&P.tg_gh, gh}, {&P.tg_gl, gl}});
  for (int l = 2; l <= P.L; ++l) P.dT[l] = P.dT_all + (size_t)(l - 2) * E * E * E * 4;
  return FMM_OK;
}

// One forward solve, cell residual and adjoint sweep down to the table
// gradients P.dT of every level; the loss is added to `loss`.  Returns an
// FMM_* code.
int table_gradient(Plan& P, const float* density, const float* target_phi, const float* target_acc, float w_phi,
                   float w_g, float* loss, void* stream) {
  const size_t n3 = (size_t)P.N * P.N * P.N;
  if (!P.train_out) {
    const int rc = alloc_train(P);
    if (rc != FMM_OK) return rc;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int rc = fmm_solve(reinterpret_cast<fmm_plan*>(&P), density, P.train_out, P.train_out + n3, stream);
  if (rc != FMM_OK) return rc;
  if (fmm::launch_residual(P.train_out, P.train_out + n3, target_phi, target_acc, n3, w_phi, w_g, P.lam_cells,
                           reinterpret_cast<double*>(P.grad_partials), loss, P.num_sms, s) != cudaSuccess ||
      fmm::launch_adjoint_and_table_grad(P, P.lam_cells, s) != cudaSuccess)
    return FMM_ERR_CUDA;
  return FMM_OK;
}

}  // namespace

int fmm::set_last_error(int code) { return set_err(code); }

extern "C" {

int fmm_last_error(void) { return g_last_error; }

const char* fmm_error_string(int code) {
  switch (code) {
    case FMM_OK: return "ok";
    case FMM_ERR_ARG: return "invalid argument";
    case FMM_ERR_CUDA: return "CUDA runtime error";
    case FMM_ERR_TIMEOUT: return "bounded device wait timed out";
    case FMM_ERR_INTERNAL: return "internal consistency check failed";
    case FMM_ERR_ALLOC: return "allocation failed";
    case FMM_ERR_UNSUPPORTED: return "unsupported by this build";
    default: return "unknown error code";
  }
}

fmm_plan* fmm_plan_create(int N, int L, int order) {
  if (L < 2 || L > fmm::kMaxLevel || order < 1 || order > fmm::kMaxOrder || N <= 0) {
    set_err(FMM_ERR_ARG);
    return nullptr;
  }
  const int n = 1 << L;
  if (N % n != 0) {
    set_err(FMM_ERR_ARG);
    return nullptr;
  }
  const int S = N / n;
  if (S != 1 && S != 2 && S != 3 && S != 4 && S != 6 && S != 8 && S != 16) {
    set_err(FMM_ERR_ARG);
    return nullptr;
  }
  Plan* P = new (std::nothrow) Plan();
  if (!P) {
    set_err(FMM_ERR_ALLOC);
    return nullptr;
  }
  P->N = N;
  P->L = L;
  P->p = order;
  P->S = S;
  if (cudaGetDevice(&P->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device) != cudaSuccess) {
    delete P;
    set_err(FMM_ERR_CUDA);
    return nullptr;
  }
  const int p = order, p3 = p * p * p;
  bool ok = true;
  for (auto& a : P->aux) ok = ok && cudaStreamCreateWithFlags(&a, cudaStreamNonBlocking) == cudaSuccess;
  for (auto& e : P->fev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    free_plan(P);
    set_err(FMM_ERR_CUDA);
    return nullptr;
  }
  P->n_partials = 4 * P->num_sms;
  ok = ok && dev_alloc(&P->d_partials, P->n_partials) && dev_alloc(&P->d_mean, 1) && dev_alloc(&P->d_err, 1) &&
       cudaMemset(P->d_err, 0, sizeof(int)) == cudaSuccess;
  for (int l = 2; l <= L && ok; ++l) {
    const size_t nodes = (size_t)1 << (3 * l);
    const size_t E = 8 * p - 1;
    ok = dev_alloc(&P->M[l], nodes * p3) && dev_alloc(&P->F[l], nodes * 4 * p3) &&
         dev_alloc(&P->tab[l], E * E * E);
    ok = ok && dev_alloc(&P->tab_lo[l], E * E * E);   // low halves: v - fl32(v)
    // FP64 gridlet masses at every level at high order (the leaf copy feeds M2M:
    // the coarse far-field sums cancel ~1000-fold there, so FP32 rounding of
    // the leaf masses alone would cost ~1e-6)
    if (ok && p >= fmm::kWideOrder) ok = dev_alloc(&P->M64[l], nodes * p3);
  }
  ok = ok && dev_alloc(&P->near_tab, (size_t)8 * S * S * S) && dev_alloc(&P->w_p2m, (size_t)p * S) &&
       dev_alloc(&P->w_m2m, (size_t)p * 2 * p);
  if (!ok) {
    free_plan(P);
    set_err(FMM_ERR_ALLOC);
    return nullptr;
  }
  // host-side constants: Lagrange weights and interaction lists
  // Lagrange weights in FP64 on the host, stored as (hi, lo) FP32 pairs
  std::vector<double> wp = lagrange_weights(p, S), wm = lagrange_weights(p, 2 * p);
  auto split = [](const std::vector<double>& v) {
    std::vector<float2> o(v.size());
    for (size_t i = 0; i < v.size(); ++i) {
      const float hi = (float)v[i];
      o[i] = make_float2(hi, (float)(v[i] - (double)hi));
    }
    return o;
  };
  std::vector<float2> wp2 = split(wp), wm2 = split(wm);
  bool cok = cudaMemcpy(P->w_p2m, wp2.data(), wp2.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(P->w_m2m, wm2.data(), wm2.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess;
  for (int l = 2; l <= L && cok; ++l) {
    std::vector<int8_t> all;
    int count = -1;
    for (int c = 0; c < 8; ++c) {
      std::vector<int8_t> o = interaction_offsets(l, c);
      const int k = (int)o.size() / 3;
      if (count >= 0 && k != count) cok = false;
      count = k;
      all.insert(all.end(), o.begin(), o.end());
    }
    P->n_off[l] = count;
    cok = cok && (l == 2 ? count == 37 : count == 189);
    cok = cok && dev_alloc(&P->offsets[l], all.size()) &&
          cudaMemcpy(P->offsets[l], all.data(), all.size(), cudaMemcpyHostToDevice) == cudaSuccess;
  }
  if (!cok) {
    free_plan(P);
    set_err(FMM_ERR_INTERNAL);
    return nullptr;
  }
  {
    // scratch for the offset-range partials of the coarse FP32 M2L levels
    bool fok = true;
    for (int l = 2; l <= L && fok; ++l)
      if (fmm::wide_level(*P, l)) fok = dev_alloc(&P->F64[l], ((size_t)1 << (3 * l)) * 4 * p3);
    int rc = fok ? make_twiddles(*P) : FMM_ERR_ALLOC;
    const size_t room = spectra_room(*P);
    if (rc == FMM_OK) rc = alloc_spec(*P, room);
    if (rc == FMM_OK) rc = alloc_near_spec(*P, room);
    if (rc != FMM_OK || alloc_m2l_part(*P) != FMM_OK) {
      free_plan(P);
      set_err(rc != FMM_OK ? rc : FMM_ERR_ALLOC);
      return nullptr;
    }
  }
  if (fmm::setup_upward(*P) != cudaSuccess || fmm::setup_m2l_fp32(*P) != cudaSuccess ||
      fmm::setup_m2l_tc(*P) != cudaSuccess || fmm::setup_learn() != cudaSuccess ||
      fmm::setup_learn_spec(*P) != cudaSuccess ||
      fmm::setup_downward(*P) != cudaSuccess || fmm::setup_p2p(*P) != cudaSuccess ||
      fmm::setup_m2l_spec(*P) != cudaSuccess || fmm::setup_spec_tc(*P) != cudaSuccess || retabulate(*P) != FMM_OK) {
    free_plan(P);
    set_err(FMM_ERR_CUDA);
    return nullptr;
  }
  set_err(FMM_OK);
  return reinterpret_cast<fmm_plan*>(P);
}

void fmm_plan_destroy(fmm_plan* plan) {
  if (!plan) return;
  cudaDeviceSynchronize();
  free_plan(reinterpret_cast<Plan*>(plan));
}

int fmm_plan_get_shape(const fmm_plan* plan, int* N, int* L, int* order, int* S) {
  if (!plan) return set_err(FMM_ERR_ARG);
  const Plan* P = reinterpret_cast<const Plan*>(plan);
  if (N) *N = P->N;
  if (L) *L = P->L;
  if (order) *order = P->p;
  if (S) *S = P->S;
  return set_err(FMM_OK);
}

namespace {
// A level of the spectral tensor-core form: split weights and sources, their
// scales and the tensor map, all of them or none (FMM_* code).
int prepare_stc(Plan& P, int l, size_t room) {
  size_t nW, nB, nS;
  fmm::stc_bytes(P, l, nW, nB, nS);
  int rc = FMM_ERR_ALLOC;
  if (spectra_fit(P, room, nW + nB + nS) &&
      set_alloc(P, {{&P.stc_W[l], nW}, {&P.stc_B[l], nB}, {&P.stc_scale[l], nS}, {&P.stc_amax[l], sizeof(float)}})) {
    // the halo of the isolated problem stays zero (fmm_plan_set_boundary clears it too)
    rc = (!P.iso || cudaMemset(P.stc_B[l], 0, nB) == cudaSuccess) && fmm::launch_stc_weights(P, l, 0) == cudaSuccess
             ? fmm::make_stc_map(P, l)
             : FMM_ERR_CUDA;
  }
  if (rc != FMM_OK) free_stc(P, l);
  return rc;
}

// Tensor-core M2L buffers of every level from the first tensor-core level down
// to the leaves (levels that already have them are kept): the spectral form's
// or, where that has no room or does not run, the dense contraction's split
// tables, split multipoles and translation tiles.  A level counts as prepared
// once it has its tensor map, which is made last.  Tabulated once, synchronously.
int prepare_tc(Plan& P) {
  const size_t E = 8 * P.p - 1, room = spectra_room(P);
  bool made = false;
  for (int l = fmm::tc_first_level(P); l <= P.L; ++l) {
    if (fmm::spec_tc_level(P, l)) {
      if (P.stc_map[l]) continue;
      const int rc = prepare_stc(P, l, room);
      if (rc == FMM_OK) {
        made = true;
        continue;
      }
      if (rc != FMM_ERR_ALLOC) return rc;
      P.stc_off[l] = true;                  // no room: spec_tc_level is false from here on
    }
    if (P.tmapB[l]) continue;
    const bool wide = fmm::tc_wide(P, l);   // wide modes: tiles from tab + tab_lo, no BF16 table
    if ((!wide && !P.tab_bf[l] && !plan_alloc(P, &P.tab_bf[l], E * E * E)) ||
        (!P.Mbf_hi[l] && !plan_alloc(P, &P.Mbf_hi[l], fmm::tc_bsplit_bytes(P.p, l, fmm::tc_splits(P, l)))) ||
        (!P.Apre[l] && !plan_alloc(P, &P.Apre[l], fmm::tc_apre_bytes(P.p, fmm::tc_splits(P, l)))))
      return FMM_ERR_ALLOC;
    if ((!wide && fmm::launch_tab_bf16(P, l, 0) != cudaSuccess) || fmm::launch_build_a(P, l, 0) != cudaSuccess)
      return FMM_ERR_CUDA;
    const int rc = fmm::make_tc_map(P, l);
    if (rc != FMM_OK) return rc;
    made = true;
  }
  if (made && cudaDeviceSynchronize() != cudaSuccess) return FMM_ERR_CUDA;
  P.tc_ready = 1;
  return FMM_OK;
}
}  // namespace

int fmm_plan_set_precision(fmm_plan* plan, int mode) {
  if (!plan) return set_err(FMM_ERR_ARG);
  if (mode != FMM_PREC_FP32 && mode != FMM_PREC_BF16 && mode != FMM_PREC_BF16X3) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (mode != FMM_PREC_FP32 && P.p >= 2) {
    const int rc = prepare_tc(P);
    if (rc != FMM_OK) return set_err(rc);
  }
  P.prec = mode;
  return set_err(FMM_OK);
}

int fmm_plan_set_spectra_limit(fmm_plan* plan, size_t bytes) {
  if (!plan) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  FMM_CUDA_TRY(cudaDeviceSynchronize());
  P.spec_limit = bytes;
  // every set again within the limit; the training step's on its next use.
  // Until all is made the plan solves nothing (P.unmade).
  for (int l = 2; l <= P.L; ++l) {
    free_spec(P, l);
    P.stc_off[l] = false;
  }
  free_near_spec(P);
  free_train(P);
  const size_t room = spectra_room(P);
  int rc = alloc_spec(P, room);
  if (rc == FMM_OK) rc = alloc_near_spec(P, P.near_fft ? SIZE_MAX : room);
  if (rc == FMM_OK && P.near_fft && !P.ns_K) rc = FMM_ERR_ALLOC;
  if (rc == FMM_OK) rc = alloc_m2l_part(P);
  if (rc == FMM_OK && P.tc_ready) rc = prepare_tc(P);
  if (rc == FMM_OK) rc = retabulate(P);
  P.unmade = rc;
  return set_err(rc);
}

int fmm_plan_get_forms(const fmm_plan* plan, int* forms, int n, size_t* spectra) {
  if (!plan || n < 0 || (n > 0 && !forms)) return set_err(FMM_ERR_ARG);
  const Plan& P = *reinterpret_cast<const Plan*>(plan);
  for (int l = 0; l < n; ++l)
    forms[l] = l == 0 ? (P.ns_K ? FMM_FORM_SPECTRAL : FMM_FORM_DENSE)
                      : (l >= 2 && l <= P.L ? m2l_form(P, l) : FMM_FORM_NONE);
  if (spectra) *spectra = spectra_bytes(P);
  return set_err(FMM_OK);
}

int fmm_plan_set_boundary(fmm_plan* plan, int boundary) {
  if (!plan || (boundary != FMM_BOUNDARY_PERIODIC && boundary != FMM_BOUNDARY_ISOLATED)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const int iso = boundary == FMM_BOUNDARY_ISOLATED ? 1 : 0;
  if (iso == P.iso) return set_err(FMM_OK);
  FMM_CUDA_TRY(cudaDeviceSynchronize());
  // level-2 interaction lists: 37 periodic nodes, or the 316 in-box offsets
  std::vector<int8_t> all;
  int count = 0;
  for (int c = 0; c < 8; ++c) {
    std::vector<int8_t> o = iso ? isolated_level2_offsets() : interaction_offsets(2, c);
    count = (int)o.size() / 3;
    all.insert(all.end(), o.begin(), o.end());
  }
  int8_t* offs = nullptr;
  if (!plan_alloc(P, &offs, all.size())) return set_err(FMM_ERR_ALLOC);
  const int was = P.n_off[2];
  P.n_off[2] = count;
  const int rc = cudaMemcpy(offs, all.data(), all.size(), cudaMemcpyHostToDevice) == cudaSuccess ? alloc_m2l_part(P)
                                                                                                  : FMM_ERR_CUDA;
  if (rc != FMM_OK) {                   // the plan keeps its boundary
    P.n_off[2] = was;
    cudaFree(offs);
    return set_err(rc);
  }
  cudaFree(P.offsets[2]);
  P.offsets[2] = offs;
  P.iso = iso;
  for (int l = 2; l <= P.L; ++l) {      // the tensor cores' sources: a periodic halo, or zeros
    size_t nW, nB, nS;
    fmm::stc_bytes(P, l, nW, nB, nS);
    if (P.stc_B[l]) FMM_CUDA_TRY(cudaMemset(P.stc_B[l], 0, nB));
  }
  return set_err(retabulate(P));
}

int fmm_plan_set_green(fmm_plan* plan, int kind, const double* a, int na) {
  if (!plan || (kind != FMM_GREEN_S1 && kind != FMM_GREEN_S && kind != FMM_GREEN_X)) return set_err(FMM_ERR_ARG);
  if (kind == FMM_GREEN_S && (na < 1 || na > fmm::green::kMaxAnsatz || !a)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  fmm::green::Spec g;
  g.kind = kind == FMM_GREEN_S ? 1 : (kind == FMM_GREEN_X ? 3 : 0);
  g.na = kind == FMM_GREEN_S ? na : 0;
  for (int k = 0; k < g.na; ++k) g.a[k] = a[k];
  P.gspec = g;
  return set_err(retabulate(P));
}

int fmm_plan_set_green_mesh(fmm_plan* plan, const double* mesh, size_t n) {
  if (!plan || !mesh) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const size_t n3 = (size_t)P.N * P.N * P.N;
  // every gridlet point of every level must sit on a mesh cell centre
  if (n != 4 * n3 || P.S % P.p != 0) return set_err(FMM_ERR_ARG);
  if (!P.gmesh && !dev_alloc(&P.gmesh, 4 * n3)) return set_err(FMM_ERR_ALLOC);
  FMM_CUDA_TRY(cudaMemcpy(P.gmesh, mesh, sizeof(double) * 4 * n3, cudaMemcpyDefault));
  fmm::green::Spec g;
  g.kind = 4;
  P.gspec = g;
  return set_err(retabulate(P));
}

int fmm_plan_set_m2l_algorithm(fmm_plan* plan, int algorithm) {
  if (!plan || (algorithm != FMM_M2L_DENSE && algorithm != FMM_M2L_FFT)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  P.m2l_fft = algorithm == FMM_M2L_FFT ? 1 : 0;
  if (P.m2l_fft) {
    const int rc = fmm::prepare_fft(P);
    if (rc != FMM_OK) {
      fmm::free_fft(P);
      P.m2l_fft = 0;
      return set_err(rc);
    }
  }
  return set_err(FMM_OK);
}

int fmm_plan_set_near_algorithm(fmm_plan* plan, int algorithm) {
  if (!plan || (algorithm != FMM_NEAR_DIRECT && algorithm != FMM_NEAR_FFT)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (algorithm == FMM_NEAR_DIRECT) {
    if (cudaDeviceSynchronize() != cudaSuccess) return set_err(FMM_ERR_CUDA);
    P.near_fft = 0;
    if (P.spec_limit != SIZE_MAX && spectra_bytes(P) > P.spec_limit) free_near_spec(P);
    return set_err(FMM_OK);
  }
  if (P.S != 8) return set_err(FMM_ERR_UNSUPPORTED);
  if (!P.ns_K) {   // over the default limit at plan creation: the caller asks for it
    const int rc = alloc_near_spec(P, SIZE_MAX);
    if (rc != FMM_OK || !P.ns_K) return set_err(rc != FMM_OK ? rc : FMM_ERR_ALLOC);
    FMM_CUDA_TRY(fmm::launch_near_spec_kernels(P, 0));
  }
  P.near_fft = 1;
  return set_err(cudaDeviceSynchronize() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA);
}

int fmm_plan_set_timeout_ms(fmm_plan* plan, int ms) {
  if (!plan || ms < 1 || ms > 600000) return set_err(FMM_ERR_ARG);
  reinterpret_cast<Plan*>(plan)->wait_ns = (uint64_t)ms * 1000000ull;
  return set_err(FMM_OK);
}

int fmm_plan_inject_fault(fmm_plan* plan, int kind) {
  const bool alloc = kind >= FMM_FAULT_ALLOC(0) && kind <= FMM_FAULT_ALLOC(255);
  if (!plan || (kind != FMM_FAULT_NONE && kind != FMM_FAULT_TC_STALL && !alloc)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  P.inject_stall = kind == FMM_FAULT_TC_STALL ? 1 : 0;
  P.fail_alloc = alloc ? kind - FMM_FAULT_ALLOC(0) : -1;
  return set_err(FMM_OK);
}

int fmm_plan_set_m2l_group(fmm_plan* plan, int offsets_per_partial) {
  if (!plan || offsets_per_partial < 1 || offsets_per_partial > fmm::kMaxOffsets) return set_err(FMM_ERR_ARG);
  reinterpret_cast<Plan*>(plan)->tc_group = offsets_per_partial;
  return set_err(FMM_OK);
}

int fmm_plan_set_tc_min_level(fmm_plan* plan, int level) {
  if (!plan || level < fmm::kTcMinLevel || level > fmm::kMaxLevel + 1) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const int was_level = P.tc_min_level, was_set = P.tc_min_set;
  P.tc_min_level = level;
  P.tc_min_set = 1;
  if (P.tc_ready) {   // a lower first level needs its tiles now
    const int rc = prepare_tc(P);
    if (rc != FMM_OK) {   // a level without them must not run
      P.tc_min_level = was_level;
      P.tc_min_set = was_set;
      return set_err(rc);
    }
  }
  return set_err(FMM_OK);
}

int fmm_plan_set_tc_tile(fmm_plan* plan, int level, int targets) {
  if (!plan || (targets != 128 && targets != 256)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (level < fmm::kTcMinLevel || level > P.L) return set_err(FMM_ERR_ARG);
  P.tc_tile[level] = targets == 128 ? 128 : 0;
  if (P.tmapB[level]) {     // the tensor loads' box follows the tile
    FMM_CUDA_TRY(cudaDeviceSynchronize());
    const int rc = fmm::make_tc_map(P, level);
    if (rc != FMM_OK) return set_err(rc);
  }
  return set_err(FMM_OK);
}

int fmm_plan_autotune_tiles(fmm_plan* plan, const float* density, int* tiles, int n, void* stream) {
  if (!plan || !density || !aligned16(density) || (n > 0 && !tiles) || n < 0) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const bool tc = P.prec != FMM_PREC_FP32 && P.tc_ready;
  const size_t n3 = (size_t)P.N * P.N * P.N;
  // levels whose kernel has a tile: the dense contraction's, but for bf16x6
  auto tiled = [&](int l) { return m2l_form(P, l) == FMM_FORM_DENSE_TC && !fmm::tc_wide(P, l); };
  bool any = false;
  for (int l = 2; l <= P.L; ++l) any = any || tiled(l);
  if (any) {
    float* out = nullptr;
    if (!dev_alloc(&out, 4 * n3)) return set_err(FMM_ERR_ALLOC);
    const int was_timing = P.timing;
    int rc = fmm_plan_set_timing(plan, 1);
    float best[fmm::kMaxLevel + 1] = {};
    int pick[fmm::kMaxLevel + 1] = {};
    for (int c = 0; c < 2 && rc == FMM_OK; ++c) {
      const int t = c == 0 ? 256 : 128;
      for (int l = fmm::tc_first_level(P); l <= P.L && rc == FMM_OK; ++l)
        if (tiled(l)) rc = fmm_plan_set_tc_tile(plan, l, t);
      float ms[FMM_TIME_SLOTS];
      float lev[fmm::kMaxLevel + 1];
      for (int l = 0; l <= fmm::kMaxLevel; ++l) lev[l] = 1e30f;
      for (int r = 0; r < 3 && rc == FMM_OK; ++r) {      // one warm-up, then the faster of two
        rc = fmm_solve(plan, density, out, out + n3, stream);
        if (rc == FMM_OK) rc = fmm_plan_stage_times(plan, ms, FMM_TIME_SLOTS);
        for (int l = 2; l <= P.L && r > 0 && rc == FMM_OK; ++l)
          lev[l] = ms[FMM_TIME_M2L_LEVEL0 + l] < lev[l] ? ms[FMM_TIME_M2L_LEVEL0 + l] : lev[l];
      }
      for (int l = 2; l <= P.L && rc == FMM_OK; ++l)
        if (c == 0 || lev[l] < best[l]) {
          best[l] = lev[l];
          pick[l] = t;
        }
    }
    for (int l = fmm::tc_first_level(P); l <= P.L && rc == FMM_OK; ++l)
      if (tiled(l)) rc = fmm_plan_set_tc_tile(plan, l, pick[l]);
    fmm_plan_set_timing(plan, was_timing);
    cudaFree(out);
    if (rc != FMM_OK) return set_err(rc);
  }
  for (int l = 0; l < n; ++l)
    tiles[l] = (tc && l <= P.L && l >= fmm::tc_first_level(P)) ? fmm::tc_targets(P, l) : 0;
  return set_err(FMM_OK);
}

int fmm_plan_set_correction_inference(fmm_plan* plan, int mode) {
  if (!plan || (mode != FMM_INFER_BF16 && mode != FMM_INFER_FP32)) return set_err(FMM_ERR_ARG);
  reinterpret_cast<Plan*>(plan)->corr_fp32 = mode == FMM_INFER_FP32 ? 1 : 0;
  return set_err(FMM_OK);
}

int fmm_plan_set_correction(fmm_plan* plan, const float* weights, size_t n) {
  if (!plan) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (weights) {
    if (n != (size_t)fmm::mlp::kParams) return set_err(FMM_ERR_ARG);
    if (!P.corr_w) {
      const std::vector<uint32_t> samples = fmm::corr_samples(P.p);
      if ((!P.corr_samples && !dev_alloc(&P.corr_samples, samples.size())) ||
          (!P.corr_val && !dev_alloc(&P.corr_val, fmm::corr_values(P))) ||
          (!P.corr_up && !dev_alloc(&P.corr_up, (size_t)(P.L - 1) * samples.size())))
        return set_err(FMM_ERR_ALLOC);
      FMM_CUDA_TRY(cudaMemcpy(P.corr_samples, samples.data(), samples.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
      P.n_corr = (int)samples.size();
      if (!dev_alloc(&P.corr_w, (size_t)fmm::mlp::kParams)) return set_err(FMM_ERR_ALLOC);
    }
    FMM_CUDA_TRY(cudaMemcpy(P.corr_w, weights, n * sizeof(float), cudaMemcpyDefault));
    P.has_corr = 1;
  } else {
    P.has_corr = 0;
  }
  return set_err(retabulate(P, false));
}

int fmm_correction_grad(fmm_plan* plan, const float* density, const float* target_phi, const float* target_acc,
                        float w_phi, float w_g, float* grad, float* loss, void* stream) {
  if (!plan || !density || !target_phi || !target_acc || !grad || !loss) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (!P.has_corr) return set_err(FMM_ERR_ARG);
  const int rc = table_gradient(P, density, target_phi, target_acc, w_phi, w_g, loss, stream);
  if (rc != FMM_OK) return set_err(rc);
  FMM_CUDA_TRY(fmm::launch_mlp_backward(P, P.corr_w, grad, reinterpret_cast<cudaStream_t>(stream)));
  return set_err(FMM_OK);
}

int fmm_plan_table_grid_size(const fmm_plan* plan, size_t* n) {
  if (!plan || !n) return set_err(FMM_ERR_ARG);
  const Plan& P = *reinterpret_cast<const Plan*>(plan);
  *n = (size_t)(P.L - 1) * fmm::grid_level_size(P.p);
  return set_err(FMM_OK);
}

int fmm_plan_set_table_grid(fmm_plan* plan, const float* theta, size_t n) {
  if (!plan) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const size_t need = (size_t)(P.L - 1) * fmm::grid_level_size(P.p);
  if (theta) {
    if (n != need) return set_err(FMM_ERR_ARG);
    if (!P.grid && !dev_alloc(&P.grid, need)) return set_err(FMM_ERR_ALLOC);
    FMM_CUDA_TRY(cudaMemcpy(P.grid, theta, need * sizeof(float), cudaMemcpyDefault));
    P.has_grid = 1;
  } else {
    P.has_grid = 0;
  }
  return set_err(retabulate(P, false));
}

int fmm_table_grid_grad(fmm_plan* plan, const float* density, const float* target_phi, const float* target_acc,
                        float w_phi, float w_g, float* grad, float* loss, void* stream) {
  if (!plan || !density || !target_phi || !target_acc || !grad || !loss) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const int rc = table_gradient(P, density, target_phi, target_acc, w_phi, w_g, loss, stream);
  if (rc != FMM_OK) return set_err(rc);
  FMM_CUDA_TRY(fmm::launch_grid_grad(P, grad, reinterpret_cast<cudaStream_t>(stream)));
  return set_err(FMM_OK);
}

int fmm_adam_step(float* w, const float* g, float* m, float* v, size_t n, int step, float lr, float beta1, float beta2,
                  float eps, void* stream) {
  if (!w || !g || !m || !v || n == 0 || step < 1) return set_err(FMM_ERR_ARG);
  FMM_CUDA_TRY(fmm::launch_adam(w, g, m, v, n, step, lr, beta1, beta2, eps, reinterpret_cast<cudaStream_t>(stream)));
  return set_err(FMM_OK);
}

int fmm_mesh_green(int N, float* out, void* stream) {
  if (N < 2 || !out) return set_err(FMM_ERR_ARG);
  int dev = 0, sms = 0;
  FMM_CUDA_TRY(cudaGetDevice(&dev));
  FMM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  FMM_CUDA_TRY(fmm::launch_mesh_green(N, out, sms, reinterpret_cast<cudaStream_t>(stream)));
  return set_err(FMM_OK);
}

int fmm_plan_mesh_green(const fmm_plan* plan, double* out, void* stream) {
  if (!plan || !out) return set_err(FMM_ERR_ARG);
  const Plan& P = *reinterpret_cast<const Plan*>(plan);
  FMM_CUDA_TRY(fmm::launch_mesh_green_plan(P, out, reinterpret_cast<cudaStream_t>(stream)));
  return set_err(FMM_OK);
}

int fmm_plan_check(fmm_plan* plan) {
  if (!plan) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  int h = 0;
  FMM_CUDA_TRY(cudaDeviceSynchronize());
  FMM_CUDA_TRY(cudaMemcpy(&h, P.d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (h) {
    FMM_CUDA_TRY(cudaMemset(P.d_err, 0, sizeof(int)));
    return set_err(FMM_ERR_TIMEOUT);
  }
  return set_err(FMM_OK);
}

int fmm_plan_set_timing(fmm_plan* plan, int enable) {
  if (!plan) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (enable && !P.ev[0]) {
    for (auto& e : P.ev) FMM_CUDA_TRY(cudaEventCreate(&e));
  }
  P.timing = enable ? 1 : 0;
  return set_err(FMM_OK);
}

int fmm_plan_stage_times(fmm_plan* plan, float* ms, int n) {
  if (!plan || !ms || n < 0) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (!P.timed) return set_err(FMM_ERR_ARG);
  const int k = n < FMM_TIME_SLOTS ? n : FMM_TIME_SLOTS;
  for (int i = 0; i < k; ++i) {
    ms[i] = 0.f;
    if (i == FMM_TIME_M2M && P.L <= 2) continue;
    if (i == FMM_TIME_L2L && P.L <= 2) continue;
    if (i >= FMM_TIME_M2L_LEVEL0 && (i - FMM_TIME_M2L_LEVEL0 < 2 || i - FMM_TIME_M2L_LEVEL0 > P.L)) continue;
    FMM_CUDA_TRY(cudaEventSynchronize(P.ev[2 * i + 1]));
    FMM_CUDA_TRY(cudaEventElapsedTime(&ms[i], P.ev[2 * i], P.ev[2 * i + 1]));
  }
  return set_err(FMM_OK);
}

int fmm_solve(fmm_plan* plan, const float* density, float* potential, float* accel, void* stream) {
  if (!plan || !density || !potential || !accel) return set_err(FMM_ERR_ARG);
  if (!aligned16(density) || !aligned16(potential) || !aligned16(accel)) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  if (P.unmade != FMM_OK) return set_err(P.unmade);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const bool t = P.timing != 0;
  auto mark = [&](int slot, int end) -> cudaError_t {
    return t ? cudaEventRecord(P.ev[2 * slot + end], s) : cudaSuccess;
  };
  FMM_CUDA_TRY(mark(FMM_TIME_MEAN, 0));
  if (P.iso)   // the isolated problem keeps every mass (m = rho / N^3)
    FMM_CUDA_TRY(cudaMemsetAsync(P.d_mean, 0, sizeof(double), s));
  else
    FMM_CUDA_TRY(fmm::launch_mean(P, density, s));
  FMM_CUDA_TRY(mark(FMM_TIME_MEAN, 1));
  // Untimed solves overlap independent stages: the near zone's spectral sums
  // need only the density and its mean (second auxiliary stream, from the mean
  // on), and fill what the small launches of the tree passes leave idle; the
  // M2L levels are independent of one another until the downward pass, so the
  // double-float levels run on the first auxiliary stream beside the FP32 and
  // tensor-core levels on `s`.  Timed solves stay serial, so that each stage's
  // events bracket it alone.
  const bool near_apart = !t && P.ns_K;
  if (near_apart) {
    FMM_CUDA_TRY(cudaEventRecord(P.fev[0], s));
    FMM_CUDA_TRY(cudaStreamWaitEvent(P.aux[1], P.fev[0], 0));
    FMM_CUDA_TRY(fmm::launch_near_spec_sums(P, density, P.aux[1]));
    FMM_CUDA_TRY(cudaEventRecord(P.fev[1], P.aux[1]));
  }
  FMM_CUDA_TRY(mark(FMM_TIME_P2M, 0));
  FMM_CUDA_TRY(fmm::launch_p2m(P, density, s));
  FMM_CUDA_TRY(mark(FMM_TIME_P2M, 1));
  FMM_CUDA_TRY(mark(FMM_TIME_M2M, 0));
  for (int l = P.L - 1; l >= 2; --l) FMM_CUDA_TRY(fmm::launch_m2m(P, l, s));
  FMM_CUDA_TRY(mark(FMM_TIME_M2M, 1));
  FMM_CUDA_TRY(mark(FMM_TIME_M2L, 0));
  auto on_tensor = [&](int l) { return m2l_form(P, l) == FMM_FORM_SPECTRAL_TC || m2l_form(P, l) == FMM_FORM_DENSE_TC; };
  auto on_spec = [&](int l) { return m2l_form(P, l) == FMM_FORM_SPECTRAL; };
  // one level on its own: FFT ablation, tensor cores or the dense CUDA-core kernels
  auto m2l_level = [&](int l, cudaStream_t q) -> cudaError_t {
    const int form = m2l_form(P, l);
    if (form == FMM_FORM_FFT) return fmm::launch_m2l_fft(P, l, q);
    if (form == FMM_FORM_SPECTRAL_TC) return fmm::launch_m2l_spec_tc(P, l, q);
    if (form == FMM_FORM_DENSE) return fmm::launch_m2l_fp32(P, l, q);
    const cudaError_t e = fmm::launch_split_bf16(P, l, q);
    return e != cudaSuccess ? e : fmm::launch_m2l_tc(P, l, P.prec, q);
  };
  if (!t) {
    // `s`: tensor-core levels, then the FP32 spectral levels; the first
    // auxiliary stream: the double-float spectral levels and the rest
    bool side = false, main = false;
    for (int l = 2; l <= P.L; ++l) {
      if (on_tensor(l) || (on_spec(l) && !fmm::wide_level(P, l))) main = true;
      else side = true;
    }
    const bool fork = side && main;
    cudaStream_t q = fork ? P.aux[0] : s;
    if (fork) FMM_CUDA_TRY(cudaEventRecord(P.fev[2], s));
    for (int l = P.L; l >= 2; --l)
      if (on_tensor(l)) FMM_CUDA_TRY(m2l_level(l, s));
    int f0 = P.L + 1, f1 = 1, d0 = P.L + 1, d1 = 1;   // spectral levels: wide_level and on_tensor split them by depth
    for (int l = 2; l <= P.L; ++l) {
      if (!on_spec(l)) continue;
      int &lo = fmm::wide_level(P, l) ? d0 : f0, &hi = fmm::wide_level(P, l) ? d1 : f1;
      lo = l < lo ? l : lo;
      hi = l;
    }
    if (f0 <= f1) FMM_CUDA_TRY(fmm::launch_m2l_spec(P, false, f0, f1, s));
    if (fork) FMM_CUDA_TRY(cudaStreamWaitEvent(q, P.fev[2], 0));
    if (d0 <= d1) FMM_CUDA_TRY(fmm::launch_m2l_spec(P, true, d0, d1, q));
    for (int l = 2; l <= P.L; ++l)
      if (!on_tensor(l) && !on_spec(l)) FMM_CUDA_TRY(m2l_level(l, q));
    if (fork) {
      FMM_CUDA_TRY(cudaEventRecord(P.fev[3], q));
      FMM_CUDA_TRY(cudaStreamWaitEvent(s, P.fev[3], 0));
    }
  } else {
    for (int l = 2; l <= P.L; ++l) {
      FMM_CUDA_TRY(mark(FMM_TIME_M2L_LEVEL0 + l, 0));
      FMM_CUDA_TRY(on_spec(l) ? fmm::launch_m2l_spec(P, fmm::wide_level(P, l), l, l, s) : m2l_level(l, s));
      FMM_CUDA_TRY(mark(FMM_TIME_M2L_LEVEL0 + l, 1));
    }
  }
  FMM_CUDA_TRY(mark(FMM_TIME_M2L, 1));
  FMM_CUDA_TRY(mark(FMM_TIME_L2L, 0));
  for (int l = 2; l < P.L; ++l) FMM_CUDA_TRY(fmm::launch_l2l(P, l, s));
  FMM_CUDA_TRY(mark(FMM_TIME_L2L, 1));
  FMM_CUDA_TRY(mark(FMM_TIME_P2P, 0));
  if (near_apart) FMM_CUDA_TRY(cudaStreamWaitEvent(s, P.fev[1], 0));
  FMM_CUDA_TRY(fmm::launch_p2p(P, density, potential, accel, s, near_apart));
  FMM_CUDA_TRY(mark(FMM_TIME_P2P, 1));
  P.solved = 1;
  if (t) P.timed = 1;
  return set_err(FMM_OK);
}

int fmm_solve_host(fmm_plan* plan, const float* density_host, float* potential_host, float* accel_host,
                   void* stream) {
  if (!plan || !density_host || !potential_host || !accel_host) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  const size_t n3 = (size_t)P.N * P.N * P.N;
  if ((!P.stage_in && !plan_alloc(P, &P.stage_in, n3)) || (!P.stage_out && !plan_alloc(P, &P.stage_out, 4 * n3)))
    return set_err(FMM_ERR_ALLOC);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  FMM_CUDA_TRY(cudaMemcpyAsync(P.stage_in, density_host, n3 * sizeof(float), cudaMemcpyHostToDevice, s));
  int rc = fmm_solve(plan, P.stage_in, P.stage_out, P.stage_out + n3, stream);
  if (rc != FMM_OK) return rc;
  FMM_CUDA_TRY(cudaMemcpyAsync(potential_host, P.stage_out, n3 * sizeof(float), cudaMemcpyDeviceToHost, s));
  FMM_CUDA_TRY(cudaMemcpyAsync(accel_host, P.stage_out + n3, 3 * n3 * sizeof(float), cudaMemcpyDeviceToHost, s));
  FMM_CUDA_TRY(cudaStreamSynchronize(s));
  return set_err(FMM_OK);
}

int fmm_plan_copy_stage(fmm_plan* plan, int stage, int level, float* dst, size_t count, void* stream) {
  if (!plan || !dst) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const size_t p3 = (size_t)P.p * P.p * P.p;
  if (stage == FMM_STAGE_MEAN) {
    if (count < 1) return set_err(FMM_ERR_ARG);
    // one-value conversion through the host keeps this path free of extra kernels
    double m = 0.0;
    FMM_CUDA_TRY(cudaMemcpyAsync(&m, P.d_mean, sizeof(double), cudaMemcpyDeviceToHost, s));
    FMM_CUDA_TRY(cudaStreamSynchronize(s));
    const float mf = (float)m;
    FMM_CUDA_TRY(cudaMemcpyAsync(dst, &mf, sizeof(float), cudaMemcpyHostToDevice, s));
    FMM_CUDA_TRY(cudaStreamSynchronize(s));
    return set_err(FMM_OK);
  }
  if (level < 2 || level > P.L) return set_err(FMM_ERR_ARG);
  const size_t nodes = (size_t)1 << (3 * level);
  const float* src = nullptr;
  size_t need = 0;
  if (stage == FMM_STAGE_MULTIPOLE) {
    src = P.M[level];
    need = nodes * p3;
  } else if (stage == FMM_STAGE_LOCAL) {
    src = P.F[level];
    need = nodes * 4 * p3;
  } else {
    return set_err(FMM_ERR_ARG);
  }
  if (count < need) return set_err(FMM_ERR_ARG);
  FMM_CUDA_TRY(cudaMemcpyAsync(dst, src, need * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return set_err(FMM_OK);
}

int fmm_plan_error_stats(fmm_plan* plan, const float* density, const float* potential, const float* accel,
                         int samples, unsigned long long seed, double* out, void* stream) {
  if (!plan || !density || !potential || !accel || !out) return set_err(FMM_ERR_ARG);
  if (!aligned16(density) || !aligned16(potential) || !aligned16(accel)) return set_err(FMM_ERR_ARG);
  if (samples < 1 || samples > fmm::error_stats_max_samples()) return set_err(FMM_ERR_ARG);
  Plan& P = *reinterpret_cast<Plan*>(plan);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const unsigned long long n3 = (unsigned long long)P.N * P.N * P.N;
  std::vector<unsigned long long> targets((size_t)samples);
  for (int i = 0; i < samples; ++i) {
    // output i of splitmix64 (Steele, Lea and Flood 2014) seeded with `seed`
    unsigned long long z = seed + (unsigned long long)(i + 1) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    z ^= z >> 31;
    targets[(size_t)i] = z % n3;
  }
  // one plan-owned block, kept between calls: partials, mean, largest value, sums, targets.
  // The call ends synchronised, so the lock covers every use of the block.
  std::lock_guard<std::mutex> hold(P.es_lock);
  const size_t np = (size_t)fmm::error_stats_grid_x(P, samples) * samples * 4, nm = (size_t)P.n_partials + 2,
               ns = 4 + 4 * (size_t)samples, bytes = sizeof(double) * (np + nm + ns + (size_t)samples);
  if (P.es_bytes < bytes) {
    cudaFree(P.es_scratch);
    P.es_scratch = nullptr;
    P.es_bytes = 0;
    if (!plan_alloc(P, &P.es_scratch, bytes)) return set_err(FMM_ERR_ALLOC);
    P.es_bytes = bytes;
  }
  double* d_partials = static_cast<double*>(P.es_scratch);
  double *d_mean = d_partials + np, *d_sums = d_mean + nm;
  unsigned long long* d_targets = reinterpret_cast<unsigned long long*>(d_sums + ns);
  FMM_CUDA_TRY(cudaMemcpyAsync(d_targets, targets.data(), sizeof(unsigned long long) * samples,
                               cudaMemcpyHostToDevice, s));
  FMM_CUDA_TRY(
      fmm::launch_error_stats(P, density, potential, accel, d_targets, samples, d_partials, d_sums, d_mean, s));
  double sums[4] = {0.0, 0.0, 0.0, 0.0};
  FMM_CUDA_TRY(cudaMemcpyAsync(sums, d_sums, sizeof(sums), cudaMemcpyDeviceToHost, s));
  FMM_CUDA_TRY(cudaStreamSynchronize(s));
  out[0] = sums[1] > 0.0 ? std::sqrt(sums[0] / sums[1]) : std::sqrt(sums[0]);
  out[1] = sums[3] > 0.0 ? std::sqrt(sums[2] / sums[3]) : std::sqrt(sums[2]);
  return set_err(FMM_OK);
}

}  // extern "C"
