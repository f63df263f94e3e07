// gm_mlp.cu -- C ABI of the learned-initialisation network: the BF16
// tensor-core GEMM and the network's forward / backward / update steps.
#include <string>

#include "gm_kernels.cuh"

extern "C" {

int gm_gemm_bf16(int32_t M, int32_t N, int32_t K, const void* A, int32_t lda, const void* B,
                 int32_t ldb, const float* bias, int32_t relu, const void* mask, int32_t ldm,
                 float* C_f32, void* C_bf16, int32_t ldc, uint32_t* err, void* stream) {
  gmcr::record_error(GM_OK, "");
  if (M < 0 || N < 0 || K < 0) return gmcr::record_error(GM_ERR_ARG, "negative GEMM size");
  if (M == 0 || N == 0 || K == 0) return GM_OK;
  if (!A || !B || (!C_f32 && !C_bf16)) return gmcr::record_error(GM_ERR_ARG, "a GEMM pointer is NULL");
  if (lda < K || ldb < K || (lda & 7) || (ldb & 7) || ldc < N)
    return gmcr::record_error(GM_ERR_ARG, "GEMM leading dimensions: lda, ldb >= K and multiples of 8; ldc >= N");
  if ((((uintptr_t)A) & 15) || (((uintptr_t)B) & 15))
    return gmcr::record_error(GM_ERR_ARG, "GEMM operands must be 16-byte aligned");
  int dev = 0, major = 0, minor = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  if (major != 10 || minor != 3)
    return gmcr::record_error(GM_ERR_UNSUPPORTED, "this library is built for sm_103a");
  cudaError_t e = gmcr::launch_tc_gemm(A, nullptr, B, M, N, K, lda, ldb, bias, relu, mask, ldm, C_f32,
                                       C_bf16, ldc, err, (cudaStream_t)stream);
  if (e != cudaSuccess)
    return gmcr::record_error(GM_ERR_CUDA, (std::string("GEMM launch: ") + cudaGetErrorString(e)).c_str());
  return GM_OK;
}

}  // extern "C"

namespace {

int check_sm103() {
  int dev = 0, major = 0, minor = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  if (major != 10 || minor != 3)
    return gmcr::record_error(GM_ERR_UNSUPPORTED, "this library is built for sm_103a");
  return GM_OK;
}

int cuda_err(cudaError_t e, const char* what) {
  return gmcr::record_error(GM_ERR_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}

size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

int check_net(const gm_mlp* net) {
  if (!net) return gmcr::record_error(GM_ERR_ARG, "net is NULL");
  if (net->D != 1 && net->D != 3) return gmcr::record_error(GM_ERR_ARG, "net->D must be 1 or 3");
  const int F = net->D == 1 ? 128 : 576;
  const int SP = 2 + 2 * net->D + net->D * (net->D - 1) / 2;
  if (net->F != F || net->H != 256 || net->O < net->Kmax * SP || (net->O & 15) || net->Kmax < 1 ||
      net->Kmax > gmcr::kMaxK)
    return gmcr::record_error(GM_ERR_ARG, "gm_mlp widths: F = 128 (D=1) / 576 (D=3), H = 256, "
                                          "O >= Kmax * slot size and a multiple of 16");
  for (int l = 0; l < 4; ++l)
    if (!net->W[l] || !net->b[l] || !net->W16[l] || !net->WT16[l])
      return gmcr::record_error(GM_ERR_ARG, "a gm_mlp weight pointer is NULL");
  return GM_OK;
}

// scratch layout for M rows.  The gradients stay until the update takes their
// column sums; those of the first two layers lie over H[1], TH[1] and H[2],
// TH[2], whose last reader has run by then (7.7 KB a row in 3V, 9.8 without).
struct MlpScratch {
  void *H[3], *hi, *lo, *TLhi, *TLlo, *TX, *TH[3];
  float* G[4];  // the loss gradient of each layer's (pre-)activations
};
size_t scratch_layout(const gm_mlp* net, int M, char* base, MlpScratch* sc) {
  const size_t H = net->H, O = net->O, F = net->F, big = H > O ? H : O;
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* p = base ? base + off : nullptr;
    off += al(bytes);
    return p;
  };
  const size_t half = (size_t)M * H * 2;  // a multiple of 256: H = 256
  for (int l = 0; l < 3; ++l) {
    char* p = take(2 * half);
    sc->H[l] = p;
    sc->TH[l] = base ? p + half : nullptr;
    if (l > 0) sc->G[l - 1] = (float*)p;
  }
  for (int l = 2; l < 4; ++l) sc->G[l] = (float*)take((size_t)M * (l < 3 ? H : O) * 4);
  sc->hi = take((size_t)M * big * 2);
  sc->lo = take((size_t)M * big * 2);
  sc->TLhi = take(big * (size_t)M * 2);
  sc->TLlo = take(big * (size_t)M * 2);
  sc->TX = take(F * (size_t)M * 2);
  return off;
}

int gemm(const void* A, const void* A2, const void* B, int M, int N, int K, int lda, int ldb,
         const float* bias, int relu, float* Cf, void* Cb, int ldc, uint32_t* err, cudaStream_t s) {
  cudaError_t e = gmcr::launch_tc_gemm(A, A2, B, M, N, K, lda, ldb, bias, relu, nullptr, 0, Cf, Cb, ldc, err, s);
  return e == cudaSuccess ? GM_OK : cuda_err(e, "GEMM launch");
}

int forward_impl(const gm_mlp* net, int M, const void* X, const MlpScratch& sc, float* out,
                 uint32_t* err, cudaStream_t s) {
  const int F = net->F, H = net->H, O = net->O;
  int rc;
  const void* in[4] = {X, sc.H[0], sc.H[1], sc.H[2]};
  for (int l = 0; l < 3; ++l) {
    const int K = l == 0 ? F : H;
    if ((rc = gemm(in[l], nullptr, net->W16[l], M, H, K, K, K, net->b[l], 1, nullptr, sc.H[l], H, err, s)))
      return rc;
  }
  return gemm(in[3], nullptr, net->W16[3], M, O, H, H, H, net->b[3], 0, out, nullptr, O, err, s);
}

}  // namespace

extern "C" {

int gm_features(const gm_config* cfg, int64_t C, int64_t n_particles, const int64_t* cell_off,
                const void* v, int32_t v_is_f64, const double* alpha, void* feat, double* wstat,
                void* stream) {
  gmcr::record_error(GM_OK, "");
  if (!cfg || (cfg->D != 1 && cfg->D != 3)) return gmcr::record_error(GM_ERR_ARG, "bad cfg");
  if (C < 0 || n_particles < 0) return gmcr::record_error(GM_ERR_ARG, "negative size");
  if (C == 0) return GM_OK;
  if (!cell_off || !v || !alpha || !feat || !wstat)
    return gmcr::record_error(GM_ERR_ARG, "a required pointer is NULL");
  int rc = check_sm103();
  if (rc) return rc;
  gmcr::trace_mark(nullptr, (cudaStream_t)stream);
  cudaError_t e = gmcr::launch_features(cfg->D, C, n_particles, cell_off, v, v_is_f64, alpha, feat,
                                        wstat, (cudaStream_t)stream);
  gmcr::trace_mark("features_kernel", (cudaStream_t)stream);
  return e == cudaSuccess ? GM_OK : cuda_err(e, "features launch");
}

int gm_mlp_targets(const gm_config* cfg, int64_t C, const int32_t* K, const double* params,
                   const double* wstat, int32_t O, float* T, float* Mk, void* stream) {
  gmcr::record_error(GM_OK, "");
  if (!cfg || (cfg->D != 1 && cfg->D != 3) || cfg->Kmax < 1 || cfg->Kmax > gmcr::kMaxK)
    return gmcr::record_error(GM_ERR_ARG, "bad cfg");
  const int SP = 2 + 2 * cfg->D + cfg->D * (cfg->D - 1) / 2;
  if (O < cfg->Kmax * SP) return gmcr::record_error(GM_ERR_ARG, "O too small");
  if (C == 0) return GM_OK;
  if (!K || !params || !wstat || !T || !Mk)
    return gmcr::record_error(GM_ERR_ARG, "a required pointer is NULL");
  int rc = check_sm103();
  if (rc) return rc;
  cudaError_t e = gmcr::launch_targets(cfg->D, C, cfg->Kmax, O, K, params, wstat, T, Mk,
                                       (cudaStream_t)stream);
  return e == cudaSuccess ? GM_OK : cuda_err(e, "targets launch");
}

int gm_mlp_sync(const gm_mlp* net, void* stream) {
  gmcr::record_error(GM_OK, "");
  int rc = check_net(net);
  if (rc || (rc = check_sm103())) return rc;
  const int rows[4] = {net->H, net->H, net->H, net->O};
  const int cols[4] = {net->F, net->H, net->H, net->H};
  for (int l = 0; l < 4; ++l) {
    cudaError_t e = gmcr::launch_cast_weights(rows[l], cols[l], net->W[l], net->W16[l],
                                              net->WT16[l], (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_err(e, "cast launch");
  }
  return GM_OK;
}

size_t gm_mlp_scratch_bytes(const gm_mlp* net, int32_t M) {
  if (!net || M <= 0) return 0;
  MlpScratch sc;
  return scratch_layout(net, M, nullptr, &sc);
}

int gm_mlp_forward(const gm_mlp* net, int32_t M, const void* X, void* scratch,
                   size_t scratch_bytes, float* out, uint32_t* err, void* stream) {
  gmcr::record_error(GM_OK, "");
  int rc = check_net(net);
  if (rc) return rc;
  if (M < 0) return gmcr::record_error(GM_ERR_ARG, "M < 0");
  if (M == 0) return GM_OK;
  if (!X || !out || !scratch) return gmcr::record_error(GM_ERR_ARG, "a required pointer is NULL");
  if (scratch_bytes < gm_mlp_scratch_bytes(net, M))
    return gmcr::record_error(GM_ERR_ARG, "scratch too small (see gm_mlp_scratch_bytes)");
  if ((rc = check_sm103())) return rc;
  MlpScratch sc;
  scratch_layout(net, M, (char*)scratch, &sc);
  gmcr::trace_mark(nullptr, (cudaStream_t)stream);
  rc = forward_impl(net, M, X, sc, out, err, (cudaStream_t)stream);
  gmcr::trace_mark("mlp_forward (tc_gemm_kernel x4)", (cudaStream_t)stream);
  return rc;
}

int gm_mlp_train_step(const gm_mlp* net, int32_t M, const void* X, const float* T,
                      const float* Mk, float lr, int32_t step, void* scratch,
                      size_t scratch_bytes, float* out, double* loss, uint32_t* err,
                      void* stream) {
  gmcr::record_error(GM_OK, "");
  int rc = check_net(net);
  if (rc) return rc;
  if (M <= 0 || (M % 64)) return gmcr::record_error(GM_ERR_ARG, "M must be a positive multiple of 64");
  if (!X || !T || !Mk || !out || !loss || !scratch)
    return gmcr::record_error(GM_ERR_ARG, "a required pointer is NULL");
  for (int l = 0; l < 4; ++l)
    if (!net->gW[l] || !net->gb[l] || (lr > 0.0f && (!net->mW[l] || !net->vW[l] || !net->mb[l] || !net->vb[l])))
      return gmcr::record_error(GM_ERR_ARG, "a gm_mlp gradient / moment pointer is NULL");
  if (lr > 0.0f && step < 1) return gmcr::record_error(GM_ERR_ARG, "step must be >= 1");
  if (scratch_bytes < gm_mlp_scratch_bytes(net, M))
    return gmcr::record_error(GM_ERR_ARG, "scratch too small (see gm_mlp_scratch_bytes)");
  if ((rc = check_sm103())) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  MlpScratch sc;
  scratch_layout(net, M, (char*)scratch, &sc);
  const int F = net->F, H = net->H, O = net->O;
  gmcr::trace_mark(nullptr, s);
  if ((rc = forward_impl(net, M, X, sc, out, err, s))) return rc;
  // The step takes 17 launches (about 50 with one for each split, transpose,
  // column sum, hi or lo product and tensor update): 1024 rows in 3V 0.78 ->
  // 0.35 ms, and 0.17 with the GEMM's idle lanes off its barrier.  Each layer's gradient dZ is fed to the tensor cores as
  // hi + lo BF16 parts, which keeps FP32-level accuracy.
  gmcr::TransposeJobs tj = {{X, sc.H[0], sc.H[1], sc.H[2]}, {sc.TX, sc.TH[0], sc.TH[1], sc.TH[2]}, {F, H, H, H}};
  cudaError_t e = gmcr::launch_transposes(M, tj, s);
  if (e != cudaSuccess) return cuda_err(e, "transpose");
  gmcr::GradOut g = {sc.hi, sc.lo, sc.TLhi, sc.TLlo, sc.G[3]};
  if ((e = gmcr::launch_loss_grad(M, O, net->D, net->Kmax, out, T, Mk, g, loss, s)) != cudaSuccess)
    return cuda_err(e, "loss launch");
  for (int l = 3; l >= 0; --l) {
    // gW = dZ^T H_prev; dZ_prev = (dZ W) where H_prev > 0
    const int C = l == 3 ? O : H, P = l == 0 ? F : H;
    if ((rc = gemm(sc.TLhi, sc.TLlo, l == 0 ? sc.TX : sc.TH[l - 1], C, P, M, M, M, nullptr, 0, net->gW[l],
                   nullptr, P, err, s)))
      return rc;
    if (l == 0) break;
    // (G[l - 1] takes the place of H[l] and TH[l] from here on, see scratch_layout)
    if ((rc = gemm(sc.hi, sc.lo, net->WT16[l], M, H, C, C, C, nullptr, 0, sc.G[l - 1], nullptr, H, err, s)))
      return rc;
    g = {l > 1 ? sc.hi : nullptr, l > 1 ? sc.lo : nullptr, sc.TLhi, sc.TLlo, sc.G[l - 1]};
    if ((e = gmcr::launch_grad_prep(M, H, sc.H[l - 1], g, s)) != cudaSuccess) return cuda_err(e, "gradient");
  }
  gmcr::UpdateJobs u;
  for (int l = 0; l < 4; ++l) {
    u.W[l] = net->W[l]; u.b[l] = net->b[l]; u.gW[l] = net->gW[l]; u.gb[l] = net->gb[l];
    u.mW[l] = net->mW[l]; u.vW[l] = net->vW[l]; u.mb[l] = net->mb[l]; u.vb[l] = net->vb[l];
    u.W16[l] = net->W16[l]; u.WT16[l] = net->WT16[l];
    u.G[l] = sc.G[l];
    u.rows[l] = l == 3 ? O : H;
    u.cols[l] = l == 0 ? F : H;
  }
  u.M = M;
  if ((e = gmcr::launch_update(u, lr, step, s)) != cudaSuccess) return cuda_err(e, "update");
  gmcr::trace_mark("mlp_train_step", s);
  return GM_OK;
}

int gm_mlp_decode(const gm_config* cfg, int64_t C, const float* out, int32_t O,
                  const double* wstat, const int64_t* cell_off, float presence_logit, int32_t* K0,
                  double* init_params, void* stream) {
  gmcr::record_error(GM_OK, "");
  if (!cfg || (cfg->D != 1 && cfg->D != 3) || cfg->Kmax < 1 || cfg->Kmax > gmcr::kMaxK)
    return gmcr::record_error(GM_ERR_ARG, "bad cfg");
  const int SP = 2 + 2 * cfg->D + cfg->D * (cfg->D - 1) / 2;
  if (O < cfg->Kmax * SP) return gmcr::record_error(GM_ERR_ARG, "O too small");
  if (C == 0) return GM_OK;
  if (!out || !wstat || !cell_off || !K0 || !init_params)
    return gmcr::record_error(GM_ERR_ARG, "a required pointer is NULL");
  int rc = check_sm103();
  if (rc) return rc;
  if (!(presence_logit == presence_logit)) return gmcr::record_error(GM_ERR_ARG, "presence_logit is NaN");
  gmcr::trace_mark(nullptr, (cudaStream_t)stream);
  cudaError_t e = gmcr::launch_decode(cfg->D, C, cfg->Kmax, O, out, wstat, cell_off, presence_logit,
                                      K0, init_params, (cudaStream_t)stream);
  gmcr::trace_mark("decode_kernel", (cudaStream_t)stream);
  return e == cudaSuccess ? GM_OK : cuda_err(e, "decode launch");
}

}  // extern "C"
