// gm_tune.cu -- launch-shape autotuner of the EM kernel (gm_autotune, C ABI
// in include/gm.h).  Trials run gm_compress itself on a sample of the
// batch, with a fixed number of sweeps so that every candidate does the
// same work.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "gm_kernels.cuh"

namespace {

int tune_fail(int code, const char* what, cudaError_t e = cudaSuccess) {
  char buf[256];
  if (e != cudaSuccess)
    snprintf(buf, sizeof buf, "gm_autotune: %s: %s", what, cudaGetErrorString(e));
  else
    snprintf(buf, sizeof buf, "gm_autotune: %s", what);
  return gmcr::record_error(code, buf);
}

// device buffers of one trial's outputs
struct TrialOut {
  void* base = nullptr;
  int32_t *K = nullptr, *sweeps = nullptr, *kwork = nullptr;
  double *params = nullptr, *W = nullptr, *rho = nullptr, *lnL = nullptr;
  uint32_t* status = nullptr;
};

size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

// candidates: lanes of a cell's sums x shared tiles; candidate i = (kTuneNT[i % 3], tile i / 3)
constexpr int kTuneThreads = 3;
constexpr int kTuneNT[kTuneThreads] = {64, 128, 256};
constexpr int kTuneCaps = 5;
constexpr int kTuneCands = kTuneThreads * kTuneCaps;
static_assert(kTuneCands == GM_TUNE_CANDIDATES, "gm.h states the number of candidates");

int tune_impl(gm_config* cfg, int64_t C, int64_t n_particles, const int64_t* cell_off,
              const double* x, const void* v, int32_t v_is_f64, const double* alpha,
              const int32_t* init_K, const double* init_params, int32_t sweeps_per_trial,
              float* timings_ms, void* stream) {
  if (!cfg || !cell_off || !x || !v || !alpha) return tune_fail(GM_ERR_ARG, "a required pointer is NULL");
  if (C < 1) return tune_fail(GM_ERR_ARG, "C must be >= 1");
  if (cfg->D != 1 && cfg->D != 3) return tune_fail(GM_ERR_ARG, "D must be 1 or 3");
  if (cfg->Kmax < 1 || cfg->Kmax > gmcr::kMaxK) return tune_fail(GM_ERR_ARG, "Kmax out of range");
  if (sweeps_per_trial < 0) return tune_fail(GM_ERR_ARG, "sweeps_per_trial < 0");
  const int spt = sweeps_per_trial > 0 ? sweeps_per_trial : 24;
  cudaStream_t s = (cudaStream_t)stream;
  const int D = cfg->D;
  const int P = 1 + D + D * (D + 1) / 2;

  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return tune_fail(GM_ERR_CUDA, "cudaGetDevice", e);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 1) sms = 1;

  // cell sizes of the sample: the first 128 cells per SM (many cells per
  // team, so that a trial measures throughput, not one wave)
  const int64_t S = std::min<int64_t>(C, (int64_t)128 * sms);
  std::vector<int64_t> off((size_t)S + 1);
  e = cudaMemcpyAsync(off.data(), cell_off, sizeof(int64_t) * (size_t)(S + 1), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return tune_fail(GM_ERR_CUDA, "reading cell_off", e);
  std::vector<int64_t> sizes((size_t)S);
  for (int64_t j = 0; j < S; ++j) sizes[(size_t)j] = off[(size_t)j + 1] - off[(size_t)j];
  std::sort(sizes.begin(), sizes.end());
  auto quant = [&](double q) {
    const size_t i = std::min(sizes.size() - 1, (size_t)(q * (double)(sizes.size() - 1) + 0.5));
    return sizes[i];
  };

  // candidate shared tiles (particles, multiple of 4, within 200 KB).  The
  // library's default is the largest one: every cell that fits the pool may have
  // a shared tile.  A smaller limit sends the cells above it to L2 and leaves
  // the pool to the others; a limit that no cell of the sample reaches is the
  // default again.
  const int64_t max_cap = (int64_t)(200 * 1024) / ((int64_t)(D + 4) * 4) & ~(int64_t)3;
  std::vector<int> caps;
  auto add_cap = [&](int64_t c) {
    c = (c + 1 + 3) & ~(int64_t)3;  // pad particle, multiple of 4
    if (c < 4) c = 4;
    if (c > max_cap) return;
    if (std::find(caps.begin(), caps.end(), (int)c) == caps.end()) caps.push_back((int)c);
  };
  add_cap(max_cap - 1);  // the library default
  for (const double q : {0.90, 0.99, 0.50})
    if (quant(q) < sizes.back()) add_cap(quant(q));
  if (caps.size() > (size_t)kTuneCaps) caps.resize(kTuneCaps);

  // trial outputs
  TrialOut o;
  const size_t bK = up256(sizeof(int32_t) * (size_t)S), bP = up256(sizeof(double) * (size_t)S * cfg->Kmax * P),
               bD = up256(sizeof(double) * (size_t)S);
  e = cudaMalloc(&o.base, 4 * bK + bP + 3 * bD);
  if (e != cudaSuccess) return tune_fail(GM_ERR_NOMEM, "trial outputs", e);
  char* b = (char*)o.base;
  o.K = (int32_t*)b;
  o.sweeps = (int32_t*)(b + bK);
  o.kwork = (int32_t*)(b + 2 * bK);
  o.status = (uint32_t*)(b + 3 * bK);
  o.params = (double*)(b + 4 * bK);
  o.W = (double*)(b + 4 * bK + bP);
  o.rho = (double*)(b + 4 * bK + bP + bD);
  o.lnL = (double*)(b + 4 * bK + bP + 2 * bD);

  cudaEvent_t t0 = nullptr, t1 = nullptr;
  e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  if (e != cudaSuccess) {
    if (t0) cudaEventDestroy(t0);
    cudaFree(o.base);
    return tune_fail(GM_ERR_CUDA, "timing events", e);
  }
  float times[kTuneCands];
  for (int i = 0; i < kTuneCands; ++i) times[i] = -1.0f;
  int best = -1;
  int rc = GM_OK;
  for (size_t ci = 0; ci < caps.size() && rc == GM_OK; ++ci) {
    for (int ti = 0; ti < kTuneThreads; ++ti) {
      gm_config tr = *cfg;
      // the paper's start: tol = 0, every candidate does the same sweeps; a
      // supplied start: the caller's tol, capped at sweeps_per_trial (0 =
      // 64): a start that leaves most cells converged in a few sweeps and
      // one that needs hundreds weigh per-cell and per-sweep costs very
      // differently, while without a cap the sample's few slowest cells
      // decide the trial (in a whole batch they are hidden among the rest)
      tr.tol = init_K ? cfg->tol : 0.0;
      tr.max_sweeps = init_K ? (sweeps_per_trial > 0 ? sweeps_per_trial : 64) : spt;
      tr.threads_per_cell = kTuneNT[ti];
      tr.smem_particles = caps[ci];
      tr.L = cfg->L * (double)S / (double)C;  // the sample keeps the cell width
      float tmin = -1.0f;
      for (int rep = 0; rep < 3; ++rep) {  // one warm-up, two timed
        cudaEventRecord(t0, s);
        const int r =
            init_K ? gm_compress_from(&tr, S, n_particles, cell_off, x, v, v_is_f64, alpha, init_K,
                                      init_params, o.K, o.params, o.W, o.rho, o.lnL, o.sweeps,
                                      o.kwork, o.status, stream)
                   : gm_compress(&tr, S, n_particles, cell_off, x, v, v_is_f64, alpha, o.K, o.params,
                                 o.W, o.rho, o.lnL, o.sweeps, o.kwork, o.status, stream);
        if (r != GM_OK) {
          tmin = -1.0f;
          break;
        }
        cudaEventRecord(t1, s);
        e = cudaEventSynchronize(t1);
        if (e != cudaSuccess) {
          rc = tune_fail(GM_ERR_CUDA, "trial", e);
          break;
        }
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, t0, t1);
        if (rep > 0 && (tmin < 0.0f || ms < tmin)) tmin = ms;
      }
      times[(int)ci * kTuneThreads + ti] = tmin;
    }
  }
  cudaEventDestroy(t0);
  cudaEventDestroy(t1);
  cudaFree(o.base);
  if (rc != GM_OK) return rc;
  // the library default (256 lanes, default tile: candidate 2) stays unless
  // another shape is faster by more than 3 %, and each number of lanes keeps
  // the default tile (candidates 0 to 2) unless another is by as much: trials closer
  // than that are within the run-to-run spread
  for (int ti = kTuneThreads - 1; ti >= 0; --ti) {
    int c = -1;
    for (int i = ti; i < kTuneCands; i += kTuneThreads)
      if (times[i] >= 0.0f && (c < 0 || times[i] < (c == ti ? 0.97f : 1.0f) * times[c])) c = i;
    if (c >= 0 && (best < 0 || times[c] < (best % kTuneThreads == kTuneThreads - 1 ? 0.97f : 1.0f) * times[best]))
      best = c;
  }
  if (best < 0) return tune_fail(GM_ERR_CUDA, "no candidate ran");
  if (timings_ms)
    for (int i = 0; i < kTuneCands; ++i) timings_ms[i] = times[i];
  cfg->threads_per_cell = kTuneNT[best % kTuneThreads];
  cfg->smem_particles = caps[(size_t)(best / kTuneThreads)];
  gmcr::record_error(GM_OK, "");
  return GM_OK;
}

}  // namespace

extern "C" int gm_autotune(gm_config* cfg, int64_t C, int64_t n_particles, const int64_t* cell_off,
                           const double* x, const void* v, int32_t v_is_f64, const double* alpha,
                           int32_t sweeps_per_trial, float* timings_ms, void* stream) {
  return tune_impl(cfg, C, n_particles, cell_off, x, v, v_is_f64, alpha, nullptr, nullptr,
                   sweeps_per_trial, timings_ms, stream);
}

extern "C" int gm_autotune_from(gm_config* cfg, int64_t C, int64_t n_particles,
                                const int64_t* cell_off, const double* x, const void* v,
                                int32_t v_is_f64, const double* alpha, const int32_t* init_K,
                                const double* init_params, int32_t sweeps_per_trial,
                                float* timings_ms, void* stream) {
  if (!init_K || !init_params) return tune_fail(GM_ERR_ARG, "init_K and init_params are required");
  return tune_impl(cfg, C, n_particles, cell_off, x, v, v_is_f64, alpha, init_K, init_params,
                   sweeps_per_trial, timings_ms, stream);
}
