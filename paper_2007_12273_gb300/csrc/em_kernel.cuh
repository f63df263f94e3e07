// em_kernel.cuh -- persistent per-cell adaptive EM (compression, Sec. 2.2-2.3)
//
// One CTA per SM holds several teams of warps; a team fits one cell at a
// time and pulls the next cell from an atomic ticket.  A cell's particles are
// staged once (whitened FP32 velocities and normalised weights) in a tile of
// the CTA's shared memory, taken from a pool for the cell's size -- or, when
// the cell does not fit, in an L2-resident global scratch with the same
// layout -- and reused by every sweep.  Each thread works on pairs of
// particles with Blackwell's packed FP32 (f32x2) arithmetic.
//
// What bounds it: a component step is a pass over the cell (four warps, 2 to
// 4 thousand cycles) and then a serial M-step in one warp (3 thousand cycles
// for D = 1, 5 thousand for D = 3, FP64 latency), with a convergence test a
// sweep (5 thousand, half of it an FP64 logarithm).  The other teams' passes
// and M-steps run meanwhile; how many there are is set by shared memory (20 or 28
// bytes per particle, 16 or 24 with equal weights) and by registers.
// 16384 3V cells of 572 particles: 285 -> 124 ms against one CTA of 256
// threads per cell with a fixed tile of 3072 particles (two per SM); 4096 1V
// cells of 2000: 113 -> 104 ms; 1024 3V cells of 1024 with unequal weights:
// 43 -> 24 ms.
//
// Component-wise EM (Sec. 2.3, Celeux et al.): the E-step of component k
// needs the normaliser s_p = sum_j omega_j f_j(v_p) with the *current*
// parameters of every component.  s_p is kept per particle (FP32, relative
// to a per-particle log2 shift m_p): a pass for component k first replaces
// the previous component's old term by its updated one, then evaluates
// f_k, the responsibility gamma_pk = alpha_p omega_k f_k / s_p and the
// per-thread FP32 sufficient statistics of component k about its old mean.
// Once per sweep an exact pass recomputes s_p and m_p and yields eq.
// (lnL-GM).  Weights are kept unnormalised (omega_j = u_j / Z), which makes
// the renormalisation after each component (step 3) implicit.
//
// The exact pass is fused with the E-step of the next sweep's first
// component, so a sweep of K components costs K passes over the particles.
//
// Precision: E-step densities / responsibilities FP32; statistics FP32 per
// thread and per warp, summed across warps in R; the M-step in R (FP32:
// precision 0, FP64: precision 1) with the component means accumulated to
// about 48 bits either way (FP64, or an unevaluated FP32 sum hi + lo when R
// is FP32, which keeps FP64 arithmetic off the M-step's critical path); the
// final unpenalised step (Sec. 2.3.1) entirely in FP64 with FP64-normalised
// responsibilities, which is what makes the moments exact.
#pragma once

#include <type_traits>

#include "gm_common.cuh"

namespace gmcr {

struct EmParams {
  int64_t C, n;
  const int64_t* cell_off;
  const void* v;
  const double* alpha;
  int32_t* K_out;
  double* params_out;
  double* W_out;
  double* lnL_out;
  int32_t* sweeps_out;
  int32_t* kwork_out;
  uint32_t* status_out;
  const int32_t* init_K;   // optional initial mixtures (original coordinates)
  const double* init_prm;  // [C][Kmax][P]
  float* scratch;          // global tile for cells without a shared one
  int64_t scratch_stride;  // floats per array of the global tile (even)
  unsigned int* queue;
  // optional work list: the queue then runs over list[0 .. *list_count)
  // (the cells that a closed-form pre-pass left to EM)
  const unsigned int* list;
  const unsigned int* list_count;
  int Kmax, max_sweeps;
  int cap;       // cells of more particles (rounded up to even) use the global tile
  int v_f64;     // velocity type: 0 = FP32, 1 = FP64
  int team;      // threads of a team (a power of two, 32 .. 256)
  int nvw;       // partial sums per cell (2, 4 or 8 groups of 32 lanes, see Team)
  int granules;  // shared-memory pool, in units of kPoolGranule bytes
  int share;     // a team's share of the pool
  int patience;  // tries for a tile of up to a share before the cell takes the global one
  double tol;
  uint64_t seed;
};

// float offset o of cell j's global tile: even, and disjoint from its
// neighbours' tiles of N_j rounded up to even length.  Its velocity arrays
// start at o (stride: scratch_stride floats), its normalisers and shifts at
// D * stride + 2 o, its terms and weights at (D + 2) * stride + 2 o.
__host__ __device__ inline int64_t scratch_offset(int64_t off, int64_t j) {
  return off + 2 * j + (off & 1);
}
// floats per array of the global tile (a multiple of 4)
__host__ inline int64_t scratch_stride(int64_t n, int64_t C) { return (n + 2 * C + 2 + 3) & ~(int64_t)3; }

constexpr double kLn2 = 0.69314718055994530942;

template <int D>
struct NConst {  // packed E constants of one component
  static constexpr int NM = D * (D + 1) / 2;
  static constexpr int N = D + NM + 1;  // -mu (D), A (D = 3) or -A^2 (D = 1), b
};

// smallest power of two >= n (n <= 32)
constexpr int pow2_at_least(int n) { return n <= 1 ? 1 : 2 * pow2_at_least((n + 1) / 2); }

// One CTA per SM holds several teams, each fitting one cell at a time.  A
// cell's particles are summed in nvw groups of 32 lanes ("virtual warps"):
// particle pair p belongs to lane p % 32 of group (p / 32) % nvw, a lane adds
// its pairs in order, a group is reduced over its lanes, and the groups are
// added in a fixed tree.  A team of nwt warps takes the groups in turn, so a
// fit does not depend on the team's size.
constexpr int kMaxVW = 8;
constexpr int kPoolGranule = 1024;
constexpr int kPoolWords = 8;
struct EmPool {  // shared-memory pool of the CTA: a bit per granule, set = taken
  unsigned int map[kPoolWords];
  int lock;
};
struct Team {
  int id, tid, nt, lane, wid, nwt, nvw;
  uint32_t buf;  // the warp's buffer of group_sum (offset in shared memory)
  // a named barrier per team (at most 16)
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nt) : "memory");
  }
};

template <int D, typename R>
struct EmCtl {
  static constexpr int NM = D * (D + 1) / 2;
  static constexpr int NS = 1 + D + NM;
  static constexpr int NRED = pow2_at_least(NS);
  // master parameters in whitened coordinates y = (v - mean) / sc
  R u[kMaxK];  // unnormalised weights, omega = u / Z (precision of the M-step)
  R Z;
  double mu[kMaxK][D];
  float mulo[kMaxK][D];  // R = FP32: mean = emu + mulo (emu the high part)
  double S0[NM];  // whitened total covariance (initial covariance of every component)
  // FP32 E-step constants: log2(u f) = b - |A (y - mu)|^2
  float emu[kMaxK][D];
  float eA[kMaxK][NM];  // lower triangle of sqrt(log2e/2) L^{-1}, row-major
  float elc[kMaxK];     // -log2|L| - (D/2) log2(2 pi)
  float eb[kMaxK];      // log2(u) + elc
  // FP64 M-step only: the product of the whitened covariance's pivots
  // (|Sigma_k|), the first-order log-likelihood error (log2 units, per unit
  // responsibility mass) of the FP32 inverse-factor diagonal the E-step
  // uses, and each component's responsibility mass N_k at its last update;
  // with them the convergence test corrects the log-likelihood for the
  // rounding of the FP32 E-step constants
  double pp[kMaxK];
  float corrA[kMaxK], Nkf[kMaxK];
  // the same, packed for the pair loop; slot kMaxK holds the previous
  // component's updated constants
  f32x2 ec[kMaxK + 1][NConst<D>::N];
  double mean[D], sc[D], isc[D];
  double sc2[D];  // sc * sc
  float meanf[D], scf[D];
  double Nd, W, L, logjac, logN;
  double rD;  // 1 / (N - T K / 2) for the current K (FP64 M-step)
  double cov0[D * (D + 1) / 2];  // the cell's weighted covariance (original coordinates)
  // convergence test on the centred log-likelihood (natural log, up to the
  // constant Lbase that c0 removes), assembled in FP64 from FP64 sums
  // of the FP32 per-lane terms: at the stopping point L changes by about
  // tol |L| per sweep, and an FP32 sum of N terms (or an FP32 log of the
  // weights' normaliser times N) errs by a tenth of that
  double Ld, Ldprev, Lbase;
  double sumAH;  // sum of the staged FP32 weights
  float c0;      // centring constant of the log-likelihood sum (log2 units)
  R NdR;
  float redf[kMaxVW][NRED];  // per-group statistics (rows >= nvw stay zero)
  // the prologue's and the final step's per-group FP64 sums; the E-step's
  // per-lane log-likelihood sums (rows >= nvw unused)
  union {
    double redd[kMaxVW][NS + 1];
    float redA[kMaxVW][32];
  };
  double res[NS + 1];
  // final step (centered original coordinates)
  double fw[kMaxK], fmu[kMaxK][D], fS[kMaxK][NM];
  int64_t cell;
  int g0, gn;  // the cell's tile in the pool (g0 < 0: the global tile)
  // the tile: pairs, stride of the velocity arrays (floats), offset in dynamic
  // shared memory or the global arrays (velocities, normalisers, terms)
  int P2, ys, eq;  // eq: every weight of the cell is the same
  uint32_t tile_off;
  float *gY, *gS, *gG;
  f32x2 ah, ah_last;  // eq: the weights of a pair, of the last pair
  int K, Kf, k, sweep, kwork, annih, done, pstate, degenerate, final_pd;
  unsigned int status;
};

// first-fit allocation of gn granules of the pool (one thread); -1 if no run
// is free, or if the lock could not be had within a bounded number of tries
__device__ inline int pool_take(EmPool& pl, int granules, int gn) {
  if (gn > granules) return -1;
  for (int it = 0; atomicCAS(&pl.lock, 0, 1) != 0; ++it)
    if (it >= (1 << 16)) return -1;
  __threadfence_block();
  volatile unsigned int* map = pl.map;
  int run = 0, at = -1;
  for (int g = 0; g < granules; ++g) {
    run = (map[g >> 5] >> (g & 31)) & 1u ? 0 : run + 1;
    if (run == gn) {
      at = g - gn + 1;
      for (int q = at; q <= g; ++q) atomicOr(&pl.map[q >> 5], 1u << (q & 31));
      break;
    }
  }
  __threadfence_block();
  atomicExch(&pl.lock, 0);
  return at;
}
// gives them back (after the team's last access to the tile); the bits are
// the team's own, so no lock is needed
__device__ inline void pool_give(EmPool& pl, int at, int gn) {
  __threadfence_block();
  for (int q = at; q < at + gn; ++q) atomicAnd(&pl.map[q >> 5], ~(1u << (q & 31)));
}

// ---------------------------------------------------------------------------
// small dense helpers (one thread)
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ int tri(int i, int j) {  // upper-triangle index, i <= j
  return D == 1 ? 0 : (i == 0 ? j : (i == 1 ? 2 + j : 5));
}

// Reciprocal and reciprocal square root for the one-thread M-step: an FP32
// hardware seed refined by Newton steps (two in FP64: relative error about
// 1e-16; one in FP32).  They avoid the long division / square-root
// sequences on the M-step's critical path.
__device__ __forceinline__ double rcp_nr(double x) {
  if (!(fabs(x) > 1e-30 && fabs(x) < 1e30)) return 1.0 / x;  // outside the FP32 seed's range
  double r = (double)rcp_approx((float)x);
  r = r * (2.0 - x * r);
  return r * (2.0 - x * r);
}
__device__ __forceinline__ float rcp_nr(float x) {
  const float r = rcp_approx(x);
  return r * (2.0f - x * r);
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ double rsqrt_nr(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / sqrt(x);  // outside the FP32 seed's range
  double y = (double)rsqrt_approx((float)x);
  y = y * (1.5 - 0.5 * x * y * y);
  return y * (1.5 - 0.5 * x * y * y);
}
__device__ __forceinline__ float rsqrt_nr(float x) {
  const float y = rsqrt_approx(x);
  return y * (1.5f - 0.5f * x * y * y);
}

// Cholesky of the upper-triangle S (precision R); returns false if a pivot
// is not positive or, measured in the original coordinates (pivots scale by
// sc_i^2), falls under rel * sum_d (Sigma_dd + mu_d^2) (rel = 1e-13: the
// covariance floor).  Lc[i][i] holds the pivot's square root and ri[i] its
// reciprocal.
template <int D, typename R, typename M>
__device__ bool chol_whitened(const R* S, const R* mu, const M* mean, const M* sc,
                              R (&Lc)[3][3], R (&ri)[3], double rel = 1e-13) {
  R scale2 = 0;
  for (int d = 0; d < D; ++d) {
    const R m = (R)mean[d] + (R)sc[d] * mu[d];
    scale2 += (R)(sc[d] * sc[d]) * S[tri<D>(d, d)] + m * m;
  }
  const R fl = (R)rel * scale2;
  for (int i = 0; i < D; ++i)
    for (int j = 0; j <= i; ++j) {
      R s = S[tri<D>(j, i)];
      for (int m = 0; m < j; ++m) s -= Lc[i][m] * Lc[j][m];
      if (i == j) {
        if (!(s * (R)(sc[i] * sc[i]) > fl) || !(s < (R)(sizeof(R) == 8 ? 1e300 : 1e30))) return false;
        ri[i] = rsqrt_nr(s);
        Lc[i][i] = s * ri[i];
      } else {
        Lc[i][j] = s * ri[j];
      }
    }
  return true;
}
template <int D, typename R, typename M>
__device__ bool chol_whitened(const R* S, const R* mu, const M* mean, const M* sc,
                              R (&Lc)[3][3]) {
  R ri[3];
  return chol_whitened<D, R, M>(S, mu, mean, sc, Lc, ri);
}

// E-step constants of a component from its Cholesky factor (ri: reciprocal
// diagonal)
template <int D, typename R>
__device__ void make_econst(const R (&Lc)[3][3], const R (&ri)[3], float* eA, float& elc) {
  const float c = 0.84932180028801904272f;  // sqrt(log2(e) / 2)
  if (D == 1) {
    eA[0] = c * (float)ri[0];
    elc = -lg2((float)Lc[0][0]) - 0.5f * 2.6514961294723187f;  // log2(2 pi) / 2
  } else {
    const R i00 = ri[0], i11 = ri[1], i22 = ri[2];
    const R i10 = -Lc[1][0] * i00 * i11;
    const R i21 = -Lc[2][1] * i11 * i22;
    const R i20 = -(Lc[2][0] * i00 + Lc[2][1] * i10) * i22;
    eA[0] = c * (float)i00;
    eA[1] = c * (float)i10;
    eA[2] = c * (float)i11;
    eA[3] = c * (float)i20;
    eA[4] = c * (float)i21;
    eA[5] = c * (float)i22;
    elc = -lg2((float)Lc[0][0]) - lg2((float)Lc[1][1]) - lg2((float)Lc[2][2]) -
          1.5f * 2.6514961294723187f;
  }
}

// packed copy of scalar E constants
template <int D>
__device__ __forceinline__ void pack_econst(const float* mu, const float* A, float b, f32x2* out) {
  constexpr int NM = D * (D + 1) / 2;
  for (int x = 0; x < D; ++x) out[x] = bc2(-mu[x]);
  if (D == 1)
    out[1] = bc2(-A[0] * A[0]);
  else
    for (int q = 0; q < NM; ++q) out[D + q] = bc2(A[q]);
  out[D + NM] = bc2(b);
}

// log2(u_k f_k(y)) (scalar), with d = y - mu returned
template <int D>
__device__ __forceinline__ float lg_eval(const float* mu, const float* A, float b, const float* y,
                                         float* d) {
  if (D == 1) {
    d[0] = y[0] - mu[0];
    const float t0 = A[0] * d[0];
    return fmaf(-t0, t0, b);
  } else {
    d[0] = y[0] - mu[0];
    d[1] = y[1] - mu[1];
    d[2] = y[2] - mu[2];
    const float t0 = A[0] * d[0];
    const float t1 = fmaf(A[1], d[0], A[2] * d[1]);
    const float t2 = fmaf(A[3], d[0], fmaf(A[4], d[1], A[5] * d[2]));
    return b - fmaf(t0, t0, fmaf(t1, t1, t2 * t2));
  }
}

// the same for a pair of particles (packed constants)
template <int D>
__device__ __forceinline__ f32x2 lg_eval2(const f32x2* e, const f32x2* y, f32x2* d) {
  constexpr int NM = D * (D + 1) / 2;
  if (D == 1) {
    d[0] = add2(y[0], e[0]);
    return fma2(e[1], mul2(d[0], d[0]), e[2]);
  } else {
    d[0] = add2(y[0], e[0]);
    d[1] = add2(y[1], e[1]);
    d[2] = add2(y[2], e[2]);
    const f32x2 t0 = mul2(e[3], d[0]);
    const f32x2 t1 = fma2(e[4], d[0], mul2(e[5], d[1]));
    const f32x2 t2 = fma2(e[6], d[0], fma2(e[7], d[1], mul2(e[8], d[2])));
    const f32x2 q = fma2(t0, t0, fma2(t1, t1, mul2(t2, t2)));
    return fma2(q, bc2(-1.0f), e[D + NM]);
  }
}

// group vw's warp totals of NV per-lane FP64 values into c.redd[vw]
template <int D, int NV, typename R>
__device__ __forceinline__ void group_sum_d(EmCtl<D, R>& c, int vw, int lane, double (&v)[NV]) {
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) c.redd[vw][i] = v[i];
}
// then the sums over the groups (NV <= NS + 1) in c.res
template <int D, int NV, typename R>
__device__ __forceinline__ void team_sum_d(EmCtl<D, R>& c, const Team& T) {
  T.sync();
  if (T.tid < NV) {
    double s = 0.0;
    for (int q = 0; q < T.nvw; ++q) s += c.redd[q][T.tid];
    c.res[T.tid] = s;
  }
  T.sync();
}

// Warp sum of NP values (NP a power of two <= 32) by recursive halving: at
// each level a lane keeps half of its values, sends the other half to its
// partner and adds what it receives, so NP values cost NP - 1 + 5 - log2(NP)
// shuffles instead of 5 NP.  On return v[0] of every lane holds the warp
// total of value warp_rs_index<NP>(lane).
template <int NP>
__device__ __forceinline__ void warp_rs(float (&v)[NP], int lane) {
  constexpr int LV = NP == 1 ? 0 : (NP == 2 ? 1 : (NP == 4 ? 2 : (NP == 8 ? 3 : (NP == 16 ? 4 : 5))));
#pragma unroll
  for (int lv = 0; lv < LV; ++lv) {
    const int h = NP >> (lv + 1), b = 16 >> lv;
    const bool up = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = up ? v[i] : v[i + h];
      const float keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, b);
    }
  }
#pragma unroll
  for (int b = 16 >> LV; b >= 1; b >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], b);
}

// warp sums of NP doubles by recursive halving (the FP64 form of warp_rs):
// lane l ends with the total of value warp_rs_index<NP>(l) in v[0]
template <int NP>
__device__ __forceinline__ void warp_rs_d(double (&v)[NP], int lane) {
  constexpr int LV = NP == 1 ? 0 : (NP == 2 ? 1 : (NP == 4 ? 2 : (NP == 8 ? 3 : (NP == 16 ? 4 : 5))));
#pragma unroll
  for (int lv = 0; lv < LV; ++lv) {
    const int h2 = NP >> (lv + 1), b = 16 >> lv;
    const bool up = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < h2; ++i) {
      const double send = up ? v[i] : v[i + h2];
      const double keep = up ? v[i + h2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, b);
    }
  }
#pragma unroll
  for (int b = 16 >> LV; b >= 1; b >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], b);
}

// group totals of NV per-lane values into red[q] (lanes added in the order
// of warp_rs's tree: lane distance 16, 8, 4, 2, 1).  Up to 4 values by
// recursive halving; more go through the warp's buffer of kRedRow floats per
// value, where a lane adds half of a value's 32 addends (the even or the odd
// lanes, in the same tree) from four 16-byte loads: 31 instructions instead
// of about 75 for ten values, and 110 cycles instead of 230.
constexpr int kRedRow = 36;  // 32 addends, rows offset by 4 banks
template <int NV, int NP>
__device__ __forceinline__ void group_sum(const float (&v)[NV], float (&red)[NP], int lane, float* buf) {
  if constexpr (NV <= 4) {
    float t[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) t[q] = q < NV ? v[q] : 0.0f;
    warp_rs<NP>(t, lane);
    if ((lane & (32 / NP - 1)) == 0) {
      const int q = warp_rs_index<NP>(lane);
      if (q < NV) red[q] = t[0];
    }
  } else {
    static_assert(NV <= 16, "a lane per value and half");
    const int pos = (lane & 1) * 16 + (lane >> 1), q = lane & 15;
#pragma unroll
    for (int i = 0; i < NV; ++i) buf[i * kRedRow + pos] = v[i];
    __syncwarp();
    const float4* h = reinterpret_cast<const float4*>(buf + (q < NV ? q : 0) * kRedRow + (lane >> 4) * 16);
    const float4 a = h[0], b = h[1], c = h[2], d = h[3];
    const float x = (a.x + c.x) + (b.x + d.x), y = (a.y + c.y) + (b.y + d.y);
    const float z = (a.z + c.z) + (b.z + d.z), w = (a.w + c.w) + (b.w + d.w);
    float t = (x + z) + (y + w);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if (lane < NV) red[lane] = t;
    __syncwarp();
  }
}

// Conversions and a reciprocal of the M-step on the integer pipe: the same
// values as the hardware conversions give, at a shorter latency (an FP64
// operation takes 64 cycles, a hardware conversion about 60; these 20 to 30)
// and off the FP64 pipe.
// FP32 -> FP64 for |f| < 2^104 (the scaling by 2^24 makes subnormals normal)
__device__ __forceinline__ double f2d_t(float f) {
  const uint32_t u = __float_as_uint(f * 16777216.0f), m = u & 0x7FFFFFFFu;
  const uint32_t hi = m == 0u ? 0u : (m >> 3) + 0x36800000u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
// rcp_nr out of line: the operands rcp_nr_q leaves out
static __device__ __noinline__ double rcp_nr_slow(double x) { return rcp_nr(x); }
// rcp_nr for a positive x (a negative or NaN x gives no useful value): the
// FP32 rounding of x, its approximate reciprocal and the conversion back
// from the bit patterns
__device__ __forceinline__ double rcp_nr_q(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  // well inside the FP32 seed's range, else rcp_nr with its own test
  if (hi - 0x39D00000u >= 0x0C500000u) return rcp_nr_slow(x);
  const uint32_t k = __funnelshift_l(lo, hi - 0x38000000u, 3);
  const uint32_t up = ((lo << 3) | (k & 1u)) > 0x80000000u ? 1u : 0u;  // nearest, ties to even
  const uint32_t u = __float_as_uint(rcp_approx(__uint_as_float(k + up)));
  double r = __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
  r = r * (2.0 - x * r);
  return r * (2.0 - x * r);
}
__device__ __forceinline__ double shfl_d(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }

// one component (thread 0): fw, fmu, fS of the final mixture = the sample
// moments; L = eq. (lnL-GM) in closed form: -(N/2)(D ln 2 pi + ln|Sigma| +
// D) - (T/2) ln N (d = T parameters, ln omega = 0); the covariance passed
// the floor in the prologue
template <int D, typename R>
__device__ void k1_closed_form(EmCtl<D, R>& c) {
  constexpr int NM = D * (D + 1) / 2;
  constexpr int T = D * (D + 3) / 2;
  c.K = 1;
  c.fw[0] = 1.0;
  for (int d = 0; d < D; ++d) c.fmu[0][d] = 0.0;
  for (int i = 0; i < NM; ++i) c.fS[0][i] = c.cov0[i];
  double L2[3][3] = {{0}}, logdet = 0.0;
  for (int x = 0; x < D; ++x)
    for (int y = 0; y <= x; ++y) {
      double sv = c.cov0[tri<D>(y, x)];
      for (int m = 0; m < y; ++m) sv -= L2[x][m] * L2[y][m];
      if (x == y) {
        L2[x][x] = sqrt(sv);
        logdet += 2.0 * log(L2[x][x]);
      } else {
        L2[x][y] = sv / L2[y][y];
      }
    }
  c.L = -0.5 * c.Nd * ((double)D * 1.8378770664093454836 + logdet + (double)D) - 0.5 * (double)T * c.logN;
  c.final_pd = 1;
}

// the cell's outputs (thread 0 writes, then a barrier)
template <int D, typename R>
__device__ __forceinline__ void write_cell(const EmParams& a, EmCtl<D, R>& c, const Team& T, int64_t j,
                                           double* prm_out) {
  constexpr int NM = D * (D + 1) / 2;
  constexpr int P = 1 + D + NM;
  if (T.tid == 0) {
    const int Kf = c.K;
    for (int k = 0; k < Kf; ++k) {
      double* r = prm_out + (size_t)k * P;
      r[0] = c.fw[k];
      for (int d = 0; d < D; ++d) r[1 + d] = c.mean[d] + c.fmu[k][d];
      for (int q = 0; q < NM; ++q) r[1 + D + q] = c.fS[k][q];
    }
    for (int i = Kf * P; i < a.Kmax * P; ++i) prm_out[i] = 0.0;
    a.K_out[j] = Kf;
    a.W_out[j] = c.W;
    a.lnL_out[j] = c.final_pd ? c.L : 0.0;
    if (a.sweeps_out) a.sweeps_out[j] = c.sweep;
    if (a.kwork_out) a.kwork_out[j] = c.kwork;
    a.status_out[j] = c.status;
  }
  T.sync();
}

// velocity element i in FP64
__device__ __forceinline__ double load_v(const EmParams& a, int64_t i) {
  return a.v_f64 ? static_cast<const double*>(a.v)[i] : to_f64(static_cast<const float*>(a.v)[i]);
}

// ---------------------------------------------------------------------------
// the particle passes
// ---------------------------------------------------------------------------
// The passes and the M-step are functions of their own: inlined together,
// twice (shared and global tile), their live ranges spilled.  They take the
// control block by its offset in dynamic shared memory, so that accesses to
// it (and to a shared tile) stay shared-memory instructions.
extern __shared__ __align__(16) unsigned char em_smem[];
template <int D, typename R>
__device__ __forceinline__ EmCtl<D, R>& em_ctl(uint32_t off) {
  return *reinterpret_cast<EmCtl<D, R>*>(em_smem + off);
}
// what a pass works on: the cell's tile (pairs) and the team
template <int D, typename R, bool kGlobal>
struct PassCtx {
  // The global tile of a 3V cell keeps a pair's term and weights in a record of
  // 16 bytes {term (2), weights (2)}: one load instead of two and no branch on
  // eq.  24 sweeps over 200 weighted cells of 20000 particles 17.1 -> 13.9 ms, 400 of
  // 10000 12.0 -> 11.2.  (In 1V the separate arrays are faster: 14000 particles 3.6
  // ms with one weight and 3.8 with a weight array, against 4.1.)
  static constexpr bool kRec = kGlobal && D == 3;
  EmCtl<D, R>* c;
  Team T;
  const f32x2 *Y2, *W2;  // velocities, weights
  ulonglong2* SM4;       // a record per pair: {s_p (2), -m_p (2)}
  f32x2* G2;             // the current component's term
  int ys2, P2;
  bool eq;  // one weight for the whole cell: no weight array
  __device__ __forceinline__ f32x2 weight(int pp) const {
    if (kRec) return G2[2 * pp + 1];
    return eq ? (pp == P2 - 1 ? c->ah_last : c->ah) : W2[pp];
  }
  __device__ __forceinline__ void put_term(int pp, f32x2 g) const { G2[kRec ? 2 * pp : pp] = g; }
};

// adds a pair's statistics: responsibilities gam, offsets d = y - mu
template <int D>
__device__ __forceinline__ void add_stats(f32x2 gam, const f32x2 (&d)[D], f32x2 (&acc)[1 + D + D * (D + 1) / 2]) {
  acc[0] = add2(acc[0], gam);
  int t = 1 + D;
#pragma unroll
  for (int x = 0; x < D; ++x) {
    const f32x2 gd = mul2(gam, d[x]);
    acc[1 + x] = add2(acc[1 + x], gd);
#pragma unroll
    for (int yy = x; yy < D; ++yy, ++t) acc[t] = fma2(gd, d[yy], acc[t]);
  }
}
// a group's statistics, reduced over its lanes
template <int D, typename R, bool kGlobal>
__device__ __forceinline__ void put_stats(const PassCtx<D, R, kGlobal>& x, int vw, const f32x2 (&acc)[EmCtl<D, R>::NS]) {
  constexpr int NS = EmCtl<D, R>::NS;
  float v[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    float lo, hi;
    upk2(acc[q], lo, hi);
    v[q] = lo + hi;
  }
  group_sum<NS, EmCtl<D, R>::NRED>(v, x.c->redf[vw], x.T.lane,
                                       reinterpret_cast<float*>(em_smem + x.T.buf));
}

// A pass: Step::run(x, pp, acc, accl) adds a lane's pair pp to acc and accl.
// A pass is bound by its instruction stream, not by a unit: a warp
// issues one instruction in about four cycles, and code beyond the
// instruction cache costs more than it hides.  Two pairs of two groups in
// one step (for independent chains) made the pass's code half as long
// again and the 3V fit slower: 176 against 138 ms for 16384 cells.
template <int D, typename R, bool kGlobal, class Step>
__device__ __forceinline__ void run_groups(const PassCtx<D, R, kGlobal>& x, const Step& st) {
  constexpr int NS = EmCtl<D, R>::NS;
  const int lane = x.T.lane, nvw = x.T.nvw, nv = 32 * nvw, P2 = x.P2;
  for (int vw = x.T.wid; vw < nvw; vw += x.T.nwt) {
    f32x2 acc[NS];
    float accl = 0.0f;
#pragma unroll
    for (int q = 0; q < NS; ++q) acc[q] = 0ull;
    for (int pp = 32 * vw + lane; pp < P2; pp += nv) st.run(x, pp, acc, accl);
    __syncwarp();
    if (st.logs()) x.c->redA[vw][lane] = accl;
    if (st.stats()) {
      if (32 * vw < P2) put_stats<D, R, kGlobal>(x, vw, acc);
      else if (lane < NS) x.c->redf[vw][lane] = 0.0f;  // no pairs
    }
  }
  x.T.sync();
}

// Exact pass: s_p, m_p and eq. (lnL-GM).
// s_p = sum_k 2^(log2(u_k f_k) - m_p).  A fresh pass (the first of a cell,
// or a pair whose sum left [1e-30, 1e30]) takes m_p = max_k log2(u_k f_k),
// so s_p >= 1; otherwise the pair keeps its previous shift m_p, which saves
// the pass for the maximum.  Either way every unchanged component's term
// stays below 1e30 until the next exact pass.  The per-particle
// log-likelihood enters the sum minus a per-cell constant c0 close to its
// mean, which keeps the FP32 partial sums small.  With stats0 the pass also
// yields component 0's E-step statistics (the first step of the next
// sweep).  Per-group partials: c.redf[vw] statistics, c.redA[vw] the lanes'
// centred sums.
template <int D, typename R, bool kGlobal>
struct ExactStep {
  int K;
  float c0;
  bool stats0, fresh;
  __device__ __forceinline__ bool logs() const { return true; }
  __device__ __forceinline__ bool stats() const { return stats0; }
  __device__ __forceinline__ void run(const PassCtx<D, R, kGlobal>& x, int pp, f32x2 (&acc)[EmCtl<D, R>::NS],
                                      float& accl) const {
    f32x2 y[D], d0[D], d[D], nm, sp, G;
    float e0, e1, s0 = 0.0f, s1 = 0.0f;
#pragma unroll
    for (int q = 0; q < D; ++q) y[q] = x.Y2[q * x.ys2 + pp];
    bool slow = fresh;
    if (!fresh) {
      nm = x.SM4[pp].y;
      upk2(add2(lg_eval2<D>(x.c->ec[0], y, d0), nm), e0, e1);
      G = pk2(ex2(e0), ex2(e1));
      sp = G;
      for (int k = 1; k < K; ++k) {
        upk2(add2(lg_eval2<D>(x.c->ec[k], y, d), nm), e0, e1);
        sp = add2(sp, pk2(ex2(e0), ex2(e1)));
      }
      upk2(sp, s0, s1);
      slow = !(s0 > 1e-30f && s0 < 1e30f && s1 > 1e-30f && s1 < 1e30f);
    }
    if (slow) {
      float m0 = -3.0e38f, m1 = -3.0e38f;
      for (int k = 0; k < K; ++k) {
        float l0, l1;
        upk2(lg_eval2<D>(x.c->ec[k], y, d), l0, l1);
        m0 = fmaxf(m0, l0);
        m1 = fmaxf(m1, l1);
      }
      nm = pk2(-m0, -m1);
      upk2(add2(lg_eval2<D>(x.c->ec[0], y, d0), nm), e0, e1);
      G = pk2(ex2(e0), ex2(e1));
      sp = G;
      for (int k = 1; k < K; ++k) {
        upk2(add2(lg_eval2<D>(x.c->ec[k], y, d), nm), e0, e1);
        sp = add2(sp, pk2(ex2(e0), ex2(e1)));
      }
      upk2(sp, s0, s1);
    }
    x.SM4[pp] = make_ulonglong2(sp, nm);
    const f32x2 ah = x.weight(pp);
    float a0, a1, n0, n1;
    upk2(ah, a0, a1);
    upk2(nm, n0, n1);
    accl = fmaf(a0, (-n0 - c0) + lg2(s0), accl);
    accl = fmaf(a1, (-n1 - c0) + lg2(s1), accl);
    if (stats0) {
      x.put_term(pp, G);
      add_stats<D>(mul2(ah, mul2(G, pk2(rcp_approx(s0), rcp_approx(s1)))), d0, acc);
    }
  }
};

// One component step's pass.
// Replaces the previous component's term in s_p (ps = 1: updated, 2:
// removed), evaluates component k and accumulates its statistics; with
// withL it also sums the centred log-likelihood of s_p after the
// replacement (the first step of a sweep without an exact pass: s_p then
// holds every component's current term).  A pair whose s_p dropped more
// than 64-fold in the replacement (cancellation), or with withL left
// [1e-30, 1e30], is recomputed exactly from all components with a fresh
// shift.  Terms are clamped at 2^100 relative to the shift.
template <int D, typename R, bool kGlobal, bool withL, bool kUpd>
struct CompStep {
  int k, ps;  // kUpd: ps = 1
  float c0;
  __device__ __forceinline__ bool logs() const { return withL; }
  __device__ __forceinline__ bool stats() const { return true; }
  __device__ __forceinline__ void run(const PassCtx<D, R, kGlobal>& x, int pp, f32x2 (&acc)[EmCtl<D, R>::NS],
                                      float& accl) const {
    f32x2 y[D], d[D];
#pragma unroll
    for (int q = 0; q < D; ++q) y[q] = x.Y2[q * x.ys2 + pp];
    const ulonglong2 sm = x.SM4[pp];
    f32x2 nm = sm.y, sp;  // -m
    ulonglong2 ga;        // the term and the weights of a record
    if constexpr (PassCtx<D, R, kGlobal>::kRec) ga = reinterpret_cast<const ulonglong2*>(x.G2)[pp];
    else ga.y = x.weight(pp);
    const f32x2 ah = ga.y;
    float so0, so1, sn0, sn1, e0, e1;
    upk2(sm.x, so0, so1);
    if (kUpd) {  // previous component updated: replace its term
      upk2(add2(lg_eval2<D>(x.c->ec[kMaxK], y, d), nm), e0, e1);
      const float gn0 = ex2(fminf(e0, 100.0f)), gn1 = ex2(fminf(e1, 100.0f));
      upk2(add2(fma2(PassCtx<D, R, kGlobal>::kRec ? ga.x : x.G2[pp], bc2(-1.0f), sm.x), pk2(gn0, gn1)), sn0, sn1);
      sn0 = fmaxf(sn0, gn0);
      sn1 = fmaxf(sn1, gn1);
    } else if (ps == 2) {  // previous component removed
      upk2(fma2(PassCtx<D, R, kGlobal>::kRec ? ga.x : x.G2[pp], bc2(-1.0f), sm.x), sn0, sn1);
    } else {
      sn0 = so0;
      sn1 = so1;
    }
    bool fix = (kUpd || ps != 0) && !(sn0 * 64.0f >= so0 && sn1 * 64.0f >= so1);
    if (withL) fix |= !(sn0 > 1e-30f && sn0 < 1e30f && sn1 > 1e-30f && sn1 < 1e30f);
    sp = pk2(sn0, sn1);
    upk2(add2(lg_eval2<D>(x.c->ec[k], y, d), nm), e0, e1);
    f32x2 G = pk2(ex2(fminf(e0, 100.0f)), ex2(fminf(e1, 100.0f)));
    if (fix) {  // exact s_p with the largest term as the shift
      const int K = x.c->K;
      f32x2 dd[D];
      float m0 = -3.0e38f, m1 = -3.0e38f;
      for (int j2 = 0; j2 < K; ++j2) {
        float l0, l1;
        upk2(lg_eval2<D>(x.c->ec[j2], y, dd), l0, l1);
        m0 = fmaxf(m0, l0);
        m1 = fmaxf(m1, l1);
      }
      nm = pk2(-m0, -m1);
      sp = 0ull;
      for (int j2 = 0; j2 < K; ++j2) {
        upk2(add2(lg_eval2<D>(x.c->ec[j2], y, dd), nm), e0, e1);
        const f32x2 t = pk2(ex2(e0), ex2(e1));
        sp = add2(sp, t);
        if (j2 == k) G = t;
      }
    }
    x.put_term(pp, G);
    x.SM4[pp] = make_ulonglong2(sp, nm);
    float s0, s1, g0, g1;
    upk2(sp, s0, s1);
    upk2(G, g0, g1);
    if (withL) {
      float a0, a1, n0, n1;
      upk2(ah, a0, a1);
      upk2(nm, n0, n1);
      accl = fmaf(a0, (-n0 - c0) + lg2(s0), accl);
      accl = fmaf(a1, (-n1 - c0) + lg2(s1), accl);
    }
    const f32x2 rr = pk2(rcp_approx(max3f(s0, g0, 1e-30f)), rcp_approx(max3f(s1, g1, 1e-30f)));
    add_stats<D>(mul2(ah, mul2(G, rr)), d, acc);
  }
};

// the context of a cell's passes; kGlobal: the tile is in global memory
template <int D, typename R, bool kGlobal>
__device__ __forceinline__ PassCtx<D, R, kGlobal> pass_ctx(uint32_t c_off, const Team& T) {
  EmCtl<D, R>& c = em_ctl<D, R>(c_off);
  PassCtx<D, R, kGlobal> x;
  x.c = &c;
  x.T = T;
  x.P2 = c.P2;
  x.ys2 = c.ys >> 1;
  float *Y, *S, *G;
  if constexpr (kGlobal) {
    Y = c.gY;
    S = c.gS;
    G = c.gG;
  } else {
    Y = reinterpret_cast<float*>(em_smem + c.tile_off);
    S = Y + D * c.ys;
    G = Y + (D + 2) * c.ys;
  }
  x.eq = c.eq != 0;
  x.Y2 = reinterpret_cast<const f32x2*>(Y);
  x.SM4 = reinterpret_cast<ulonglong2*>(S);
  x.G2 = reinterpret_cast<f32x2*>(G);
  x.W2 = x.G2 + x.P2;
  return x;
}
template <int D, typename R, bool kGlobal>
__device__ __noinline__ void exact_pass(uint32_t c_off, Team T, bool stats0, bool fresh) {
  const PassCtx<D, R, kGlobal> x = pass_ctx<D, R, kGlobal>(c_off, T);
  run_groups<D, R, kGlobal>(x, ExactStep<D, R, kGlobal>{x.c->K, x.c->c0, stats0, fresh});
}
template <int D, typename R, bool kGlobal, bool withL>
__device__ __forceinline__ void comp_pass_here(uint32_t c_off, const Team& T, int k) {
  const PassCtx<D, R, kGlobal> x = pass_ctx<D, R, kGlobal>(c_off, T);
  const int ps = x.c->pstate;
  const float c0 = withL ? x.c->c0 : 0.0f;
  if (ps == 1) run_groups<D, R, kGlobal>(x, CompStep<D, R, kGlobal, withL, true>{k, ps, c0});
  else
  run_groups<D, R, kGlobal>(x, CompStep<D, R, kGlobal, withL, false>{k, ps, c0});
}

template <int D, typename R, bool kGlobal, bool withL>
__device__ __noinline__ void comp_pass(uint32_t c_off, Team T, int k) {
  comp_pass_here<D, R, kGlobal, withL>(c_off, T, k);
}

// Annihilation of component k (one thread): compaction, eq. (omegak)'s
// renormalisation through Z
template <int D, typename R>
__device__ void remove_comp(EmCtl<D, R>& c, int k) {
  constexpr int NM = D * (D + 1) / 2, NC = NConst<D>::N;
  const double halfT = 0.5 * (D * (D + 3) / 2);
  const int K = c.K;
  c.Z -= c.u[k];
  for (int m = k; m < K - 1; ++m) {
    c.u[m] = c.u[m + 1];
    for (int x = 0; x < D; ++x) {
      c.mu[m][x] = c.mu[m + 1][x];
      c.emu[m][x] = c.emu[m + 1][x];
      c.mulo[m][x] = c.mulo[m + 1][x];
    }
    for (int q = 0; q < NM; ++q) c.eA[m][q] = c.eA[m + 1][q];
    for (int q = 0; q < NC; ++q) c.ec[m][q] = c.ec[m + 1][q];
    c.elc[m] = c.elc[m + 1];
    c.eb[m] = c.eb[m + 1];
    c.pp[m] = c.pp[m + 1];
    c.corrA[m] = c.corrA[m + 1];
    c.Nkf[m] = c.Nkf[m + 1];
  }
  c.K = K - 1;
  if constexpr (sizeof(R) == 8) c.rD = rcp_nr((double)c.NdR - halfT * (K - 1));
  c.annih = 1;
  c.pstate = 2;
}

// M-step for component k (eqs. muk, sigmak, omegak), one thread.
// sv: N_k, the first moments and the second moments about the FP32 mean
// the E-step used.
template <int D, typename R>
__device__ void mstep(EmCtl<D, R>& c, int k, const R (&sv)[2 + D + D * (D + 1) / 2]) {
  constexpr int NM = D * (D + 1) / 2, NC = NConst<D>::N;
  const double halfT = 0.5 * (D * (D + 3) / 2);
  c.kwork++;
  const int K = c.K;
  const R Nk = sv[0];
  bool removed = false;
  if (K > 1 && Nk - (R)halfT <= (R)0) {
    removed = true;
  } else {
    const R rN = rcp_nr(Nk);
    R dl[D], mun[D], Sn[NM];
    // The shift of the mean is added to a ~48-bit master copy (FP64, or
    // hi + lo FP32 when R is FP32), which keeps the sub-ulp part of every
    // update: the FP32 copy then follows the FP64 trajectory instead of
    // stalling when an update is below its resolution.
    double mu64[D];
    float mlo[D];
    for (int x = 0; x < D; ++x) {
      dl[x] = sv[1 + x] * rN;
      if constexpr (sizeof(R) == 4) {
        const float hi = c.emu[k][x];
        const float sm = hi + (float)dl[x];  // two-sum of hi and the shift
        const float bb = sm - hi;
        const float er = (hi - (sm - bb)) + ((float)dl[x] - bb);
        const float lo = c.mulo[k][x] + er;
        const float h2 = sm + lo;  // renormalise
        mlo[x] = lo - (h2 - sm);
        mun[x] = (R)h2;
      } else {
        mu64[x] = c.mu[k][x] + (double)dl[x];
        mun[x] = (R)mu64[x];
      }
    }
    int t = 0;
    for (int x = 0; x < D; ++x)
      for (int yy = x; yy < D; ++yy, ++t) Sn[t] = sv[1 + D + t] * rN - dl[x] * dl[yy];
    R Lc[3][3], ri[3];
    bool pd;
    if constexpr (sizeof(R) == 4)
      pd = chol_whitened<D, R, float>(Sn, mun, c.meanf, c.scf, Lc, ri);
    else
      pd = chol_whitened<D, R, double>(Sn, mun, c.mean, c.sc, Lc, ri);
    if (!pd) {
      c.status |= GM_ST_COV_NOT_PD;
      if (K > 1) {
        removed = true;
      } else {
        c.pstate = 0;  // a lone component keeps its parameters
        c.k = k + 1;
      }
    } else {
      // eq. (omegak), then the renormalisation of step 3 through Z
      const R wn = (K == 1) ? (R)1 : (Nk - (R)halfT) * rcp_nr(c.NdR - (R)halfT * (R)K);
      const R un = wn * c.Z;
      c.Z = c.Z - c.u[k] + un;
      c.u[k] = un;
      float eA[NM], elc;
      make_econst<D, R>(Lc, ri, eA, elc);
      for (int x = 0; x < D; ++x) {
        if constexpr (sizeof(R) == 4)
          c.mulo[k][x] = mlo[x];
        else
          c.mu[k][x] = mu64[x];
        c.emu[k][x] = (float)mun[x];
      }
      for (int q = 0; q < NM; ++q) c.eA[k][q] = eA[q];
      c.elc[k] = elc;
      const float eb = lg2((float)un) + elc;
      c.eb[k] = eb;
      float emu[D];
      for (int x = 0; x < D; ++x) emu[x] = (float)mun[x];
      f32x2 ec[NC];
      pack_econst<D>(emu, eA, eb, ec);
      for (int q = 0; q < NC; ++q) {
        c.ec[k][q] = ec[q];
        c.ec[kMaxK][q] = ec[q];
      }
      c.pstate = 1;
      c.k = k + 1;
    }
  }
  if (removed) remove_comp<D, R>(c, k);
}

// The same M-step in FP64 by the team's first warp.
// What bounds it is the chain of dependent FP64 operations (64 cycles each;
// the pipe, shared by the SM's teams, takes one warp instruction in 19
// cycles however few lanes are active): the group sums, three reciprocals,
// the covariance and its factor.  The chain runs the same on every lane,
// without shuffles or selects between its steps; what is off it -- the
// group sums, S_t / N_k, the floor test's terms, the conversions to FP32,
// the correction's terms -- runs lane-parallel, and the reciprocals' seeds
// are converted on the integer pipe.  There is no branch before the results
// are known, so the floor test and the E constants overlap.
// D = 3: 54 FP64 instructions.
// Lane t < NS holds the statistic S_t (reduce_stats).
// The covariance about the new mean is factored as L~ diag(p) L~^T
// (pivots p_i = the squared Cholesky diagonal); the FP32 E-step
// constants are then c diag(p)^-1/2 L~^-1 with c = sqrt(log2(e) / 2) and
// eb = log2(u) - log2|L| - (D/2) log2(2 pi) (FP32 logarithms: their error
// is what the convergence test corrects for).  The floor test is
// chol_whitened's: p_i sc_i^2 > 1e-13 sum_d (sc_d^2 S_dd + m_d^2) and
// p_i < 1e300.  With gate the team waits for the convergence test, which
// another warp runs meanwhile, and nothing is stored if the cell is done.
template <int D, typename R>
__device__ __forceinline__ double reduce_stats(const EmCtl<D, R>& c, int lane) {
  constexpr int NS = EmCtl<D, R>::NS;
  if constexpr (D == 3) {
    const int q = lane & 15, g = lane >> 4;
    double s = 0.0;
    if (q < NS)
      s = (f2d_t(c.redf[g][q]) + f2d_t(c.redf[g + 4][q])) + (f2d_t(c.redf[g + 2][q]) + f2d_t(c.redf[g + 6][q]));
    return s + __shfl_xor_sync(0xffffffffu, s, 16);
  } else {
    const int q = lane & 7, g = lane >> 3;
    double s = 0.0;
    if (q < NS) s = f2d_t(c.redf[g][q]) + f2d_t(c.redf[g + 4][q]);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s + __shfl_xor_sync(0xffffffffu, s, 8);
  }
}
// Lane roles.  A value chosen by lane goes through selp in inline PTX and
// lane tables in a constant's nibbles: written as conditions on the lane
// number the compiler threads them into a branch per role and runs the M-step
// once for each (5400 cycles a step for D = 3 instead of 2900).
// a on the lanes of kSet (bit = 1 << role), else b
template <uint32_t kSet>
__device__ __forceinline__ double lane_sel(uint32_t bit, double a, double b) {
  double r;
  asm("{\n .reg .pred p;\n .reg .b32 t;\n and.b32 t, %3, %4;\n setp.ne.u32 p, t, 0;\n selp.f64 %0, %1, %2, p;\n}"
      : "=d"(r)
      : "d"(a), "d"(b), "r"(bit), "n"(kSet));
  return r;
}
template <uint32_t kSet>
__device__ __forceinline__ float lane_sel(uint32_t bit, float a, float b) {
  float r;
  asm("{\n .reg .pred p;\n .reg .b32 t;\n and.b32 t, %3, %4;\n setp.ne.u32 p, t, 0;\n selp.f32 %0, %1, %2, p;\n}"
      : "=f"(r)
      : "f"(a), "f"(b), "r"(bit), "n"(kSet));
  return r;
}
// nibble q of a table
__device__ __forceinline__ int lane_tab(uint64_t tab, int q) { return (int)(tab >> (4 * q)) & 15; }

template <int D, typename R>
__device__ __noinline__ void mstep64(uint32_t c_off, int k, Team TM, bool gate) {
  constexpr int NM = D * (D + 1) / 2, NS = 1 + D + NM, NC = NConst<D>::N;
  const double halfT = 0.5 * (D * (D + 3) / 2);
  const int lane = TM.lane;
  EmCtl<D, R>& c = em_ctl<D, R>(c_off);
  const double S = reduce_stats<D, R>(c, lane);
  const int K = c.K;
  const double Zold = (double)c.Z, uold = (double)c.u[k];
  const double kBig = 1e300;
  const double Nk = shfl_d(S, 0);
  const double nkh = Nk - halfT;
  const double rN = rcp_nr_q(Nk);
  // eq. (omegak), then the renormalisation of step 3 through Z
  const double un = (K == 1 ? 1.0 : nkh * c.rD) * Zold;
  const double Zn = (Zold - uold) + un;
  const bool drop = K > 1 && nkh <= 0.0;
  const float cc = 0.84932180028801904272f;  // sqrt(log2(e) / 2)
  float F, A, uf, ppf;
  double caf, pp, mv;
  int bad;
  if constexpr (D == 1) {
    const double S1 = shfl_d(S, 1), S2 = shfl_d(S, 2);
    const double dl = S1 * rN;
    pp = fma(-dl, dl, S2 * rN);  // the new variance
    mv = c.mu[k][0] + dl;
    ppf = (float)pp;
    F = (float)mv;
    uf = (float)un;
    A = cc * rsqrt_nr(ppf);
    // the packed constant is -A^2 (one FP32 product)
    caf = fma(f2d_t(A * A), pp, -0.72134752044448170368);
    const double sc2 = c.sc2[0], md = fma(c.sc[0], mv, c.mean[0]);
    const double fl = 1e-13 * fma(sc2, pp, md * md);
    bad = (pp * sc2 > fl ? 0 : 1) | (__double_as_longlong(pp) < __double_as_longlong(kBig) ? 0 : 1);
  } else {
    const int q = lane & 15;
    const uint32_t bit = 1u << q;
    constexpr uint32_t kMean = 14u;  // lanes 1-3: a coordinate each
    const int x = lane_tab(0x2100u, q);
    const double t = S * rN;  // lanes 1-3: the mean's shift; 4-9: S_t / N_k
    mv = c.mu[k][x] + t;      // lanes 1-3: the new mean
    const double sc2x = c.sc2[x], md = fma(c.sc[x], mv, c.mean[x]);  // in original coordinates
    const double md2 = md * md;
    if (lane < NS) c.res[lane] = t;
    __syncwarp();
    const double d0 = c.res[1], d1 = c.res[2], d2 = c.res[3];
    // covariance about the new mean, L~ diag(p) L~^T
    const double p0 = fma(-d0, d0, c.res[4]);
    const double S01 = fma(-d0, d1, c.res[5]), S02 = fma(-d0, d2, c.res[6]);
    const double S11 = fma(-d1, d1, c.res[7]), S12 = fma(-d1, d2, c.res[8]), S22 = fma(-d2, d2, c.res[9]);
    const double r0 = rcp_nr_q(p0);
    const double term = fma(sc2x, lane_sel<2u>(bit, p0, lane_sel<4u>(bit, S11, S22)), md2);
    const double fl = 1e-13 * ((shfl_d(term, 1) + shfl_d(term, 2)) + shfl_d(term, 3));
    // FP32 values by lane: 0 u; 1-3 the pivots; 4, 7, 9 the means; 5 -l10;
    // 6 l10 l21 - l20; 8 -l21; 10 the pivots' product
    double X = lane_sel<1u>(bit, un, shfl_d(mv, lane_tab(0x3020010000ull, q)));
    X = lane_sel<2u>(bit, p0, X);
    const double l10 = S01 * r0, l20 = S02 * r0;
    const double p1 = fma(-l10, S01, S11), e12 = fma(-l20, S01, S12), t22 = fma(-l20, S02, S22);
    const double r1 = rcp_nr_q(p1);
    X = lane_sel<1u << 5>(bit, -l10, X);
    X = lane_sel<4u>(bit, p1, X);
    const double l21 = e12 * r1, p01 = p0 * p1;
    const double p2 = fma(-l21, e12, t22), x20 = fma(l10, l21, -l20);
    X = lane_sel<1u << 8>(bit, -l21, X);
    X = lane_sel<1u << 6>(bit, x20, X);
    X = lane_sel<8u>(bit, p2, X);
    pp = p01 * p2;
    X = lane_sel<1u << 10>(bit, pp, X);
    F = (float)X;
    const double px = lane_sel<2u>(bit, p0, lane_sel<4u>(bit, p1, p2));
    bad = ((px * sc2x > fl ? 0 : 1) | (__double_as_longlong(px) < __double_as_longlong(kBig) ? 0 : 1)) &
          (int)(kMean >> q) & 1;
    uf = __shfl_sync(0xffffffffu, F, 0);
    ppf = __shfl_sync(0xffffffffu, F, 10);
    const float rr = rsqrt_nr(F);  // lanes 1-3: p_i^-1/2
    // factor entry q - 4 (row-major lower triangle) on lane q; 4, 6, 9 the diagonal
    const float ri = __shfl_sync(0xffffffffu, rr, lane_tab(0x3332210000ull, q));
    const float off = __shfl_sync(0xffffffffu, F, lane_tab(0x860500000ull, q));
    A = (cc * lane_sel<(1u << 4) | (1u << 6) | (1u << 9)>(bit, 1.0f, off)) * ri;
    const double Ad = f2d_t(A);
    const double ct = fma(Ad * Ad, lane_sel<1u << 4>(bit, p0, lane_sel<1u << 6>(bit, p1, p2)),
                          -0.72134752044448170368);
    caf = (shfl_d(ct, 4) + shfl_d(ct, 6)) + shfl_d(ct, 9);
  }
  // eb = log2(u) - (1/2) log2(prod p) - (D/2) log2(2 pi) (FP32); caf: the
  // first-order log-likelihood error of the FP32 inverse factor's diagonal:
  // the quadratic form's error summed over the component's
  // responsibilities is N_k sum_i (A_ii^2 p_i - c^2), A_ii as used
  const float lu = lg2(uf);
  const float eb = lu - 0.5f * lg2(ppf) - (float)D * 1.3257480647361593f;
  const float caff = (float)caf, Nkf = (float)Nk;
  const bool not_pd = __any_sync(0xffffffffu, bad);
  if (gate) {
    TM.sync();
    if (c.done) return;
  }
  if (lane == 0) c.kwork++;
  if (drop || not_pd) {
    if (lane == 0) {
      if (!drop) c.status |= GM_ST_COV_NOT_PD;
      if (K > 1) {
        remove_comp<D, R>(c, k);
      } else {
        c.pstate = 0;  // a lone component keeps its parameters
        c.k = k + 1;
      }
    }
    __syncwarp();
    return;
  }
  if constexpr (D == 1) {
    if (lane == 1) {
      c.mu[k][0] = mv;
      c.emu[k][0] = F;
      c.ec[k][0] = bc2(-F);
      c.ec[kMaxK][0] = bc2(-F);
    }
    if (lane == 2) {
      c.eA[k][0] = A;
      c.ec[k][1] = bc2(-A * A);
      c.ec[kMaxK][1] = bc2(-A * A);
    }
  } else {
    if (lane >= 1 && lane <= 3) c.mu[k][lane - 1] = mv;
    if (lane == 4 || lane == 7 || lane == 9) {
      const int d = (lane - 4) >> 1;  // 0, 1, 2
      c.emu[k][d] = F;
      c.ec[k][d] = bc2(-F);
      c.ec[kMaxK][d] = bc2(-F);
    }
    if (lane >= 4 && lane < 10) {
      c.eA[k][lane - 4] = A;
      c.ec[k][lane - 1] = bc2(A);
      c.ec[kMaxK][lane - 1] = bc2(A);
    }
  }
  if (lane == 10) {
    c.pp[k] = pp;
    c.corrA[k] = caff;
    c.Nkf[k] = Nkf;
  }
  if (lane == 0) {
    c.Z = (R)Zn;
    c.u[k] = (R)un;
    c.elc[k] = eb - lu;
    c.eb[k] = eb;
    c.ec[k][NC - 1] = bc2(eb);
    c.ec[kMaxK][NC - 1] = bc2(eb);
    c.pstate = 1;
    c.k = k + 1;
  }
  __syncwarp();
}

// the statistics' sums over the groups for the FP32 M-step (R = FP32),
// returned in sv by every lane
template <int D, typename R>
__device__ __forceinline__ void gather_stats(const EmCtl<D, R>& c, int lane, R (&sv)[2 + D + D * (D + 1) / 2]) {
  constexpr int NS = EmCtl<D, R>::NS;
  R st[kMaxVW];
#pragma unroll
  for (int q = 0; q < kMaxVW; ++q) st[q] = lane < NS ? (R)c.redf[q][lane] : (R)0;
#pragma unroll
  for (int h = kMaxVW / 2; h >= 1; h >>= 1)
#pragma unroll
    for (int q = 0; q < h; ++q) st[q] += st[q + h];
#pragma unroll
  for (int q = 0; q < NS; ++q) sv[q] = __shfl_sync(0xffffffffu, st[0], q);
  sv[NS] = (R)0;
}

// the first warp after a pass that summed the log-likelihood: eq. (lnL-GM)
// (lane 0, FP64): the centred value c.Ld for the convergence test,
// and with full the value c.L.  The first pass of a cell fixes c0 at the
// mean per-particle term, so that later passes sum small deviations.  The
// weights enter as omega_k = u_k / Z with Z = sum_k u_k summed afresh in
// FP64 (the running Z of the M-step carries its rounding).
template <int D, typename R>
__device__ __noinline__ void finish_exact(uint32_t c_off, bool full, int nvw, int lane) {
  constexpr int T = D * (D + 3) / 2;
  EmCtl<D, R>& c = em_ctl<D, R>(c_off);
  const int K = c.K;
  // the lanes' FP32 sums in FP64 (conversions on the integer pipe), the
  // tree over lanes of every group at once: lane 4 g + r sums group g's
  // lanes r, r + 4, .., then the four lanes of a group
  double lw;
  {
    const int g = lane >> 2, r = lane & 3;
    double e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = g < nvw ? f2d_t(c.redA[g][r + 4 * i]) : 0.0;
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1)
#pragma unroll
      for (int i = 0; i < h; ++i) e[i] += e[i + h];
    lw = e[0];
    lw += __shfl_xor_sync(0xffffffffu, lw, 2);
    lw += __shfl_xor_sync(0xffffffffu, lw, 1);
  }
  const double ud = lane < K ? (double)c.u[lane] : 0.0;
  double Zd = ud;  // lanes K and up hold zeros
  for (int o = K > 4 ? (K > 8 ? 8 : 4) : 2; o > 0; o >>= 1) Zd += __shfl_xor_sync(0xffffffffu, Zd, o);
  Zd = shfl_d(Zd, 0);
  float pen = lane < K ? lg2((float)ud / (float)Zd) : 0.0f;  // log2 omega_k
  pen = warp_sum(pen) * (float)kLn2;
  // FP64 logarithms in one lane-parallel sequence: lane k < K log2 u_k,
  // lane 16 + k log2 |Sigma_k|, lane K (K < 16) log2 Z
  const int kk = lane & 15;
  double arg = 1.0;
  if (lane < K) arg = ud;
  else if (lane >= 16 && kk < K) arg = (sizeof(R) == 8) ? c.pp[kk] : 1.0;
  else if (lane == K) arg = Zd;
  const double lg = log2(arg);
  const double lz = K < 16 ? __shfl_sync(0xffffffffu, lg, K < 16 ? K : 0) : log2(Zd);
  // FP64 M-step, convergence test: the first-order correction
  // sum_k N_k corr_k (log2 units) of the log-likelihood for the rounding of
  // the FP32 E-step constants, corr_k = (eb_k exact - eb_k as used) +
  // corrA_k (see mstep64).  Not for the reported value after the final
  // step (full), whose constants the final step rebuilt.
  float cor = 0.0f;
  if (sizeof(R) == 8 && !full) {
    const double lpp = __shfl_sync(0xffffffffu, lg, (lane + 16) & 31);
    float ck = 0.0f;
    if (lane < K) {
      const double b64 = lg - 0.5 * lpp - D * 1.3257480647361593;
      ck = c.Nkf[lane] * ((float)(b64 - f2d_t(c.eb[lane])) + c.corrA[lane]);
    }
    cor = warp_sum(ck);
  }
  const int dpar = K * (T + 1) - 1;
  double lsum = f2d_t(cor);
#pragma unroll
  for (int q = 0; q < kMaxVW; ++q) lsum += shfl_d(lw, 4 * q);  // zeros from nvw on
  if (lane == 0) {
    lsum -= c.sumAH * lz;
    const double pc = -0.5 * dpar * c.logN - 0.5 * T * (double)pen;
    if (full || c.sweep == 0) {
      const double ls = lsum + (double)c.c0 * c.sumAH;
      c.L = ls * kLn2 - c.Nd * c.logjac + pc;
      if (!full) {
        const float c0n = c.sumAH > 0.0 ? (float)(ls / c.sumAH) : c.c0;
        c.c0 = c0n;
        c.Ld = (ls - (double)c0n * c.sumAH) * kLn2 + pc;
        c.Lbase = (double)c0n * c.sumAH * kLn2 - c.Nd * c.logjac;
      }
    } else {
      c.Ld = kLn2 * lsum + pc;
    }
  }
}

// ---------------------------------------------------------------------------
// one cell, after its moments are known and it is not degenerate.  The
// particle tile (shared or global) holds N rounded up to even particles (a
// zero-weight pad particle), an FP32 value per particle and array, read a
// pair at a time: the whitened velocities Y (array d at Y + d * ys), at S
// 16 bytes per pair with the normalisers and shifts {s_p (2), -m_p (2)}, at
// G the current component's terms, then -- unless the cell has one weight --
// the normalised weights (a 3V cell's global tile: {terms, weights} records at G).
// ---------------------------------------------------------------------------
template <int D, typename R, bool kGlobal>
__device__ __forceinline__ void em_cell_body(const EmParams& a, uint32_t c_off, const Team& TM,
                                             int64_t j, int64_t off, int N, float* Y, int ys,
                                             float* SMT, float* GAT) {
  EmCtl<D, R>& c = em_ctl<D, R>(c_off);
  constexpr bool kRec = PassCtx<D, R, kGlobal>::kRec;
  constexpr int NM = D * (D + 1) / 2;
  constexpr int NS = 1 + D + NM;
  constexpr int T = D * (D + 3) / 2;
  constexpr int P = 1 + D + NM;
  const double halfT = 0.5 * T;
  const int tid = TM.tid, lane = TM.lane, nvw = TM.nvw, nv = 32 * TM.nvw;
  double* prm_out = a.params_out + (size_t)j * a.Kmax * P;
  const int P2 = (N + 1) >> 1;  // particle pairs

  // ---- initialisation --------------------------------------------------
  // A supplied initial mixture (learned initialisation) is used when given:
  // components failing the Cholesky floor are dropped, the count is capped
  // so that N - T K / 2 > 0, and an empty result falls back to the paper's
  // initialisation (Sec. 2.3): Kmax components at random particles.
  if (tid == 0) {
    int K = 0;
    if (a.init_K) {
      const int K0 = a.init_K[j] < a.Kmax ? a.init_K[j] : a.Kmax;
      double wsum = 0.0;
      for (int k = 0; k < K0; ++k) {
        const double* r = a.init_prm + ((size_t)j * a.Kmax + k) * P;
        double mw[D], Sw[NM], Lw[3][3], rw[3];
        for (int d = 0; d < D; ++d) mw[d] = (r[1 + d] - c.mean[d]) * c.isc[d];
        int q = 0;
        for (int x = 0; x < D; ++x)
          for (int yy = x; yy < D; ++yy, ++q) Sw[q] = r[1 + D + q] * c.isc[x] * c.isc[yy];
        if (!(r[0] > 0.0) || !chol_whitened<D, double, double>(Sw, mw, c.mean, c.sc, Lw, rw))
          continue;
        float eA[NM], elc;
        make_econst<D, double>(Lw, rw, eA, elc);
        for (int d = 0; d < D; ++d) {
          c.mu[K][d] = mw[d];
          c.emu[K][d] = (float)mw[d];
          c.mulo[K][d] = (float)(mw[d] - (double)c.emu[K][d]);
        }
        for (int i = 0; i < NM; ++i) c.eA[K][i] = eA[i];
        c.elc[K] = elc;
        c.u[K] = (R)r[0];
        wsum += r[0];
        ++K;
      }
      while (K > 1 && c.Nd - halfT * K <= 0.0) {
        --K;
        wsum -= (double)c.u[K];
      }
      for (int k = 0; k < K; ++k) {
        c.u[k] = (R)((double)c.u[k] / wsum);
        c.eb[k] = lg2((float)c.u[k]) + c.elc[k];
        c.pp[k] = 1.0;
        c.corrA[k] = c.Nkf[k] = 0.0f;
        pack_econst<D>(c.emu[k], c.eA[k], c.eb[k], c.ec[k]);
      }
      c.K = K;
      c.Z = (R)1;
    }
  }
  TM.sync();
  if (tid == 0 && c.K == 0) {
    int K = a.Kmax < N ? a.Kmax : N;
    while (K > 1 && c.Nd - halfT * K <= 0.0) --K;
    int picks[kMaxK];
    int got = 0;
    for (uint32_t t = 0; got < K; ++t) {
      int idx;
      if (t < 100000u) {
        const u32x4 r = philox_draw(a.seed, t, kTagInit, j);
        const double uu = uniform52(r.x, r.y);
        idx = (int)floor(uu * c.Nd);
        if (idx >= N) idx = N - 1;
      } else {
        idx = 0;
        for (;;) {
          bool used = false;
          for (int m = 0; m < got; ++m) used |= (picks[m] == idx);
          if (!used) break;
          ++idx;
        }
      }
      bool dup = false;
      for (int m = 0; m < got; ++m) dup |= (picks[m] == idx);
      if (!dup) picks[got++] = idx;
    }
    c.K = K;
    c.Z = (R)1;
    R Lc[3][3], ri[3];
    R S0[NM], m0[D];
    for (int i = 0; i < NM; ++i) S0[i] = (R)c.S0[i];
    for (int d = 0; d < D; ++d) m0[d] = 0;
    chol_whitened<D, R, double>(S0, m0, c.mean, c.sc, Lc, ri);  // the total covariance passed
    float eA[NM], elc;
    make_econst<D, R>(Lc, ri, eA, elc);
    for (int k = 0; k < K; ++k) {
      c.u[k] = (R)1 / (R)K;
      for (int d = 0; d < D; ++d) {
        c.mu[k][d] = (load_v(a, (int64_t)d * a.n + off + picks[k]) - c.mean[d]) * c.isc[d];
        c.emu[k][d] = (float)c.mu[k][d];
        c.mulo[k][d] = (float)(c.mu[k][d] - (double)c.emu[k][d]);
      }
      for (int i = 0; i < NM; ++i) c.eA[k][i] = eA[i];
      c.elc[k] = elc;
      c.eb[k] = lg2((float)c.u[k]) + elc;
      c.pp[k] = 1.0;
      c.corrA[k] = c.Nkf[k] = 0.0f;
      pack_econst<D>(c.emu[k], c.eA[k], c.eb[k], c.ec[k]);
    }
  }
  TM.sync();
  // ---- one component: the EM's fixed point in closed form ----------------
  // With K = 1 every responsibility is the particle's weight, so one EM step
  // from any start gives the weighted sample mean and covariance (Sec.
  // 2.3.1), and eq. (lnL-GM) is -(N/2)(D ln 2 pi + ln|Sigma| + D) - (T/2) ln N.
  // Reported as one sweep without component E-steps (kwork 0).
  if (c.K == 1) {
    if (tid == 0) {
      c.sweep = 1;
      c.kwork = 0;
      k1_closed_form<D, R>(c);
    }
    TM.sync();
    write_cell<D, R>(a, c, TM, j, prm_out);
    return;
  }
  // ---- stage whitened velocities and normalised weights ------------------
  {
    const double nw = c.Nd / c.W;
    for (int vw = TM.wid; vw < nvw; vw += TM.nwt) {
      double sa[1] = {0.0};
      for (int p = 32 * vw + lane; p < 2 * P2; p += nv) {
        if (p < N) {
#pragma unroll
          for (int d = 0; d < D; ++d)
            Y[d * ys + p] = (float)((load_v(a, (int64_t)d * a.n + off + p) - c.mean[d]) * c.isc[d]);
          const float ah = (float)(a.alpha[off + p] * nw);
          if (kRec) GAT[4 * (p >> 1) + 2 + (p & 1)] = ah;
          else if (!c.eq) GAT[2 * P2 + p] = ah;
          sa[0] += (double)ah;
        } else {  // zero-weight pad particle
#pragma unroll
          for (int d = 0; d < D; ++d) Y[d * ys + p] = 0.0f;
          if (kRec) GAT[4 * (p >> 1) + 2 + (p & 1)] = 0.0f;
          else if (!c.eq) GAT[2 * P2 + p] = 0.0f;
        }
      }
      group_sum_d<D, 1, R>(c, vw, lane, sa);
    }
    team_sum_d<D, 1, R>(c, TM);
    if (tid == 0) {
      if (c.eq) {
        const float ah = (float)(a.alpha[off] * nw);
        c.ah = bc2(ah);
        c.ah_last = pk2(ah, N & 1 ? 0.0f : ah);
      }
      c.sumAH = c.res[0];
      c.c0 = -2.0471975511965976f * D;  // mean log2 density of a standard normal
      c.NdR = (R)c.Nd;
      if constexpr (sizeof(R) == 8) c.rD = rcp_nr(c.Nd - halfT * c.K);
    }
  }
  if (tid == 0) {
    c.sweep = 0;
    c.kwork = 0;
    c.done = 0;
    c.annih = 0;
  }
  TM.sync();

  // ---- sweeps -------------------------------------------------------------
  // Every kExactEvery-th sweep starts with the exact pass (after the weights
  // are normalised); the others start with the first component step, which
  // also yields the log-likelihood of the previous sweep's parameters.
  constexpr int kExactEvery = 8;
  for (;;) {
    if (c.sweep % kExactEvery == 0) {
      if (c.sweep > 0) {
        if (tid < c.K) {
          const R un = c.u[tid] / c.Z;
          c.u[tid] = un;
          c.eb[tid] = lg2((float)un) + c.elc[tid];
          pack_econst<D>(c.emu[tid], c.eA[tid], c.eb[tid], c.ec[tid]);
        }
        TM.sync();
        if (tid == 0) c.Z = (R)1;
        TM.sync();
      }
      exact_pass<D, R, kGlobal>(c_off, TM, true, c.sweep == 0);
    } else {
      comp_pass<D, R, kGlobal, true>(c_off, TM, 0);
    }
    // the convergence test (one warp) beside the first component's M-step
    // (the first warp), whose results wait for it; a team of one warp and
    // the FP32 M-step run them in turn
    const bool beside = sizeof(R) == 8 && TM.nwt > 1;
    if (TM.wid == (beside ? 1 : 0)) {
      finish_exact<D, R>(c_off, false, nvw, lane);
      if (lane == 0) {
        if (c.sweep > 0 && !c.annih && fabs(c.Ld - c.Ldprev) <= a.tol * fabs(c.Ldprev + c.Lbase))
          c.done = 1;
        else if (c.sweep >= a.max_sweeps)
          c.done = 2;
        c.Ldprev = c.Ld;
        if (!c.done) {
          c.sweep = c.sweep + 1;
          c.annih = 0;
          c.k = 0;
          c.pstate = 0;
        }
      }
      __syncwarp();
    }
    if (sizeof(R) == 8) {
      if (TM.wid == 0) {
        if (beside || !c.done) mstep64<D, R>(c_off, 0, TM, beside);
      } else {
        TM.sync();
      }
    } else if (TM.wid == 0 && !c.done) {
      R sv[NS + 1];
      gather_stats<D, R>(c, lane, sv);
      if (lane == 0) mstep<D, R>(c, 0, sv);
    }
    TM.sync();
    if (c.done) break;
    while (c.k < c.K) {
      const int k = c.k;
      // (in place beside the FP32 M-step: a call and its return take 260 cycles,
      // 2 to 5 % of a fit; with the FP64 one the 3V kernel spills more than that)
      if constexpr (sizeof(R) == 4 && !kGlobal) comp_pass_here<D, R, kGlobal, false>(c_off, TM, k);
      else comp_pass<D, R, kGlobal, false>(c_off, TM, k);
      if (tid < 32) {
        if constexpr (sizeof(R) == 8) {
          mstep64<D, R>(c_off, k, TM, false);
        } else {
          R sv[NS + 1];
          gather_stats<D, R>(c, lane, sv);
          if (lane == 0) mstep<D, R>(c, k, sv);
        }
      }
      TM.sync();
    }
  }
  if (tid == 0 && c.done == 2) c.status |= GM_ST_EM_MAXSWEEPS;
  if constexpr (sizeof(R) == 4) {  // FP64 means from the hi + lo pairs
    if (tid < c.K)
      for (int x = 0; x < D; ++x) c.mu[tid][x] = (double)c.emu[tid][x] + (double)c.mulo[tid][x];
    TM.sync();
  }

  // ---- final unpenalised step (Sec. 2.3.1), FP64 ---------------------------
  if (c.K == 1) {  // the final step of one component: the sample moments
    if (tid == 0) k1_closed_form<D, R>(c);
    TM.sync();
    write_cell<D, R>(a, c, TM, j, prm_out);
    return;
  }
  if (tid == 0) c.Kf = 0;
  TM.sync();
  {
    const int K = c.K;
    const double nw = c.Nd / c.W;
    // Normaliser pass: per particle the shift m_p = max_j log2(u_j f_j) and
    // r_p = alpha_p (N / W) / S_p with S_p = sum_j 2^(log2(u_j f_j) - m_p)
    // summed in FP64.  r_p goes over the tile's s_p and m_p arrays (8 bytes per
    // particle) and m_p over its terms; the weights stay for the last exact
    // pass.
    // The whole team shares this pass, so that a team of more warps than the
    // cell has groups idles none; the groups' warps read other warps' particles
    // after the barrier.  The component passes recompute
    // 2^(log2(u_k f_k) - m_p) with the same instructions on the same operands,
    // so sum_k gamma_pk = alpha_p N / W to FP64 rounding.
    double* Rd = reinterpret_cast<double*>(SMT);
    float* Mf = GAT;
    for (int p = tid; p < N; p += TM.nt) {
      float y[D], d[D];
#pragma unroll
      for (int q = 0; q < D; ++q) y[q] = Y[q * ys + p];
      float m = -3.0e38f;
      for (int jj = 0; jj < K; ++jj) m = fmaxf(m, lg_eval<D>(c.emu[jj], c.eA[jj], c.eb[jj], y, d));
      double Ssum = 0.0;
      for (int jj = 0; jj < K; ++jj)
        Ssum += (double)ex2(lg_eval<D>(c.emu[jj], c.eA[jj], c.eb[jj], y, d) - m);
      Rd[p] = a.alpha[off + p] * nw / Ssum;
      Mf[kRec ? 4 * (p >> 1) + (p & 1) : p] = m;
    }
    TM.sync();
    for (int k = 0; k < K; ++k) {
      double ck[D];
#pragma unroll
      for (int q = 0; q < D; ++q) ck[q] = c.mu[k][q] * c.sc[q];
      for (int vw = TM.wid; vw < nvw; vw += TM.nwt) {
      double acc[NS];
#pragma unroll
      for (int q = 0; q < NS; ++q) acc[q] = 0.0;
      for (int p = 32 * vw + lane; p < N; p += nv) {
        float y[D], d[D];
#pragma unroll
        for (int q = 0; q < D; ++q) y[q] = Y[q * ys + p];
        const float m = Mf[kRec ? 4 * (p >> 1) + (p & 1) : p];
        const double gk = (double)ex2(lg_eval<D>(c.emu[k], c.eA[k], c.eb[k], y, d) - m);
        const double gam = Rd[p] * gk;
        double dv[D];
#pragma unroll
        for (int q = 0; q < D; ++q) dv[q] = (load_v(a, (int64_t)q * a.n + off + p) - c.mean[q]) - ck[q];
        acc[0] += gam;
        int t = 1 + D;
#pragma unroll
        for (int x = 0; x < D; ++x) {
          const double gd = gam * dv[x];
          acc[1 + x] += gd;
#pragma unroll
          for (int yy = x; yy < D; ++yy, ++t) acc[t] += gd * dv[yy];
        }
      }
      group_sum_d<D, NS, R>(c, vw, lane, acc);
      }
      team_sum_d<D, NS, R>(c, TM);
      if (tid == 0 && c.res[0] > 0.0) {
        const int f = c.Kf;
        const double n = c.res[0];
        double dl[D];
        for (int x = 0; x < D; ++x) {
          dl[x] = c.res[1 + x] / n;
          c.fmu[f][x] = ck[x] + dl[x];
        }
        int t = 0;
        for (int x = 0; x < D; ++x)
          for (int yy = x; yy < D; ++yy, ++t) c.fS[f][t] = c.res[1 + D + t] / n - dl[x] * dl[yy];
        c.fw[f] = n / c.Nd;
        c.Kf = f + 1;
      }
      TM.sync();
    }
  }
  // ---- final parameters: E constants, Cholesky floor, eq. (lnL-GM) -------
  if (tid == 0) {
    const int Kf = c.Kf;
    int pd = 1;
    double one[D];
    for (int d = 0; d < D; ++d) one[d] = 1.0;
    for (int k = 0; k < Kf; ++k) {
      // floor test in the original coordinates
      double So[NM], mo[D], Lo[3][3];
      for (int q = 0; q < NM; ++q) So[q] = c.fS[k][q];
      for (int d = 0; d < D; ++d) mo[d] = 0.0;
      double meano[D];
      for (int d = 0; d < D; ++d) meano[d] = c.mean[d] + c.fmu[k][d];
      if (!chol_whitened<D, double, double>(So, mo, meano, one, Lo)) pd = 0;
      // whitened copy for the likelihood pass
      double Sw[NM], mw[D], Lw[3][3];
      for (int x = 0; x < D; ++x) {
        mw[x] = c.fmu[k][x] * c.isc[x];
        for (int yy = x; yy < D; ++yy) Sw[tri<D>(x, yy)] = c.fS[k][tri<D>(x, yy)] * c.isc[x] * c.isc[yy];
      }
      double rw[3];
      if (chol_whitened<D, double, double>(Sw, mw, c.mean, c.sc, Lw, rw)) {
        float eA[NM], elc;
        make_econst<D, double>(Lw, rw, eA, elc);
        for (int q = 0; q < NM; ++q) c.eA[k][q] = eA[q];
        c.elc[k] = elc;
      } else {
        pd = 0;
      }
      for (int x = 0; x < D; ++x) c.emu[k][x] = (float)mw[x];
      c.eb[k] = lg2((float)c.fw[k]) + c.elc[k];
      c.u[k] = (R)c.fw[k];
      pack_econst<D>(c.emu[k], c.eA[k], c.eb[k], c.ec[k]);
    }
    if (!pd) c.status |= GM_ST_COV_NOT_PD;
    c.final_pd = pd;
    c.K = Kf;
    c.Z = (R)1;
  }
  TM.sync();
  if (c.final_pd) {
    exact_pass<D, R, kGlobal>(c_off, TM, false, true);
    if (tid < 32) finish_exact<D, R>(c_off, true, nvw, lane);
    TM.sync();
  }
  write_cell<D, R>(a, c, TM, j, prm_out);
}

// ---------------------------------------------------------------------------
// the kernel: work queue, per-cell moments, degenerate cells, dispatch of
// the cell body on the shared or the global tile.  One CTA per SM of up to
// kEmThreads threads, split into teams; dynamic shared
// memory: the pool's map, a control block per team, then the pool.
// ---------------------------------------------------------------------------
constexpr int kEmThreads = 640;  // threads of a CTA, at most (96 registers each)
template <int D, typename R>
__host__ __device__ constexpr size_t em_ctl_bytes() { return (sizeof(EmCtl<D, R>) + 15) & ~(size_t)15; }
__host__ __device__ constexpr int em_buf_bytes(int D) { return D == 1 ? 0 : 10 * kRedRow * (int)sizeof(float); }
// bytes of the shared tile of N particles: D + 4 arrays (D + 3 without weights)
__host__ __device__ constexpr int64_t em_tile_bytes(int D, int64_t N, bool eq) {
  return ((N + 3) & ~(int64_t)3) * (D + (eq ? 3 : 4)) * 4;
}

template <int D, typename R>
__global__ void __launch_bounds__(kEmThreads, 1) em_kernel(EmParams a) {
  constexpr int NM = D * (D + 1) / 2;
  constexpr int P = 1 + D + NM;
  using Ctl = EmCtl<D, R>;
  EmPool& pool = *reinterpret_cast<EmPool*>(em_smem);
  const int teams = (int)blockDim.x / a.team;
  Team TM;
  TM.nt = a.team;
  TM.id = (int)threadIdx.x / a.team;
  TM.tid = (int)threadIdx.x - TM.id * a.team;
  TM.lane = TM.tid & 31;
  TM.wid = TM.tid >> 5;
  TM.nwt = a.team >> 5;
  TM.nvw = a.nvw;
  const uint32_t c_off = 64u + (uint32_t)TM.id * (uint32_t)em_ctl_bytes<D, R>();
  Ctl& c = em_ctl<D, R>(c_off);
  const uint32_t bufs = 64u + (uint32_t)teams * (uint32_t)em_ctl_bytes<D, R>();
  TM.buf = bufs + (threadIdx.x >> 5) * (uint32_t)em_buf_bytes(D);
  const uint32_t arena = bufs + (blockDim.x >> 5) * (uint32_t)em_buf_bytes(D);
  const int tid = TM.tid, lane = TM.lane, nvw = TM.nvw, nv = 32 * TM.nvw;
  if (threadIdx.x < kPoolWords) pool.map[threadIdx.x] = 0u;
  if (threadIdx.x == 0) pool.lock = 0;
  for (int i = tid; i < kMaxVW * Ctl::NRED; i += TM.nt) c.redf[i / Ctl::NRED][i % Ctl::NRED] = 0.0f;
  __syncthreads();

  // the first cells go round the SMs, then the teams draw tickets
  for (int64_t first = (int64_t)TM.id * gridDim.x + blockIdx.x;; first = -1) {
    if (tid == 0) {
      const int64_t t = first >= 0 ? first : (int64_t)teams * gridDim.x + atomicAdd(a.queue, 1u);
      c.cell = a.list ? (t < (int64_t)*a.list_count ? (int64_t)a.list[t] : a.C) : t;
    }
    TM.sync();
    const int64_t j = c.cell;
    if (j >= a.C) break;
    const int64_t off = a.cell_off[j];
    const int N = (int)(a.cell_off[j + 1] - off);
    double* prm_out = a.params_out + (size_t)j * a.Kmax * P;

    // ---- total weight, mean and covariance (FP64, one pass) ----------------
    // sums of alpha, alpha d and alpha d d^T with d = v - s, s the cell's
    // first particle (d is exact in FP64, and s lies within the cell's
    // spread, so mean = s + sum(alpha d) / W and cov = sum(alpha d d^T) / W
    // - (mean - s)(mean - s)^T lose no more than a few ulps to cancellation)
    {
      double sh[D];
#pragma unroll
      for (int d = 0; d < D; ++d) sh[d] = N > 0 ? load_v(a, (int64_t)d * a.n + off) : 0.0;
      // equal weights (bit for bit) need no weight array
      const long long al0 = N > 0 ? __double_as_longlong(a.alpha[off]) : 0;
      bool same = true;
      if (tid == 0) c.eq = 1;
      TM.sync();
      for (int vw = TM.wid; vw < nvw; vw += TM.nwt) {
        double acc[1 + D + NM];
#pragma unroll
        for (int i = 0; i < 1 + D + NM; ++i) acc[i] = 0.0;
        for (int p = 32 * vw + lane; p < N; p += nv) {
          const double al = a.alpha[off + p];
          same &= __double_as_longlong(al) == al0;
          double dv[D];
#pragma unroll
          for (int d = 0; d < D; ++d) dv[d] = load_v(a, (int64_t)d * a.n + off + p) - sh[d];
          acc[0] += al;
          int t = 1 + D;
#pragma unroll
          for (int x = 0; x < D; ++x) {
            const double ad = al * dv[x];
            acc[1 + x] += ad;
#pragma unroll
            for (int y = x; y < D; ++y, ++t) acc[t] = fma(ad, dv[y], acc[t]);
          }
        }
        group_sum_d<D, 1 + D + NM, R>(c, vw, lane, acc);
      }
      if (!same) c.eq = 0;
      team_sum_d<D, 1 + D + NM, R>(c, TM);
      if (tid == 0) {
        c.W = c.res[0];
        c.Nd = (double)N;
        c.status = (N <= 10) ? GM_ST_TOO_FEW : 0u;
        const double rW = 1.0 / c.res[0];
        double dm[D];
        for (int d = 0; d < D; ++d) {
          dm[d] = c.res[1 + d] * rW;
          c.mean[d] = sh[d] + dm[d];
        }
        double cov[NM];
        int t = 0;
        for (int x = 0; x < D; ++x)
          for (int y = x; y < D; ++y, ++t) cov[t] = fma(-dm[x], dm[y], c.res[1 + D + t] * rW);
        c.degenerate = 0;
        if (N == 0 || !(c.W > 0.0)) {
          c.degenerate = 2;  // empty: handled below
        } else {
          // degenerate cell: the total covariance fails the Cholesky floor
          // 1e-13 * sum_d (cov_dd + mean_d^2)
          double scale2 = 0.0;
          for (int d = 0; d < D; ++d) scale2 += cov[tri<D>(d, d)] + c.mean[d] * c.mean[d];
          const double fl = 1e-13 * scale2;
          bool ok = true;
          double L2[3][3] = {{0}};
          for (int x = 0; x < D && ok; ++x)
            for (int y = 0; y <= x && ok; ++y) {
              double sv = cov[tri<D>(y, x)];
              for (int m = 0; m < y; ++m) sv -= L2[x][m] * L2[y][m];
              if (x == y) {
                if (!(sv > fl) || !(sv < 1e300)) ok = false;
                else L2[x][x] = sqrt(sv);
              } else {
                L2[x][y] = sv / L2[y][y];
              }
            }
          c.degenerate = ok ? 0 : 1;
          if (c.degenerate) {
            for (int i = 0; i < NM; ++i) c.fS[0][i] = cov[i];
          } else {
            for (int i = 0; i < NM; ++i) c.cov0[i] = cov[i];
            c.logN = log(c.Nd);
            double prod = 1.0;
            for (int d = 0; d < D; ++d) {
              c.sc[d] = sqrt(cov[tri<D>(d, d)]);
              c.isc[d] = 1.0 / c.sc[d];
              c.sc2[d] = c.sc[d] * c.sc[d];
              prod *= c.sc[d];
              c.meanf[d] = (float)c.mean[d];
              c.scf[d] = (float)c.sc[d];
            }
            c.logjac = log(prod);
            // whitened total covariance (correlation matrix) for the init
            for (int x = 0; x < D; ++x)
              for (int y = x; y < D; ++y)
                c.S0[tri<D>(x, y)] = (x == y) ? 1.0 : cov[tri<D>(x, y)] * c.isc[x] * c.isc[y];
          }
        }
      }
      TM.sync();
    }
    if (c.degenerate == 2) {
      for (int i = tid; i < a.Kmax * P; i += TM.nt) prm_out[i] = 0.0;
      if (tid == 0) {
        a.K_out[j] = 0;
        a.W_out[j] = N == 0 ? 0.0 : c.W;
        a.lnL_out[j] = 0.0;
        if (a.sweeps_out) a.sweeps_out[j] = 0;
        if (a.kwork_out) a.kwork_out[j] = 0;
        a.status_out[j] = N == 0 ? GM_ST_EMPTY : (GM_ST_EMPTY | GM_ST_DEGENERATE);
      }
      TM.sync();
      continue;
    }
    if (c.degenerate) {
      for (int i = tid; i < a.Kmax * P; i += TM.nt) prm_out[i] = 0.0;
      TM.sync();
      if (tid == 0) {
        prm_out[0] = 1.0;
        for (int d = 0; d < D; ++d) prm_out[1 + d] = c.mean[d];
        for (int i = 0; i < NM; ++i) prm_out[1 + D + i] = c.fS[0][i];
        a.K_out[j] = 1;
        a.W_out[j] = c.W;
        a.lnL_out[j] = 0.0;
        if (a.sweeps_out) a.sweeps_out[j] = 0;
        if (a.kwork_out) a.kwork_out[j] = 0;
        a.status_out[j] = c.status | GM_ST_DEGENERATE | GM_ST_COV_NOT_PD;
      }
      TM.sync();
      continue;
    }
    if (tid == 0) {
      c.K = 0;
      const int Np = N + (N & 1);
      c.gn = (int)((em_tile_bytes(D, Np, c.eq != 0) + kPoolGranule - 1) / kPoolGranule);
      c.g0 = -1;
      // A cell within its team's share waits for a hole (the others' cells are
      // of its kind, and free one in a few ms at most); a larger one takes what
      // is free now or works in L2, where it would otherwise wait for the
      // other teams' whole fits.
      if (Np <= a.cap && c.gn <= a.granules) {
        const int tries = c.gn <= a.share ? a.patience : 1;
        for (int it = 0; it < tries && (c.g0 = pool_take(pool, a.granules, c.gn)) < 0; ++it)
          if (it + 1 < tries) __nanosleep(2000);
      }
    }
    TM.sync();
    if (tid == 0) {
      c.P2 = (N + 1) >> 1;
      if (c.g0 >= 0) {
        c.ys = (N + 3) & ~3;
        c.tile_off = arena + (uint32_t)c.g0 * kPoolGranule;
      } else {
        const int64_t o = scratch_offset(off, j), ss = a.scratch_stride;
        c.ys = (int)ss;
        c.gY = a.scratch + o;
        c.gS = a.scratch + D * ss + 2 * o;
        c.gG = a.scratch + (D + 2) * ss + 2 * o;
      }
    }
    TM.sync();
    if (c.g0 >= 0) {
      float* tile = reinterpret_cast<float*>(em_smem + c.tile_off);
      const int ys = c.ys;
      em_cell_body<D, R, false>(a, c_off, TM, j, off, N, tile, ys, tile + D * ys, tile + (D + 2) * ys);
      if (tid == 0) pool_give(pool, c.g0, c.gn);
    } else {
      em_cell_body<D, R, true>(a, c_off, TM, j, off, N, c.gY, c.ys, c.gS, c.gG);
    }
  }
}

}  // namespace gmcr
