// recon_sampler.cuh -- the counter-based particle sampler of the
// reconstruction (Sec. 2.4, eq. mix-dist-1) and the Lemons projection
// coefficients (Sec. 2.4.2, eqs. alpha, beta), shared by the 1D and 2D
// meshes.  A particle is regenerated bit-identically from (seed, cell,
// index); FP64 is kept for the position and for the velocity's offset from
// the mixture mean, the categorical choice is decided on integers and the
// Gaussian draw is FP32.
#pragma once

#include "gm_kernels.cuh"

namespace gmcr {

// Cell j's output range [o, o + n) of the caller's particle arrays (n_out
// particles).  A range that does not lie inside [0, n_out) -- a negative
// count, or a start or an end outside the arrays -- is replaced by the empty
// range, and the function returns false: the cell is then treated as a cell
// without resampled particles and flagged GM_ST_BAD_RANGE, so that no kernel
// writes outside the caller's buffers.
__device__ __forceinline__ bool out_range(const int64_t* out_off, int64_t j, int64_t n_out,
                                          int64_t& o, int64_t& n) {
  o = out_off[j];
  n = out_off[j + 1] - o;
  if (o < 0 || n < 0 || o > n_out - n) {
    o = 0;
    n = 0;
    return false;
  }
  return true;
}
__device__ __forceinline__ int64_t out_count(const int64_t* out_off, int64_t j, int64_t n_out) {
  int64_t o, n;
  out_range(out_off, j, n_out, o, n);
  return n;
}

template <int D>
struct RecCell {
  static constexpr int NM = D * (D + 1) / 2;
  // categorical thresholds: u < cw_k  <=>  2 m + 1 < thr_k, where
  // u = (m + 1/2) 2^-52 and thr_k = ceil(cw_k 2^53) (cw_k the cumulative
  // weights summed in component order): the FP64 comparison, decided on
  // integers
  long long thr[kMaxK];
  double dz[kMaxK][D];      // mu_k - u
  float Lf[kMaxK][NM];      // lower-triangular Cholesky factor (FP32), row-major
  double u[D];              // mixture mean sum_k w_k mu_k
  double theta;             // sum_k w_k (tr Sigma_k + |mu_k - u|^2)
  int K;
};

// FP32 lower-triangular Cholesky factor (row-major) of a component's
// covariance r[1 + D ..] (upper triangle), factored in FP64 with no floor: a
// non-positive pivot gives a zero column, as for a degenerate stored
// covariance
template <int D>
__device__ __forceinline__ void chol_f(const double* r, float* Lf) {
  if (D == 1) {
    const double s = r[2];
    Lf[0] = (float)(s > 0.0 ? sqrt(s) : 0.0);
  } else {
    // S upper: [s00 s01 s02 s11 s12 s22]
    const double s00 = r[4], s01 = r[5], s02 = r[6], s11 = r[7], s12 = r[8], s22 = r[9];
    const double l00 = s00 > 0.0 ? sqrt(s00) : 0.0;
    const double l10 = l00 > 0.0 ? s01 / l00 : 0.0;
    const double l20 = l00 > 0.0 ? s02 / l00 : 0.0;
    const double t11 = s11 - l10 * l10;
    const double l11 = t11 > 0.0 ? sqrt(t11) : 0.0;
    const double l21 = l11 > 0.0 ? (s12 - l20 * l10) / l11 : 0.0;
    const double t22 = s22 - l20 * l20 - l21 * l21;
    const double l22 = t22 > 0.0 ? sqrt(t22) : 0.0;
    Lf[0] = (float)l00; Lf[1] = (float)l10; Lf[2] = (float)l11;
    Lf[3] = (float)l20; Lf[4] = (float)l21; Lf[5] = (float)l22;
  }
}

// the mixture-wide quantities of a cell's Kj components rj (records of P
// values): the categorical thresholds (put_thr(k, t)), dz_k = mu_k - u
// (put_dz(k, d, value)), the mean u and the spread theta
template <int D, class PutThr, class PutDz>
__device__ __forceinline__ void mix_head(const double* rj, int Kj, PutThr put_thr, PutDz put_dz,
                                         double* u_out, double& theta) {
  constexpr int P = 1 + D + D * (D + 1) / 2;
  double cum = 0.0, u[D], th = 0.0;
  for (int d = 0; d < D; ++d) u[d] = 0.0;
  for (int q = 0; q < Kj; ++q) {
    const double* r = rj + (size_t)q * P;
    cum += r[0];
    const double t = ceil(cum * 9007199254740992.0);  // 2^53
    put_thr(q, t < 4.0e18 ? (long long)t : 4000000000000000000ll);
    for (int d = 0; d < D; ++d) u[d] += r[0] * r[1 + d];
  }
  for (int q = 0; q < Kj; ++q) {
    const double* r = rj + (size_t)q * P;
    double tr = 0.0, dd = 0.0;
    int t = 1 + D;
    for (int x = 0; x < D; ++x)
      for (int y = x; y < D; ++y, ++t) {
        if (x == y) tr += r[t];
      }
    for (int d = 0; d < D; ++d) {
      put_dz(q, d, r[1 + d] - u[d]);
      dd += (r[1 + d] - u[d]) * (r[1 + d] - u[d]);
    }
    th += r[0] * (tr + dd);
  }
  for (int d = 0; d < D; ++d) u_out[d] = u[d];
  theta = th;
}

// A cell's mixture data computed once per cell, by one thread per cell (the
// FP64 square roots and divisions then run 32 cells to a warp instruction),
// and kept in the workspace for the two particle passes: per cell a head
// (u, theta, K) and Kmax component records (threshold, dz, FP32 factor).
template <int D>
struct RecHead {
  double u[D];
  double theta;
  int K;
  int pad;
};
template <int D>
struct RecComp {
  long long thr;
  double dz[D];
  float Lf[D * (D + 1) / 2];
};
template <int D>
__device__ __forceinline__ void prep_cell(int64_t j, int Kmax, const int32_t* K, const double* prm,
                                          RecHead<D>* head, RecComp<D>* comp) {
  constexpr int P = 1 + D + D * (D + 1) / 2;
  const int Kj = K[j];
  const double* rj = prm + (size_t)j * Kmax * P;
  RecComp<D>* cj = comp + (size_t)j * Kmax;
  RecHead<D> h;
  mix_head<D>(
      rj, Kj, [&](int q, long long t) { cj[q].thr = t; },
      [&](int q, int d, double x) { cj[q].dz[d] = x; }, h.u, h.theta);
  h.K = Kj;
  h.pad = 0;
  head[j] = h;
  for (int q = 0; q < Kj; ++q) {
    float Lf[D * (D + 1) / 2];
    chol_f<D>(rj + (size_t)q * P, Lf);
    for (int m = 0; m < D * (D + 1) / 2; ++m) cj[q].Lf[m] = Lf[m];
  }
}
// copy cell j's prepared mixture into the warp's RecCell (lanes k < K copy
// component k, lane 0 the head)
template <int D>
__device__ __forceinline__ void load_prepped(RecCell<D>& rc, int64_t j, int Kmax,
                                             const RecHead<D>* head, const RecComp<D>* comp,
                                             int lane) {
  constexpr int NM = D * (D + 1) / 2;
  const int Kj = head[j].K;
  if (lane < Kj) {
    const RecComp<D>& c = comp[(size_t)j * Kmax + lane];
    rc.thr[lane] = c.thr;
#pragma unroll
    for (int d = 0; d < D; ++d) rc.dz[lane][d] = c.dz[d];
#pragma unroll
    for (int m = 0; m < NM; ++m) rc.Lf[lane][m] = c.Lf[m];
  }
  if (lane == 0) {
    const RecHead<D>& h = head[j];
    rc.K = Kj;
#pragma unroll
    for (int d = 0; d < D; ++d) rc.u[d] = h.u[d];
    rc.theta = h.theta;
  }
}

// the 52 leading bits of (hi, lo), as uniform52 uses them
__device__ __forceinline__ uint64_t bits52(uint32_t hi, uint32_t lo) {
  return ((uint64_t)hi << 20) | (uint64_t)(lo >> 12);
}
// (t + 1/2) 2^-52 in FP32 (relative error ~2^-24) for a 52-bit t, without
// FP64 arithmetic: t = hi26 2^26 + lo26
__device__ __forceinline__ float half_ulp52_f(uint64_t t) {
  const float hi = (float)(uint32_t)(t >> 26), lo = (float)(uint32_t)(t & 0x3FFFFFFull);
  return fmaf(hi, 1.4901161193847656e-08f /* 2^-26 */, (lo + 0.5f) * 2.220446049250313e-16f);
}
// Box-Muller radius sqrt(-2 ln u) for u = (m + 1/2) 2^-52, in FP32 from the
// integer: below 1/2, ln u; above, log1p(-(1 - u)) with 1 - u =
// (2^52 - 1 - m + 1/2) 2^-52 formed exactly on integers, so the radius
// keeps FP32 relative accuracy where its derivative is unbounded
__device__ __forceinline__ float bm_radius(uint64_t m) {
  const float lnu = m < (1ull << 51) ? logf(half_ulp52_f(m))
                                     : log1pf(-half_ulp52_f((1ull << 52) - 1ull - m));
  return sqrtf(-2.0f * lnu);
}

// (w + 1/2) 2^-32 in FP32 (relative error ~2^-24) for a 32-bit w
__device__ __forceinline__ float half_ulp32_f(uint32_t w) {
  return fmaf((float)w, 2.3283064365386963e-10f /* 2^-32 */, 1.1641532182693481e-10f /* 2^-33 */);
}
// the same radius for a 32-bit uniform (w + 1/2) 2^-32
__device__ __forceinline__ float bm_radius32(uint32_t w) {
  const float lnu = w < 0x80000000u ? logf(half_ulp32_f(w)) : log1pf(-half_ulp32_f(0xFFFFFFFFu - w));
  return sqrtf(-2.0f * lnu);
}

// particle i of cell j (Sec. 2.4, eq. mix-dist-1): the 52-bit integer m0
// of its position's uniform u0 = (m0 + 1/2) 2^-52 (x = (j + u0) dx), its
// component z (the categorical draw) and f = L_z xi (FP32), so that
// w = v - u = (mu_z - u) + f
template <int D>
__device__ __forceinline__ void sample_f(const RecCell<D>& rc, int64_t j, int64_t i, uint64_t seed,
                                         uint64_t& m0, int& z, float (&f)[D]) {
  const u32x4 r0 = philox_draw(seed, (uint32_t)i, kTagSample | 0u, j);
  m0 = bits52(r0.x, r0.y);
  const int K = rc.K;
  z = K - 1;  // the only choice when K <= 1
  if (K > 1) {
    const long long m1x2 = 2 * (long long)bits52(r0.z, r0.w) + 1;
    for (int k = 0; k < K; ++k)
      if (m1x2 < rc.thr[k]) { z = k; break; }
  }
  // Box-Muller (Box & Muller 1958) on block 1: for D = 1 one (radius,
  // angle) pair of 52-bit uniforms, for D = 3 two pairs of 32-bit uniforms
  // (words x, y and z, w), so that a 3V particle takes two Philox blocks
  float xi[3];
  const u32x4 r1 = philox_draw(seed, (uint32_t)i, kTagSample | 1u, j);
  if (D == 1) {
    const float rr = bm_radius(bits52(r1.x, r1.y));
    xi[0] = rr * cospif(2.0f * half_ulp52_f(bits52(r1.z, r1.w)));
  } else {
    const float rr = bm_radius32(r1.x);
    float sn, cs;
    sincospif(2.0f * half_ulp32_f(r1.y), &sn, &cs);
    xi[0] = rr * cs;
    xi[1] = rr * sn;
    xi[2] = bm_radius32(r1.z) * cospif(2.0f * half_ulp32_f(r1.w));
  }
  if (K == 0) {
    for (int d = 0; d < D; ++d) f[d] = 0.0f;
    return;
  }
  const float* L = rc.Lf[z];
  if (D == 1) {
    f[0] = L[0] * xi[0];
  } else {
    f[0] = L[0] * xi[0];
    f[1] = fmaf(L[2], xi[1], L[1] * xi[0]);
    f[2] = fmaf(L[5], xi[2], fmaf(L[4], xi[1], L[3] * xi[0]));
  }
}

// the particle's w = v - u in FP64 from its draw (z, f): (mu_z - u) + f
// (w = -u for a cell without a mixture)
template <int D>
__device__ __forceinline__ void draw_offset(const RecCell<D>& rc, int z, const float (&f)[D],
                                            double (&w)[D]) {
  if (rc.K == 0) {
    for (int d = 0; d < D; ++d) w[d] = -rc.u[d];
    return;
  }
#pragma unroll
  for (int d = 0; d < D; ++d) w[d] = rc.dz[z][d] + f2d_exact(f[d]);
}
// the 52 leading bits of the y uniform of particle i of cell j on a 2D mesh
// (Philox block 3, words 0-1)
__device__ __forceinline__ uint64_t sample_y_bits(int64_t j, int64_t i, uint64_t seed) {
  const u32x4 r3 = philox_draw(seed, (uint32_t)i, kTagSample | 3u, j);
  return bits52(r3.x, r3.y);
}

// (m + 1/2) 2^-52 - 1/2, the in-cell offset of a position from the cell
// centre in cell units (exact in FP64)
__device__ __forceinline__ double centred52(uint64_t m) {
  // ((m - 2^51) + 1/2) 2^-52 = (2 m - 2^52 + 1) 2^-53, built on the integer pipe
  return m >= (1ull << 51) ? odd_2m53(2ull * m - (1ull << 52) + 1ull, false)
                           : odd_2m53((1ull << 52) - 2ull * m - 1ull, true);
}
// j + u0 rounded to the nearest double (ties to even), as the FP64 addition
// (double)j + u0 gives it, on the integer pipe, for 0 <= j < 2^52: with L
// the leading bit of j the sum's 53-bit significand in units of 2^(L - 52)
// is j 2^(52 - L) + t / 2^(L + 1), t = 2 m + 1; the fraction t mod 2^(L+1)
// decides the rounding, and a carry to 2^53 moves the exponent up by one
__device__ __forceinline__ double cell_plus_u0(uint64_t j, uint64_t m) {
  const unsigned long long t = 2ull * m + 1ull;
  if (j == 0) return odd_2m53(t, false);
  const int L = 63 - __clzll((long long)j);
  unsigned long long M = (j << (52 - L)) + (t >> (L + 1));
  const unsigned long long rem = t & ((2ull << L) - 1ull), half = 1ull << L;
  M += (rem > half || (rem == half && (M & 1ull))) ? 1ull : 0ull;
  const int e = M >> 53 ? L + 1 : L;
  M = M >> 53 ? (1ull << 52) : M;
  return __longlong_as_double((long long)(((unsigned long long)(1023 + e) << 52) | (M & ((1ull << 52) - 1ull))));
}

// Lemons projection of a cell with n resampled particles: the corrected
// weight alpha' = W_j / n + dA_j and, from the sums sw[d] = sum_p w_d and
// sw[D] = sum_p |w|^2 (w = v - u), the scale a and shift beta of eqs.
// (alpha), (beta) in the frame of the mixture mean u:
// 2 E N' - p^2 = W (N' theta + (N' - W) |u|^2),
// 2 E' N' - p'^2 = alpha'^2 (n sum|w|^2 - |sum w|^2).
template <int D>
struct ProjCoef {
  double a, beta[D], alpha_new;
  int skip;
  unsigned int status;
};
template <int D>
__device__ __forceinline__ ProjCoef<D> proj_coeffs(int K, const double* u, double theta, int64_t n,
                                                   double Wj, double dAj, const double* sw) {
  ProjCoef<D> pc;
  unsigned int st = 0;
  if (n == 0) st |= GM_ST_MM_EMPTY_COL;
  const double an = (n > 0 ? Wj / (double)n : 0.0) + dAj;
  pc.alpha_new = an;
  if (n > 0 && !(an > 0.0)) st |= GM_ST_NEG_WEIGHT;
  pc.skip = 1;
  pc.a = 1.0;
  for (int d = 0; d < D; ++d) pc.beta[d] = 0.0;
  if (n > 0 && K == 0) st |= GM_ST_NO_MIXTURE;
  if (n > 0 && K > 0) {
    const double Np = (double)n * an;
    double u2 = 0.0, sw2 = 0.0;
    for (int d = 0; d < D; ++d) {
      u2 += u[d] * u[d];
      sw2 += sw[d] * sw[d];
    }
    const double num = Wj * (Np * theta + (Np - Wj) * u2);
    const double den = an * an * ((double)n * sw[D] - sw2);
    if (num > 0.0 && den > 0.0 && Np > 0.0) {
      const double aa = sqrt(num / den);
      pc.a = aa;
      for (int d = 0; d < D; ++d) pc.beta[d] = ((Wj - Np) * u[d] - aa * an * sw[d]) / (aa * Np);
      pc.skip = 0;
    } else {
      st |= GM_ST_PROJ_SKIPPED;
    }
  }
  pc.status = st;
  return pc;
}
// ---------------------------------------------------------------------------
// Pass 1's per-cell record and the staged draws (both meshes)
// ---------------------------------------------------------------------------
// Sums of a cell's resampled particles.  A cell with components and at most
// kFixMaxN particles keeps integer sums (fixed = 1), every other cell FP64
// sums:
//   integer: sum t as (low, high) 64-bit halves in words (2t, 2t+1): first
//            the NP position sums, then D sums of f_d (one component) or
//            w_d (several) in units of 2^eq_d, then D sums of their squares;
//   FP64:    words 0 .. NP-1 the position sums, then the D sums of f_d (one
//            component) or w_d (otherwise) and the sum of |f|^2 or |w|^2.
// w = v - u = dz + f with f = L_z xi.  An FP64 addition costs as much as some
// sixty integer instructions here, and the integer sums carry no rounding
// from particle to particle.
template <int D, int NP>
struct alignas(16) RecRaw {
  static constexpr int NS = NP + 2 * D;
  double w[2 * NS];
  int eq[3];
  int fixed;
};
__device__ __forceinline__ __int128 load_i128(const double* p) {
  const longlong2 v = *reinterpret_cast<const longlong2*>(p);
  return ((__int128)v.y << 64) | (__int128)(unsigned long long)v.x;
}
// bound of |f_d| by the factor's rows: |xi| <= sqrt(-2 ln 2^-53) = 8.6 < 9
template <int D>
__device__ __forceinline__ void row_bounds(const float* L, float (&bnd)[D]) {
  if (D == 1) {
    bnd[0] = 9.0f * fabsf(L[0]);
  } else {
    bnd[0] = 9.0f * fabsf(L[0]);
    bnd[1] = 9.0f * (fabsf(L[1]) + fabsf(L[2]));
    bnd[D - 1] = 9.0f * (fabsf(L[3]) + fabsf(L[4]) + fabsf(L[5]));
  }
}
// exponent eq with v / 2^eq below 2^bits for |v| <= b
__device__ __forceinline__ int fix_exponent(float b, int bits) {
  const int eb = (int)((__float_as_uint(b) >> 23) & 0xFFu);
  return (eb ? eb - 127 : -126) + 1 - bits;
}
// The fixed-point plan of a cell in the warp's RecCell: the exponents eq and
// (several components) dzq[k] = dz_k / 2^eq.  One component: f alone, kFixBits
// bits, so that a lane's kFixMaxN / 32 = 512 terms (0.96 x 2^54 each) stay
// below 2^63; several: w, one bit less.  False (no component, too many
// particles, or offsets beyond FP32) for the FP64 sums.
template <int D>
__device__ __forceinline__ bool fix_plan(const RecCell<D>& rc, int64_t n, int lane, int (&eq)[D],
                                         long long (*dzq)[D]) {
  const int K = rc.K;
  if (K < 1 || n > kFixMaxN) return false;
  float b[D];
  row_bounds<D>(rc.Lf[lane < K ? lane : 0], b);
  if (K == 1) {
#pragma unroll
    for (int d = 0; d < D; ++d) eq[d] = fix_exponent(b[d], kFixBits);
    return true;
  }
  bool ok = true;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    b[d] = lane < K ? (fabsf((float)rc.dz[lane][d]) + b[d]) * 1.00001f : 0.0f;
    b[d] = warp_max(b[d]);
    ok = ok && b[d] < 1e38f;
    eq[d] = fix_exponent(b[d], kFixBits - 1);
  }
  if (!__all_sync(0xffffffffu, ok)) return false;
  if (lane < K)
#pragma unroll
    for (int d = 0; d < D; ++d) dzq[lane][d] = fixq(rc.dz[lane][d], eq[d]);
  __syncwarp();
  return true;
}
// the warp's integer sums sm into cell record r
template <int D, int NP>
__device__ __forceinline__ void put_fixed(RecRaw<D, NP>& r, const __int128 (&sm)[NP + 2 * D], const int (&eq)[D],
                                          int lane) {
  constexpr int NS = NP + 2 * D, NQ = NS <= 4 ? 4 : (NS <= 8 ? 8 : 16);
  __int128 w[NQ];
#pragma unroll
  for (int t = 0; t < NQ; ++t) w[t] = t < NS ? sm[t < NS ? t : 0] : (__int128)0;
  const __int128 mine = warp_rs_i128<NQ>(w, lane);
  const int t = warp_rs_index<NQ>(lane);
  if (t < NS && lane == warp_rs_lane<NQ>(t))  // the first of the lanes that hold the sum
    *reinterpret_cast<longlong2*>(&r.w[2 * t]) =
        make_longlong2((long long)(unsigned long long)mine, (long long)(mine >> 64));
  if (lane == 0) {
#pragma unroll
    for (int d = 0; d < D; ++d) r.eq[d] = eq[d];
    r.fixed = 1;
  }
}
// Pass 1 stages each particle's draw in the caller's output slots of that
// same particle, and pass 2 reads it back before it overwrites them with
// the final values (one thread reads, then writes, each particle's slots,
// so no other particle's staging is ever touched): x_out[p] holds the
// position integer m0 (52 bits) and the component z (bits 56-63),
// alpha_out[p] the FP32 pair (f_0, f_1), v_out[0][p] (D = 3) the FP32 f_2.
// The second pass then needs neither the Philox draws nor the Box-Muller
// transform of the first.
template <int D>
__device__ __forceinline__ void stage_draw(double* x_out, double* v_out, double* alpha_out,
                                           int64_t p, uint64_t m0, int z, const float (&f)[D]) {
  reinterpret_cast<unsigned long long*>(x_out)[p] = m0 | ((unsigned long long)(z & 0xFF) << 56);
  reinterpret_cast<float2*>(alpha_out)[p] = make_float2(f[0], D == 3 ? f[1] : 0.0f);
  if (D == 3) reinterpret_cast<float2*>(v_out)[p] = make_float2(f[D - 1], 0.0f);
}
template <int D>
__device__ __forceinline__ void load_draw(const double* x_out, const double* v_out,
                                          const double* alpha_out, int64_t p, uint64_t& m0, int& z,
                                          float (&f)[D]) {
  const unsigned long long t = reinterpret_cast<const unsigned long long*>(x_out)[p];
  m0 = t & ((1ull << 52) - 1ull);
  z = (int)(t >> 56);
  const float2 a = reinterpret_cast<const float2*>(alpha_out)[p];
  f[0] = a.x;
  if (D == 3) {
    f[1] = a.y;
    f[D - 1] = reinterpret_cast<const float2*>(v_out)[p].x;
  }
}

// sum w (sw[0 .. D-1]) and sum |w|^2 (sw[D]) of a cell; for one component
// w = dz + f with one dz, so sum w = n dz + sum f and
// sum |w|^2 = n |dz|^2 + 2 dz . sum f + sum |f|^2
template <int D, int NP>
__device__ __forceinline__ void velocity_sums(const RecRaw<D, NP>& r, int Kj, const RecComp<D>& c0,
                                              int64_t n, double (&sw)[D + 1]) {
  if (r.fixed) {
    sw[D] = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      sw[d] = i128_to_f64(load_i128(&r.w[2 * (NP + d)]), r.eq[d]);
      sw[D] += i128_to_f64(load_i128(&r.w[2 * (NP + D + d)]), 2 * r.eq[d]);
    }
  } else {
#pragma unroll
    for (int t = 0; t <= D; ++t) sw[t] = r.w[NP + t];
  }
  if (Kj == 1) {
    const double nd = (double)n;
    double dzf = 0.0, dz2 = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const double dz = c0.dz[d];
      dzf = fma(dz, sw[d], dzf);
      dz2 = fma(dz, dz, dz2);
      sw[d] = fma(nd, dz, sw[d]);
    }
    sw[D] = fma(nd, dz2, fma(2.0, dzf, sw[D]));
  }
}

// Pass 0, one thread per cell: each cell's mixture data for the two particle
// passes (prep_cell).
template <int D>
__global__ void recon_prep_kernel(int64_t C, int Kmax, const int32_t* K, const double* prm,
                                  RecHead<D>* head, RecComp<D>* comp) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < C;
       j += (int64_t)gridDim.x * blockDim.x)
    prep_cell<D>(j, Kmax, K, prm, head, comp);
}

// a cell's projection for pass 2: the scale a and shift beta, the corrected
// weight and, for one component, cv = u + a (dz + beta), so that the particle
// pass writes v = cv + a f (a = 1 and beta = 0 when the projection is skipped)
template <int D>
struct RecCoef {
  double a, beta[D], alpha_new, cv[D];
};
template <int D>
__device__ __forceinline__ RecCoef<D> make_coef(const ProjCoef<D>& pc, const RecHead<D>& h,
                                                const RecComp<D>& c0) {
  RecCoef<D> cf;
  cf.a = pc.a;
  cf.alpha_new = pc.alpha_new;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    cf.beta[d] = pc.beta[d];
    cf.cv[d] = h.K == 1 ? fma(pc.a, c0.dz[d] + pc.beta[d], h.u[d]) : 0.0;
  }
  return cf;
}

// Pass 2, one warp per cell: the final particles (positions, projected
// velocities, corrected weights) from the draws that pass 1 staged (on the 2D
// mesh y_out holds the y uniform's 52 bits).
template <int D, int NW, bool kMesh2d>
__global__ void __launch_bounds__(NW * 32) recon_emit_kernel(
    int64_t C, int Kmax, const RecHead<D>* head, const RecComp<D>* comp, const RecCoef<D>* coef,
    const int64_t* out_off, int64_t Cx, double dx, double dy, int64_t n_out, double* x_out, double* y_out,
    double* v_out, double* alpha_out) {
  __shared__ RecCell<D> rcs[NW];
  __shared__ double cvs[NW][kMaxK][D];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  RecCell<D>& rc = rcs[wid];
  for (int64_t j = (int64_t)blockIdx.x * NW + wid; j < C; j += (int64_t)gridDim.x * NW) {
    load_prepped<D>(rc, j, Kmax, head, comp, lane);
    const RecCoef<D> cf = coef[j];
    __syncwarp();
    int64_t o, n;
    out_range(out_off, j, n_out, o, n);
    const double aa = cf.a, an = cf.alpha_new;
    const uint64_t jx = kMesh2d ? (uint64_t)(j % Cx) : (uint64_t)j, jy = kMesh2d ? (uint64_t)(j / Cx) : 0;
    if (rc.K == 1) {
      // four particles per lane per step: their staged draws are all loaded
      // before any of their slots is overwritten, so the loads of a step
      // are in flight together
      constexpr int U = 4;
      int64_t i = lane;
      for (; i + 32 * (U - 1) < n; i += 32 * U) {
        uint64_t m0[U], my[U];
        int z[U];
        float f[U][D];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          load_draw<D>(x_out, v_out, alpha_out, o + i + 32 * u, m0[u], z[u], f[u]);
          my[u] = kMesh2d ? reinterpret_cast<const unsigned long long*>(y_out)[o + i + 32 * u] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t p = o + i + 32 * u;
          x_out[p] = __dmul_rn(cell_plus_u0(jx, m0[u]), dx);
          if (kMesh2d) y_out[p] = __dmul_rn(cell_plus_u0(jy, my[u]), dy);
          alpha_out[p] = an;
#pragma unroll
          for (int d = 0; d < D; ++d) v_out[(int64_t)d * n_out + p] = fma(aa, f2d_exact(f[u][d]), cf.cv[d]);
        }
      }
      for (; i < n; i += 32) {
        uint64_t m0, my = 0;
        int z;
        float f[D];
        load_draw<D>(x_out, v_out, alpha_out, o + i, m0, z, f);
        if (kMesh2d) my = reinterpret_cast<const unsigned long long*>(y_out)[o + i];
        x_out[o + i] = __dmul_rn(cell_plus_u0(jx, m0), dx);
        if (kMesh2d) y_out[o + i] = __dmul_rn(cell_plus_u0(jy, my), dy);
        alpha_out[o + i] = an;
#pragma unroll
        for (int d = 0; d < D; ++d) v_out[(int64_t)d * n_out + o + i] = fma(aa, f2d_exact(f[d]), cf.cv[d]);
      }
    } else {
      // several components: v = c_z + a f with c_k = u + a (dz_k + beta) once
      // per component (one FP64 operation per dimension instead of three:
      // 0.47 -> 0.26 ms for 18.8 M particles in 3V, 0.12 -> 0.07 for 8.2 M in 1V); no component: v = 0
      if (lane < rc.K)
#pragma unroll
        for (int d = 0; d < D; ++d) cvs[wid][lane][d] = fma(aa, rc.dz[lane][d] + cf.beta[d], rc.u[d]);
      if (rc.K == 0 && lane < D) cvs[wid][0][lane] = 0.0;
      __syncwarp();
      const int zmax = rc.K > 0 ? rc.K - 1 : 0;
      constexpr int U = 2;
      int64_t i = lane;
      for (; i + 32 * (U - 1) < n; i += 32 * U) {
        uint64_t m0[U], my[U];
        int z[U];
        float f[U][D];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          load_draw<D>(x_out, v_out, alpha_out, o + i + 32 * u, m0[u], z[u], f[u]);
          my[u] = kMesh2d ? reinterpret_cast<const unsigned long long*>(y_out)[o + i + 32 * u] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t p = o + i + 32 * u;
          const double* cv = cvs[wid][z[u] < zmax ? z[u] : zmax];
          x_out[p] = __dmul_rn(cell_plus_u0(jx, m0[u]), dx);
          if (kMesh2d) y_out[p] = __dmul_rn(cell_plus_u0(jy, my[u]), dy);
          alpha_out[p] = an;
#pragma unroll
          for (int d = 0; d < D; ++d) v_out[(int64_t)d * n_out + p] = fma(aa, f2d_exact(f[u][d]), cv[d]);
        }
      }
      for (; i < n; i += 32) {
        uint64_t m0, my = 0;
        int z;
        float f[D];
        load_draw<D>(x_out, v_out, alpha_out, o + i, m0, z, f);
        if (kMesh2d) my = reinterpret_cast<const unsigned long long*>(y_out)[o + i];
        const double* cv = cvs[wid][z < zmax ? z : zmax];
        x_out[o + i] = __dmul_rn(cell_plus_u0(jx, m0), dx);
        if (kMesh2d) y_out[o + i] = __dmul_rn(cell_plus_u0(jy, my), dy);
        alpha_out[o + i] = an;
#pragma unroll
        for (int d = 0; d < D; ++d) v_out[(int64_t)d * n_out + o + i] = fma(aa, f2d_exact(f[d]), cv[d]);
      }
    }
    __syncwarp();
  }
}

}  // namespace gmcr
