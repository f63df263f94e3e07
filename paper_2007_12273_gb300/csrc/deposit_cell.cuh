// deposit_cell.cuh -- one cell's charge-deposit sums (Sec. 2.4.1), computed
// by one warp: the record that deposit_combine_kernel turns into rho.  Used
// by the deposit kernel and, fused with the closed-form pre-pass of
// gm_compress_from, by em_k1_kernel (both read the cell's weights).
//
// Per cell, the partial deposits on nodes j-1, j, j+1 follow from
// A0 = sum alpha, A1 = sum alpha s, A2 = sum alpha s^2 (quadratic
// B-spline) or the CIC parts sum alpha max(-s, 0), sum alpha max(s, 0),
// with s = xi - 1/2 the particle's offset from the cell centre.  Record of
// kDepWords 64-bit words:
//   equal weights: [k0 (low, high), k1 (low, high), alpha bits, n], the
//     exact 128-bit sums of k and k^2 (or of the CIC parts) with
//     s = k 2^-53;
//   otherwise: [A0, A1, A2 (FP64 bits), -, -, -1].
#pragma once

#include "gm_common.cuh"

namespace gmcr {

constexpr int kDepWords = 6;

// the weights of a cell's n particles equal bit for bit (every lane gets the
// answer; alpha = NULL means unit weights)
__device__ __forceinline__ bool equal_weights(const double* alpha, int64_t o, int64_t n, int lane) {
  if (!alpha) return true;
  const long long wb = __double_as_longlong(alpha[o]);
  bool same = true;
#pragma unroll 4
  for (int64_t p = lane; p < n; p += 32) same &= (__double_as_longlong(alpha[o + p]) == wb);
  return __all_sync(0xffffffffu, same);
}

// k = round(xi 2^53) - 2^52 of an FP64 xi in [0, 1), from its bits
__device__ __forceinline__ long long frac_k(double xi) {
  // xi = m 2^(e - 1075) (m with its implicit bit)
  const unsigned long long u = (unsigned long long)__double_as_longlong(xi);
  const int e = (int)((u >> 52) & 0x7FFull);
  const long long m = (long long)((u & ((1ull << 52) - 1ull)) | (e ? (1ull << 52) : 0ull));
  const int sh = (e ? e : 1) - 1022;  // xi 2^53 = m 2^sh, sh <= 0
  long long rr = 0;
  if (sh == 0) rr = m;
  else if (sh > -60) rr = (m + (1ll << (-sh - 1))) >> (-sh);
  return rr - (1ll << 52);
}

// a lane's sums of k and k^2 (quadratic B-spline) or of the CIC parts
// max(-k, 0) and max(k, 0), |k| <= 2^52, over up to kFixMaxN / 32 = 512
// particles: k = h 2^27 + l has |h| <= 2^25, so that SplitSum's parts stay
// below 2^63 for 512 terms
struct DepSums {
  long long k0 = 0;
  SplitSum q;
  __device__ __forceinline__ void add(long long k, int order) {
    if (order == 1) {
      k0 += k < 0 ? -k : 0;
      q.ll += k > 0 ? k : 0;
    } else {
      k0 += k;
      q.add_square(SplitInt(k));
    }
  }
  // the equal-weight record r (weight bits wb) of the warp's cell
  __device__ __forceinline__ void put(long long wb, int64_t n, int order, long long* r, int lane) const {
    __int128 s0 = (__int128)k0, s1 = order == 1 ? (__int128)q.ll : q.total_square();
#pragma unroll
    for (int b = 16; b > 0; b >>= 1) {
      s0 += shfl_xor_i128(s0, b);
      s1 += shfl_xor_i128(s1, b);
    }
    // lanes 0-5 write the record's words
    long long wv = (long long)(unsigned long long)s0;
    wv = lane == 1 ? (long long)(s0 >> 64) : wv;
    wv = lane == 2 ? (long long)(unsigned long long)s1 : wv;
    wv = lane == 3 ? (long long)(s1 >> 64) : wv;
    wv = lane == 4 ? wb : wv;
    wv = lane == 5 ? (long long)n : wv;
    if (lane < kDepWords) r[lane] = wv;
  }
};

// cell j's record r; same = equal_weights(...) for 0 < n <= kFixMaxN
__device__ __forceinline__ void deposit_cell(int64_t j, int64_t o, int64_t n, const double* x,
                                             const double* alpha, double inv_dx, int order,
                                             long long* r, int lane, bool same) {
  const double jd = (double)j;
  // equal weights (bit for bit) and at most 2^14 particles: the sums of s
  // and s^2 (or of the CIC parts) exactly on the integer pipe, s = k 2^-53
  // with k = round(xi 2^53) - 2^52 from the bits of the FP64 in-cell
  // position xi in [0, 1); the weight multiplies the sums once
  if (n > 0 && n <= kFixMaxN && same) {
    const long long wb = alpha ? __double_as_longlong(alpha[o]) : __double_as_longlong(1.0);
    DepSums t;
#pragma unroll 2
    for (int64_t p = lane; p < n; p += 32) t.add(frac_k(cell_frac(x[o + p], jd, inv_dx)), order);
    t.put(wb, n, order, r, lane);
    return;
  }
  // otherwise by chunks of kSumChunk particles: in fixed point (see
  // kScaleBits), or in FP64 where a weight is not finite or the weights spread
  // too far (keeps_bits): the sum of the weights, to which the quadratic
  // B-spline's parts add up, and for CIC each side's part, which stands alone
  ChunkSum tot;  // sum t on lane t < 3
  for (int64_t c0 = o; c0 < o + n; c0 += kSumChunk) {
    const int m = (int)(o + n - c0 < kSumChunk ? o + n - c0 : kSumChunk);
    int ea = 0;
#pragma unroll 4
    for (int p = lane; p < m; p += 32) ea = max(ea, exp_field(alpha ? alpha[c0 + p] : 1.0));
    ea = warp_imax(ea);
    bool fixed = exp_finite(ea, 0.0);
    double mine;
    if (fixed) {
      const int eq = scale_exp(ea, 0.0);
      const TermShift sh(m, 62);
      long long s0 = 0, s1 = 0, s2 = 0;  // units of 2^(eq + sh.s)
      for (int p0 = lane; p0 < m; p0 += 128) {  // the loads of four particles together
        double xp[4], ap[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = min(p0 + 32 * u, m - 1);
          xp[u] = x[c0 + p];
          ap[u] = alpha ? alpha[c0 + p] : 1.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (p0 + 32 * u >= m) break;
          const long long k = frac_k(cell_frac(xp[u], jd, inv_dx));
          const long long a = fixq(ap[u], eq), X = k << 11;  // s = X 2^-64
          const long long as = __mul64hi(a, X);
          s0 += sh(a);
          if (order == 1) {
            const long long t = sh(as);
            s1 -= k < 0 ? t : 0;
            s2 += k > 0 ? t : 0;
          } else {
            s1 += sh(as);
            s2 += sh(__mul64hi(as, X));
          }
        }
      }
      __int128 t0 = s0, t1 = s1, t2 = s2;
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) {
        t0 += shfl_xor_i128(t0, q);
        t1 += shfl_xor_i128(t1, q);
        t2 += shfl_xor_i128(t2, q);
      }
      mine = i128_to_f64(lane == 0 ? t0 : (lane == 1 ? t1 : t2), eq + sh.s);
      fixed = keeps_bits(t0, m, 62, sh) &&
              (order != 1 || (keeps_bits(t1, m, 62, sh) && keeps_bits(t2, m, 62, sh)));
    }
    if (!fixed) {
      double a0 = 0.0, a1 = 0.0, a2 = 0.0;
      for (int p = lane; p < m; p += 32) {
        const double sx = cell_frac(x[c0 + p], jd, inv_dx) - 0.5;
        const double al = alpha ? alpha[c0 + p] : 1.0;
        if (order == 1) {
          a0 += al;
          a1 = sx < 0.0 ? fma(-al, sx, a1) : a1;
          a2 = sx > 0.0 ? fma(al, sx, a2) : a2;
        } else {
          const double as = al * sx;
          a0 += al;
          a1 += as;
          a2 = fma(as, sx, a2);
        }
      }
      a0 = warp_sum(a0);
      a1 = warp_sum(a1);
      a2 = warp_sum(a2);
      mine = lane == 0 ? a0 : (lane == 1 ? a1 : a2);
    }
    tot.add(mine, c0 == o);
  }
  long long wv = __double_as_longlong(tot.value());
  wv = lane == 5 ? -1ll : wv;
  if (lane < kDepWords) r[lane] = wv;
}

}  // namespace gmcr
