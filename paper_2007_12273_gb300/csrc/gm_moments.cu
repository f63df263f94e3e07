// gm_moments.cu -- charge deposition (Sec. 2.4.1) and per-cell moments.
#include "deposit_cell.cuh"
#include "gm_kernels.cuh"

namespace gmcr {

// Per-cell partial deposits: part[j] = sum_{p in j} alpha_p S(x_i - x_p)
// for i = j-1, j, j+1 (alpha = NULL means unit weights).  With s = xi - 1/2
// (xi the position inside the cell) the quadratic B-spline weights are
// (1/2 - s)^2 / 2, 3/4 - s^2, (1/2 + s)^2 / 2, so the three sums follow
// from A0 = sum alpha, A1 = sum alpha s, A2 = sum alpha s^2; for CIC they
// are sum alpha max(-s, 0), A0 - (the other two), sum alpha max(s, 0).
//
// deposit_partials_kernel, one warp per cell, writes each cell's sums to a
// record (deposit_cell.cuh); deposit_combine_kernel, one thread per node,
// turns the records of the node's three cells into the charge, so the
// per-cell FP64 work runs 32 cells to a warp instruction.
size_t deposit_ws_bytes(int64_t C) { return (size_t)kDepWords * 8 * (size_t)(C > 0 ? C : 0) + 256; }

template <int NW>
__global__ void __launch_bounds__(NW * 32) deposit_partials_kernel(int64_t C, const int64_t* cell_off,
                                                                   const double* x, const double* alpha,
                                                                   double inv_dx, int order,
                                                                   long long* rec) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t j = (int64_t)blockIdx.x * NW + wid; j < C; j += (int64_t)gridDim.x * NW) {
    const int64_t o = cell_off[j], n = cell_off[j + 1] - o;
    const bool same = n > 0 && n <= kFixMaxN && equal_weights(alpha, o, n, lane);
    deposit_cell(j, o, n, x, alpha, inv_dx, order, rec + (size_t)j * kDepWords, lane, same);
  }
}

// the three partial deposits of a cell (on its nodes j-1, j, j+1) from its
// record
__device__ __forceinline__ void dep_parts(const long long* r, int order, double (&pt)[3]) {
  double a0, a1, a2;
  if (r[5] >= 0) {
    const double al = __longlong_as_double(r[4]);
    const __int128 k0 = ((__int128)r[1] << 64) | (__int128)(unsigned long long)r[0];
    const __int128 k1 = ((__int128)r[3] << 64) | (__int128)(unsigned long long)r[2];
    a0 = al * (double)r[5];
    a1 = al * i128_to_f64(k0, -53);
    a2 = al * i128_to_f64(k1, order == 1 ? -53 : -106);
  } else {
    a0 = __longlong_as_double(r[0]);
    a1 = __longlong_as_double(r[1]);
    a2 = __longlong_as_double(r[2]);
  }
  if (order == 1) {
    pt[0] = a1;
    pt[1] = a0 - a1 - a2;
    pt[2] = a2;
  } else {
    pt[0] = 0.5 * (0.25 * a0 - a1 + a2);
    pt[1] = 0.75 * a0 - a2;
    pt[2] = 0.5 * (0.25 * a0 + a1 + a2);
  }
}

// rho_i = (q/dx) (part[i-1][+] + part[i][0] + part[i+1][-]), periodic
__global__ void deposit_combine_kernel(int64_t C, const long long* rec, int order, double q_over_dx,
                                       double* rho) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < C;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t im = (i == 0) ? C - 1 : i - 1;
    const int64_t ip = (i == C - 1) ? 0 : i + 1;
    double pm[3], p0[3], pp[3];
    dep_parts(rec + (size_t)im * kDepWords, order, pm);
    dep_parts(rec + (size_t)i * kDepWords, order, p0);
    dep_parts(rec + (size_t)ip * kDepWords, order, pp);
    rho[i] = q_over_dx * (pm[2] + p0[1] + pp[0]);
  }
}

// W, p, M2 (upper triangle), E of each cell's particles, one warp per cell, by
// chunks of kSumChunk particles.  A chunk of finite particles takes fixed-point
// sums (see kScaleBits): a pass for the largest exponents, then alpha, alpha v
// and alpha v v^T on the integer pipe, converted to FP64 a sum per lane.  A
// chunk in which one of them does not keep the bits of its own terms
// (keeps_bits) sums in FP64 (13 operations a particle for D = 3): the weight
// and the diagonal of alpha v v^T by their totals, an off-diagonal by the sum of
// its terms' magnitudes (a light x-velocity may meet every heavy y-velocity);
// alpha v follows from the diagonal, as |v| >= v^2 / max|v|.  A CTA per cell with 28 FP64 operations a particle and
// FP64 sums over its warps took 2.83 ms for 65536 3V cells of 572 weighted
// particles (FP64 pipe); moments and deposit together went from 3.55 to 1.09 ms
// (1.1 GB; issue and the latency of the loads share it: one load in flight a
// lane took 1.25).  Six CTAs an SM (80 registers) hide the
// loads and the reductions better than five (95).  E = tr(M2) / 2.
// A cell of more than kBigCell particles is left to a whole CTA, after the
// others: its chunks go round the CTA's warps, whose sums are added in their
// order.  With a warp for every cell 152 3V cells of 1e5 particles took 3.66 ms
// and one of 1e7 338; now 2.15 and 200 (with the deposit, a warp a cell).
constexpr int kBigCell = 2 * kSumChunk;
constexpr int kLoads = 4;  // particles a lane whose loads are issued together
template <int D, int NW, typename VT>
__global__ void __launch_bounds__(NW * 32, D == 3 ? 6 : 8) moments_kernel(int64_t C, int64_t n, const int64_t* cell_off,
                                                          const VT* v, const double* alpha, double* W,
                                                          double* p, double* M2, double* E) {
  constexpr int NM = D * (D + 1) / 2;
  constexpr int NS = 1 + D + NM;
  constexpr int NP = NS <= 4 ? 4 : 16;
  __shared__ double parts[NW][NS][2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // the CTA's cells: groups of NW, a warp each, or one where the grid has a CTA per cell
  const int per = C <= (int64_t)gridDim.x ? 1 : NW;
  const int64_t step = (int64_t)gridDim.x * per;
  bool big = false, met = false;  // the second turn, for the CTA's big cells; whether it has any
  int w = 0;                      // place in the group (second turn)
  int64_t j = wid < per ? (int64_t)blockIdx.x * per + wid : C;
  for (;;) {
    if (j >= C) {
      // every warp gets here once, and they take the second turn together
      if (big || !__syncthreads_or(met)) break;
      big = true;
      j = (int64_t)blockIdx.x * per;
    }
    const int64_t jc = j, o = cell_off[jc], end = cell_off[jc + 1];
    j += step;
    if (big) {
      j = ++w == per ? j - per + 1 : jc + 1;
      w = w == per ? 0 : w;
    }
    if ((end - o > kBigCell) != big) {
      met = true;
      continue;
    }
    const int64_t first = big ? o + (int64_t)wid * kSumChunk : o;
    ChunkSum tot;  // sum t on lane t < NS
    for (int64_t c0 = first; c0 < end; c0 += (big ? NW : 1) * kSumChunk) {
      const int cnt = (int)(end - c0 < kSumChunk ? end - c0 : kSumChunk);
      const double* al = alpha + c0;
      const VT* vj = v ? v + c0 : nullptr;  // no velocities: the weights' sum alone
      // the largest exponents
      int ea = 0, ev[D];
      bool moves[D];  // whether any velocity is not zero
#pragma unroll
      for (int d = 0; d < D; ++d) ev[d] = 0;
#pragma unroll 4
      for (int q = lane; q < cnt; q += 32) {
        ea = max(ea, exp_field(al[q]));
        if (vj)
#pragma unroll
          for (int d = 0; d < D; ++d) ev[d] = max(ev[d], top_bits(vj[(int64_t)d * n + q]));
      }
      ea = warp_imax(ea);
      bool fixed = exp_finite(ea, 0.0);
#pragma unroll
      for (int d = 0; d < D; ++d) {
        ev[d] = warp_imax(ev[d]);
        moves[d] = ev[d] != 0;
        ev[d] = top_exp(ev[d], VT(0));
        fixed = fixed && exp_finite(ev[d], VT(0));
      }
      double mine;
      if (fixed) {
        const int qa = scale_exp(ea, 0.0);
        int qv[D];
#pragma unroll
        for (int d = 0; d < D; ++d) qv[d] = scale_exp(ev[d], VT(0));
        const TermShift s0(cnt, 62), s1(cnt, 60);
        // units: 2^(qa + s0.s); 2^(qa + qv + 64 + s1.s); 2^(qa + qv + qv' + 126 + s1.s)
        long long s[NP];
        int mag[D == 3 ? 3 : 1];  // the off-diagonal terms' magnitudes, high words (below 2^30)
#pragma unroll
        for (int t = 0; t < NP; ++t) s[t] = 0;
#pragma unroll
        for (int t = 0; t < (D == 3 ? 3 : 1); ++t) mag[t] = 0;
        for (int q0 = lane; q0 < cnt; q0 += 32 * kLoads) {
          double ap[kLoads];
          VT vp[kLoads][D];
#pragma unroll
          for (int u = 0; u < kLoads; ++u) {
            const int q = min(q0 + 32 * u, cnt - 1);
            ap[u] = al[q];
#pragma unroll
            for (int d = 0; d < D; ++d) vp[u][d] = vj ? vj[(int64_t)d * n + q] : VT(0);
          }
#pragma unroll
          for (int u = 0; u < kLoads; ++u) {
            if (q0 + 32 * u >= cnt) break;
            const long long a = fixq(ap[u], qa);
            s[0] += s0(a);
            if (vj) {
              long long vq[D], av[D];
#pragma unroll
              for (int d = 0; d < D; ++d) {
                vq[d] = fixq<kScaleBits>(vp[u][d], qv[d]);
                av[d] = __mul64hi(a, vq[d]);  // below 2^60, units of 2^(qa + qv + 64)
                s[1 + d] += s1(av[d]);
              }
              int t = 1 + D;
#pragma unroll
              for (int x = 0; x < D; ++x)
#pragma unroll
                for (int y = x; y < D; ++y, ++t) {
                  const long long w = s1(__mul64hi(av[x] << 2, vq[y]));
                  s[t] += w;
                  if (y > x) mag[x + y - 1] += abs((int)(w >> 32));
                }
            }
          }
        }
        const int i = warp_rs_index<NP>(lane);
        int unit = qa + s0.s, t = 1 + D;
#pragma unroll
        for (int d = 0; d < D; ++d) unit = i == 1 + d ? qa + qv[d] + 64 + s1.s : unit;
#pragma unroll
        for (int x = 0; x < D; ++x)
#pragma unroll
          for (int y = x; y < D; ++y, ++t) unit = i == t ? qa + qv[x] + qv[y] + 126 + s1.s : unit;
        const __int128 sum = warp_rs_i128<NP>(s, lane);
        mine = i128_to_f64(sum, unit);
        bool kept = i != 0 || keeps_bits(sum, cnt, 62, s0);
#pragma unroll
        for (int x = 0, t = 1 + D; x < D; t += D - x, ++x)
          kept = kept && (i != t || !moves[x] || keeps_bits(sum, cnt, 60, s1));
        fixed = __all_sync(0xffffffffu, kept);
        if (D == 3) {
#pragma unroll
          for (int x = 0; x < D; ++x)
#pragma unroll
            for (int y = x + 1; y < D; ++y) {
              const int q = x + y - 1;
              const long long m = (long long)__reduce_add_sync(0xffffffffu, mag[q] >> 5) << 37;
              fixed = fixed && (!moves[x] || !moves[y] || keeps_bits(m, cnt, 60, s1));
            }
        }
      }
      if (!fixed) {
        double acc[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i] = 0.0;
        for (int q = lane; q < cnt; q += 32) {
          const double a = al[q];
          acc[0] += a;
          if (vj) {
            double vv[D];
#pragma unroll
            for (int d = 0; d < D; ++d) vv[d] = to_f64(vj[(int64_t)d * n + q]);
            int t = 1 + D;
#pragma unroll
            for (int x = 0; x < D; ++x) {
              const double ax = a * vv[x];
              acc[1 + x] += ax;
#pragma unroll
              for (int y = x; y < D; ++y, ++t) acc[t] = fma(ax, vv[y], acc[t]);
            }
          }
        }
        warp_rs_d<NP>(acc, lane);
        mine = acc[0];
      }
      mine = __shfl_sync(0xffffffffu, mine, warp_rs_lane<NP>(lane & (NP - 1)));
      tot.add(mine, c0 == first);
    }
    if (big) {
      if (lane < NS) {
        parts[wid][lane][0] = tot.s;
        parts[wid][lane][1] = tot.e;
      }
      __syncthreads();
      if (wid == 0 && lane < NS)
        for (int q = 1; q < NW; ++q) {
          tot.add(parts[q][lane][0], false);
          tot.e += parts[q][lane][1];
        }
      __syncthreads();
      if (wid != 0) continue;
    }
    const double mine = tot.value();
    if (W && lane == 0) W[jc] = mine;
    if (p && lane >= 1 && lane <= D) p[jc * D + lane - 1] = mine;
    if (M2 && lane > D && lane < NS) M2[jc * NM + lane - 1 - D] = mine;
    if (E) {
      double tr = __shfl_sync(0xffffffffu, mine, 1 + D);
      if (D == 3)
        tr = (tr + __shfl_sync(0xffffffffu, mine, 7 < NS ? 7 : 0)) + __shfl_sync(0xffffffffu, mine, 9 < NS ? 9 : 0);
      if (lane == 0) E[jc] = 0.5 * tr;
    }
  }
}

// the same moments of the mixtures (one thread per cell)
template <int D>
__global__ void mixture_moments_kernel(int64_t C, int Kmax, const int32_t* K, const double* prm,
                                       const double* Wc, double* W, double* p, double* M2,
                                       double* E) {
  constexpr int NM = D * (D + 1) / 2;
  constexpr int P = 1 + D + NM;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < C;
       j += (int64_t)gridDim.x * blockDim.x) {
    double pm[D], m2[NM];
    for (int a = 0; a < D; ++a) pm[a] = 0.0;
    for (int t = 0; t < NM; ++t) m2[t] = 0.0;
    const double w = Wc[j];
    for (int k = 0; k < K[j]; ++k) {
      const double* r = prm + ((size_t)j * Kmax + k) * P;
      int t = 0;
      for (int a = 0; a < D; ++a) {
        pm[a] += w * r[0] * r[1 + a];
        for (int b = a; b < D; ++b, ++t) m2[t] += w * r[0] * (r[1 + D + t] + r[1 + a] * r[1 + b]);
      }
    }
    if (W) W[j] = w;
    double e = 0.0;
    int t = 0;
    for (int a = 0; a < D; ++a) {
      if (p) p[j * D + a] = pm[a];
      for (int b = a; b < D; ++b, ++t) {
        if (a == b) e += 0.5 * m2[t];
        if (M2) M2[j * NM + t] = m2[t];
      }
    }
    if (E) E[j] = e;
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int grid_for(int64_t C, int cap) { return (int)(C < cap ? (C > 0 ? C : 1) : cap); }

cudaError_t launch_deposit(int64_t C, const int64_t* cell_off, const double* x,
                           const double* alpha, double dx, double q, int order, void* ws,
                           double* rho, cudaStream_t s) {
  if (C == 0) return cudaSuccess;
  long long* rec = (long long*)ws;
  deposit_partials_kernel<4><<<grid_for((C + 3) / 4, 152 * 16), 128, 0, s>>>(C, cell_off, x, alpha,
                                                                              1.0 / dx, order, rec);
  deposit_combine_kernel<<<grid_for((C + 255) / 256, 1024), 256, 0, s>>>(C, rec, order, q / dx, rho);
  return cudaGetLastError();
}

cudaError_t launch_deposit_combine(int64_t C, double dx, double q, int order, const void* ws,
                                   double* rho, cudaStream_t s) {
  if (C == 0) return cudaSuccess;
  deposit_combine_kernel<<<grid_for((C + 255) / 256, 1024), 256, 0, s>>>(C, (const long long*)ws, order,
                                                                          q / dx, rho);
  return cudaGetLastError();
}

cudaError_t launch_moments(int D, int64_t C, int64_t n, const int64_t* cell_off, const void* v,
                           int v_f64, const double* alpha, double* W, double* p, double* M2,
                           double* E, cudaStream_t s) {
  if (C == 0) return cudaSuccess;
  constexpr int NW = 4;
  // a CTA per cell as long as that leaves no more than a few on an SM
  const int g = C <= 152 * 4 ? (int)C : grid_for((C + NW - 1) / NW, 152 * 16);
  if (D == 1) {
    if (v_f64)
      moments_kernel<1, NW, double><<<g, NW * 32, 0, s>>>(C, n, cell_off, (const double*)v, alpha, W, p, M2, E);
    else
      moments_kernel<1, NW, float><<<g, NW * 32, 0, s>>>(C, n, cell_off, (const float*)v, alpha, W, p, M2, E);
  } else {
    if (v_f64)
      moments_kernel<3, NW, double><<<g, NW * 32, 0, s>>>(C, n, cell_off, (const double*)v, alpha, W, p, M2, E);
    else
      moments_kernel<3, NW, float><<<g, NW * 32, 0, s>>>(C, n, cell_off, (const float*)v, alpha, W, p, M2, E);
  }
  return cudaGetLastError();
}

cudaError_t launch_mixture_moments(int D, int64_t C, int Kmax, const int32_t* K, const double* prm,
                                   const double* Wc, double* W, double* p, double* M2, double* E,
                                   cudaStream_t s) {
  if (C == 0) return cudaSuccess;
  const int g = grid_for((C + 127) / 128, 4096);
  if (D == 1)
    mixture_moments_kernel<1><<<g, 128, 0, s>>>(C, Kmax, K, prm, Wc, W, p, M2, E);
  else
    mixture_moments_kernel<3><<<g, 128, 0, s>>>(C, Kmax, K, prm, Wc, W, p, M2, E);
  return cudaGetLastError();
}

}  // namespace gmcr
