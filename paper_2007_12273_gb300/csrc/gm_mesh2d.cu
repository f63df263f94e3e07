// gm_mesh2d.cu -- the reconstruction on a 2D doubly periodic mesh (Sec. 2.4
// with the tensor-product shape function S(x) S(y), the geometry of the
// 2D-3V Weibel runs of Sec. 3.2).  Cells and nodes are numbered
// j = jy Cx + jx; node (ix, iy) sits at the cell centre.
//
// Sampling, the per-cell velocity sums and the Lemons projection are those
// of the 1D path (recon_sampler.cuh), with one more uniform per particle for
// y.  The mass matrix M_ij = q sum_{p in j} S(x_i - x_p) S(y_i - y_p) has a
// 3 x 3 column per cell.  With the quadratic B-spline it is not diagonally
// dominant in 2D (a uniformly filled cell keeps (2/3)^2 of its weight on
// its own node), so M dA = dx dy (rho' - rho) is solved by defect
// correction with the operator of uniformly filled cells as preconditioner:
// P = (Tx (x) Ty) diag(q N'_j), T the circulant tridiagonal matrix of the
// mean shape weights (e, d0, e) = (1/6, 2/3, 1/6); CIC (1/8, 3/4, 1/8).
// T^-1 is circulant with entries c_k = (r^k + r^(n-k)) / ((1 - r^n) s),
// s = sqrt(d0^2 - 4 e^2), r = (s - d0) / (2 e) (r = -(2 - sqrt 3) for the
// quadratic B-spline: the images of the bi-infinite inverse), so P^-1 is a
// convolution along every row and then every column: all n entries for
// lines of at most 33 cells, else the 33 central ones (the first one left
// out is below 2e-10 of c_0; the residual is always formed with the true M,
// so the preconditioner's truncation changes the rate, not the solution).
// Each iteration is a residual pass, an x pass and a y pass over the nodes,
// separated by grid barriers inside one cooperative launch.  A cell
// without resampled particles has a unit column: its unknown appears in its
// own row only, so it is left out of the iteration and found afterwards
// from its row.
#include "recon_sampler.cuh"

namespace gmcr {

// shape weights of an in-cell offset s = u - 1/2 on the nodes -1, 0, +1 of
// its cell (the B-spline S(a - s)): quadratic (1/2 - s)^2 / 2, 3/4 - s^2,
// (1/2 + s)^2 / 2; CIC max(-s, 0), 1 - |s|, max(s, 0)
__device__ __forceinline__ void shape3(int order, double s, double (&w)[3]) {
  if (order == 1) {
    w[0] = s < 0.0 ? -s : 0.0;
    w[2] = s > 0.0 ? s : 0.0;
    w[1] = 1.0 - (w[0] + w[2]);
  } else {
    const double a = 0.5 - s, b = 0.5 + s;
    w[0] = 0.5 * a * a;
    w[1] = 0.75 - s * s;
    w[2] = 0.5 * b * b;
  }
}

// part[j][3 (b + 1) + (a + 1)] = sum_{p in j} alpha_p S(x-weight a) S(y-weight b):
// what cell j's particles put on node (jx + a, jy + b).  One warp per cell;
// alpha = NULL means unit weights.
template <int NW>
__global__ void __launch_bounds__(NW * 32) deposit2d_partials_kernel(
    int64_t Cx, int64_t C, const int64_t* cell_off, const double* x, const double* y,
    const double* alpha, double inv_dx, double inv_dy, int order, double* part) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t j = (int64_t)blockIdx.x * NW + wid; j < C; j += (int64_t)gridDim.x * NW) {
    const int64_t jx = j % Cx, jy = j / Cx;
    const int64_t o = cell_off[j], n = cell_off[j + 1] - o;
    double acc[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[t] = 0.0;
    for (int64_t p = lane; p < n; p += 32) {
      double wx[3], wy[3];
      shape3(order, cell_frac(x[o + p], (double)jx, inv_dx) - 0.5, wx);
      shape3(order, cell_frac(y[o + p], (double)jy, inv_dy) - 0.5, wy);
      const double al = alpha ? alpha[o + p] : 1.0;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const double ab = al * wy[b];
#pragma unroll
        for (int a = 0; a < 3; ++a) acc[3 * b + a] = fma(ab, wx[a], acc[3 * b + a]);
      }
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[t] = warp_sum(acc[t]);
    if (lane == 0)
#pragma unroll
      for (int t = 0; t < 9; ++t) part[9 * j + t] = acc[t];
  }
}

// the cell whose entry (a, b) lands on node (ix, iy): (ix - a, iy - b), periodic
__device__ __forceinline__ int64_t src_cell(int64_t ix, int64_t iy, int a, int b, int64_t Cx,
                                            int64_t Cy) {
  int64_t sx = ix - a, sy = iy - b;
  sx = sx < 0 ? sx + Cx : (sx >= Cx ? sx - Cx : sx);
  sy = sy < 0 ? sy + Cy : (sy >= Cy ? sy - Cy : sy);
  return sy * Cx + sx;
}

// rho_i = q / (dx dy) sum over the 3 x 3 cells around node i of their entry on it
__global__ void deposit2d_combine_kernel(int64_t Cx, int64_t Cy, const double* part,
                                         double q_over_dv, double* rho) {
  const int64_t C = Cx * Cy;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < C;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ix = i % Cx, iy = i / Cx;
    double s = 0.0;
    for (int b = -1; b <= 1; ++b)
      for (int a = -1; a <= 1; ++a) s += part[9 * src_cell(ix, iy, a, b, Cx, Cy) + 3 * (b + 1) + (a + 1)];
    rho[i] = q_over_dv * s;
  }
}

// Position sums of the 2D mesh (the first 8 sums of RecRaw<D, 8>), s_x and
// s_y the particle's offsets from the cell centre:
//   quadratic B-spline: sum of s_x, s_y (units of 2^-53), s_x^2, s_y^2, s_x s_y,
//     s_x^2 s_y, s_x s_y^2, s_x^2 s_y^2 (2^-54): every S(x) S(y) is a
//     combination of them;
//   CIC, a = max(-s, 0), b = max(s, 0): sum of a_x, b_x, a_y, b_y (2^-53),
//     a_x a_y, b_x a_y, a_x b_y, b_x b_y (2^-54).
// The products are taken to 2^-64 (high halves of 64 x 64-bit products) and
// rounded to 2^-54 each, so that a lane's 512 terms fit in 64 bits; FP64 sums
// of this size carry 2^-48.  A cell that takes FP64 sums has the 9 shape
// sums in words 0 .. 8 and the sums of w and |w|^2 in words 9 .. 9 + D.
constexpr int kPos2d = 8;
__device__ __forceinline__ long long mulhi64(long long a, long long b) { return __mul64hi(a, b); }
__device__ __forceinline__ long long to_2m54(long long v) { return (v + 512) >> 10; }  // from 2^-64

// Pass 1, one warp per cell: draws every particle once, stages the draw in
// its output slots and sums it (RecRaw).  On the integer pipe throughout:
// with the shape weights, their 9 products and w in FP64 the pass took 32 FP64
// instructions a particle, each 19 cycles of the SM's pipe.
template <int D, int NW>
__global__ void __launch_bounds__(NW * 32) recon2d_stats_kernel(
    int64_t C, int Kmax, const RecHead<D>* head, const RecComp<D>* comp, const int64_t* out_off,
    int64_t n_out, uint64_t seed, int order, RecRaw<D, kPos2d>* raw, double* x_out, double* y_out,
    double* v_out, double* alpha_out) {
  constexpr int NS = kPos2d + 2 * D;
  constexpr int NV = 9 + D + 1;
  __shared__ RecCell<D> rcs[NW];
  __shared__ long long dzqs[NW][kMaxK][D];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  RecCell<D>& rc = rcs[wid];
  for (int64_t j = (int64_t)blockIdx.x * NW + wid; j < C; j += (int64_t)gridDim.x * NW) {
    load_prepped<D>(rc, j, Kmax, head, comp, lane);
    __syncwarp();
    int64_t o, n;
    out_range(out_off, j, n_out, o, n);
    RecRaw<D, kPos2d>& rw = raw[j];
    int eq[D];
    if (fix_plan<D>(rc, n, lane, eq, dzqs[wid])) {
      const bool several = rc.K > 1;
      long long sp[kPos2d], sf[D];
      SplitSum sq[D];
#pragma unroll
      for (int t = 0; t < kPos2d; ++t) sp[t] = 0;
#pragma unroll
      for (int d = 0; d < D; ++d) sf[d] = 0;
      for (int64_t i = lane; i < n; i += 32) {
        uint64_t m0;
        int z;
        float f[D];
        sample_f<D>(rc, j, i, seed, m0, z, f);
        const uint64_t my = sample_y_bits(j, i, seed);
        stage_draw<D>(x_out, v_out, alpha_out, o + i, m0, z, f);
        reinterpret_cast<unsigned long long*>(y_out)[o + i] = my;
        const long long kx = 2ll * (long long)m0 - (1ll << 52) + 1ll;
        const long long ky = 2ll * (long long)my - (1ll << 52) + 1ll;
        if (order == 1) {
          const bool xp = kx > 0, yp = ky > 0;
          const long long ax = xp ? kx : -kx, ay = yp ? ky : -ky;
          const long long r = to_2m54(mulhi64(ax << 11, ay << 11));
          sp[0] += xp ? 0 : ax;
          sp[1] += xp ? ax : 0;
          sp[2] += yp ? 0 : ay;
          sp[3] += yp ? ay : 0;
          sp[4] += !xp && !yp ? r : 0;
          sp[5] += xp && !yp ? r : 0;
          sp[6] += !xp && yp ? r : 0;
          sp[7] += xp && yp ? r : 0;
        } else {
          const long long X = kx << 11, Y = ky << 11;  // s in units of 2^-64
          const long long xx = mulhi64(X, X), yy = mulhi64(Y, Y);
          sp[0] += kx;
          sp[1] += ky;
          sp[2] += to_2m54(xx);
          sp[3] += to_2m54(yy);
          sp[4] += to_2m54(mulhi64(X, Y));
          sp[5] += to_2m54(mulhi64(xx, Y));
          sp[6] += to_2m54(mulhi64(X, yy));
          sp[7] += to_2m54(mulhi64(xx, yy));
        }
#pragma unroll
        for (int d = 0; d < D; ++d) {
          long long fq = fixq(f[d], eq[d]);
          if (several) fq += dzqs[wid][z][d];
          sf[d] += fq;
          sq[d].add_square(SplitInt(fq));
        }
      }
      __int128 sm[NS];
#pragma unroll
      for (int t = 0; t < kPos2d; ++t) sm[t] = (__int128)sp[t];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        sm[kPos2d + d] = (__int128)sf[d];
        sm[kPos2d + D + d] = sq[d].total_square();
      }
      put_fixed<D, kPos2d>(rw, sm, eq, lane);
    } else {
      double acc[NV];
#pragma unroll
      for (int t = 0; t < NV; ++t) acc[t] = 0.0;
      for (int64_t i = lane; i < n; i += 32) {
        uint64_t m0;
        int z;
        float f[D];
        double w[D], wx[3], wy[3];
        sample_f<D>(rc, j, i, seed, m0, z, f);
        const uint64_t my = sample_y_bits(j, i, seed);
        stage_draw<D>(x_out, v_out, alpha_out, o + i, m0, z, f);
        reinterpret_cast<unsigned long long*>(y_out)[o + i] = my;
        draw_offset<D>(rc, z, f, w);
        shape3(order, centred52(m0), wx);
        shape3(order, centred52(my), wy);
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int a = 0; a < 3; ++a) acc[3 * b + a] = fma(wy[b], wx[a], acc[3 * b + a]);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          acc[9 + d] += w[d];
          acc[9 + D] = fma(w[d], w[d], acc[9 + D]);
        }
      }
#pragma unroll
      for (int t = 0; t < NV; ++t) acc[t] = warp_sum(acc[t]);
      if (lane == 0) {
#pragma unroll
        for (int t = 0; t < NV; ++t) rw.w[t] = acc[t];
        rw.fixed = 0;
      }
    }
    __syncwarp();
  }
}

// one thread per cell: cstat[j] = [the 9 unit-weight shape sums (layout of
// part above), sum w (D), sum |w|^2] from the cell's record
template <int D>
__global__ void recon2d_sums_kernel(int64_t C, int Kmax, const RecHead<D>* head, const RecComp<D>* comp,
                                    const RecRaw<D, kPos2d>* raw, const int64_t* out_off, int64_t n_out,
                                    int order, double* cstat) {
  constexpr int NV = 9 + D + 1;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < C;
       j += (int64_t)gridDim.x * blockDim.x) {
    const RecRaw<D, kPos2d>& r = raw[j];
    double* cs = cstat + (size_t)j * NV;
    if (!r.fixed) {
      for (int t = 0; t < NV; ++t) cs[t] = r.w[t];
      continue;
    }
    const int64_t n = out_count(out_off, j, n_out);
    const double nd = (double)n;
    double p[kPos2d];
#pragma unroll
    for (int t = 0; t < kPos2d; ++t) p[t] = i128_to_f64(load_i128(&r.w[2 * t]), t < (order == 1 ? 4 : 2) ? -53 : -54);
    if (order == 1) {
      cs[0] = p[4];
      cs[2] = p[5];
      cs[6] = p[6];
      cs[8] = p[7];
      cs[1] = p[2] - (p[4] + p[5]);
      cs[7] = p[3] - (p[6] + p[7]);
      cs[3] = p[0] - (p[4] + p[6]);
      cs[5] = p[1] - (p[5] + p[7]);
      cs[4] = (nd - (p[0] + p[1])) - (cs[1] + cs[7]);
    } else {
      // weights of the nodes -1, 0, +1: 1/8 -+ s/2 + s^2/2, 3/4 - s^2; first
      // along x (rows: y moments 0, 1, 2), then along y
      const double m[3][3] = {{nd, p[0], p[2]}, {p[1], p[4], p[5]}, {p[3], p[6], p[7]}};
      double h[3][3];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const double e = 0.5 * (0.25 * m[b][0] + m[b][2]);
        h[b][0] = e - 0.5 * m[b][1];
        h[b][1] = 0.75 * m[b][0] - m[b][2];
        h[b][2] = e + 0.5 * m[b][1];
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double e = 0.5 * (0.25 * h[0][a] + h[2][a]);
        cs[a] = e - 0.5 * h[1][a];
        cs[3 + a] = 0.75 * h[0][a] - h[2][a];
        cs[6 + a] = e + 0.5 * h[1][a];
      }
    }
    double sw[D + 1];
    velocity_sums<D, kPos2d>(r, head[j].K, comp[(size_t)j * Kmax], n, sw);
#pragma unroll
    for (int t = 0; t <= D; ++t) cs[9 + t] = sw[t];
  }
}

// order-preserving bits of a non-negative double (for atomicMax)
__device__ __forceinline__ unsigned long long pos_bits(double v) {
  return (unsigned long long)__double_as_longlong(v);
}

constexpr int kCircTaps = 33;  // entries of T^-1 kept per direction
constexpr int kCircHalf = 16;  // window half-width for lines of more than kCircTaps cells

struct Mesh2dSolve {
  int64_t Cx, Cy;
  const double* cstat;   // [C][NV]
  int nv;                // 9 + D + 1
  const int64_t* out_off;
  int64_t n_out;
  double q;
  double* b;             // [C] right-hand side dx dy (rho' - rho)
  double* dA;            // [C]
  double* r;             // [C] residual
  double* t;             // [C] after the x sweep
  unsigned long long* norm;  // [max_iter + 1] max |r| per iteration (as bits)
  unsigned long long* scale; // [1] max |dx dy rho'| (as bits)
  unsigned int* arrived;     // [1] the solve's grid barrier (zero at the launch)
  double tol;
};

// rows of the right-hand side, dA = 0
__global__ void assemble2d_kernel(Mesh2dSolve m, const double* W, const double* rho_target,
                                  double dv) {
  const int64_t C = m.Cx * m.Cy;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < C;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ix = i % m.Cx, iy = i / m.Cx;
    double s = 0.0;
    for (int b = -1; b <= 1; ++b)
      for (int a = -1; a <= 1; ++a) {
        const int64_t src = src_cell(ix, iy, a, b, m.Cx, m.Cy);
        const int64_t ns = out_count(m.out_off, src, m.n_out);
        if (ns > 0) s += (W[src] / (double)ns) * m.cstat[(size_t)src * m.nv + 3 * (b + 1) + (a + 1)];
      }
    const double tgt = dv * rho_target[i];
    m.b[i] = tgt - m.q * s;
    m.dA[i] = 0.0;
    atomicMax(m.scale, pos_bits(fabs(tgt)));
  }
}

// entries of T^-1 along one direction (host-computed, passed by value)
struct CircTaps {
  int full;        // 1: all n entries c_0 .. c_{n-1}; 0: c_0 .. c_16 (window)
  double c[kCircTaps];
};

// (T^-1 line)_i for a line of n values at stride st
__device__ __forceinline__ double circ_apply(const CircTaps& T, const double* line, int64_t n,
                                             int64_t i, int64_t st) {
  double s = 0.0;
  if (T.full) {
#pragma unroll
    for (int k = 0; k < kCircTaps; ++k)
      if (k < n) {
        int64_t j = i - k;
        j = j < 0 ? j + n : j;
        s = fma(T.c[k], __ldcg(line + j * st), s);
      }
    return s;
  }
  s = T.c[0] * __ldcg(line + i * st);
#pragma unroll
  for (int k = 1; k <= kCircHalf; ++k) {
    int64_t jm = i - k, jp = i + k;
    jm = jm < 0 ? jm + n : jm;
    jp = jp >= n ? jp - n : jp;
    s = fma(T.c[k], __ldcg(line + jm * st) + __ldcg(line + jp * st), s);
  }
  return s;
}

// all CTAs of the cooperative grid: phase p (0, 1, ..) ends when every CTA has
// arrived p + 1 times.  False if that takes more than about a second.
__device__ __forceinline__ bool grid_barrier(unsigned int* arrived, unsigned int phase) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrived, 1u);
    const unsigned int want = (phase + 1u) * gridDim.x;
    ok = 0;
    for (int it = 0; it < (1 << 22); ++it) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
      if (v >= want) {
        ok = 1;
        break;
      }
      __nanosleep(100);
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// the sum of row i over the cells with particles
__device__ __forceinline__ double mm2d_row(const Mesh2dSolve& m, int64_t i) {
  const int64_t ix = i % m.Cx, iy = i / m.Cx;
  double s = 0.0;
  for (int b = -1; b <= 1; ++b)
    for (int a = -1; a <= 1; ++a) {
      const int64_t src = src_cell(ix, iy, a, b, m.Cx, m.Cy);
      if (out_count(m.out_off, src, m.n_out) > 0)
        s = fma(m.cstat[(size_t)src * m.nv + 3 * (b + 1) + (a + 1)], __ldcg(m.dA + src), s);
    }
  return s;
}

// The whole solve in one cooperative launch, one thread per node (strided on
// large meshes).  An iteration's work is small (9 + 66 FP64 operations per
// node: 2 us over the GPU for 16384 nodes) against the launches it took as
// three kernels, and launching the rest of the iterations after convergence
// cost as much again: 16384 cells of 512 particles, 10 iterations of at most
// 64, reconstruct in 2.02 ms with 193 launches and FP64 sums, in 0.58 ms with
// this kernel (0.16 ms) and the integer sums.  CTAs of 64 threads spread the FP64 work of a
// small mesh over the SMs.
constexpr int kSolveThreads = 64;
__global__ void __launch_bounds__(kSolveThreads) mm2d_solve_kernel(Mesh2dSolve m, CircTaps tx, CircTaps ty,
                                                                  int max_iter, int* converged) {
  __shared__ unsigned long long red[kSolveThreads / 32];
  const double thr = m.tol * __longlong_as_double((long long)*m.scale);
  const int64_t C = m.Cx * m.Cy, step = (int64_t)gridDim.x * kSolveThreads;
  const int64_t i0 = blockIdx.x * (int64_t)kSolveThreads + threadIdx.x;
  unsigned int phase = 0;
  int conv = 0;
  for (int it = 0;; ++it) {
    // r_i = b_i - (M dA)_i on the rows of cells with particles (empty rows 0)
    // (the largest |r| by its bits, in which NaN lies above infinity)
    unsigned long long mx = 0ull;
    for (int64_t i = i0; i < C; i += step) {
      const double ri = out_count(m.out_off, i, m.n_out) > 0 ? m.b[i] - m.q * mm2d_row(m, i) : 0.0;
      m.r[i] = ri;
      mx = max(mx, pos_bits(fabs(ri)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 1; q < kSolveThreads / 32; ++q) mx = max(mx, red[q]);
      atomicMax(m.norm + it, mx);
    }
    if (!grid_barrier(m.arrived, phase++)) break;
    const double norm = __longlong_as_double((long long)__ldcg(m.norm + it));
    conv = isfinite(norm) && norm <= thr;
    if (conv || it == max_iter) break;
    // t = (Tx^-1 along every row) r
    for (int64_t i = i0; i < C; i += step) {
      const int64_t ix = i % m.Cx, row = i - ix;
      m.t[i] = circ_apply(tx, m.r + row, m.Cx, ix, 1);
    }
    if (!grid_barrier(m.arrived, phase++)) break;
    // dA_j += (Ty^-1 along every column of t)_j / (q N'_j) on cells with particles
    for (int64_t i = i0; i < C; i += step) {
      const int64_t n = out_count(m.out_off, i, m.n_out);
      if (n == 0) continue;
      const int64_t ix = i % m.Cx, iy = i / m.Cx;
      m.dA[i] = __ldcg(m.dA + i) + circ_apply(ty, m.t + ix, m.Cy, iy, m.Cx) / (m.q * (double)n);
    }
    if (!grid_barrier(m.arrived, phase++)) break;
  }
  // the unknowns of empty cells from their own rows (unit diagonal); they
  // enter no other row
  for (int64_t i = i0; i < C; i += step)
    if (out_count(m.out_off, i, m.n_out) == 0) m.dA[i] = m.b[i] - m.q * mm2d_row(m, i);
  if (i0 == 0) *converged = conv;
}

// the entries of T^-1 for a periodic line of n cells (closed form above)
static CircTaps circ_taps(int64_t n, double e, double d0) {
  CircTaps T;
  const double sq = sqrt(d0 * d0 - 4.0 * e * e), r = (sq - d0) / (2.0 * e);
  const double rn = pow(r, (double)n);
  T.full = n <= kCircTaps ? 1 : 0;
  const int cnt = T.full ? (int)n : kCircHalf + 1;
  for (int k = 0; k < kCircTaps; ++k) T.c[k] = 0.0;
  for (int k = 0; k < cnt; ++k)
    T.c[k] = (pow(r, (double)k) + pow(r, (double)(n - k))) / ((1.0 - rn) * sq);
  return T;
}

// one thread per cell: the projection coefficients and the cell's status
template <int D>
__global__ void recon2d_coeffs_kernel(int64_t C, int Kmax, const RecHead<D>* head, const RecComp<D>* comp,
                                      const double* cstat, const int64_t* out_off, int64_t n_out,
                                      const double* W, const double* dA, const int* converged,
                                      RecCoef<D>* coef, uint32_t* status_out) {
  constexpr int NV = 9 + D + 1;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < C;
       j += (int64_t)gridDim.x * blockDim.x) {
    int64_t o, n;
    const bool in_range = out_range(out_off, j, n_out, o, n);
    const RecHead<D> h = head[j];
    const ProjCoef<D> pc = proj_coeffs<D>(h.K, h.u, h.theta, n, W[j], dA[j], cstat + (size_t)j * NV + 9);
    coef[j] = make_coef<D>(pc, h, comp[(size_t)j * Kmax]);
    status_out[j] = pc.status | (*converged ? 0u : GM_ST_MM_NOT_CONVERGED) | (in_range ? 0u : GM_ST_BAD_RANGE);
  }
}

// ---------------------------------------------------------------------------
static int grid_cap(int64_t units, int per, int cap) {
  const int64_t g = (units + per - 1) / per;
  return (int)(g < 1 ? 1 : (g < cap ? g : cap));
}

cudaError_t launch_deposit2d(int64_t Cx, int64_t Cy, const int64_t* cell_off, const double* x,
                             const double* y, const double* alpha, double dx, double dy, double q,
                             int order, double* part, double* rho, cudaStream_t s) {
  const int64_t C = Cx * Cy;
  if (C == 0) return cudaSuccess;
  deposit2d_partials_kernel<4><<<grid_cap(C, 4, 152 * 16), 128, 0, s>>>(
      Cx, C, cell_off, x, y, alpha, 1.0 / dx, 1.0 / dy, order, part);
  deposit2d_combine_kernel<<<grid_cap(C, 256, 1024), 256, 0, s>>>(Cx, Cy, part, q / (dx * dy), rho);
  return cudaGetLastError();
}

// workspace: FP64 arrays (the per-cell sums, right-hand side, dA, residual and
// sweep arrays, the norms, the scale and the barrier's counter), then the
// records, the mixture heads and components and the coefficients
struct Ws2d {
  size_t head, comp, coef, raw, total;
};
template <int D>
static Ws2d ws2d(int64_t C, int Kmax) {
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  Ws2d w;
  w.raw = up(((size_t)(9 + D + 1) * C + 4 * (size_t)C + (kMesh2dMaxIter + 1) + 3) * sizeof(double));
  w.head = w.raw + up((size_t)C * sizeof(RecRaw<D, kPos2d>));
  w.comp = w.head + up((size_t)C * sizeof(RecHead<D>));
  w.coef = w.comp + up((size_t)C * Kmax * sizeof(RecComp<D>));
  w.total = w.coef + up((size_t)C * sizeof(RecCoef<D>));
  return w;
}

size_t reconstruct2d_ws_bytes(int D, int64_t Cx, int64_t Cy, int Kmax) {
  return D == 1 ? ws2d<1>(Cx * Cy, Kmax).total : ws2d<3>(Cx * Cy, Kmax).total;
}

template <int D>
static cudaError_t recon2d_passes(int64_t Cx, int64_t Cy, int Kmax, const int32_t* K, const double* prm,
                                  const double* W, const double* rho_target, int64_t n_out,
                                  const int64_t* out_off, uint64_t seed, double dx, double dy, double q,
                                  int order, double* x_out, double* y_out, double* v_out,
                                  double* alpha_out, uint32_t* status_out, double* dA_user, void* ws,
                                  cudaStream_t s) {
  const int64_t C = Cx * Cy;
  const Ws2d w = ws2d<D>(C, Kmax);
  unsigned char* base = (unsigned char*)ws;
  RecRaw<D, kPos2d>* raw = (RecRaw<D, kPos2d>*)(base + w.raw);
  RecHead<D>* head = (RecHead<D>*)(base + w.head);
  RecComp<D>* comp = (RecComp<D>*)(base + w.comp);
  RecCoef<D>* coef = (RecCoef<D>*)(base + w.coef);
  Mesh2dSolve m;
  m.Cx = Cx;
  m.Cy = Cy;
  m.nv = 9 + D + 1;
  double* cstat = (double*)ws;
  m.cstat = cstat;
  m.out_off = out_off;
  m.n_out = n_out;
  m.q = q;
  m.b = cstat + (size_t)m.nv * C;
  m.dA = m.b + C;
  m.r = m.dA + C;
  m.t = m.r + C;
  m.norm = (unsigned long long*)(m.t + C);
  m.scale = m.norm + kMesh2dMaxIter + 1;
  m.arrived = (unsigned int*)(m.scale + 1);
  int* converged = (int*)(m.scale + 2);
  m.tol = kMesh2dTol;
  if (dA_user) m.dA = dA_user;
  const double e = order == 1 ? 0.125 : 1.0 / 6.0;
  const double d0 = order == 1 ? 0.75 : 2.0 / 3.0;
  CircTaps tx = circ_taps(Cx, e, d0), ty = circ_taps(Cy, e, d0);

  trace_mark(nullptr, s);
  // the norms, the scale and the barrier's counter start at zero
  cudaError_t err = cudaMemsetAsync(m.norm, 0, sizeof(unsigned long long) * (kMesh2dMaxIter + 3), s);
  if (err != cudaSuccess) return err;
  constexpr int NW = 4;
  const int g = grid_cap(C, NW, 152 * 16), gc = grid_cap(C, 128, 2048);
  recon_prep_kernel<D><<<gc, 128, 0, s>>>(C, Kmax, K, prm, head, comp);
  recon2d_stats_kernel<D, NW><<<g, NW * 32, 0, s>>>(C, Kmax, head, comp, out_off, n_out, seed, order, raw,
                                                    x_out, y_out, v_out, alpha_out);
  trace_mark("recon2d_stats_kernel", s);
  recon2d_sums_kernel<D><<<gc, 128, 0, s>>>(C, Kmax, head, comp, raw, out_off, n_out, order, cstat);
  assemble2d_kernel<<<gc, 128, 0, s>>>(m, W, rho_target, dx * dy);
  trace_mark("recon2d_sums_kernel, assemble2d_kernel", s);
  // cooperative: every CTA resident (two of 64 threads per SM always are)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid_cap(C, kSolveThreads, 152 * 2));
  cfg.blockDim = dim3(kSolveThreads);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  err = cudaLaunchKernelEx(&cfg, mm2d_solve_kernel, m, tx, ty, kMesh2dMaxIter, converged);
  if (err != cudaSuccess) return err;
  trace_mark("mm2d_solve_kernel", s);
  recon2d_coeffs_kernel<D><<<gc, 128, 0, s>>>(C, Kmax, head, comp, cstat, out_off, n_out, W, m.dA, converged,
                                              coef, status_out);
  recon_emit_kernel<D, NW, true><<<g, NW * 32, 0, s>>>(C, Kmax, head, comp, coef, out_off, Cx, dx, dy, n_out,
                                                       x_out, y_out, v_out, alpha_out);
  trace_mark("recon_emit_kernel", s);
  return cudaGetLastError();
}

cudaError_t launch_reconstruct2d(int D, int64_t Cx, int64_t Cy, int Kmax, const int32_t* K,
                                 const double* prm, const double* W, const double* rho_target,
                                 int64_t n_out, const int64_t* out_off, uint64_t seed, double dx,
                                 double dy, double q, int order, double* x_out, double* y_out,
                                 double* v_out, double* alpha_out, uint32_t* status_out,
                                 double* dA_user, void* ws, cudaStream_t s) {
  if (Cx * Cy == 0) return cudaSuccess;
  return D == 1 ? recon2d_passes<1>(Cx, Cy, Kmax, K, prm, W, rho_target, n_out, out_off, seed, dx, dy, q,
                                    order, x_out, y_out, v_out, alpha_out, status_out, dA_user, ws, s)
                : recon2d_passes<3>(Cx, Cy, Kmax, K, prm, W, rho_target, n_out, out_off, seed, dx, dy, q,
                                    order, x_out, y_out, v_out, alpha_out, status_out, dA_user, ws, s);
}

}  // namespace gmcr
