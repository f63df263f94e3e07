// em_launch.cuh -- launch of one EM kernel instantiation (em_kernel<D, R>).
// Each is compiled in a translation unit of its own (gm_em<D>_fp<bits>.cu)
// so that the library's heaviest kernels build in parallel; gm_em.cu picks
// the instantiation and the launch shape.
#pragma once

#include "gm_kernels.cuh"

namespace gmcr {

struct EmShape {
  int teams, team, grid;  // teams of a CTA, threads of a team, CTAs
};

template <int D, typename R>
size_t em_ctl_size();
template <int D, typename R>
cudaError_t em_go(const EmParams& p, const EmShape& sh, size_t smem, cudaStream_t s);

#define GM_EM_DECLARE(D, R)                                                                    \
  template <>                                                                                  \
  size_t em_ctl_size<D, R>();                                                                  \
  template <>                                                                                  \
  cudaError_t em_go<D, R>(const EmParams& p, const EmShape& sh, size_t smem, cudaStream_t s);
GM_EM_DECLARE(1, float)
GM_EM_DECLARE(1, double)
GM_EM_DECLARE(3, float)
GM_EM_DECLARE(3, double)

#define GM_EM_DEFINE(D, R)                                                                     \
  template <>                                                                                  \
  size_t em_ctl_size<D, R>() {                                                                 \
    return em_ctl_bytes<D, R>();                                                               \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t em_go<D, R>(const EmParams& p, const EmShape& sh, size_t smem, cudaStream_t s) { \
    auto k = em_kernel<D, R>;                                                                  \
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    if (e != cudaSuccess) return e;                                                            \
    k<<<sh.grid, sh.teams * sh.team, smem, s>>>(p);                                            \
    return cudaGetLastError();                                                                 \
  }

}  // namespace gmcr
