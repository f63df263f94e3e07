// gm_em3_fp64.cu -- the EM kernel for D = 3 with the FP64 M-step.
#include "em_launch.cuh"

namespace gmcr {
GM_EM_DEFINE(3, double)
}  // namespace gmcr
