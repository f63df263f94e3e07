// gm_em1_fp64.cu -- the EM kernel for D = 1 with the FP64 M-step.
#include "em_launch.cuh"

namespace gmcr {
GM_EM_DEFINE(1, double)
}  // namespace gmcr
