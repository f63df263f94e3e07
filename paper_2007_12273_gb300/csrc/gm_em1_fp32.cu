// gm_em1_fp32.cu -- the EM kernel for D = 1 with the FP32 M-step.
#include "em_launch.cuh"

namespace gmcr {
GM_EM_DEFINE(1, float)
}  // namespace gmcr
