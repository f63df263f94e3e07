// gm_em3_fp32.cu -- the EM kernel for D = 3 with the FP32 M-step.
#include "em_launch.cuh"

namespace gmcr {
GM_EM_DEFINE(3, float)
}  // namespace gmcr
