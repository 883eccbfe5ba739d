// FP32 pass kernels of radius 1.
#include "pass_fp32.cuh"

namespace rpiv {

RPIV_PASS_RADIUS(1)

}  // namespace rpiv
