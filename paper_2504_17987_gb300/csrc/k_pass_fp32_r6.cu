// FP32 pass kernels of radius 6.
#include "pass_fp32.cuh"

namespace rpiv {

RPIV_PASS_RADIUS(6)

}  // namespace rpiv
