// FP32 pass kernels of radius 4.
#include "pass_fp32.cuh"

namespace rpiv {

RPIV_PASS_RADIUS(4)

}  // namespace rpiv
