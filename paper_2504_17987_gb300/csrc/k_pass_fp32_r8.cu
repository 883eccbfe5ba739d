// FP32 pass kernels of radius 8.
#include "pass_fp32.cuh"

namespace rpiv {

RPIV_PASS_RADIUS(8)

}  // namespace rpiv
