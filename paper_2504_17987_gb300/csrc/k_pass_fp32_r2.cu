// FP32 pass kernels of radii 2 and 3.
#include "pass_fp32.cuh"

namespace rpiv {

RPIV_PASS_RADIUS(2)
RPIV_PASS_RADIUS(3)

}  // namespace rpiv
