// The x transforms in FP32 (mixed precision).
#include "poisson_xpass.cuh"

namespace tribo {
TRIBO_XPASS_INSTANTIATE(float)
}  // namespace tribo
