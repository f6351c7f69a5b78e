// The z transforms in FP32 (mixed precision).
#include "poisson_zpass.cuh"

namespace tribo {
TRIBO_ZPASS_INSTANTIATE(float)
}  // namespace tribo
