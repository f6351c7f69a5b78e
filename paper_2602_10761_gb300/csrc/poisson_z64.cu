// The z transforms in FP64.
#include "poisson_zpass.cuh"

namespace tribo {
TRIBO_ZPASS_INSTANTIATE(double)
}  // namespace tribo
