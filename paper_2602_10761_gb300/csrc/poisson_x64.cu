// The x transforms in FP64.
#include "poisson_xpass.cuh"

namespace tribo {
TRIBO_XPASS_INSTANTIATE(double)
}  // namespace tribo
