// FP32 storage and arithmetic instantiation of the fused sweep.
#include "band.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(float, float)
BTRIRT_INSTANTIATE_TILE(float, float)
BTRIRT_INSTANTIATE_BAND(float)
}  // namespace btrirt
