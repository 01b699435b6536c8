// FP32 storage and arithmetic instantiation of the fused sweep.
#include "band.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(float, float)
BTRIRT_INSTANTIATE_TILE(float, float)
BTRIRT_INSTANTIATE_BATCH_TILE(float)
BTRIRT_INSTANTIATE_BATCH_BAND(float)
BTRIRT_INSTANTIATE_BAND(float)
}  // namespace btrirt
