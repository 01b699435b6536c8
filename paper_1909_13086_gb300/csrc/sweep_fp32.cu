// FP32 storage and arithmetic instantiation of the fused sweep.
#include "tile.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(float, float)
BTRIRT_INSTANTIATE_TILE(float, float)
}  // namespace btrirt
