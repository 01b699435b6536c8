// FP64 storage and arithmetic instantiation of the fused sweep (parity path).
#include "tile.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(double, double)
BTRIRT_INSTANTIATE_TILE(double, double)
}  // namespace btrirt
