// BF16 population storage with FP32 arithmetic (round to nearest / stochastic).
#include "band.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(float, BF16<false>)
BTRIRT_INSTANTIATE_TILE(float, BF16<false>)
BTRIRT_INSTANTIATE_BATCH_TILE(BF16<false>)
BTRIRT_INSTANTIATE_BATCH_BAND(BF16<false>)
BTRIRT_INSTANTIATE(float, BF16<true>)
BTRIRT_INSTANTIATE_TILE(float, BF16<true>)
BTRIRT_INSTANTIATE_BATCH_TILE(BF16<true>)
BTRIRT_INSTANTIATE_BATCH_BAND(BF16<true>)
}  // namespace btrirt
