// FP16 population storage with FP32 arithmetic (round to nearest / stochastic).
#include "band.cuh"

namespace btrirt {
BTRIRT_INSTANTIATE(float, F16<false>)
BTRIRT_INSTANTIATE_TILE(float, F16<false>)
BTRIRT_INSTANTIATE_BATCH_TILE(F16<false>)
BTRIRT_INSTANTIATE_BATCH_BAND(F16<false>)
BTRIRT_INSTANTIATE(float, F16<true>)
BTRIRT_INSTANTIATE_TILE(float, F16<true>)
BTRIRT_INSTANTIATE_BATCH_TILE(F16<true>)
BTRIRT_INSTANTIATE_BATCH_BAND(F16<true>)
}  // namespace btrirt
