// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_HASH) and up to kFewStages stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_few_fn fused_few_hash(bool mul, bool hash) { return fused_variant<RunParamsFew, AGG_HASH>(mul, hash); }

} // namespace sjq
