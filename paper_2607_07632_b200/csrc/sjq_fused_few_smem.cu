// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_SMEM) and up to kFewStages stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_few_fn fused_few_smem(bool mul, bool hash) { return fused_variant<RunParamsFew, AGG_SMEM>(mul, hash); }

} // namespace sjq
