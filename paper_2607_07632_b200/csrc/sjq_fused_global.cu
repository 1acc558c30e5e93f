// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_GLOBAL); one translation unit per
// path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_fn fused_variant_global(bool mul, bool hash) { return fused_variant<RunParams, AGG_GLOBAL>(mul, hash); }

} // namespace sjq
