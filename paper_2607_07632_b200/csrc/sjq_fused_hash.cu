// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_HASH); one translation unit per
// path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_fn fused_variant_hash(bool mul, bool hash) { return fused_variant<RunParams, AGG_HASH>(mul, hash); }

} // namespace sjq
