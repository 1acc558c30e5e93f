// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_SMEM); one translation unit per
// path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_fn fused_variant_smem(bool mul, bool hash) { return fused_variant<RunParams, AGG_SMEM>(mul, hash); }

} // namespace sjq
