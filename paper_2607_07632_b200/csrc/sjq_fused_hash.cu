// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_HASH) and any number of stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_fn fused_variant_hash(bool mul, int form)
{
    switch (form) {
    case 0: return fused_of<RunParams, AGG_HASH, 0>(mul);
    case kFormHash: return fused_of<RunParams, AGG_HASH, kFormHash>(mul);
    case kFormDirect: return fused_of<RunParams, AGG_HASH, kFormDirect>(mul);
    default: return fused_of<RunParams, AGG_HASH, kFormDirect | kFormHash>(mul);
    }
}

} // namespace sjq
