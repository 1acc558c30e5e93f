// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_SCALAR) and any number of stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_fn fused_variant_scalar(bool mul, int form)
{
    switch (form) {
    case 0: return fused_of<RunParams, AGG_SCALAR, 0>(mul);
    case kFormHash: return fused_of<RunParams, AGG_SCALAR, kFormHash>(mul);
    case kFormDirect: return fused_of<RunParams, AGG_SCALAR, kFormDirect>(mul);
    default: return fused_of<RunParams, AGG_SCALAR, kFormDirect | kFormHash>(mul);
    }
}

} // namespace sjq
