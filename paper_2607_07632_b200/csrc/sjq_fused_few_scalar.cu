// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_SCALAR) and up to kFewStages stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_few_fn fused_few_scalar(bool mul, int form)
{
    switch (form) {
    case 0: return fused_of<RunParamsFew, AGG_SCALAR, 0>(mul);
    case kFormHash: return fused_of<RunParamsFew, AGG_SCALAR, kFormHash>(mul);
    case kFormDirect: return fused_of<RunParamsFew, AGG_SCALAR, kFormDirect>(mul);
    case kFormDirect | kFormHash: return fused_of<RunParamsFew, AGG_SCALAR, kFormDirect | kFormHash>(mul);
    case kFormNarrow: return fused_of<RunParamsFew, AGG_SCALAR, kFormNarrow>(mul);
    case kFormDirect | kFormNarrow: return fused_of<RunParamsFew, AGG_SCALAR, kFormDirect | kFormNarrow>(mul);
    case kFormHash | kFormNarrow: return fused_of<RunParamsFew, AGG_SCALAR, kFormHash | kFormNarrow>(mul);
    default: return fused_of<RunParamsFew, AGG_SCALAR, kFormDirect | kFormHash | kFormNarrow>(mul);
    }
}

} // namespace sjq
