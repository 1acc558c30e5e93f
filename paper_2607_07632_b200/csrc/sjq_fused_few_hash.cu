// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_HASH) and up to kFewStages stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_few_fn fused_few_hash(bool mul, int form)
{
    switch (form) {
    case 0: return fused_of<RunParamsFew, AGG_HASH, 0>(mul);
    case kFormHash: return fused_of<RunParamsFew, AGG_HASH, kFormHash>(mul);
    case kFormDirect: return fused_of<RunParamsFew, AGG_HASH, kFormDirect>(mul);
    case kFormDirect | kFormHash: return fused_of<RunParamsFew, AGG_HASH, kFormDirect | kFormHash>(mul);
    case kFormNarrow: return fused_of<RunParamsFew, AGG_HASH, kFormNarrow>(mul);
    case kFormDirect | kFormNarrow: return fused_of<RunParamsFew, AGG_HASH, kFormDirect | kFormNarrow>(mul);
    case kFormHash | kFormNarrow: return fused_of<RunParamsFew, AGG_HASH, kFormHash | kFormNarrow>(mul);
    default: return fused_of<RunParamsFew, AGG_HASH, kFormDirect | kFormHash | kFormNarrow>(mul);
    }
}

} // namespace sjq
