// Ahead-of-time instantiations of the fused kernel for one aggregation path (AGG_SMEM) and up to kFewStages stages;
// one translation unit per path and size of the parameter block so that they compile in parallel.
#include "sjq_fused_device.cuh"

namespace sjq {

fused_few_fn fused_few_smem(bool mul, int form)
{
    switch (form) {
    case 0: return fused_of<RunParamsFew, AGG_SMEM, 0>(mul);
    case kFormHash: return fused_of<RunParamsFew, AGG_SMEM, kFormHash>(mul);
    case kFormDirect: return fused_of<RunParamsFew, AGG_SMEM, kFormDirect>(mul);
    case kFormDirect | kFormHash: return fused_of<RunParamsFew, AGG_SMEM, kFormDirect | kFormHash>(mul);
    case kFormNarrow: return fused_of<RunParamsFew, AGG_SMEM, kFormNarrow>(mul);
    case kFormDirect | kFormNarrow: return fused_of<RunParamsFew, AGG_SMEM, kFormDirect | kFormNarrow>(mul);
    case kFormHash | kFormNarrow: return fused_of<RunParamsFew, AGG_SMEM, kFormHash | kFormNarrow>(mul);
    default: return fused_of<RunParamsFew, AGG_SMEM, kFormDirect | kFormHash | kFormNarrow>(mul);
    }
}

} // namespace sjq
