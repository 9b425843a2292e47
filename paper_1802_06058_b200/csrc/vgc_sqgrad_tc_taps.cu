// Forms of the tensor-core kernel: tiles of 192 columns, the B tile gathered several taps at a time.
#include "vgc_sqgrad_tc.cuh"

namespace vgc {
namespace tc {

KernelFn wide_taps_kernel(int mode, bool per_example)
{
    switch (mode) {
        case kGatherTaps4: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps4, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps4, true, false, true, kWideN>;
        case kGatherTaps2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps2, true, false, true, kWideN>;
        case kGatherTaps4S2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps4S2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps4S2, true, false, true, kWideN>;
        case kGatherTaps2S2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps2S2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps2S2, true, false, true, kWideN>;
        case kGatherTaps7S2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps7S2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kGatherTaps7S2, true, false, true, kWideN>;
        default: return nullptr;
    }
}

}  // namespace tc
}  // namespace vgc
