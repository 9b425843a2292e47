// Forms of the tensor-core kernel: tiles of 192 columns, the B tile gathered several taps at a time.
#include "vgc_sqgrad_tc.cuh"

namespace vgc {
namespace tc {

template <int kMode>
static KernelFn form(bool per_example, bool bf16_cross)
{
    if (per_example) return sqgrad_tc<kMajorK, kTma, kMode, true, true, false, kWideN>;
    return bf16_cross ? sqgrad_tc<kMajorK, kTma, kMode, true, false, true, kWideN> : sqgrad_tc<kMajorK, kTma, kMode, true, false, false, kWideN>;
}

KernelFn wide_taps_kernel(int mode, bool per_example, bool bf16_cross)
{
    switch (mode) {
        case kGatherTaps4: return form<kGatherTaps4>(per_example, bf16_cross);
        case kGatherTaps2: return form<kGatherTaps2>(per_example, bf16_cross);
        case kGatherTaps4S2: return form<kGatherTaps4S2>(per_example, bf16_cross);
        case kGatherTaps2S2: return form<kGatherTaps2S2>(per_example, bf16_cross);
        case kGatherTaps7S2: return form<kGatherTaps7S2>(per_example, bf16_cross);
        default: return nullptr;
    }
}

}  // namespace tc
}  // namespace vgc
