// Forms of the tensor-core kernel: tiles of whole tuples of five or seven taps, input rows by TMA.
#include "vgc_sqgrad_tc.cuh"

namespace vgc {
namespace tc {

template <int kMode>
static KernelFn form(bool per_example, bool bf16_cross)
{
    if (per_example) return sqgrad_tc<kMajorK, kTma, kMode, true, true, false, kWideN>;
    return bf16_cross ? sqgrad_tc<kMajorK, kTma, kMode, true, false, true, kWideN> : sqgrad_tc<kMajorK, kTma, kMode, true, false, false, kWideN>;
}

KernelFn wide_halo_kernel(int mode, bool per_example, bool bf16_cross)
{
    switch (mode) {
        case kHalo5x4: return form<kHalo5x4>(per_example, bf16_cross);
        case kHalo5x2: return form<kHalo5x2>(per_example, bf16_cross);
        case kHalo7x4: return form<kHalo7x4>(per_example, bf16_cross);
        case kHalo7x2: return form<kHalo7x2>(per_example, bf16_cross);
        default: return nullptr;
    }
}

}  // namespace tc
}  // namespace vgc
