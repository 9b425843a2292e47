// Forms of the tensor-core kernel: tiles of whole tuples of five or seven taps, input rows by TMA.
#include "vgc_sqgrad_tc.cuh"

namespace vgc {
namespace tc {

KernelFn wide_halo_kernel(int mode, bool per_example)
{
    switch (mode) {
        case kHalo5x4: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo5x4, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo5x4, true, false, true, kWideN>;
        case kHalo5x2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo5x2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo5x2, true, false, true, kWideN>;
        case kHalo7x4: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo7x4, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo7x4, true, false, true, kWideN>;
        case kHalo7x2: return per_example ? (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo7x2, true, true, false, kWideN> : (KernelFn)sqgrad_tc<kMajorK, kTma, kHalo7x2, true, false, true, kWideN>;
        default: return nullptr;
    }
}

}  // namespace tc
}  // namespace vgc
