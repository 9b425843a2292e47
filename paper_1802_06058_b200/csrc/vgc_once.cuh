// Which kernels have been set up on which device (plain C++, no CUDA): a kernel's limit on dynamic shared memory belongs to
// the device that was current when it was raised, and calls come from any thread.
#pragma once

#include <atomic>

namespace vgc {

class OncePerDevice {
public:
    static constexpr int kDevices = 64, kKernels = 64;

    // Runs setup() -- which returns 0 when it succeeded -- unless it has succeeded for this kernel and device before; its
    // result.  Calls that meet may run it twice.  Further devices and kernels than there is room for run it every time.
    template <class Setup>
    int operator()(const void *kernel, int device, Setup setup)
    {
        if (device < 0 || device >= kDevices) return setup();
        std::atomic<const void *> *const done = done_[device];
        for (int i = 0; i < kKernels; ++i) {
            const void *const k = done[i].load(std::memory_order_acquire);
            if (k == kernel) return 0;
            if (!k) break;
        }
        const int result = setup();
        for (int i = 0; result == 0 && i < kKernels; ++i) {
            const void *empty = nullptr;
            if (done[i].compare_exchange_strong(empty, kernel, std::memory_order_release, std::memory_order_relaxed) || empty == kernel) break;
        }
        return result;
    }

private:
    std::atomic<const void *> done_[kDevices][kKernels] = {};
};

}  // namespace vgc
