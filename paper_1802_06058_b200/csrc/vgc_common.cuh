// Shared device/host helpers of the vgc CUDA library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <cstdlib>
#include <utility>

#include "vgc.h"
#include "vgc_once.cuh"

#ifndef __CUDA_ARCH__
#define VGC_HOST_ONLY 1
#endif

namespace vgc {

constexpr int kWarp = 32;
constexpr int kSmCount = 148;       // SMs of a B200: work is cut by this number, so that results do not depend on the device

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// VGC_DEBUG=1 in the environment (read once): a failing CUDA call is named on stderr before the status is returned
inline bool debug_enabled()
{
    static const bool on = getenv("VGC_DEBUG") != nullptr;
    return on;
}
inline void report_cuda_error(cudaError_t e, const char *what, const char *file, int line)
{
    if (debug_enabled()) fprintf(stderr, "vgc: %s:%d: %s -> %s\n", file, line, what, cudaGetErrorString(e));
}
#define VGC_CUDA_OK(expr)                                                  \
    do {                                                                   \
        const cudaError_t vgc_e_ = (expr);                                 \
        if (vgc_e_ != cudaSuccess) {                                       \
            ::vgc::report_cuda_error(vgc_e_, #expr, __FILE__, __LINE__);   \
            return VGC_ERR_CUDA;                                           \
        }                                                                  \
    } while (0)

// Number of kernels this library has enqueued since it was loaded (benchmark bookkeeping).
extern unsigned long long g_launches;
inline void count_launch(unsigned k = 1) { g_launches += k; }

// ---- launches that follow one another closely ---------------------------------------------------------------------
// A kernel launched with `overlap` may start while the kernel before it on the stream is still running (programmatic
// dependent launch): its blocks take the SMs as they become free, and everything before its grid_wait() hides under that
// kernel's end.  grid_wait() returns once the kernel before has finished and its writes are visible.  Every kernel launched
// that way executes it in all its threads, before it touches memory that work ahead of it on the stream may write -- every
// array of the caller's, the tensor offsets too.  The one exception: the second kernel of a call may read what only the
// caller writes, where the first one calls grid_release() after its own grid_wait().
// A kernel launched that way may be alive while the one ahead writes what it is going to read.  The non-coherent loads
// (__ldg, const __restrict__ parameters) are defined only for data that nobody writes during the kernel's life, so these
// kernels use ordinary ones.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// lets the next kernel of the stream start now, where it was launched with `overlap`
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;"); }

// carveout >= 0: percent of an SM's on-chip memory that shall be shared memory while the kernel runs there, the rest L1.  A kernel
// that starts under the end of the one ahead otherwise runs with what that one left: behind a kernel that takes all the shared
// memory, 28 KB of L1, too little for the loads that a streaming kernel keeps in flight.  (It costs small kernels some of the
// overlap, since an SM changes over only when nothing runs there.)
struct Carveout { int percent; };
template <class... Params, class... Given>
cudaError_t launch_kernel(Carveout carveout, void (*fn)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool overlap,
                          Given &&...given)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = 0;
    if (overlap) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (carveout.percent >= 0) {
        attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[cfg.numAttrs++].val.sharedMemCarveout = (unsigned)carveout.percent;
    }
    return cudaLaunchKernelEx(&cfg, fn, static_cast<Params>(given)...);
}

template <class... Params, class... Given>
cudaError_t launch_kernel(void (*fn)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool overlap,
                          Given &&...given)
{
    return launch_kernel(Carveout{-1}, fn, grid, block, smem, st, overlap, std::forward<Given>(given)...);
}

// Lets a kernel use `bytes` of dynamic shared memory on the current device.  regs > 0: it has to have been compiled to that
// many registers (its code shares them out); cudaErrorInvalidKernelImage where it was not.
inline cudaError_t allow_dynamic_smem(const void *kernel, size_t bytes, int regs = 0)
{
    static OncePerDevice once;
    int device = -1;
    const cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    return (cudaError_t)once(kernel, device, [&]() -> int {
        if (regs > 0) {
            cudaFuncAttributes attr;
            const cudaError_t a = cudaFuncGetAttributes(&attr, kernel);
            if (a != cudaSuccess) return (int)a;
            if (attr.numRegs != regs) return (int)cudaErrorInvalidKernelImage;
        }
        return (int)cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    });
}

// Streaming (evict-first) 128-bit load for data touched once per call.
__device__ __forceinline__ float4 ld_stream_f4(const float *p)
{
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
// Index of the weight tensor holding flat index i: the k with offs[k] <= i < offs[k+1].
// offs has K+1 non-decreasing entries, offs[0] = 0; empty tensors are skipped.
__device__ __forceinline__ int group_of(const uint32_t *offs, int K, uint32_t i)
{
    int lo = 0, hi = K;   // invariant: offs[lo] <= i, answer in [lo, hi)
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (offs[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t x)
{
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    return x;
}

}  // namespace vgc
