// Shared device/host helpers of the vgc CUDA library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <cstdlib>

#include "vgc.h"

#ifndef __CUDA_ARCH__
#define VGC_HOST_ONLY 1
#endif

namespace vgc {

constexpr int kWarp = 32;

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

// How many blocks of a kernel the current device holds at a time -- what a cooperative launch may use.  Looked up once
// per device (a race between two threads looks it up twice); 0 on an error.
struct ResidentBlocks {
    static constexpr int kMaxDevices = 64;
    uint32_t blocks[kMaxDevices];
    uint32_t get(const void *fn, int threads, size_t smem)
    {
        int dev = -1, per_sm = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
        if (dev < kMaxDevices && blocks[dev]) return blocks[dev];
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 0;
        const uint32_t all = (uint32_t)(per_sm * sms);
        if (dev < kMaxDevices) blocks[dev] = all;
        return all;
    }
};

// A buffer of n parameters cut into one contiguous range per block: `least` parameters each while there are fewer of
// those than blocks to hold them; beyond that every block takes the same share (a multiple of 128 parameters: 512 B of
// every stream), cut into tiles of equal size.
struct Ranges {
    uint32_t grid, per_block, tile;
};
inline Ranges even_ranges(size_t n, uint32_t most_blocks, uint32_t tile_max, uint32_t least)
{
    Ranges R;
    const size_t tiles = (n + least - 1) / least;
    const size_t blocks = tiles < most_blocks ? tiles : most_blocks;
    const size_t per = round_up((n + blocks - 1) / blocks, 128);
    const size_t tiles_per = (per + tile_max - 1) / tile_max;
    R.per_block = (uint32_t)per;
    R.grid = (uint32_t)((n + per - 1) / per);
    R.tile = (uint32_t)round_up((per + tiles_per - 1) / tiles_per, 128);
    return R;
}

// ---- values that the blocks of one cooperative launch hand each other ---------------------------------------------
// A slot is 16 bytes, {tag, two 32-bit values}, written and read as one 128-bit access: a block publishes its slot, the
// others poll it until it carries the launch's tag -- one store and one load of latency, the values included, where a
// grid barrier costs 2.4 us with 16 blocks and 5 us with 592 and is followed by the loads of whatever it guarded.
// Slots live in the caller's workspace, whose contents are arbitrary, so nothing may depend on their being cleared:
//   - the tag is 64 bits, unique to the call on the host (leftovers of anything else do not match);
//   - a captured launch is replayed with the same tag, so a launch leaves no slot behind that carries it: a launch uses
//     two sets, `first` and `second`.  A block clears its `second` slot, then (a fence between them) publishes its
//     `first`; it waits for ALL `first` slots (and a fence) before it publishes its `second` and before it looks at
//     anyone's `second`, so a stale `second` is never seen; the last block, once it has every `second`, clears all of
//     `first` (everybody has read them by then).
// Apart from that order the values in a slot are all that is handed over, so publishing and polling are relaxed: a
// release store would wait for every store the block has in flight, an acquire load would empty the L1 cache.
// The polls are bounded: a wait that runs out makes the block raise VGC_DEV_TIMEOUT and leave.
struct __align__(16) Slot {
    unsigned long long tag;
    uint32_t a, b;
};
constexpr uint32_t kSlotPolls = 1u << 22;

__device__ __forceinline__ void slot_publish(Slot *s, unsigned long long tag, uint32_t a, uint32_t b)
{
    const unsigned long long v = (unsigned long long)b << 32 | a;
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}"
                 ::"l"(s), "l"(tag), "l"(v) : "memory");
}
__device__ __forceinline__ bool slot_read(const Slot *s, unsigned long long tag, uint32_t &a, uint32_t &b)
{
    unsigned long long t, v;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(t), "=l"(v) : "l"(s) : "memory");
    a = (uint32_t)v;
    b = (uint32_t)(v >> 32);
    return t == tag;
}
// waits until the slot carries the tag; false if it never did
__device__ __forceinline__ bool slot_wait(const Slot *s, unsigned long long tag, uint32_t &a, uint32_t &b)
{
    for (uint32_t i = 0; i < kSlotPolls; ++i) {
        if (slot_read(s, tag, a, b)) return true;
        if (i >= 4) __nanosleep(32);
    }
    a = b = 0;
    return false;
}
// host: a tag no other call of this process uses (never 0, which cleared slots carry)
unsigned long long next_tag();

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ uint64_t ld_volatile_u64(const uint64_t *p)
{
    uint64_t v;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_volatile_u64(uint64_t *p, uint64_t v)
{
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Streaming (evict-first) 128-bit accesses for data touched once per call.
__device__ __forceinline__ float4 ld_stream_f4(const float *p)
{
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream_f4(float *p, float4 v)
{
    asm volatile("st.global.cs.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
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
