// C ABI of the compressor: one step of Algorithm 1 ("Basic") over the flat parameter buffer followed by Encode() -- the
// 4-bit quantiser of Sec. 4.2 in the bit-level form of Sec. 4.4 and the 32-bit (value, index) word.  The kernel is in
// vgc_step.cuh.
#include <atomic>

#include "vgc_step.cuh"

using namespace vgc;

namespace {
struct CompressLayout {
    size_t records, rec_max, stage, total;
};

static CompressLayout compress_layout(size_t n, int K)
{
    CompressLayout L;
    size_t off = 0;
    L.records = off;       off = round_up(off + step::kRecordBytes, 256);
    L.rec_max = off;       off = round_up(off + sizeof(uint32_t) * ((size_t)K + step::kMaxGrid), 256);
    L.stage = off;         off = round_up(off + sizeof(uint32_t) * n, 256);
    // the interface states about 8 bytes per parameter; the staging area takes 4 of them
    L.total = round_up(off + sizeof(uint32_t) * n, 256);
    return L;
}
}  // namespace

extern "C" size_t vgc_compress_workspace_bytes(size_t n, int K)
{
    if (K < 1) K = 1;
    return compress_layout(n, K).total;
}

extern "C" vgc_status vgc_compress(const float *g, const float *s, float *r, float *v, size_t n,
                                   const uint32_t *group_offsets, int K, float alpha, float zeta,
                                   const vgc_message *out, void *ws, size_t ws_bytes, vgc_stream_t stream)
{
    if (n == 0) return VGC_OK;
    if (n > VGC_MAX_PARAMS || K < 1 || !out) return VGC_ERR_INVALID_ARG;
    if (!(alpha >= 0.f) || !(alpha <= 3.402823466e38f) || !(zeta == zeta) || !(zeta >= -3.402823466e38f) ||
        !(zeta <= 3.402823466e38f))
        return VGC_ERR_INVALID_ARG;
    if (!g || !r || !v || !group_offsets || !ws) return VGC_ERR_INVALID_ARG;
    if (!out->group_exp || !out->nnz || !out->n_criterion || !out->n_dropped || !out->dev_status)
        return VGC_ERR_INVALID_ARG;
    if (out->capacity && !out->words) return VGC_ERR_INVALID_ARG;
    if (!aligned16(g) || (s && !aligned16(s)) || !aligned16(r) || !aligned16(v) || !aligned16(ws) ||
        (out->mask && (reinterpret_cast<uintptr_t>(out->mask) & 3u)))
        return VGC_ERR_INVALID_ARG;
    const CompressLayout L = compress_layout(n, K);
    if (ws_bytes < L.total) return VGC_ERR_WORKSPACE;

    char *base = static_cast<char *>(ws);
    step::Args args = {};
    args.g = g; args.s = s; args.r = r; args.v = v; args.n = n;
    args.group_offsets = group_offsets; args.K = K; args.alpha = alpha; args.zeta = zeta;
    args.rec_max = reinterpret_cast<uint32_t *>(base + L.rec_max);
    args.stage = reinterpret_cast<uint32_t *>(base + L.stage);
    args.out = *out;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return s ? step::launch<true, step::kBasic>(args, base + L.records, st) : step::launch<false, step::kBasic>(args, base + L.records, st);
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant of vgc_compress: the scratch lives in the library image
// ------------------------------------------------------------------------------------------
// Some callers cannot hand the library a workspace because they cannot allocate device memory at the
// point where they call it: code running under a memory plan fixed ahead of time (every byte of the
// device budget already assigned), plug-ins called from inside another framework's step where
// cudaMalloc would synchronise the device or is simply forbidden, and embedding hosts that expose
// only the tensors they pass in.  For them the scratch of vgc_compress is a fixed array that every
// GPU loading this library reserves until the process exits; its size bounds the buffer length.
namespace vgc {
constexpr size_t kStaticMaxParams = VGC_COMPRESS_STATIC_MAX_PARAMS;
constexpr int kStaticMaxGroups = VGC_COMPRESS_STATIC_MAX_GROUPS;
// worst-case layout: extremes per (block, tensor), block totals, 8 bytes of staging per parameter
constexpr size_t kStaticScratchBytes = 8 * kStaticMaxParams + kStaticMaxGroups * 8 + 1024 * 1024;
static __device__ __align__(256) unsigned char g_compress_scratch[kStaticScratchBytes];
}  // namespace vgc

extern "C" vgc_status vgc_compress_static(const float *g, const float *s, float *r, float *v, size_t n,
                                          const uint32_t *group_offsets, int K, float alpha, float zeta,
                                          const vgc_message *out, vgc_stream_t stream)
{
    if (n > kStaticMaxParams || K > kStaticMaxGroups) return VGC_ERR_UNSUPPORTED;
    if (n == 0) return VGC_OK;
    if (K < 1) return VGC_ERR_INVALID_ARG;
    if (compress_layout(n, K).total > kStaticScratchBytes) return VGC_ERR_UNSUPPORTED;
    // Host code sees g_compress_scratch only as a stand-in for the device array: the address a kernel can
    // use has to be asked for, once per device, with that device current.
    constexpr int kMaxDevices = 64;
    static std::atomic<void *> scratch_of_device[kMaxDevices] = {};
    int dev = -1;
    VGC_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return VGC_ERR_UNSUPPORTED;
    void *scratch = scratch_of_device[dev];
    if (!scratch) {
        VGC_CUDA_OK(cudaGetSymbolAddress(&scratch, g_compress_scratch));
        if (!scratch) return VGC_ERR_CUDA;
        scratch_of_device[dev] = scratch;
    }
    return vgc_compress(g, s, r, v, n, group_offsets, K, alpha, zeta, out, scratch, kStaticScratchBytes, stream);
}
