// C ABI of the hybrid algorithm (Algorithm 2): variance criterion on top of the fixed threshold tau of Strom's method,
// with the variance correction of Sec. 4.5.  The streaming pass is the basic compressor's (vgc_step.cuh), minus maxima
// and quantiser: a sent element's word is index << 4 | sign << 3.
#include "vgc_step.cuh"

using namespace vgc;

// the blocks' records, then the staged values: 4 bytes per parameter
extern "C" size_t vgc_compress_hybrid_workspace_bytes(size_t n)
{
    return round_up(step::kRecordBytes, 256) + round_up(sizeof(uint32_t) * n, 256);
}

extern "C" vgc_status vgc_compress_hybrid(const float *g, const float *s, float *r, float *v, size_t n,
                                          float alpha, float zeta, float tau, int correction_from_updated_r,
                                          const vgc_hybrid_message *out, void *ws, size_t ws_bytes,
                                          vgc_stream_t stream)
{
    if (n == 0) return VGC_OK;
    if (n > VGC_MAX_PARAMS || !out) return VGC_ERR_INVALID_ARG;
    const float fmax = 3.402823466e38f;
    if (!(alpha >= 0.f) || !(alpha <= fmax) || !(zeta >= -fmax) || !(zeta <= fmax) || !(tau >= 0.f) || !(tau <= fmax))
        return VGC_ERR_INVALID_ARG;
    if (!g || !r || !v || !ws || !out->nnz || !out->dev_status) return VGC_ERR_INVALID_ARG;
    if (out->capacity && !out->words) return VGC_ERR_INVALID_ARG;
    if (!aligned16(g) || (s && !aligned16(s)) || !aligned16(r) || !aligned16(v) || !aligned16(ws) ||
        (out->mask && (reinterpret_cast<uintptr_t>(out->mask) & 3u)))
        return VGC_ERR_INVALID_ARG;
    if (ws_bytes < vgc_compress_hybrid_workspace_bytes(n)) return VGC_ERR_WORKSPACE;

    step::Args args = {};
    args.g = g; args.s = s; args.r = r; args.v = v; args.n = n;
    args.alpha = alpha; args.zeta = zeta; args.tau = tau;
    args.stage = reinterpret_cast<uint32_t *>(static_cast<char *>(ws) + round_up(step::kRecordBytes, 256));
    args.out.words = out->words; args.out.capacity = out->capacity; args.out.nnz = out->nnz;
    args.out.mask = out->mask; args.out.dev_status = out->dev_status;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (correction_from_updated_r)
        return s ? step::launch<true, step::kHybridAfter>(args, ws, st) : step::launch<false, step::kHybridAfter>(args, ws, st);
    return s ? step::launch<true, step::kHybridBefore>(args, ws, st) : step::launch<false, step::kHybridBefore>(args, ws, st);
}
