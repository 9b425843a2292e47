// vgc_step_host: one worker step driven from HOST buffers -- the end-to-end form of the path.
// Copies each layer's x and delta (and the step's mean gradient g) from host memory into caller-provided
// device buffers, runs the squared-gradient sums of every layer and one compressor step on the device,
// and copies the message back to host memory.
//
// Bound: the copies (PCIe).  They go back to back on a stream of the library's own, and a layer's kernels wait for that
// layer's copies only, so that all but the last layer's run under the copies that follow (with everything on the caller's
// stream every switch between copy and kernel cost 2 - 10 us besides; MLP 784-1024-1024-10, 128 examples, 9.5 MB:
// 351 -> 261 us, of which the copies are 205).  Where a staging buffer lies over another one or over memory that an earlier
// layer's kernels write, copies and kernels take turns on the caller's stream.
// The message goes home by a kernel that writes the counters and, up to kDirectWords, the words to host memory, where that memory is
// page-locked as far as the message can reach: the call waits for the stream once.  Copies need the word count on the host first: two waits (MLP as above: 258 against 245 us).
#include <cuda.h>

#include <mutex>

#include "vgc_common.cuh"

namespace {

// A stream for the copies and an event, kept between calls: a free list for all threads (one entry per call that runs at a
// time), of kKept entries at most -- more are destroyed when their call ends, the kept ones when the process does.
struct CopyLane {
    int device = -1;
    cudaStream_t stream = nullptr;
    cudaEvent_t event = nullptr;
};
constexpr int kKept = 8;
std::mutex g_lane_mutex;
CopyLane g_lanes[kKept];
int g_lanes_kept = 0;

void destroy(CopyLane &lane)
{
    if (lane.event) cudaEventDestroy(lane.event);
    if (lane.stream) cudaStreamDestroy(lane.stream);
    lane = CopyLane();
}

bool acquire(CopyLane &lane)
{
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return false;
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        for (int i = 0; i < g_lanes_kept; ++i)
            if (g_lanes[i].device == device) {
                lane = g_lanes[i];
                g_lanes[i] = g_lanes[--g_lanes_kept];
                return true;
            }
    }
    lane.device = device;
    if (cudaStreamCreateWithFlags(&lane.stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&lane.event, cudaEventDisableTiming) != cudaSuccess) {
        destroy(lane);
        return false;
    }
    return true;
}

void release(CopyLane &lane)
{
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        if (g_lanes_kept < kKept) {
            g_lanes[g_lanes_kept++] = lane;
            return;
        }
    }
    destroy(lane);
}

// Copies of one call.  Not `overlap`, or no stream to be had: all on the caller's stream.
class Copies {
public:
    Copies(cudaStream_t caller, bool overlap) : caller_(caller), own_(overlap && acquire(lane_))
    {
        if (own_) ok_ = order(caller_, lane_.stream);            // after what the caller's stream holds already
    }
    ~Copies()
    {
        if (!own_) return;
        if (pending_) arrived();                                 // (an error return: the caller's stream still covers the copies)
        release(lane_);
    }
    bool in(void *dst, const void *src, size_t bytes)
    {
        pending_ = true;
        return ok_ && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, own_ ? lane_.stream : caller_) == cudaSuccess;
    }
    // what the caller's stream holds from here on comes after the copies so far
    bool arrived()
    {
        pending_ = false;
        return !own_ || order(lane_.stream, caller_);
    }

private:
    // (a wait refers to the event's last record when it is enqueued, so one event serves all)
    bool order(cudaStream_t first, cudaStream_t then)
    {
        return cudaEventRecord(lane_.event, first) == cudaSuccess && cudaStreamWaitEvent(then, lane_.event, 0) == cudaSuccess;
    }
    cudaStream_t caller_;
    CopyLane lane_;
    bool own_, ok_ = true, pending_ = false;
};

// ---- the message's way home -----------------------------------------------------------------------------------------
constexpr uint32_t kDirectWords = 1u << 18;          // longer messages take a copy: its engine, no SM waits for PCIe
__global__ void __launch_bounds__(256)
message_to_host(const vgc_message out, uint32_t *words_host, uint32_t *counters_host)
{
    vgc::grid_wait();
    const uint32_t nnz = *out.nnz, kept = min(nnz, out.capacity);
    if (blockIdx.x == 0 && threadIdx.x < 4) {
        const uint32_t *const from[4] = {out.nnz, out.n_criterion, out.n_dropped, out.dev_status};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (threadIdx.x == i) counters_host[i] = *from[i];
    }
    if (kept > kDirectWords) return;
    const uint32_t step = gridDim.x * 256, first = blockIdx.x * 256 + threadIdx.x;
    const bool vec = ((reinterpret_cast<uintptr_t>(out.words) | reinterpret_cast<uintptr_t>(words_host)) & 15u) == 0;
    const uint32_t whole = vec ? kept / 4 : 0;
    for (uint32_t i = first; i < whole; i += step) reinterpret_cast<uint4 *>(words_host)[i] = reinterpret_cast<const uint4 *>(out.words)[i];
    for (uint32_t i = 4 * whole + first; i < kept; i += step) words_host[i] = out.words[i];
}

// The address under which kernels reach `bytes` bytes of host memory: all of them in one page-locked allocation or registration
// (the runtime says of the first byte only whether it is), on a 4-byte boundary.  nullptr for other memory.
uint32_t *device_view(const void *host, size_t bytes)
{
    typedef CUresult (*AttributesFn)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const AttributesFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttributes", &p, cudaEnableDefault, &found) == cudaSuccess;
        return ok && found == cudaDriverEntryPointSuccess ? reinterpret_cast<AttributesFn>(p) : nullptr;
    }();
    const uintptr_t first = reinterpret_cast<uintptr_t>(host);
    if (!fn || (first & 3u)) return nullptr;
    unsigned type = 0, managed = 0;
    CUdeviceptr seen = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *into[5] = {&type, &managed, &seen, &start, &size};
    // (memory that CUDA does not know: all of them zero)
    if (fn(5, what, into, (CUdeviceptr)first) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed || seen != (CUdeviceptr)first) return nullptr;
    return first >= start && first - start <= size && bytes <= size - (first - start) ? reinterpret_cast<uint32_t *>(seen) : nullptr;
}

struct LayerSizes {
    size_t n_x, n_d, n_w;
};
bool layer_sizes(const vgc_layer_host &L, LayerSizes &z)
{
    if (!L.x_host || !L.delta_host || !L.x_dev || !L.delta_dev) return false;
    if (L.is_conv) {
        if (L.H + 2 * L.pad_h < L.Kh || L.W + 2 * L.pad_w < L.Kw || L.stride_h < 1 || L.stride_w < 1) return false;
        const size_t Ho = (L.H + 2 * L.pad_h - L.Kh) / L.stride_h + 1, Wo = (L.W + 2 * L.pad_w - L.Kw) / L.stride_w + 1;
        z.n_x = (size_t)L.B * L.C * L.H * L.W;
        z.n_d = (size_t)L.B * L.Cout * Ho * Wo;
        z.n_w = (size_t)L.Cout * L.C * L.Kh * L.Kw;
    } else {
        z.n_x = (size_t)L.B * L.C;
        z.n_d = (size_t)L.B * L.Cout;
        z.n_w = (size_t)L.Cout * L.C;
    }
    return true;
}

struct Span {
    uintptr_t begin, end;
    Span(const void *p, size_t bytes) : begin(reinterpret_cast<uintptr_t>(p)), end(begin + bytes) {}
    bool meets(const Span &o) const { return begin < o.end && o.begin < end; }
};

// Copies may run beside the kernels of the layers before: no two of the copies' destinations overlap, and none lies over what
// those kernels write (the squared sums, the workspace).
bool copies_may_overlap(const vgc_layer_host *layers, int n_layers, const float *g_dev, size_t n, const float *s_dev, const void *ws,
                        size_t ws_bytes)
{
    // 0: sums, 1: workspace, 2: g, then x and delta of every layer
    auto span = [&](int i) {
        if (i == 0) return Span(s_dev, n * sizeof(float));
        if (i == 1) return Span(ws, ws_bytes);
        if (i == 2) return Span(g_dev, n * sizeof(float));
        const vgc_layer_host &L = layers[(i - 3) / 2];
        LayerSizes z;
        layer_sizes(L, z);
        return i % 2 ? Span(L.x_dev, z.n_x * sizeof(float)) : Span(L.delta_dev, z.n_d * sizeof(float));
    };
    for (int i = 2; i < 3 + 2 * n_layers; ++i)
        for (int j = 0; j < i; ++j)
            if (span(i).meets(span(j))) return false;
    return true;
}

}  // namespace

extern "C" vgc_status vgc_step_host(const vgc_layer_host *layers, int n_layers, const float *g_host, float *g_dev,
                                    float *s_dev, float *r, float *v, size_t n, const uint32_t *group_offsets,
                                    int K, float alpha, float zeta, float scale, const vgc_message *out,
                                    uint32_t *words_host, uint32_t *counters_host, void *ws_sqgrad,
                                    size_t ws_sqgrad_bytes, void *ws_compress, size_t ws_compress_bytes,
                                    vgc_stream_t stream)
{
    if (n_layers < 0 || (n_layers && !layers) || !g_host || !g_dev || !s_dev || !out || !words_host || !counters_host)
        return VGC_ERR_INVALID_ARG;
    if (K != n_layers) return VGC_ERR_INVALID_ARG;        // one weight tensor (group) per layer, in order
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    size_t offset = 0;
    for (int l = 0; l < n_layers; ++l) {
        LayerSizes z;
        if (!layer_sizes(layers[l], z) || offset + z.n_w > n) return VGC_ERR_INVALID_ARG;
        offset += z.n_w;
    }
    if (offset != n) return VGC_ERR_INVALID_ARG;
    const bool beside = copies_may_overlap(layers, n_layers, g_dev, n, s_dev, ws_sqgrad, ws_sqgrad_bytes);
    Copies copies(st, beside);
    offset = 0;
    for (int l = 0; l < n_layers; ++l) {
        const vgc_layer_host &L = layers[l];
        LayerSizes z;
        layer_sizes(L, z);
        if (!copies.in(L.x_dev, L.x_host, z.n_x * sizeof(float)) || !copies.in(L.delta_dev, L.delta_host, z.n_d * sizeof(float)) ||
            !copies.arrived())
            return VGC_ERR_CUDA;
        // g under the last layer's kernels
        if (beside && l == n_layers - 1 && !copies.in(g_dev, g_host, n * sizeof(float))) return VGC_ERR_CUDA;
        vgc_status rc = L.is_conv
                            ? vgc_sqgrad_conv(L.x_dev, L.delta_dev, L.B, L.C, L.H, L.W, L.Cout, L.Kh, L.Kw, L.stride_h,
                                              L.stride_w, L.pad_h, L.pad_w, scale, 0, s_dev + offset, ws_sqgrad,
                                              ws_sqgrad_bytes, stream)
                            : vgc_sqgrad_linear(L.x_dev, L.delta_dev, L.B, L.C, L.Cout, scale, 0, s_dev + offset,
                                                ws_sqgrad, ws_sqgrad_bytes, stream);
        if (rc != VGC_OK) return rc;
        offset += z.n_w;
    }
    if ((!beside || n_layers == 0) && !copies.in(g_dev, g_host, n * sizeof(float))) return VGC_ERR_CUDA;
    if (!copies.arrived()) return VGC_ERR_CUDA;
    vgc_status rc = vgc_compress(g_dev, s_dev, r, v, n, group_offsets, K, alpha, zeta, out, ws_compress, ws_compress_bytes,
                                 stream);
    if (rc != VGC_OK) return rc;
    const uint32_t most_words = out->capacity < kDirectWords ? out->capacity : kDirectWords;        // that the kernel may write
    uint32_t *const words_view = most_words ? device_view(words_host, (size_t)most_words * 4) : nullptr;
    uint32_t *const counters_view = device_view(counters_host, 16);
    if (words_view && counters_view) {
        VGC_CUDA_OK(vgc::launch_kernel(message_to_host, dim3(64), dim3(256), 0, st, true, *out, words_view, counters_view));
        vgc::count_launch();
        VGC_CUDA_OK(cudaStreamSynchronize(st));
        const uint32_t kept = counters_host[0] < out->capacity ? counters_host[0] : out->capacity;
        if (kept > kDirectWords) {
            VGC_CUDA_OK(cudaMemcpyAsync(words_host, out->words, (size_t)kept * 4, cudaMemcpyDeviceToHost, st));
            VGC_CUDA_OK(cudaStreamSynchronize(st));
        }
        return VGC_OK;
    }
    // counters: nnz, n_criterion, n_dropped, dev_status -- one copy where they lie side by side
    if (out->n_criterion == out->nnz + 1 && out->n_dropped == out->nnz + 2 && out->dev_status == out->nnz + 3) {
        VGC_CUDA_OK(cudaMemcpyAsync(counters_host, out->nnz, 16, cudaMemcpyDeviceToHost, st));
    } else {
        VGC_CUDA_OK(cudaMemcpyAsync(counters_host + 0, out->nnz, 4, cudaMemcpyDeviceToHost, st));
        VGC_CUDA_OK(cudaMemcpyAsync(counters_host + 1, out->n_criterion, 4, cudaMemcpyDeviceToHost, st));
        VGC_CUDA_OK(cudaMemcpyAsync(counters_host + 2, out->n_dropped, 4, cudaMemcpyDeviceToHost, st));
        VGC_CUDA_OK(cudaMemcpyAsync(counters_host + 3, out->dev_status, 4, cudaMemcpyDeviceToHost, st));
    }
    VGC_CUDA_OK(cudaStreamSynchronize(st));
    const uint32_t kept = counters_host[0] < out->capacity ? counters_host[0] : out->capacity;
    if (kept) {
        VGC_CUDA_OK(cudaMemcpyAsync(words_host, out->words, (size_t)kept * 4, cudaMemcpyDeviceToHost, st));
        VGC_CUDA_OK(cudaStreamSynchronize(st));
    }
    return VGC_OK;
}
