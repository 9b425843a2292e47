// vgc_pack_indices / vgc_unpack_indices: the index field of a packed message stored as differences in a
// variable-length code (Sec. 4.2, last paragraph: "we can further reduce the number of bits by compressing
// parameter indexes" -- the paper names the idea and does not fix a format; the format is this library's).
//
// The words of a message come in ascending index order.  They are taken in runs of 256; word i of a run becomes
//     v = (idx_i - idx_{i-1}) << 4 | (word_i & 15)        (idx_{-1} = 0 at the start of every run)
// -- the difference above the unchanged 4-bit value field -- written in the base-128 code: seven bits per byte, least
// significant group first, the top bit of a byte set when another byte follows (1 to 5 bytes).  The stream is
//     [table: (runs + 1) x uint32, little endian][payload],   table[j] = offset of run j inside the payload,
// table[runs] = payload length, runs = ceil(nnz / 256).  Runs restart so that they can be coded and decoded side by
// side: one warp per run.
//
//   pack:   pack_count   every lane sizes 8 consecutive words of its warp's run; the totals of chunks of 8 runs are stored
//           pack_emit    starts under pack_count and codes its words into shared memory; then a block adds up the totals of the
//                        chunks before its own (no waiting on other blocks), and its bytes leave as whole words, shifted to the
//                        alignment they have in the stream
//   unpack: one kernel   a warp brings its run's bytes into shared memory, 4 at a time; a byte with a clear top bit ends a
//                        number: a warp scan of their counts gives every end its place, every lane reads the 8 numbers
//                        between its ends, and a second scan over the differences gives the indices
// Bound: latency (launch, the counter, the table, the bytes follow one another).  Measured (B200, 765 thousand words, 2 bytes
// each): pack and unpack together 28.7 us byte by byte (31 M warp instructions), 13.6 with whole words, 12.9 with the code written
// before the wait.
#include "vgc_common.cuh"

namespace vgc {

constexpr int kPackRun = VGC_PACK_RUN;                  // words per run
constexpr int kPackWarps = 8;                           // runs per chunk, a block's work at a time
constexpr int kPackThreads = 32 * kPackWarps;
constexpr int kPerLane = kPackRun / 32;                 // 8 words per lane
constexpr int kRunBytesMax = 5 * kPackRun;              // 1280

__device__ __forceinline__ uint32_t code_length(uint32_t v)
{
    return v < (1u << 7) ? 1u : v < (1u << 14) ? 2u : v < (1u << 21) ? 3u : v < (1u << 28) ? 4u : 5u;
}

// the numbers of this lane's 8 words of run `run` and how many of them exist; `bytes`: what they take
__device__ __forceinline__ uint32_t lane_numbers(const uint32_t *words, uint32_t n, uint32_t run, uint32_t lane,
                                                 uint32_t (&v)[kPerLane], uint32_t &bytes)
{
    const uint32_t first = run * kPackRun + lane * kPerLane;
    const uint32_t have = first >= n ? 0u : min((uint32_t)kPerLane, n - first);
    if (have == kPerLane && (reinterpret_cast<uintptr_t>(words) & 15u) == 0u) {
        const uint4 a = *reinterpret_cast<const uint4 *>(words + first), b = *reinterpret_cast<const uint4 *>(words + first + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) v[j] = (uint32_t)j < have ? words[first + j] : 0u;
    }
    uint32_t prev = __shfl_up_sync(0xffffffffu, v[kPerLane - 1], 1) >> 4;
    if (lane == 0) prev = 0;
    bytes = 0;
#pragma unroll
    for (int j = 0; j < kPerLane; ++j) {
        const uint32_t idx = v[j] >> 4;
        v[j] = ((idx - prev) << 4) | (v[j] & 15u);
        prev = idx;
        bytes += (uint32_t)j < have ? code_length(v[j]) : 0u;
    }
    return have;
}

__device__ __forceinline__ uint32_t warp_inclusive(uint32_t x, uint32_t lane)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += up;
    }
    return x;
}

__global__ void __launch_bounds__(kPackThreads, 6)
pack_count(const uint32_t *words, const uint32_t *nnz, uint32_t max_words, uint32_t *chunk_bytes)
{
    __shared__ uint32_t sm_tot[2][kPackWarps];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_wait();
    grid_release();                                     // in this order: pack_emit reads the words before it waits for us
    const uint32_t n = min(*nnz, max_words), runs = (n + kPackRun - 1) / kPackRun;
    uint32_t buf = 0;
    for (uint32_t chunk = blockIdx.x; chunk * kPackWarps < runs; chunk += gridDim.x, buf ^= 1) {
        uint32_t v[kPerLane], bytes;
        lane_numbers(words, n, chunk * kPackWarps + warp, lane, v, bytes);
        bytes = __reduce_add_sync(0xffffffffu, bytes);
        if (lane == 0) sm_tot[buf][warp] = bytes;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
#pragma unroll
            for (int w = 0; w < kPackWarps; ++w) t += sm_tot[buf][w];
            chunk_bytes[chunk] = t;
        }
    }
}

__global__ void __launch_bounds__(kPackThreads, 6)
pack_emit(const uint32_t *words, const uint32_t *nnz, uint32_t max_words,
          const uint32_t *chunk_bytes, uint8_t *packed, size_t capacity, uint32_t *packed_bytes, uint32_t *dev_status)
{
    __shared__ uint32_t sm_code[kPackWarps * kRunBytesMax / 4 + 1];     // (and a word to read past)
    __shared__ unsigned long long sm_part[kPackWarps];
    __shared__ uint32_t sm_run[kPackWarps];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_release();
    const uint32_t n = min(*nnz, max_words);
    const uint32_t runs = (n + kPackRun - 1) / kPackRun;
    const size_t table_bytes = 4 * ((size_t)runs + 1);
    // a chunk's code in shared memory, from its first byte on: all of it before the wait where the chunk is the block's first
    uint32_t in_chunk = 0, chunk_total = 0;
    auto code = [&](uint32_t chunk) {
        uint32_t v[kPerLane], mine;
        const uint32_t have = lane_numbers(words, n, chunk * kPackWarps + warp, lane, v, mine);
        const uint32_t incl = warp_inclusive(mine, lane);
        if (lane == 31) sm_run[warp] = incl;
        __syncthreads();
        in_chunk = chunk_total = 0;
#pragma unroll
        for (int w = 0; w < kPackWarps; ++w) {
            in_chunk += (uint32_t)w < warp ? sm_run[w] : 0u;
            chunk_total += sm_run[w];
        }
        uint8_t *at = reinterpret_cast<uint8_t *>(sm_code) + in_chunk + (incl - mine);
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            if ((uint32_t)j < have) {
                const uint32_t x = v[j], len = code_length(x);
                at[0] = (uint8_t)((x & 0x7Fu) | (len > 1 ? 0x80u : 0u));
                if (len > 1) at[1] = (uint8_t)((x >> 7 & 0x7Fu) | (len > 2 ? 0x80u : 0u));
                if (len > 2) at[2] = (uint8_t)((x >> 14 & 0x7Fu) | (len > 3 ? 0x80u : 0u));
                if (len > 3) at[3] = (uint8_t)((x >> 21 & 0x7Fu) | (len > 4 ? 0x80u : 0u));
                if (len > 4) at[4] = (uint8_t)(x >> 28);
                at += len;
            }
        }
    };
    if (blockIdx.x * kPackWarps <= runs) code(blockIdx.x);
    grid_wait();                                                        // pack_count's totals
    unsigned long long before = 0;                                      // payload bytes of all chunks before this one
    uint32_t summed = 0;                                                // chunks summed so far
    // one chunk more than the runs need: the warp that writes table[runs]
    for (uint32_t chunk = blockIdx.x; chunk * kPackWarps <= runs; chunk += gridDim.x) {
        if (chunk != blockIdx.x) {
            __syncthreads();                                            // the chunk before has left shared memory
            code(chunk);
        }
        unsigned long long more = 0;
        for (uint32_t b = summed + threadIdx.x; b < chunk; b += kPackThreads) more += __ldcg(chunk_bytes + b);
        summed = chunk;
        more = warp_sum_u64(more);
        const uint32_t run = chunk * kPackWarps + warp;
        if (lane == 0) sm_part[warp] = more;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kPackWarps; ++w) before += sm_part[w];
        const unsigned long long run_off = before + in_chunk;           // this run's first byte inside the payload
        if (run <= runs && lane < 4) {                                  // table[run]
            const size_t at = 4 * (size_t)run + lane;
            if (at < capacity) packed[at] = (uint8_t)((uint32_t)run_off >> (8 * lane));
        }
        if (run == runs && lane == 0) {
            // table[runs] is the payload length: written by the warp whose run number is `runs` (its offset is the total)
            const unsigned long long total = table_bytes + run_off;
            *packed_bytes = (uint32_t)total;
            if (total > capacity) atomicOr(dev_status, VGC_DEV_CAPACITY);
        }
        // whole words of the stream, each out of two of the chunk's; the first and last one, which neighbouring chunks share,
        // byte by byte
        const size_t dst0 = table_bytes + before;                       // of the chunk's first byte
        const uint32_t skew = (uint32_t)((reinterpret_cast<uintptr_t>(packed) + dst0) & 3u), span = skew + chunk_total;
        uint8_t *const base = packed + dst0 - skew;                     // 4-byte aligned
        for (uint32_t i = 4 * threadIdx.x; i < span; i += 4 * kPackThreads) {
            if (i >= skew && i + 4 <= span && dst0 - skew + i + 4 <= capacity) {
                const uint32_t *const from = sm_code + ((i - skew) >> 2);
                *reinterpret_cast<uint32_t *>(base + i) = __funnelshift_r(from[0], from[1], 8 * ((i - skew) & 3u));
            } else {
                for (uint32_t b = i < skew ? skew : i; b < i + 4 && b < span; ++b)
                    if (dst0 - skew + b < capacity) base[b] = reinterpret_cast<const uint8_t *>(sm_code)[b - skew];
            }
        }
    }
}

__global__ void __launch_bounds__(kPackThreads, 6)
unpack_runs(const uint8_t *packed, const uint32_t *nnz, uint32_t max_words, uint32_t *words, uint32_t *dev_status)
{
    constexpr int kWordsMax = kRunBytesMax / 4 + 4;                     // a run's bytes at any alignment, and a word to read past
    __shared__ uint32_t sm_words[kPackWarps][kWordsMax];
    __shared__ __align__(16) uint16_t sm_end[kPackWarps][kPackRun];     // where the numbers end
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_release();
    grid_wait();
    const uint32_t n = min(*nnz, max_words);
    const uint32_t runs = (n + kPackRun - 1) / kPackRun;
    const size_t table_bytes = 4 * ((size_t)runs + 1);
    for (uint32_t run = blockIdx.x * kPackWarps + warp; run < runs; run += gridDim.x * kPackWarps) {
        __syncwarp();                                                   // the run before has left shared memory
        uint32_t begin = 0, end = 0;
        if ((reinterpret_cast<uintptr_t>(packed) & 3u) == 0u) {
            begin = reinterpret_cast<const uint32_t *>(packed)[run];
            end = reinterpret_cast<const uint32_t *>(packed)[run + 1];
        } else {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                begin |= (uint32_t)packed[4 * (size_t)run + b] << (8 * b);
                end |= (uint32_t)packed[4 * (size_t)run + 4 + b] << (8 * b);
            }
        }
        const uint32_t in_run = min((uint32_t)kPackRun, n - run * kPackRun);   // words this run holds
        const uint32_t nb = end - begin;
        uint32_t *const out = words + (size_t)run * kPackRun;
        auto refuse = [&]() {
            if (lane == 0) atomicOr(dev_status, VGC_DEV_RANGE);
            for (uint32_t i = lane; i < in_run; i += 32) out[i] = 0xFFFFFFFFu;  // an index no buffer has
        };
        // a run of k words takes k .. 5 k bytes; anything else is not a stream this library wrote
        if (end < begin || nb < in_run || nb > 5 * in_run) { refuse(); continue; }
        const uint8_t *src = packed + table_bytes + begin;
        // the bytes keep their alignment in shared memory (byte i sits at off + i), so whole words can be copied; the word that
        // holds the first byte starts up to 3 bytes earlier (inside the stream: the table is before it), the bytes after the
        // last whole word come one by one
        const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 3u), limit = off + nb, n_words = (limit + 3u) / 4u;
        const uint32_t *src_w = reinterpret_cast<const uint32_t *>(src - off);
        uint32_t found = 0;                                                  // numbers that end in the words so far
        bool bad = false;
        for (uint32_t i0 = 0; i0 < n_words; i0 += 128) {                     // four words per lane, 32 apart
            uint32_t w[4], ends[4], counts = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + 32 * u + lane;
                w[u] = 0;
                if (4 * i + 4 <= limit) w[u] = src_w[i];
                else for (uint32_t b = 4 * i; b < limit; ++b) w[u] |= (uint32_t)src[b - off] << (8 * (b & 3u));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + 32 * u + lane;
                if (i < n_words) sm_words[warp][i] = w[u];
                ends[u] = ~w[u] & 0x80808080u;                               // bytes of the run that end a number
                if (i == 0) ends[u] &= 0xFFFFFFFFu << (8 * off);
                if (4 * i + 4 > limit) ends[u] &= 4 * i < limit ? (1u << (8 * (limit - 4 * i))) - 1u : 0u;
                counts |= (uint32_t)__popc(ends[u]) << (8 * u);
            }
            // 32 lanes x 4 ends: a scan of four bytes at a time, then the four rows one after the other
            const uint32_t incl = warp_inclusive(counts, lane), total = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t k = found + ((incl >> (8 * u)) & 0xFFu) - ((counts >> (8 * u)) & 0xFFu);
                for (uint32_t e = ends[u]; e; e &= e - 1u, ++k)
                    if (k < (uint32_t)kPackRun) sm_end[warp][k] = (uint16_t)(4 * (i0 + 32 * u + lane) + ((__ffs(e) - 1) >> 3));
                found += (total >> (8 * u)) & 0xFFu;
            }
        }
        if (lane == 0) sm_words[warp][n_words] = 0;
        __syncwarp();
        // as many numbers as the run has words, the last byte ending one
        if (found != in_run || sm_end[warp][in_run - 1] != limit - 1) { refuse(); continue; }
        const uint4 e4 = *reinterpret_cast<const uint4 *>(&sm_end[warp][lane * kPerLane]);
        const uint32_t pair[4] = {e4.x, e4.y, e4.z, e4.w};
        uint32_t start = __shfl_up_sync(0xffffffffu, e4.w >> 16, 1) + 1u;
        if (lane == 0) start = off;
        uint32_t v[kPerLane], sum = 0;
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            v[j] = 0;
            if (lane * kPerLane + j < in_run) {
                const uint32_t last = (pair[j >> 1] >> (16 * (j & 1))) & 0xFFFFu, len = last - start + 1u;
                if (len > 5u) bad = true;
                else {
                    const uint32_t *p = &sm_words[warp][start >> 2];
                    uint32_t x = __funnelshift_r(p[0], p[1], 8 * (start & 3u));
                    if (len < 4u) x &= (1u << (8 * len)) - 1u;
                    v[j] = (x & 0x7Fu) | (x >> 1 & 0x3F80u) | (x >> 2 & 0x1FC000u) | (x >> 3 & 0xFE00000u);
                    if (len == 5u) v[j] |= (sm_words[warp][last >> 2] >> (8 * (last & 3u))) << 28;
                    sum += v[j] >> 4;
                }
                start = last + 1u;
            }
        }
        if (__any_sync(0xffffffffu, bad)) { refuse(); continue; }
        // indices: running sum of the differences, 8 consecutive words per lane
        uint32_t idx = warp_inclusive(sum, lane) - sum;
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            idx += v[j] >> 4;
            v[j] = (idx << 4) | (v[j] & 15u);
        }
        if (in_run == kPackRun && (reinterpret_cast<uintptr_t>(words) & 15u) == 0u) {
            *reinterpret_cast<uint4 *>(out + lane * kPerLane) = make_uint4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<uint4 *>(out + lane * kPerLane + 4) = make_uint4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int j = 0; j < kPerLane; ++j)
                if (lane * kPerLane + j < in_run) out[lane * kPerLane + j] = v[j];
        }
    }
}

}  // namespace vgc

using namespace vgc;

namespace {
struct PackLayout { size_t total; uint32_t chunks; };
// At most this many blocks, which then take several chunks each: a message may be much shorter than its buffer, and a block
// that starts only to find nothing to do costs a round trip to memory (7.6 M words in a buffer of 61 M: pack 83 us with a block
// per chunk of the buffer).  Eight times what is resident at a time: with once that many, 7.6 M words in a buffer of their
// own length took 39 us instead of 34.
constexpr uint32_t kPackGrid = 8 * kSmCount * (2048 / kPackThreads);
PackLayout pack_layout(uint32_t max_words)
{
    PackLayout L;
    const uint32_t runs = (max_words + kPackRun - 1) / kPackRun;
    L.chunks = runs / kPackWarps + 1;                      // one more than the runs need: the warp that writes table[runs]
    L.total = round_up(sizeof(uint32_t) * (size_t)L.chunks, 256);
    return L;
}
}  // namespace

extern "C" size_t vgc_pack_bound_bytes(uint32_t max_words)
{
    return 4 * ((size_t)(max_words + kPackRun - 1) / kPackRun + 1) + 5 * (size_t)max_words;
}

extern "C" size_t vgc_pack_workspace_bytes(uint32_t max_words) { return pack_layout(max_words).total; }

extern "C" vgc_status vgc_pack_indices(const uint32_t *words, const uint32_t *nnz, uint32_t max_words, uint8_t *packed,
                                       size_t packed_capacity, uint32_t *packed_bytes, uint32_t *dev_status, void *ws,
                                       size_t ws_bytes, vgc_stream_t stream)
{
    if (!nnz || !packed || !packed_bytes || !dev_status || (max_words && !words)) return VGC_ERR_INVALID_ARG;
    if (max_words > VGC_MAX_PARAMS || packed_capacity < 4) return VGC_ERR_INVALID_ARG;
    const PackLayout L = pack_layout(max_words);
    if (!ws || ws_bytes < L.total) return VGC_ERR_WORKSPACE;
    uint32_t *chunk_bytes = static_cast<uint32_t *>(ws);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const unsigned blocks = L.chunks < kPackGrid ? L.chunks : kPackGrid;
    VGC_CUDA_OK(launch_kernel(pack_count, dim3(blocks), dim3(kPackThreads), 0, st, true, words, nnz, max_words, chunk_bytes));
    VGC_CUDA_OK(launch_kernel(pack_emit, dim3(blocks), dim3(kPackThreads), 0, st, true, words, nnz, max_words, chunk_bytes, packed,
                              packed_capacity, packed_bytes, dev_status));
    count_launch(2);
    VGC_CUDA_OK(cudaGetLastError());
    return VGC_OK;
}

extern "C" vgc_status vgc_unpack_indices(const uint8_t *packed, const uint32_t *nnz, uint32_t max_words, uint32_t *words,
                                         uint32_t *dev_status, vgc_stream_t stream)
{
    if (!packed || !nnz || !dev_status || (max_words && !words)) return VGC_ERR_INVALID_ARG;
    if (max_words > VGC_MAX_PARAMS) return VGC_ERR_INVALID_ARG;
    if (max_words == 0) return VGC_OK;
    const uint32_t chunks = ((max_words + kPackRun - 1) / kPackRun + kPackWarps - 1) / kPackWarps;
    VGC_CUDA_OK(launch_kernel(unpack_runs, dim3(chunks < kPackGrid ? chunks : kPackGrid), dim3(kPackThreads), 0,
                              reinterpret_cast<cudaStream_t>(stream), true, packed, nnz, max_words, words, dev_status));
    count_launch();
    VGC_CUDA_OK(cudaGetLastError());
    return VGC_OK;
}
