// vgc_compress: one step of Algorithm 1 ("Basic") over the flat parameter buffer followed by
// Encode() -- the 4-bit quantiser of Sec. 4.2 in the bit-level form of Sec. 4.4 and the
// 32-bit (value, index) word.
//
// One cooperative kernel.  Every thread block owns one contiguous range of the buffer and goes through three
// steps with a grid-wide barrier between them (the per-tensor maximum has to be complete before any value can be
// quantised, and the number of words before a block's own before it can write them):
//   1  streams g, s, r, v once (16 B read + 8 B written per parameter), applies the send test, writes r, v back and
//      keeps the selected (index, value) pairs in index order: the first kStagePairs of them in shared memory, the
//      rest in the block's part of the workspace.  For every weight tensor the range touches it records the largest
//      and the smallest |value| sent, and it publishes them.
//   2  E_k = floor(log2 M_k) of the tensors at the range's two ends from the records of the blocks that share them
//      (tensors inside the range are complete already); how many pairs survive the quantiser (d <= 7): all of them
//      unless a recorded minimum says otherwise, so the pairs are rarely looked at here.
//   3  adds up the counts of the blocks before its own and writes its words.
// The records of (block b, tensor k) live at index b + k: blocks and the tensors they touch advance together, so no
// two share a slot, and nothing has to be cleared by a launch of its own.
//
// Bound: HBM, 24 B per parameter, for large buffers -- launches and barriers for small ones.  Before, this was a
// memset and three kernels whose pairs went through global memory; measured (B200, time of one call among others):
//   n = 25.5 M, density 1e-2: 125.8 us -> @R50@ us;   n = 32768: @SMALL@.
#include <cooperative_groups.h>

#include "vgc_common.cuh"

namespace cg = cooperative_groups;

namespace vgc {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / kWarp;             // 8
constexpr int kBlocksPerSm = 4;                      // 64 registers: 1024 threads with eight 16-byte loads each in flight
constexpr int kRowsA = 2;                            // float4 vectors per thread per tile
constexpr int kTileA = kThreads * kRowsA * 4;        // at most 2048 parameters per tile
constexpr int kMaxGrid = 148 * kBlocksPerSm;
constexpr int kOffsSmem = 1024;                      // group offsets cached in shared memory
constexpr uint32_t kStagePairs = 4096;               // selected pairs a block keeps in shared memory (32 KB)

struct CompressLayout {
    size_t rec_max, rec_min, block_total, stage_idx, stage_val, total;
};

static CompressLayout compress_layout(size_t n, int K)
{
    CompressLayout L;
    size_t off = 0;
    L.rec_max = off;       off = round_up(off + sizeof(uint32_t) * ((size_t)K + kMaxGrid), 256);
    L.rec_min = off;       off = round_up(off + sizeof(uint32_t) * ((size_t)K + kMaxGrid), 256);
    L.block_total = off;   off = round_up(off + sizeof(uint64_t) * kMaxGrid, 256);
    L.stage_idx = off;     off = round_up(off + sizeof(uint32_t) * n, 256);
    L.stage_val = off;     off = round_up(off + sizeof(uint32_t) * n, 256);
    L.total = off;
    return L;
}

struct CompressArgs {
    const float *g, *s;
    float *r, *v;
    size_t n;
    const uint32_t *group_offsets;
    int K;
    float alpha, zeta;
    uint32_t *rec_max, *rec_min;         // per (block, tensor) at [block + tensor]: |value| bit patterns
    uint64_t *block_total;               // per block: passed << 32 | kept
    uint32_t *stage_idx, *stage_val;     // pairs past kStagePairs of a block, from its first parameter's index on
    uint32_t per_block, tile;
    vgc_message out;
};

constexpr uint64_t kPassedShift = 32;
constexpr uint32_t kNoMin = 0x7FFFFFFFu;

__device__ __forceinline__ int32_t exponent_of(uint32_t max_bits)       // floor(log2 M_k)
{
    return max_bits ? (int32_t)((max_bits >> 23) & 0xFFu) - 127 : VGC_EXP_NONE;
}
__device__ __forceinline__ int32_t rounded_exponent(uint32_t bits)      // nearer power of two, midpoint up
{
    return (int32_t)((bits + 0x00400000u) >> 23) - 127;
}

// kHasS = false: the caller accumulated this step's squared-gradient sums straight into v (the sqgrad entry
// points with accumulate = 1), so the pass reads 12 instead of 16 bytes per parameter.
template <bool kHasS>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
compress_step(const __grid_constant__ CompressArgs a)
{
    extern __shared__ uint2 sm_pairs[];                 // kStagePairs (index, value bits)
    __shared__ uint32_t sm_offs[kOffsSmem];
    __shared__ uint32_t sm_part[2][32];                 // per-(row, warp) counts, double buffered
    __shared__ uint32_t sm_wmax[2][kWarps];
    __shared__ uint32_t sm_wmin[2][kWarps];             // smallest |value| bit pattern sent by each warp
    __shared__ uint32_t sm_end_max[2];                  // M_k bits of the range's first and last tensor
    __shared__ uint32_t sm_kept[kWarps];
    __shared__ unsigned long long sm_tot[kWarps];

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    const int K = a.K;
    const bool offs_in_smem = (K + 1) <= kOffsSmem;
    if (offs_in_smem)
        for (int i = tid; i <= K; i += kThreads) sm_offs[i] = a.group_offsets[i];
    const uint32_t *offs = offs_in_smem ? sm_offs : a.group_offsets;
    if (tid < 64) (&sm_part[0][0])[tid] = 0;            // entries past kRowsA*kWarps stay zero
    __syncthreads();

    const uint32_t lo = b * a.per_block;
    const uint32_t hi = (uint32_t)((size_t)lo + a.per_block < a.n ? (size_t)lo + a.per_block : a.n);
    const int k_first = group_of(offs, K, lo), k_last = group_of(offs, K, hi - 1);
    uint32_t *const rec_max = a.rec_max + b, *const rec_min = a.rec_min + b;     // this block's records, by tensor
    for (int k = k_first + (int)tid; k <= k_last; k += kThreads) { rec_max[k] = 0; rec_min[k] = kNoMin; }
    __syncthreads();

    // ---- step 1
    uint32_t run = 0;                                   // pairs of the block so far
    int k_tile = k_first;                               // tensor of the tile's first parameter
    int k_held = k_first;                               // thread 0: the tensor whose extremes it holds
    uint32_t held_max = 0, held_min = kNoMin;
    auto release = [&]() {
        if (held_max) { atomicMax(rec_max + k_held, held_max); atomicMin(rec_min + k_held, held_min); }
    };
    uint32_t buf = 0;
    for (uint32_t base = lo; base < hi; base += a.tile, buf ^= 1) {
        const uint32_t end = hi - base < a.tile ? hi : base + a.tile;

        // load: thread t owns elements base + (j*256 + t)*4 + {0..3}
        float4 G[kRowsA], S[kRowsA], R[kRowsA], V[kRowsA];
#pragma unroll
        for (int j = 0; j < kRowsA; ++j) {
            const uint32_t e = base + (j * kThreads + tid) * 4;
            if (e + 3 < end) {
                G[j] = ld_stream_f4(a.g + e);
                if (kHasS) S[j] = ld_stream_f4(a.s + e);
                R[j] = *reinterpret_cast<const float4 *>(a.r + e);
                V[j] = *reinterpret_cast<const float4 *>(a.v + e);
            } else {
                float tg[4], ts[4], tr[4], tv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const bool in = e + q < end;
                    tg[q] = in ? a.g[e + q] : 0.f;  ts[q] = (kHasS && in) ? a.s[e + q] : 0.f;
                    tr[q] = in ? a.r[e + q] : 0.f;  tv[q] = in ? a.v[e + q] : 0.f;
                }
                G[j] = make_float4(tg[0], tg[1], tg[2], tg[3]);  S[j] = make_float4(ts[0], ts[1], ts[2], ts[3]);
                R[j] = make_float4(tr[0], tr[1], tr[2], tr[3]);  V[j] = make_float4(tv[0], tv[1], tv[2], tv[3]);
            }
        }
        while (offs[k_tile + 1] <= base) ++k_tile;      // block-uniform
        const int grp = end <= offs[k_tile + 1] ? k_tile : -1;          // -1: the tile spans several tensors

        // Algorithm 1 loop body; every operation rounded on its own (no FMA)
        uint32_t send_bits = 0;          // bit j*4+q
        uint32_t packed = 0;             // per-row counts, 8 bits each
        uint32_t my_max = 0, my_min = kNoMin;
#pragma unroll
        for (int j = 0; j < kRowsA; ++j) {
            const uint32_t e = base + (j * kThreads + tid) * 4;
            float *Gj = reinterpret_cast<float *>(&G[j]);
            const float *Sj = reinterpret_cast<const float *>(&S[j]);
            float *Rj = reinterpret_cast<float *>(&R[j]);
            float *Vj = reinterpret_cast<float *>(&V[j]);
            uint32_t row_bits = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float r1 = __fadd_rn(Rj[q], Gj[q]);
                const float v1 = kHasS ? __fadd_rn(Vj[q], Sj[q]) : Vj[q];
                const float lhs = __fmul_rn(r1, r1);
                const float rhs = __fmul_rn(a.alpha, v1);
                const bool send = (lhs > rhs) && (e + q < end);
                Gj[q] = r1;                                       // value handed to Encode()
                Rj[q] = send ? 0.f : r1;
                Vj[q] = send ? 0.f : __fmul_rn(v1, a.zeta);
                if (send) {
                    row_bits |= 1u << q;
                    my_max = max(my_max, __float_as_uint(r1) & 0x7FFFFFFFu);
                    my_min = min(my_min, __float_as_uint(r1) & 0x7FFFFFFFu);
                }
            }
            send_bits |= row_bits << (4 * j);
            packed |= (uint32_t)__popc(row_bits) << (8 * j);
            if (e + 3 < end) {
                *reinterpret_cast<float4 *>(a.r + e) = R[j];
                *reinterpret_cast<float4 *>(a.v + e) = V[j];
                if (a.out.mask) {
                    const uint32_t m4 = (row_bits & 1u) | ((row_bits & 2u) << 7) | ((row_bits & 4u) << 14) |
                                        ((row_bits & 8u) << 21);
                    *reinterpret_cast<uint32_t *>(a.out.mask + e) = m4;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (e + q < end) {
                        a.r[e + q] = Rj[q];
                        a.v[e + q] = Vj[q];
                        if (a.out.mask) a.out.mask[e + q] = (row_bits >> q) & 1u;
                    }
            }
        }

        // ordered positions inside the tile: warp scan of the packed per-row counts, then every warp scans the 16
        // (row, warp) totals by itself (one barrier per tile)
        uint32_t incl = packed;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += up;
        }
        const uint32_t warp_max = __reduce_max_sync(0xffffffffu, my_max);
        const uint32_t warp_min = __reduce_min_sync(0xffffffffu, my_min);
        if (lane == 31) {
#pragma unroll
            for (int j = 0; j < kRowsA; ++j) sm_part[buf][j * kWarps + warp] = (incl >> (8 * j)) & 0xFFu;
            sm_wmax[buf][warp] = warp_max;
            sm_wmin[buf][warp] = warp_min;
        }
        __syncthreads();
        const uint32_t part = sm_part[buf][lane];
        uint32_t pincl = part;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, pincl, d);
            if (lane >= d) pincl += up;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, pincl, 31);
        const uint32_t pexcl = pincl - part;
#pragma unroll
        for (int j = 0; j < kRowsA; ++j) {
            const uint32_t row_base = __shfl_sync(0xffffffffu, pexcl, j * kWarps + warp);
            const uint32_t row_bits = (send_bits >> (4 * j)) & 0xFu;
            if (row_bits) {
                const uint32_t e = base + (j * kThreads + tid) * 4;
                uint32_t at = run + row_base + ((incl >> (8 * j)) & 0xFFu) - (uint32_t)__popc(row_bits);
                const float *Gj = reinterpret_cast<const float *>(&G[j]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (row_bits & (1u << q)) {
                        const uint32_t bits = __float_as_uint(Gj[q]);
                        if (at < kStagePairs) sm_pairs[at] = make_uint2(e + q, bits);
                        else { a.stage_idx[lo + at] = e + q; a.stage_val[lo + at] = bits; }
                        ++at;
                        if (grp < 0) {
                            const int k = group_of(offs, K, e + q);
                            atomicMax(rec_max + k, bits & 0x7FFFFFFFu);
                            atomicMin(rec_min + k, bits & 0x7FFFFFFFu);
                        }
                    }
            }
        }
        if (tid == 0 && grp >= 0 && total) {
            if (grp != k_held) { release(); k_held = grp; held_max = 0; held_min = kNoMin; }
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                held_max = max(held_max, sm_wmax[buf][w]);
                held_min = min(held_min, sm_wmin[buf][w]);
            }
        }
        run += total;
    }
    if (tid == 0) release();
    cg::this_grid().sync();

    // ---- step 2: M_k of the tensors that other blocks may share (the range's first and last one)
    if (warp < 2) {
        const int k = warp == 0 ? k_first : k_last;
        const uint32_t b0 = offs[k] / a.per_block, b1 = (offs[k + 1] - 1) / a.per_block;
        uint32_t m = 0;
        for (uint32_t c = b0 + lane; c <= b1; c += 32) m = max(m, __ldcg(a.rec_max + c + k));
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) sm_end_max[warp] = m;
    }
    __syncthreads();
    auto max_of = [&](int k) -> uint32_t {
        return k == k_first ? sm_end_max[0] : k == k_last ? sm_end_max[1] : __ldcg(rec_max + k);
    };
    {
        // exponents of the tensors that begin in this range (empty tensors at the buffer's end belong to the last block)
        int k0 = 0, k1 = K;                             // first k with offs[k] >= lo
        while (k0 < k1) {
            const int mid = (k0 + k1) >> 1;
            if (offs[mid] < lo) k0 = mid + 1; else k1 = mid;
        }
        const bool last = b == gridDim.x - 1;
        for (int k = k0 + (int)tid; k < K && (last || offs[k] < hi); k += kThreads)
            a.out.group_exp[k] = offs[k] < offs[k + 1] ? exponent_of(max_of(k)) : VGC_EXP_NONE;
    }
    // nothing is dropped when even the smallest value sent from each tensor is within 7 binades of its exponent
    bool drops = false;
    for (int k = k_first + (int)tid; k <= k_last; k += kThreads) {
        const uint32_t m = __ldcg(rec_min + k);
        if (m != kNoMin && rounded_exponent(m) < exponent_of(max_of(k)) - 7) drops = true;
    }
    drops = __syncthreads_or(drops);

    // pair i of the block -> its word; true if a word is emitted.  k: the tensor of the last pair looked at
    auto pair_at = [&](uint32_t i) -> uint2 {
        return i < kStagePairs ? sm_pairs[i] : make_uint2(a.stage_idx[lo + i], a.stage_val[lo + i]);
    };
    auto encode = [&](uint2 p, int &k, int32_t &Ek, uint32_t &word) -> bool {
        if (p.x < offs[k] || p.x >= offs[k + 1] || Ek == INT32_MIN) {
            k = k_first == k_last ? k_first : group_of(offs, K, p.x);
            Ek = exponent_of(max_of(k));
        }
        const int32_t e1 = rounded_exponent(p.y & 0x7FFFFFFFu);
        const int32_t d = Ek - (e1 < Ek ? e1 : Ek);                        // cut at 2^E_k
        word = (p.x << 4) | ((p.y >> 31) << 3) | (uint32_t)(d & 7);
        return d <= 7;
    };
    // with drops every warp walks a section of the pairs, four 32-wide slices per round
    const uint32_t section = ((run + kWarps - 1) / kWarps + 31u) & ~31u;
    const uint32_t s0 = min(run, warp * section), s1 = min(run, s0 + section);
    auto walk = [&](auto emit) {
        int k = k_first;
        int32_t Ek = INT32_MIN;
        uint32_t kept = 0;
        for (uint32_t i0 = s0; i0 < s1; i0 += 128) {
            uint2 p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * 32 + lane;
                p[u] = i < s1 ? pair_at(i) : make_uint2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                bool keep = false;
                uint32_t word = 0;
                if (i0 + u * 32 + lane < s1) keep = encode(p[u], k, Ek, word);
                const uint32_t ballot = __ballot_sync(0xffffffffu, keep);
                if (keep) emit(kept + __popc(ballot & ((1u << lane) - 1u)), word);
                kept += __popc(ballot);
            }
        }
        return kept;
    };
    uint32_t kept = run;
    if (drops) {
        const uint32_t mine = walk([](uint32_t, uint32_t) {});
        if (lane == 0) sm_kept[warp] = mine;
        __syncthreads();
        kept = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) kept += sm_kept[w];
    }
    const unsigned long long own = ((unsigned long long)run << kPassedShift) | kept;
    if (tid == 0) a.block_total[b] = own;
    cg::this_grid().sync();

    // ---- step 3: totals of the blocks before this one, then the words
    unsigned long long before = 0;
    for (uint32_t c = tid; c < b; c += kThreads) before += __ldcg(reinterpret_cast<unsigned long long *>(a.block_total) + c);
    before = warp_sum_u64(before);
    if (lane == 0) sm_tot[warp] = before;
    __syncthreads();
    before = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) before += sm_tot[w];
    uint32_t pos = (uint32_t)(before & 0xFFFFFFFFull);
    if (tid == 0) {
        if (pos + kept > a.out.capacity) atomicOr(a.out.dev_status, VGC_DEV_CAPACITY);
        if (b == gridDim.x - 1) {
            const unsigned long long all = before + own;
            *a.out.nnz = (uint32_t)(all & 0xFFFFFFFFull);
            *a.out.n_criterion = (uint32_t)(all >> kPassedShift);
            *a.out.n_dropped = (uint32_t)(all >> kPassedShift) - (uint32_t)(all & 0xFFFFFFFFull);
        }
    }
    if (drops) {
#pragma unroll
        for (uint32_t w = 0; w < kWarps; ++w) pos += w < warp ? sm_kept[w] : 0u;
        walk([&](uint32_t at, uint32_t word) {
            if (pos + at < a.out.capacity) a.out.words[pos + at] = word;
        });
    } else {
        int k = k_first;
        int32_t Ek = INT32_MIN;
        for (uint32_t i = tid; i < run; i += kThreads) {
            uint32_t word;
            encode(pair_at(i), k, Ek, word);
            if (pos + i < a.out.capacity) a.out.words[pos + i] = word;
        }
    }
}

}  // namespace vgc

// ------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------
using namespace vgc;

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

    const void *fn = s ? reinterpret_cast<const void *>(compress_step<true>) : reinterpret_cast<const void *>(compress_step<false>);
    constexpr size_t smem = kStagePairs * sizeof(uint2);
    static ResidentBlocks resident[2];
    const uint32_t most = resident[s ? 1 : 0].get(fn, kThreads, smem);
    if (most == 0) return VGC_ERR_CUDA;
    const Ranges R = even_ranges(n, most < (uint32_t)kMaxGrid ? most : (uint32_t)kMaxGrid, kTileA);

    char *base = static_cast<char *>(ws);
    CompressArgs args;
    args.g = g; args.s = s; args.r = r; args.v = v; args.n = n;
    args.group_offsets = group_offsets; args.K = K; args.alpha = alpha; args.zeta = zeta;
    args.rec_max = reinterpret_cast<uint32_t *>(base + L.rec_max);
    args.rec_min = reinterpret_cast<uint32_t *>(base + L.rec_min);
    args.block_total = reinterpret_cast<uint64_t *>(base + L.block_total);
    args.stage_idx = reinterpret_cast<uint32_t *>(base + L.stage_idx);
    args.stage_val = reinterpret_cast<uint32_t *>(base + L.stage_val);
    args.per_block = R.per_block; args.tile = R.tile;
    args.out = *out;
    void *params[] = {&args};
    VGC_CUDA_OK(cudaLaunchCooperativeKernel(fn, dim3(R.grid), dim3(kThreads), params, smem,
                                            reinterpret_cast<cudaStream_t>(stream)));
    count_launch();
    return VGC_OK;
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
    static void *scratch_of_device[kMaxDevices] = {};
    int dev = -1;
    VGC_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return VGC_ERR_UNSUPPORTED;
    if (!scratch_of_device[dev]) {
        void *p = nullptr;
        VGC_CUDA_OK(cudaGetSymbolAddress(&p, g_compress_scratch));
        if (!p) return VGC_ERR_CUDA;
        scratch_of_device[dev] = p;
    }
    return vgc_compress(g, s, r, v, n, group_offsets, K, alpha, zeta, out, scratch_of_device[dev], kStaticScratchBytes,
                        stream);
}
