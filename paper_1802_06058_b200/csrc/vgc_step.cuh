// The streaming pass shared by vgc_compress (Algorithm 1, "Basic") and vgc_compress_hybrid (Algorithm 2): one step over
// the flat parameter buffer and the message it sends.
//
// Every thread block owns one contiguous range of the buffer:
//   1  it streams g, s, r, v once (16 B read + 8 B written per parameter), applies the send test, writes r, v back and
//      stages what was selected in index order, 32 bits each -- position in the range, sign, rounded exponent: all the
//      quantiser needs.  For every weight tensor the range touches it records the largest |value| sent.
//   2  E_k = floor(log2 M_k) needs the records of every block that shares tensor k, and a block's first word's place
//      needs to know how many staged values of the blocks before it survive the quantiser (d <= 7).
//   3  it writes its words.
// Steps 2 and 3 are a second kernel: at the end of its range a block of the first one counts how many of the staged values
// of the range's first and last tensor (the two that other blocks may share) survive for each exponent E_k can turn out to
// have, nine at most.  (Counting them as they are selected, in a shared-memory histogram, cost 20 % at density 0.15.)
// With these the second kernel's blocks work out E_k, every block's surviving count and their own place from the records
// alone: no block waits for another, and nothing has to be cleared by a launch of its own.  It is launched so that it
// starts under the end of the first.
// The hybrid algorithm has neither maxima nor quantiser.
//
// Bound: HBM, 24 B per parameter, for large buffers (the first kernel: 612 MB in 101.5 us, 0.92 of the measured copy
// rate) -- the latency of launches and exchanges for small ones.  Measured against the memset and three kernels this
// replaces (B200, one call among others, Algorithm 1, density 1e-2): n = 25.5 M  125.9 -> 110.0 us,
// n = 138 M at density 0.05  627 -> 563 us,  n = 3e4 .. 4e5  19 -> 9 us.
// In between stood one kernel: cooperative, its grid barriers cost 2.4 us each with 16 blocks and 5 us with 592, polled
// slots 2 us and 4 us, the cooperative launch itself 2.5 us on either side; as one cluster of 16 blocks with distributed
// shared memory it took as long as these two kernels at n = 8192 and 22 % longer at 131072.
#pragma once

#include "vgc_common.cuh"

namespace vgc {
namespace step {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / kWarp;             // 16
constexpr int kBlocksPerSm = 2;                      // 64 registers: 1024 threads with eight 16-byte loads each in flight
constexpr int kRowsA = 2;                            // float4 vectors per thread per tile
constexpr int kTileA = kThreads * kRowsA * 4;        // at most 4096 parameters per tile
constexpr int kLeastPerBlock = 2048;
constexpr int kMaxGrid = 148 * kBlocksPerSm;
static_assert(kMaxGrid <= kThreads, "the second kernel reads one record per thread");
constexpr int kOffsSmem = 1024;                      // group offsets cached in shared memory
constexpr uint32_t kStagedCopy = 2048;
// a staged value: position in the block's range << 10 | sign << 9 | (rounded exponent + 127)
constexpr uint32_t kPosShift = 10;
static_assert(((size_t)VGC_MAX_PARAMS + kMaxGrid - 1) / kMaxGrid + 128 <= (size_t)1 << (32 - kPosShift), "a block's range");

enum { kBasic = 0, kHybridBefore = 1, kHybridAfter = 2 };     // the hybrid's correction uses |r| from before / after r -= Sign(r) tau

// What the first kernel leaves about a block's range.
struct __align__(16) Record {
    uint32_t max_first, max_last;        // largest |value| bits sent from the range's first and last tensor
    uint32_t head;                       // block where the first tensor begins; top bit: it is also the last tensor
    uint32_t passed;                     // values staged
};
constexpr uint32_t kSame = 0x80000000u;
// how many of the staged values survive, per exponent E_k above the block's own one ([0] = the same): first tensor, last
// tensor; then those of the tensors between them, which no other block shares
constexpr int kLevels = 9, kCounts = 2 * kLevels + 1;
constexpr size_t kRecordBytes = (sizeof(Record) + sizeof(uint32_t) * kCounts) * kMaxGrid;

struct Args {
    const float *g, *s;
    float *r, *v;
    size_t n;
    const uint32_t *group_offsets;
    int K;
    float alpha, zeta;
    Record *records;                     // [block]
    uint32_t *counts;                    // [block][kCounts]
    uint32_t *rec_max;                   // per (block, tensor) at [block + tensor]: |value| bits of the tensors inside
    uint32_t *stage;                     // staged values of a block from its first parameter's index on
    uint32_t per_block, tile;
    float tau;                           // hybrid only
    vgc_message out;                     // (hybrid: no exponents, nnz only)
};

// Blocks and the tensors they touch advance together, so that index block + tensor of rec_max is nobody else's.

__device__ __forceinline__ int32_t exponent_of(uint32_t max_bits)       // floor(log2 M_k)
{
    return max_bits ? (int32_t)((max_bits >> 23) & 0xFFu) - 127 : VGC_EXP_NONE;
}
__device__ __forceinline__ int32_t rounded_exponent(uint32_t bits)      // nearer power of two, midpoint up
{
    return (int32_t)((bits + 0x00400000u) >> 23) - 127;
}

// exponents of the tensors that begin in [lo, hi) (empty tensors at the buffer's end belong to the last block)
template <class MaxOf>
__device__ __forceinline__ void write_exponents(const Args &a, const uint32_t *offs, uint32_t lo, uint32_t hi, bool last,
                                                const MaxOf &max_of)
{
    int k0 = 0, k1 = a.K;                               // first k with offs[k] >= lo
    while (k0 < k1) {
        const int mid = (k0 + k1) >> 1;
        if (offs[mid] < lo) k0 = mid + 1; else k1 = mid;
    }
    for (int k = k0 + (int)threadIdx.x; k < a.K && (last || offs[k] < hi); k += kThreads)
        a.out.group_exp[k] = offs[k] < offs[k + 1] ? exponent_of(max_of(k)) : VGC_EXP_NONE;
}

// staged value -> word; true if the word is emitted (d <= 7).  Holds the tensor of the last value it saw.
template <bool kQuantise>
struct Encoder {
    const uint32_t *offs;
    int K, k_first, k_last, k;
    uint32_t lo;
    int32_t Ek;
    __device__ __forceinline__ Encoder(const uint32_t *offs_, int K_, uint32_t lo_, int k_first_, int k_last_)
        : offs(offs_), K(K_), k_first(k_first_), k_last(k_last_), k(-1), lo(lo_), Ek(0) {}
    template <class MaxOf>
    __device__ __forceinline__ bool operator()(uint32_t staged, const MaxOf &max_of, uint32_t &word)
    {
        const uint32_t idx = lo + (staged >> kPosShift);
        word = (idx << 4) | ((staged >> 6) & 8u);
        if (!kQuantise) return true;
        if (k < 0 || (k_first != k_last && (idx < offs[k] || idx >= offs[k + 1]))) {
            k = k_first == k_last ? k_first : group_of(offs, K, idx);
            Ek = exponent_of(max_of(k));
        }
        const int32_t e1 = (int32_t)(staged & 0x1FFu) - 127;
        const int32_t d = Ek - (e1 < Ek ? e1 : Ek);                        // cut at 2^E_k
        word |= (uint32_t)(d & 7);
        return d <= 7;
    }
};

// counters of the message: passed and kept values up to and with this block's
__device__ __forceinline__ void finish(const Args &a, bool last, bool quantise, uint32_t passed, uint32_t kept)
{
    if (threadIdx.x != 0) return;
    if (kept > a.out.capacity) atomicOr(a.out.dev_status, VGC_DEV_CAPACITY);
    if (last) {
        *a.out.nnz = kept;
        if (quantise) {
            *a.out.n_criterion = passed;
            *a.out.n_dropped = passed - kept;
        }
    }
}

// kHasS = false: the caller accumulated this step's squared-gradient sums straight into v (the sqgrad entry
// points with accumulate = 1), so the pass reads 12 instead of 16 bytes per parameter.
template <bool kHasS, int kAlgorithm>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
compress_step(const __grid_constant__ Args a)
{
    constexpr bool kQuantise = kAlgorithm == kBasic;
    __shared__ uint32_t sm_offs[kOffsSmem];
    __shared__ uint32_t sm_part[2][kRowsA * kWarps];    // per-(row, warp) counts, double buffered
    __shared__ uint32_t sm_wmax[2][kWarps];
    __shared__ uint32_t sm_rec_max[2];                  // maxima of the range's first and last tensor
    __shared__ uint32_t sm_fields[kWarps][7];
    __shared__ uint32_t sm_staged[kStagedCopy];         // the first staged values once more, for the count at the end

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    const int K = a.K;
    grid_wait();
    grid_release();                                     // in this order: encode_step reads the offsets before it waits for us
    const bool offs_in_smem = kQuantise && (K + 1) <= kOffsSmem;
    if (offs_in_smem) {                                 // asynchronously: the first tile's loads go out before they arrive
        for (int i = tid; i <= K; i += kThreads)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                         ::"r"((uint32_t)__cvta_generic_to_shared(sm_offs + i)), "l"(a.group_offsets + i) : "memory");
    }
    const uint32_t *offs = offs_in_smem ? sm_offs : a.group_offsets;
    const uint32_t lo = b * a.per_block;
    const uint32_t hi = (uint32_t)((size_t)lo + a.per_block < a.n ? (size_t)lo + a.per_block : a.n);
    if (tid < 2) sm_rec_max[tid] = 0;
    uint32_t *const rec_max = a.rec_max + b;            // this block's records, by tensor
    int k_first = 0, k_last = 0;

    const float tau_sq = __fmul_rn(a.tau, a.tau);
    uint32_t run = 0;                                   // values staged by the block so far
    int k_tile = 0;                                     // tensor of the tile's first parameter
    int k_held = 0;                                     // thread 0: the tensor whose maximum it holds
    uint32_t held_max = 0;
    // largest |value| bits of tensor k: the range's first and last tensor in shared memory (all there is, mostly), the
    // ones between them in the workspace
    auto record = [&](int k, uint32_t most) {
        atomicMax(k == k_first ? sm_rec_max : k == k_last ? sm_rec_max + 1 : rec_max + k, most);
    };
    uint32_t buf = 0;
    for (uint32_t base = lo; base < hi; base += a.tile, buf ^= 1) {
        const uint32_t end = hi - base < a.tile ? hi : base + a.tile;

        // load: thread t owns elements base + (j*512 + t)*4 + {0..3}
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
        if (base == lo) {
            if (offs_in_smem) asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
            __syncthreads();
        }
        if (kQuantise && base == lo) {
            k_first = group_of(offs, K, lo);
            k_last = hi <= offs[k_first + 1] ? k_first : group_of(offs, K, hi - 1);
            k_tile = k_held = k_first;
            for (int k = k_first + 1 + (int)tid; k < k_last; k += kThreads) rec_max[k] = 0;
        }
        if (kQuantise)
            while (offs[k_tile + 1] <= base) ++k_tile;  // block-uniform
        const int grp = !kQuantise || end <= offs[k_tile + 1] ? k_tile : -1;      // -1: the tile spans several tensors

        // loop body of Algorithm 1 / Algorithm 2; every operation rounded on its own (no FMA)
        uint32_t send_bits = 0;          // bit j*4+q
        uint32_t packed = 0;             // per-row counts, 8 bits each
        uint32_t my_max = 0;
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
                const bool send = (lhs > rhs) && (e + q < end) && (kQuantise || fabsf(r1) > a.tau);
                Gj[q] = r1;                                       // value handed to Encode()
                if (kQuantise) {
                    Rj[q] = send ? 0.f : r1;
                    Vj[q] = send ? 0.f : __fmul_rn(v1, a.zeta);
                    if (send) my_max = max(my_max, __float_as_uint(r1) & 0x7FFFFFFFu);
                } else {
                    const float r2 = r1 < 0.f ? __fadd_rn(r1, a.tau) : __fsub_rn(r1, a.tau);     // r -= Sign(r) tau
                    const float cross = __fmul_rn(__fmul_rn(2.0f, kAlgorithm == kHybridBefore ? fabsf(r1) : fabsf(r2)), a.tau);
                    const float corr = __fadd_rn(__fsub_rn(v1, cross), tau_sq);                  // v - 2|r|tau + tau^2
                    Rj[q] = send ? r2 : r1;
                    Vj[q] = __fmul_rn(send ? (corr > 0.f ? corr : 0.f) : v1, a.zeta);            // decay at every step
                }
                row_bits |= (send ? 1u : 0u) << q;
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

        // ordered positions inside the tile: warp scan of the packed per-row counts, then every warp scans the 32
        // (row, warp) totals by itself (one barrier per tile)
        uint32_t incl = packed;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += up;
        }
        const uint32_t warp_max = kQuantise ? __reduce_max_sync(0xffffffffu, my_max) : 0u;
        if (lane == 31) {
#pragma unroll
            for (int j = 0; j < kRowsA; ++j) sm_part[buf][j * kWarps + warp] = (incl >> (8 * j)) & 0xFFu;
            sm_wmax[buf][warp] = warp_max;
        }
        __syncthreads();
        static_assert(kRowsA * kWarps == 32, "one count per lane");
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
                        const uint32_t staged = (e + q - lo) << kPosShift | (bits >> 31) << 9 |
                                                (uint32_t)(rounded_exponent(bits & 0x7FFFFFFFu) + 127);
                        a.stage[lo + at] = staged;
                        if (kQuantise && at < kStagedCopy) sm_staged[at] = staged;
                        ++at;
                    }
            }
        }
        if (kQuantise && grp < 0 && send_bits) {         // a thread's values mostly share a tensor: one search, one maximum
            int k_mine = k_tile;
            uint32_t mine_max = 0;
#pragma unroll 1
            for (uint32_t left = send_bits; left; left &= left - 1u) {
                const uint32_t c = (uint32_t)__ffs(left) - 1u, i = base + ((c >> 2) * kThreads + tid) * 4 + (c & 3u);
                uint32_t bits = 0;
#pragma unroll
                for (int j = 0; j < kRowsA; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (c == (uint32_t)(4 * j + q)) bits = __float_as_uint(reinterpret_cast<const float *>(&G[j])[q]) & 0x7FFFFFFFu;
                if (i < offs[k_mine] || i >= offs[k_mine + 1]) {
                    if (mine_max) record(k_mine, mine_max);
                    k_mine = group_of(offs, K, i); mine_max = 0;
                }
                mine_max = max(mine_max, bits);
            }
            record(k_mine, mine_max);
        }
        if (kQuantise && tid == 0 && grp >= 0 && total) {
            if (grp != k_held) {
                if (held_max) record(k_held, held_max);
                k_held = grp; held_max = 0;
            }
#pragma unroll
            for (int w = 0; w < kWarps; ++w) held_max = max(held_max, sm_wmax[buf][w]);
        }
        run += total;
    }
    if (tid == 0 && held_max) record(k_held, held_max);
    __syncthreads();
    const bool same = k_first == k_last;

    // ---- what the second kernel needs to know
    if (kQuantise) {
        // a value survives E_k = own + j (own: this block's exponent for the tensor) if e >= own + j - 7, and e <= own + 1.
        // A thread counts its values by e - own + 7 in nine 7-bit fields per tensor; a warp adds them in fields of ten
        // bits (at most 24 values per thread in between), three to a word
        const uint32_t first_end = offs[k_first + 1], last_begin = offs[k_last];
        const int own_first = (int)(sm_rec_max[0] >> 23), own_last = (int)(sm_rec_max[1] >> 23);         // biased
        constexpr uint32_t kBatch = 8, kRound = 3 * kBatch * kThreads;
        uint32_t sums = 0;                               // thread j of the first kCounts: entry j
        int k_in = -1, own_in = 0;                       // the tensor looked at last of those between the first and the last one
        for (uint32_t i0 = 0; i0 < run; i0 += kRound) {  // block-uniform
            unsigned long long of_first = 0, of_last = 0;
            uint32_t inside = 0;
            const uint32_t i1 = min(run, i0 + kRound);
            for (uint32_t i = i0 + tid; i < i1; i += kBatch * kThreads) {
                uint32_t staged[kBatch];
#pragma unroll
                for (uint32_t u = 0; u < kBatch; ++u) {
                    const uint32_t at = i + u * kThreads;
                    staged[u] = at >= i1 ? 0u : at < kStagedCopy ? sm_staged[at] : __ldcg(a.stage + lo + at);
                }
#pragma unroll
                for (uint32_t u = 0; u < kBatch; ++u) {
                    if (i + u * kThreads >= i1) break;
                    const uint32_t idx = lo + (staged[u] >> kPosShift);
                    const int e = (int)(staged[u] & 0x1FFu);
                    if (idx < first_end) {
                        const int level = e - own_first + 7;
                        if (level >= 0) of_first += 1ull << (7 * level);
                    } else if (idx >= last_begin) {
                        const int level = e - own_last + 7;
                        if (level >= 0) of_last += 1ull << (7 * level);
                    } else {                             // a tensor wholly inside: E_k is this block's
                        if (k_in < 0 || idx < offs[k_in] || idx >= offs[k_in + 1]) {
                            k_in = group_of(offs, K, idx);
                            own_in = (int)(__ldcg(rec_max + k_in) >> 23);
                        }
                        inside += e >= own_in - 7 ? 1u : 0u;
                    }
                }
            }
            auto add_up = [&](unsigned long long f, uint32_t *to) {
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const uint32_t g = (uint32_t)(f >> (21 * w));
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, (g & 0x7Fu) | (g & 0x3F80u) << 3 | (g & 0x1FC000u) << 6);
                    if (lane == 0) to[w] = sum;
                }
            };
            add_up(of_first, sm_fields[warp]);
            if (!same) {
                add_up(of_last, sm_fields[warp] + 3);
                inside = __reduce_add_sync(0xffffffffu, inside);
                if (lane == 0) sm_fields[warp][6] = inside;
            }
            __syncthreads();
            if (tid < (uint32_t)kCounts && !(same && tid >= (uint32_t)kLevels)) {
                const int j = (int)tid % kLevels;
                const uint32_t at = tid < 2u * kLevels ? 3 * (tid / kLevels) + j / 3 : 6, shift = tid < 2u * kLevels ? 10 * (j % 3) : 0;
                const uint32_t field = tid < 2u * kLevels ? 0x3FFu : 0xFFFFFFFFu;
#pragma unroll
                for (int w = 0; w < kWarps; ++w) sums += (sm_fields[w][at] >> shift) & field;
            }
            if (i0 + kRound < run) __syncthreads();
        }
        // entry j of a tensor: the values of levels >= j
        if (warp == 0) {
            const int level = (int)lane % kLevels;
#pragma unroll
            for (int d = 1; d < kLevels; d <<= 1) {
                const uint32_t up = __shfl_down_sync(0xffffffffu, sums, d);
                if (lane < 2u * kLevels && level + d < kLevels) sums += up;
            }
            if (lane < (uint32_t)kCounts) a.counts[b * kCounts + lane] = sums;
        }
    }
    if (tid == 0) {
        Record rec;
        rec.max_first = sm_rec_max[0];
        rec.max_last = sm_rec_max[same ? 0 : 1];
        rec.head = (kQuantise ? offs[k_first] / a.per_block : 0u) | (same ? kSame : 0u);
        rec.passed = run;
        a.records[b] = rec;
    }
}

// The second kernel: same blocks, same ranges.  Before its grid_wait() it reads the offsets only (from L2), which nothing
// writes any more: it starts when every block of the first kernel has passed its own.
template <bool kQuantise>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
encode_step(const __grid_constant__ Args a)
{
    __shared__ uint32_t sm_offs[kOffsSmem];
    __shared__ uint32_t sm_begun[kMaxGrid];             // M_k bits of the last tensor of every block
    __shared__ uint32_t sm_end_max[2];                  // ... of this block's first and last tensor
    __shared__ uint32_t sm_passed[kWarps], sm_kept[kWarps], sm_own[2];
    constexpr int kPerRound = 4;
    __shared__ __align__(8) uint32_t sm_part[2][kPerRound * kWarps];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x, blocks = gridDim.x;
    const int K = a.K;
    const bool offs_in_smem = kQuantise && (K + 1) <= kOffsSmem;
    if (offs_in_smem)
        for (int i = tid; i <= K; i += kThreads) sm_offs[i] = __ldcg(a.group_offsets + i);
    else if (kQuantise) grid_wait();                    // read where they are, through L1
    const uint32_t *offs = offs_in_smem ? sm_offs : a.group_offsets;
    const uint32_t lo = b * a.per_block;
    const uint32_t hi = (uint32_t)((size_t)lo + a.per_block < a.n ? (size_t)lo + a.per_block : a.n);
    if (kQuantise && tid < blocks) sm_begun[tid] = 0;
    __syncthreads();
    int k_first = 0, k_last = 0;
    if (kQuantise) { k_first = group_of(offs, K, lo); k_last = hi <= offs[k_first + 1] ? k_first : group_of(offs, K, hi - 1); }
    grid_wait();

    // the values of the first round are asked for together with the records
    const uint32_t *staged = a.stage + lo;
    uint32_t next[kPerRound];
#pragma unroll
    for (int u = 0; u < kPerRound; ++u) next[u] = u * kThreads + tid < hi - lo ? __ldcg(staged + u * kThreads + tid) : 0u;
    Record rec = {0, 0, 0, 0};
    if (tid < blocks) {
        const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(a.records) + tid);
        rec.max_first = q.x; rec.max_last = q.y; rec.head = q.z; rec.passed = q.w;
    }
    const uint32_t head = rec.head & ~kSame;
    const bool same = rec.head & kSame, shared_first = head < tid;
    uint32_t kept = rec.passed;
    if (kQuantise) {
        if (tid < blocks) {
            // a tensor that spans several blocks is the last one of the block it begins in and the first one of the others
            if (shared_first) atomicMax(&sm_begun[head], rec.max_first);
            if (!(same && shared_first)) atomicMax(&sm_begun[tid], rec.max_last);
        }
        __syncthreads();
        kept = 0;
        if (tid <= b) {
            const uint32_t m_first = shared_first ? sm_begun[head] : same ? sm_begun[tid] : rec.max_first;
            const uint32_t m_last = same ? m_first : sm_begun[tid];
            const uint32_t *counts = a.counts + tid * kCounts;
            const uint32_t up_first = (m_first >> 23) - (rec.max_first >> 23), up_last = (m_last >> 23) - (rec.max_last >> 23);
            const uint32_t of_first = up_first < kLevels ? __ldcg(counts + up_first) : 0u;
            const uint32_t of_last = !same && up_last < kLevels ? __ldcg(counts + kLevels + up_last) : 0u;
            kept = of_first + of_last + __ldcg(counts + 2 * kLevels);
            if (tid == b) { sm_end_max[0] = m_first; sm_end_max[1] = m_last; }
        }
    }
    if (tid == b) { sm_own[0] = rec.passed; sm_own[1] = kept; }
    const uint32_t passed_w = __reduce_add_sync(0xffffffffu, tid < b ? rec.passed : 0u);
    const uint32_t kept_w = __reduce_add_sync(0xffffffffu, tid < b ? kept : 0u);
    if (lane == 0) { sm_passed[warp] = passed_w; sm_kept[warp] = kept_w; }
    __syncthreads();
    uint32_t passed_before = 0, pos = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { passed_before += sm_passed[w]; pos += sm_kept[w]; }
    const uint32_t run = sm_own[0];
    finish(a, b == blocks - 1, kQuantise, passed_before + run, pos + sm_own[1]);
    const uint32_t *rec_max = a.rec_max + b;
    auto max_of = [&](int k) -> uint32_t {
        return k == k_first ? sm_end_max[0] : k == k_last ? sm_end_max[1] : __ldcg(rec_max + k);
    };
    if (kQuantise) write_exponents(a, offs, lo, hi, b == blocks - 1, max_of);

    // words, 4 x 512 values a round (a thread's are 512 apart: neighbouring lanes write neighbouring words); where some are
    // dropped, a scan over the (512 values, warp) counts of the survivors gives the places
    Encoder<kQuantise> enc(offs, K, lo, k_first, k_last);
    const bool drops = kQuantise && sm_own[1] != run;
    uint32_t buf = 0;
    for (uint32_t i0 = 0; i0 < run; i0 += kPerRound * kThreads, buf ^= 1) {
        uint32_t now[kPerRound], word[kPerRound], ballot[kPerRound];
#pragma unroll
        for (int u = 0; u < kPerRound; ++u) {
            now[u] = next[u];
            const uint32_t i = i0 + (kPerRound + u) * kThreads + tid;
            next[u] = i < run ? __ldcg(staged + i) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kPerRound; ++u) {
            const bool keep = i0 + u * kThreads + tid < run && enc(now[u], max_of, word[u]);
            ballot[u] = __ballot_sync(0xffffffffu, keep);
        }
        if (!drops) {
#pragma unroll
            for (int u = 0; u < kPerRound; ++u) {
                const uint32_t i = i0 + u * kThreads + tid;
                if (i < run && pos + i < a.out.capacity) a.out.words[pos + i] = word[u];
            }
            continue;
        }
        if (lane < (uint32_t)kPerRound) {
            uint32_t c = 0;
#pragma unroll
            for (int u = 0; u < kPerRound; ++u) c = lane == (uint32_t)u ? (uint32_t)__popc(ballot[u]) : c;
            sm_part[buf][lane * kWarps + warp] = c;
        }
        __syncthreads();
        static_assert(kPerRound * kWarps == 64, "two counts per lane");
        const uint2 two = *reinterpret_cast<const uint2 *>(&sm_part[buf][2 * lane]);
        uint32_t incl = two.x + two.y;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += up;
        }
        const uint32_t before_two = incl - two.x - two.y;
#pragma unroll
        for (int u = 0; u < kPerRound; ++u) {
            const uint32_t entry = u * kWarps + warp;
            uint32_t at = __shfl_sync(0xffffffffu, before_two, entry >> 1);
            const uint32_t even = __shfl_sync(0xffffffffu, two.x, entry >> 1);
            at += pos + (entry & 1u ? even : 0u) + __popc(ballot[u] & ((1u << lane) - 1u));
            if ((ballot[u] >> lane & 1u) && at < a.out.capacity) a.out.words[at] = word[u];
        }
        pos += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// Buffers from which on the streaming kernel asks for L1.  Steps of one dense layer, 60 examples, without / with, us: 131 thousand
// parameters 12.9 / 13.9, 262 and 524 thousand the same, 1.05 M 19.4 / 19.0 (added to v 19.4 / 19.6), 2.1 M 25.4 / 23.6, 8.4 M 69.0 / 58.8.
constexpr size_t kCarveLeast = 1 << 20;

// Enqueues one step.  a: everything but the ranges; records: kRecordBytes, 16-byte aligned.
template <bool kHasS, int kAlgorithm>
vgc_status launch(Args a, void *records, cudaStream_t st)
{
    a.records = static_cast<Record *>(records);
    a.counts = reinterpret_cast<uint32_t *>(a.records + kMaxGrid);
    // every block the same share (to 128 parameters: 512 B of every stream), cut into tiles of equal size
    const size_t shares = (a.n + kLeastPerBlock - 1) / kLeastPerBlock;
    const size_t blocks = shares < (size_t)kMaxGrid ? shares : (size_t)kMaxGrid;
    const size_t per = round_up((a.n + blocks - 1) / blocks, 128);
    const size_t tiles = (per + kTileA - 1) / kTileA;
    a.per_block = (uint32_t)per;
    a.tile = (uint32_t)round_up((per + tiles - 1) / tiles, 128);
    const dim3 grid((unsigned)((a.n + per - 1) / per));
    // Two blocks' 26 KB, the rest L1: 1024 threads with eight 16-byte loads each.  Behind a dense layer's kernel without it (119.6 M
    // parameters, B200): 531 us for this kernel, 383 with it.  Not the hybrid, which asks for next to no shared memory and would
    // rather start under a decoder (25 M, 8 messages: 129.7 us a step, 131.1 with it).
    const Carveout carveout{kAlgorithm == kBasic && a.n >= kCarveLeast ? 15 : -1};
    VGC_CUDA_OK(launch_kernel(carveout, compress_step<kHasS, kAlgorithm>, grid, dim3(kThreads), 0, st, true, a));
    VGC_CUDA_OK(launch_kernel(encode_step<kAlgorithm == kBasic>, grid, dim3(kThreads), 0, st, true, a));
    count_launch(2);
    return VGC_OK;
}

}  // namespace step
}  // namespace vgc
