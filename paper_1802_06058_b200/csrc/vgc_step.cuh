// The streaming pass shared by vgc_compress (Algorithm 1, "Basic") and vgc_compress_hybrid (Algorithm 2): one step over
// the flat parameter buffer and the message it sends.
//
// One cooperative kernel.  Every thread block owns one contiguous range of the buffer and goes through three steps;
// between them the blocks hand each other 16-byte slots (the per-tensor maximum has to be complete before any value can
// be quantised, and the number of words before a block's own before it can write them):
//   1  streams g, s, r, v once (16 B read + 8 B written per parameter), applies the send test, writes r, v back and
//      keeps what was selected in index order, 32 bits each -- position in the range, sign, rounded exponent: all the
//      quantiser needs.  The first kStaged of them stay in shared memory, the rest goes to the block's part of the
//      workspace.  For every weight tensor the range touches it records the largest and the smallest |value| sent.
//   2  E_k = floor(log2 M_k) of the tensors at the range's two ends from the other blocks' slots (tensors inside the
//      range are complete already); how many selected values survive the quantiser (d <= 7): all of them unless a
//      recorded minimum says otherwise.
//   3  adds up the counts of the blocks before its own and writes its words.
// The hybrid algorithm has neither maxima nor quantiser: its step 2 is only the hand-shake that the slots ask for.
//
// Bound: HBM, 24 B per parameter, for large buffers -- the latency of the launch and of the two exchanges (about 2 us
// each with 16 blocks, 4 us with 296) for small ones.  The contiguous ranges keep everything a block selects in its own
// shared memory; two blocks of 512 threads per SM stream as fast as four of 256 (612 MB in 101.5 us, 0.92 of the
// measured copy rate) and halve the slots every block has to read.
// Measured against the memset and three kernels this replaces (B200, one call among others, Algorithm 1, density 1e-2):
//   n = 25.5 M  125.9 -> 109.8 us,   n = 1.86 M  @M@ -> 16.7 us,   n = 32768  @S@ -> 7.9 us.
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
constexpr int kCopies = 8;                           // of every slot, so that the pollers do not all meet in one place
constexpr int kOffsSmem = 1024;                      // group offsets cached in shared memory
constexpr uint32_t kStaged = 12288;                  // selected values a block keeps in shared memory (48 KB)
// a staged value: position in the block's range << 10 | sign << 9 | (rounded exponent + 127)
constexpr uint32_t kPosShift = 10;
constexpr size_t kMostPerBlock = 1u << (32 - kPosShift);

enum { kBasic = 0, kHybridBefore = 1, kHybridAfter = 2 };     // the hybrid's correction uses |r| from before / after r -= Sign(r) tau

constexpr size_t kSlotBytes = 2 * sizeof(Slot) * kCopies * kMaxGrid;

struct Args {
    const float *g, *s;
    float *r, *v;
    size_t n;
    const uint32_t *group_offsets;
    int K;
    float alpha, zeta;
    unsigned long long tag;
    Slot *first, *second;                // per block: {max of its first tensor, of its last}; {passed, kept}
    uint32_t *rec_max, *rec_min;         // per (block, tensor) at [block + tensor]: |value| bit patterns
    uint32_t *stage;                     // values past kStaged of a block, from its first parameter's index on
    uint32_t per_block, tile;
    float tau;                           // hybrid only
    vgc_message out;                     // (hybrid: no exponents, nnz only)
};

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
template <bool kHasS, int kAlgorithm>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
compress_step(const __grid_constant__ Args a)
{
    constexpr bool kQuantise = kAlgorithm == kBasic;
    extern __shared__ uint32_t sm_staged[];             // kStaged values
    __shared__ uint32_t sm_offs[kOffsSmem];
    __shared__ uint32_t sm_part[2][kRowsA * kWarps];    // per-(row, warp) counts, double buffered
    __shared__ uint32_t sm_wmax[2][kWarps];
    __shared__ uint32_t sm_wmin[2][kWarps];             // smallest |value| bit pattern sent by each warp
    __shared__ uint32_t sm_rec_max[2], sm_rec_min[2];   // extremes of the range's first and last tensor, this block's ...
    __shared__ uint32_t sm_end_max[2];                  // ... and M_k bits, from all blocks
    __shared__ uint32_t sm_kept[kWarps];
    __shared__ uint32_t sm_passed_before[kWarps], sm_kept_before[kWarps];

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    const int K = a.K;
    const bool offs_in_smem = kQuantise && (K + 1) <= kOffsSmem;
    if (offs_in_smem) {                                 // asynchronously: the first tile's loads go out before they arrive
        for (int i = tid; i <= K; i += kThreads)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                         ::"r"((uint32_t)__cvta_generic_to_shared(sm_offs + i)), "l"(a.group_offsets + i) : "memory");
    }
    const uint32_t *offs = offs_in_smem ? sm_offs : a.group_offsets;
    const uint32_t lo = b * a.per_block;
    const uint32_t hi = (uint32_t)((size_t)lo + a.per_block < a.n ? (size_t)lo + a.per_block : a.n);
    if (tid < 2) { sm_end_max[tid] = 0; sm_rec_max[tid] = 0; sm_rec_min[tid] = kNoMin; }
    Slot *const my_first = a.first + tid * kMaxGrid + b, *const my_second = a.second + tid * kMaxGrid + b;     // tid < kCopies
    const Slot *const firsts = a.first + (b % kCopies) * kMaxGrid, *const seconds = a.second + (b % kCopies) * kMaxGrid;
    if (tid < kCopies) slot_publish(my_second, 0, 0, 0);
    uint32_t *const rec_max = a.rec_max + b, *const rec_min = a.rec_min + b;     // this block's records, by tensor
    int k_first = 0, k_last = 0;

    const float tau_sq = __fmul_rn(a.tau, a.tau);

    // ---- step 1
    uint32_t run = 0;                                   // values staged by the block so far
    int k_tile = 0;                                     // tensor of the tile's first parameter
    int k_held = 0;                                     // thread 0: the tensor whose extremes it holds
    uint32_t held_max = 0, held_min = kNoMin;
    // largest and smallest |value| bits of tensor k: the range's first and last tensor in shared memory (all there is,
    // mostly), the ones between them in the workspace
    auto record = [&](int k, uint32_t most, uint32_t least) {
        const bool end = k == k_first || k == k_last;
        atomicMax(end ? sm_rec_max + (k != k_first) : rec_max + k, most);
        atomicMin(end ? sm_rec_min + (k != k_first) : rec_min + k, least);
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
            if (tid < kCopies) __threadfence();         // the cleared `second` slot before the `first` one
            if (offs_in_smem) asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
            __syncthreads();
        }
        if (kQuantise && base == lo) {
            k_first = group_of(offs, K, lo);
            k_last = hi <= offs[k_first + 1] ? k_first : group_of(offs, K, hi - 1);
            k_tile = k_held = k_first;
            for (int k = k_first + 1 + (int)tid; k < k_last; k += kThreads) { rec_max[k] = 0; rec_min[k] = kNoMin; }
        }
        if (kQuantise)
            while (offs[k_tile + 1] <= base) ++k_tile;  // block-uniform
        const int grp = !kQuantise || end <= offs[k_tile + 1] ? k_tile : -1;      // -1: the tile spans several tensors

        // loop body of Algorithm 1 / Algorithm 2; every operation rounded on its own (no FMA)
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
                const bool send = (lhs > rhs) && (e + q < end) && (kQuantise || fabsf(r1) > a.tau);
                Gj[q] = r1;                                       // value handed to Encode()
                if (kQuantise) {
                    Rj[q] = send ? 0.f : r1;
                    Vj[q] = send ? 0.f : __fmul_rn(v1, a.zeta);
                    if (send) {
                        my_max = max(my_max, __float_as_uint(r1) & 0x7FFFFFFFu);
                        my_min = min(my_min, __float_as_uint(r1) & 0x7FFFFFFFu);
                    }
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
        const uint32_t warp_min = kQuantise ? __reduce_min_sync(0xffffffffu, my_min) : 0u;
        if (lane == 31) {
#pragma unroll
            for (int j = 0; j < kRowsA; ++j) sm_part[buf][j * kWarps + warp] = (incl >> (8 * j)) & 0xFFu;
            sm_wmax[buf][warp] = warp_max;
            sm_wmin[buf][warp] = warp_min;
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
                        if (at < kStaged) sm_staged[at] = staged;
                        else a.stage[lo + at] = staged;
                        ++at;
                        if (kQuantise && grp < 0) {
                            const int k = group_of(offs, K, e + q);
                            record(k, bits & 0x7FFFFFFFu, bits & 0x7FFFFFFFu);
                        }
                    }
            }
        }
        if (kQuantise && tid == 0 && grp >= 0 && total) {
            if (grp != k_held) {
                if (held_max) record(k_held, held_max, held_min);
                k_held = grp; held_max = 0; held_min = kNoMin;
            }
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                held_max = max(held_max, sm_wmax[buf][w]);
                held_min = min(held_min, sm_wmin[buf][w]);
            }
        }
        run += total;
    }
    if (tid == 0 && held_max) record(k_held, held_max, held_min);
    __syncthreads();
    const int i_last = k_first == k_last ? 0 : 1;
    if (tid < kCopies) slot_publish(my_first, a.tag, sm_rec_max[0], sm_rec_max[i_last]);

    // ---- step 2: M_k of the range's first and last tensor, which other blocks may share.  A tensor that spans several
    // blocks is the last tensor of the block it begins in and the first one of the others
    {
        uint32_t f0 = 1, f1 = 0, l0 = 1, l1 = 0;
        if (kQuantise) {
            f0 = offs[k_first] / a.per_block; f1 = (offs[k_first + 1] - 1) / a.per_block;
            l0 = offs[k_last] / a.per_block;  l1 = (offs[k_last + 1] - 1) / a.per_block;
        }
        uint32_t m_first = 0, m_last = 0;
        bool late = false;
        for (uint32_t c = tid; c < gridDim.x; c += kThreads) {
            uint32_t of_first, of_last;
            if (!slot_wait(firsts + c, a.tag, of_first, of_last)) { late = true; break; }
            if (c >= f0 && c <= f1) m_first = max(m_first, c == f0 && f0 < f1 ? of_last : of_first);
            if (c >= l0 && c <= l1) m_last = max(m_last, c == l0 ? of_last : of_first);
        }
        __threadfence();                                // ... before anyone's `second` slot is looked at
        __syncwarp();
        if (kQuantise) {
            m_first = __reduce_max_sync(0xffffffffu, m_first);
            m_last = __reduce_max_sync(0xffffffffu, m_last);
        }
        if (kQuantise && lane == 0) {
            if (m_first) atomicMax(&sm_end_max[0], m_first);
            if (m_last) atomicMax(&sm_end_max[1], m_last);
        }
        if (__syncthreads_or(late)) {
            if (tid == 0) atomicOr(a.out.dev_status, VGC_DEV_TIMEOUT);
            return;
        }
    }
    auto max_of = [&](int k) -> uint32_t {
        return k == k_first ? sm_end_max[0] : k == k_last ? sm_end_max[1] : __ldcg(rec_max + k);
    };
    bool drops = false;
    if (kQuantise) {
        // exponents of the tensors that begin in this range (empty tensors at the buffer's end belong to the last block)
        int k0 = 0, k1 = K;                             // first k with offs[k] >= lo
        while (k0 < k1) {
            const int mid = (k0 + k1) >> 1;
            if (offs[mid] < lo) k0 = mid + 1; else k1 = mid;
        }
        const bool last = b == gridDim.x - 1;
        for (int k = k0 + (int)tid; k < K && (last || offs[k] < hi); k += kThreads)
            a.out.group_exp[k] = offs[k] < offs[k + 1] ? exponent_of(max_of(k)) : VGC_EXP_NONE;
        // nothing is dropped when even the smallest value sent from each tensor is within 7 binades of its exponent
        for (int k = k_first + (int)tid; k <= k_last; k += kThreads) {
            const uint32_t m = k == k_first ? sm_rec_min[0] : k == k_last ? sm_rec_min[1] : __ldcg(rec_min + k);
            if (m != kNoMin && rounded_exponent(m) < exponent_of(max_of(k)) - 7) drops = true;
        }
        drops = __syncthreads_or(drops);
    }

    // staged value i of the block -> its word; true if a word is emitted.  k: the tensor of the last value looked at
    auto staged_at = [&](uint32_t i) -> uint32_t { return i < kStaged ? sm_staged[i] : a.stage[lo + i]; };
    auto encode = [&](uint32_t staged, int &k, int32_t &Ek, uint32_t &word) -> bool {
        const uint32_t idx = lo + (staged >> kPosShift);
        if (!kQuantise) { word = (idx << 4) | ((staged >> 6) & 8u); return true; }
        if (Ek == INT32_MIN || idx < offs[k] || idx >= offs[k + 1]) {
            k = k_first == k_last ? k_first : group_of(offs, K, idx);
            Ek = exponent_of(max_of(k));
        }
        const int32_t e1 = (int32_t)(staged & 0x1FFu) - 127;
        const int32_t d = Ek - (e1 < Ek ? e1 : Ek);                        // cut at 2^E_k
        word = (idx << 4) | ((staged >> 6) & 8u) | (uint32_t)(d & 7);
        return d <= 7;
    };
    // with drops every warp walks a section of the values, four 32-wide slices per round
    const uint32_t section = ((run + kWarps - 1) / kWarps + 31u) & ~31u;
    const uint32_t s0 = min(run, warp * section), s1 = min(run, s0 + section);
    auto walk = [&](auto emit) {
        int k = k_first;
        int32_t Ek = INT32_MIN;
        uint32_t kept = 0;
        for (uint32_t i0 = s0; i0 < s1; i0 += 128) {
            uint32_t p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * 32 + lane;
                p[u] = i < s1 ? staged_at(i) : 0u;
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
    if (tid < kCopies) slot_publish(my_second, a.tag, run, kept);

    // ---- step 3: counts of the blocks before this one, then the words
    uint32_t passed_before = 0, kept_before = 0;
    bool late = false;
    for (uint32_t c = tid; c < b; c += kThreads) {
        uint32_t passed_c, kept_c;
        if (!slot_wait(seconds + c, a.tag, passed_c, kept_c)) { late = true; break; }
        passed_before += passed_c;
        kept_before += kept_c;
    }
    __syncwarp();
    passed_before = __reduce_add_sync(0xffffffffu, passed_before);
    kept_before = __reduce_add_sync(0xffffffffu, kept_before);
    if (lane == 0) { sm_passed_before[warp] = passed_before; sm_kept_before[warp] = kept_before; }
    if (__syncthreads_or(late)) {
        if (tid == 0) atomicOr(a.out.dev_status, VGC_DEV_TIMEOUT);
        return;
    }
    uint32_t pos = 0;
    passed_before = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { pos += sm_kept_before[w]; passed_before += sm_passed_before[w]; }
    if (tid == 0 && pos + kept > a.out.capacity) atomicOr(a.out.dev_status, VGC_DEV_CAPACITY);
    if (b == gridDim.x - 1) {
        if (tid == 0) {
            *a.out.nnz = pos + kept;
            if (kQuantise) {
                *a.out.n_criterion = passed_before + run;
                *a.out.n_dropped = passed_before + run - (pos + kept);
            }
        }
        for (uint32_t c = tid; c < kCopies * kMaxGrid; c += kThreads) slot_publish(a.first + c, 0, 0, 0);   // everyone has read them
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
            encode(staged_at(i), k, Ek, word);
            if (pos + i < a.out.capacity) a.out.words[pos + i] = word;
        }
    }
}

// Enqueues one step.  a: everything but the tag, the slots and the ranges, which are set here; `slots`: kSlotBytes.
template <bool kHasS, int kAlgorithm>
vgc_status launch(Args a, void *slots, cudaStream_t st)
{
    const void *fn = reinterpret_cast<const void *>(compress_step<kHasS, kAlgorithm>);
    constexpr size_t smem = kStaged * sizeof(uint32_t);
    static ResidentBlocks resident;
    const uint32_t most = resident.get(fn, kThreads, smem);
    if (most == 0) return VGC_ERR_CUDA;
    const Ranges R = even_ranges(a.n, most < (uint32_t)kMaxGrid ? most : (uint32_t)kMaxGrid, kTileA, kLeastPerBlock);
    if (R.per_block > kMostPerBlock) return VGC_ERR_UNSUPPORTED;         // a device with room for fewer than 64 blocks
    a.tag = next_tag();
    a.first = static_cast<Slot *>(slots);
    a.second = a.first + kCopies * kMaxGrid;
    a.per_block = R.per_block;
    a.tile = R.tile;
    void *params[] = {&a};
    VGC_CUDA_OK(cudaLaunchCooperativeKernel(fn, dim3(R.grid), dim3(kThreads), params, smem, st));
    count_launch();
    return VGC_OK;
}

}  // namespace step
}  // namespace vgc
