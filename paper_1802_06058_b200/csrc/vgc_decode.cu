// vgc_decode_accumulate / vgc_decode_sum: the decode-and-sum half of CommunicateAndUpdate (Sec. 4.3).
//
// Every 32-bit word (index << 4 | sign << 3 | d) of W packed messages is expanded to
// (-1)^sign * 2^(E_k - d), E_k the per-tensor exponent that travels with the message (Sec. 4.2),
// scaled, and added into the dense update buffer.  One launch covers up to kMaxViews messages (their
// pointers travel in the kernel parameters, so nothing is allocated).
//
// Messages are sorted by index, so the words that fall into a contiguous range of u are a contiguous run of every
// message.  Three ways, by how many words the messages hold together:
//   flat      few words, added to u: every warp takes pieces of the messages and adds them to u with fp32 atomics -- u is
//             touched only where a word points (decode_flat);
//   scatter   few words, u written: a block owns a range of u, writes zeros piece by piece and adds the piece's words while
//             it is still in L2 (scatter_range);
//   dense     a block owns a range of u and walks it in tiles held in shared memory; u is read and written once, coalesced:
//             exact_range where every word of a tensor is a multiple of one power of two, ordered_range where no tensor's
//             are, many_range where some are and some are not, or where the tensors are many.
// kOverwrite: the range starts from zero instead of the old contents of u (u = scale * sum of the messages).
// kHybrid: messages of the hybrid algorithm (Algorithm 2) -- every word stands for +-tau, no exponents.
#include <type_traits>

#include "vgc_common.cuh"

namespace vgc {

constexpr int kMaxViews = 64;
constexpr int kDecOffsSmem = 1024;

struct DecodeViews {
    const uint32_t *words[kMaxViews];
    const uint32_t *nnz[kMaxViews];
    const int32_t *group_exp[kMaxViews];
    uint32_t max_words[kMaxViews];
};

// Below one word per this many elements (all messages together) a call is not dense.  Added: an atomic costs two DRAM
// accesses, a dense pass reads and writes all of u (n = 138 M, one word per 16: 172 us flat, 330 us dense; per 6: 250 us
// dense).  Written: small buffers take scatter up to one word per eight, larger ones up to one per 16.  Measured just below /
// above the line (4 messages; 32 messages), us: around one per 8, n = 1.86 M 5.6 / 7.0 and 8.1 / 12.9, n = 4 M 8.3 / 8.3 and
// 10.3 / 13.6; around one per 16, n = 12 M 16.5 / 13.6 and 16.0 / 21.9, n = 25.5 M 43.4 / 23.7 and 34.0 / 37.7, n = 138 M 238 / 120
// and 219 / 183.  (Between 4 and 12 M elements many messages would gain from scatter beyond one per 16: 8 M, 32 messages,
// 12.4 / 20.2.)
constexpr size_t kSparseAdd = 8;
__host__ __device__ constexpr size_t sparse_write(size_t n) { return n <= ((size_t)4 << 20) ? 8 : 16; }

// three blocks of eight warps per SM: while one block waits at a barrier or for its first words, the others add
constexpr int kTileThreads = 256;
constexpr int kBlocksPerSm = 3;
constexpr int kTileWarps = kTileThreads / 32;
constexpr int kTileMax = 15360;                  // elements per tile: three tiles and the tables fit in shared memory
constexpr int kTensors = kTileWarps;             // weight tensors of a range that exact_range takes
constexpr int kTilePre = 8;                      // ordered form: words per thread in one batch

__device__ __forceinline__ void cp_async_16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ float value_at(uint32_t word, int32_t tensor_exp, float scale)
{
    const int32_t e = tensor_exp - (int32_t)(word & 7u);
    return __fmul_rn(scale, __uint_as_float(((uint32_t)(e + 127) << 23) | ((word & 8u) << 28)));
}
template <bool kHybrid>
__device__ __forceinline__ float value_of(uint32_t word, const int32_t *gexp, const uint32_t *offs, int K, float scale, float tau,
                                          int &k)
{
    if (kHybrid) return __fmul_rn(scale, (word & 8u) ? -tau : tau);
    const uint32_t idx = word >> 4;
    if (idx < offs[k] || idx >= offs[k + 1]) k = group_of(offs, K, idx);
    return value_at(word, gexp[k], scale);
}

// ---- flat -----------------------------------------------------------------------------------------------------------
// Every warp takes pieces of up to 32 words and adds their values to u with fp32 atomics (reductions: nothing comes
// back), the next piece's words already on their way.  Messages of about one length (within a factor of two) are cut into
// the same number of pieces, and the pieces go round by place first and message second, so that what is in flight at a time
// lies in one stretch of u: DRAM pages are opened once for the words of all of them.  Shorter messages make groups of their
// own, so that a piece is at least about half full whatever the lengths (one group for all took 4.5 ms for 64
// messages into 138 M elements, one of 6.9 M words and the others empty; now 127 us).
// Warps: two and a half blocks' per SM; one block's where three things hold: a large buffer (kFlatLarge), less than one word per kFlatThin
// elements, and words enough that what they touch does not stay in L2 (kFlatMany).  us, one block per SM / two: 16 M elements, 0.35 M
// words 11.7 / 7.3; 68 M, 1.5 M 51.9 / 50.0; 100 M, 1.9 M 69.0 / 72.2; 138 M, 0.22 M 6.4 / 4.6; 138 M, 0.9 M 40.7 / 43.1.  (The line between 68 M
// and 138 M elements is drawn at 100.7 M: just below it one block would be 4 % faster.)  DRAM is what bounds it, with accesses of 32 to
// 64 bytes in random order -- 138 M elements, 2.7 M words: 76 bytes read and up to 34 written per 64 touched, 92 us for what a copy moves
// in 40 --, and more in flight only widens the stretch.  138 M elements, us, with 1 / 2 / 2.5 / 3 / 4 blocks per SM: 64 messages, 2.7 M words
// 95 / 103 / 103 / 103 / 102, 8.9 M words 230 / 173 / 172 / 223 / 271; 4 messages, 11 M words 272 / 189 / 175 / 170 / 200; 32 M elements, 7 messages,
// 2 M words 55 / 41 / 39 / 40 / 40.
constexpr int kFlatThreads = 256, kPiece = 32, kFlatFewest = kSmCount, kFlatMost = kSmCount * 5 / 2;
constexpr uint32_t kFlatThin = 40;
constexpr uint32_t kFlatMany = 1u << 19;             // words
constexpr size_t kFlatLarge = (size_t)3 << 25;       // elements
__device__ __forceinline__ uint32_t flat_blocks(uint32_t words, size_t n)
{
    return n >= kFlatLarge && words >= kFlatMany && (size_t)words * kFlatThin < n ? kFlatFewest : kFlatMost;
}

struct FlatGroup {
    uint32_t first, members, pieces, end;                        // place in order[]; messages; pieces of each; end of its units
};
struct FlatPlan {
    FlatGroup group[32];                                         // (a message has less than 2^29 words)
    uint32_t units, words;                                       // all pieces, all words
    uint8_t order[kMaxViews];                                    // messages, longest group first
};
struct FlatShared {
    const uint32_t *words[kMaxViews];
    const int32_t *gexp[kMaxViews];
    uint32_t count[kMaxViews];
    FlatPlan plan;
};

// One warp; counts in shared memory, W <= 64.
__device__ __forceinline__ void plan_flat(FlatPlan &plan, const uint32_t *count, int W)
{
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
    const uint32_t c0 = lane < (uint32_t)W ? count[lane] : 0u, c1 = lane + 32u < (uint32_t)W ? count[lane + 32] : 0u;
    const uint32_t longest = __reduce_max_sync(0xffffffffu, max(c0, c1));
    // group of a message: the largest s with c <= longest >> s
    auto level_of = [&](uint32_t c) -> uint32_t {
        if (c == 0) return 32u;
        const uint32_t s = (uint32_t)(__clz(c) - __clz(longest));
        return (longest >> s) < c ? s - 1u : s;
    };
    uint32_t s0 = level_of(c0), s1 = level_of(c1), first = 0, units = 0;
    for (int g = 0;; ++g) {
        const uint32_t s = __reduce_min_sync(0xffffffffu, min(s0, s1));
        if (s == 32u) break;
        const uint32_t b0 = __ballot_sync(0xffffffffu, s0 == s), b1 = __ballot_sync(0xffffffffu, s1 == s);
        const uint32_t members = __popc(b0) + __popc(b1), pieces = ((longest >> s) + kPiece - 1) / kPiece;
        if (s0 == s) { plan.order[first + __popc(b0 & below)] = (uint8_t)lane; s0 = 32u; }
        if (s1 == s) { plan.order[first + __popc(b0) + __popc(b1 & below)] = (uint8_t)(lane + 32u); s1 = 32u; }
        units += pieces * members;
        if (lane == 0) plan.group[g] = FlatGroup{first, members, pieces, units};
        first += members;
    }
    const uint32_t words = __reduce_add_sync(0xffffffffu, c0 + c1);       // (fewer than one per eight elements)
    if (lane == 0) { plan.units = units; plan.words = words; }
}

template <bool kHybrid, class Shared>
__device__ __forceinline__ void add_flat(const Shared &sm, const FlatPlan &plan, const uint32_t *offs, int K, float scale, float tau,
                                         float *u, size_t n, uint32_t *dev_status, uint32_t warp, uint32_t warps)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t units = plan.units;
    FlatGroup at = plan.group[0];                                // the group of the unit asked for last
    uint32_t begin = 0;
    int g = 0;
    bool bad = false;
    // this lane's word of a piece; `in`: the piece reaches this lane and the word's index lies inside u (in a buffer of 2^28
    // elements no word could serve as filler: every index is an element)
    auto fetch = [&](uint32_t unit, const int32_t *&ge, bool &in) -> uint32_t {
        while (unit >= at.end) { begin = at.end; at = plan.group[++g]; }
        const uint32_t piece = (unit - begin) / at.members, w = plan.order[at.first + (unit - begin) - piece * at.members];
        const uint32_t c = sm.count[w], len = (c + at.pieces - 1) / at.pieces;    // at most kPiece
        const uint32_t p = piece * len + lane, end = min((piece + 1) * len, c);
        ge = kHybrid ? nullptr : sm.gexp[w];
        const uint32_t word = p < end ? sm.words[w][p] : 0u;
        in = p < end && (word >> 4) < n;
        if (p < end && !in) bad = true;
        return word;
    };
    const int32_t *ge_next = nullptr;
    bool in_next = false;
    uint32_t next = warp < units ? fetch(warp, ge_next, in_next) : 0u;
    int k = 0;
    for (uint32_t unit = warp; unit < units; unit += warps) {
        const int32_t *ge = ge_next;
        const bool in = in_next;
        const uint32_t word = next;
        if (unit + warps < units) next = fetch(unit + warps, ge_next, in_next);
        if (in) atomicAdd(u + (word >> 4), value_of<kHybrid>(word, ge, offs, K, scale, tau, k));
    }
    if (bad) atomicOr(dev_status, VGC_DEV_RANGE);
}

template <bool kHybrid>
__global__ void __launch_bounds__(kFlatThreads, 3)
decode_flat(const __grid_constant__ DecodeViews views, int W, const uint32_t *group_offsets, int K, float scale,
            float tau, float *u, size_t n, uint32_t *dev_status)
{
    __shared__ uint32_t sm_offs[kDecOffsSmem];
    __shared__ FlatShared sm;
    const uint32_t tid = threadIdx.x;
    const bool in_smem = !kHybrid && (K + 1) <= kDecOffsSmem;
    grid_wait();
    if (in_smem)
        for (int i = tid; i <= K; i += kFlatThreads) sm_offs[i] = group_offsets[i];
    if (tid < (uint32_t)W) {
        sm.words[tid] = views.words[tid];
        sm.gexp[tid] = views.group_exp[tid];
        const uint32_t said = *views.nnz[tid], have = views.max_words[tid];
        sm.count[tid] = said < have ? said : have;
        if (said > have && blockIdx.x == 0) atomicOr(dev_status, VGC_DEV_CAPACITY);
    }
    __syncthreads();
    if (tid < 32) plan_flat(sm.plan, sm.count, W);
    __syncthreads();
    const uint32_t blocks = min(gridDim.x, flat_blocks(sm.plan.words, n));
    if (blockIdx.x < blocks)
        add_flat<kHybrid>(sm, sm.plan, in_smem ? sm_offs : group_offsets, K, scale, tau, u, n, dev_status,
                          blockIdx.x * (kFlatThreads / 32) + (tid >> 5), blocks * (kFlatThreads / 32));
}

// ---- a block's range --------------------------------------------------------------------------------------------------
struct TileShared {
    uint32_t offs[kDecOffsSmem];
    uint32_t cur[kMaxViews], end[kMaxViews], taken[kMaxViews], count[kMaxViews];
    // the messages' pointers, copied out of the kernel parameters once: parameters cannot be indexed with a
    // run-time value (the compiler turns such an access into a chain of selects over all kMaxViews entries)
    const uint32_t *words[kMaxViews];
    const int32_t *gexp[kMaxViews];
    int32_t base[kTensors];                                      // exact form: 2^base is the unit of the range's tensors
    float lut[2][kMaxViews * 16];                                // values of the words of two tensors, 16 per message
    uint32_t unfit;                                              // what the range's tensors are like: kOrdered, ...
};
enum : uint32_t { kOrdered = 1, kCrowded = 2, kSomeUnfit = 4, kSomeFit = 8 };

// Where every message's run enters the range: sm.cur[w] becomes the first position of message w whose index is >= bound
// (its count if none).  Warp j looks after the messages j, j + 8, ...; lane i holds the state of the i-th of them.
// Random accesses are what a search costs -- all blocks search at the same time, every round is a memory latency under
// that load -- so it interpolates: one probe at the place that uniform indices would give (after it the place is known to
// some dozens of words), then kWindow neighbouring words around the next guess.  Where the indices are not uniform and the
// window misses, 32 evenly spaced probes and further windows take turns.  (Five rounds of evenly spaced probes took 10 us
// of a 43 us call.)  `meanwhile` runs while the first probes are on their way.
template <int kWords, int kTogether, class Meanwhile>       // words per lane of a window; messages whose windows go out together
__device__ __forceinline__ void find_runs(TileShared &sm, int W, uint32_t bound, uint32_t most_index, Meanwhile meanwhile)
{
    constexpr uint32_t kWindow = 32 * kWords;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t mine = warp + kTileWarps * lane;              // this lane's message
    uint32_t lo = 0, hi = mine < (uint32_t)W ? sm.count[mine] : 0u;   // positions < lo are below the bound, >= hi are not
    uint32_t key_lo = 0, key_hi = most_index;                    // indices at those ends
    const uint32_t *words = mine < (uint32_t)W ? sm.words[mine] : nullptr;
    if (bound == 0) hi = 0;
    auto guess = [&]() -> uint32_t {
        const uint32_t len = hi - lo;
        const float part = key_hi > key_lo ? __fdividef((float)(bound - key_lo), (float)(key_hi - key_lo)) : 0.5f;
        return lo + min((uint32_t)(part * (float)len), len - 1u);
    };
    const bool probe = hi > kWindow;
    uint32_t g = 0, key = 0;
    if (probe) { g = guess(); key = words[g] >> 4; }
    meanwhile();
    if (probe) {
        if (key < bound) { lo = g + 1; key_lo = key; }
        else { hi = g; key_hi = max(key, key_lo); }
    }
    for (uint32_t round = 0;; ++round) {
        const uint32_t open = __ballot_sync(0xffffffffu, lo < hi);
        if (open == 0) break;
        const uint32_t place = lo < hi ? guess() : 0u;
        for (uint32_t j0 = 0; j0 < 32 && (open >> j0); j0 += kTogether) {
            uint32_t base[kTogether], step[kTogether], key_at[kTogether][kWords];
#pragma unroll
            for (int t = 0; t < kTogether; ++t) {
                const uint32_t j = j0 + t;
                const uint32_t l = __shfl_sync(0xffffffffu, lo, j), h = __shfl_sync(0xffffffffu, hi, j);
                const uint32_t at = __shfl_sync(0xffffffffu, place, j), len = h - l;
                const uint32_t *from = reinterpret_cast<const uint32_t *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(words), j));
                const bool spread = (round & 1u) && len > kWindow;        // all of this is warp-uniform
                step[t] = spread ? len / kWindow + 1 : 1u;
                base[t] = (spread || at - l <= kWindow / 2 || len <= kWindow) ? l : min(at - kWindow / 2, h - kWindow);
#pragma unroll
                for (int i = 0; i < kWords; ++i) {
                    const uint32_t pos = base[t] + step[t] * (32 * i + lane);
                    key_at[t][i] = (open >> j & 1u) && pos < h ? from[pos] >> 4 : 0xFFFFFFFFu;
                }
            }
#pragma unroll
            for (int t = 0; t < kTogether; ++t) {
                const uint32_t j = j0 + t;
                uint32_t nb = 0, below = 0, above = 0xFFFFFFFFu;          // probes below the bound; the keys around it
#pragma unroll
                for (int i = 0; i < kWords; ++i) {
                    const uint32_t b = __popc(__ballot_sync(0xffffffffu, key_at[t][i] < bound));      // sorted: a prefix
                    nb += b;
                    const uint32_t last = __shfl_sync(0xffffffffu, key_at[t][i], (b + 31u) & 31u);
                    if (b > 0) below = last;
                    const uint32_t first = __shfl_sync(0xffffffffu, key_at[t][i], b & 31u);
                    if (b < 32 && above == 0xFFFFFFFFu) above = first;
                }
                if (lane == j && (open >> j & 1u)) {
                    const uint32_t new_lo = nb > 0 ? base[t] + step[t] * (nb - 1) + 1 : lo;
                    const uint32_t new_hi = nb < kWindow ? min(base[t] + step[t] * nb, hi) : hi;
                    if (nb > 0) key_lo = below;
                    if (new_hi < hi) key_hi = max(above, key_lo);
                    lo = new_lo;
                    hi = max(new_lo, new_hi);
                }
            }
        }
    }
    if (mine < (uint32_t)W) sm.cur[mine] = lo;
}

// ---- scatter: few words, u written --------------------------------------------------------------------------------------
// Zeros and additions piece by piece: the pieces of all blocks together (444 x 128 KB) stay in L2 between the two.
constexpr uint32_t kScatterPiece = 32768;

template <bool kHybrid>
__device__ __forceinline__ bool scatter_range(TileShared &sm, int W, const uint32_t *offs, int K, float scale, float tau,
                                              float *u, uint32_t lo, uint32_t hi)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool bad = false;
    auto load = [&](uint32_t w, uint32_t at) { return at + lane < sm.count[w] ? sm.words[w][at + lane] : 0xFFFFFFFFu; };
    for (uint32_t p0 = lo; p0 < hi; p0 += kScatterPiece) {
        const uint32_t p1 = min(hi, p0 + kScatterPiece);
        uint32_t next = warp < (uint32_t)W ? load(warp, sm.cur[warp]) : 0u;
        for (uint32_t i = p0 + 4 * tid; i < p1; i += 4 * kTileThreads) {
            if (i + 3 < p1) *reinterpret_cast<float4 *>(u + i) = make_float4(0.f, 0.f, 0.f, 0.f);
            else for (uint32_t c = i; c < p1; ++c) u[c] = 0.f;
        }
        __syncthreads();                                            // this piece's zeros before its additions
        for (uint32_t w = warp; w < (uint32_t)W; w += kTileWarps) {
            uint32_t word = next, at = sm.cur[w];
            if (w + kTileWarps < (uint32_t)W) next = load(w + kTileWarps, sm.cur[w + kTileWarps]);
            const int32_t *gexp = sm.gexp[w];
            int k = 0;
            for (;;) {
                const uint32_t idx = word >> 4;
                const bool in = at + lane < sm.count[w] && idx < p1;
                if (in) {
                    if (idx >= p0) atomicAdd(u + idx, value_of<kHybrid>(word, gexp, offs, K, scale, tau, k));
                    else bad = true;                                // behind the piece's start: the message is not sorted
                }
                const uint32_t out = __ballot_sync(0xffffffffu, !in);
                if (out) { at += __ffs(out) - 1; break; }           // sorted: the rest belongs to later pieces
                at += 32;
                word = load(w, at);
            }
            __syncwarp();
            if (lane == 0) sm.cur[w] = at;
        }
        __syncwarp();
    }
    return bad;
}

// ---- dense, ordered form --------------------------------------------------------------------------------------------------
// Tile by tile, the messages' runs are added one after the other by the whole block, 8 x 256 words at a time with the next
// batch's loads in flight (indices inside a message are distinct, so plain read-modify-writes, a block barrier between
// messages): an element receives its additions in message order, the fp32 sequence of a sequential sum.
// Returns whether a word was out of place.
// This and many_range are functions of their own, given shared-memory addresses: inlined, their registers make the other forms
// spill (messages that are not aligned, K = 1, W = 64, added to 25.5 M elements: 294 -> 324 us).
template <bool kHybrid, bool kOverwrite>
__device__ __noinline__ bool ordered_range(uint32_t sm_addr, uint32_t tile_addr, int W, const uint32_t *offs, int K, float scale,
                                           float tau, float *u, uint32_t lo, uint32_t hi, uint32_t tile_elems)
{
    TileShared &sm = *static_cast<TileShared *>(__cvta_shared_to_generic(sm_addr));
    float *const tile = static_cast<float *>(__cvta_shared_to_generic(tile_addr));
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *const cur = sm.cur, *const end = sm.end;
    bool bad = false;
    uint32_t t_len = 0;
    for (uint32_t t0 = lo; t0 < hi; t0 += t_len) {
        t_len = min(hi - t0, tile_elems);
        int tile_group = kHybrid ? 0 : -1;                          // weight tensor of the tile, -1 if it spans several
        int g0 = -1;                                                // its first tensor, where the exponents of all fit into exps
        int32_t *const exps = reinterpret_cast<int32_t *>(sm.lut);  // [tensor of the tile][message]
        if (!kHybrid) {
            const int g = group_of(offs, K, t0);
            const uint32_t rem = offs[g + 1] - t0;
            if (rem >= t_len) tile_group = g;
            else {
                const int all = (group_of(offs, K, t0 + t_len - 1) - g + 1) * W;
                if (all <= (int)(sizeof(sm.lut) / sizeof(int32_t))) {
                    g0 = g;
                    for (int i = tid; i < all; i += kTileThreads) exps[i] = sm.gexp[i % W][g + i / W];
                }
            }
        }
        const uint32_t t_hi = t0 + t_len;
        const uint32_t n_vec = t_len / 4;                           // t0 is a multiple of 4 elements
        if (!kOverwrite) {                                          // the tile's old content
            for (uint32_t q = tid; q < n_vec; q += kTileThreads) cp_async_16(tile + 4 * q, u + t0 + 4 * q);
            if (tid < t_len - 4 * n_vec) tile[4 * n_vec + tid] = u[t0 + 4 * n_vec + tid];
        }
        // where every message's run leaves the tile: at most t_len of its words can lie inside
        for (int w = warp; w < W; w += kTileWarps) {
            const uint32_t *words = sm.words[w] + cur[w];
            const uint32_t left = sm.count[w] - cur[w];
            uint32_t a = 0, b = left < t_len ? left : t_len;        // positions < a are below t_hi, >= b are not
            while (a < b) {                                         // 32 probes a, a + step, ... reach past b
                const uint32_t step = (b - a) / 32 + 1, pos = a + step * lane;
                const uint32_t nb = __popc(__ballot_sync(0xffffffffu, pos < b && (words[pos] >> 4) < t_hi));
                if (nb == 0) break;
                const uint32_t new_b = a + step * nb;
                a += step * (nb - 1) + 1;
                b = new_b < b ? new_b : b;
            }
            if (lane == 0) end[w] = cur[w] + a;
        }
        // the 16 values a word's low four bits (sign, d) can stand for, per message
        if (tile_group >= 0)
            for (int i = tid; i < W * 16; i += kTileThreads) {
                const uint32_t code = (uint32_t)i & 15u;
                const uint32_t ebits = kHybrid ? 0u : (uint32_t)(sm.gexp[i >> 4][tile_group] + 127) << 23;
                const float val = kHybrid ? ((code & 8u) ? -tau : tau)
                                          : __uint_as_float((ebits - ((code & 7u) << 23)) | ((code & 8u) << 28));
                sm.lut[0][i] = __fmul_rn(scale, val);
            }
        if (!kOverwrite) cp_async_wait_all();
        __syncthreads();

        constexpr uint32_t kBatchWords = kTilePre * kTileThreads;
        auto batches_of = [&](int w) -> uint32_t { return (end[w] - cur[w] + kBatchWords - 1) / kBatchWords; };
        auto load_batch = [&](int w, uint32_t b, uint32_t (&dst)[kTilePre]) {
            const uint32_t first = cur[w] + b * kBatchWords + tid, e = end[w];
            const uint32_t *p = sm.words[w] + first;
#pragma unroll
            for (int j = 0; j < kTilePre; ++j) dst[j] = first + j * kTileThreads < e ? p[j * kTileThreads] : 0u;
        };
        int w = 0;
        uint32_t b = 0;
        while (w < W && batches_of(w) == 0) ++w;
        uint32_t held[kTilePre], next[kTilePre];
        uint32_t nb = w < W ? batches_of(w) : 0;                     // batches of the current message
        if (w < W) load_batch(w, 0, held);
        int k = 0;
        while (w < W) {
            int w2 = w;
            uint32_t b2 = b + 1, nb2 = nb;
            if (b2 >= nb) {
                w2 = w + 1; b2 = 0;
                while (w2 < W && (nb2 = batches_of(w2)) == 0) ++w2;
            }
            if (w2 < W) load_batch(w2, b2, next);
            const uint32_t first = cur[w] + b * kBatchWords + tid, e = end[w];
            const float *lut = sm.lut[0] + 16 * w;
            const int32_t *gexp = sm.gexp[w];
#pragma unroll
            for (int j = 0; j < kTilePre; ++j) {
                const uint32_t word = held[j], at = (word >> 4) - t0;
                if (first + j * kTileThreads >= e) continue;
                // a word of a sorted message lies inside the tile; one that does not (the message is not sorted) is skipped
                if (at >= t_len) { bad = true; continue; }
                float v;
                if (tile_group >= 0) v = lut[word & 15u];
                else if (g0 >= 0) {
                    if ((word >> 4) < offs[k] || (word >> 4) >= offs[k + 1]) k = group_of(offs, K, word >> 4);
                    v = value_at(word, exps[(k - g0) * W + w], scale);
                } else v = value_of<kHybrid>(word, gexp, offs, K, scale, tau, k);
                tile[at] = __fadd_rn(tile[at], v);
            }
            if (w2 != w) __syncthreads();                            // the next message may hit the same elements
#pragma unroll
            for (int j = 0; j < kTilePre; ++j) held[j] = next[j];
            w = w2; b = b2; nb = nb2;
        }
        __syncthreads();
        if (tid < (uint32_t)W) cur[tid] = end[tid];
        for (uint32_t q = tid; q < n_vec; q += kTileThreads) {
            *reinterpret_cast<float4 *>(u + t0 + 4 * q) = reinterpret_cast<const float4 *>(tile)[q];
            if (kOverwrite) reinterpret_cast<float4 *>(tile)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (tid < t_len - 4 * n_vec) {
            u[t0 + 4 * n_vec + tid] = tile[4 * n_vec + tid];
            if (kOverwrite) tile[4 * n_vec + tid] = 0.f;
        }
        __syncthreads();                                             // cursors, and the tile before it is loaded again
    }
    return bad;
}

// ---- dense, the exact form's words --------------------------------------------------------------------------------------
// Warps stream the messages' words from their cursors.  Message m is shared by the warps m, m + W, ... (W < 8) in turns of
// 256 words -- or a warp takes the messages warp, warp + 8, ... -- and a warp stops at its first turn that reaches past the
// tile (or the message's end); the words it found inside are added to the message's count (sm.taken), which moves the cursor
// once all warps are done.
// A word minus t0 << 4 keeps its low four bits and turns its index into the offset inside the tile; one unsigned comparison
// then says "inside the tile" (a word behind the tile wraps around to a huge number, and so does the filler 0xFFFFFFFF,
// because the range ends before 2^28).  add(word, message, count) makes that comparison, adds the word and counts it.
template <class Add>
__device__ __forceinline__ void stream_tile(TileShared &sm, int W, uint32_t t0, uint32_t t_len, bool &bad, Add add)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t t0s = t0 << 4, t_len16 = t_len << 4;
    const int sharers = W < kTileWarps ? kTileWarps / W : 1;       // warps per message
    for (int m = (int)warp % W; m < W; m += kTileWarps) {
        if (W < kTileWarps && (int)warp >= sharers * W) break;     // warps left over when W does not divide the warps
        const uint32_t turn0 = W < kTileWarps ? warp / (uint32_t)W : 0u;
        const uint32_t *words = sm.words[m];
        const uint32_t c = sm.cur[m], cnt = sm.count[m];
        const uint32_t a = c & ~3u;                                // 16-byte loads: start at the boundary before the cursor
        uint32_t inside = 0, n_in = 0;                             // words up to the tile's end; words added
        // a turn is 256 consecutive words, two 16-byte loads per lane; the next turn's loads are issued before
        // this turn's words are looked at, so the latency of one turn hides under the work of the other
        constexpr int kVecs = 2, kAhead = 4;
        constexpr uint32_t kTurnWords = 128u * kVecs;
        uint4 nxt[kVecs];
        auto fetch = [&](uint32_t turn, uint4 (&dst)[kVecs]) {
            const uint32_t p0 = a + turn * kTurnWords + 4u * lane;
            if (a + (turn + 1u) * kTurnWords <= cnt) {             // warp-uniform: the whole turn lies inside the message
#pragma unroll
                for (int v = 0; v < kVecs; ++v) dst[v] = *reinterpret_cast<const uint4 *>(words + p0 + 128u * v);
            } else {
#pragma unroll
                for (int v = 0; v < kVecs; ++v) {
                    const uint32_t p = p0 + 128u * v;
                    dst[v].x = p < cnt ? words[p] : 0xFFFFFFFFu;
                    dst[v].y = p + 1u < cnt ? words[p + 1] : 0xFFFFFFFFu;
                    dst[v].z = p + 2u < cnt ? words[p + 2] : 0xFFFFFFFFu;
                    dst[v].w = p + 3u < cnt ? words[p + 3] : 0xFFFFFFFFu;
                }
            }
            // ... and the turns after it are asked into L2 (no registers held): a turn's loads then find their lines there
            const uint32_t ahead = a + (turn + (uint32_t)(kAhead * sharers)) * kTurnWords + 32u * lane;
            if (lane < kTurnWords / 32u && ahead < cnt) asm volatile("prefetch.global.L2 [%0];" ::"l"(words + ahead));
        };
        fetch(turn0, nxt);
        for (uint32_t turn = turn0;; turn += (uint32_t)sharers) {
            uint4 wd[kVecs];
#pragma unroll
            for (int v = 0; v < kVecs; ++v) wd[v] = nxt[v];
            fetch(turn + (uint32_t)sharers, nxt);
#pragma unroll
            for (int v = 0; v < kVecs; ++v) {
                add(wd[v].x, (uint32_t)m, n_in); add(wd[v].y, (uint32_t)m, n_in);
                add(wd[v].z, (uint32_t)m, n_in); add(wd[v].w, (uint32_t)m, n_in);
            }
            // sorted words: the turn lies inside the tile when its last word does (and the message goes on)
            const uint32_t turn_end = a + (turn + 1u) * kTurnWords;
            const bool last_in = wd[kVecs - 1].w - t0s < t_len16;
            if (turn_end <= cnt && (__ballot_sync(0xffffffffu, last_in) >> 31)) {
                inside += kTurnWords - (turn == 0u ? c - a : 0u);
                continue;
            }
            // the last turn of this warp: count the words from the cursor on that lie before the tile's end
            uint32_t mine = 0;
            const uint32_t p0 = a + turn * kTurnWords + 4u * lane, t_hi = t0 + t_len;
#pragma unroll
            for (int v = 0; v < kVecs; ++v) {
                const uint32_t p = p0 + 128u * v;
                const uint32_t x[4] = {wd[v].x, wd[v].y, wd[v].z, wd[v].w};
#pragma unroll
                for (uint32_t i = 0; i < 4; ++i) mine += (p + i >= c && p + i < cnt && (x[i] >> 4) < t_hi) ? 1u : 0u;
            }
            inside += __reduce_add_sync(0xffffffffu, mine);
            break;
        }
        // a word before the tile's end that was not added lies behind the tile: the message is not sorted
        if (__reduce_add_sync(0xffffffffu, n_in) != inside) bad = true;
        if (lane == 0 && inside) atomicAdd(&sm.taken[m], inside);
    }
}

constexpr int32_t kUnfit = INT32_MIN;

// Unit of a tensor whose exponents (of this lane's two messages: ex[0], ex[1]) lie close enough together; else kUnfit.
// With a scale that is a power of two 2^s_exp (pow2) the result is the sequential sum's, bit for bit.
__device__ __forceinline__ int32_t unit_of_tensor(const int32_t (&ex)[2], int W, bool pow2, int s_exp)
{
    const bool some0 = ex[0] != VGC_EXP_NONE, some1 = ex[1] != VGC_EXP_NONE;
    const int e_max = __reduce_max_sync(0xffffffffu, max(some0 ? ex[0] : INT32_MIN, some1 ? ex[1] : INT32_MIN));
    const int e_min = __reduce_min_sync(0xffffffffu, min(some0 ? ex[0] : INT32_MAX, some1 ? ex[1] : INT32_MAX));
    if (e_max < e_min) return 0;                                 // (nothing was sent from this tensor)
    const int b = e_min - 7;                                     // the smallest value a word can stand for
    // 2^base and every sum of multiples are normal numbers; with a power-of-two scale so are their products
    const bool fits = e_max - b + (32 - __clz((W - 1) | 1)) <= 22 && b >= -126 && b + 22 <= 127 &&
                      (!pow2 || (b + s_exp >= -126 && b + 22 + s_exp <= 127));
    return fits ? b : kUnfit;
}
// A sum of multiples (at most 2^22 either way, so 1.5 * 2^23 plus it is a float whose bits are 0x4B400000 plus it) times
// the unit (exact).
__device__ __forceinline__ float times_unit(int mult, float unit)
{
    return __fmul_rn(__fsub_rn(__int_as_float(0x4B400000 + mult), 12582912.f), unit);
}
__device__ __forceinline__ float power_of_two(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

// ---- dense, exact form ----------------------------------------------------------------------------------------------------
// When the exponents of all messages for a tensor lie close enough together, every word is an integer multiple of one power
// of two, 2^base, and every partial sum of up to W of them stays within 2^22 multiples: all of them are exact fp32 numbers,
// fp32 addition of them is associative, and the sequential sum of the words equals the exact sum (with a power-of-two scale
// that is the decoder's result bit for bit; otherwise the scale is applied to the exact sum, one rounding instead of one
// per message, and vgc_decode_accumulate adds the scaled sum to u in one addition).  A tile is then accumulated as int32
// multiples of 2^base with shared-memory integer atomics, in any order: no barrier between messages, no search for the
// runs' ends -- the warps stream every message's words from its cursor until the indices leave the tile -- and one
// conversion at the end.  Same bits, much less waiting.  exact_range is for ranges of few tensors, all of which fit: its tiles
// hold two at most, and a word's multiple is one look-up.
// Returns whether a word was out of place.
template <bool kHybrid, bool kOverwrite>
__device__ __forceinline__ bool exact_range(TileShared &sm, float *tile, int W, const uint32_t *offs, int g_first, float scale,
                                            float tau, float *u, uint32_t lo, uint32_t hi, uint32_t tile_elems)
{
    const uint32_t tid = threadIdx.x;
    const uint32_t tile_addr = (uint32_t)__cvta_generic_to_shared(tile);
    bool bad = false;
    int g = g_first, made = -1;        // tensor of the tile's first element; the last tensor whose table was made
    int slot = 1;                      // the table of the tile's first tensor
    uint32_t t_len = 0;
    for (uint32_t t0 = lo; t0 < hi; t0 += t_len) {
        // A tile inside one tensor or across the border of two; one that would reach a third ends before it, at a multiple
        // of four elements
        t_len = min(hi - t0, tile_elems);
        uint32_t split = t_len;                                     // elements of the first tensor
        if (!kHybrid) {
            while (offs[g + 1] <= t0) ++g;                          // block-uniform, as all of this
            if (offs[g + 1] - t0 < t_len) {
                split = offs[g + 1] - t0;
                int g1 = g + 1;
                while (offs[g1 + 1] == offs[g1]) ++g1;
                if (offs[g1 + 1] - t0 < t_len) t_len = (offs[g1 + 1] - t0) & ~3u;
                split = min(split, t_len);
            }
        }
        // the 16 values a word's low four bits (sign, d) can stand for, per message, as multiples of the tensor's unit; the
        // tables of two neighbouring tensors take turns
        auto table = [&](int which, int k) {
            const int base = kHybrid ? 0 : sm.base[k - g_first];
            for (int i = tid; i < W * 16; i += kTileThreads) {
                const int e = kHybrid ? 0 : sm.gexp[i >> 4][k];
                const int mult = kHybrid ? 1 : e == VGC_EXP_NONE ? 0 : 1 << (e - (i & 7) - base);
                reinterpret_cast<int *>(sm.lut[which])[i] = (i & 8) ? -mult : mult;
            }
        };
        if (made < g) { slot ^= 1; table(slot, g); made = g; }      // (the tile before ended with its tensor)
        int next = g;
        if (split < t_len) {
            ++next;
            while (offs[next + 1] == offs[next]) ++next;
            table(slot ^ 1, next);
            made = next;
        }
        const uint32_t n_vec = t_len / 4;                           // t0 is a multiple of 4 elements
        if (!kOverwrite)                                            // u is read at the tile's end: ask it into L2 now
            for (uint32_t line = tid; line < (t_len + 31u) / 32u; line += kTileThreads)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(u + t0 + 32u * line));
        if (tid < (uint32_t)W) sm.taken[tid] = 0;
        __syncthreads();

        const uint32_t t0s = t0 << 4, t_len16 = t_len << 4, split16 = split << 4;
        auto stream = [&](auto two) {
            constexpr bool kTwo = decltype(two)::value;             // the tile has elements of two tensors
            const uint32_t lut_addr = (uint32_t)__cvta_generic_to_shared(sm.lut[slot]);
            const uint32_t lut_other = (uint32_t)__cvta_generic_to_shared(sm.lut[slot ^ 1]) - lut_addr;
            // one word: inside the tile -> look its multiple up and add it; all of it predicated, no branch
            stream_tile(sm, W, t0, t_len, bad, [&](uint32_t word, uint32_t m, uint32_t &n_in) {
                const uint32_t lut_m = lut_addr + 64u * m;
                if (kTwo)
                    asm volatile("{\n\t"
                                 ".reg .pred p, second;\n\t"
                                 ".reg .s32 iv;\n\t"
                                 ".reg .u32 o, at, l;\n\t"
                                 "sub.u32 o, %1, %2;\n\t"
                                 "setp.lt.u32 p, o, %3;\n\t"
                                 "setp.ge.u32 second, o, %6;\n\t"
                                 "and.b32 l, %1, 15;\n\t"
                                 "shl.b32 l, l, 2;\n\t"
                                 "add.u32 l, l, %4;\n\t"
                                 "@second add.u32 l, l, %7;\n\t"
                                 "shr.u32 at, o, 2;\n\t"
                                 "and.b32 at, at, 0xFFFFFFFC;\n\t"
                                 "add.u32 at, at, %5;\n\t"
                                 "@p ld.shared.s32 iv, [l];\n\t"
                                 "@p red.shared.add.s32 [at], iv;\n\t"
                                 "@p add.u32 %0, %0, 1;\n\t"
                                 "}"
                                 : "+r"(n_in)
                                 : "r"(word), "r"(t0s), "r"(t_len16), "r"(lut_m), "r"(tile_addr), "r"(split16), "r"(lut_other)
                                 : "memory");
                else
                    asm volatile("{\n\t"
                                 ".reg .pred p;\n\t"
                                 ".reg .s32 iv;\n\t"
                                 ".reg .u32 o, at, l;\n\t"
                                 "sub.u32 o, %1, %2;\n\t"
                                 "setp.lt.u32 p, o, %3;\n\t"
                                 "and.b32 l, %1, 15;\n\t"
                                 "shl.b32 l, l, 2;\n\t"
                                 "add.u32 l, l, %4;\n\t"
                                 "shr.u32 at, o, 2;\n\t"
                                 "and.b32 at, at, 0xFFFFFFFC;\n\t"
                                 "add.u32 at, at, %5;\n\t"
                                 "@p ld.shared.s32 iv, [l];\n\t"
                                 "@p red.shared.add.s32 [at], iv;\n\t"
                                 "@p add.u32 %0, %0, 1;\n\t"
                                 "}"
                                 : "+r"(n_in)
                                 : "r"(word), "r"(t0s), "r"(t_len16), "r"(lut_m), "r"(tile_addr)
                                 : "memory");
            });
        };
        if (split < t_len) stream(std::true_type());
        else stream(std::false_type());
        __syncthreads();
        if (tid < (uint32_t)W) sm.cur[tid] += sm.taken[tid];

        // ---- multiples of 2^base -> fp32 (a sum is at most 2^22 multiples either way, so 1.5 * 2^23 plus it is a float
        // whose bits are 0x4B400000 plus it), times 2^base (exact), times the scale: one rounding, none when the scale is a
        // power of two.  vgc_decode_accumulate adds the result to u; an element no word points at keeps its bits.
        auto unit_of = [&](int k) {
            return kHybrid ? __fmul_rn(scale, tau) : power_of_two(sm.base[k - g_first]);
        };
        const float unit_a = unit_of(g), unit_b = unit_of(next);
        auto value = [&](int mult, float unit) {
            const float m = times_unit(mult, unit);
            return kHybrid ? m : __fmul_rn(m, scale);           // hybrid: a word is worth scale * tau, rounded once
        };
        // vector q of the tile: the units of its elements (they differ inside the one vector that holds the border)
        auto values = [&](const int4 &mult, uint32_t q) {
            const uint32_t left = split - min(split, 4 * q);    // elements of the first tensor from here on
            return make_float4(value(mult.x, left > 0 ? unit_a : unit_b), value(mult.y, left > 1 ? unit_a : unit_b),
                               value(mult.z, left > 2 ? unit_a : unit_b), value(mult.w, left > 3 ? unit_a : unit_b));
        };
        float *const dst = u + t0;
        if (kOverwrite) {
            for (uint32_t q = tid; q < n_vec; q += kTileThreads) {
                const int4 mlt = reinterpret_cast<const int4 *>(tile)[q];
                reinterpret_cast<int4 *>(tile)[q] = make_int4(0, 0, 0, 0);
                *reinterpret_cast<float4 *>(dst + 4 * q) = values(mlt, q);
            }
        } else {
            constexpr int kHeld = 4;                            // vectors of u per thread in flight
            for (uint32_t q0 = tid; q0 < n_vec; q0 += kHeld * kTileThreads) {
                float4 o[kHeld];
#pragma unroll
                for (int j = 0; j < kHeld; ++j) {
                    const uint32_t q = q0 + j * kTileThreads;
                    if (q < n_vec) o[j] = *reinterpret_cast<const float4 *>(dst + 4 * q);
                }
#pragma unroll
                for (int j = 0; j < kHeld; ++j) {
                    const uint32_t q = q0 + j * kTileThreads;
                    if (q >= n_vec) break;
                    const int4 mlt = reinterpret_cast<const int4 *>(tile)[q];
                    if ((mlt.x | mlt.y | mlt.z | mlt.w) == 0) continue;
                    reinterpret_cast<int4 *>(tile)[q] = make_int4(0, 0, 0, 0);
                    const float4 add = values(mlt, q);
                    if (mlt.x) o[j].x = __fadd_rn(o[j].x, add.x);
                    if (mlt.y) o[j].y = __fadd_rn(o[j].y, add.y);
                    if (mlt.z) o[j].z = __fadd_rn(o[j].z, add.z);
                    if (mlt.w) o[j].w = __fadd_rn(o[j].w, add.w);
                    *reinterpret_cast<float4 *>(dst + 4 * q) = o[j];
                }
            }
        }
        if (tid < t_len - 4 * n_vec) {                          // the buffer's last elements
            const uint32_t i = 4 * n_vec + tid;
            const int mult = reinterpret_cast<const int *>(tile)[i];
            const float v = value(mult, i < split ? unit_a : unit_b);
            if (kOverwrite) dst[i] = v;
            else if (mult) dst[i] = __fadd_rn(dst[i], v);
            tile[i] = 0.f;
        }
        // every thread put zeros back where it read, and the next tile's barrier orders them before the next additions
        if (next != g) { g = next; slot ^= 1; }
    }
    return bad;
}

// ---- dense, many tensors ----------------------------------------------------------------------------------------------------
// Tiles of any number of tensors, each in its own form: words of a tensor whose exponents fit are added as multiples of its
// unit, in any order, in one pass over all messages; then, where a tensor of the tile does not fit, the words of such
// tensors are added message after message, a block barrier between messages.  Both share the tile: an element belongs to
// one tensor.  A word's tensor is searched among the tile's (kept from word to word: neighbours mostly share it), its
// multiple made from the exponent's distance to the tensor's unit.
// Measured (B200, ResNet-50 with its normalisation vectors: 161 tensors, 25.6 M elements, written): 8 messages of density
// 0.05 47 us, 64 of 0.01 99 us; with the range in the ordered form 103 and 472, with tiles in it 81 and 315.
// What a tile needs to know about its tensors; in the place of the exact form's tables.
constexpr int kMany = 511, kAbove = 4096;
struct ManyTensors {
    uint8_t above[kAbove];                       // [tensor][message]: exponent above the unit's; kNothing: nothing was sent
    uint32_t begin[kMany + 1];                   // first element, counted from the tile's; [tensors]: behind the last one
    int32_t base[kMany + 1];                     // 2^base is the unit; kUnfit: the tensor is added in message order
};
static_assert(sizeof(ManyTensors) <= sizeof(TileShared::lut), "in the place of the tables");
constexpr uint8_t kNothing = 255;

// Walks [lo, hi) from lo on.  Returns where it stopped -- hi, but where more tensors than a tile has room for begin within
// four elements (the ordered form does the rest) -- and whether a word was out of place (kBad).
constexpr uint32_t kBad = 1u << 31;
template <bool kOverwrite>
__device__ __noinline__ uint32_t many_range(uint32_t sm_addr, uint32_t tile_addr, int W, const uint32_t *offs, int K, float scale, bool pow2,
                                            int s_exp, float *u, uint32_t lo, uint32_t hi, uint32_t tile_elems)
{
    TileShared &sm = *static_cast<TileShared *>(__cvta_shared_to_generic(sm_addr));
    float *const tile = static_cast<float *>(__cvta_shared_to_generic(tile_addr));
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    ManyTensors &mt = *reinterpret_cast<ManyTensors *>(sm.lut);
    const int room = min(kMany, kAbove / W);
    int *const sums = reinterpret_cast<int *>(tile);
    bool bad = false;
    int g = group_of(offs, K, lo);                                  // tensor of the tile's first element
    uint32_t t0 = lo, t_len = 0;
    for (; t0 < hi; t0 += t_len) {
        t_len = min(hi - t0, tile_elems);
        for (int j = tid; j <= room; j += kTileThreads) mt.begin[j] = j == 0 ? 0u : g + j <= K ? offs[g + j] - t0 : 0xFFFFFFFFu;
        if (tid == 0) sm.unfit = 0;
        if (tid < (uint32_t)W) sm.taken[tid] = 0;
        __syncthreads();
        // last of the first `last + 1` tensors that begins at or before element i
        auto tensor_at = [&](uint32_t i, int last) -> int {
            int a = 0, b = last + 1;
            while (b - a > 1) {
                const int mid = (a + b) >> 1;
                if (mt.begin[mid] <= i) a = mid; else b = mid;
            }
            return a;
        };
        if (mt.begin[room] < t_len) t_len = mt.begin[room] & ~3u;
        if (t_len == 0) { __syncthreads(); break; }
        const int T = tensor_at(t_len - 1, room - 1) + 1;
        // units and exponents, four tensors per warp at a time
        for (int j0 = warp; j0 < T; j0 += 4 * kTileWarps) {
            int32_t ex[4][2];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + q * kTileWarps;
                ex[q][0] = j < T && lane < (uint32_t)W ? sm.gexp[lane][g + j] : VGC_EXP_NONE;
                ex[q][1] = j < T && lane + 32u < (uint32_t)W ? sm.gexp[lane + 32][g + j] : VGC_EXP_NONE;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + q * kTileWarps;
                if (j >= T) break;
                const int32_t b = unit_of_tensor(ex[q], W, pow2, s_exp);
                if (lane == 0) {
                    mt.base[j] = b;
                    if (b == kUnfit) sm.unfit = 1;
                }
                if (lane < (uint32_t)W) mt.above[j * W + lane] = ex[q][0] == VGC_EXP_NONE ? kNothing : (uint8_t)(ex[q][0] - b);
                if (lane + 32u < (uint32_t)W) mt.above[j * W + lane + 32] = ex[q][1] == VGC_EXP_NONE ? kNothing : (uint8_t)(ex[q][1] - b);
            }
        }
        __syncthreads();
        const bool unfit = sm.unfit;
        if (!kOverwrite) {                                          // u is read at the tile's end: ask it into L2 now
            for (uint32_t line = tid; line < (t_len + 31u) / 32u; line += kTileThreads)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(u + t0 + 32u * line));
        }
        int j = 0;                                                  // tensor of the word looked at last, its elements
        uint32_t from = 0, len = T > 1 ? mt.begin[1] : t_len;
        auto look_up = [&](uint32_t at) {
            if (at - from >= len) {
                j = tensor_at(at, T - 1);
                from = mt.begin[j];
                len = mt.begin[j + 1] - from;
            }
        };
        if (!kOverwrite && unfit) {                                 // the old content that is added to in message order
            for (uint32_t i = 4 * tid; i < t_len; i += 4 * kTileThreads) {
                look_up(i);
                if (i + 4 <= t_len && i + 3 - from < len) {
                    if (mt.base[j] == kUnfit) cp_async_16(tile + i, u + t0 + i);
                } else {
                    for (uint32_t c = i; c < min(i + 4, t_len); ++c) {
                        look_up(c);
                        if (mt.base[j] == kUnfit) tile[c] = u[t0 + c];
                    }
                }
            }
            cp_async_wait_all();                                    // (before the barrier behind the words that fit)
        }
        stream_tile(sm, W, t0, t_len, bad, [&](uint32_t word, uint32_t m, uint32_t &n_in) {
            const uint32_t at = (word - (t0 << 4)) >> 4;
            if (at >= t_len) return;
            ++n_in;
            look_up(at);
            const uint32_t above = mt.above[j * W + (int)m];
            if (mt.base[j] == kUnfit || above == kNothing) return;
            const int mult = 1 << (above - (word & 7u));
            atomicAdd(sums + at, (word & 8u) ? -mult : mult);
        });
        __syncthreads();
        if (unfit) {
            for (int w = 0; w < W; ++w) {
                const uint32_t words = sm.taken[w], *run = sm.words[w] + sm.cur[w];
                if (words == 0) continue;
                const int32_t *gexp = sm.gexp[w] + g;
                for (uint32_t i = tid; i < words; i += kTileThreads) {
                    const uint32_t word = run[i], at = (word >> 4) - t0;
                    if (at >= t_len) continue;                      // (counted as out of place above)
                    look_up(at);
                    if (mt.base[j] != kUnfit) continue;
                    tile[at] = __fadd_rn(tile[at], value_at(word, gexp[j], scale));
                }
                __syncthreads();                                    // the next message may hit the same elements
            }
        }
        if (tid < (uint32_t)W) sm.cur[tid] += sm.taken[tid];

        // ---- the tile leaves, zeros stay behind
        auto result = [&](int mult, int jj, float old) -> float {
            const int32_t b = mt.base[jj];
            if (b == kUnfit) return __int_as_float(mult);
            if (!kOverwrite && mult == 0) return old;
            const float v = __fmul_rn(times_unit(mult, power_of_two(b)), scale);
            return kOverwrite ? v : __fadd_rn(old, v);
        };
        float *const dst = u + t0;
        constexpr int kHeld = 4;                                    // vectors of u per thread in flight
        const uint32_t n_vec = t_len / 4;
        for (uint32_t q0 = tid; q0 < n_vec; q0 += kHeld * kTileThreads) {
            float4 o[kHeld];
#pragma unroll
            for (int h = 0; h < kHeld; ++h) {
                o[h] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!kOverwrite && q0 + h * kTileThreads < n_vec) o[h] = *reinterpret_cast<const float4 *>(dst + 4 * (q0 + h * kTileThreads));
            }
#pragma unroll
            for (int h = 0; h < kHeld; ++h) {
                const uint32_t q = q0 + h * kTileThreads;
                if (q >= n_vec) break;
                const int4 mlt = reinterpret_cast<const int4 *>(sums)[q];
                reinterpret_cast<int4 *>(sums)[q] = make_int4(0, 0, 0, 0);
                float4 v;
                look_up(4 * q);
                v.x = result(mlt.x, j, o[h].x);
                if (4 * q + 3 - from < len) {
                    v.y = result(mlt.y, j, o[h].y);
                    v.z = result(mlt.z, j, o[h].z);
                    v.w = result(mlt.w, j, o[h].w);
                } else {                                            // a border inside the vector
                    look_up(4 * q + 1); v.y = result(mlt.y, j, o[h].y);
                    look_up(4 * q + 2); v.z = result(mlt.z, j, o[h].z);
                    look_up(4 * q + 3); v.w = result(mlt.w, j, o[h].w);
                }
                *reinterpret_cast<float4 *>(dst + 4 * q) = v;
            }
        }
        if (tid < t_len - 4 * n_vec) {                              // the buffer's last elements
            const uint32_t i = 4 * n_vec + tid;
            look_up(i);
            dst[i] = result(sums[i], j, kOverwrite ? 0.f : dst[i]);
            sums[i] = 0;
        }
        g += tensor_at(t_len, room);
        __syncthreads();                                            // cursors, tensors, and the tile's zeros
    }
    return t0 | (bad ? kBad : 0u);
}

// Bound: HBM for the dense forms (4 B per word, 4 or 8 B per element), DRAM accesses for the sparse ones, latency for small
// buffers.  Measured (B200, one call among others, W messages): n = 25.5 M, W = 8, density 0.05, written: 45.2 -> 33.7 us
// (143 MB, 0.65 of the measured copy rate); added: 64.2 -> 58.0; W = 64, density 0.01: 107.8 -> 73.0; n = 123.6 M, W = 4,
// density 0.03: 345 -> 114 us; n = 32768: 4.3 -> 3.3 us.  The gain is the search (five rounds of scattered probes -> two),
// tiles that may span two tensors, tables made once per tensor, and the sparse forms.
template <bool kHybrid, bool kOverwrite>
__global__ void __launch_bounds__(kTileThreads, kBlocksPerSm)
decode_tiles(const __grid_constant__ DecodeViews views, int W, const uint32_t *group_offsets, int K,
             float scale, float tau, float *u, size_t n, uint32_t chunk_elems, uint32_t tile_elems,
             uint32_t *dev_status)
{
    extern __shared__ __align__(16) float tile[];                // kTileMax floats
    __shared__ TileShared sm;

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool in_smem = !kHybrid && (K + 1) <= kDecOffsSmem;
    const uint32_t *offs = in_smem ? sm.offs : group_offsets;
    if (tid == 0) sm.unfit = 0;
    if (tid < (uint32_t)W) {
        sm.words[tid] = views.words[tid];
        sm.gexp[tid] = views.group_exp[tid];
    }
    grid_wait();
    if (in_smem)
        for (int i = tid; i <= K; i += kTileThreads) sm.offs[i] = group_offsets[i];
    if (tid < (uint32_t)W) {
        // never read past the buffer the caller says it has: a truncated message (VGC_DEV_CAPACITY at the sender)
        // carries the count that was needed, not the count that was written
        const uint32_t said = *views.nnz[tid], have = views.max_words[tid];
        sm.count[tid] = said < have ? said : have;
        if (said > have && blockIdx.x == 0) atomicOr(dev_status, VGC_DEV_CAPACITY);
    }
    __syncthreads();

    const uint32_t lo = blockIdx.x * chunk_elems;
    const uint32_t hi = (uint32_t)((size_t)lo + chunk_elems < n ? (size_t)lo + chunk_elems : n);
    uint32_t total;                                              // words, in units of 64
    {
        const uint32_t c0 = lane < (uint32_t)W ? sm.count[lane] : 0u, c1 = lane + 32u < (uint32_t)W ? sm.count[lane + 32] : 0u;
        total = __reduce_add_sync(0xffffffffu, (uint32_t)(((uint64_t)c0 + c1 + 63u) >> 6));
    }
    if (total == 0 && !kOverwrite) return;
    if (hi == n && tid < (uint32_t)W) {
        const uint32_t count = sm.count[tid];
        if (count && (sm.words[tid][count - 1] >> 4) >= n) atomicOr(dev_status, VGC_DEV_RANGE);   // skipped
    }
    bool bad;
    if ((size_t)total * 64 * (kOverwrite ? sparse_write(n) : kSparseAdd) < n) {
        if constexpr (kOverwrite) {
            if (W <= kTileWarps) find_runs<8, 1>(sm, W, lo, (uint32_t)n, [] {});
            else find_runs<4, 4>(sm, W, lo, (uint32_t)n, [] {});
            __syncwarp();                                        // (a warp's cursors are its own)
            bad = scatter_range<kHybrid>(sm, W, offs, K, scale, tau, u, lo, hi);
            if (bad) atomicOr(dev_status, VGC_DEV_RANGE);
        } else {
            FlatPlan &plan = *reinterpret_cast<FlatPlan *>(sm.lut);      // (no tables in this form)
            static_assert(sizeof(FlatPlan) <= sizeof(sm.lut) && alignof(FlatPlan) <= alignof(float), "the plan takes the tables' place");
            if (warp == 0) plan_flat(plan, sm.count, W);
            __syncthreads();
            const uint32_t blocks = min(gridDim.x, flat_blocks(plan.words, n));
            if (blockIdx.x < blocks)
                add_flat<kHybrid>(sm, plan, offs, K, scale, tau, u, n, dev_status, blockIdx.x * kTileWarps + warp, blocks * kTileWarps);
        }
        return;
    }

    // ---- dense: whether the exact form applies
    // with a scale that is a positive, normal power of two its result is the sequential sum's, bit for bit
    const int s_exp = (int)((__float_as_uint(scale) >> 23) & 0xFFu) - 127;
    const bool pow2 = (__float_as_uint(scale) & 0x807FFFFFu) == 0u && s_exp > -127 && s_exp < 128;
    const int g_first = kHybrid ? 0 : group_of(offs, K, lo);
    const int g_last = kHybrid ? 0 : hi <= offs[g_first + 1] ? g_first : group_of(offs, K, hi - 1);
    // kOrdered: read 16 bytes at a time; a scale that is not finite; the filler's index would be an element
    if (tid < (uint32_t)W && (reinterpret_cast<uintptr_t>(sm.words[tid]) & 15u)) atomicOr(&sm.unfit, kOrdered);
    if (tid == 0 && (s_exp >= 128 || hi == (1u << 28))) atomicOr(&sm.unfit, kOrdered);
    if (tid == 0 && g_last - g_first >= kTensors) atomicOr(&sm.unfit, kCrowded);
    int32_t ex[2] = {VGC_EXP_NONE, VGC_EXP_NONE};                // warp j looks at the range's j-th tensor
    const int g_mine = g_first + (int)warp;
    if (!kHybrid && g_mine <= g_last) {                          // on their way during the search
        if (lane < (uint32_t)W) ex[0] = sm.gexp[lane][g_mine];
        if (lane + 32u < (uint32_t)W) ex[1] = sm.gexp[lane + 32][g_mine];
    }
    // the tile buffer starts as zeros; from then on whoever writes a tile out leaves zeros behind
    auto clear = [&] {
        for (uint32_t q = tid; q < kTileMax / 4; q += kTileThreads)
            reinterpret_cast<float4 *>(tile)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    if (W <= kTileWarps) find_runs<8, 1>(sm, W, lo, (uint32_t)n, clear);
    else find_runs<4, 4>(sm, W, lo, (uint32_t)n, clear);
    __syncwarp();
    for (uint32_t w = warp; w < (uint32_t)W; w += kTileWarps) {  // the runs' first words into L2
        const uint32_t at = sm.cur[w] + 32u * lane, count = sm.count[w];
        if (at < count && (float)(32u * lane) * (float)n < (float)count * (float)(hi - lo))
            asm volatile("prefetch.global.L2 [%0];" ::"l"(sm.words[w] + at));
    }
    if (!kHybrid && g_mine <= g_last) {
        const int32_t b = unit_of_tensor(ex, W, pow2, s_exp);
        if (lane == 0) {
            // a tile of exact_range takes elements of two tensors at most and begins at a multiple of four elements: a
            // tensor of fewer than seven between two others would make it three
            const uint32_t size = offs[g_mine + 1] - offs[g_mine];
            uint32_t about = b == kUnfit ? kSomeUnfit : kSomeFit;
            if (g_mine > g_first && g_mine < g_last && size > 0 && size < 7) about |= kCrowded;
            atomicOr(&sm.unfit, about);
            sm.base[warp] = b;
        }
    }
    __syncthreads();
    const uint32_t about = sm.unfit;
    const uint32_t sm_addr = (uint32_t)__cvta_generic_to_shared(&sm), tile_addr = (uint32_t)__cvta_generic_to_shared(tile);
    uint32_t from = lo;                                          // what is left to the ordered form
    bad = false;
    if (!(about & (kOrdered | kCrowded | kSomeUnfit))) {
        bad = exact_range<kHybrid, kOverwrite>(sm, tile, W, offs, g_first, scale, tau, u, lo, hi, tile_elems);
        from = hi;
    } else if constexpr (!kHybrid) {
        if (!(about & kOrdered) && (about & (kCrowded | kSomeFit))) {
            __syncthreads();                                     // (everybody has read sm.unfit)
            const uint32_t end = many_range<kOverwrite>(sm_addr, tile_addr, W, offs, K, scale, pow2, s_exp, u, lo, hi, tile_elems);
            from = end & ~kBad;
            bad = (end & kBad) != 0;
        }
    }
    if (from < hi) bad |= ordered_range<kHybrid, kOverwrite>(sm_addr, tile_addr, W, offs, K, scale, tau, u, from, hi, tile_elems);
    if (bad) atomicOr(dev_status, VGC_DEV_RANGE);
}

}  // namespace vgc

using namespace vgc;

namespace {
typedef void (*TilesFn)(const DecodeViews, int, const uint32_t *, int, float, float, float *, size_t, uint32_t, uint32_t,
                        uint32_t *);

vgc_status decode_launch(bool hybrid, bool overwrite, const vgc_message_view *msgs, int W, const uint32_t *group_offsets,
                         int K, float scale, float tau, float *u, size_t n, uint32_t *dev_status, cudaStream_t st)
{
    if (W == 0) {                                                // vgc_decode_sum of nothing
        VGC_CUDA_OK(cudaMemsetAsync(u, 0, n * sizeof(float), st));
        return VGC_OK;
    }
    for (int w0 = 0; w0 < W; w0 += kMaxViews) {
        const int wb = W - w0 < kMaxViews ? W - w0 : kMaxViews;
        DecodeViews views;
        for (int w = 0; w < kMaxViews; ++w) {
            const vgc_message_view &m = msgs[w0 + (w < wb ? w : 0)];
            views.words[w] = m.words;
            views.nnz[w] = m.nnz;
            views.group_exp[w] = m.group_exp;
            views.max_words[w] = m.max_words;
        }
        const bool ow = overwrite && w0 == 0;                    // later groups of messages add to the first
        size_t most_words = 0, longest = 0;
        for (int w = 0; w < wb; ++w) {
            most_words += views.max_words[w];
            longest = longest > views.max_words[w] ? longest : views.max_words[w];
        }
        if (!ow && most_words * kSparseAdd < n) {                // whatever the counts on the device say
            const size_t want = ((longest + kPiece - 1) / kPiece * wb + kFlatThreads / 32 - 1) / (kFlatThreads / 32);
            const unsigned blocks = (unsigned)(want < 1 ? 1 : want < (size_t)kFlatMost ? want : (size_t)kFlatMost);
            VGC_CUDA_OK(launch_kernel(hybrid ? decode_flat<true> : decode_flat<false>, dim3(blocks), dim3(kFlatThreads), 0, st, true,
                                      views, wb, group_offsets, K, scale, tau, u, n, dev_status));
            count_launch();
            continue;
        }
        // one contiguous range per block, kBlocksPerSm blocks per SM, tiles of equal size; not less than 2048 elements
        // each: a range costs its search
        size_t chunk = (n + (size_t)kSmCount * kBlocksPerSm - 1) / ((size_t)kSmCount * kBlocksPerSm);
        chunk = chunk > 2048 ? chunk : 2048;
        chunk = (chunk + 3) / 4 * 4;
        const size_t tiles = (chunk + kTileMax - 1) / kTileMax;
        const uint32_t tile_elems = (uint32_t)(((chunk + tiles - 1) / tiles + 3) / 4 * 4);
        const unsigned blocks = (unsigned)((n + chunk - 1) / chunk);
        TilesFn fn = hybrid ? (ow ? decode_tiles<true, true> : decode_tiles<true, false>)
                            : (ow ? decode_tiles<false, true> : decode_tiles<false, false>);
        VGC_CUDA_OK(allow_dynamic_smem(reinterpret_cast<const void *>(fn), (size_t)kTileMax * 4));
        VGC_CUDA_OK(launch_kernel(fn, dim3(blocks), dim3(kTileThreads), (size_t)kTileMax * 4, st, true, views, wb, group_offsets, K,
                                  scale, tau, u, n, (uint32_t)chunk, tile_elems, dev_status));
        count_launch();
    }
    VGC_CUDA_OK(cudaGetLastError());
    return VGC_OK;
}

bool views_ok(const vgc_message_view *msgs, int W, bool need_exp)
{
    for (int w = 0; w < W; ++w)
        if (!msgs[w].words || !msgs[w].nnz || (need_exp && !msgs[w].group_exp)) return false;
    return true;
}
}  // namespace

extern "C" vgc_status vgc_decode_accumulate(const vgc_message_view *msgs, int W,
                                            const uint32_t *group_offsets, int K, float scale,
                                            float *u, size_t n, uint32_t *dev_status, vgc_stream_t stream)
{
    if (W == 0 || n == 0) return VGC_OK;
    if (W < 0 || K < 1 || n > VGC_MAX_PARAMS || !msgs || !group_offsets || !u || !dev_status || !aligned16(u))
        return VGC_ERR_INVALID_ARG;
    if (!(scale == scale) || !views_ok(msgs, W, true)) return VGC_ERR_INVALID_ARG;
    return decode_launch(false, false, msgs, W, group_offsets, K, scale, 0.f, u, n, dev_status,
                         reinterpret_cast<cudaStream_t>(stream));
}

extern "C" vgc_status vgc_decode_accumulate_hybrid(const vgc_message_view *msgs, int W, float tau, float scale,
                                                   float *u, size_t n, uint32_t *dev_status, vgc_stream_t stream)
{
    if (W == 0 || n == 0) return VGC_OK;
    if (W < 0 || n > VGC_MAX_PARAMS || !msgs || !u || !dev_status || !aligned16(u)) return VGC_ERR_INVALID_ARG;
    if (!(scale == scale) || !(tau == tau) || !views_ok(msgs, W, false)) return VGC_ERR_INVALID_ARG;
    return decode_launch(true, false, msgs, W, nullptr, 0, scale, tau, u, n, dev_status,
                         reinterpret_cast<cudaStream_t>(stream));
}

extern "C" vgc_status vgc_decode_sum(const vgc_message_view *msgs, int W, const uint32_t *group_offsets, int K,
                                     float scale, float *u, size_t n, uint32_t *dev_status, vgc_stream_t stream)
{
    if (n == 0) return VGC_OK;
    if (W < 0 || K < 1 || n > VGC_MAX_PARAMS || (W > 0 && !msgs) || !group_offsets || !u || !dev_status || !aligned16(u))
        return VGC_ERR_INVALID_ARG;
    if (!(scale == scale) || !views_ok(msgs, W, true)) return VGC_ERR_INVALID_ARG;
    return decode_launch(false, true, msgs, W, group_offsets, K, scale, 0.f, u, n, dev_status,
                         reinterpret_cast<cudaStream_t>(stream));
}

extern "C" vgc_status vgc_decode_sum_hybrid(const vgc_message_view *msgs, int W, float tau, float scale, float *u,
                                            size_t n, uint32_t *dev_status, vgc_stream_t stream)
{
    if (n == 0) return VGC_OK;
    if (W < 0 || n > VGC_MAX_PARAMS || (W > 0 && !msgs) || !u || !dev_status || !aligned16(u)) return VGC_ERR_INVALID_ARG;
    if (!(scale == scale) || !(tau == tau) || !views_ok(msgs, W, false)) return VGC_ERR_INVALID_ARG;
    return decode_launch(true, true, msgs, W, nullptr, 0, scale, tau, u, n, dev_status,
                         reinterpret_cast<cudaStream_t>(stream));
}
