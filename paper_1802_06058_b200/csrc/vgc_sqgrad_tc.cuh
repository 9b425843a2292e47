// Squared per-example gradient sums on the 5th-generation tensor cores (tcgen05, sm_100a).
//
//   D[m][n] = sum_k A(k,m)^2 * B(k,n)^2          (the contraction behind Eq. 2 / Algorithm 1's
//                                                  "v_i +=" line; N_params*|B| multiply-adds, Sec. 5)
// Operands stay fp32 in global memory.  Per 32-deep k slice a thread block
//   1. TMA-loads the raw fp32 tiles of A (128 rows) and B (kBN rows) into a pipeline stage
//      (128-byte swizzle, out-of-range parts filled with zeros),
//   2. squares every element in fp32 and splits the square into two TF32 numbers hi + lo
//      (hi = x*x rounded to 11 significant bits, lo = x*x - hi, of which the tensor core reads the
//      leading 11 bits); the transform is elementwise
//      and in place (hi overwrites the raw tile, lo goes beside it), so both inherit the swizzled
//      layout the tensor core wants,
//   3. issues three tcgen05.mma per 8-deep step -- hi*hi, hi*lo, lo*hi -- into a TMEM
//      accumulator (the dropped lo*lo term is 2^-22 relative).  In the TMA-fed K-major form, and in the
//      wide form where accumulator runs are long and terms many (bf16_cross_better), the two cross terms
//      use bf16 copies of hi and lo instead (kind::f16, 16 deep per instruction): a cross term is 2^-11 of
//      the product, so 8-bit operands leave an error below 2^-18 of it, of either sign -- in such sums less
//      than the third of the instructions saves of the accumulator's truncation bias (largest error of 128
//      channels 28 x 28, batch 16: 2.9e-6 -> 2.4e-6).
// The tensor core's fp32 accumulation is not trusted over long reductions: every kChunk k slices
// the accumulator is drained by four epilogue warps (tcgen05.ld) and added, round-to-nearest, to
// fp32 registers while the next chunk accumulates into the second TMEM buffer.
// Work distribution: the (layer, tile, k slice) space of a launch is laid out linearly and cut into one
// contiguous range per thread block, with at most one block per SM; a block walks its range segment by
// segment (a segment = consecutive slices of one output tile) with the pipeline running across segment
// borders.  A segment that covers a tile's whole reduction writes the result; otherwise it writes a partial
// tile to scratch and a second kernel adds the partial tiles of a tile in a fixed order.
//
// Operand layouts:
//   dense layer: A = delta[z][out], B = x[z][in]  (m / n innermost: MN-major tiles, both by TMA)
//   conv layer:  the error tile is delta[z][o][p], p = (ho,wo) innermost (K-major); the input tile is
//                the im2col view of x, row (c,kh,kw), column k = (z,ho,wo).  Each example contributes
//                ceil(P/32) slices.  Error tile: TMA when the row pitch P*4 is a multiple of 16 bytes,
//                else gathered.  Input tile: TMA for a 1x1 / stride 1 / unpadded kernel (then it is
//                just x[z][c][p]); otherwise the transform warps gather it straight from global
//                memory, four consecutive k per thread, zero outside the image -- im2col is never
//                materialised.  With few output channels (Cout <= 64) the roles are swapped: the
//                im2col rows become the 128-row A tile and the errors the narrow B tile.
//
// Warp roles (512 threads): 0 TMA producer, 1 MMA issuer + TMEM owner, 4-11 transform, 12-15 epilogue.
// While the epilogue warps write a segment's tile out, the other roles are already working on the next one.
// Every wait on an mbarrier is bounded; on expiry the block raises an abort flag, all roles fall
// through to the common exit, outstanding TMA loads are waited for (bounded) and TMEM is freed.
#pragma once

#include "vgc_rows.cuh"
#include "vgc_tc.cuh"

namespace vgc {

namespace tc {

#ifndef VGC_TC_RAW_SLOTS
#define VGC_TC_RAW_SLOTS 5
#endif
#ifndef VGC_TC_LO_SLOTS
#define VGC_TC_LO_SLOTS 2
#endif
// The pipeline is bound by how many bytes are in flight, so the raw tiles get as many slots as fit:
// a raw slot holds the fp32 tiles of one slice (overwritten in place by their hi parts), a lo slot the
// lo parts, which only exist between the transform and the MMAs that consume them.
constexpr int kRawSlots = VGC_TC_RAW_SLOTS;
constexpr int kLoSlots = VGC_TC_LO_SLOTS;
#ifndef VGC_TC_GROUPS
#define VGC_TC_GROUPS 2
#endif
// Transform warps: groups of four warps; in the forms whose slices are taken by one group each, the groups work on
// consecutive slices side by side (a slice's transform is a chain of shared-memory round trips, waits and fences: its
// latency, not the arithmetic, sets the pace, so slices in flight are what counts).  The element-wise gathers share a
// slice among eight warps (the first two groups).
constexpr int kGroups = VGC_TC_GROUPS;
constexpr int kTransformWarps = 4 * kGroups;
constexpr int kGatherThreads = 256;                                 // threads sharing a slice in the one-group forms
constexpr int kEpilogueWarps = 4;
// Warps 0 and 1 are the producer and the issuer, 2 and 3 idle, so that the transform groups and the epilogue are warpgroups
// and can be given different shares of the registers: the epilogue holds 128 sums per lane and spilled 1.4 KB of loads per
// lane and chunk at the 128 registers that an even split leaves.
constexpr int kFirstTransform = 4, kFirstEpilogue = kFirstTransform + kTransformWarps;
constexpr int kThreadsTc = 32 * (kFirstEpilogue + kEpilogueWarps);
constexpr int kRegsLaunch = 65536 / kThreadsTc, kRegsFew = 40, kRegsTransform = 112, kRegsEpilogue = 232;
constexpr int kRegsTransformWide = 120, kRegsEpilogueWide = 232;
static_assert(kGroups == 2 && 128 * (kRegsFew + kGroups * kRegsTransform + kRegsEpilogue) <= kRegsLaunch * kThreadsTc &&
              128 * (kRegsFew + kGroups * kRegsTransformWide + kRegsEpilogueWide) <= kRegsLaunch * kThreadsTc,
              "the shares come out of what the block was launched with");
template <int kRegs> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs)); }
template <int kRegs> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs)); }
constexpr uint32_t kRawBytesA = kBM * kBK * 4;                      // 16 KB
constexpr uint32_t kRawBytesB = kBN * kBK * 4;                      // 16 KB
constexpr uint32_t kRawStageBytes = kRawBytesA + kRawBytesB;        // 32 KB: [A raw/hi][B raw/hi], same for lo
constexpr uint32_t kLoBase = kRawSlots * kRawStageBytes;            // lo slots follow the raw slots
constexpr uint32_t kSmemBytes = (kRawSlots + kLoSlots) * kRawStageBytes + 1024 /*align*/ + 128;
// With the A operand in tensor memory a lo slot holds the B tile only, so twice as many fit; the A
// operand ring in TMEM has the same number of slots and shares their barrier.
constexpr int kLoSlotsAT = 2 * kLoSlots;
// Pure TMA form with A in tensor memory ("split rings"): the raw A tile is dead as soon as the transform has
// read it, long before the MMAs of its slice retire.  It therefore gets a ring of its own that is freed
// early, and the 16-KB units this saves hold more B tiles: more slices in flight from the same shared memory.
constexpr int kSplitA = 4, kSplitB = 7, kSplitLo = 3;   // 16-KB units: A raw, B raw/hi, B lo (+ A in TMEM)
static_assert((kSplitA + kSplitB + kSplitLo) * kRawBytesA <= (kRawSlots + kLoSlots) * kRawStageBytes, "smem budget");
// Wide form (the kernels that gather several taps at a time, tiles of 192 columns): the tensor core takes an N = 192
// instruction in no more time than an N = 128 one (98 busy cycles by the counters, 110), and 192 rows of the im2col view are 64 whole triples.  The raw A
// tiles have a ring of two, the B tile and its lo part one of four, A in tensor memory two slots beside two accumulators.
constexpr int kWideN = 192, kWideA = 2, kWideB = 4, kWideTmemA = 2;
static_assert(kWideA * kRawBytesA + 2 * kWideB * kWideN * kBK * 4 <= (kRawSlots + kLoSlots) * kRawStageBytes, "smem budget");
static_assert(2 * kWideN + kWideTmemA * 64 <= 512, "tensor memory");
// With the input rows by TMA a ring of four slots of them (8 KB) takes the place of the fourth B tile.
constexpr int kHaloB = 3, kHaloSlots = 4;
constexpr uint32_t kHaloSlotMost = 8192;
constexpr uint32_t kHaloBase = kWideA * kRawBytesA + 2 * kHaloB * kWideN * kBK * 4;
static_assert(kHaloBase + kHaloSlots * kHaloSlotMost <= (kRawSlots + kLoSlots) * kRawStageBytes, "smem budget");
constexpr uint32_t kTmemColsA = 64;                                 // per slot: 32 columns hi + 32 columns lo
constexpr uint32_t kTmemCols = 512;                                 // two accumulator buffers + the A operand ring

// how a tile gets its rows; kGatherTaps4 / kGatherTaps2: im2col rows of a Kw = 3, stride 1, pad_w = 1 kernel
// gathered three taps at a time (output width a multiple of 4 / of 2)
// kGatherTaps4S2 / kGatherTaps2S2: the same for stride 2 along w (input width twice the output width)
// kGatherTaps7S2: seven taps at a time for a Kw = 7, stride-2, pad-3 kernel (the first layer of the ImageNet networks)
// kHalo...: im2col rows of a square kernel of 5 or 7 taps that keeps the width (stride 1), from input rows that TMA brings
// into shared memory (width a multiple of 4 / of 2)
enum { kTma = 0, kGatherErr = 1, kGatherIm2col = 2, kGatherTaps4 = 3, kGatherTaps2 = 4, kGatherTaps4S2 = 5,
       kGatherTaps2S2 = 6, kGatherTaps7S2 = 7, kHalo5x4 = 8, kHalo5x2 = 9, kHalo7x4 = 10, kHalo7x2 = 11 };

struct Params {
    int M, N;                // rows of the A tile space / of the B tile space
    int k_slices;            // 32-deep slices of one tile's reduction
    int p_slices;            // conv: slices per example (ceil(P/32)); dense: 1
    int chunk;               // slices per accumulator drain
    int unit;                // slices that stay in one block: the reduction is cut between units only
    int units_per_tile;      // k_slices / unit
    int parts, part_slices;  // per-example form, examples cut up: parts of an example (0: whole examples), slices of one; a block each
    int units_total;         // layers * tiles * units_per_tile: the launch's work, cut evenly over the blocks:
    int units_q, units_r;    // block b owns units [b q + min(b, r), ...) with q = total / blocks, r = total % blocks
    int tile_n;              // columns of a tile: 128, or 192 (wide form)
    int tiles_x, tiles_y;    // tiles of one layer's result
    uint32_t tx_bytes;       // bytes the TMA loads of one slice deliver
    uint32_t tx_bytes_a;     // of which the A tile's
    float scale;
    int accumulate;
    int C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, Wo, P;     // conv geometry (gathered tiles)
    int chw;                 // C*H*W
    unsigned wo_magic;       // p / Wo == row_of(p, wo_magic, wo_shift); Wo >= 2
    int wo_shift;
    long long ld_m, ld_n;    // result: element (m, n) lives at S[m*ld_m + n*ld_n]; one of the two is 1
    float *partial;          // scratch for partial tiles [2 * block + (0: a block's first segment, 1: its last)][column / 4][row][column % 4]
    uint32_t *status;        // device word; VGC_DEV_TIMEOUT is OR-ed in if a wait expired
};

// Layers of one geometry computed by one launch: their tensor maps and pointers.
constexpr int kMaxBatch = 8;
struct Batch {
    CUtensorMap a[kMaxBatch], b[kMaxBatch];
    const float *x[kMaxBatch], *delta[kMaxBatch];   // raw operands (gathered tiles)
    float *S[kMaxBatch];
};

// One 16-byte chunk (4 consecutive k of one row) of a K-major 128-byte-swizzled tile.
__device__ __forceinline__ uint32_t chunk_offset(int row, int kq) { return (uint32_t)row * 128u + (uint32_t)((kq ^ (row & 7)) << 4); }

// Four consecutive k of one row of a K-major tile of bf16: 64-byte rows, 64-byte swizzle.
__device__ __forceinline__ uint32_t bf_offset(int row, int kq)
{
    return (uint32_t)row * 64u + (uint32_t)((((kq >> 1) ^ (row >> 1)) & 3) << 4) + (uint32_t)((kq & 1) << 3);
}

constexpr int kRowsPerThread = kBM * 8 / kGatherThreads;        // 4 gathered chunks per thread per tile

// The four rows (row0 + 32*i) of a gathered tile that one transform thread owns.
template <int kMode>
struct GatherRows {
    int base[kRowsPerThread], dh[kRowsPerThread], dw[kRowsPerThread];
    bool ok[kRowsPerThread];
    const float *src;       // x (im2col rows) or delta (error rows) of this block's layer

    __device__ __forceinline__ void init(const Params &prm, const float *x, const float *delta, int first_row, int limit)
    {
        if (kMode == kTma) return;
        src = kMode == kGatherIm2col ? x : delta;
        const int khw = prm.Kh * prm.Kw;
#pragma unroll
        for (int i = 0; i < kRowsPerThread; ++i) {
            const int idx = first_row + 32 * i;
            ok[i] = idx < limit;
            const int ii = ok[i] ? idx : 0;
            if (kMode == kGatherIm2col) {
                const int c = ii / khw, rem = ii - c * khw;
                const int kh = rem / prm.Kw, kw = rem - kh * prm.Kw;
                dh[i] = kh - prm.ph;
                dw[i] = kw - prm.pw;
                base[i] = (c * prm.H + dh[i]) * prm.W + dw[i];
            } else {
                base[i] = ii * prm.P;   // offset of the output channel's plane
                dh[i] = dw[i] = 0;
            }
        }
    }
    // loads this thread's 4 rows x 4 consecutive k: example z, output positions pbase .. pbase+3
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, float (&v)[kRowsPerThread][4]) const
    {
        if (kMode == kGatherIm2col) {
            const float *xz = src + (size_t)z * prm.chw;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = pbase + j;
                const int ho = prm.Wo == 1 ? p : (int)row_of((unsigned)p, prm.wo_magic, prm.wo_shift), wo = p - ho * prm.Wo;
                const int hs = ho * prm.sh, ws = wo * prm.sw;
                const float *xp = xz + (hs * prm.W + ws);
                const bool pv = p < prm.P;
#pragma unroll
                for (int i = 0; i < kRowsPerThread; ++i) {
                    const bool in = pv && (unsigned)(hs + dh[i]) < (unsigned)prm.H &&
                                    (unsigned)(ws + dw[i]) < (unsigned)prm.W;
                    v[i][j] = in ? xp[base[i]] : 0.f;
                }
            }
        } else if (kMode == kGatherErr) {
            const float *dz = src + (size_t)z * prm.Cout * prm.P + pbase;
#pragma unroll
            for (int i = 0; i < kRowsPerThread; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[i][j] = (ok[i] && pbase + j < prm.P) ? dz[base[i] + j] : 0.f;
        }
    }
};

// Kw = 3, stride 1, pad_w = 1: the three rows (c, kh, kw = 0..2) of the im2col view read the same input row
// shifted by one, so a thread takes whole triples: for 4 (or 2 + 2) consecutive output positions it loads
// the input row segment once -- one aligned vector and its two neighbours -- and feeds all three rows from
// it.  A thread owns the triples first_triple + grp + 32*i (i = 0, 1) of the tile's rows; triples that
// straddle the tile's first or last row are handled by the row test at store time.
// kTriples = 2: 256 threads share a slice (triples grp + 32 i); kTriples = 3: 128 threads do (grp + 16 i).
template <int kSpan, int kTriples>      // kSpan: output positions covered by one aligned vector load, 4 or 2
struct GatherTaps {
    static constexpr int kStride = kTriples == 2 ? 32 : 16;
    static constexpr int kKw = 3;
    static constexpr int kSlots = 8;                         // registers per triple
    static constexpr int kLoaded = kSpan == 4 ? 6 : 8;       // of which loaded
    // register that holds the input of tap kw for the j-th of the thread's four output positions
    __device__ __forceinline__ static constexpr int idx(int kw, int j) { return kSpan == 4 ? kw + j : (j >> 1) * 4 + (j & 1) + kw; }
    int base[kTriples], dh[kTriples], row0;      // dh: far outside where the tuple has no rows; row0: tile row of the first tuple
    __device__ __forceinline__ int row(int i) const { return row0 + kKw * kStride * i; }
    const float *src;

    __device__ __forceinline__ void init(const Params &prm, const float *x, int tile_origin, int grp, int limit)
    {
        src = x;
        const int first_triple = tile_origin / 3;
        row0 = 3 * (first_triple + grp) - tile_origin;               // (may be -2, -1)
#pragma unroll
        for (int i = 0; i < kTriples; ++i) {
            const int T = first_triple + grp + kStride * i;          // triple = (c, kh)
            const bool ok = 3 * T < limit;
            const int tt = ok ? T : 0;
            const int c = tt / prm.Kh, kh = tt - c * prm.Kh;
            base[i] = (c * prm.H + kh - prm.ph) * prm.W;
            dh[i] = ok ? kh - prm.ph : INT32_MIN / 2;
        }
    }
    // v[i][0..7]: kSpan = 4: {left, m0, m1, m2, m3, right, -, -} for positions pbase..pbase+3;
    //             kSpan = 2: {left, m0, m1, right} for pbase, pbase+1 and the same for pbase+2, pbase+3
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, float (&v)[kTriples][8]) const
    {
        const float *xz = src + (size_t)z * prm.chw;
#pragma unroll
        for (int s = 0; s < 4 / kSpan; ++s) {
            const int p = pbase + s * kSpan;
            const int ho = (int)row_of((unsigned)p, prm.wo_magic, prm.wo_shift), wo = p - ho * prm.Wo;
            const bool pv = p < prm.P;
            const float *xp = xz + (ho * prm.W + wo);
#pragma unroll
            for (int i = 0; i < kTriples; ++i) {
                const bool in = pv && (unsigned)(ho + dh[i]) < (unsigned)prm.H;
                const float *q = xp + base[i];
                float *o = &v[i][s * 4];
                if (kSpan == 4) {
                    const float4 m = in ? *reinterpret_cast<const float4 *>(q) : make_float4(0.f, 0.f, 0.f, 0.f);
                    o[0] = (in && wo > 0) ? q[-1] : 0.f;
                    o[1] = m.x; o[2] = m.y; o[3] = m.z; o[4] = m.w;
                    o[5] = (in && wo + 4 < prm.W) ? q[4] : 0.f;
                } else {
                    const float2 m = in ? *reinterpret_cast<const float2 *>(q) : make_float2(0.f, 0.f);
                    o[0] = (in && wo > 0) ? q[-1] : 0.f;
                    o[1] = m.x; o[2] = m.y;
                    o[3] = (in && wo + 2 < prm.W) ? q[2] : 0.f;
                }
            }
        }
    }
    // the four k of tap kw of triple i
    __device__ __forceinline__ static void tap(const float (&v)[kTriples][8], int i, int kw, float (&out)[4])
    {
        if (kSpan == 4) {
            out[0] = v[i][kw]; out[1] = v[i][kw + 1]; out[2] = v[i][kw + 2]; out[3] = v[i][kw + 3];
        } else {
            out[0] = v[i][kw]; out[1] = v[i][kw + 1]; out[2] = v[i][4 + kw]; out[3] = v[i][4 + kw + 1];
        }
    }
};

// Stride 2 along w with Kw = 3, pad_w = 1 and W == 2 Wo: the 4 (or 2) output positions of a span read the input
// columns 2 wo - 1 .. 2 wo + 7 (or + 3): one neighbour on the left and two (one) aligned 4-vectors, never past the
// row's end.  Tap kw of output j is element 2 j + kw of that segment.
template <int kSpan, int kTriples>
struct GatherTapsS2 {
    static constexpr int kStride = kTriples == 2 ? 32 : 16;
    static constexpr int kPerSpan = kSpan == 4 ? 9 : 5;
    static constexpr int kKw = 3;
    static constexpr int kSlots = 10;
    static constexpr int kLoaded = kSpan == 4 ? 9 : 10;
    __device__ __forceinline__ static constexpr int idx(int kw, int j)
    {
        return kSpan == 4 ? 2 * j + kw : (j >> 1) * 5 + 2 * (j & 1) + kw;
    }
    int base[kTriples], dh[kTriples], row0;      // dh: far outside where the tuple has no rows; row0: tile row of the first tuple
    __device__ __forceinline__ int row(int i) const { return row0 + kKw * kStride * i; }
    const float *src;

    __device__ __forceinline__ void init(const Params &prm, const float *x, int tile_origin, int grp, int limit)
    {
        src = x;
        const int first_triple = tile_origin / 3;
        row0 = 3 * (first_triple + grp) - tile_origin;               // (may be -2, -1)
#pragma unroll
        for (int i = 0; i < kTriples; ++i) {
            const int T = first_triple + grp + kStride * i;          // triple = (c, kh)
            const bool ok = 3 * T < limit;
            const int tt = ok ? T : 0;
            const int c = tt / prm.Kh, kh = tt - c * prm.Kh;
            base[i] = (c * prm.H + kh - prm.ph) * prm.W;
            dh[i] = ok ? kh - prm.ph : INT32_MIN / 2;
        }
    }
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, float (&v)[kTriples][kSlots]) const
    {
        const float *xz = src + (size_t)z * prm.chw;
#pragma unroll
        for (int s = 0; s < 4 / kSpan; ++s) {
            const int p = pbase + s * kSpan;
            const int ho = (int)row_of((unsigned)p, prm.wo_magic, prm.wo_shift), wo = p - ho * prm.Wo;
            const bool pv = p < prm.P;
            const int hs = ho * prm.sh;
            const float *xp = xz + (hs * prm.W + 2 * wo);
#pragma unroll
            for (int i = 0; i < kTriples; ++i) {
                const bool in = pv && (unsigned)(hs + dh[i]) < (unsigned)prm.H;
                const float *q = xp + base[i];
                float *o = &v[i][s * kPerSpan];
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 m0 = in ? *reinterpret_cast<const float4 *>(q) : zero;
                o[0] = (in && wo > 0) ? q[-1] : 0.f;
                o[1] = m0.x; o[2] = m0.y; o[3] = m0.z; o[4] = m0.w;
                if (kSpan == 4) {
                    const float4 m1 = in ? reinterpret_cast<const float4 *>(q)[1] : zero;
                    o[5] = m1.x; o[6] = m1.y; o[7] = m1.z; o[8] = m1.w;
                }
            }
        }
    }
};

// Kw = 7, stride 2, pad_w = 3, W == 2 Wo, Wo a multiple of 4: the seven rows (c, kh, kw = 0..6) read, for four
// consecutive output positions, the input columns 2 wo - 3 .. 2 wo + 9.  Four aligned 4-vectors from column 2 wo - 4
// on cover them (each wholly inside or wholly outside the row); tap kw of output j is element 1 + 2 j + kw.
// 128 threads share a slice; a thread owns the tuples first_tuple + grp + 16 i, i = 0, 1 (at most 20 touch a tile).
template <int kTuples>
struct GatherTaps7S2 {
    static_assert(kTuples == 2, "used by the two-group form only");
    static constexpr int kStride = 16;
    static constexpr int kKw = 7;
    static constexpr int kSlots = 16;
    static constexpr int kLoaded = 14;
    __device__ __forceinline__ static constexpr int idx(int kw, int j) { return 1 + 2 * j + kw; }
    int base[kTuples], dh[kTuples], row0;      // dh: far outside where the tuple has no rows; row0: tile row of the first tuple
    __device__ __forceinline__ int row(int i) const { return row0 + kKw * kStride * i; }
    const float *src;

    __device__ __forceinline__ void init(const Params &prm, const float *x, int tile_origin, int grp, int limit)
    {
        src = x;
        const int first_tuple = tile_origin / 7;
        row0 = 7 * (first_tuple + grp) - tile_origin;
#pragma unroll
        for (int i = 0; i < kTuples; ++i) {
            const int T = first_tuple + grp + kStride * i;           // tuple = (c, kh)
            const bool ok = 7 * T < limit;
            const int tt = ok ? T : 0;
            const int c = tt / prm.Kh, kh = tt - c * prm.Kh;
            base[i] = (c * prm.H + kh - prm.ph) * prm.W;
            dh[i] = ok ? kh - prm.ph : INT32_MIN / 2;
        }
    }
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, float (&v)[kTuples][kSlots]) const
    {
        const int ho = (int)row_of((unsigned)pbase, prm.wo_magic, prm.wo_shift), wo = pbase - ho * prm.Wo;
        const int hs = ho * prm.sh;
        const bool pv = pbase < prm.P;
        const float *xp = src + (size_t)z * prm.chw + (hs * prm.W + 2 * wo - 4);
        const int col0 = 2 * wo - 4;
#pragma unroll
        for (int i = 0; i < kTuples; ++i) {
            const bool in = pv && (unsigned)(hs + dh[i]) < (unsigned)prm.H;
            const float4 *q = reinterpret_cast<const float4 *>(xp + base[i]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool inside = in && (unsigned)(col0 + 4 * u) < (unsigned)prm.W;
                const float4 m = inside ? q[u] : make_float4(0.f, 0.f, 0.f, 0.f);
                v[i][4 * u] = m.x; v[i][4 * u + 1] = m.y; v[i][4 * u + 2] = m.z; v[i][4 * u + 3] = m.w;
            }
        }
    }
};

template <int kMode> struct IsTaps {
    static constexpr bool value = kMode == kGatherTaps4 || kMode == kGatherTaps2 || kMode == kGatherTaps4S2 ||
                                  kMode == kGatherTaps2S2 || kMode == kGatherTaps7S2;
};
template <int kMode, int kTriples> struct TapsOf { typedef GatherTaps<kMode == kGatherTaps4 ? 4 : 2, kTriples> type; };
template <int kTriples> struct TapsOf<kGatherTaps4S2, kTriples> { typedef GatherTapsS2<4, kTriples> type; };
template <int kTriples> struct TapsOf<kGatherTaps2S2, kTriples> { typedef GatherTapsS2<2, kTriples> type; };
template <int kTriples> struct TapsOf<kGatherTaps7S2, kTriples> { typedef GatherTaps7S2<2> type; };

// ---- input rows by TMA ("halo" forms) -----------------------------------------------------------------------------------
// A kernel of K x K taps, stride 1, that keeps the width (2 pad_w = K - 1): in the flattened input plane, tap (kh, kw) of output
// position p reads p + (kh - pad_h) W + kw - pad_w, so the K rows (c, kh, 0..K-1) of a slice's 32 positions are 32 + K - 1 consecutive
// floats of the plane.  TMA brings them, zeros outside the plane (rows above and below the image); what wraps around the image's
// sides is masked here.  A TMA copy starts at a multiple of four floats, so a row holds up to three floats more in front.
// A tile is kTuples whole tuples (c, kh); its rows in shared memory go by kh first, a box of kChannels channels each.
// Bound: shared memory, as the other wide forms, with 15 KB more traffic a slice.  Element by element the same layers took (B200, us,
// before / now): 32 channels 64 x 64 to 19, 5 taps, 16 examples 110 / 62; 659 channels 8 x 8 to 32, 5 taps, 62 examples 121 / 72; 16 channels
// 28 x 28 to 65, 7 taps, 45 examples 62 / 40.  Three taps are faster gathered straight from global memory (128 channels 28 x 28, batch
// 32: 38.6 against 43.4; 14 x 14, per-example statistic: 47.4 against 51.5).
template <int kMode> struct IsHalo { static constexpr bool value = kMode >= kHalo5x4 && kMode <= kHalo7x2; };
template <int kMode>
struct Halo {
    static constexpr int kKw = kMode <= kHalo5x2 ? 5 : 7, kPad = kKw / 2;
    static constexpr int kSpan = kMode % 2 == 0 ? 4 : 2;             // outputs of a thread that surely share an image row
    static constexpr int kTuples = kWideN / kKw, kCols = kTuples * kKw;          // 38, 27 tuples; 190, 189 columns
    static constexpr int kChannels = (kTuples + kKw - 2) / kKw + 1;             // 9, 5
    static constexpr int kPos = kKw == 7 ? 44 : 40;                             // floats of a row
    static constexpr uint32_t kRowBytes = kPos * 4, kBoxBytes = (kChannels * kRowBytes + 127) / 128 * 128;
    static constexpr uint32_t kSlotBytes = kKw * kBoxBytes;
    static constexpr int kPerThread = (kTuples + 15) / 16;                      // 16 threads side by side per eight k
    static constexpr int kValues = kSpan == 4 ? kKw + 3 : 2 * (kKw + 1);        // split values of a tuple
    // where the input of tap kw for the j-th of a thread's four outputs is
    __device__ __forceinline__ static constexpr int idx(int kw, int j) { return kSpan == 4 ? kw + j : (j >> 1) * (kKw + 1) + (j & 1) + kw; }
    // floats in front of the first one a row needs; the same for all slices (their first positions are multiples of 32)
    __device__ __forceinline__ static int lead(const Params &prm, int kh) { return ((kh - prm.ph) * prm.W - kPad) & 3; }

    uint32_t at[kPerThread];         // byte offset of the thread's first float of tuple i within a slot
    int left;                        // tuples of this tile from this thread's first one on

    __device__ __forceinline__ void init(const Params &prm, int origin, int grp, int kq, int limit)
    {
        const int first = origin / kKw, c0 = first / kKw;
        left = min(kTuples, limit / kKw - first) - grp;
#pragma unroll
        for (int i = 0; i < kPerThread; ++i) {
            const int T = first + grp + 16 * i, c = T / kKw, kh = T - c * kKw;
            at[i] = i * 16 < left ? (uint32_t)kh * kBoxBytes + (uint32_t)(c - c0) * kRowBytes + 16u * kq + 4u * (kSpan == 4 ? 0 : lead(prm, kh) & 2) : 0u;
        }
    }
    // the four outputs from pbase on: which of a tuple's values lie inside the image row (bit per value)
    __device__ __forceinline__ static uint32_t inside(const Params &prm, int pbase)
    {
        if (pbase >= prm.P) return 0;                                // past the example's last position (P is a multiple of 4)
        uint32_t bits = 0;
#pragma unroll
        for (int s = 0; s < 4 / kSpan; ++s) {
            const int p = pbase + s * kSpan;
            const int ho = (int)row_of((unsigned)p, prm.wo_magic, prm.wo_shift), wo = p - ho * prm.Wo;
#pragma unroll
            for (int i = 0; i < kSpan + kKw - 1; ++i)
                bits |= ((i >= kPad && i < kSpan + kPad) || (unsigned)(wo + i - kPad) < (unsigned)prm.W ? 1u : 0u) << (s * (kKw + 1) + i);
        }
        return bits;
    }
    // a tuple's floats of the thread's four outputs
    __device__ __forceinline__ static void read(const uint8_t *from, uint32_t bits, float (&v)[kValues])
    {
        constexpr int kFloats = kKw + 3;
        float e[kFloats];
        if (kSpan == 4) {            // lead 2 or 1: the middle vector is aligned
            const float4 m = *reinterpret_cast<const float4 *>(from + 16);
            e[kPad] = m.x; e[kPad + 1] = m.y; e[kPad + 2] = m.z; e[kPad + 3] = m.w;
            if (kKw == 5) {
                const float2 a = *reinterpret_cast<const float2 *>(from + 8), b = *reinterpret_cast<const float2 *>(from + 32);
                e[0] = a.x; e[1] = a.y; e[kFloats - 2] = b.x; e[kFloats - 1] = b.y;
            } else {
                const float4 a = *reinterpret_cast<const float4 *>(from), b = *reinterpret_cast<const float4 *>(from + 32);
                e[0] = a.y; e[1] = a.z; e[2] = a.w; e[kFloats - 3] = b.x; e[kFloats - 2] = b.y; e[kFloats - 1] = b.z;
            }
        } else {                     // lead 1 or 3 (0 or 2 for five taps): pairs from an even place
            constexpr int kOdd = kKw == 5 ? 0 : 1;
#pragma unroll
            for (int i = 0; i < (kFloats + kOdd + 1) / 2; ++i) {
                const float2 a = *reinterpret_cast<const float2 *>(from + 8 * i);
                if (2 * i - kOdd >= 0) e[2 * i - kOdd] = a.x;
                if (2 * i + 1 - kOdd < kFloats) e[2 * i + 1 - kOdd] = a.y;
            }
        }
#pragma unroll
        for (int s = 0; s < 4 / kSpan; ++s)
#pragma unroll
            for (int i = 0; i < kSpan + kKw - 1; ++i) {
                const int to = s * (kKw + 1) + i;
                v[to] = (bits >> to & 1u) ? e[s * kSpan + i] : 0.f;
            }
    }
};

// One interface over both gather forms: the registers of one slice, how they are loaded and where their
// squared, split values go in a K-major swizzled tile.  row0 = t >> 3 and kq = t & 7 of transform thread t.
// kHalf: the slice is shared by 128 threads instead of 256 (two transform groups on alternate slices)
template <int kMode, bool kHalf = false, int kRows = kBM, bool kTaps = IsTaps<kMode>::value>
struct Gatherer {
    struct Regs { float v[kRowsPerThread][4]; };
    GatherRows<kMode> g;
    __device__ __forceinline__ void init(const Params &prm, const float *x, const float *delta, int origin, int row0, int limit)
    {
        g.init(prm, x, delta, origin + row0, limit);
    }
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, Regs &r) const { g.load(prm, z, pbase, r.v); }
    template <bool kSquare>
    __device__ __forceinline__ void store(uint8_t *hi, uint8_t *lo, int row0, int kq, const Regs &r) const
    {
#pragma unroll
        for (int i = 0; i < kRowsPerThread; ++i)
            split_store<kSquare>(hi, lo, chunk_offset(row0 + 32 * i, kq), r.v[i][0], r.v[i][1], r.v[i][2], r.v[i][3]);
    }
};
// A tuple's values, squared and split once, into the tile's rows row .. row + kKw - 1: the taps are views of the same parts.
// kBf: `lo` takes hi and lo as bf16, tiles of 64-byte rows one behind the other; a thread's four k are half of a 16-byte chunk.
template <class Impl, bool kSquare, bool kBf, int kRows, bool kWhole, int kN>
__device__ __forceinline__ void store_tuple(uint8_t *hi, uint8_t *lo, int row0, int kq, const float (&v)[kN], int loaded)
{
    uint32_t h[kN], l[kN];
#pragma unroll
    for (int e = 0; e < kN; ++e) {
        if (e >= loaded) break;
        const float q = kSquare ? __fmul_rn(v[e], v[e]) : v[e];
        h[e] = to_tf32(q);
        l[e] = __float_as_uint(__fsub_rn(q, __uint_as_float(h[e])));
    }
#pragma unroll
    for (int kw = 0; kw < Impl::kKw; ++kw) {
        const int row = row0 + kw;
        if (!kWhole && (unsigned)row >= (unsigned)kRows) continue;
        const uint32_t off = chunk_offset(row, kq);
        *reinterpret_cast<uint4 *>(hi + off) = make_uint4(h[Impl::idx(kw, 0)], h[Impl::idx(kw, 1)], h[Impl::idx(kw, 2)], h[Impl::idx(kw, 3)]);
        if (kBf) {
            auto pair = [&](const uint32_t (&w)[kN], int j) {
                return pack_bf16(__uint_as_float(w[Impl::idx(kw, j)]), __uint_as_float(w[Impl::idx(kw, j + 1)]));
            };
            uint8_t *const at = lo + bf_offset(row, kq);
            *reinterpret_cast<uint2 *>(at) = make_uint2(pair(h, 0), pair(h, 2));
            *reinterpret_cast<uint2 *>(at + kRows * 64) = make_uint2(pair(l, 0), pair(l, 2));
        } else {
            *reinterpret_cast<uint4 *>(lo + off) = make_uint4(l[Impl::idx(kw, 0)], l[Impl::idx(kw, 1)], l[Impl::idx(kw, 2)], l[Impl::idx(kw, 3)]);
        }
    }
}
template <int kMode, bool kHalf, int kRows>
struct Gatherer<kMode, kHalf, kRows, true> {
    // tuples of rows per thread; with 192 rows (16 threads side by side) 64 whole triples, no remainder
    static constexpr int kTriples = kMode == kGatherTaps7S2 ? 2 : kRows == kWideN ? 4 : kHalf ? 3 : 2;
    typedef typename TapsOf<kMode, kTriples>::type Impl;
    // the tile is whole tuples (192 rows of a three-tap kernel, its origin a multiple of 192): no row to test, and a
    // thread's rows are 48 apart, so that their swizzled places differ by constants
    static constexpr bool kWhole = Impl::kKw * Impl::kStride * kTriples == kRows;
    struct Regs { float v[kTriples][Impl::kSlots]; };
    Impl g;
    __device__ __forceinline__ void init(const Params &prm, const float *x, const float *, int origin, int row0, int limit)
    {
        g.init(prm, x, origin, row0, limit);
    }
    __device__ __forceinline__ void load(const Params &prm, int z, int pbase, Regs &r) const { g.load(prm, z, pbase, r.v); }
    template <bool kSquare, bool kBf = false>
    __device__ __forceinline__ void store(uint8_t *hi, uint8_t *lo, int, int kq, const Regs &r) const
    {
#pragma unroll
        for (int i = 0; i < kTriples; ++i) {
            if (!kWhole && (g.row(i) >= kRows || g.row(i) <= -Impl::kKw)) continue;   // no row of this tuple in the tile
            store_tuple<Impl, kSquare, kBf, kRows, kWhole>(hi, lo, g.row(i), kq, r.v[i], Impl::kLoaded);
        }
    }
};

// ---- work distribution -----------------------------------------------------------------------
// One segment of a block's range: slices [s_begin, s_end) of the reduction of one output tile.
struct Seg {
    int layer, m0, n0;       // layer of the batch, first row / column of the tile
    int n_valid, n_act;      // columns of the tile that exist; the MMAs' N (rounded up to a multiple of 16)
    int s_begin, s_end;
    bool whole;              // the segment is the tile's whole reduction: its block writes the result itself
    int slot;                // otherwise: which partial tile of the scratch it writes
};

// The launch's work is the sequence (layer, tile, unit of the tile's reduction), units_total long; block b owns
// units [b U / G, (b + 1) U / G).  Every role of a block walks the same segments with an iterator of its own.
template <bool kPerExample>
struct SegIter {
    int pos, end;
    int index;
    __device__ __forceinline__ SegIter(const Params &prm)
    {
        const int b = (int)blockIdx.x;
        pos = b * prm.units_q + min(b, prm.units_r);
        end = pos + prm.units_q + (b < prm.units_r ? 1 : 0);
        index = 0;
    }
    __device__ __forceinline__ bool next(const Params &prm, Seg &sg)
    {
        if (pos >= end) return false;
        const int upt = prm.units_per_tile;
        const int tile = pos / upt;
        const int u0 = pos - tile * upt;
        const int u1 = min(end - tile * upt, upt);
        const int tiles_layer = prm.tiles_x * prm.tiles_y;
        const bool cut = kPerExample && prm.parts > 0;
        sg.layer = tile / tiles_layer;
        const int rem = tile - sg.layer * tiles_layer;
        const int tile_m = rem / prm.tiles_x, tile_n = rem - tile_m * prm.tiles_x;
        sg.m0 = tile_m * kBM;
        sg.n0 = tile_n * prm.tile_n;
        sg.n_valid = min(prm.tile_n, prm.N - sg.n0);
        sg.n_act = (sg.n_valid + 15) & ~15;
        if (cut) {                                               // one part of one example
            const int z = u0 / prm.parts, part = u0 - z * prm.parts;
            sg.s_begin = z * prm.p_slices + part * prm.part_slices;
            sg.s_end = min(sg.s_begin + prm.part_slices, (z + 1) * prm.p_slices);
        } else {
            sg.s_begin = u0 * prm.unit;
            sg.s_end = u1 * prm.unit;
        }
        sg.whole = !cut && u0 == 0 && u1 == upt;
        // a block's partial segments: its first and / or its last; with parts of examples its only one
        sg.slot = cut ? (int)blockIdx.x : 2 * (int)blockIdx.x + (index > 0 ? 1 : 0);
        pos += u1 - u0;
        ++index;
        return true;
    }
};

// ---- the kernel ------------------------------------------------------------------------------
// kExact: the per-example statistic of a conv layer, S = scale * sum_z (sum_p delta x)^2 -- operands are split without
// squaring, an accumulator is drained at least at every example's end, the epilogue sums the drains of one example
// in registers and adds the square of that sum into a third accumulator kept in tensor memory.
// kBf: the two cross terms hi*lo and lo*hi are taken with bf16 operands (half the shared-memory reads and half the
// tensor-pipe time of a tf32 product each; their rounding, 2^-9 relative on a term that is itself 2^-11 of the
// product, stays below 2^-18 of the result).  A lo slot then holds [B hi as bf16][B lo as bf16], 8 KB each with
// 64-byte rows, and an A slot in tensor memory [hi tf32: 32 columns][hi bf16: 16][lo bf16: 16].
// The wide form's B tile is split as it is gathered: a thread's four k are 16 bytes of the tf32 tile and 8 of each bf16 tile
// (12 KB each, in the same lo slot); five conversions of pairs serve three taps.  Twelve instructions a slice were what the
// tensor pipe and the power cap allowed (1290 cycles a slice at 1.6 GHz); with eight, 128 channels 28 x 28, batch 32, take
// 41.6 -> 38.6 us a call, the ResNet-50 pass 1920 -> 1871.
// kN: columns of a tile, 128 or (wide form) 192.  The wide per-example form keeps the sum of squares in the epilogue's
// registers: it takes layers whose examples fit one accumulator run (at most kChunk slices).
// Where examples are cut into parts (Params::parts), kExact writes a part's plain sums and a kernel of its own adds an example's
// parts up, squares and adds.
template <int kMajor, int kModeA, int kModeB, bool kATmem, bool kExact = false, bool kBf = false, int kN = kBN>
__global__ void __launch_bounds__(kThreadsTc, 1)
sqgrad_tc(const __grid_constant__ Batch bt, const Params prm)
{
    static_assert(kMajor == kMajorK || (kModeA == kTma && kModeB == kTma), "gathered tiles are K-major");
    static_assert(!kATmem || (kMajor == kMajorK && kModeA == kTma), "A goes to tensor memory from a K-major TMA tile");
    constexpr bool kGatherA = kModeA != kTma, kGatherB = kModeB != kTma;
    constexpr bool kAnyTma = !kGatherA || !kGatherB;
    constexpr bool kAnyGather = kGatherA || kGatherB;
    constexpr bool kWide = kN != kBN;
    constexpr bool kHalo = IsHalo<kModeB>::value;
    typedef Halo<kHalo ? kModeB : (int)kHalo5x4> HaloB;
    static_assert(!kWide || (kN == kWideN && kATmem && (IsTaps<kModeB>::value || kHalo)), "wide tiles: several taps at a time");
    static_assert(!kHalo || kWide, "input rows by TMA: wide tiles");
    constexpr bool kSplit = kATmem && (!kAnyGather || kWide);              // A raw tiles in a ring of their own
    static_assert(!kBf || (kSplit && !kExact), "bf16 cross terms: A in tensor memory, sums of squares");
    constexpr bool kTmaB = kSplit && !kGatherB;                            // split form: the B tile comes by TMA, too
    constexpr int kNA = kWide ? kWideA : kSplitA;                                           // slots of the raw A ring (split form)
    // the transform warps work as two groups of four on alternate slices (else all eight on every slice)
    constexpr bool kTwoGroups = !kAnyGather || ((IsTaps<kModeB>::value || kHalo) && kModeA == kTma);
    constexpr int kWideNB = kHalo ? kHaloB : kWideB;
    constexpr int kNB = kWide ? kWideNB : kSplit ? kSplitB : kRawSlots;     // slots of the raw / hi ring
    // lo slots (and A slots in TMEM); the per-example form needs 128 TMEM columns for its sum of squares
    constexpr int kLoN = kWide ? kWideNB : (kExact && kATmem) ? 2 : kSplit ? kSplitLo : (kATmem ? kLoSlotsAT : kLoSlots);
    constexpr int kAN = kWide ? kWideTmemA : kLoN;                         // A slots in tensor memory
    constexpr uint32_t kBBytes = kN * kBK * 4;                             // bytes of a B tile
    constexpr uint32_t kSqCol = 2 * kBN + (kATmem ? 2 * kTmemColsA : 0);         // where that sum lives
    constexpr uint32_t kLoBytes = kATmem ? kRawBytesB : kRawStageBytes;  // bytes of one lo slot
    // byte offsets of slot s: the [A][B] pair of the raw / hi ring (split form: only its B half exists, the
    // offset points one A tile below it), the lo ring likewise, and the split form's A ring
    auto pair_off = [](int s) -> uint32_t { return kWide ? kWideA * kRawBytesA + (uint32_t)s * kBBytes - kRawBytesA : kSplit ? (uint32_t)(kSplitA + s - 1) * kRawBytesA : (uint32_t)s * kRawStageBytes; };
    auto lo_off = [](int s) -> uint32_t {
        return kWide ? kWideA * kRawBytesA + (uint32_t)(kWideNB + s) * kBBytes - kRawBytesA
               : kSplit ? (uint32_t)(kSplitA + kSplitB + s - 1) * kRawBytesA
                      : kLoBase + (uint32_t)s * kLoBytes - (kATmem ? kRawBytesA : 0u);
    };
    // bf16-cross form: where the B tile of raw slot s and the [hi bf16][lo bf16] tiles of lo slot s live
    auto b_tile = [&](int s) -> uint32_t { return pair_off(s) + kRawBytesA; };
    auto bf_tile = [&](int s) -> uint32_t { return lo_off(s) + kRawBytesA; };

    extern __shared__ uint8_t smem_raw_[];
    __shared__ __align__(8) uint64_t bars[3 * kSplitB + 5 + 2 * kSplitA];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile uint32_t abort_flag;

    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = (smem_u32(smem_raw_) + 1023u) & ~1023u;     // 1024-byte aligned tiles
    uint8_t *smem_gen = smem_raw_ + (smem_base - smem_u32(smem_raw_));

    // per raw slot: raw_full (TMA landed) -> op_full (hi/lo written) -> empty (MMAs that read it retired);
    // a lo slot (and its A slot in tensor memory) is free when the MMAs of the slice that used it last have
    // retired, which is what that slice's `empty` barrier says: no barrier of its own, one commit per slice
    uint64_t *raw_full = bars, *op_full = bars + kNB, *empty = bars + 2 * kNB;
    uint64_t *acc_full = bars + 3 * kNB, *acc_empty = acc_full + 2, *drain = acc_empty + 2;
    uint64_t *a_full = drain + 1, *a_empty = a_full + kNA;                 // split form: the A ring
    uint64_t *h_full = a_empty + kNA, *h_empty = h_full + kHaloSlots;      // input rows by TMA: their ring
    static_assert(!kHalo || (3 * kNB + 5 + 2 * kNA + 2 * kHaloSlots <= 3 * kSplitB + 5 + 2 * kSplitA && HaloB::kSlotBytes <= kHaloSlotMost), "barriers, slots");

    grid_release();
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < kNB; ++i) {
            mbar_init(smem_u32(&raw_full[i]), 1);
            mbar_init(smem_u32(&op_full[i]), kTwoGroups ? 4 : kGatherThreads / 32);
            mbar_init(smem_u32(&empty[i]), 1);
        }
        if (kSplit)
            for (int i = 0; i < kNA; ++i) {
                mbar_init(smem_u32(&a_full[i]), 1);
                mbar_init(smem_u32(&a_empty[i]), 4);
            }
        if (kHalo)
            for (int i = 0; i < kHaloSlots; ++i) {
                mbar_init(smem_u32(&h_full[i]), 1);
                mbar_init(smem_u32(&h_empty[i]), 4);
            }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&acc_full[i]), 1); mbar_init(smem_u32(&acc_empty[i]), kEpilogueWarps); }
        mbar_init(smem_u32(drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {      // TMEM: this warp allocates and, at the end, frees
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;

    // Every role works its first segment out (divisions, cold instructions: 2 us) before it waits for the work ahead, as it
    // does with all else that follows from the parameters alone.
    // `it` below is the running number of a slice within this block (over all of its segments): ring slots and
    // barrier phases follow it, so the pipeline does not drain between segments.
    if (warp < kFirstTransform) regs_dec<kRegsFew>();
    if (warp == 0) {
        // ================= TMA producer (one thread) =================
        if (lane == 0 && kAnyTma) {
            SegIter<kExact> iter(prm);
            Seg sg;
            bool more = iter.next(prm, sg);
            if (!kGatherA) prefetch_map(&bt.a[sg.layer]);
            if (!kGatherB) prefetch_map(&bt.b[sg.layer]);
            grid_wait();
            int it = 0;
            bool ok = true;
            for (; ok && more; more = iter.next(prm, sg)) {
                const CUtensorMap *map_a = &bt.a[sg.layer], *map_b = &bt.b[sg.layer];
                const int m0 = sg.m0, n0 = sg.n0;
                for (int slice = sg.s_begin; slice < sg.s_end; ++slice, ++it) {
                    const int st = it % kNB;
                    const uint32_t ph = (uint32_t)(it / kNB) & 1u;
                    if (!(kSplit && !kTmaB) && !mbar_wait(smem_u32(&empty[st]), ph ^ 1u, &abort_flag, 64)) { ok = false; break; }
                    const uint32_t full = smem_u32(&raw_full[st]);
                    const uint32_t dst_a = smem_base + pair_off(st), dst_b = dst_a + kRawBytesA;
                    if (kSplit) {
                        const int sa = it % kNA;
                        if (!mbar_wait(smem_u32(&a_empty[sa]), ((uint32_t)(it / kNA) & 1u) ^ 1u, &abort_flag, 64)) { ok = false; break; }
                        const uint32_t full_a = smem_u32(&a_full[sa]);
                        const int z = slice / prm.p_slices, p0 = (slice - z * prm.p_slices) * kBK;
                        mbar_expect_tx(full_a, prm.tx_bytes_a);
                        tma_load_3d(smem_base + (uint32_t)sa * kRawBytesA, map_a, full_a, p0, m0, z);
                        if (!kTmaB) continue;
                        mbar_expect_tx(full, prm.tx_bytes - prm.tx_bytes_a);
                        if (kBf) tma_load_3d(smem_base + b_tile(st), map_b, full, p0, n0, z);
                        else tma_load_3d(dst_b, map_b, full, p0, n0, z);
                        continue;
                    }
                    mbar_expect_tx(full, prm.tx_bytes);
                    if (kMajor == kMajorK) {
                        const int z = slice / prm.p_slices, p0 = (slice - z * prm.p_slices) * kBK;
                        if (!kGatherA) tma_load_3d(dst_a, map_a, full, p0, m0, z);
                        if (!kGatherB) tma_load_3d(dst_b, map_b, full, p0, n0, z);
                    } else {
                        const int k0 = slice * kBK;
#pragma unroll
                        for (int j = 0; j < kBM / 32; ++j) tma_load_2d(dst_a + j * 4096, map_a, full, m0 + 32 * j, k0);
#pragma unroll
                        for (int j = 0; j < kBN / 32; ++j) tma_load_2d(dst_b + j * 4096, map_b, full, n0 + 32 * j, k0);
                    }
                }
            }
            // on an abort: loads already issued (slices 0 .. it-1) must land before the block may exit
            if (abort_flag) {
                const int issued = it;
                const int first = kSplit && !kTmaB ? issued : issued > kNB ? issued - kNB : 0;
                for (int i = first; i < issued; ++i) {
                    const uint32_t bar = smem_u32(&raw_full[i % kNB]);
                    const uint32_t ph = (uint32_t)(i / kNB) & 1u;
                    for (uint32_t t = 0; t < kWaitLimit && !mbar_try(bar, ph); ++t) {}
                }
                if (kSplit) {
                    const int first_a = issued > kNA ? issued - kNA : 0;
                    for (int i = first_a; i < issued; ++i) {
                        const uint32_t bar = smem_u32(&a_full[i % kNA]);
                        const uint32_t ph = (uint32_t)(i / kNA) & 1u;
                        for (uint32_t t = 0; t < kWaitLimit && !mbar_try(bar, ph); ++t) {}
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (one thread) =================
        if (lane == 0) {
            // K-major: rows of 128 B, 8-row groups 1024 B apart (SBO); LBO unused.
            // MN-major: 32-wide column blocks 4096 B apart (LBO); 4-deep k groups 512 B apart (SBO).
            const uint32_t lbo = kMajor == kMajorK ? 16u : 4096u;
            const uint32_t sbo = kMajor == kMajorK ? 1024u : 512u;
            const uint32_t layout = kMajor == kMajorK ? 2u : 1u;
            constexpr uint32_t k_step16 = (kMajor == kMajorK ? 32u : 1024u) >> 4;   // 16-byte units per 8-deep MMA step
            // This one thread feeds the tensor pipe, so its instruction stream is kept short: the descriptor's
            // upper word and the LBO field never change, the start-address field (address >> 4; shared memory
            // is < 256 KB, so it cannot overflow its 14 bits) is one addition per operand and step.
            const uint32_t desc_hi = (uint32_t)(smem_desc(0, lbo, sbo, layout) >> 32);
            const uint32_t desc_lo0 = (uint32_t)smem_desc(0, lbo, sbo, layout);
            auto desc_at = [&](uint32_t lo16) -> uint64_t { return ((uint64_t)desc_hi << 32) | (desc_lo0 + lo16); };
            // bf16 tiles: K-major rows of 64 B with the 64-byte swizzle (mode 4), 8-row groups 512 B apart
            const uint32_t desc_bf_hi = (uint32_t)(smem_desc(0, 16u, 512u, 4u) >> 32);
            const uint32_t desc_bf_lo0 = (uint32_t)smem_desc(0, 16u, 512u, 4u);
            auto desc_bf = [&](uint32_t lo16) -> uint64_t { return ((uint64_t)desc_bf_hi << 32) | (desc_bf_lo0 + lo16); };
            int st = 0, ls = 0, as = 0;                  // the current slice's raw / hi slot, lo slot and A slot
            uint32_t st_phase = 0;
            int c = 0;                                   // running number of the chunk (accumulator buffer c & 1)
            bool ok = true;
            SegIter<kExact> iter(prm);
            Seg sg;
            bool more = iter.next(prm, sg);
            for (; ok && more; more = iter.next(prm, sg)) {
                const uint32_t idesc = instr_desc(kMajor, sg.n_act, kBM);
                const uint32_t idesc_bf = instr_desc_bf16(sg.n_act, kBM);
                // an accumulator is drained every prm.chunk slices, and (kExact) at the end of every example: the
                // segment's slices are runs of seg_len slices (whole examples -- the work is cut that way), each cut
                // into cps chunks
                const int n_slices = sg.s_end - sg.s_begin;
                const int seg_len = kExact && prm.parts == 0 ? prm.p_slices : n_slices;
                const int cps = (seg_len + prm.chunk - 1) / prm.chunk;
                const int n_chunks = (n_slices / seg_len) * cps;
                int i = 0;                               // slice within the segment
                for (int cc = 0; cc < n_chunks && ok; ++cc, ++c) {
                    const int b = c & 1;
                    ok = mbar_wait(smem_u32(&acc_empty[b]), ((uint32_t)(c >> 1) & 1u) ^ 1u, &abort_flag, 0);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)b * kN;
                    const int run = cc / cps, cq = cc - run * cps;              // run (example) and chunk inside it
                    const int chunk_end = run * seg_len + min(seg_len, (cq + 1) * prm.chunk);
                    for (bool first = true; i < chunk_end; ++i) {
                        ok = mbar_wait(smem_u32(&op_full[st]), st_phase, &abort_flag, 0);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t hi_a16 = (smem_base + pair_off(st)) >> 4, hi_b16 = hi_a16 + (kRawBytesA >> 4);
                        const uint32_t lo_a16 = (smem_base + lo_off(ls)) >> 4, lo_b16 = lo_a16 + (kRawBytesA >> 4);   // lo_a unused with A in TMEM
                        const uint32_t ta_hi = tmem_base + 2 * kN + as * kTmemColsA, ta_lo = ta_hi + 32;
                        if (kBf) {
                            const uint32_t b16 = (smem_base + b_tile(st)) >> 4;
#pragma unroll
                            for (int kk = 0; kk < kBK / 8; ++kk) {
                                const uint64_t db_hi = desc_at(b16 + kk * k_step16);
                                if (kk == 0) tc_mma_tf32_ts(d_tmem, ta_hi, db_hi, idesc, first ? 0u : 1u);
                                else tc_mma_tf32_ts_acc(d_tmem, ta_hi + kk * 8, db_hi, idesc);
                            }
                            // cross terms, 16 k (32 bytes of a 64-byte row, 8 columns of tensor memory) per instruction
                            const uint32_t bf_hi16 = (smem_base + bf_tile(ls)) >> 4, bf_lo16 = bf_hi16 + (kBBytes >> 5);
#pragma unroll
                            for (int kk = 0; kk < kBK / 16; ++kk) {
                                tc_mma_bf16_ts_acc(d_tmem, ta_hi + 32 + kk * 8, desc_bf(bf_lo16 + kk * 2), idesc_bf);
                                tc_mma_bf16_ts_acc(d_tmem, ta_hi + 48 + kk * 8, desc_bf(bf_hi16 + kk * 2), idesc_bf);
                            }
                        } else
#pragma unroll
                        for (int kk = 0; kk < kBK / 8; ++kk) {
                            const uint64_t db_hi = desc_at(hi_b16 + kk * k_step16);
                            const uint64_t db_lo = desc_at(lo_b16 + kk * k_step16);
                            if (kATmem) {
                                if (kk == 0) tc_mma_tf32_ts(d_tmem, ta_hi, db_hi, idesc, first ? 0u : 1u);
                                else tc_mma_tf32_ts_acc(d_tmem, ta_hi + kk * 8, db_hi, idesc);
                                tc_mma_tf32_ts_acc(d_tmem, ta_hi + kk * 8, db_lo, idesc);
                                tc_mma_tf32_ts_acc(d_tmem, ta_lo + kk * 8, db_hi, idesc);
                            } else {
                                const uint64_t da_hi = desc_at(hi_a16 + kk * k_step16);
                                const uint64_t da_lo = desc_at(lo_a16 + kk * k_step16);
                                if (kk == 0) tc_mma_tf32(d_tmem, da_hi, db_hi, idesc, first ? 0u : 1u);
                                else tc_mma_tf32_acc(d_tmem, da_hi, db_hi, idesc);
                                tc_mma_tf32_acc(d_tmem, da_hi, db_lo, idesc);
                                tc_mma_tf32_acc(d_tmem, da_lo, db_hi, idesc);
                            }
                        }
                        first = false;
                        tc_commit(smem_u32(&empty[st]));              // raw, lo and TMEM-A slots are free once these MMAs retire
                        if (++st == kNB) { st = 0; st_phase ^= 1u; }
                        if (++ls == kLoN) ls = 0;
                        if (++as == kAN) as = 0;
                    }
                    if (ok) tc_commit(smem_u32(&acc_full[b]));
                }
            }
            if (!ok) {      // abort: MMAs already issued must retire before TMEM is freed
                tc_commit(smem_u32(drain));
                for (uint32_t t = 0; t < kWaitLimit && !mbar_try(smem_u32(drain), 0); ++t) {}
            }
        }
    } else if (warp == 2 && kHalo) {
        // ================= producer of the input rows (one thread), ahead of the A tiles, whose ring is shorter =================
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            SegIter<kExact> iter(prm);
            Seg sg;
            bool more = iter.next(prm, sg);
            prefetch_map(&bt.b[sg.layer]);
            grid_wait();
            for (; ok && more; more = iter.next(prm, sg)) {
                const CUtensorMap *map = &bt.b[sg.layer];
                const int c0 = sg.n0 / (HaloB::kKw * HaloB::kKw);
                int z = sg.s_begin / prm.p_slices, p0 = (sg.s_begin - z * prm.p_slices) * kBK;
                for (int slice = sg.s_begin; slice < sg.s_end; ++slice, ++it) {
                    const int sh = it % kHaloSlots;
                    if (!mbar_wait(smem_u32(&h_empty[sh]), ((uint32_t)(it / kHaloSlots) & 1u) ^ 1u, &abort_flag, 64)) { ok = false; break; }
                    const uint32_t full = smem_u32(&h_full[sh]), dst = smem_base + kHaloBase + (uint32_t)sh * HaloB::kSlotBytes;
                    mbar_expect_tx(full, prm.tx_bytes - prm.tx_bytes_a);
#pragma unroll
                    for (int kh = 0; kh < HaloB::kKw; ++kh)        // (a start below zero rounds down, too)
                        tma_load_3d(dst + kh * HaloB::kBoxBytes, map, full, (p0 + (kh - prm.ph) * prm.W - HaloB::kPad) & ~3, c0, z);
                    p0 += kBK;
                    if (p0 >= prm.p_slices * kBK) { p0 = 0; ++z; }
                }
            }
            if (abort_flag)                              // loads already issued must land before the block may exit
                for (int i = it > kHaloSlots ? it - kHaloSlots : 0; i < it; ++i)
                    for (uint32_t t = 0; t < kWaitLimit && !mbar_try(smem_u32(&h_full[i % kHaloSlots]), (uint32_t)(i / kHaloSlots) & 1u); ++t) {}
        }
    } else if (warp < kFirstTransform) {
        // nothing: the rest of the first warpgroup
    } else if (warp < kFirstEpilogue) {
        // ================= transform warps: square and split into TF32 hi / lo =================
        regs_dec<kWide ? kRegsTransformWide : kRegsTransform>();
        const int t = (int)threadIdx.x - 32 * kFirstTransform;                               // 0 .. 128 * kGroups - 1
        // With nothing to gather the warps work as groups of four that take consecutive slices in turn: the waits,
        // fences and tensor-memory stores of one slice then overlap the arithmetic of the others.  The same split
        // is used when the B tile is gathered several taps at a time next to a TMA-fed A tile.  The element-wise
        // gathers share every slice among the first eight warps; further warps have nothing to do there.
        constexpr int kTT = kTwoGroups ? 128 : kGatherThreads;             // threads sharing a slice
        const int group = kTwoGroups ? (t >> 7) : 0;
        const int tt = kTwoGroups ? (t & 127) : t;
        const int kq = tt & 7, row0 = tt >> 3;                             // gathered chunks: rows row0 + 32*i, k = 4*kq..4*kq+3
        typedef Gatherer<kModeA, kTwoGroups> GatherA;
        typedef Gatherer<kHalo ? (int)kTma : kModeB, kTwoGroups, kN> GatherB;
        HaloB halo;
        GatherA rows_a;
        GatherB rows_b;
        typedef typename GatherA::Regs RegsA;
        typedef typename GatherB::Regs RegsB;
        // where the current slice sits: example z, 32-wide block pblk of that example's output positions
        int z = 0, pblk = 0;
        auto advance = [&]() {
            if (++pblk == prm.p_slices) { pblk = 0; ++z; }
        };
        auto gather = [&](RegsA &ga, RegsB &gb) {
            const int pbase = pblk * kBK + kq * 4;
            rows_a.load(prm, z, pbase, ga);
            if (!kHalo) rows_b.load(prm, z, pbase, gb);
        };
        // transform of the block's slice number i; gathered elements come in registers, TMA tiles from the raw stage
        // (`gathered`: called once the registers have been read)
        auto process = [&](int i, const RegsA &ga, const RegsB &gb, auto gathered) -> bool {
            const int st = i % kNB, ls = i % kLoN;
            const uint32_t ph = (uint32_t)(i / kNB) & 1u;
            const int sa = kSplit ? i % kNA : 0;
            if (kSplit && !kWide && !mbar_wait(smem_u32(&a_full[sa]), (uint32_t)(i / kNA) & 1u, &abort_flag)) return false;
            // a raw slot is ours once its TMA tiles landed (the producer waited for it to be empty), or, with
            // nothing coming by TMA, once the MMAs that last read it retired; likewise the lo slot
            if (kAnyTma && !kWide ? !mbar_wait(smem_u32(&raw_full[st]), ph, &abort_flag)
                                  : !mbar_wait(smem_u32(&empty[st]), ph ^ 1u, &abort_flag))
                return false;
            if (!kWide && i >= kLoN) {      // the lo slot's previous user: slice i - kLoN (wide: B and lo slots go together)
                const int j = i - kLoN;
                if (!mbar_wait(smem_u32(&empty[j % kNB]), (uint32_t)(j / kNB) & 1u, &abort_flag)) return false;
            }
            uint8_t *hi = smem_gen + pair_off(st);               // raw tiles live here and become the hi tiles
            // lo tiles: [A lo][B lo], or the B tile alone when A lives in tensor memory (then `lo` points
            // one A tile below the slot so that the same chunk offsets address the B part)
            uint8_t *lo = smem_gen + lo_off(ls);
            if constexpr (kWide) {
                // the B tile first: only two A slots in tensor memory, so the A tile waits for slice i - 2 to retire
                if constexpr (kHalo) {
                    const uint32_t bits = HaloB::inside(prm, pblk * kBK + kq * 4);
                    const int sh = i % kHaloSlots;
                    if (!mbar_wait(smem_u32(&h_full[sh]), (uint32_t)(i / kHaloSlots) & 1u, &abort_flag)) return false;
                    const uint8_t *const from = smem_gen + kHaloBase + (uint32_t)sh * HaloB::kSlotBytes;
#pragma unroll
                    for (int u = 0; u < HaloB::kPerThread; ++u) {
                        if (16 * u >= halo.left) break;
                        float v[HaloB::kValues];
                        HaloB::read(from + halo.at[u], bits, v);
                        store_tuple<HaloB, !kExact, kBf, kN, true>(hi + kRawBytesA, lo + kRawBytesA, HaloB::kKw * (row0 + 16 * u), kq, v, HaloB::kValues);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&h_empty[sh]));
                } else {
                    rows_b.template store<!kExact, kBf>(hi + kRawBytesA, lo + kRawBytesA, row0, kq, gb);
                }
                gathered();
                if (!mbar_wait(smem_u32(&a_full[sa]), (uint32_t)(i / kNA) & 1u, &abort_flag)) return false;
                if (i >= kAN) {
                    const int j = i - kAN;
                    if (!mbar_wait(smem_u32(&empty[j % kNB]), (uint32_t)(j / kNB) & 1u, &abort_flag)) return false;
                }
            }
            if (kATmem) {
                // A: this thread's row (TMEM lane) and 16 of the slice's 32 k at a time -> hi / lo straight into
                // TMEM (a warp of the two-group form takes both halves, otherwise its group number picks one)
                tc_fence_after();
                const uint32_t q = warp & 3;
                const int m_local = (int)(q * 32 + lane);
                const uint8_t *arow = (kSplit ? smem_gen + (uint32_t)sa * kRawBytesA : hi) + m_local * 128;
                if (kWide) {         // 8 k at a time: the next slice's gathered values are held in registers meanwhile
                    const uint32_t taddr = tmem_base + ((q * 32u) << 16) + 2 * kN + (i % kAN) * kTmemColsA;
#pragma unroll
                    for (int k8 = 0; k8 < kBK / 8; ++k8) {
                        uint32_t h8[8], l8[8];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float4 c = *reinterpret_cast<const float4 *>(arow + (((2 * k8 + u) ^ (m_local & 7)) << 4));
                            const float e[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float sq = kExact ? e[j] : __fmul_rn(e[j], e[j]);
                                h8[4 * u + j] = to_tf32(sq);
                                l8[4 * u + j] = __float_as_uint(__fsub_rn(sq, __uint_as_float(h8[4 * u + j])));
                            }
                        }
                        tc_st_32x8(taddr + 8 * k8, h8);
                        if (kBf) {
                            uint32_t hb[4], lb[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                hb[j] = pack_bf16(__uint_as_float(h8[2 * j]), __uint_as_float(h8[2 * j + 1]));
                                lb[j] = pack_bf16(__uint_as_float(l8[2 * j]), __uint_as_float(l8[2 * j + 1]));
                            }
                            tc_st_32x4(taddr + 32 + 4 * k8, hb);
                            tc_st_32x4(taddr + 48 + 4 * k8, lb);
                        } else
                        tc_st_32x8(taddr + 32 + 8 * k8, l8);
                    }
                } else
#pragma unroll
                for (int hh = 0; hh < (kTwoGroups ? 2 : 1); ++hh) {
                    const uint32_t h = kTwoGroups ? (uint32_t)hh : (warp - kFirstTransform) >> 2;
                    float4 c4[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        c4[u] = *reinterpret_cast<const float4 *>(arow + (((4 * h + u) ^ (m_local & 7)) << 4));
                    uint32_t h16[16], l16[16];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float e[4] = {c4[u].x, c4[u].y, c4[u].z, c4[u].w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float sq = kExact ? e[j] : __fmul_rn(e[j], e[j]);
                            h16[4 * u + j] = to_tf32(sq);
                            l16[4 * u + j] = __float_as_uint(__fsub_rn(sq, __uint_as_float(h16[4 * u + j])));
                        }
                    }
                    const uint32_t taddr = tmem_base + ((q * 32u) << 16) + 2 * kN + (i % kAN) * kTmemColsA + 16 * h;
                    tc_st_32x16(taddr, h16);
                    if (kBf) {
                        uint32_t hb[8], lb[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            hb[j] = pack_bf16(__uint_as_float(h16[2 * j]), __uint_as_float(h16[2 * j + 1]));
                            lb[j] = pack_bf16(__uint_as_float(l16[2 * j]), __uint_as_float(l16[2 * j + 1]));
                        }
                        const uint32_t tb = taddr - 16 * h + 32 + 8 * h;
                        tc_st_32x8(tb, hb);
                        tc_st_32x8(tb + 16, lb);
                    } else
                    tc_st_32x16(taddr + 32, l16);
                }
                if (kSplit) {                     // the raw A tile has been read: its slot may be refilled
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&a_empty[sa]));
                }
            }
            if (kBf && !kWide) {
                // B tile: a thread takes pairs of adjacent 16-byte chunks (8 consecutive k of one row: the 128-byte
                // swizzle permutes the two chunks of a pair only among themselves).  hi goes back in place as tf32;
                // hi and lo as bf16 make one 16-byte chunk each, and under the 64-byte swizzle that chunk's place in
                // its tile is the pair's place in the raw tile.  Half of each quarter-warp reads the second chunk of
                // its pair first, which keeps the 16-byte accesses free of bank conflicts.
                uint8_t *braw = smem_gen + b_tile(st), *bf_hi = smem_gen + bf_tile(ls), *bf_lo = bf_hi + kBBytes / 2;
                const uint32_t s1 = (lane >> 2) & 1u;
#pragma unroll
                for (int u = 0; u < (int)(kBBytes / 32) / kTT; ++u) {
                    const uint32_t p = (uint32_t)tt + (uint32_t)u * kTT;          // pair index = 4 * row + pair of the row
                    const uint32_t offx = 32 * p + 16 * s1, offy = 32 * p + 16 * (s1 ^ 1u);
                    const float4 x4 = *reinterpret_cast<const float4 *>(braw + offx);
                    const float4 y4 = *reinterpret_cast<const float4 *>(braw + offy);
                    const float ex[8] = {x4.x, x4.y, x4.z, x4.w, y4.x, y4.y, y4.z, y4.w};
                    uint32_t h[8];
                    float l[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float sq = __fmul_rn(ex[j], ex[j]);
                        h[j] = to_tf32(sq);
                        l[j] = __fsub_rn(sq, __uint_as_float(h[j]));
                    }
                    *reinterpret_cast<uint4 *>(braw + offx) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4 *>(braw + offy) = make_uint4(h[4], h[5], h[6], h[7]);
                    const uint32_t hx0 = pack_bf16(__uint_as_float(h[0]), __uint_as_float(h[1]));
                    const uint32_t hx1 = pack_bf16(__uint_as_float(h[2]), __uint_as_float(h[3]));
                    const uint32_t hy0 = pack_bf16(__uint_as_float(h[4]), __uint_as_float(h[5]));
                    const uint32_t hy1 = pack_bf16(__uint_as_float(h[6]), __uint_as_float(h[7]));
                    const uint32_t lx0 = pack_bf16(l[0], l[1]), lx1 = pack_bf16(l[2], l[3]);
                    const uint32_t ly0 = pack_bf16(l[4], l[5]), ly1 = pack_bf16(l[6], l[7]);
                    // the chunk read first holds the lower k iff its place in the pair equals the row's parity
                    const bool x_first = s1 == ((p >> 2) & 1u);
                    *reinterpret_cast<uint4 *>(bf_hi + 16 * p) =
                        x_first ? make_uint4(hx0, hx1, hy0, hy1) : make_uint4(hy0, hy1, hx0, hx1);
                    *reinterpret_cast<uint4 *>(bf_lo + 16 * p) =
                        x_first ? make_uint4(lx0, lx1, ly0, ly1) : make_uint4(ly0, ly1, lx0, lx1);
                }
            } else
            if (kAnyTma && !kWide) {      // tiles that came by TMA: elementwise, in place, over their 16-byte chunks
                constexpr uint32_t c_begin = (kGatherA || kATmem) ? kRawBytesA / 16 : 0;
                constexpr uint32_t c_end = kGatherB ? kRawBytesA / 16 : kRawStageBytes / 16;
                constexpr int kPerThread = c_end > c_begin ? (c_end - c_begin) / kTT : 1;
                constexpr int kBatch = kPerThread < 4 ? kPerThread : 4;              // chunks in registers at a time
                if (c_end > c_begin) {
#pragma unroll
                    for (int u0 = 0; u0 < kPerThread; u0 += kBatch) {
                        float4 v[kBatch];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u)
                            v[u] = *reinterpret_cast<const float4 *>(hi + 16 * (c_begin + (uint32_t)tt + (u0 + u) * kTT));
#pragma unroll
                        for (int u = 0; u < kBatch; ++u)
                            split_store<!kExact>(hi, lo, 16 * (c_begin + (uint32_t)tt + (u0 + u) * kTT), v[u].x, v[u].y, v[u].z, v[u].w);
                    }
                }
            }
            if (kGatherA) rows_a.template store<!kExact>(hi, lo, row0, kq, ga);
            if (kGatherB && !kWide) rows_b.template store<!kExact>(hi + kRawBytesA, lo + kRawBytesA, row0, kq, gb);
            if (kATmem) { tc_wait_st(); tc_fence_before(); }      // TMEM stores complete and ordered before the signal
            fence_async_smem();                                   // generic-proxy writes -> tensor core reads
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&op_full[st]));
            return true;
        };

        RegsA a0, a1;
        RegsB b0, b1;
        int it0 = 0;                                 // block-wide number of the segment's first slice
        bool ok = true;
        if (!kTwoGroups && t >= kGatherThreads) ok = false;
        SegIter<kExact> iter(prm);
        Seg sg;
        bool more = iter.next(prm, sg);
        for (; ok && more; more = iter.next(prm, sg)) {
            const int n_slices = sg.s_end - sg.s_begin;
            if (kAnyGather) {
                rows_a.init(prm, bt.x[sg.layer], bt.delta[sg.layer], sg.m0, row0, prm.M);
                if (kHalo) halo.init(prm, sg.n0, row0, kq, prm.N);
                else rows_b.init(prm, bt.x[sg.layer], bt.delta[sg.layer], sg.n0, row0, prm.N);
                z = sg.s_begin / prm.p_slices;
                pblk = sg.s_begin - z * prm.p_slices;
            }
            grid_wait();                             // (returns at once from the second segment on)
            if (kTwoGroups) {
                // this group's slices: those whose block-wide number is the group's modulo kGroups.  With a gathered
                // tile: one register set per thread -- the other groups' work covers this group's load latency
                // (measured faster than two sets in turn)
                const int i_first = (group - it0 % kGroups + kGroups) % kGroups;
                if (kAnyGather)
                    for (int sk = 0; sk < i_first; ++sk) advance();
                auto skip = [&]() {
                    for (int sk = 0; sk < kGroups; ++sk) advance();
                };
                if (kWide) {
                    // the registers are free as soon as the B tile is written: the next slice's loads go out there and are
                    // on their way during the A tile, the signal and the wait for the next slot
                    if (i_first < n_slices) gather(a0, b0);
                    for (int i = i_first; i < n_slices; i += kGroups)
                        if (!process(it0 + i, a0, b0, [&]() { if (i + kGroups < n_slices) { skip(); gather(a0, b0); } })) { ok = false; break; }
                } else {
                    for (int i = i_first; i < n_slices; i += kGroups) {
                        if (kAnyGather) gather(a0, b0);
                        if (!process(it0 + i, a0, b0, []() {})) { ok = false; break; }
                        if (kAnyGather) skip();
                    }
                }
            } else {
                // two register sets in turn: the loads of slice i+1 are in flight while slice i is transformed
                if (kAnyGather) gather(a0, b0);
                for (int i = 0; i < n_slices; i += 2) {
                    if (kAnyGather && i + 1 < n_slices) { advance(); gather(a1, b1); }
                    if (!process(it0 + i, a0, b0, []() {})) { ok = false; break; }
                    if (i + 1 < n_slices) {
                        if (kAnyGather && i + 2 < n_slices) { advance(); gather(a0, b0); }
                        if (!process(it0 + i + 1, a1, b1, []() {})) { ok = false; break; }
                    }
                }
            }
            it0 += n_slices;
        }
    } else {
        // ================= epilogue warps: drain chunks, accumulate in fp32 registers =================
        regs_inc<kWide ? kRegsEpilogueWide : kRegsEpilogue>();
        const uint32_t q = warp & 3;                                      // TMEM lane quarter of this warp
        const int r_local = (int)(q * 32u + lane);
        float acc[kN];
        const uint32_t sq_addr = tmem_base + ((q * 32u) << 16) + kSqCol;  // kExact: this warp's rows of the sum of squares
        int c = 0;                                                        // running number of the chunk
        bool ok = true;
        SegIter<kExact> iter(prm);
        Seg sg;
        bool more = iter.next(prm, sg);
        grid_wait();
        for (; ok && more; more = iter.next(prm, sg)) {
#pragma unroll
            for (int j = 0; j < kN; ++j) acc[j] = 0.f;
            const bool square = kExact && prm.parts == 0;
            if (kExact && !kWide && square) {
                uint32_t zero[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) zero[j] = 0u;
#pragma unroll
                for (int j0 = 0; j0 < kN; j0 += 16) tc_st_32x16(sq_addr + j0, zero);
                tc_wait_st();
            }
            const int n_act = sg.n_act, n_valid = sg.n_valid;
            const int n_slices = sg.s_end - sg.s_begin;
            const int seg_len = kExact && prm.parts == 0 ? prm.p_slices : n_slices;
            const int cps = (seg_len + prm.chunk - 1) / prm.chunk;
            const int n_chunks = (n_slices / seg_len) * cps;
            for (int cc = 0; cc < n_chunks && ok; ++cc, ++c) {
                const int b = c & 1;
                ok = mbar_wait(smem_u32(&acc_full[b]), (uint32_t)(c >> 1) & 1u, &abort_flag, 256);
                if (!ok) break;
                tc_fence_after();
                const uint32_t taddr = tmem_base + ((q * 32u) << 16) + (uint32_t)b * kN;
#pragma unroll
                for (int j0 = 0; j0 < kN; j0 += 32) {
                    if (j0 < n_act) {
                        uint32_t r[32];
                        tc_ld_32x32(taddr + j0, r);
                        tc_wait_ld();
                        if (kExact && kWide && square) {                // the example's whole sum
#pragma unroll
                            for (int j = 0; j < 32; ++j) acc[j0 + j] = __fadd_rn(acc[j0 + j], __fmul_rn(__uint_as_float(r[j]), __uint_as_float(r[j])));
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j) acc[j0 + j] = __fadd_rn(acc[j0 + j], __uint_as_float(r[j]));
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
                if (kExact && !kWide && square && (cc + 1) % cps == 0) {
                    // end of an example: acc holds its sum over positions; add the squares to the running sum in TMEM
#pragma unroll
                    for (int j0 = 0; j0 < kN; j0 += 32) {
                        if (j0 < n_act) {
                            uint32_t r[32];
                            tc_ld_32x32(sq_addr + j0, r);
                            tc_wait_ld();
                            uint32_t w0[16], w1[16];
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                w0[j] = __float_as_uint(__fadd_rn(__uint_as_float(r[j]), __fmul_rn(acc[j0 + j], acc[j0 + j])));
                                w1[j] = __float_as_uint(__fadd_rn(__uint_as_float(r[16 + j]), __fmul_rn(acc[j0 + 16 + j], acc[j0 + 16 + j])));
                            }
                            tc_st_32x16(sq_addr + j0, w0);
                            tc_st_32x16(sq_addr + j0 + 16, w1);
                        }
                    }
                    tc_wait_st();
#pragma unroll
                    for (int j = 0; j < kN; ++j) acc[j] = 0.f;
                }
            }
            if (!ok) break;
            if (kExact && !kWide && square) {        // the result is the sum of squares
#pragma unroll
                for (int j0 = 0; j0 < kN; j0 += 32) {
                    uint32_t r[32];
                    tc_ld_32x32(sq_addr + j0, r);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) acc[j0 + j] = __uint_as_float(r[j]);
                }
            }
            // ---- the segment's 128 x 128 sums leave the registers (the other roles are already on the next segment)
            const int m = sg.m0 + r_local;
            float *const S = bt.S[sg.layer];
            if (!sg.whole) {
                // partial tile, [four columns][row][column]: a lane's four columns in one store, lanes side by side; rows past
                // the result's end (few output channels) are nobody's
                float *dst = prm.partial + (size_t)sg.slot * (kBM * kN) + 4 * r_local;
                if (sg.m0 + (int)(q * 32u) < prm.M)
#pragma unroll
                    for (int j = 0; j < kN; j += 4)
                        if (j < n_valid) *reinterpret_cast<float4 *>(dst + j * kBM) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
            } else if (prm.ld_m == 1) {
                // result is contiguous along m: lanes write neighbouring addresses directly
                if (m < prm.M) {
                    float *col = S + (size_t)m + (size_t)sg.n0 * prm.ld_n;
#pragma unroll
                    for (int j0 = 0; j0 < kN; j0 += 16) {        // old values sixteen at a time, all loads in flight
                        float old[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            old[j] = (prm.accumulate && j0 + j < n_valid) ? col[(size_t)(j0 + j) * prm.ld_n] : 0.f;
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j0 + j < n_valid) {
                                const float res = __fmul_rn(prm.scale, acc[j0 + j]);
                                col[(size_t)(j0 + j) * prm.ld_n] = prm.accumulate ? __fadd_rn(old[j], res) : res;
                            }
                    }
                }
            } else if (iter.pos >= iter.end) {
                // result is contiguous along n, and this is the block's last segment: the pipeline stages are idle
                // (the last accumulator was complete before we got here), so this warp's 32 x 128 block is transposed
                // through shared memory and written row by row with consecutive lanes on consecutive addresses
                float *tile = reinterpret_cast<float *>(smem_gen) + q * (32 * (kN + 1));
#pragma unroll
                for (int j = 0; j < kN; ++j) tile[lane * (kN + 1) + j] = __fmul_rn(prm.scale, acc[j]);
                __syncwarp();
                for (int r0 = 0; r0 < 32; r0 += 8) {              // eight rows at a time, all loads in flight
                    float old[8][kN / 32];
#pragma unroll
                    for (int rr = 0; rr < 8; ++rr) {
                        const int mr = sg.m0 + (int)(q * 32u) + r0 + rr;
                        const float *src = S + (size_t)mr * prm.ld_m + sg.n0;
#pragma unroll
                        for (int cblk = 0; cblk < kN / 32; ++cblk) {
                            const int j = cblk * 32 + (int)lane;
                            old[rr][cblk] = (prm.accumulate && mr < prm.M && j < n_valid) ? src[j] : 0.f;
                        }
                    }
#pragma unroll
                    for (int rr = 0; rr < 8; ++rr) {
                        const int mr = sg.m0 + (int)(q * 32u) + r0 + rr;
                        float *dst = S + (size_t)mr * prm.ld_m + sg.n0;
#pragma unroll
                        for (int cblk = 0; cblk < kN / 32; ++cblk) {
                            const int j = cblk * 32 + (int)lane;
                            if (mr < prm.M && j < n_valid) {
                                const float res = tile[(r0 + rr) * (kN + 1) + j];
                                dst[j] = prm.accumulate ? __fadd_rn(old[rr][cblk], res) : res;
                            }
                        }
                    }
                }
            } else if (m < prm.M) {
                // result is contiguous along n, more segments follow (the pipeline is busy with the next one): every
                // lane owns a row and writes it 16 bytes at a time (the halves of a
                // 32-byte sector arrive in consecutive instructions and are merged in L2); rows whose pitch is not a
                // multiple of 16 bytes go element by element
                float *row = S + (size_t)m * prm.ld_m + sg.n0;
                if (((prm.ld_m | sg.n0) & 3) == 0) {
#pragma unroll
                    for (int j0 = 0; j0 < kN; j0 += 16) {
                        float4 old[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            old[u] = (prm.accumulate && j0 + 4 * u + 3 < n_valid) ? *reinterpret_cast<const float4 *>(row + j0 + 4 * u)
                                                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int j = j0 + 4 * u;
                            if (j + 3 < n_valid) {
                                float4 res = make_float4(__fmul_rn(prm.scale, acc[j]), __fmul_rn(prm.scale, acc[j + 1]),
                                                         __fmul_rn(prm.scale, acc[j + 2]), __fmul_rn(prm.scale, acc[j + 3]));
                                if (prm.accumulate) {
                                    res.x = __fadd_rn(old[u].x, res.x); res.y = __fadd_rn(old[u].y, res.y);
                                    res.z = __fadd_rn(old[u].z, res.z); res.w = __fadd_rn(old[u].w, res.w);
                                }
                                *reinterpret_cast<float4 *>(row + j) = res;
                            } else {
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    if (j + e < n_valid) {
                                        const float res = __fmul_rn(prm.scale, acc[j + e]);
                                        row[j + e] = prm.accumulate ? __fadd_rn(row[j + e], res) : res;
                                    }
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < kN; ++j)
                        if (j < n_valid) {
                            const float res = __fmul_rn(prm.scale, acc[j]);
                            row[j] = prm.accumulate ? __fadd_rn(row[j], res) : res;
                        }
                }
            }
        }
    }

    // ---- common exit ----
    grid_wait();                                          // (the threads without a role that touches memory)
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicOr(prm.status, VGC_DEV_TIMEOUT);
}

typedef void (*KernelFn)(const Batch, const Params);
// The kernel's forms are compiled in several files: tiles of 192 columns whose B tile is gathered several taps at a time, the same with
// the input rows by TMA, and 128-column tiles gathered several taps at a time.  mode: how the B tile gets its rows.
KernelFn wide_taps_kernel(int mode, bool per_example, bool bf16_cross);
KernelFn wide_halo_kernel(int mode, bool per_example, bool bf16_cross);
KernelFn narrow_taps_kernel(int mode, bool per_example);

}  // namespace tc
}  // namespace vgc
