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
//      accumulator (the dropped lo*lo term is 2^-22 relative).  In the TMA-fed K-major form and the
//      wide form the two cross terms use bf16 copies of hi and lo instead (kind::f16, 16 deep per
//      instruction): a cross term is 2^-11 of the product, so 8-bit operands leave an error below
//      2^-18 of it, of either sign -- less than the third of the instructions saves of the
//      accumulator's truncation bias (largest error of 3x3 layers 2.9e-6 -> 2.4e-6).
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
#include <cstdlib>

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
constexpr uint32_t kTmemColsA = 64;                                 // per slot: 32 columns hi + 32 columns lo
constexpr uint32_t kTmemCols = 512;                                 // two accumulator buffers + the A operand ring

// how a tile gets its rows; kGatherTaps4 / kGatherTaps2: im2col rows of a Kw = 3, stride 1, pad_w = 1 kernel
// gathered three taps at a time (output width a multiple of 4 / of 2)
// kGatherTaps4S2 / kGatherTaps2S2: the same for stride 2 along w (input width twice the output width)
// kGatherTaps7S2: seven taps at a time for a Kw = 7, stride-2, pad-3 kernel (the first layer of the ImageNet networks)
enum { kTma = 0, kGatherErr = 1, kGatherIm2col = 2, kGatherTaps4 = 3, kGatherTaps2 = 4, kGatherTaps4S2 = 5,
       kGatherTaps2S2 = 6, kGatherTaps7S2 = 7 };

struct Params {
    int M, N;                // rows of the A tile space / of the B tile space
    int k_slices;            // 32-deep slices of one tile's reduction
    int p_slices;            // conv: slices per example (ceil(P/32)); dense: 1
    int chunk;               // slices per accumulator drain
    int unit;                // slices that stay in one block: the reduction is cut between units only
    int units_per_tile;      // k_slices / unit
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
    unsigned wo_magic;       // floor(2^32 / Wo) + 1: p / Wo == umulhi(p, wo_magic) for p * Wo < 2^32
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
                const int ho = prm.Wo == 1 ? p : (int)__umulhi((unsigned)p, prm.wo_magic), wo = p - ho * prm.Wo;
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
            const int ho = (int)__umulhi((unsigned)p, prm.wo_magic), wo = p - ho * prm.Wo;
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
            const int ho = (int)__umulhi((unsigned)p, prm.wo_magic), wo = p - ho * prm.Wo;
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
        const int ho = (int)__umulhi((unsigned)pbase, prm.wo_magic), wo = pbase - ho * prm.Wo;
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
    // kBf: `lo` takes hi and lo as bf16, tiles of 64-byte rows one behind the other; a thread's four k are half of a 16-byte chunk
    template <bool kSquare, bool kBf = false>
    __device__ __forceinline__ void store(uint8_t *hi, uint8_t *lo, int, int kq, const Regs &r) const
    {
#pragma unroll
        for (int i = 0; i < kTriples; ++i) {
            if (!kWhole && (g.row(i) >= kRows || g.row(i) <= -Impl::kKw)) continue;   // no row of this tuple in the tile
            // square and split every loaded element once; the three taps are views of the same parts
            uint32_t h[Impl::kSlots], l[Impl::kSlots];
#pragma unroll
            for (int e = 0; e < Impl::kLoaded; ++e) {
                const float q = kSquare ? __fmul_rn(r.v[i][e], r.v[i][e]) : r.v[i][e];
                h[e] = to_tf32(q);
                l[e] = __float_as_uint(__fsub_rn(q, __uint_as_float(h[e])));
            }
#pragma unroll
            for (int kw = 0; kw < Impl::kKw; ++kw) {
                const int row = g.row(i) + kw;
                if (kWhole || (unsigned)row < (unsigned)kRows) {
                    const uint32_t off = chunk_offset(row, kq);
                    *reinterpret_cast<uint4 *>(hi + off) =
                        make_uint4(h[Impl::idx(kw, 0)], h[Impl::idx(kw, 1)], h[Impl::idx(kw, 2)], h[Impl::idx(kw, 3)]);
                    if (kBf) {
                        auto pair = [&](const uint32_t (&v)[Impl::kSlots], int j) {
                            return pack_bf16(__uint_as_float(v[Impl::idx(kw, j)]), __uint_as_float(v[Impl::idx(kw, j + 1)]));
                        };
                        uint8_t *const at = lo + bf_offset(row, kq);
                        *reinterpret_cast<uint2 *>(at) = make_uint2(pair(h, 0), pair(h, 2));
                        *reinterpret_cast<uint2 *>(at + kRows * 64) = make_uint2(pair(l, 0), pair(l, 2));
                    } else
                    *reinterpret_cast<uint4 *>(lo + off) =
                        make_uint4(l[Impl::idx(kw, 0)], l[Impl::idx(kw, 1)], l[Impl::idx(kw, 2)], l[Impl::idx(kw, 3)]);
                }
            }
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
        sg.layer = tile / tiles_layer;
        const int rem = tile - sg.layer * tiles_layer;
        const int tile_m = rem / prm.tiles_x, tile_n = rem - tile_m * prm.tiles_x;
        sg.m0 = tile_m * kBM;
        sg.n0 = tile_n * prm.tile_n;
        sg.n_valid = min(prm.tile_n, prm.N - sg.n0);
        sg.n_act = (sg.n_valid + 15) & ~15;
        sg.s_begin = u0 * prm.unit;
        sg.s_end = u1 * prm.unit;
        sg.whole = u0 == 0 && u1 == upt;
        sg.slot = 2 * (int)blockIdx.x + (index > 0 ? 1 : 0);     // a block's partial segments: its first and / or its last
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
    static_assert(!kWide || (kN == kWideN && kATmem && IsTaps<kModeB>::value), "wide tiles: several taps at a time");
    constexpr bool kSplit = kATmem && (!kAnyGather || kWide);              // A raw tiles in a ring of their own
    static_assert(!kBf || (kSplit && !kExact), "bf16 cross terms: A in tensor memory, sums of squares");
    constexpr bool kTmaB = kSplit && !kGatherB;                            // split form: the B tile comes by TMA, too
    constexpr int kNA = kWide ? kWideA : kSplitA;                                           // slots of the raw A ring (split form)
    // the transform warps work as two groups of four on alternate slices (else all eight on every slice)
    constexpr bool kTwoGroups = !kAnyGather || (IsTaps<kModeB>::value && kModeA == kTma);
    constexpr int kNB = kWide ? kWideB : kSplit ? kSplitB : kRawSlots;     // slots of the raw / hi ring
    // lo slots (and A slots in TMEM); the per-example form needs 128 TMEM columns for its sum of squares
    constexpr int kLoN = kWide ? kWideB : (kExact && kATmem) ? 2 : kSplit ? kSplitLo : (kATmem ? kLoSlotsAT : kLoSlots);
    constexpr int kAN = kWide ? kWideTmemA : kLoN;                         // A slots in tensor memory
    constexpr uint32_t kBBytes = kN * kBK * 4;                             // bytes of a B tile
    constexpr uint32_t kSqCol = 2 * kBN + (kATmem ? 2 * kTmemColsA : 0);         // where that sum lives
    constexpr uint32_t kLoBytes = kATmem ? kRawBytesB : kRawStageBytes;  // bytes of one lo slot
    // byte offsets of slot s: the [A][B] pair of the raw / hi ring (split form: only its B half exists, the
    // offset points one A tile below it), the lo ring likewise, and the split form's A ring
    auto pair_off = [](int s) -> uint32_t { return kWide ? kWideA * kRawBytesA + (uint32_t)s * kBBytes - kRawBytesA : kSplit ? (uint32_t)(kSplitA + s - 1) * kRawBytesA : (uint32_t)s * kRawStageBytes; };
    auto lo_off = [](int s) -> uint32_t {
        return kWide ? kWideA * kRawBytesA + (uint32_t)(kWideB + s) * kBBytes - kRawBytesA
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
            SegIter iter(prm);
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
            SegIter iter(prm);
            Seg sg;
            bool more = iter.next(prm, sg);
            for (; ok && more; more = iter.next(prm, sg)) {
                const uint32_t idesc = instr_desc(kMajor, sg.n_act, kBM);
                const uint32_t idesc_bf = instr_desc_bf16(sg.n_act, kBM);
                // an accumulator is drained every prm.chunk slices, and (kExact) at the end of every example: the
                // segment's slices are runs of seg_len slices (whole examples -- the work is cut that way), each cut
                // into cps chunks
                const int n_slices = sg.s_end - sg.s_begin;
                const int seg_len = kExact ? prm.p_slices : n_slices;
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
        typedef Gatherer<kModeB, kTwoGroups, kN> GatherB;
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
            rows_b.load(prm, z, pbase, gb);
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
                rows_b.template store<!kExact, kBf>(hi + kRawBytesA, lo + kRawBytesA, row0, kq, gb);
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
        SegIter iter(prm);
        Seg sg;
        bool more = iter.next(prm, sg);
        for (; ok && more; more = iter.next(prm, sg)) {
            const int n_slices = sg.s_end - sg.s_begin;
            if (kAnyGather) {
                rows_a.init(prm, bt.x[sg.layer], bt.delta[sg.layer], sg.m0, row0, prm.M);
                rows_b.init(prm, bt.x[sg.layer], bt.delta[sg.layer], sg.n0, row0, prm.N);
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
        SegIter iter(prm);
        Seg sg;
        bool more = iter.next(prm, sg);
        grid_wait();
        for (; ok && more; more = iter.next(prm, sg)) {
#pragma unroll
            for (int j = 0; j < kN; ++j) acc[j] = 0.f;
            if (kExact && !kWide) {
                uint32_t zero[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) zero[j] = 0u;
#pragma unroll
                for (int j0 = 0; j0 < kN; j0 += 16) tc_st_32x16(sq_addr + j0, zero);
                tc_wait_st();
            }
            const int n_act = sg.n_act, n_valid = sg.n_valid;
            const int n_slices = sg.s_end - sg.s_begin;
            const int seg_len = kExact ? prm.p_slices : n_slices;
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
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float d = __uint_as_float(r[j]);      // wide per-example form: the example's whole sum
                            acc[j0 + j] = __fadd_rn(acc[j0 + j], kExact && kWide ? __fmul_rn(d, d) : d);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
                if (kExact && !kWide && (cc + 1) % cps == 0) {
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
            if (kExact && !kWide) {        // the result is the sum of squares
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
                if ((prm.ld_m & 3) == 0) {
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

// Adds the partial tiles of every tile that more than one block worked on, in the order of the blocks (a fixed
// order: the result does not depend on scheduling).  One thread block per 32 x 32 patch of a tile: a warp takes
// four columns, a lane one row of them -- 16 bytes per lane and partial tile, four sums -- and the result is written along
// whichever of m / n has unit stride.  Tiles that one block covered alone were written by that block; their patches return
// at once.  Which partial tiles they are is worked out before the wait for the kernel that writes them.
struct ResultPtrs { float *S[kMaxBatch]; };

// What both combine kernels need to know about a tile of the launch.
struct TileParts {
    int b_first, b_last;     // the blocks that hold the tile's first and last unit
    int tx, ty;
    bool first_is_last;      // the first block's part of this tile is that block's last segment (slot 1), not its first;
                             // every later block's part is its first segment
    __device__ __forceinline__ TileParts(int units_q, int units_r, int units_per_tile, int tiles_x, int tiles_y, int layer, int tile)
    {
        // the first units_r blocks own units_q + 1 units each, the others units_q
        const int t_lo = (layer * (tiles_x * tiles_y) + tile) * units_per_tile, t_hi = t_lo + units_per_tile - 1;
        const int big = units_r * (units_q + 1);
        auto block_of = [&](int u) -> int { return u < big ? u / (units_q + 1) : units_r + (u - big) / units_q; };
        b_first = block_of(t_lo);
        b_last = block_of(t_hi);
        first_is_last = b_first * units_q + min(b_first, units_r) < t_lo;
        ty = tile / tiles_x;
        tx = tile - ty * tiles_x;
    }
};
__device__ __forceinline__ float4 add4(const float4 &a, const float4 &b)
{
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}

__global__ void __launch_bounds__(256)
sqgrad_tc_combine(const float *partial, int units_q, int units_r, int units_per_tile,
                  int tile_n, int tiles_x, int tiles_y, int M, int N, float scale, int accumulate, const ResultPtrs results,
                  long long ld_m, long long ld_n)
{
    __shared__ float patch[32][33];
    grid_release();
    const int tile = blockIdx.x / (tile_n >> 3), sub = blockIdx.x - tile * (tile_n >> 3);
    const TileParts parts(units_q, units_r, units_per_tile, tiles_x, tiles_y, (int)blockIdx.y, tile);
    const int tx = parts.tx, ty = parts.ty;
    float *S = results.S[blockIdx.y];                                      // blockIdx.y: layer of the batch
    const int r0 = (sub & 3) * 32, j0 = (sub >> 2) * 32;                  // patch origin inside the tile
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;              // lane -> row, warp -> four columns
    const size_t step = (size_t)2 * kBM * tile_n;                         // from a block's first segment to the next block's
    const float *src = partial + ((size_t)(j0 / 4 + w) * kBM + r0 + lane) * 4 + (size_t)parts.b_first * step;
    const float *src0 = src + (parts.first_is_last ? step / 2 : 0);
    grid_wait();
    if (parts.b_first == parts.b_last || ty * kBM + r0 >= M || tx * tile_n + j0 >= N) return;
    float4 sum = __ldcs(reinterpret_cast<const float4 *>(src0));
    const int n = parts.b_last - parts.b_first;
    int b = 1;
    for (; b + 4 <= n + 1; b += 4) {                     // four loads in flight, summed in block order
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldcs(reinterpret_cast<const float4 *>(src + (size_t)(b + u) * step));
#pragma unroll
        for (int u = 0; u < 4; ++u) sum = add4(sum, v[u]);
    }
    {
        float4 v[3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (b + u <= n) v[u] = __ldcs(reinterpret_cast<const float4 *>(src + (size_t)(b + u) * step));
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (b + u <= n) sum = add4(sum, v[u]);
    }
    const float sums[4] = {sum.x, sum.y, sum.z, sum.w};
    if (ld_m == 1) {
        const int m = ty * kBM + r0 + lane;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int n = tx * tile_n + j0 + 4 * w + c;
            if (m < M && n < N) {
                float *dst = S + (size_t)m + (size_t)n * ld_n;
                const float res = __fmul_rn(scale, sums[c]);
                *dst = accumulate ? __fadd_rn(*dst, res) : res;
            }
        }
        return;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) patch[4 * w + c][lane] = __fmul_rn(scale, sums[c]);      // patch[column][row]
    __syncthreads();
    {
        const int c0 = (threadIdx.x & 7) * 4, r = threadIdx.x >> 3;       // four consecutive columns of one row
        const int m = ty * kBM + r0 + r, n = tx * tile_n + j0 + c0;
        if (m < M) {
            float *dst = S + (size_t)m * ld_m + n;
            if ((ld_m & 3) == 0 && n + 3 < N) {
                float4 out = make_float4(patch[c0][r], patch[c0 + 1][r], patch[c0 + 2][r], patch[c0 + 3][r]);
                if (accumulate) out = add4(*reinterpret_cast<const float4 *>(dst), out);
                *reinterpret_cast<float4 *>(dst) = out;
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (n + c < N) dst[c] = accumulate ? __fadd_rn(dst[c], patch[c0 + c][r]) : patch[c0 + c][r];
            }
        }
    }
}

// The same for tiles that many blocks worked on: a thread block per 32 rows x 4 columns, the partial tiles dealt out to its
// eight warps in turn and their sums added in the order of the warps (a fixed order as well).  A chain of 148 partial tiles
// took 22 us in the kernel above.
__global__ void __launch_bounds__(256)
sqgrad_tc_combine_many(const float *partial, int units_q, int units_r, int units_per_tile,
                       int tile_n, int tiles_x, int tiles_y, int M, int N, float scale, int accumulate, const ResultPtrs results,
                       long long ld_m, long long ld_n)
{
    __shared__ float sums[8][4][32];
    grid_release();
    const int tile = blockIdx.x / tile_n, sub = blockIdx.x - tile * tile_n;
    const TileParts parts(units_q, units_r, units_per_tile, tiles_x, tiles_y, (int)blockIdx.y, tile);
    const int r0 = (sub & 3) * 32, j0 = (sub >> 2) * 4;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // thread of the first four warps: one element of the patch, lanes along whichever of m / n has unit stride; its old
    // content is on its way during the sums
    const int row = ld_m == 1 ? lane : 8 * w + (lane >> 2), col = ld_m == 1 ? w : lane & 3;
    const int m = parts.ty * kBM + r0 + row, n = parts.tx * tile_n + j0 + col;
    const bool mine = w < 4 && m < M && n < N;
    float *const dst = results.S[blockIdx.y] + (size_t)m * ld_m + (size_t)n * ld_n;
    const size_t step = (size_t)2 * kBM * tile_n;
    const float *src = partial + ((size_t)(j0 / 4) * kBM + r0 + lane) * 4 + (size_t)parts.b_first * step;
    grid_wait();
    if (parts.b_first == parts.b_last || parts.ty * kBM + r0 >= M || parts.tx * tile_n + j0 >= N) return;
    const float old = accumulate && mine ? *dst : 0.f;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    const int last = parts.b_last - parts.b_first;
#pragma unroll 4
    for (int b = w; b <= last; b += 8)
        sum = add4(sum, __ldcs(reinterpret_cast<const float4 *>(src + (size_t)b * step + (b == 0 && parts.first_is_last ? step / 2 : 0))));
    sums[w][0][lane] = sum.x; sums[w][1][lane] = sum.y; sums[w][2][lane] = sum.z; sums[w][3][lane] = sum.w;
    __syncthreads();
    if (!mine) return;
    float total = sums[0][col][row];
#pragma unroll
    for (int i = 1; i < 8; ++i) total = __fadd_rn(total, sums[i][col][row]);
    const float res = __fmul_rn(scale, total);
    *dst = accumulate ? __fadd_rn(old, res) : res;
}

// ---- host side --------------------------------------------------------------------------------
// Slices per accumulator drain.  The tensor core's fp32 accumulation truncates (a one-sided bias of about 1.3e-8 of the
// sum per instruction), so an accumulator is handed to the round-to-nearest register sums after at most 8 slices
// (96 instructions): results then sit 1 - 3e-6 below the exact sum, against the 1e-5 bound.
constexpr int kChunk = 8;
// how many sqgrad launches the caller keeps in flight side by side (vgc_sqgrad_plan_hint)
static int g_concurrent = 1;

struct Plan {
    int unit, units_per_tile, blocks, tiles_x, tiles_y;
    int units_total;
    bool partials;           // some tile is shared by several blocks: partial tiles go through the scratch
};

// How a launch's work -- n_layers x tiles x k_slices slices -- is cut into one contiguous range per block.
// `unit_min`: slices that must stay in one block (the per-example form cuts the reduction between examples only).
// Two candidates: whole tiles per block (no scratch, no second kernel, but the blocks' loads are as even as the
// tile count allows), or an even cut of the slices over all SMs (tiles at the cuts are shared, their partial
// sums combined by a second kernel).  Costs in slice times: a block's longest range, plus what the combine pass
// adds to the call (its launch and the partial tiles' round trip, about 14 slices' worth: measured with tiles of 128 columns
// and before launches overlapped; not measured again for the wide form and for chains that several warps share).
static Plan make_plan(int M, int N, int k_slices, int n_layers, int unit_min, int tile_n)
{
    Plan p;
    p.tiles_x = (N + tile_n - 1) / tile_n;
    p.tiles_y = (M + kBM - 1) / kBM;
    const long long tiles = (long long)p.tiles_x * p.tiles_y * n_layers;
    const long long upt = k_slices / unit_min, units = tiles * upt;
    bool even;
    long long blocks;
    if (g_concurrent > 1) {
        // Next to other launches the hardware's block scheduler does the balancing: blocks of all launches in flight
        // queue for the SMs and a partly filled wave costs nothing (the neighbours' blocks take the idle SMs).  Each
        // tile's reduction is cut into as many parts as make about half a wave of blocks per launch: shorter blocks
        // pay their start and tail more often, longer ones balance worse (measured on the ResNet-50 pass with 3 to 8
        // launches in flight: 148 blocks per launch 1.90 ms, 111: 1.86, 74: 1.80 - 1.85, 50: 1.99).
        long long parts = (kSmCount / 2) / tiles;
        parts = parts > upt ? upt : (parts < 1 ? 1 : parts);
        even = parts > 1;
        blocks = tiles * parts;
    } else {
        // Alone, the launch is one block per SM at most.  Two candidates, costs in slice times: whole tiles per block
        // (a block's longest range), or an even cut of all slices (plus what the combine pass adds to the call: its
        // launch and the partial tiles' round trip, about 14 slices' worth).
        const long long waves = (tiles + kSmCount - 1) / kSmCount;
        const long long blocks_a = (tiles + waves - 1) / waves;
        const long long cost_a = ((tiles + blocks_a - 1) / blocks_a) * k_slices;
        const long long blocks_b = units < kSmCount ? units : kSmCount;
        const long long cost_b = ((units + blocks_b - 1) / blocks_b) * unit_min + 14;
        even = cost_b < cost_a;
        blocks = even ? blocks_b : blocks_a;
    }
    if (even && units >= (1LL << 31)) {          // unit positions are 32-bit in the kernel: whole tiles then
        even = false;
        blocks = tiles < kSmCount ? tiles : kSmCount;
    }
    p.unit = even ? unit_min : k_slices;
    p.units_per_tile = even ? (int)upt : 1;
    p.units_total = (int)(even ? units : tiles);
    p.blocks = (int)blocks;
    p.partials = false;
    const int q = p.units_total / p.blocks, r = p.units_total % p.blocks;
    for (int b = 1; b < p.blocks && !p.partials; ++b) p.partials = (b * q + (b < r ? b : r)) % p.units_per_tile != 0;
    return p;
}

}  // namespace tc

using namespace tc;

void tc_plan_hint(int concurrent_launches)
{
    g_concurrent = concurrent_launches > 1 ? concurrent_launches : 1;
}

bool tc_linear_supported(int B, int in, int out)
{
    return B >= 32 && in >= 32 && out >= 32 && in % 4 == 0 && out % 4 == 0;
}
bool tc_conv_supported(int B, int C, int H, int W, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw)
{
    const long Ho = (H + 2 * ph - Kh) / sh + 1, Wo = (W + 2 * pw - Kw) / sw + 1;
    const long P = Ho * Wo, N = (long)C * Kh * Kw;
    // 32-bit index arithmetic inside the kernel
    return B >= 1 && C >= 1 && Cout >= 1 && (long)C * H * W < (1L << 30) && N < (1L << 24) &&
           (long)B * ((P + kBK - 1) / kBK) < (1L << 30);
}

static size_t tc_workspace_bytes(int M, int N, int k_slices, int n_layers = 1, int unit = 1, int tile_n = kBN)
{
    const Plan p = make_plan(M, N, k_slices, n_layers, unit, tile_n);
    // status word (256 bytes) + two partial tiles per block (the first and the last segment of its range)
    return 256 + (p.partials ? (size_t)2 * p.blocks * kBM * tile_n * sizeof(float) : 0);
}

typedef void (*KernelFn)(const Batch, const Params);

static vgc_status tc_launch(KernelFn kernel, const Batch &bt, int n_layers, Params prm, int M, int N,
                            int k_slices, void *ws, size_t ws_bytes, cudaStream_t st, int unit = 1, int tile_n = kBN)
{
    const Plan plan = make_plan(M, N, k_slices, n_layers, unit, tile_n);
    if (ws_bytes < tc_workspace_bytes(M, N, k_slices, n_layers, unit, tile_n)) return VGC_ERR_WORKSPACE;
    VGC_CUDA_OK(allow_dynamic_smem(reinterpret_cast<const void *>(kernel), kSmemBytes, kRegsLaunch));
    prm.M = M; prm.N = N; prm.k_slices = k_slices;
    prm.unit = plan.unit; prm.units_per_tile = plan.units_per_tile; prm.units_total = plan.units_total;
    prm.units_q = plan.units_total / plan.blocks; prm.units_r = plan.units_total % plan.blocks;
    prm.tile_n = tile_n; prm.tiles_x = plan.tiles_x; prm.tiles_y = plan.tiles_y;
    prm.chunk = kChunk;
    prm.status = static_cast<uint32_t *>(ws);
    prm.partial = reinterpret_cast<float *>(static_cast<char *>(ws) + 256);
    VGC_CUDA_OK(launch_kernel(kernel, dim3((unsigned)plan.blocks), dim3(kThreadsTc), kSmemBytes, st, true, bt, prm));
    count_launch();
    if (plan.partials) {
        ResultPtrs results = {};
        for (int l = 0; l < n_layers; ++l) results.S[l] = bt.S[l];
        // eight and more partial tiles per tile: the warps share the chain
        const bool many = plan.units_per_tile >= 8 * (prm.units_q + 1);
        const unsigned patches = (unsigned)(plan.tiles_x * plan.tiles_y) * (unsigned)(many ? tile_n : tile_n / 8);
        const auto combine = many ? sqgrad_tc_combine_many : sqgrad_tc_combine;
        // L1 for the loads of eight blocks (34 KB of shared memory) behind the kernel above, which takes all shared memory;
        // with the same for sqgrad_repack, a pass over ResNet-50, batch 32, takes 1853 us instead of 1880
        VGC_CUDA_OK(prefer_carveout(reinterpret_cast<const void *>(combine), 18));
        VGC_CUDA_OK(launch_kernel(combine, dim3(patches, (unsigned)n_layers), dim3(256), 0, st,
                                  true, prm.partial, prm.units_q, prm.units_r, plan.units_per_tile, tile_n, plan.tiles_x, plan.tiles_y, M, N,
                                  prm.scale, prm.accumulate, results, prm.ld_m, prm.ld_n));
        count_launch();
    }
    VGC_CUDA_OK(cudaGetLastError());
    return VGC_OK;
}

size_t tc_linear_workspace_bytes(int B, int in, int out) { return tc_workspace_bytes(out, in, (B + kBK - 1) / kBK); }

vgc_status tc_sqgrad_linear(const float *x, const float *delta, int B, int in, int out, float scale, int accumulate,
                            float *S, void *ws, size_t ws_bytes, cudaStream_t st)
{
    Batch bt = {};
    const cuuint32_t box[2] = {32, (cuuint32_t)kBK};
    const cuuint64_t dims_a[2] = {(cuuint64_t)out, (cuuint64_t)B}, str_a[1] = {(cuuint64_t)out * 4};
    const cuuint64_t dims_b[2] = {(cuuint64_t)in, (cuuint64_t)B}, str_b[1] = {(cuuint64_t)in * 4};
    if (!make_map(&bt.a[0], delta, 2, dims_a, str_a, box, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B) ||
        !make_map(&bt.b[0], x, 2, dims_b, str_b, box, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B))
        return VGC_ERR_CUDA;
    bt.x[0] = x; bt.delta[0] = delta; bt.S[0] = S;
    Params prm = {};
    prm.p_slices = 1; prm.tx_bytes = kRawStageBytes; prm.tx_bytes_a = kRawBytesA; prm.scale = scale;
    prm.accumulate = accumulate;
    prm.ld_m = in; prm.ld_n = 1;
    return tc_launch(sqgrad_tc<kMajorMN, kTma, kTma, false>, bt, 1, prm, out, in, (B + kBK - 1) / kBK, ws, ws_bytes, st);
}

// Set for the duration of a per-example (exact) call: planning, repacking and kernel choice consult it.
static thread_local bool t_exact = false;
struct ExactScope {
    bool saved;
    explicit ExactScope(bool on) : saved(t_exact) { t_exact = on; }
    ~ExactScope() { t_exact = saved; }
};

// Cout <= 64: the im2col rows take the 128-row A tile and the errors the narrow B tile
static bool conv_swapped(int Cout, int n_im2col) { return Cout <= 64 && n_im2col > Cout; }

// ---- repacking pre-pass for 1x1 convolutions whose tiles TMA cannot address in place ----------
// A strided 1x1 convolution reads every (sh, sw)-th input position, and planes of P positions with P not
// a multiple of 4 (7x7) have a row pitch TMA does not accept.  One small copy kernel per operand puts
// them into a layout the TMA-fed kernel takes:
//   kRepackPlanes   x_s[z][c][p] = x[z][c][(p / Wo) sh][(p % Wo) sw]: the input subsampled, examples kept
//                   apart (the errors are used where they are)
//   kRepackFlat     x_r[c][z P + p], d_r[o][z P + p]: channel-major, the (example, position) pairs of one
//                   channel back to back -- the layer becomes a 1x1 convolution over ONE example with
//                   B P positions, and its reduction has no per-example padding to whole slices
//   kRepackPadW     a Kw = 3, pad_w = 1 kernel with stride 1 (W == Wo) or 2 (W == 2 Wo) whose output planes have
//                   an odd width (7x7): the errors are copied into planes of width Wo4 = Wo rounded up to 4 and x
//                   into planes of width stride * Wo4, new columns zero.  Zero input columns are what the padding
//                   supplies anyway, zero error columns contribute nothing, so the statistic is unchanged -- and
//                   the padded layer has TMA-able error planes and takes the three-tap gather
enum { kRepackNone = 0, kRepackPlanes = 1, kRepackFlat = 2, kRepackPadW = 3 };

static int repack_mode(int B, int C, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int P, int W = 0, int Ho = 0,
                       int Wo = 0)
{
    if ((long)B * C >= (1L << 31) || (long)B * Cout >= (1L << 31)) return kRepackNone;      // 32-bit row index
    if (Kw == 3 && pw == 1 && Wo % 2 == 1 && Wo >= 3 && (long)Ho * ((Wo + 3) / 4 * 4) >= kBK &&
        ((sw == 1 && sh == 1 && W == Wo) || (sw == 2 && W == 2 * Wo)))
        return kRepackPadW;
    if (Kh != 1 || Kw != 1 || ph != 0 || pw != 0) return kRepackNone;
    const bool planes_ok = P >= kBK && P % 4 == 0;
    if (planes_ok) return (sh > 1 || sw > 1) ? kRepackPlanes : kRepackNone;
    const long flat = (long)B * P;
    if (t_exact) return kRepackNone;                 // the flat form merges the examples' positions
    return (flat >= kBK && flat % 4 == 0 && flat < (1L << 30)) ? kRepackFlat : kRepackNone;
}

// One tensor to repack: out[a][b][p] = in[z][c][(p / Wo) sh W + (p % Wo) sw], zero where p % Wo >= wo_valid, with
// (a, b) = (z, c), or (c, z) when channel_major.  All tensors of a layer group go into one launch.
struct RepackJob {
    const float *in;
    float *out;
    int C, HW, W, Wo, P, sh, sw, channel_major, wo_valid;
};
struct RepackJobs {
    RepackJob job[2 * kMaxBatch];
    int B;
};

// n / d for n <= most: one multiplication where it is exact (n d < 2^32), which is everywhere but in huge planes.
struct Divisor {
    uint32_t d, magic;
    __device__ __forceinline__ Divisor(uint32_t v, uint32_t most)
        : d(v), magic(v > 1 && ((unsigned long long)most * v >> 32) == 0 ? 0xffffffffu / v + 1u : 0u) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t n) const { return magic ? __umulhi(n, magic) : n / d; }
};

// out[a][b][p] = in[z][c][(p / Wo) sh W + (p % Wo) sw] with (a, b) = (z, c), or (c, z) when channel_major.
// Bound: HBM latency.  The output is one contiguous run whatever the planes' size; a warp takes 512 of it, lanes side by
// side, all 16 loads of a lane in flight before the first store (with a warp per four planes, eight loads and a grid of one
// small wave, 256 channels 56 x 56 to 28 x 28, batch 32, took 20 us longer a call: 89 -> 69 us with its contraction).
constexpr int kRepackRun = 512;
__global__ void __launch_bounds__(256)
sqgrad_repack(const __grid_constant__ RepackJobs jobs)
{
    grid_release();
    // blockIdx.y picks the tensor; its description is read once (a run-time index into kernel parameters
    // is expensive, so nothing below touches `jobs` again)
    const RepackJob job = jobs.job[blockIdx.y];
    const uint32_t lane = threadIdx.x & 31, B = (uint32_t)jobs.B, P = (uint32_t)job.P;
    const size_t total = (size_t)B * job.C * P;
    const Divisor by_P(P, P + kRepackRun), by_B(B, B + kRepackRun), by_Wo((uint32_t)job.Wo, P);
    const uint32_t row_step = (uint32_t)job.sh * job.W;
    const bool whole = job.channel_major && job.sh == 1 && job.sw == 1 && job.W == job.Wo && job.wo_valid == job.Wo;
    grid_wait();
    for (size_t base = (size_t)(blockIdx.x * 8 + (threadIdx.x >> 5)) * kRepackRun; base < total;
         base += (size_t)gridDim.x * 8 * kRepackRun) {
        const uint32_t row0 = base >> 32 ? (uint32_t)(base / P) : (uint32_t)base / P;
        const uint32_t p0 = (uint32_t)(base - (size_t)row0 * P);
        // channel-major rows: row = c B + z
        const uint32_t c0 = job.channel_major ? row0 / B : 0, z0 = job.channel_major ? row0 - c0 * B : 0;
        const uint32_t left = total - base < kRepackRun ? (uint32_t)(total - base) : kRepackRun;
        float v[kRepackRun / 32];
        if (whole) {      // planes as they are, channel-major (2048 + 512 channels, 7 x 7, three layers: 28.4 -> 21.8 us)
#pragma unroll
            for (int u = 0; u < kRepackRun / 32; ++u) {
                const uint32_t i = lane + 32u * u, q = p0 + i;
                const uint32_t dr = by_P(q), dc = by_B(z0 + dr), plane = (z0 + dr - dc * B) * job.C + (c0 + dc);
                v[u] = i < left ? job.in[(size_t)plane * P + (q - dr * P)] : 0.f;
            }
        } else
#pragma unroll
        for (int u = 0; u < kRepackRun / 32; ++u) {
            const uint32_t i = lane + 32u * u, q = p0 + i;
            const uint32_t dr = by_P(q), p = q - dr * P;
            size_t plane;
            if (job.channel_major) {
                const uint32_t dc = by_B(z0 + dr);
                plane = (size_t)(z0 + dr - dc * B) * job.C + (c0 + dc);
            } else plane = row0 + dr;
            const uint32_t ho = by_Wo(p), wo = p - ho * job.Wo;
            // columns wo >= wo_valid are zero padding
            v[u] = i < left && wo < (uint32_t)job.wo_valid ? job.in[plane * job.HW + (ho * row_step + wo * job.sw)] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kRepackRun / 32; ++u)
            if (lane + 32u * u < left) job.out[base + lane + 32u * u] = v[u];
    }
}

static size_t conv_workspace_plain(int n_layers, int B, int C, int Kh, int Kw, int P, int Cout)
{
    const int p_slices = (P + kBK - 1) / kBK, n_im2col = C * Kh * Kw, k_slices = B * p_slices;
    const int unit = t_exact ? p_slices : 1;
    // the wide and the narrow form of a layer that gathers several taps at a time: either can be chosen at call time
    const size_t narrow = conv_swapped(Cout, n_im2col) ? tc_workspace_bytes(n_im2col, Cout, k_slices, n_layers, unit)
                                                       : tc_workspace_bytes(Cout, n_im2col, k_slices, n_layers, unit);
    const size_t wide = Kw > 1 ? tc_workspace_bytes(Cout, n_im2col, k_slices, n_layers, unit, kWideN) : 0;
    return narrow > wide ? narrow : wide;
}

// Workspace of one launch over n_layers layers of this geometry (n_layers <= kMaxBatch).
static size_t conv_workspace_group(int n_layers, int B, int C, int Kh, int Kw, int sh, int sw, int ph, int pw, int P,
                                   int Cout, int H, int W, int Ho, int Wo)
{
    // the larger of the in-place form and the repacked one, so that either can be chosen at call time
    size_t need = conv_workspace_plain(n_layers, B, C, Kh, Kw, P, Cout);
    const int mode = repack_mode(B, C, Cout, Kh, Kw, sh, sw, ph, pw, P, W, Ho, Wo);
    const size_t x_bytes = round_up(sizeof(float) * (size_t)B * C * P, 256);
    const size_t d_bytes = round_up(sizeof(float) * (size_t)B * Cout * P, 256);
    if (mode == kRepackPadW) {
        const int Wo4 = (Wo + 3) / 4 * 4;
        const size_t xp = round_up(sizeof(float) * (size_t)B * C * H * (sw * Wo4), 256);
        const size_t dp = round_up(sizeof(float) * (size_t)B * Cout * Ho * Wo4, 256);
        const size_t r = round_up(conv_workspace_plain(n_layers, B, C, Kh, Kw, Ho * Wo4, Cout), 256) + n_layers * (xp + dp);
        need = need > r ? need : r;
    } else if (mode == kRepackPlanes) {
        const size_t r = round_up(conv_workspace_plain(n_layers, B, C, 1, 1, P, Cout), 256) + n_layers * x_bytes;
        need = need > r ? need : r;
    } else if (mode == kRepackFlat) {
        const size_t r = round_up(conv_workspace_plain(n_layers, 1, C, 1, 1, B * P, Cout), 256) +
                         n_layers * (x_bytes + d_bytes);
        need = need > r ? need : r;
    }
    return need;
}

size_t tc_conv_workspace_bytes(int n_layers, int B, int C, int H, int W, int Kh, int Kw, int sh, int sw, int ph, int pw,
                               int Ho, int Wo, int Cout, bool exact)
{
    const int P = Ho * Wo;
    ExactScope scope(exact);
    // more layers than one launch takes are processed group after group in the same workspace
    const int first = n_layers < kMaxBatch ? n_layers : kMaxBatch;
    size_t need = conv_workspace_group(first, B, C, Kh, Kw, sh, sw, ph, pw, P, Cout, H, W, Ho, Wo);
    const int rest = n_layers > kMaxBatch ? n_layers % kMaxBatch : 0;
    if (rest) {
        const size_t r = conv_workspace_group(rest, B, C, Kh, Kw, sh, sw, ph, pw, P, Cout, H, W, Ho, Wo);
        need = need > r ? need : r;
    }
    return need;
}

static vgc_status conv_group(int n_layers, const float *const *x, const float *const *delta, float *const *S, int B,
                             int C, int H, int W, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int Ho,
                             int Wo, float scale, int accumulate, void *ws, size_t ws_bytes, cudaStream_t st)
{
    const int P = Ho * Wo, n_im2col = C * Kh * Kw;
    const int mode = repack_mode(B, C, Cout, Kh, Kw, sh, sw, ph, pw, P, W, Ho, Wo);
    if (mode != kRepackNone) VGC_CUDA_OK(prefer_carveout(reinterpret_cast<const void *>(sqgrad_repack), 5));      // no shared memory: all L1
    // one run of the output per warp; more when there are many
    auto blocks_for = [](size_t values) { const size_t b = (values + 8 * kRepackRun - 1) / (8 * kRepackRun); return (unsigned)(b < 1 ? 1 : (b > 148 * 32 ? 148 * 32 : b)); };
    if (mode == kRepackPadW) {
        const int Wo4 = (Wo + 3) / 4 * 4, Wx = sw * Wo4;              // padded widths of the errors and of x
        const size_t inner = round_up(conv_workspace_plain(n_layers, B, C, Kh, Kw, Ho * Wo4, Cout), 256);
        const size_t xp = round_up(sizeof(float) * (size_t)B * C * H * Wx, 256);
        const size_t dp = round_up(sizeof(float) * (size_t)B * Cout * Ho * Wo4, 256);
        if (ws_bytes < inner + n_layers * (xp + dp)) return VGC_ERR_WORKSPACE;
        const float *xr[kMaxBatch], *dr[kMaxBatch];
        RepackJobs jobs = {};
        jobs.B = B;
        for (int l = 0; l < n_layers; ++l) {
            char *base = static_cast<char *>(ws) + inner + (size_t)l * (xp + dp);
            float *x_p = reinterpret_cast<float *>(base), *d_p = reinterpret_cast<float *>(base + xp);
            jobs.job[2 * l] = RepackJob{x[l], x_p, C, H * W, W, Wx, H * Wx, 1, 1, 0, W};
            jobs.job[2 * l + 1] = RepackJob{delta[l], d_p, Cout, Ho * Wo, Wo, Wo4, Ho * Wo4, 1, 1, 0, Wo};
            xr[l] = x_p; dr[l] = d_p;
        }
        VGC_CUDA_OK(launch_kernel(sqgrad_repack, dim3(blocks_for((size_t)B * ((size_t)C * H * Wx > (size_t)Cout * Ho * Wo4 ? (size_t)C * H * Wx : (size_t)Cout * Ho * Wo4)), 2 * n_layers), dim3(256), 0, st, true, jobs));
        count_launch();
        return conv_group(n_layers, xr, dr, S, B, C, H, Wx, Cout, Kh, Kw, sh, sw, ph, 1, Ho, Wo4, scale, accumulate, ws, inner, st);
    }
    if (mode != kRepackNone) {
        const bool flat = mode == kRepackFlat;
        const size_t inner = round_up(flat ? conv_workspace_plain(n_layers, 1, C, 1, 1, B * P, Cout)
                                           : conv_workspace_plain(n_layers, B, C, 1, 1, P, Cout), 256);
        const size_t x_bytes = round_up(sizeof(float) * (size_t)B * C * P, 256);
        const size_t d_bytes = flat ? round_up(sizeof(float) * (size_t)B * Cout * P, 256) : 0;
        if (ws_bytes < inner + n_layers * (x_bytes + d_bytes)) return VGC_ERR_WORKSPACE;
        const float *xr[kMaxBatch], *dr[kMaxBatch];
        RepackJobs jobs = {};
        jobs.B = B;
        int n_jobs = 0;
        for (int l = 0; l < n_layers; ++l) {
            char *base = static_cast<char *>(ws) + inner + (size_t)l * (x_bytes + d_bytes);
            float *x_r = reinterpret_cast<float *>(base), *d_r = reinterpret_cast<float *>(base + x_bytes);
            jobs.job[n_jobs++] = RepackJob{x[l], x_r, C, H * W, W, Wo, P, sh, sw, flat ? 1 : 0, Wo};
            if (flat) jobs.job[n_jobs++] = RepackJob{delta[l], d_r, Cout, P, Wo, Wo, P, 1, 1, 1, Wo};
            xr[l] = x_r;
            dr[l] = flat ? d_r : delta[l];
        }
        VGC_CUDA_OK(launch_kernel(sqgrad_repack, dim3(blocks_for((size_t)B * (flat && Cout > C ? Cout : C) * P), n_jobs), dim3(256), 0, st, true, jobs));
        count_launch();
        if (flat)
            return conv_group(n_layers, xr, dr, S, 1, C, B * P, 1, Cout, 1, 1, 1, 1, 0, 0, B * P, 1, scale, accumulate, ws,
                              inner, st);
        return conv_group(n_layers, xr, dr, S, B, C, Ho, Wo, Cout, 1, 1, 1, 1, 0, 0, Ho, Wo, scale, accumulate, ws, inner, st);
    }
    // which tiles TMA can deliver: rows of P positions with a 16-byte pitch, at least one slice long; the input
    // tile only when the im2col view is the tensor itself (1x1 kernel, stride 1, no padding)
    const bool err_tma = P >= kBK && P % 4 == 0;
    const bool in_tma = err_tma && Kh == 1 && Kw == 1 && sh == 1 && sw == 1 && ph == 0 && pw == 0;
    const int p_slices = (P + kBK - 1) / kBK;
    const int k_slices = B * p_slices;
    // three taps at a time: Kw = 3, stride 1 along w with pad 1 (then Wo == W), output width even, errors by TMA
    const int taps = (!in_tma && err_tma && Kw == 3 && sw == 1 && sh == 1 && pw == 1 && Wo == W && W % 2 == 0)
                         ? (W % 4 == 0 ? 4 : 2) : 0;
    // the same with stride 2 along w: W == 2 Wo, output width even
    const int taps_s2 = (!in_tma && err_tma && Kw == 3 && sw == 2 && pw == 1 && W == 2 * Wo && Wo % 2 == 0)
                            ? (Wo % 4 == 0 ? 4 : 2) : 0;
    // seven taps at a time: Kw = 7, stride 2, pad 3
    const bool taps7 = !in_tma && err_tma && Kw == 7 && sw == 2 && pw == 3 && W == 2 * Wo && Wo % 4 == 0;
    // with few output channels the roles are swapped -- except in the three-tap form, where keeping the errors as
    // the A operand (in tensor memory, half of its rows unused) measures faster than both operands in shared memory
    const bool swapped = conv_swapped(Cout, n_im2col) && !taps && !taps_s2 && !taps7;
    // both tiles by TMA: A in tensor memory, cross terms in bf16 (the per-example form keeps tf32 cross terms)
    const bool tma_bf = err_tma && in_tma && !t_exact;
    const int rows_err = swapped ? kBN : kBM, rows_in = swapped ? kBM : kBN;
    Batch bt = {};
    uint32_t tx_err = 0, tx_in = 0;
    for (int l = 0; l < n_layers; ++l) {
        CUtensorMap *m_err = swapped ? &bt.b[l] : &bt.a[l], *m_in = swapped ? &bt.a[l] : &bt.b[l];
        if (err_tma) {
            const cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)(Cout < rows_err ? Cout : rows_err), 1};
            const cuuint64_t dims[3] = {(cuuint64_t)P, (cuuint64_t)Cout, (cuuint64_t)B};
            const cuuint64_t str[2] = {(cuuint64_t)P * 4, (cuuint64_t)Cout * P * 4};
            if (!make_map(m_err, delta[l], 3, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B)) return VGC_ERR_CUDA;
            tx_err = box[1] * kBK * 4;
        }
        if (in_tma) {
            const cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)(C < rows_in ? C : rows_in), 1};
            const cuuint64_t dims[3] = {(cuuint64_t)P, (cuuint64_t)C, (cuuint64_t)B};
            const cuuint64_t str[2] = {(cuuint64_t)P * 4, (cuuint64_t)C * P * 4};
            if (!make_map(m_in, x[l], 3, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B)) return VGC_ERR_CUDA;
            tx_in = box[1] * kBK * 4;
        }
        bt.x[l] = x[l]; bt.delta[l] = delta[l]; bt.S[l] = S[l];
    }
    Params prm = {};
    prm.p_slices = p_slices; prm.tx_bytes = tx_err + tx_in; prm.scale = scale;
    prm.tx_bytes_a = swapped ? tx_in : tx_err; prm.accumulate = accumulate;
    prm.C = C; prm.H = H; prm.W = W; prm.Cout = Cout; prm.Kh = Kh; prm.Kw = Kw; prm.sh = sh; prm.sw = sw;
    prm.ph = ph; prm.pw = pw; prm.Wo = Wo; prm.P = P;
    prm.chw = C * H * W;
    prm.wo_magic = (unsigned)(0x100000000ull / (unsigned)Wo) + 1u;
    const bool ex = t_exact;
    const int unit = ex ? p_slices : 1;
    KernelFn fn = nullptr;
#define VGC_TC_FN(A, B_, AT) (ex ? (KernelFn)sqgrad_tc<kMajorK, A, B_, AT, true> : (KernelFn)sqgrad_tc<kMajorK, A, B_, AT, false>)
    if (!swapped) {     // S[o][idx]: m = o, n = idx
        prm.ld_m = n_im2col; prm.ld_n = 1;
        // wide tiles where they are fewer than narrow ones: a slice of one takes about 1750 cycles, of the other 1390 - 1500,
        // for 1.5 times the columns (B200, one call: 128 channels 28 x 28, batch 32: 47.9 -> 43.0 us; all of ResNet-50,
        // batch 32: 2167 -> 2020 us).  The wide per-example form adds an example's sums up within one accumulator run.
        const bool any_taps = taps || taps_s2 || taps7;
        const bool wide = any_taps && (n_im2col + kWideN - 1) / kWideN < (n_im2col + kBN - 1) / kBN && (!ex || p_slices <= kChunk);
#define VGC_TAPS_FN(B_) (wide ? (ex ? (KernelFn)sqgrad_tc<kMajorK, kTma, B_, true, true, false, kWideN>                          \
                                    : (KernelFn)sqgrad_tc<kMajorK, kTma, B_, true, false, true, kWideN>)                         \
                              : VGC_TC_FN(kTma, B_, true))
        if (any_taps) {
            if (taps) fn = taps == 4 ? VGC_TAPS_FN(kGatherTaps4) : VGC_TAPS_FN(kGatherTaps2);
            else if (taps_s2) fn = taps_s2 == 4 ? VGC_TAPS_FN(kGatherTaps4S2) : VGC_TAPS_FN(kGatherTaps2S2);
            else fn = VGC_TAPS_FN(kGatherTaps7S2);
            return tc_launch(fn, bt, n_layers, prm, Cout, n_im2col, k_slices, ws, ws_bytes, st, unit, wide ? kWideN : kBN);
        }
#undef VGC_TAPS_FN
        if (tma_bf) fn = sqgrad_tc<kMajorK, kTma, kTma, true, false, true>;
        else if (err_tma && in_tma) fn = sqgrad_tc<kMajorK, kTma, kTma, true, true>;
        else if (err_tma) fn = VGC_TC_FN(kTma, kGatherIm2col, true);
        else fn = VGC_TC_FN(kGatherErr, kGatherIm2col, false);
        return tc_launch(fn, bt, n_layers, prm, Cout, n_im2col, k_slices, ws, ws_bytes, st, unit);
    }
    prm.ld_m = 1; prm.ld_n = n_im2col;   // m = idx, n = o
    if (tma_bf) fn = sqgrad_tc<kMajorK, kTma, kTma, true, false, true>;
    else if (err_tma && in_tma) fn = sqgrad_tc<kMajorK, kTma, kTma, true, true>;
    else if (err_tma) fn = VGC_TC_FN(kGatherIm2col, kTma, false);
    else fn = VGC_TC_FN(kGatherIm2col, kGatherErr, false);
#undef VGC_TC_FN
    return tc_launch(fn, bt, n_layers, prm, n_im2col, Cout, k_slices, ws, ws_bytes, st, unit);
}

// n_layers layers of one geometry; x, delta, S are host arrays of device pointers
vgc_status tc_sqgrad_conv(int n_layers, const float *const *x, const float *const *delta, float *const *S, int B, int C,
                          int H, int W, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int Ho, int Wo,
                          float scale, int accumulate, void *ws, size_t ws_bytes, cudaStream_t st, bool exact)
{
    ExactScope scope(exact);
    for (int l0 = 0; l0 < n_layers; l0 += kMaxBatch) {
        const int nl = n_layers - l0 < kMaxBatch ? n_layers - l0 : kMaxBatch;
        const vgc_status rc = conv_group(nl, x + l0, delta + l0, S + l0, B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, Ho, Wo,
                                         scale, accumulate, ws, ws_bytes, st);
        if (rc != VGC_OK) return rc;
    }
    return VGC_OK;
}

}  // namespace vgc
