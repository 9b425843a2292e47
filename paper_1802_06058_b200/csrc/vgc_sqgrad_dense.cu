// Squared per-example gradient sums of a dense layer whose reduction is short (up to 512 examples), on the tensor cores:
//
//   S[m][n] (+)= scale * sum_z delta[z][m]^2 * x[z][n]^2
//
// With few examples the result is what costs: a 128 x 128 tile is one to sixteen 32-deep slices of work and 64 KB to write
// (64 KB more to read when it is added to what is there).  The general kernel drains a tile through registers into
// row-by-row accesses of global memory, 17 us a tile for 64 examples; here the tile leaves (and the old one arrives) by TMA:
//   warp 0       one thread: TMA loads of the operand slices (A plain, B MN-major with the 128-byte swizzle of 32-byte units)
//   warp 1       one thread: 12 tcgen05.mma per slice (3xTF32: hi hi + hi lo + lo hi, A from tensor memory), or 8 (hi lo and lo hi
//                with bf16 copies)
//   warps 2-9    square and split, two groups of four on alternate slices: A into tensor memory (a lane per row: 32 loads of
//                neighbouring floats), B in place with its lo part (or bf16 copies of both parts) beside it
//   the others   epilogue: 32 x 32 boxes, one accumulator row per lane, through a shared-memory buffer of their own; the
//                box's old contents were loaded by TMA while the tile before was written, the result is stored by TMA
// An accumulator takes at most 8 slices (96 instructions: the bias of the tensor core's truncating accumulation is about
// 1.3e-8 of the sum per instruction); a tile uses one or both of the two accumulators, added by the epilogue.
//
// Bound: the pipeline's round trip per slice, shared-memory bandwidth (416 KB a tile of 64 examples) and HBM: 8 bytes per
// weight when S is added to, 4 when it is written.  Measured (B200, one call among others): 64 examples, 25088 x 4096 added
// to: 741 -> 178 us (822 MB, 0.70 of the measured copy rate); 4096 x 4096 written: 81 -> 19.8; 128 examples, 1024 x 1024:
// 14.5 -> 6.4; 512 examples, 2048 x 2048: 43 -> 29.
#include <type_traits>

#include "vgc_tc.cuh"

namespace vgc {
namespace dense {

using namespace tc;

constexpr int kRawSlots = 3, kLoSlots = 4;           // [A raw][B raw / hi]; [B lo] and the A slots in tensor memory
constexpr int kTransformWarps = 8;
constexpr uint32_t kTileBytes = kBM * kBK * 4;                      // 16 KB: one operand of one slice
constexpr uint32_t kStageBytes = 2 * kTileBytes;
constexpr uint32_t kBfBytes = kTileBytes / 2;                       // a bf16 copy of B; a lo slot takes two, [hi][lo]
constexpr uint32_t kLoBase = kRawSlots * kStageBytes;
constexpr uint32_t kBoxBase = kLoBase + kLoSlots * kTileBytes;
constexpr uint32_t kBoxBytes = 32 * 32 * 4;
constexpr uint32_t kSmemBytes = kBoxBase + kBM * kBN * 4 + 1024 /*align*/;
constexpr int kAccumulators = 2, kChunk = 8;                         // slices per accumulator
constexpr uint32_t kTmemA = kAccumulators * kBN, kTmemColsA = 64;    // A slots: 32 columns hi, 32 columns lo (16 hi as bf16, 16 lo as bf16)
constexpr uint32_t kTmemCols = kTmemA + kLoSlots * kTmemColsA;
static_assert(kTmemCols == 512, "tensor memory");
// Epilogue warps: with eight (two halves of the columns per lane quarter) a written tile leaves sooner (4096 x 4096, 16
// examples: 15.0 us against 19.9); an added one needs the longer lead that four buffers per warp give its loads (25088 x
// 4096, 64 examples: 178 us with four warps, 199 with eight).
// kN: columns of a tile, 128 or (layers of few tiles) 64.
template <bool kAccumulate, int kN> struct Shape {
    static constexpr int kHalves = kAccumulate ? 1 : 2, kEpilogueWarps = 4 * kHalves, kBoxes = kN / 32 / kHalves;
    static constexpr int kThreads = 32 * (2 + kTransformWarps + kEpilogueWarps);
};

// Where the bf16 copy of the raw tile's i-th 16 bytes goes.  Raw: boxes of 32 columns, 128 bytes a row k, whose 32-byte units were put
// in place unit ^ (k & 3).  Copy: blocks of 64 columns, 128 bytes a row, 16-byte units in place unit ^ (k & 7).
__device__ __forceinline__ uint32_t bf_place(uint32_t i)
{
    const uint32_t k = (i >> 3) & 31u, n = 32 * (i >> 8) + 8 * (((i >> 1) ^ k) & 3u) + 4 * (i & 1u);
    return (n >> 6) * 4096u + k * 128u + (((n >> 3) ^ k) & 7u) * 16u + (n & 4u) * 2u;
}

struct Params {
    int k_slices, tiles, tiles_x;
    float scale;
    uint32_t *status;
    const float *x, *delta;
    int examples, in, out;
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int kLeft>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kLeft) : "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// kFew: fewer than 32 examples (see the epilogue; the check costs an added layer 6 %, so it is compiled for these only)
// kBf: the two cross terms take bf16 copies of hi and lo, 16 deep an instruction: a third fewer instructions and so less of the
// accumulator's bias, but their rounding shows in sums of few terms: largest error, of 1024 x 1024 to 2048 x 2048 sums and 4096 x 1024,
// squares of normals (of positive parts of normals), in tf32 / with bf16: 64 examples 1.7e-6 / 2.9e-6; 192 4.1e-6 / 4.0e-6 (3.7e-6 / 3.9e-6);
// 256, a whole run of the accumulator, 5.1e-6 / 4.6e-6 (4.6e-6 / 4.3e-6); 512 4.5e-6 / 4.0e-6 (3.8e-6 / 3.7e-6).  Hence from kBfLeast examples
// on (512 examples, 2048 x 2048: 27.9 -> 26.0 us; 256 examples, 1024 x 1024: 9.4 -> 8.7).
constexpr int kBfLeast = 256;
template <bool kAccumulate, int kN, bool kFew, bool kBf>
__global__ void __launch_bounds__(Shape<kAccumulate, kN>::kThreads, 1)
sqgrad_dense(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
             const __grid_constant__ CUtensorMap map_s, const Params prm)
{
    constexpr int kEpilogueWarps = Shape<kAccumulate, kN>::kEpilogueWarps, kBoxes = Shape<kAccumulate, kN>::kBoxes;
    constexpr uint32_t kBytesB = kN * kBK * 4;
    extern __shared__ uint8_t smem_raw_[];
    __shared__ __align__(8) uint64_t bars[3 * kRawSlots + 2 * kAccumulators + 1];
    __shared__ __align__(8) uint64_t box_full[kEpilogueWarps][kBoxes];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile uint32_t abort_flag;

    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = (smem_u32(smem_raw_) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw_ + (smem_base - smem_u32(smem_raw_));
    uint64_t *raw_full = bars, *op_full = bars + kRawSlots, *empty = bars + 2 * kRawSlots;
    uint64_t *acc_full = bars + 3 * kRawSlots, *acc_empty = acc_full + kAccumulators, *drain = acc_empty + kAccumulators;

    grid_release();
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < kRawSlots; ++i) {
            mbar_init(smem_u32(&raw_full[i]), 1);
            mbar_init(smem_u32(&op_full[i]), 4);
            mbar_init(smem_u32(&empty[i]), 1);
        }
        for (int i = 0; i < kAccumulators; ++i) {
            mbar_init(smem_u32(&acc_full[i]), 1);
            mbar_init(smem_u32(&acc_empty[i]), kEpilogueWarps);
        }
        mbar_init(smem_u32(drain), 1);
        for (int e = 0; e < kEpilogueWarps; ++e)
            for (int j = 0; j < kBoxes; ++j) mbar_init(smem_u32(&box_full[e][j]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    if (threadIdx.x == 0) { prefetch_map(&map_a); prefetch_map(&map_b); prefetch_map(&map_s); }
    grid_wait();

    const int k_slices = prm.k_slices, step = (int)gridDim.x, first_tile = (int)blockIdx.x;
    if (warp == 0) {
        // ================= TMA producer (one thread) =================
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int t = first_tile; ok && t < prm.tiles; t += step) {
                const int ty = t / prm.tiles_x, m0 = ty * kBM, n0 = (t - ty * prm.tiles_x) * kN;
                for (int s = 0; s < k_slices; ++s, ++it) {
                    const int st = it % kRawSlots;
                    if (!mbar_wait(smem_u32(&empty[st]), ((uint32_t)(it / kRawSlots) & 1u) ^ 1u, &abort_flag, 32)) { ok = false; break; }
                    const uint32_t full = smem_u32(&raw_full[st]), dst = smem_base + (uint32_t)st * kStageBytes;
                    mbar_expect_tx(full, kTileBytes + kBytesB);
#pragma unroll
                    for (int j = 0; j < 4; ++j) tma_load_2d(dst + j * 4096, &map_a, full, m0 + 32 * j, s * kBK);
#pragma unroll
                    for (int j = 0; j < kN / 32; ++j) tma_load_2d(dst + kTileBytes + j * 4096, &map_b, full, n0 + 32 * j, s * kBK);
                }
            }
            if (abort_flag) {                            // loads already issued must land before the block may exit
                for (int i = it > kRawSlots ? it - kRawSlots : 0; i < it; ++i)
                    for (uint32_t n = 0; n < kWaitLimit && !mbar_try(smem_u32(&raw_full[i % kRawSlots]), (uint32_t)(i / kRawSlots) & 1u); ++n) {}
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (one thread) =================
        if (lane == 0) {
            // B MN-major: 32-wide column blocks 4096 B apart (LBO), 4-deep k groups 512 B apart (SBO), 8-deep steps 1024 B
            const uint32_t desc_hi = (uint32_t)(smem_desc(0, 4096u, 512u, 1u) >> 32);
            const uint32_t desc_lo0 = (uint32_t)smem_desc(0, 4096u, 512u, 1u);
            auto desc_at = [&](uint32_t lo16) -> uint64_t { return ((uint64_t)desc_hi << 32) | (desc_lo0 + lo16); };
            const uint32_t idesc = instr_desc(kMajorK, kN, kBM) | (1u << 16);        // A K-major (tensor memory), B MN-major
            // the bf16 copies: 64-wide column blocks 4096 B apart (LBO), 8-deep k groups 1024 B apart (SBO), 128-byte swizzle
            const uint32_t bf_hi = (uint32_t)(smem_desc(0, 4096u, 1024u, 2u) >> 32), bf_lo0 = (uint32_t)smem_desc(0, 4096u, 1024u, 2u);
            auto desc_bf = [&](uint32_t lo16) -> uint64_t { return ((uint64_t)bf_hi << 32) | (bf_lo0 + lo16); };
            const uint32_t idesc_bf = instr_desc_bf16(kN, kBM) | (1u << 16);
            int it = 0, c = 0;                           // running numbers of the slice and of the chunk
            bool ok = true;
            for (int t = first_tile; ok && t < prm.tiles; t += step) {
                for (int s0 = 0; ok && s0 < k_slices; s0 += kChunk, ++c) {
                    const int b = c % kAccumulators;
                    ok = mbar_wait(smem_u32(&acc_empty[b]), ((uint32_t)(c / kAccumulators) & 1u) ^ 1u, &abort_flag, 0);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)b * kBN;
                    const int s1 = min(k_slices, s0 + kChunk);
                    for (int s = s0; s < s1; ++s, ++it) {
                        const int st = it % kRawSlots, ls = it % kLoSlots;
                        ok = mbar_wait(smem_u32(&op_full[st]), (uint32_t)(it / kRawSlots) & 1u, &abort_flag, 0);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t hi_b = (smem_base + (uint32_t)st * kStageBytes + kTileBytes) >> 4;
                        const uint32_t lo_b = (smem_base + kLoBase + (uint32_t)ls * kTileBytes) >> 4;
                        const uint32_t ta = tmem_base + kTmemA + (uint32_t)ls * kTmemColsA;
#pragma unroll
                        for (int kk = 0; kk < kBK / 8; ++kk) {
                            const uint64_t db_hi = desc_at(hi_b + kk * 64), db_lo = desc_at(lo_b + kk * 64);
                            if (kk == 0) tc_mma_tf32_ts(d_tmem, ta, db_hi, idesc, s == s0 ? 0u : 1u);
                            else tc_mma_tf32_ts_acc(d_tmem, ta + kk * 8, db_hi, idesc);
                            if (kBf) continue;
                            tc_mma_tf32_ts_acc(d_tmem, ta + kk * 8, db_lo, idesc);
                            tc_mma_tf32_ts_acc(d_tmem, ta + 32 + kk * 8, db_hi, idesc);
                        }
                        if constexpr (kBf) {
#pragma unroll
                            for (int kk = 0; kk < kBK / 16; ++kk) {
                                tc_mma_bf16_ts_acc(d_tmem, ta + 32 + kk * 8, desc_bf(lo_b + (kBfBytes >> 4) + kk * 128), idesc_bf);
                                tc_mma_bf16_ts_acc(d_tmem, ta + 48 + kk * 8, desc_bf(lo_b + kk * 128), idesc_bf);
                            }
                        }
                        tc_commit(smem_u32(&empty[st]));
                    }
                    if (ok) tc_commit(smem_u32(&acc_full[b]));
                }
            }
            if (!ok) {                                   // MMAs already issued must retire before tensor memory is freed
                tc_commit(smem_u32(drain));
                for (uint32_t n = 0; n < kWaitLimit && !mbar_try(smem_u32(drain), 0); ++n) {}
            }
        }
    } else if (warp < 2 + kTransformWarps) {
        // ================= transform: square and split =================
        const int tt = (int)(threadIdx.x - 64) & 127, group = (int)(threadIdx.x - 64) >> 7;
        const int my_tiles = first_tile < prm.tiles ? (prm.tiles - first_tile - 1) / step + 1 : 0;
        const int total = my_tiles * k_slices;
        for (int i = group; i < total; i += 2) {
            const int st = i % kRawSlots, ls = i % kLoSlots;
            // the slot's user before, slice i - kRawSlots, belongs to the other group: its phase has to be over before the
            // parity of raw_full says anything about slice i
            if (!mbar_wait(smem_u32(&empty[st]), ((uint32_t)(i / kRawSlots) & 1u) ^ 1u, &abort_flag)) break;
            if (!mbar_wait(smem_u32(&raw_full[st]), (uint32_t)(i / kRawSlots) & 1u, &abort_flag)) break;
            // (the lo slots' previous user, slice i - kLoSlots, has retired as well)
            static_assert(kLoSlots >= kRawSlots, "no wait of its own for a lo slot");
            tc_fence_after();
            const uint32_t q = warp & 3;                 // lane quarter of tensor memory = 32-row block of the A tile
            const float *a_raw = reinterpret_cast<const float *>(smem_gen + (uint32_t)st * kStageBytes + q * 4096) + lane;
            const uint32_t ta = tmem_base + ((q * 32u) << 16) + kTmemA + (uint32_t)ls * kTmemColsA;
#pragma unroll
            for (int k0 = 0; k0 < kBK; k0 += 16) {
                float e[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) e[k] = a_raw[(k0 + k) * 32];
                uint32_t h[16], l[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const float sq = __fmul_rn(e[k], e[k]);
                    h[k] = to_tf32(sq);
                    l[k] = __float_as_uint(__fsub_rn(sq, __uint_as_float(h[k])));
                }
                tc_st_32x16(ta + k0, h);
                if constexpr (kBf) {
                    uint32_t hb[8], lb[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        hb[k] = pack_bf16(__uint_as_float(h[2 * k]), __uint_as_float(h[2 * k + 1]));
                        lb[k] = pack_bf16(__uint_as_float(l[2 * k]), __uint_as_float(l[2 * k + 1]));
                    }
                    tc_st_32x8(ta + 32 + k0 / 2, hb);
                    tc_st_32x8(ta + 48 + k0 / 2, lb);
                } else {
                    tc_st_32x16(ta + 32 + k0, l);
                }
            }
            uint8_t *hi = smem_gen + (uint32_t)st * kStageBytes + kTileBytes, *lo = smem_gen + kLoBase + (uint32_t)ls * kTileBytes;
#pragma unroll
            for (int u0 = 0; u0 < (int)(kBytesB / 16 / 128); u0 += 4) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const float4 *>(hi + 16 * (tt + (u0 + u) * 128));
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = (uint32_t)(tt + (u0 + u) * 128);
                    if (!kBf) { split_store<true>(hi, lo, 16 * i, v[u].x, v[u].y, v[u].z, v[u].w); continue; }
                    const float e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                    uint32_t h[4], l[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float sq = __fmul_rn(e[j], e[j]);
                        h[j] = to_tf32(sq);
                        l[j] = __float_as_uint(__fsub_rn(sq, __uint_as_float(h[j])));
                    }
                    *reinterpret_cast<uint4 *>(hi + 16 * i) = make_uint4(h[0], h[1], h[2], h[3]);
                    uint8_t *const bf = lo + bf_place(i);
                    *reinterpret_cast<uint2 *>(bf) = make_uint2(pack_bf16(__uint_as_float(h[0]), __uint_as_float(h[1])), pack_bf16(__uint_as_float(h[2]), __uint_as_float(h[3])));
                    *reinterpret_cast<uint2 *>(bf + kBfBytes) = make_uint2(pack_bf16(__uint_as_float(l[0]), __uint_as_float(l[1])), pack_bf16(__uint_as_float(l[2]), __uint_as_float(l[3])));
                }
            }
            tc_wait_st();
            tc_fence_before();
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&op_full[st]));
        }
    } else {
        // ================= epilogue =================
        const uint32_t q = warp & 3;                     // lane quarter of tensor memory
        const uint32_t e = warp - (2 + kTransformWarps), first_col = (e >> 2) * kBoxes * 32;
        const uint32_t box0 = smem_base + kBoxBase + e * kBoxes * kBoxBytes;
        uint8_t *const box_gen = smem_gen + kBoxBase + e * kBoxes * kBoxBytes;
        auto load_box = [&](int t, int j) {              // old contents of box j of tile t; lane 0
            const int ty = t / prm.tiles_x;
            const uint32_t full = smem_u32(&box_full[e][j]);
            mbar_expect_tx(full, kBoxBytes);
            tma_load_2d(box0 + j * kBoxBytes, &map_s, full, (t - ty * prm.tiles_x) * kN + (int)first_col + 32 * j, ty * kBM + 32 * (int)q);
        };
        int waited[kBoxes] = {};                         // loads of box j waited for (lane 0: for an abort)
        if (kAccumulate && lane == 0 && first_tile < prm.tiles)
            for (int j = 0; j < kBoxes; ++j) load_box(first_tile, j);
        const int chunks = (k_slices + kChunk - 1) / kChunk;          // 1 or 2 accumulators per tile
        int c = 0;                                       // running number of the tile
        bool ok = true;
        for (int t = first_tile; ok && t < prm.tiles; t += step, ++c) {
            const int ty = t / prm.tiles_x, m0 = ty * kBM + 32 * (int)q, n0 = (t - ty * prm.tiles_x) * kN + (int)first_col;
            const int a0 = c * chunks, b = a0 % kAccumulators;
            for (int i = 0; ok && i < chunks; ++i)
                ok = mbar_wait(smem_u32(&acc_full[(a0 + i) % kAccumulators]), (uint32_t)((a0 + i) / kAccumulators) & 1u, &abort_flag, 32);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((q * 32u) << 16) + first_col;
#pragma unroll
            for (int j = 0; j < kBoxes; ++j) {
                uint32_t r[32];
                tc_ld_32x32(taddr + (uint32_t)b * kBN + 32 * j, r);
                if (kAccumulate) {
                    if (!mbar_wait(smem_u32(&box_full[e][j]), (uint32_t)c & 1u, &abort_flag, 32)) ok = false;
                    else ++waited[j];
                } else {                                 // the box's last store has been read out
                    if (lane == 0) bulk_wait_read<kBoxes - 1>();
                    __syncwarp();
                }
                tc_wait_ld();
                if (!ok) break;
                if (chunks > 1) {
                    uint32_t r2[32];
                    tc_ld_32x32(taddr + (uint32_t)(b ^ 1) * kBN + 32 * j, r2);
                    tc_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__fadd_rn(__uint_as_float(r[i]), __uint_as_float(r2[i])));
                }
                // Fewer examples than the general tensor-core kernel takes: a layer is infinite where a square or a sum is, as
                // on the CUDA cores.  The three products make NaN of that (infinity times a zero low part, infinity minus
                // infinity), so what comes out NaN is summed again in plain fp32.
                uint32_t top = 0;                        // (sums of squares: NaN is what lies above infinity's bits)
                if (kFew) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) top = max(top, r[i]);
                }
                if (kFew && top > 0x7F800000u) {
                    uint32_t nan = 0;
#pragma unroll
                    for (int i = 0; i < 32; ++i) nan |= (__uint_as_float(r[i]) != __uint_as_float(r[i]) ? 1u : 0u) << i;
                    const int m = m0 + (int)lane;
                    while (nan) {
                        const int at = __ffs(nan) - 1, n = n0 + 32 * j + at;
                        nan &= nan - 1u;
                        float sum = 0.f;
                        for (int z = 0; z < prm.examples && m < prm.out && n < prm.in; ++z) {
                            const float d = prm.delta[(size_t)z * prm.out + m], v = prm.x[(size_t)z * prm.in + n];
                            sum = fmaf(__fmul_rn(d, d), __fmul_rn(v, v), sum);
                        }
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (i == at) r[i] = __float_as_uint(sum);
                    }
                }
                if (kFew) __syncwarp();
                uint8_t *const row = box_gen + j * kBoxBytes + lane * 128;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    float4 *const at = reinterpret_cast<float4 *>(row + ((u ^ (lane & 7)) << 4));
                    float4 v = make_float4(__fmul_rn(prm.scale, __uint_as_float(r[4 * u])), __fmul_rn(prm.scale, __uint_as_float(r[4 * u + 1])),
                                           __fmul_rn(prm.scale, __uint_as_float(r[4 * u + 2])), __fmul_rn(prm.scale, __uint_as_float(r[4 * u + 3])));
                    if (kAccumulate) {
                        const float4 old = *at;
                        v.x = __fadd_rn(old.x, v.x); v.y = __fadd_rn(old.y, v.y);
                        v.z = __fadd_rn(old.z, v.z); v.w = __fadd_rn(old.w, v.w);
                    }
                    *at = v;
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&map_s, box0 + j * kBoxBytes, n0 + 32 * j, m0);      // parts past the edges are clipped
                    if (kAccumulate) {
                        // the box stored before this one is free once that store has been read out: its next contents
                        const int tp = j > 0 ? t + step : t, jp = j > 0 ? j - 1 : kBoxes - 1;
                        if ((j > 0 || c > 0) && tp < prm.tiles) {
                            bulk_wait_read<1>();
                            load_box(tp, jp);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (ok && lane == 0)
                for (int i = 0; i < chunks; ++i) mbar_arrive(smem_u32(&acc_empty[(a0 + i) % kAccumulators]));
        }
        if (lane == 0) {
            if (!ok && kAccumulate) {                    // loads in flight must land before the block may exit
                for (int j = 0; j < kBoxes; ++j)
                    for (uint32_t n = 0; n < kWaitLimit && !mbar_try(smem_u32(&box_full[e][j]), (uint32_t)waited[j] & 1u); ++n) {}
            }
            bulk_wait_all();
        }
    }

    // ---- common exit ----
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicOr(prm.status, VGC_DEV_TIMEOUT);
}

}  // namespace dense

// 16-byte row pitches for TMA; the reduction fits the accumulators (fewer examples than a slice is deep: zeros)
bool dense_supported(int B, int in, int out)
{
    return B >= 1 && B <= dense::kAccumulators * dense::kChunk * tc::kBK && in % 4 == 0 && out % 4 == 0;
}

vgc_status dense_sqgrad_linear(const float *x, const float *delta, int B, int in, int out, float scale, int accumulate,
                               float *S, void *ws, cudaStream_t st)
{
    using namespace dense;
    CUtensorMap map_a, map_b, map_s;
    const cuuint32_t box[2] = {32, (cuuint32_t)kBK}, box_s[2] = {32, 32};
    const cuuint64_t dims_a[2] = {(cuuint64_t)out, (cuuint64_t)B}, str_a[1] = {(cuuint64_t)out * 4};
    const cuuint64_t dims_b[2] = {(cuuint64_t)in, (cuuint64_t)B}, str_b[1] = {(cuuint64_t)in * 4};
    const cuuint64_t dims_s[2] = {(cuuint64_t)in, (cuuint64_t)out};
    if (!make_map(&map_a, delta, 2, dims_a, str_a, box, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map(&map_b, x, 2, dims_b, str_b, box, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B) ||
        !make_map(&map_s, S, 2, dims_s, str_b, box_s, CU_TENSOR_MAP_SWIZZLE_128B))
        return VGC_ERR_CUDA;
    // 64 columns where tiles of 128 leave half of the SMs idle: half of B's transform and of the result per block
    // (128 examples, 1024 x 1024: 7.2 -> 6.4 us; from there on it is the slices one after another, twelve instructions of about
    // 100 cycles whatever their columns: rings of twice the depth changed nothing)
    const long long rows_m = (out + kBM - 1) / kBM;
    const bool narrow = rows_m * ((in + kBN - 1) / kBN) <= 74;
    const int tile_n = narrow ? 64 : kBN;
    auto pick = [&](auto few, auto bf) {
        constexpr bool kFew = decltype(few)::value, kBf = decltype(bf)::value;
        return accumulate ? (narrow ? sqgrad_dense<true, 64, kFew, kBf> : sqgrad_dense<true, kBN, kFew, kBf>)
                          : (narrow ? sqgrad_dense<false, 64, kFew, kBf> : sqgrad_dense<false, kBN, kFew, kBf>);
    };
    const std::true_type yes;
    const std::false_type no;
    auto fn = B < 32 ? pick(yes, no) : B < kBfLeast ? pick(no, no) : pick(no, yes);
    VGC_CUDA_OK(allow_dynamic_smem(reinterpret_cast<const void *>(fn), kSmemBytes));
    Params prm;
    prm.k_slices = (B + kBK - 1) / kBK;
    prm.tiles_x = (in + tile_n - 1) / tile_n;
    const long long tiles = (long long)prm.tiles_x * rows_m;
    if (tiles >= (1LL << 26)) return VGC_ERR_UNSUPPORTED;
    prm.tiles = (int)tiles;
    prm.scale = scale;
    prm.status = static_cast<uint32_t *>(ws);
    prm.x = x; prm.delta = delta; prm.examples = B; prm.in = in; prm.out = out;
    // as few rounds as there have to be, of equal length
    const int rounds = (prm.tiles + 147) / 148, blocks = (prm.tiles + rounds - 1) / rounds;
    const int threads = accumulate ? Shape<true, kBN>::kThreads : Shape<false, kBN>::kThreads;
    VGC_CUDA_OK(launch_kernel(fn, dim3((unsigned)blocks), dim3((unsigned)threads), kSmemBytes, st, true, map_a, map_b, map_s, prm));
    count_launch();
    return VGC_OK;
}

}  // namespace vgc
