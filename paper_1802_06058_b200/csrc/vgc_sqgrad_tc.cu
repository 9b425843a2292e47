// Squared per-example gradient sums on the tensor cores: the pass that adds partial tiles, the repacking pre-pass, planning and
// launches.  The kernel is in vgc_sqgrad_tc.cuh.
#include <atomic>
#include <cstdlib>

#include "vgc_sqgrad_tc.cuh"

namespace vgc {

namespace tc {

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
                  int tile_n, int slot_n, int tiles_x, int tiles_y, int M, int N, float scale, int accumulate, const ResultPtrs results,
                  long long ld_m, long long ld_n)
{
    __shared__ float patch[32][33];
    grid_release();
    const int tile = blockIdx.x / (slot_n >> 3), sub = blockIdx.x - tile * (slot_n >> 3);
    const TileParts parts(units_q, units_r, units_per_tile, tiles_x, tiles_y, (int)blockIdx.y, tile);
    const int tx = parts.tx, ty = parts.ty;
    float *S = results.S[blockIdx.y];                                      // blockIdx.y: layer of the batch
    const int r0 = (sub & 3) * 32, j0 = (sub >> 2) * 32;                  // patch origin inside the tile
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;              // lane -> row, warp -> four columns
    const size_t step = (size_t)2 * kBM * slot_n;                         // from a block's first segment to the next block's
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
        const int m = ty * kBM + r0 + lane, n_end = min(N, (tx + 1) * tile_n);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int n = tx * tile_n + j0 + 4 * w + c;
            if (m < M && n < n_end) {
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
        const int m = ty * kBM + r0 + r, n = tx * tile_n + j0 + c0, n_end = min(N, (tx + 1) * tile_n);
        if (m < M) {
            float *dst = S + (size_t)m * ld_m + n;
            if (((ld_m | n) & 3) == 0 && n + 3 < n_end) {
                float4 out = make_float4(patch[c0][r], patch[c0 + 1][r], patch[c0 + 2][r], patch[c0 + 3][r]);
                if (accumulate) out = add4(*reinterpret_cast<const float4 *>(dst), out);
                *reinterpret_cast<float4 *>(dst) = out;
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (n + c < n_end) dst[c] = accumulate ? __fadd_rn(dst[c], patch[c0 + c][r]) : patch[c0 + c][r];
            }
        }
    }
}

// The same for tiles that many blocks worked on: a thread block per 32 rows x 4 columns, the partial tiles dealt out to its
// eight warps in turn and their sums added in the order of the warps (a fixed order as well).  A chain of 148 partial tiles
// took 22 us in the kernel above.
__global__ void __launch_bounds__(256)
sqgrad_tc_combine_many(const float *partial, int units_q, int units_r, int units_per_tile,
                       int tile_n, int slot_n, int tiles_x, int tiles_y, int M, int N, float scale, int accumulate, const ResultPtrs results,
                       long long ld_m, long long ld_n)
{
    __shared__ float sums[8][4][32];
    grid_release();
    const int tile = blockIdx.x / slot_n, sub = blockIdx.x - tile * slot_n;
    const TileParts parts(units_q, units_r, units_per_tile, tiles_x, tiles_y, (int)blockIdx.y, tile);
    const int r0 = (sub & 3) * 32, j0 = (sub >> 2) * 4;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // thread of the first four warps: one element of the patch, lanes along whichever of m / n has unit stride; its old
    // content is on its way during the sums
    const int row = ld_m == 1 ? lane : 8 * w + (lane >> 2), col = ld_m == 1 ? w : lane & 3;
    const int m = parts.ty * kBM + r0 + row, n = parts.tx * tile_n + j0 + col;
    const bool mine = w < 4 && m < M && n < min(N, (parts.tx + 1) * tile_n);
    float *const dst = results.S[blockIdx.y] + (size_t)m * ld_m + (size_t)n * ld_n;
    const size_t step = (size_t)2 * kBM * slot_n;
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

// Examples cut into parts: S = scale * sum_z (sum of the example's parts)^2.  A thread block per 32 rows x 4 columns of a tile, its
// eight warps take the examples in turn; their sums are added in the order of the warps.
__global__ void __launch_bounds__(256)
sqgrad_tc_combine_examples(const float *partial, int examples, int n_parts, int tile_n, int slot_n, int tiles_x, int tiles_y, int M, int N,
                           float scale, int accumulate, const ResultPtrs results, long long ld_m, long long ld_n)
{
    __shared__ float sums[8][4][32];
    grid_release();
    const int tile = blockIdx.x / slot_n, sub = blockIdx.x - tile * slot_n;
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const int r0 = (sub & 3) * 32, j0 = (sub >> 2) * 4;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int row = ld_m == 1 ? lane : 8 * w + (lane >> 2), col = ld_m == 1 ? w : lane & 3;
    const int m = ty * kBM + r0 + row, n = tx * tile_n + j0 + col;
    const bool mine = w < 4 && m < M && n < min(N, (tx + 1) * tile_n);
    float *const dst = results.S[blockIdx.y] + (size_t)m * ld_m + (size_t)n * ld_n;
    const size_t slot = (size_t)kBM * slot_n;
    const float *src = partial + ((size_t)blockIdx.y * tiles_x * tiles_y + tile) * examples * n_parts * slot +
                       ((size_t)(j0 / 4) * kBM + r0 + lane) * 4;
    grid_wait();
    if (ty * kBM + r0 >= M || tx * tile_n + j0 >= N) return;
    const float old = accumulate && mine ? *dst : 0.f;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z = w; z < examples; z += 8) {
        const float *at = src + (size_t)z * n_parts * slot;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int i = 0; i < n_parts; ++i) d = add4(d, __ldcs(reinterpret_cast<const float4 *>(at + (size_t)i * slot)));
        sum = add4(sum, make_float4(__fmul_rn(d.x, d.x), __fmul_rn(d.y, d.y), __fmul_rn(d.z, d.z), __fmul_rn(d.w, d.w)));
    }
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
static std::atomic<int> g_concurrent{1};

// What one call of the library goes by from its beginning to its end: plans, workspace and the kernel's form have to agree, and
// another thread may change the hint meanwhile.
struct Call {
    bool exact;              // the per-example statistic
    int concurrent;
    explicit Call(bool per_example) : exact(per_example), concurrent(g_concurrent.load(std::memory_order_relaxed)) {}
};

struct Plan {
    int M, N, k_slices, n_layers, tile_n;
    int unit, units_per_tile, blocks, tiles_x, tiles_y;
    int units_total;
    int parts, part_slices;  // examples cut up: parts of each (0: not), slices of a part
    bool partials;           // some tile is shared by several blocks: partial tiles go through the scratch
};

// How a launch's work -- n_layers x tiles x k_slices slices -- is cut into one contiguous range per block.
// `unit_min`: slices that must stay in one block (the per-example form cuts the reduction between examples only).
// Two candidates: whole tiles per block (no scratch, no second kernel, but the blocks' loads are as even as the
// tile count allows), or an even cut of the slices over all SMs (tiles at the cuts are shared, their partial
// sums combined by a second kernel).  Costs in slice times: a block's longest range, plus what the combine pass
// adds to the call: its launch and the partial tiles' round trip, kCombineSlices.  Measured over 40 convolutions and small
// networks (B200): 6 is 5 % faster than 14 (which held before launches overlapped and partial tiles left in 16-byte
// stores), up to 1.6 times (9 examples, 544 channels 14 x 14 to 48, 3x3 stride 2: 31.5 -> 19.3 us), none slower by more than the runs of
// one side differ; 10 is 2 % faster than 14, 4 as fast as 6 but for small networks (ResNet-50, 128 x 128, 3 examples: 378 -> 367).
constexpr int kCombineSlices = 4;
// The price of a combine pass where examples may be cut into parts (either candidate there ends in one).  Its blocks have a warp per
// example and few examples to share, so that many tiles take long: one example, 512 channels 32 x 32 to 300, 3 taps (72 tiles), 30.6 us in
// whole tiles, 57.8 in two parts, which a price of 4 chooses; 256 channels 24 x 24 to 16, 5 taps (34 tiles), 26.5, 25.9; 3 channels 24 x 24
// to 48, 7 taps (1 tile), 27.2, 10.4.  Of 61 such layers 4 makes 38 faster and 23 up to 1.9 times slower; no drawn size of four
// examples and more depends on it.
constexpr int kPartsCombineSlices = 14;
static Plan make_plan(const Call &call, int M, int N, int k_slices, int n_layers, int unit_min, int tile_n)
{
    Plan p;
    p.M = M; p.N = N; p.k_slices = k_slices; p.n_layers = n_layers; p.tile_n = tile_n;
    p.tiles_x = (N + tile_n - 1) / tile_n;
    p.tiles_y = (M + kBM - 1) / kBM;
    const long long tiles = (long long)p.tiles_x * p.tiles_y * n_layers;
    const long long upt = k_slices / unit_min, units = tiles * upt;
    bool even;
    long long blocks;
    if (call.concurrent > 1) {
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
        // (a block's longest range), or an even cut of all slices (plus what the combine pass adds to the call).
        const long long waves = (tiles + kSmCount - 1) / kSmCount;
        const long long blocks_a = (tiles + waves - 1) / waves;
        const long long cost_a = ((tiles + blocks_a - 1) / blocks_a) * k_slices;
        const long long blocks_b = units < kSmCount ? units : kSmCount;
        const long long cost_b = ((units + blocks_b - 1) / blocks_b) * unit_min + kCombineSlices;
        even = cost_b < cost_a;
        blocks = even ? blocks_b : blocks_a;
    }
    p.parts = p.part_slices = 0;
    if (unit_min > 1 && call.concurrent == 1) {
        // Few long examples, which the form that adds up an example's products before it squares them keeps whole, leave SMs
        // idle: parts of an example, a block each, at most two waves of them; a wave's start costs about 5 slices.
        const long long waves_now = even ? (units + blocks - 1) / blocks : ((tiles + blocks - 1) / blocks) * upt;
        long long best = waves_now * unit_min + (even ? kPartsCombineSlices : 0);
        const long long most = 2 * kSmCount / units;
        for (long long want = most < unit_min ? most : unit_min; want > 1; --want) {          // parts of ever more slices
            const int q = (int)((unit_min + want - 1) / want);
            const long long n_parts = (unit_min + q - 1) / q, n = units * n_parts;
            const long long cost = ((n + kSmCount - 1) / kSmCount) * (q + 5) + kPartsCombineSlices;
            if (cost < best) { best = cost; p.parts = (int)n_parts; p.part_slices = q; }
        }
        if (p.parts) {
            p.unit = p.part_slices;
            p.units_per_tile = (int)(upt * p.parts);
            p.units_total = (int)(units * p.parts);
            p.blocks = p.units_total;
            p.partials = true;
            return p;
        }
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
    g_concurrent.store(concurrent_launches > 1 ? concurrent_launches : 1, std::memory_order_relaxed);
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

// columns of an accumulator and of a partial tile, whatever part of them a tile uses
static int slot_columns(int tile_n) { return tile_n > kBN ? kWideN : kBN; }

static size_t tc_workspace_bytes(const Plan &p)
{
    // status word (256 bytes) + two partial tiles per block (the first and the last segment of its range)
    return 256 + (p.partials ? (size_t)(p.parts ? 1 : 2) * p.blocks * kBM * slot_columns(p.tile_n) * sizeof(float) : 0);
}

// Whether the cross terms of a layer of 192-column tiles take bf16 copies: where that loses nothing.  The copies' rounding adds up to
// 2^-18 of a product, of either sign, so that it averages out over many terms; a third fewer instructions save up to 4 x 2^-23 of the
// accumulator's truncation for every slice it runs.  From six slices a run on the second outweighs the first in the worst case.  Largest
// error of squared sums of normals (positive parts of normals), 3 and 5 taps, 1 to 128 tiles, bf16 over tf32 (B200): runs of one slice,
// 768 to 2048 terms 0.96 - 1.5 (1.12 - 2.3); of four slices, 128 terms 0.94 - 1.2 (1.09 - 1.66); of six to eight, 192 to 384 terms 0.86 - 1.02
// (0.89 - 1.16), 512 to 768 terms 0.79 - 0.88 (0.80 - 0.97), 1024 and more 0.79 - 0.88 (0.77 - 0.95).  Root mean square: 0.77 - 0.84 there.
static bool bf16_cross_better(const Plan &p, long long terms)
{
    const long long range = (long long)p.units_total / p.blocks * p.unit;         // slices of a block
    const long long run = range < p.k_slices ? range : p.k_slices;               // in one tile, the drains every kChunk apart
    return run >= 6 && terms >= 1024;
}

static vgc_status tc_launch(KernelFn kernel, const Batch &bt, const Plan &plan, Params prm, void *ws, size_t ws_bytes, cudaStream_t st)
{
    const int M = plan.M, N = plan.N, n_layers = plan.n_layers, tile_n = plan.tile_n;
    if (ws_bytes < tc_workspace_bytes(plan)) return VGC_ERR_WORKSPACE;
    VGC_CUDA_OK(allow_dynamic_smem(reinterpret_cast<const void *>(kernel), kSmemBytes, kRegsLaunch));
    prm.M = M; prm.N = N; prm.k_slices = plan.k_slices;
    prm.unit = plan.unit; prm.units_per_tile = plan.units_per_tile; prm.units_total = plan.units_total;
    prm.units_q = plan.units_total / plan.blocks; prm.units_r = plan.units_total % plan.blocks;
    prm.parts = plan.parts; prm.part_slices = plan.part_slices;
    prm.tile_n = tile_n; prm.tiles_x = plan.tiles_x; prm.tiles_y = plan.tiles_y;
    prm.chunk = kChunk;
    prm.status = static_cast<uint32_t *>(ws);
    // partial tiles are read and written 16 bytes at a time, the caller's workspace may start anywhere: the status word's 256 bytes
    // have room to round down
    prm.partial = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(ws) + 256) & ~(uintptr_t)15);
    VGC_CUDA_OK(launch_kernel(kernel, dim3((unsigned)plan.blocks), dim3(kThreadsTc), kSmemBytes, st, true, bt, prm));
    count_launch();
    if (plan.partials) {
        ResultPtrs results = {};
        for (int l = 0; l < n_layers; ++l) results.S[l] = bt.S[l];
        if (plan.parts) {
            const int slot_n = slot_columns(tile_n);
            VGC_CUDA_OK(launch_kernel(Carveout{18}, sqgrad_tc_combine_examples, dim3((unsigned)(plan.tiles_x * plan.tiles_y * slot_n), (unsigned)n_layers), dim3(256), 0,
                                      st, true, prm.partial, plan.k_slices / prm.p_slices, plan.parts, tile_n, slot_n, plan.tiles_x, plan.tiles_y, M, N,
                                      prm.scale, prm.accumulate, results, prm.ld_m, prm.ld_n));
            count_launch();
            VGC_CUDA_OK(cudaGetLastError());
            return VGC_OK;
        }
        // eight and more partial tiles per tile: the warps share the chain
        const bool many = plan.units_per_tile >= 8 * (prm.units_q + 1);
        const int slot_n = slot_columns(tile_n);
        const unsigned patches = (unsigned)(plan.tiles_x * plan.tiles_y) * (unsigned)(many ? slot_n : slot_n / 8);
        const auto combine = many ? sqgrad_tc_combine_many : sqgrad_tc_combine;
        // L1 for the loads of eight blocks (34 KB of shared memory) behind the kernel above, which takes all shared memory;
        // with the same for sqgrad_repack, a pass over ResNet-50, batch 32, takes 1853 us instead of 1880
        VGC_CUDA_OK(launch_kernel(Carveout{18}, combine, dim3(patches, (unsigned)n_layers), dim3(256), 0, st,
                                  true, prm.partial, prm.units_q, prm.units_r, plan.units_per_tile, tile_n, slot_n, plan.tiles_x, plan.tiles_y, M, N,
                                  prm.scale, prm.accumulate, results, prm.ld_m, prm.ld_n));
        count_launch();
    }
    VGC_CUDA_OK(cudaGetLastError());
    return VGC_OK;
}

static Plan linear_plan(int B, int in, int out) { return make_plan(Call(false), out, in, (B + kBK - 1) / kBK, 1, 1, kBN); }

size_t tc_linear_workspace_bytes(int B, int in, int out) { return tc_workspace_bytes(linear_plan(B, in, out)); }

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
    return tc_launch(sqgrad_tc<kMajorMN, kTma, kTma, false>, bt, linear_plan(B, in, out), prm, ws, ws_bytes, st);
}

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

static int repack_mode(const Call &call, int B, int C, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int P, int W = 0, int Ho = 0,
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
    if (call.exact) return kRepackNone;                 // the flat form merges the examples' positions
    return (flat >= kBK && flat % 4 == 0 && flat < (1L << 30)) ? kRepackFlat : kRepackNone;
}

constexpr Carveout kAllL1{5};       // sqgrad_repack has no shared memory

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

static size_t conv_workspace_plain(const Call &call, int n_layers, int B, int C, int Kh, int Kw, int P, int Cout)
{
    const int p_slices = (P + kBK - 1) / kBK, n_im2col = C * Kh * Kw, k_slices = B * p_slices;
    auto bytes = [&](int M, int N, int tile_n) {
        return tc_workspace_bytes(make_plan(call, M, N, k_slices, n_layers, call.exact ? p_slices : 1, tile_n));
    };
    // the wide and the narrow form of a layer that gathers several taps at a time: either can be chosen at call time
    const size_t narrow = conv_swapped(Cout, n_im2col) ? bytes(n_im2col, Cout, kBN) : bytes(Cout, n_im2col, kBN);
    size_t wide = Kw > 1 ? bytes(Cout, n_im2col, kWideN) : 0;
    if (Kw == 5 || Kw == 7) {           // whole tuples of five or seven columns
        const size_t w = bytes(Cout, n_im2col, kWideN / Kw * Kw);
        wide = wide > w ? wide : w;
    }
    return narrow > wide ? narrow : wide;
}

// Workspace of one launch over n_layers layers of this geometry (n_layers <= kMaxBatch).
static size_t conv_workspace_group(const Call &call, int n_layers, int B, int C, int Kh, int Kw, int sh, int sw, int ph, int pw, int P,
                                   int Cout, int H, int W, int Ho, int Wo)
{
    // the larger of the in-place form and the repacked one, so that either can be chosen at call time
    size_t need = conv_workspace_plain(call, n_layers, B, C, Kh, Kw, P, Cout);
    const int mode = repack_mode(call, B, C, Cout, Kh, Kw, sh, sw, ph, pw, P, W, Ho, Wo);
    const size_t x_bytes = round_up(sizeof(float) * (size_t)B * C * P, 256);
    const size_t d_bytes = round_up(sizeof(float) * (size_t)B * Cout * P, 256);
    if (mode == kRepackPadW) {
        const int Wo4 = (Wo + 3) / 4 * 4;
        const size_t xp = round_up(sizeof(float) * (size_t)B * C * H * (sw * Wo4), 256);
        const size_t dp = round_up(sizeof(float) * (size_t)B * Cout * Ho * Wo4, 256);
        const size_t r = round_up(conv_workspace_plain(call, n_layers, B, C, Kh, Kw, Ho * Wo4, Cout), 256) + n_layers * (xp + dp);
        need = need > r ? need : r;
    } else if (mode == kRepackPlanes) {
        const size_t r = round_up(conv_workspace_plain(call, n_layers, B, C, 1, 1, P, Cout), 256) + n_layers * x_bytes;
        need = need > r ? need : r;
    } else if (mode == kRepackFlat) {
        const size_t r = round_up(conv_workspace_plain(call, n_layers, 1, C, 1, 1, B * P, Cout), 256) +
                         n_layers * (x_bytes + d_bytes);
        need = need > r ? need : r;
    }
    return need;
}

size_t tc_conv_workspace_bytes(int n_layers, int B, int C, int H, int W, int Kh, int Kw, int sh, int sw, int ph, int pw,
                               int Ho, int Wo, int Cout, bool exact)
{
    const int P = Ho * Wo;
    const Call call(exact);
    // more layers than one launch takes are processed group after group in the same workspace
    const int first = n_layers < kMaxBatch ? n_layers : kMaxBatch;
    size_t need = conv_workspace_group(call, first, B, C, Kh, Kw, sh, sw, ph, pw, P, Cout, H, W, Ho, Wo);
    const int rest = n_layers > kMaxBatch ? n_layers % kMaxBatch : 0;
    if (rest) {
        const size_t r = conv_workspace_group(call, rest, B, C, Kh, Kw, sh, sw, ph, pw, P, Cout, H, W, Ho, Wo);
        need = need > r ? need : r;
    }
    return need;
}

static vgc_status conv_group(const Call &call, int n_layers, const float *const *x, const float *const *delta, float *const *S, int B,
                             int C, int H, int W, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int Ho,
                             int Wo, float scale, int accumulate, void *ws, size_t ws_bytes, cudaStream_t st)
{
    const int P = Ho * Wo, n_im2col = C * Kh * Kw;
    const int mode = repack_mode(call, B, C, Cout, Kh, Kw, sh, sw, ph, pw, P, W, Ho, Wo);
    // one run of the output per warp; more when there are many
    auto blocks_for = [](size_t values) { const size_t b = (values + 8 * kRepackRun - 1) / (8 * kRepackRun); return (unsigned)(b < 1 ? 1 : (b > 148 * 32 ? 148 * 32 : b)); };
    if (mode == kRepackPadW) {
        const int Wo4 = (Wo + 3) / 4 * 4, Wx = sw * Wo4;              // padded widths of the errors and of x
        const size_t inner = round_up(conv_workspace_plain(call, n_layers, B, C, Kh, Kw, Ho * Wo4, Cout), 256);
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
        VGC_CUDA_OK(launch_kernel(kAllL1, sqgrad_repack, dim3(blocks_for((size_t)B * ((size_t)C * H * Wx > (size_t)Cout * Ho * Wo4 ? (size_t)C * H * Wx : (size_t)Cout * Ho * Wo4)), 2 * n_layers), dim3(256), 0, st, true, jobs));
        count_launch();
        return conv_group(call, n_layers, xr, dr, S, B, C, H, Wx, Cout, Kh, Kw, sh, sw, ph, 1, Ho, Wo4, scale, accumulate, ws, inner, st);
    }
    if (mode != kRepackNone) {
        const bool flat = mode == kRepackFlat;
        const size_t inner = round_up(flat ? conv_workspace_plain(call, n_layers, 1, C, 1, 1, B * P, Cout)
                                           : conv_workspace_plain(call, n_layers, B, C, 1, 1, P, Cout), 256);
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
        VGC_CUDA_OK(launch_kernel(kAllL1, sqgrad_repack, dim3(blocks_for((size_t)B * (flat && Cout > C ? Cout : C) * P), n_jobs), dim3(256), 0, st, true, jobs));
        count_launch();
        if (flat)
            return conv_group(call, n_layers, xr, dr, S, 1, C, B * P, 1, Cout, 1, 1, 1, 1, 0, 0, B * P, 1, scale, accumulate, ws,
                              inner, st);
        return conv_group(call, n_layers, xr, dr, S, B, C, Ho, Wo, Cout, 1, 1, 1, 1, 0, 0, Ho, Wo, scale, accumulate, ws, inner, st);
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
    const bool ex = call.exact;
    const int unit = ex ? p_slices : 1;
    // the launch's plan: made once, it decides between forms below and is what is launched
    auto plan_of = [&](int M, int N, int tile_n) { return make_plan(call, M, N, k_slices, n_layers, unit, tile_n); };
    // wide tiles of the per-example form: an example fits one accumulator run, or parts of examples leave as plain sums
    auto wide_fits = [&](const Plan &p) { return !ex || p_slices <= kChunk || p.parts > 0; };
    auto bf_cross = [&](const Plan &p) { return bf16_cross_better(p, (long long)B * P); };
    Plan plan = {};
    // a square kernel that keeps the width: its input rows by TMA, however few its columns (280 layers of 1 to 8 channels, 8 x 8 to 64 x 64,
    // against the element-wise gather: 0.65 - 0.86 of its time on average for each number of channels and taps, at worst 1.02)
    bool halo = !in_tma && err_tma && (Kw == 5 || Kw == 7) && Kh == Kw && sh == 1 && sw == 1 && 2 * pw == Kw - 1 && Wo == W &&
                W % 2 == 0 && H * W % 4 == 0;
    if (halo) {
        plan = plan_of(Cout, n_im2col, kWideN / Kw * Kw);
        halo = wide_fits(plan);
    }
    // with few output channels the roles are swapped -- except where several taps are gathered at a time: there keeping the errors
    // as the A operand (in tensor memory, half of its rows unused) measures faster than both operands in shared memory
    const bool swapped = conv_swapped(Cout, n_im2col) && !taps && !taps_s2 && !taps7 && !halo;
    // both tiles by TMA: A in tensor memory, cross terms in bf16 (the per-example form keeps tf32 cross terms)
    const bool tma_bf = err_tma && in_tma && !ex;
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
        if (halo) {
            const cuuint32_t channels = Kw == 5 ? Halo<kHalo5x4>::kChannels : Halo<kHalo7x4>::kChannels;
            const cuuint32_t box[3] = {(cuuint32_t)(Kw == 5 ? Halo<kHalo5x4>::kPos : Halo<kHalo7x4>::kPos), (cuuint32_t)C < channels ? (cuuint32_t)C : channels, 1};
            const cuuint64_t dims[3] = {(cuuint64_t)H * W, (cuuint64_t)C, (cuuint64_t)B};
            const cuuint64_t str[2] = {(cuuint64_t)H * W * 4, (cuuint64_t)C * H * W * 4};
            if (!make_map(m_in, x[l], 3, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE)) return VGC_ERR_CUDA;
            tx_in = (uint32_t)Kh * box[0] * box[1] * 4;
        }
        bt.x[l] = x[l]; bt.delta[l] = delta[l]; bt.S[l] = S[l];
    }
    Params prm = {};
    prm.p_slices = p_slices; prm.tx_bytes = tx_err + tx_in; prm.scale = scale;
    prm.tx_bytes_a = swapped ? tx_in : tx_err; prm.accumulate = accumulate;
    prm.C = C; prm.H = H; prm.W = W; prm.Cout = Cout; prm.Kh = Kh; prm.Kw = Kw; prm.sh = sh; prm.sw = sw;
    prm.ph = ph; prm.pw = pw; prm.Wo = Wo; prm.P = P;
    prm.chw = C * H * W;
    if (Wo > 1) {
        const RowDivisor by_wo = row_divisor((uint32_t)Wo);
        prm.wo_magic = by_wo.magic;
        prm.wo_shift = by_wo.shift;
    }
    KernelFn fn = nullptr;
#define VGC_TC_FN(A, B_, AT) (ex ? (KernelFn)sqgrad_tc<kMajorK, A, B_, AT, true> : (KernelFn)sqgrad_tc<kMajorK, A, B_, AT, false>)
    if (!swapped) {     // S[o][idx]: m = o, n = idx
        prm.ld_m = n_im2col; prm.ld_n = 1;
        if (halo) {
            const bool by4 = W % 4 == 0;
            fn = wide_halo_kernel(Kw == 5 ? (by4 ? kHalo5x4 : kHalo5x2) : (by4 ? kHalo7x4 : kHalo7x2), ex, bf_cross(plan));
            return tc_launch(fn, bt, plan, prm, ws, ws_bytes, st);
        }
        if (taps || taps_s2 || taps7) {
            // Wide tiles where they are fewer than narrow ones (128 channels 28 x 28, batch 32: 47.9 -> 43.0 us, now 38.6; but 9 channels
            // 16 x 16 to 958, 81 columns: 25.0 us narrow, 28.7 wide).  The wide per-example form adds an example's sums up within
            // one accumulator run.
            const int mode = taps ? (taps == 4 ? kGatherTaps4 : kGatherTaps2) : taps_s2 ? (taps_s2 == 4 ? kGatherTaps4S2 : kGatherTaps2S2) : kGatherTaps7S2;
            bool wide = (n_im2col + kWideN - 1) / kWideN < (n_im2col + kBN - 1) / kBN;
            if (wide) {
                plan = plan_of(Cout, n_im2col, kWideN);
                wide = wide_fits(plan);
            }
            if (!wide) plan = plan_of(Cout, n_im2col, kBN);
            fn = wide ? wide_taps_kernel(mode, ex, bf_cross(plan)) : narrow_taps_kernel(mode, ex);
            return tc_launch(fn, bt, plan, prm, ws, ws_bytes, st);
        }
        if (tma_bf) fn = sqgrad_tc<kMajorK, kTma, kTma, true, false, true>;
        else if (err_tma && in_tma) fn = sqgrad_tc<kMajorK, kTma, kTma, true, true>;
        else if (err_tma) fn = VGC_TC_FN(kTma, kGatherIm2col, true);
        else fn = VGC_TC_FN(kGatherErr, kGatherIm2col, false);
        return tc_launch(fn, bt, plan_of(Cout, n_im2col, kBN), prm, ws, ws_bytes, st);
    }
    prm.ld_m = 1; prm.ld_n = n_im2col;   // m = idx, n = o
    if (tma_bf) fn = sqgrad_tc<kMajorK, kTma, kTma, true, false, true>;
    else if (err_tma && in_tma) fn = sqgrad_tc<kMajorK, kTma, kTma, true, true>;
    else if (err_tma) fn = VGC_TC_FN(kGatherIm2col, kTma, false);
    else fn = VGC_TC_FN(kGatherIm2col, kGatherErr, false);
#undef VGC_TC_FN
    return tc_launch(fn, bt, plan_of(n_im2col, Cout, kBN), prm, ws, ws_bytes, st);
}

// n_layers layers of one geometry; x, delta, S are host arrays of device pointers
vgc_status tc_sqgrad_conv(int n_layers, const float *const *x, const float *const *delta, float *const *S, int B, int C,
                          int H, int W, int Cout, int Kh, int Kw, int sh, int sw, int ph, int pw, int Ho, int Wo,
                          float scale, int accumulate, void *ws, size_t ws_bytes, cudaStream_t st, bool exact)
{
    const Call call(exact);
    for (int l0 = 0; l0 < n_layers; l0 += kMaxBatch) {
        const int nl = n_layers - l0 < kMaxBatch ? n_layers - l0 : kMaxBatch;
        const vgc_status rc = conv_group(call, nl, x + l0, delta + l0, S + l0, B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, Ho, Wo,
                                         scale, accumulate, ws, ws_bytes, st);
        if (rc != VGC_OK) return rc;
    }
    return VGC_OK;
}

}  // namespace vgc
