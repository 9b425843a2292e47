// Squared per-example gradient sums on the CUDA cores (fp32 FMA), used for shapes the
// tensor-core kernel does not take and as its cross-check.
//
//   S[m][n] = scale * sum_k A(k,m)^2 * B(k,n)^2
// dense layer:  A = delta [K=B][M=out],  B = x [K=B][N=in]
// conv layer:   k = (example z, output position ho, wo), m = output channel,
//               n = (input channel c, kh, kw);  B(k,n) is the im2col view of x, zero outside.
// This is the right-hand side of Eq. 2 / the "v_i +=" line of Algorithm 1 obtained as one
// contraction of squared operands (N_params * |B| multiply-adds, Sec. 5).
//
// 64x64 output tile per block, 4x4 outputs per thread, 16-deep k slices through shared
// memory.  Partial sums run 256 terms in fp32 and are then promoted to fp64, so the
// accumulated rounding error stays near 1e-6 relative for any K.  Long reductions are split
// across blockIdx.z; the slices are combined in a fixed order by a second kernel.
#include "vgc_common.cuh"

namespace vgc {

constexpr int kBM = 64, kBN = 64, kBK = 16, kSimtThreads = 256;
constexpr int kPromote = 16;        // k slices (of 16) between promotions to fp64

struct LinearOperands {
    const float *x, *delta;
    int in, out;
    static constexpr bool kInnerIsK = false;
    __device__ __forceinline__ float a(int k, int m) const { return delta[(size_t)k * out + m]; }
    __device__ __forceinline__ float b(int k, int n) const { return x[(size_t)k * in + n]; }
    struct NCoord { int n; };
    __device__ __forceinline__ NCoord ncoord(int n) const { return {n}; }
    __device__ __forceinline__ float b(int k, const NCoord &c) const { return x[(size_t)k * in + c.n]; }
};

struct ConvOperands {
    const float *x, *delta;
    int C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, Ho, Wo;
    static constexpr bool kInnerIsK = true;
    __device__ __forceinline__ float a(int k, int m) const
    {
        const int P = Ho * Wo;
        const int z = k / P, p = k - z * P;
        return delta[((size_t)z * Cout + m) * P + p];
    }
    struct NCoord { int c, kh, kw; };
    __device__ __forceinline__ NCoord ncoord(int n) const
    {
        const int kw = n % Kw, t = n / Kw;
        return {t / Kh, t % Kh, kw};
    }
    __device__ __forceinline__ float b(int k, const NCoord &nc) const
    {
        const int P = Ho * Wo;
        const int z = k / P, p = k - z * P;
        const int ho = p / Wo, wo = p - ho * Wo;
        const int hi = ho * sh + nc.kh - ph, wi = wo * sw + nc.kw - pw;
        if (hi < 0 || hi >= H || wi < 0 || wi >= W) return 0.f;
        return x[(((size_t)z * C + nc.c) * H + hi) * W + wi];
    }
};

// out_partial: [gridDim.z][M][N] fp32 when gridDim.z > 1, else the final S.
template <class Ops>
__global__ void __launch_bounds__(kSimtThreads)
sqgrad_simt(const Ops ops, int M, int N, int K, int k_per_split, float scale, int accumulate,
            float *__restrict__ S, float *__restrict__ partial)
{
    __shared__ float As[kBK][kBM + 4];
    __shared__ float Bs[kBK][kBN + 4];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * kBN;
    const int k_begin = blockIdx.z * k_per_split;
    const int k_end = min(K, k_begin + k_per_split);

    // which 4 elements of each operand tile this thread fetches
    int lk[4], lmn[4];
    typename Ops::NCoord nco[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = tid + kSimtThreads * i;
        if (Ops::kInnerIsK) { lk[i] = e % kBK; lmn[i] = e / kBK; }
        else                { lk[i] = e / kBM; lmn[i] = e % kBM; }
        nco[i] = ops.ncoord(min(n0 + lmn[i], N - 1));
    }

    float acc[4][4];
    double acc2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = 0.f; acc2[i][j] = 0.0; }

    int slice = 0;
    for (int k0 = k_begin; k0 < k_end; k0 += kBK) {
        float av[4], bv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + lk[i];
            const bool kin = k < k_end;
            av[i] = (kin && m0 + lmn[i] < M) ? ops.a(k, m0 + lmn[i]) : 0.f;
            bv[i] = (kin && n0 + lmn[i] < N) ? ops.b(k, nco[i]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            As[lk[i]][lmn[i]] = __fmul_rn(av[i], av[i]);
            Bs[lk[i]][lmn[i]] = __fmul_rn(bv[i], bv[i]);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            const float4 a4 = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (++slice == kPromote) {
            slice = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) { acc2[i][j] += (double)acc[i][j]; acc[i][j] = 0.f; }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
            if (m >= M || n >= N) continue;
            const double sum = acc2[i][j] + (double)acc[i][j];
            if (gridDim.z > 1) {
                partial[((size_t)blockIdx.z * M + m) * N + n] = (float)sum;
            } else {
                const size_t at = (size_t)m * N + n;
                const double res = (double)scale * sum;
                S[at] = accumulate ? __fadd_rn(S[at], (float)res) : (float)res;      // one fp32 addition, as everywhere
            }
        }
}

__global__ void __launch_bounds__(256)
sqgrad_combine_splits(const float *__restrict__ partial, int splits, size_t mn, float scale, int accumulate,
                      float *__restrict__ S)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= mn) return;
    double sum = 0.0;
    for (int z = 0; z < splits; ++z) sum += (double)partial[(size_t)z * mn + i];
    const double res = (double)scale * sum;
    S[i] = accumulate ? __fadd_rn(S[i], (float)res) : (float)res;
}

// ---- dense layers: few enough multiply-adds for the CUDA cores, or sizes the tensor-core kernels do not take ------------
//
// One block of 256 threads per kTile x kTile tile of S, 4 x 4 results per thread; 32 (64) examples at a time through shared
// memory, squared on the way in, the next ones already in registers.  kTile = 64: one thread per result block.  kTile = 32
// (where 64 x 64 tiles would leave SMs idle): four groups of 64 threads take every fourth example each and add up at the
// end.  fp32 sums of at most 64 examples, fp64 above that.
//
// Bound: the launch and one round trip to memory for small layers, fp32 multiply-adds for large ones.  Measured (B200, one
// call among others): 32 examples, 256 x 128: 11.2 us on the tensor-core kernel, 2.5 here; 128 examples, 1024 x 10: 10.5 us
// on the kernel above, 4.6 here.
constexpr int kDenseFlush = 2;                        // rounds per fp32 sum

template <int kTile, bool kVec>                        // kVec: in and out are multiples of 4
__global__ void __launch_bounds__(kSimtThreads)
sqgrad_dense_simt(const float *x, const float *delta, int B, int in, int out, float scale, int accumulate, float *S)
{
    constexpr int kDenseK = kTile == 32 ? 64 : 32;                     // examples per round
    constexpr int kThreadsPerTile = (kTile / 4) * (kTile / 4), kGroups = kSimtThreads / kThreadsPerTile;
    constexpr int kVecs = kDenseK * kTile / 4 / kSimtThreads;          // float4 per thread, operand and round
    __shared__ __align__(16) float As[kDenseK][kTile];
    __shared__ __align__(16) float Bs[kDenseK][kTile];
    const int tid = threadIdx.x, group = tid / kThreadsPerTile, t = tid % kThreadsPerTile;
    const int tx = t % (kTile / 4), ty = t / (kTile / 4);
    const int m0 = blockIdx.y * kTile, n0 = blockIdx.x * kTile;
    grid_release();
    grid_wait();
    if (accumulate && tid < kTile && m0 + tid < out) {                 // the old contents, needed at the end
#pragma unroll
        for (int j = 0; j < kTile; j += 32)
            if (n0 + j < in) asm volatile("prefetch.global.L2 [%0];" ::"l"(S + (size_t)(m0 + tid) * in + n0 + j));
    }
    float4 a[kVecs], b[kVecs];
    auto load4 = [&](const float *row, int at, int limit, bool valid) -> float4 {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!valid) return v;
        if (kVec) {
            if (at < limit) v = *reinterpret_cast<const float4 *>(row + at);
        } else {
            if (at < limit) v.x = row[at];
            if (at + 1 < limit) v.y = row[at + 1];
            if (at + 2 < limit) v.z = row[at + 2];
            if (at + 3 < limit) v.w = row[at + 3];
        }
        return v;
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int e = tid + i * kSimtThreads, k = k0 + e / (kTile / 4), c = e % (kTile / 4) * 4;
            a[i] = load4(delta + (size_t)k * out, m0 + c, out, k < B);
            b[i] = load4(x + (size_t)k * in, n0 + c, in, k < B);
        }
    };
    auto square = [](const float4 &v) {
        return make_float4(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y), __fmul_rn(v.z, v.z), __fmul_rn(v.w, v.w));
    };
    float acc[4][4];
    double sum[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = 0.f; sum[i][j] = 0.0; }
    fetch(0);
    int rounds = 0;
    for (int k0 = 0; k0 < B; k0 += kDenseK) {
        if (k0) __syncthreads();
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int e = tid + i * kSimtThreads, k = e / (kTile / 4), c = e % (kTile / 4) * 4;
            *reinterpret_cast<float4 *>(&As[k][c]) = square(a[i]);
            *reinterpret_cast<float4 *>(&Bs[k][c]) = square(b[i]);
        }
        if (k0 + kDenseK < B) fetch(k0 + kDenseK);                      // (before the barrier: ordinary loads stay behind it)
        __syncthreads();
        auto step = [&](int kk) {
            const float4 a4 = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
            const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        };
        if (k0 + kDenseK <= B) {
#pragma unroll 8
            for (int kk = group; kk < kDenseK; kk += kGroups) step(kk);
        } else {
            for (int kk = group; kk < B - k0; kk += kGroups) step(kk);
        }
        if (++rounds == kDenseFlush) {
            rounds = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) { sum[i][j] += (double)acc[i][j]; acc[i][j] = 0.f; }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[i][j] += (double)acc[i][j];
    if (kGroups > 1) {
        __shared__ double part[kGroups > 1 ? kGroups - 1 : 1][kGroups > 1 ? 16 : 1][kThreadsPerTile];
        if (group > 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) part[group - 1][i][t] = sum[i >> 2][i & 3];
        }
        __syncthreads();
        if (group > 0) return;
#pragma unroll
        for (int g = 0; g < kGroups - 1; ++g)
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i >> 2][i & 3] += part[g][i][t];
    }
    const int n = n0 + tx * 4;
    float old[4][4];                                                    // all of it asked for before the first store
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        const float *src = S + (size_t)m * in + n;
        if (kVec) {
            const float4 o = accumulate && m < out && n < in ? *reinterpret_cast<const float4 *>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
            old[i][0] = o.x; old[i][1] = o.y; old[i][2] = o.z; old[i][3] = o.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) old[i][j] = accumulate && m < out && n + j < in ? src[j] : 0.f;
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= out || n >= in) continue;
        float *dst = S + (size_t)m * in + n;
        float res[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            res[j] = (float)((double)scale * sum[i][j]);
            if (accumulate) res[j] = __fadd_rn(old[i][j], res[j]);
        }
        if (kVec) {
            *reinterpret_cast<float4 *>(dst) = make_float4(res[0], res[1], res[2], res[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (n + j < in) dst[j] = res[j];
        }
    }
}

// Whether the kernel above is faster than what else takes the layer; tensor_cores: that is the general tensor-core kernel
// (sqgrad_tc), else sqgrad_simt with its split reduction.  Measured on both sides (B200, one call among others, us above / else):
//   sqgrad_tc, up to 2^27 multiply-adds: 640 examples 500 x 256 15.9 / 17.8, 768 18.6 / 19.7, 896 21.3 / 20.0, 1024 24.1 / 21.2
//   sqgrad_simt: 149 to 296 tiles leave SMs with one or two blocks that nothing hides behind: 1031 x 1009, 64 examples faster
//   above, 128 17.4 / 16.8, 256 31.9 / 27.8, 1024 119 / 93; more tiles are as fast above (2049 x 1023, 1024 examples: 171 / 174);
//   fewer: 333 x 257, 768 examples 20.5 / 23.0, 896 23.7 / 21.0; less than half of the other kernel's tile used: 1024
//   examples, 1000 x 10: 20.3 / 22.9
bool dense_simt_better(int B, int in, int out, bool tensor_cores)
{
    if (tensor_cores) return B <= 768 && (long long)in * out * B <= (1ll << 27);
    const long long tiles = (long long)((in + 63) / 64) * ((out + 63) / 64);
    if (tiles > 148 && tiles <= 296) return B < 128;
    return B <= 768 || (B <= 1024 && (tiles > 296 || in < 32 || out < 32));
}

vgc_status dense_simt(const float *x, const float *delta, int B, int in, int out, float scale, int accumulate, float *S,
                      cudaStream_t st)
{
    auto tiles = [&](int tile) { return (long long)((in + tile - 1) / tile) * ((out + tile - 1) / tile); };
    const bool vec = in % 4 == 0 && out % 4 == 0, small = tiles(64) < 148;
    const int tile = small ? 32 : 64;
    const dim3 grid((in + tile - 1) / tile, (out + tile - 1) / tile);
    if (grid.y > 65535u) return VGC_ERR_UNSUPPORTED;
    auto fn = small ? (vec ? sqgrad_dense_simt<32, true> : sqgrad_dense_simt<32, false>)
                    : (vec ? sqgrad_dense_simt<64, true> : sqgrad_dense_simt<64, false>);
    VGC_CUDA_OK(launch_kernel(fn, grid, dim3(kSimtThreads), 0, st, true, x, delta, B, in, out, scale, accumulate, S));
    count_launch();
    return VGC_OK;
}

int simt_splits(int M, int N, int K)
{
    const long tiles = (long)((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN);
    long want = (4L * 148 + tiles - 1) / tiles;
    const long max_by_k = (K + kBK * kPromote - 1) / (kBK * kPromote);
    if (want > max_by_k) want = max_by_k;
    if (want > 1024) want = 1024;
    if (want < 1) want = 1;
    return (int)want;
}

size_t simt_workspace_bytes(int M, int N, int K)
{
    const int splits = simt_splits(M, N, K);
    return splits > 1 ? (size_t)splits * M * N * sizeof(float) : 0;
}

template <class Ops>
vgc_status simt_launch(const Ops &ops, int M, int N, int K, float scale, int accumulate, float *S,
                       void *ws, size_t ws_bytes, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return VGC_ERR_INVALID_ARG;     // empty sums are the caller's business
    int splits = simt_splits(M, N, K);
    if (splits > 1 && ws_bytes < (size_t)splits * M * N * sizeof(float)) return VGC_ERR_WORKSPACE;
    int k_per_split = (K + splits - 1) / splits;
    k_per_split = (k_per_split + kBK - 1) / kBK * kBK;
    splits = (K + k_per_split - 1) / k_per_split;
    dim3 grid((N + kBN - 1) / kBN, (M + kBM - 1) / kBM, splits);
    if (grid.y > 65535u) return VGC_ERR_UNSUPPORTED;
    sqgrad_simt<Ops><<<grid, kSimtThreads, 0, st>>>(ops, M, N, K, k_per_split, scale, accumulate, S,
                                                    static_cast<float *>(ws));
    count_launch();
    if (splits > 1) {
        count_launch();
        const size_t mn = (size_t)M * N;
        sqgrad_combine_splits<<<(unsigned)((mn + 255) / 256), 256, 0, st>>>(static_cast<const float *>(ws), splits,
                                                                            mn, scale, accumulate, S);
    }
    return cudaGetLastError() == cudaSuccess ? VGC_OK : VGC_ERR_CUDA;
}

vgc_status simt_sqgrad_linear(const float *x, const float *delta, int B, int in, int out, float scale,
                              int accumulate, float *S, void *ws, size_t ws_bytes, cudaStream_t st)
{
    LinearOperands ops{x, delta, in, out};
    return simt_launch(ops, out, in, B, scale, accumulate, S, ws, ws_bytes, st);
}

vgc_status simt_sqgrad_conv(const float *x, const float *delta, int B, int C, int H, int W, int Cout,
                            int Kh, int Kw, int sh, int sw, int ph, int pw, int Ho, int Wo, float scale,
                            int accumulate, float *S, void *ws, size_t ws_bytes, cudaStream_t st)
{
    ConvOperands ops{x, delta, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, Ho, Wo};
    return simt_launch(ops, Cout, C * Kh * Kw, B * Ho * Wo, scale, accumulate, S, ws, ws_bytes, st);
}

}  // namespace vgc
