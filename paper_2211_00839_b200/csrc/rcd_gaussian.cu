// Gaussian-kernel similarity (Section 4, item 2: "a Gaussian kernel with L2 distance" whose
// bandwidth is sigma = sum_{v,v'} ||v - v'||_2 / n^2).  Reading taken (the paper gives neither the
// exponent nor what n counts): n = |V_l|, all ordered pairs of the class, and
//     sim(v, v') = exp(-||v - v'||^2 / (2 sigma^2)).
//
// Built on the dot-product matrix the similarity kernels have already written:
//     ||v - v'||^2 = ||v||^2 + ||v'||^2 - 2 <v, v'>,
// exact in integers for int8 features.  Four small kernels: row norms, per-row-block sums of the
// distances (fp64, fixed order), sigma per class, and the in-place transform of S to fp32 kernel
// values.  The sums are reduced in a fixed order so that sigma, and with it every similarity, is
// reproducible from run to run.
#include "rcd_internal.h"

namespace rcd {

constexpr int kGaussRows = 64;       // rows of S per CTA, sums of distances
constexpr int kGaussApplyRows = 16;  // ... and kernel values
constexpr int kGaussBatch = 4;       // rows a lane has in flight
constexpr int kGaussWarps = 8;
constexpr int kGaussFixedExp = 29;   // the largest value of the kernel, 1, at 2^29 (as fixed_exponent_kernel would have it)

__device__ __forceinline__ float bf16_bits_as_float(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

// ||x_r||^2 of every class-sorted row: int32 for int8 features (exact), fp32 for bf16.
template <bool kInt8>
__global__ void __launch_bounds__(256, 4) row_norms_kernel(const void *__restrict__ Xs, int64_t N, int64_t d, void *__restrict__ norms)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= N) return;
    if constexpr (kInt8) {
        const int8_t *x = reinterpret_cast<const int8_t *>(Xs) + row * d;
        int acc = 0;
        for (int64_t k = lane; k < d; k += 32) acc += (int)x[k] * (int)x[k];
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) reinterpret_cast<int32_t *>(norms)[row] = acc;
    } else {
        const uint16_t *x = reinterpret_cast<const uint16_t *>(Xs) + row * d;
        float acc = 0.f;
        for (int64_t k = lane; k < d; k += 32) { const float v = bf16_bits_as_float(x[k]); acc = fmaf(v, v, acc); }
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) reinterpret_cast<float *>(norms)[row] = acc;
    }
}

// Squared distance of two samples of a class from their norms and dot product.  int8: exact, one rounding; in 32 bits while
// 255^2 d fits them (sums and differences modulo 2^32), else in 64.
constexpr int64_t kGaussNarrowDim = 66051;
template <bool kInt8, bool kWide>
__device__ __forceinline__ float squared_distance(uint32_t ni, uint32_t nj, uint32_t dotBits)
{
    if constexpr (kInt8 && kWide) {
        return (float)((long long)(int32_t)ni + (long long)(int32_t)nj - 2ll * (long long)(int32_t)dotBits);
    } else if constexpr (kInt8) {
        return (float)(ni + nj - 2u * dotBits);
    } else {
        return fmaxf(__uint_as_float(ni) + __uint_as_float(nj) - 2.f * __uint_as_float(dotBits), 0.f);
    }
}

// Square root within a unit in the last place of fp64: Heron's step s += (v - s s) / (2 s) twice, with the fp32 reciprocal root standing in for
// 1 / s: 22 bits right, then 44, then all that the format holds.  No branches (zeros and infinities are their own roots).
__device__ __forceinline__ double root_fp64(float v)
{
    const float y = rsqrtf(v);
    const double d = (double)v, h = (double)(0.5f * y);
    double s = 2.0 * d * h;
    s = fma(fma(-s, s, d), h, s);
    s = fma(fma(-s, s, d), h, s);
    return v > 0.f && v < INFINITY ? s : d;
}

// Both passes over S below give a CTA some rows of a class (sums 64, values 16) and its warps 128 columns at a time, four per
// lane: the norms of a lane's columns stay in registers down the rows, those of the rows sit in shared memory, and S moves in
// 128-bit pieces.

// Sums of distances.  They are symmetric, so only the columns right of the diagonal are read and rooted (sigma counts each
// pair twice).  Bound by the square roots in fp64: 212 us at 10 classes of 5000, 1 GB of S (338 with one row in flight per
// lane, 408 with sqrt(double) as well).  Classes run fastest in the grid, so that the long row groups start first.
template <bool kInt8, bool kWide>
__global__ void __launch_bounds__(kGaussWarps * 32, 4) gauss_dist_sum_kernel(DescSource src, const uint32_t *__restrict__ S,
                                                                            const uint32_t *__restrict__ norms, int32_t maxBlocks,
                                                                            double *__restrict__ partial)
{
    __shared__ double shWarp[kGaussWarps];
    __shared__ uint32_t shNorm[kGaussRows];
    const int l = blockIdx.x;
    const ClassDesc c = src.get(l);
    const int first = blockIdx.y * kGaussRows;
    if (first >= c.M) return;
    const int rows = min(kGaussRows, c.M - first);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < rows) shNorm[threadIdx.x] = norms[c.row0 + first + threadIdx.x];
    __syncthreads();
    double acc = 0.0;
    for (int col = (first / 128 + warp) * 128 + lane * 4; col < c.M; col += kGaussWarps * 128) {
        uint32_t nj[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) nj[e] = col + e < c.M ? norms[c.row0 + col + e] : 0u;
        const uint32_t *p = S + c.sOff + (int64_t)first * c.ld + col;
        const int last = min(rows, col + 3 - first);       // rows above this piece's last column
        for (int r0 = 0; r0 < last; r0 += kGaussBatch) {
            uint4 x[kGaussBatch];
#pragma unroll
            for (int b = 0; b < kGaussBatch; ++b)
                if (r0 + b < last) x[b] = __ldcs(reinterpret_cast<const uint4 *>(p + (int64_t)(r0 + b) * c.ld));
#pragma unroll
            for (int b = 0; b < kGaussBatch; ++b) {
                const int r = r0 + b;
                if (r >= last) break;
                const uint32_t dots[4] = {x[b].x, x[b].y, x[b].z, x[b].w};
                const uint32_t ni = shNorm[r];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    acc += root_fp64(col + e > first + r && col + e < c.M ? squared_distance<kInt8, kWide>(ni, nj[e], dots[e]) : 0.f);
            }
        }
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) shWarp[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kGaussWarps; ++w) s += shWarp[w];
        partial[(int64_t)l * maxBlocks + blockIdx.y] = 2.0 * s;
    }
}

// sigma_l = (sum of all pairwise distances) / M^2 ; scale_l = 1 / (2 sigma^2)  (0 when sigma = 0)
__global__ void gauss_sigma_kernel(DescSource src, int32_t L, const double *__restrict__ partial, int32_t maxBlocks,
                                   float *__restrict__ sigma, float *__restrict__ scale)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= L) return;
    const ClassDesc c = src.get(l);
    const int nb = (c.M + kGaussRows - 1) / kGaussRows;
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += partial[(int64_t)l * maxBlocks + b];
    const double sg = c.M > 0 ? s / ((double)c.M * (double)c.M) : 0.0;
    sigma[l] = (float)sg;
    scale[l] = sg > 0.0 ? (float)(1.0 / (2.0 * sg * sg)) : 0.f;
}

// Dot products to kernel values, in place: fp32, or (fixedExp given) the fixed-point integers that the cluster form of the
// greedy loop reads.  Every class has 1 on its diagonal and nothing above it, so their scale needs no look at S and S no
// further pass: round(sim * 2^29).  Bound by reading and writing S and by the conversions: 437 us at 10 classes of 5000, 2 GB
// (630 with one row in flight per lane and 64 rows per CTA, 1.3 waves of them).  Both passes over whole rows with four bytes
// per lane and load, and a third to fixed point, took 2.1 ms.
template <bool kInt8, bool kWide>
__global__ void __launch_bounds__(kGaussWarps * 32, 4) gauss_apply_kernel(DescSource src, uint32_t *__restrict__ S,
                                                                         const uint32_t *__restrict__ norms,
                                                                         const float *__restrict__ scale, int32_t *__restrict__ fixedExp)
{
    __shared__ uint32_t shNorm[kGaussApplyRows];
    const int l = blockIdx.x;
    const ClassDesc c = src.get(l);
    const int first = blockIdx.y * kGaussApplyRows;
    if (fixedExp && blockIdx.y == 0 && threadIdx.x == 0) fixedExp[l] = kGaussFixedExp;
    if (first >= c.M) return;
    const float k = scale[l];
    const float unit = fixedExp ? (float)(1 << kGaussFixedExp) : 0.f;
    const int rows = min(kGaussApplyRows, c.M - first);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < rows) shNorm[threadIdx.x] = norms[c.row0 + first + threadIdx.x];
    __syncthreads();
    for (int col = warp * 128 + lane * 4; col < c.M; col += kGaussWarps * 128) {
        uint32_t nj[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) nj[e] = col + e < c.M ? norms[c.row0 + col + e] : 0u;
        uint32_t *p = S + c.sOff + (int64_t)first * c.ld + col;
        for (int r0 = 0; r0 < rows; r0 += kGaussBatch) {
            uint4 x[kGaussBatch];
#pragma unroll
            for (int b = 0; b < kGaussBatch; ++b)
                if (r0 + b < rows) x[b] = __ldcs(reinterpret_cast<const uint4 *>(p + (int64_t)(r0 + b) * c.ld));
#pragma unroll
            for (int b = 0; b < kGaussBatch; ++b) {
                const int r = r0 + b;
                if (r >= rows) break;
                uint32_t v[4] = {x[b].x, x[b].y, x[b].z, x[b].w};
                const uint32_t ni = shNorm[r];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float d2 = col + e == first + r ? 0.f : squared_distance<kInt8, kWide>(ni, nj[e], v[e]);
                    const float sim = k > 0.f ? expf(-d2 * k) : 1.0f;              // sigma = 0: all points coincide
                    const uint32_t bits = unit > 0.f ? (uint32_t)__float2int_rn(sim * unit) : __float_as_uint(sim);
                    v[e] = col + e < c.M ? bits : 0u;                              // (pad columns stay zero)
                }
                *reinterpret_cast<uint4 *>(p + (int64_t)r * c.ld) = make_uint4(v[0], v[1], v[2], v[3]);
            }
        }
    }
}

rcd_status launch_gaussian(rcd_ctx *ctx, const void *Xs, rcd_feat_dtype dtype, int64_t N, int64_t d, const SimClasses &cls,
                           void *S, void *norms, double *partial, float *sigma, float *scale, int32_t *fixedExp, cudaStream_t st)
{
    if (N == 0 || cls.L == 0 || cls.maxM == 0) return RCD_OK;
    if (cls.L > 65535) return fail(ctx, RCD_ERR_UNSUPPORTED, "Gaussian similarity: more than 65535 classes");
    const int maxBlocks = (int)((cls.maxM + kGaussRows - 1) / kGaussRows);
    const unsigned normBlocks = (unsigned)((N + 7) / 8);
    const dim3 grid(cls.L, maxBlocks), applyGrid(cls.L, (unsigned)((cls.maxM + kGaussApplyRows - 1) / kGaussApplyRows));
    if (applyGrid.y > 65535) return fail(ctx, RCD_ERR_UNSUPPORTED, "Gaussian similarity: more than 65535 row groups");
    const bool wide = d > kGaussNarrowDim;
    auto *sums = dtype != RCD_FEAT_I8 ? gauss_dist_sum_kernel<false, false> : wide ? gauss_dist_sum_kernel<true, true> : gauss_dist_sum_kernel<true, false>;
    auto *apply = dtype != RCD_FEAT_I8 ? gauss_apply_kernel<false, false> : wide ? gauss_apply_kernel<true, true> : gauss_apply_kernel<true, false>;
    if (dtype == RCD_FEAT_I8) row_norms_kernel<true><<<normBlocks, 256, 0, st>>>(Xs, N, d, norms);
    else row_norms_kernel<false><<<normBlocks, 256, 0, st>>>(Xs, N, d, norms);
    sums<<<grid, kGaussWarps * 32, 0, st>>>(cls.src, (const uint32_t *)S, (const uint32_t *)norms, maxBlocks, partial);
    gauss_sigma_kernel<<<(cls.L + 127) / 128, 128, 0, st>>>(cls.src, cls.L, partial, maxBlocks, sigma, scale);
    apply<<<applyGrid, kGaussWarps * 32, 0, st>>>(cls.src, (uint32_t *)S, (const uint32_t *)norms, scale, fixedExp);
    ctx->kernelLaunches += 4;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

size_t gaussian_scratch_bytes(int64_t N, int32_t L, int64_t maxM)
{
    const size_t maxBlocks = (size_t)((maxM + kGaussRows - 1) / kGaussRows);
    return align_up((size_t)(N > 0 ? N : 1) * 4) + align_up((size_t)L * (maxBlocks ? maxBlocks : 1) * 8) + 2 * align_up((size_t)L * 4);
}

}  // namespace rcd
