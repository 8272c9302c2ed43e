// f(A_j^l) = sum_{i in V_l} max(0, max_{v' in A_j^l} S[i][v'])  for every class l and block j,
// straight from the definition (Section 4, item 2), given an assignment vector.  Independent of
// the greedy state: one pass over S, then sums in a fixed order so that the fp64 result is reproducible.
//
// S is symmetric, so the maximum over a block's members may be taken down the members' rows: a thread owns four columns
// and keeps their running maximum, nothing is shared and every load is coalesced.  The rows are walked in block order (a
// counting sort of each class's samples); where the block changes, or at the end of a unit of work, the maxima join the
// block's coverage vector by atomic maxima.  Bound by reading S once (1 GB for ten classes of 5000: 1.25 ms with a
// shared-memory atomic maximum per element, 0.2 ms now, of which 0.15 ms is the copy bandwidth's share).
#include "rcd_internal.h"

#include <type_traits>

namespace rcd {

constexpr int kObjThreads = 128;          // x 4 columns
constexpr int kObjRows = 128;             // rows of S per unit of work

// Class-sorted positions of a class's samples, sorted by block (samples in no block left out); counts[l][W] members.
__global__ void __launch_bounds__(512) objective_members_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ perm,
                                                               const int32_t *__restrict__ assignment, int32_t W,
                                                               int32_t *__restrict__ members, int32_t *__restrict__ counts)
{
    extern __shared__ int32_t shCount[];
    const ClassDesc c = desc[blockIdx.x];
    const int32_t *pl = perm + c.row0;
    for (int p = threadIdx.x; p < W; p += 512) shCount[p] = 0;
    __syncthreads();
    for (int v = threadIdx.x; v < c.M; v += 512) {
        const int a = assignment[pl[v]];
        if (a >= 0 && a < W) atomicAdd(&shCount[a], 1);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int run = 0;
        for (int p0 = 0; p0 < W; p0 += 32) {
            const int p = p0 + threadIdx.x;
            const int n = p < W ? shCount[p] : 0;
            int sum = n;
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, sum, off);
                if ((int)threadIdx.x >= off) sum += up;
            }
            if (p < W) {
                counts[(int64_t)blockIdx.x * W + p] = n;
                shCount[p] = run + sum - n;
            }
            run += __shfl_sync(0xffffffffu, sum, 31);
        }
    }
    __syncthreads();
    // (the order inside a block does not matter: a maximum is taken over it)
    for (int v = threadIdx.x; v < c.M; v += 512) {
        const int a = assignment[pl[v]];
        if (a >= 0 && a < W) members[c.row0 + atomicAdd(&shCount[a], 1)] = v;
    }
}

template <typename SV>
__device__ __forceinline__ int32_t above_zero(SV s)
{
    // positive int32 and positive fp32 both order like their bit patterns
    if constexpr (std::is_integral<SV>::value) return max((int32_t)s, 0);
    else return s > 0.f ? __float_as_int(s) : 0;
}

template <typename SV>
__global__ void __launch_bounds__(kObjThreads, 8) objective_cover_kernel(const ClassDesc *__restrict__ desc, const SV *__restrict__ S,
                                                                        const int32_t *__restrict__ members, const int32_t *__restrict__ counts,
                                                                        int32_t W, int32_t *__restrict__ cover)
{
    __shared__ int32_t shMember[kObjRows];
    __shared__ int32_t shBlock[kObjRows];
    const int l = blockIdx.z;
    const ClassDesc c = desc[l];
    const int first = blockIdx.y * kObjRows;
    if (first >= c.M || (int)blockIdx.x * kObjThreads * 4 >= c.ld) return;
    // the block of every row of this unit
    {
        const int32_t *cnt = counts + (int64_t)l * W;
        const int k = first + threadIdx.x;
        int run = 0, p = 0;
        for (; p < W; ++p) {
            const int n = cnt[p];
            if (k < run + n) break;
            run += n;
        }
        shBlock[threadIdx.x] = p < W ? p : -1;
        shMember[threadIdx.x] = p < W ? members[c.row0 + k] : 0;
    }
    __syncthreads();
    const int q = blockIdx.x * kObjThreads + threadIdx.x;
    if (4 * q >= c.ld) return;
    typedef typename std::conditional<std::is_integral<SV>::value, int4, float4>::type V4;
    const V4 *col = reinterpret_cast<const V4 *>(S + c.sOff) + q;
    const int ld4 = c.ld >> 2;
    int4 m = make_int4(0, 0, 0, 0);
    int block = shBlock[0];
    auto flush = [&] {
        int32_t *to = cover + c.vOff + (int64_t)block * c.ld + 4 * q;
        if (m.x) atomicMax(to, m.x);
        if (m.y) atomicMax(to + 1, m.y);
        if (m.z) atomicMax(to + 2, m.z);
        if (m.w) atomicMax(to + 3, m.w);
        m = make_int4(0, 0, 0, 0);
    };
    for (int k0 = 0; k0 < kObjRows && shBlock[k0] >= 0; k0 += 8) {
        V4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = __ldcs(col + (int64_t)shMember[k0 + u] * ld4);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int b = shBlock[k0 + u];
            if (b < 0) break;
            if (b != block) { flush(); block = b; }
            m.x = max(m.x, above_zero<SV>(x[u].x));
            m.y = max(m.y, above_zero<SV>(x[u].y));
            m.z = max(m.z, above_zero<SV>(x[u].z));
            m.w = max(m.w, above_zero<SV>(x[u].w));
        }
    }
    if (block >= 0) flush();
}

// f of one (class, block): the sum of its coverage vector, by one warp.
template <typename SV, typename FV>
__global__ void __launch_bounds__(256) objective_sum_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ cover, int32_t L, int32_t W,
                                                           FV *__restrict__ partValues)
{
    const int lane = threadIdx.x & 31;
    const int64_t idx = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (idx >= (int64_t)L * W) return;
    const ClassDesc c = desc[idx / W];
    const int4 *v = reinterpret_cast<const int4 *>(cover + c.vOff + (idx % W) * c.ld);
    FV s = (FV)0;
    for (int q = lane; q < c.ld / 4; q += 32) {
        const int4 x = v[q];
        if constexpr (std::is_integral<SV>::value) s += (FV)x.x + (FV)x.y + (FV)x.z + (FV)x.w;
        else s += (FV)__int_as_float(x.x) + (FV)__int_as_float(x.y) + (FV)__int_as_float(x.z) + (FV)__int_as_float(x.w);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) partValues[idx] = s;
}

// one CTA, fixed strided partials then a fixed tree: reproducible
template <typename FV>
__global__ void __launch_bounds__(256, 1) objective_total_kernel(const FV *__restrict__ partValues, int64_t n,
                                                             FV *__restrict__ total)
{
    __shared__ FV sh[256];
    FV s = (FV)0;
    for (int64_t i = threadIdx.x; i < n; i += 256) s += partValues[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = sh[0];
}

template <typename SV, typename FV>
static rcd_status run_objective(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const int32_t *assignment, void *partValues, void *total,
                                cudaStream_t st)
{
    const int64_t rowBlocks = (sz.maxM + kObjRows - 1) / kObjRows;
    if (sz.L > 65535 || rowBlocks > 65535) return fail(ctx, RCD_ERR_UNSUPPORTED, "objective: more than 65535 classes or row blocks");
    int32_t *members = ws.cand, *counts = ws.cnt, *cover = (int32_t *)ws.cover;
    if (sz.maxM > 0) {
        RCD_CUDA(ctx, cudaMemsetAsync(cover, 0, (size_t)sz.vElems * sizeof(int32_t), st));
        objective_members_kernel<<<sz.L, 512, (size_t)sz.W * 4, st>>>(ws.desc, ws.perm, assignment, sz.W, members, counts);
        const dim3 grid((unsigned)((pad_row(sz.maxM) + 4 * kObjThreads - 1) / (4 * kObjThreads)), (unsigned)rowBlocks, (unsigned)sz.L);
        objective_cover_kernel<SV><<<grid, kObjThreads, 0, st>>>(ws.desc, (const SV *)ws.S, members, counts, sz.W, cover);
        ctx->kernelLaunches += 2;
    }
    const int64_t n = (int64_t)sz.L * sz.W;
    objective_sum_kernel<SV, FV><<<(unsigned)((n + 7) / 8), 256, 0, st>>>(ws.desc, cover, sz.L, sz.W, (FV *)partValues);
    objective_total_kernel<FV><<<1, 256, 0, st>>>((const FV *)partValues, n, (FV *)total);
    ctx->kernelLaunches += 2;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_objective(rcd_ctx *ctx, rcd_feat_dtype dtype, const Sizes &sz, const Workspace &ws, const int32_t *assignment,
                            void *partValues, void *total, cudaStream_t st)
{
    if (dtype == RCD_FEAT_I8) return run_objective<int32_t, long long>(ctx, sz, ws, assignment, partValues, total, st);
    return run_objective<float, double>(ctx, sz, ws, assignment, partValues, total, st);
}

}  // namespace rcd
