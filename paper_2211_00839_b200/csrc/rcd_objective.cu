// f(A_j^l) = sum_{i in V_l} max(0, max_{v' in A_j^l} S[i][v'])  for every class l and block j,
// straight from the definition (Section 4, item 2), given an assignment vector.  Independent of
// the greedy state: one pass over S, then sums in a fixed order so that the fp64 result is reproducible.
//
// With dot products S is never written: the rows of every class are brought into block order (objective_order_kernel, gather), the
// similarity kernel's epilogue keeps the maxima of its tiles (keep_maxima in rcd_similarity_tc.cu) and joins them to the blocks'
// coverage, and only the sums are left (ten classes of 5000 into 8 blocks: 440 us through S, 172 without).
//
// Otherwise (Gaussian kernel, whose bandwidth needs all distances first, and the generic similarity kernel) the maxima are taken
// from S.  S is symmetric, so the maximum over a block's members may be taken down the members' rows: a thread owns four columns
// and keeps their running maximum, nothing is shared and every load is coalesced.  The rows are walked in block order (a
// counting sort of each class's samples); where the block changes, or at the end of a unit of work, the maxima join the
// block's coverage vector by atomic maxima.  Bound by reading S once (1 GB for ten classes of 5000: 1.25 ms with a
// shared-memory atomic maximum per element, 0.2 ms now, of which 0.15 ms is the copy bandwidth's share).
#include "rcd_internal.h"

#include <algorithm>
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

// Every class's samples in block order, those in no block last: a stable counting sort by one CTA (the sums over a coverage vector
// run in this order, so it has to be the same on every call).  Each warp takes a run of consecutive samples and has counters of its own.
constexpr int kOrderSteps = 8;            // of 32 samples whose trips to memory a warp has under way together
__global__ void __launch_bounds__(1024) objective_order_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ perm,
                                                              const int32_t *__restrict__ assignment, int32_t W,
                                                              int32_t *__restrict__ order, int32_t *__restrict__ blockOf)
{
    extern __shared__ int32_t shCount[];                   // [warps][W + 1]
    const ClassDesc c = desc[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5, B = W + 1;
    const int per = ((c.M + warps - 1) / warps + 31) & ~31, v0 = min(c.M, warp * per), v1 = min(c.M, v0 + per);
    int32_t *const mine = shCount + warp * B;
    for (int p = lane; p < B; p += 32) mine[p] = 0;
    __syncwarp();
    int sample[kOrderSteps], block[kOrderSteps];
    auto load = [&](int v) {
#pragma unroll
        for (int u = 0; u < kOrderSteps; ++u) sample[u] = v + u * 32 + lane < v1 ? perm[c.row0 + v + u * 32 + lane] : -1;
#pragma unroll
        for (int u = 0; u < kOrderSteps; ++u) {
            const int a = sample[u] >= 0 ? assignment[sample[u]] : W;
            block[u] = a >= 0 && a < W ? a : W;
        }
    };
    for (int v = v0; v < v1; v += kOrderSteps * 32) {
        load(v);
#pragma unroll
        for (int u = 0; u < kOrderSteps; ++u) {
            if (v + u * 32 >= v1) break;
            const unsigned same = __match_any_sync(0xffffffffu, sample[u] >= 0 ? block[u] : -1);
            if (sample[u] >= 0 && (same & ((1u << lane) - 1u)) == 0) mine[block[u]] += __popc(same);
            __syncwarp();
        }
    }
    __syncthreads();
    if (warp == 0) {                                       // first places: block after block, in each warp after warp
        int run = 0;
        for (int p0 = 0; p0 < B; p0 += 32) {
            const int p = p0 + lane;
            int n = 0;
            if (p < B)
                for (int w = 0; w < warps; ++w) n += shCount[w * B + p];
            int sum = n;
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, sum, off);
                if (lane >= off) sum += up;
            }
            if (p < B) {
                int at = run + sum - n;
                for (int w = 0; w < warps; ++w) {
                    const int k = shCount[w * B + p];
                    shCount[w * B + p] = at;
                    at += k;
                }
            }
            run += __shfl_sync(0xffffffffu, sum, 31);
        }
    }
    __syncthreads();
    for (int v = v0; v < v1; v += kOrderSteps * 32) {
        if (per > kOrderSteps * 32) load(v);               // (else they are still in the registers)
#pragma unroll
        for (int u = 0; u < kOrderSteps; ++u) {
            if (v + u * 32 >= v1) break;
            const unsigned same = __match_any_sync(0xffffffffu, sample[u] >= 0 ? block[u] : -1);
            const int rank = __popc(same & ((1u << lane) - 1u));
            const int at = sample[u] >= 0 ? mine[block[u]] + rank : 0;
            __syncwarp();
            if (sample[u] >= 0) {
                if (rank == 0) mine[block[u]] = at + __popc(same);
                order[c.row0 + at] = sample[u];
                blockOf[c.row0 + at] = block[u] < W ? block[u] : -1;
            }
            __syncwarp();
        }
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

// f of one (class, block): the sum of its coverage vector, by `team` warps (1 or 8), in a fixed order.
template <typename SV, typename FV>
__global__ void __launch_bounds__(256) objective_sum_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ cover, int32_t L, int32_t W, int32_t team,
                                                           FV *__restrict__ partValues)
{
    __shared__ FV sh[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t idx = team == 1 ? (int64_t)blockIdx.x * 8 + warp : (int64_t)blockIdx.x;
    if (idx >= (int64_t)L * W) return;
    const ClassDesc c = desc[idx / W];
    const int4 *v = reinterpret_cast<const int4 *>(cover + c.vOff + (idx % W) * c.ld);
    FV s = (FV)0;
    for (int q = team == 1 ? lane : (int)threadIdx.x; q < c.ld / 4; q += 32 * team) {
        const int4 x = v[q];
        if constexpr (std::is_integral<SV>::value) s += (FV)x.x + (FV)x.y + (FV)x.z + (FV)x.w;
        else s += (FV)__int_as_float(x.x) + (FV)__int_as_float(x.y) + (FV)__int_as_float(x.z) + (FV)__int_as_float(x.w);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (team == 1) {
        if (lane == 0) partValues[idx] = s;
        return;
    }
    if (lane == 0) sh[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += sh[w];
        partValues[idx] = s;
    }
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
static rcd_status run_objective(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const int32_t *assignment, bool covered, void *partValues, void *total,
                                cudaStream_t st)
{
    const int64_t rowBlocks = (sz.maxM + kObjRows - 1) / kObjRows;
    if (!covered && (sz.L > 65535 || rowBlocks > 65535)) return fail(ctx, RCD_ERR_UNSUPPORTED, "objective: more than 65535 classes or row blocks");
    int32_t *members = ws.cand, *counts = ws.cnt, *cover = (int32_t *)ws.cover;
    if (sz.maxM > 0 && !covered) {
        RCD_CUDA(ctx, cudaMemsetAsync(cover, 0, (size_t)sz.vElems * sizeof(int32_t), st));
        objective_members_kernel<<<sz.L, 512, (size_t)sz.W * 4, st>>>(ws.desc, ws.perm, assignment, sz.W, members, counts);
        const dim3 grid((unsigned)((pad_row(sz.maxM) + 4 * kObjThreads - 1) / (4 * kObjThreads)), (unsigned)rowBlocks, (unsigned)sz.L);
        objective_cover_kernel<SV><<<grid, kObjThreads, 0, st>>>(ws.desc, (const SV *)ws.S, members, counts, sz.W, cover);
        ctx->kernelLaunches += 2;
    }
    const int64_t n = (int64_t)sz.L * sz.W;
    // (few long vectors: 8 warps each; 80 of 5000 entries 12.4 us by one)
    const int team = n <= 2048 && sz.maxM > 512 ? 8 : 1;
    objective_sum_kernel<SV, FV><<<(unsigned)((n * team + 7) / 8), 256, 0, st>>>(ws.desc, cover, sz.L, sz.W, team, (FV *)partValues);
    objective_total_kernel<FV><<<1, 256, 0, st>>>((const FV *)partValues, n, (FV *)total);
    ctx->kernelLaunches += 2;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_objective_order(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const int32_t *assignment, cudaStream_t st)
{
    if (sz.L > 65535 || (sz.maxM + kObjRows - 1) / kObjRows > 65535) return fail(ctx, RCD_ERR_UNSUPPORTED, "objective: more than 65535 classes or row blocks");
    if (sz.maxM == 0) return RCD_OK;
    RCD_CUDA(ctx, cudaMemsetAsync(ws.cover, 0, (size_t)sz.vElems * sizeof(int32_t), st));
    // as many warps as the counters leave room for in 48 KB (W = 1024: 11), no more than a class of this size keeps busy
    const int warps = (int)std::min<int64_t>(std::min(32, 48 * 1024 / (4 * (sz.W + 1))), (sz.maxM + 31) / 32);
    objective_order_kernel<<<sz.L, warps * 32, (size_t)warps * (sz.W + 1) * 4, st>>>(ws.desc, ws.perm, assignment, sz.W, ws.cand, ws.pos);
    ctx->kernelLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_objective(rcd_ctx *ctx, rcd_feat_dtype dtype, const Sizes &sz, const Workspace &ws, const int32_t *assignment,
                            bool covered, void *partValues, void *total, cudaStream_t st)
{
    if (dtype == RCD_FEAT_I8) return run_objective<int32_t, long long>(ctx, sz, ws, assignment, covered, partValues, total, st);
    return run_objective<float, double>(ctx, sz, ws, assignment, covered, partValues, total, st);
}

}  // namespace rcd
