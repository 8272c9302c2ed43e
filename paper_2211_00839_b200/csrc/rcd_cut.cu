// Algorithm 1 with the graph-cut objective of Section 4, item 2:
//     f(A) = sum_{v in V_l \ A} sum_{v' in A} S[v][v'].
// With S symmetric and tie_p[u] = sum_{a in A_p} S[u][a],
//     f(A_p u {u}) - f(A_p) = (sum_v S[v][u] - S[u][u]) - 2 tie_p[u] = base[u] - 2 tie_p[u],
// so a pick needs no pass over S at all: an argmax over M values, then tie_p += row v* of S.
// One CTA per class runs the class to completion (classes are independent); the whole objective
// costs O(M) per pick.  Values: int64 for int8 features (exact), double otherwise.
// The objective is not monotone (a sample that joins A stops being cut), gains may be negative;
// Algorithm 1 runs unchanged: least-f non-full block, argmax with lowest-index ties.
#include "rcd_cut_plan.h"
#include "rcd_exact.cuh"

#include <limits.h>
#include <algorithm>
#include <type_traits>

namespace rcd {

constexpr int kCutThreads = 512;
constexpr int kCutMaxBlocks = 1024;

template <typename SV> struct CutArith { using FV = double; };
template <> struct CutArith<int32_t> { using FV = long long; };

template <typename SV>
struct CutParams {
    using FV = typename CutArith<SV>::FV;
    const ClassDesc *desc;
    const SV *S;
    FV *tie;            // [sum W*ld] tie_p[u]
    FV *base;           // [N]        column sum minus the diagonal entry, class-sorted order
    FV *fval;           // [L][W]
    const int32_t *quota;
    int32_t *pos;       // [N] >= 0 while the sample is unassigned
    const int32_t *perm;
    int32_t *assignment;
    int32_t *order;     // may be null
    int32_t *status;
    int32_t L, W;
};

template <typename SV>
__global__ void __launch_bounds__(kCutThreads, 2) cut_chain_kernel(CutParams<SV> prm)
{
    using FV = typename CutArith<SV>::FV;
    __shared__ FV shF[kCutMaxBlocks];
    __shared__ int32_t shRoom[kCutMaxBlocks];
    __shared__ unsigned long long shG[kCutThreads / 32];      // order-preserving images of the warps' best gains
    __shared__ int shV[kCutThreads / 32];
    __shared__ int shPick, shBlock;
    const int l = blockIdx.x;
    const ClassDesc c = prm.desc[l];
    const int W = prm.W;
    if (c.M == 0) {                                           // empty class: every block has value 0
        for (int p = threadIdx.x; p < W; p += kCutThreads) prm.fval[(int64_t)l * W + p] = 0;
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const SV *Sl = prm.S + c.sOff;
    FV *base = prm.base + c.row0;
    FV *tie = prm.tie + c.vOff;
    int32_t *pos = prm.pos + c.row0;

    // base[u] = sum_v S[v][u] - S[u][u]  (row sum of the symmetric S, one warp per row, lanes in fixed order)
    for (int u = warp; u < c.M; u += kCutThreads / 32) {
        const SV *row = Sl + (int64_t)u * c.ld;
        FV acc = 0;
        for (int j = lane; j < c.M; j += 32) acc += (FV)row[j];
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) base[u] = acc - (FV)row[u];
    }
    for (int64_t i = threadIdx.x; i < (int64_t)W * c.ld; i += kCutThreads) tie[i] = 0;
    for (int u = threadIdx.x; u < c.M; u += kCutThreads) pos[u] = u;
    for (int p = threadIdx.x; p < W; p += kCutThreads) { shF[p] = 0; shRoom[p] = prm.quota[(int64_t)l * W + p]; }
    __syncthreads();

    for (int t = 0; t < c.M; ++t) {
        // j* = argmin over non-full blocks of f, ties -> lowest index
        if (warp == 0) {
            FV bestF = 0;
            int bestP = INT_MAX;
            for (int p = lane; p < W; p += 32)
                if (shRoom[p] > 0 && (bestP == INT_MAX || shF[p] < bestF)) { bestF = shF[p]; bestP = p; }
            // (three warp-wide reductions on an order-preserving image of f: least f, lowest index among equals)
            unsigned long long of = ordered_u64(bestF);
            warp_argmin_ordered(of, bestP);
            if (lane == 0) shBlock = bestP;
        }
        __syncthreads();
        const int j = shBlock;
        if (j == INT_MAX) {                                   // samples left but every block is full
            if (threadIdx.x == 0) atomicOr(prm.status, kDevNoCandidate);
            return;
        }
        // v* = argmax over the unassigned samples of base[u] - 2 tie_j[u], ties -> lowest index
        const FV *tj = tie + (int64_t)j * c.ld;
        FV bestG = 0;
        int bestV = INT_MAX;
#pragma unroll 4
        for (int u = threadIdx.x; u < c.M; u += kCutThreads) {
            const FV g = base[u] - 2 * tj[u];
            if (pos[u] >= 0 && (bestV == INT_MAX || g > bestG)) { bestG = g; bestV = u; }
        }
        // greatest gain, lowest index among equals: over the warp, then over the warps' results
        unsigned long long og = ordered_u64(bestG);
        warp_argmax_ordered(og, bestV);
        if (lane == 0) { shG[warp] = og; shV[warp] = bestV; }
        __syncthreads();
        if (warp == 0) {
            og = lane < kCutThreads / 32 ? shG[lane] : 0ull;
            bestV = lane < kCutThreads / 32 ? shV[lane] : INT_MAX;
            warp_argmax_ordered(og, bestV);
            if constexpr (std::is_same<FV, double>::value) bestG = from_ordered_u64_d(og);
            else bestG = from_ordered_u64_ll(og);
            if (lane == 0) {
                shPick = bestV;
                if (bestV != INT_MAX) {
                    shF[j] += bestG;
                    shRoom[j] -= 1;
                    pos[bestV] = -1;
                    const int global = prm.perm[c.row0 + bestV];
                    prm.assignment[global] = j;
                    if (prm.order) prm.order[c.row0 + t] = global;
                }
            }
        }
        __syncthreads();
        const int vstar = shPick;
        if (vstar == INT_MAX) {
            if (threadIdx.x == 0) atomicOr(prm.status, kDevBadState);
            return;
        }
        // tie_j[u] += S[v*][u]
        {
            FV *tw = tie + (int64_t)j * c.ld;
            const SV *row = Sl + (int64_t)vstar * c.ld;
            for (int u = threadIdx.x; u < c.M; u += kCutThreads) tw[u] += (FV)row[u];
        }
        __syncthreads();
    }
    for (int p = threadIdx.x; p < W; p += kCutThreads) prm.fval[(int64_t)l * W + p] = shF[p];
}

// ---- integer similarities: a cluster per class, all warps in step ------------------------------
// What bounds the alternatives.  One CTA per class with everything in global memory (cut_chain_kernel) takes 7.6 us per pick.  In the
// cluster form (rcd_cluster.cu) picks of different blocks overlap, but under this objective all blocks want the same samples, so half the
// notes of 10 classes of 5000 into 8 blocks are stale when their block's turn comes, and a pick takes 1.8 us.  Here a thread keeps some
// columns of the class, with their gains for every block in shared memory, and nothing goes stale: all warps post their best unassigned
// candidate for the block that is next to every CTA, and when all have arrived everybody knows the pick.  The sample's row of S is asked for
// then, and taken off the block's gains two picks later (or where the block comes again before), so that the trip to memory passes under
// other picks.  One more warp per CTA keeps the blocks' values and prepares the choice of the next block.
//
// What bounds it (10 classes of 5000 into 8 blocks, 8 CTAs each, 2700 cycles a pick): instructions of one warp after another, half of them
// for the candidates and the row's loads.  Whole calls, before and now: 3 classes of 1300 into 20 blocks 2103 and 1120 us, 30 of 2500 into 8
// blocks 5060 and 3644, 200 of 700 into 8 blocks 2886 and 1247.
struct LockParams {
    const ClassDesc *desc;
    const int32_t *S;
    long long *base;           // [N] column sum minus the diagonal entry, class-sorted order
    unsigned long long *top;   // [L] zero at the start: largest sum of |S| over a row
    long long *fval;           // [L][W]
    const int32_t *quota;
    const int32_t *perm;
    const int32_t *classOrder;
    uint32_t *picks;           // [N] sample | block << 16, in the order picked
    int32_t *assignment;
    int32_t *order;            // may be null
    int32_t *status;
    unsigned long long *stats; // phase words
    int32_t W;
    int32_t columns;           // of a CTA (its gains: [W][columns])
    uint32_t one;              // the value 1, opaque to the compiler
};

__device__ __forceinline__ void lock_barrier(bool alone)
{
    if (alone) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Over a cluster the candidates travel as asynchronous stores that count towards an mbarrier of the CTA they reach (phases of two picks in
// turn).  A cluster's own barrier for every pick, whose release waits for the rows on their way, cost 700 cycles of 3200.
__device__ __forceinline__ uint32_t lock_remote(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void lock_send(const unsigned long long *to, unsigned long long v, uint32_t bar, uint32_t rank)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" :: "r"(lock_remote(smem32(to), rank)), "l"(v), "r"(lock_remote(bar, rank)) : "memory");
}
__device__ __forceinline__ bool lock_wait(uint32_t bar, uint32_t parity)
{
    for (unsigned k = 0; k < (1u << 28); ++k) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) {
            // (what the stores brought is not read before this; only shared memory: an acquire of everything would drop the L1's lines)
            asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
            return true;
        }
    }
    return false;
}

// K: columns per thread; KW: blocks per lane of the leader.
template <int K, int KW>
__global__ void __launch_bounds__((kLockWarps + 1) * 32) cut_lockstep_kernel(const __grid_constant__ LockParams prm)
{
    extern __shared__ __align__(16) unsigned char shared[];
    __shared__ unsigned long long shBest[2][kLockCtas * kLockWarps];           // the warps' best candidates, for two picks in turn
    // by the leader of each CTA: the least value << 7 | block among the blocks with room but the next | 1 << 63: the next has room for one only
    __shared__ unsigned long long shOthers[2][kLockCtas];
    __shared__ __align__(8) unsigned long long shBars[2];
    uint32_t rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const bool alone = C == 1;
    const int l = prm.classOrder[blockIdx.x / C], W = prm.W, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int NW = (int)(blockDim.x >> 5) - 1, NT = NW * 32, entries = NW * (int)C;
    const ClassDesc c = prm.desc[l];
    const int M = c.M;
    if (M == 0) {                                          // empty class: every block has value 0
        if (rank == 0) for (int p = threadIdx.x; p < W; p += blockDim.x) prm.fval[(int64_t)l * W + p] = 0;
        return;
    }
    const int32_t *const Sl = prm.S + c.sOff;
    long long *const base = prm.base + c.row0;
    unsigned long long *const gains = reinterpret_cast<unsigned long long *>(shared) + threadIdx.x;  // of block j, k-th column: [j * prm.columns + k * NT]
    const int column = (int)rank * prm.columns + threadIdx.x;

    const uint32_t bars = smem32(shBars);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 2; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bars + 8 * k) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp < NW) {
        unsigned long long top = 0;
        for (int u = (int)rank * NW + warp; u < M; u += entries) {
            unsigned long long neg;
            const unsigned long long pos = row_value<true>(reinterpret_cast<const int4 *>(Sl + (int64_t)u * c.ld), c.ld >> 2, lane, prm.one, neg);
            top = umax(top, pos + neg);
            if (lane == 0) __stcg(base + u, (long long)(pos - neg) - (long long)Sl[(int64_t)u * c.ld + u]);
        }
        if (lane == 0 && top) atomicMax(prm.top + l, top);
    }
    unsigned long long f[KW], least;                       // value << 7 | block; least: of the block that is next
    int room[KW];
    auto least_but = [&](int but) {
        unsigned long long m = ~0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k) m = room[k] > 0 && lane + 32 * k != but ? umin(m, f[k]) : m;
        return ~warp_max_u64(~m);
    };
#pragma unroll
    for (int k = 0; k < KW; ++k) {                         // (every warp finds the first block; the leader goes on with these)
        f[k] = (kTrackedZero << 7) | (unsigned long long)(lane + 32 * k);
        room[k] = lane + 32 * k < W ? prm.quota[(int64_t)l * W + lane + 32 * k] : 0;
    }
    least = least_but(-1);
    lock_barrier(alone);
    // gains lie within three times the largest sum of |S| over a row, either way
    const unsigned long long bias = 3 * __ldcg(prm.top + l) + 1;
    unsigned gone = 0;                                     // columns that are assigned or beyond the class
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int u = column + k * NT;
        const bool own = warp < NW && k * NT + (int)threadIdx.x < prm.columns;
        const unsigned long long g = own && u < M ? (unsigned long long)__ldcg(base + u) + bias : 0ull;
        if (own)
            for (int p = 0; p < W; ++p) gains[p * prm.columns + k * NT] = g;
        gone |= own && u < M ? 0u : 1u << k;
    }
    struct Owed {                                          // the row of a sample picked lately, for its block (-1: none)
        int32_t row[K];
        int block;
    } even, odd;
    even.block = odd.block = -1;
    auto settle = [&](Owed &o) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k * NT + (int)threadIdx.x < prm.columns) gains[o.block * prm.columns + k * NT] -= 2ll * o.row[k];
        o.block = -1;
    };
    // (mine: of the pick before the last, and then of this one; last: of the pick before)
    auto make_pick = [&](int t, Owed &mine, Owed &last) {
        const int j = (int)(least & 127);
        const uint32_t bar = bars + 8 * (t & 1);
        if (!alone && threadIdx.x == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"((uint32_t)((entries + (int)C) * 8)) : "memory");
        if (warp < NW) {
            if (last.block == j) settle(last);
            if (mine.block == j) settle(mine);
            unsigned long long best = 0;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (!(gone >> k & 1)) best = umax(best, make_key(gains[j * prm.columns + k * NT], column + k * NT));
            best = warp_max_u64(best);
            unsigned long long *const to = &shBest[t & 1][rank * NW + warp];
            if (!alone) {
                if (lane < (int)C) lock_send(to, best, bar, lane);
            } else if (lane == 0) {
                *to = best;
            }
            if (mine.block >= 0) settle(mine);
        } else {
            const unsigned long long others = least_but(j);
            int left = room[0];
#pragma unroll
            for (int k = 1; k < KW; ++k) left ^= (left ^ room[k]) & (j >> 5 == k ? ~0 : 0);
            left = __shfl_sync(0xffffffffu, left, j & 31);
            // (to every CTA: nobody writes to candidates that a leader may still be reading)
            const unsigned long long word = others & ~(1ull << 63) | (left > 1 ? 0ull : 1ull << 63);
            if (!alone) {
                if (lane < (int)C) lock_send(&shOthers[t & 1][rank], word, bar, lane);
            } else if (lane == 0) {
                shOthers[t & 1][0] = word;
            }
        }
        if (alone) {
            __syncthreads();
        } else if (!lock_wait(bar, (uint32_t)t >> 1 & 1)) {
            if (lane == 0) atomicOr(prm.status, kDevTimeout);
            return false;
        }
        unsigned long long best = 0;
        for (int i = lane; i < entries; i += 32) best = umax(best, shBest[t & 1][i]);
        best = warp_max_u64(best);
        unsigned long long others = shOthers[t & 1][rank];
        const unsigned long long inc = ((best >> 16) - bias) << 7;
        const bool more = !(others >> 63);
        others &= ~(1ull << 63);
        others = others == ~(1ull << 63) ? ~0ull : others;     // (none)
        const int v = key_sample(best);
        least = umin(others, more ? least + inc : ~0ull);
        if (warp < NW) {
            if (more) {                                    // (a full block needs no gains any more)
                const int32_t *const from = Sl + (int64_t)v * c.ld + column;
#pragma unroll
                for (int k = 0; k < K; ++k) mine.row[k] = k * NT + (int)threadIdx.x < prm.columns && column + k * NT < M ? __ldg(from + k * NT) : 0;
                mine.block = j;
            }
#pragma unroll
            for (int k = 0; k < K; ++k) gone |= column + k * NT == v ? 1u << k : 0u;
        } else {
#pragma unroll
            for (int k = 0; k < KW; ++k) {
                f[k] += lane + 32 * k == j ? inc : 0ull;
                room[k] -= lane + 32 * k == j ? 1 : 0;
            }
            // (a load in front of the stores that need it would hold up every pick)
            if (rank == 0 && lane == 0) prm.picks[c.row0 + t] = (uint32_t)v | (uint32_t)j << 16;
        }
        if (best == 0 || (least == ~0ull && t + 1 < M)) {  // (cannot be: samples are left, and the quotas add up to M)
            if (threadIdx.x == 0) atomicOr(prm.status, kDevNoCandidate);
            return false;
        }
        return true;
    };
    for (int t = 0; t < M; t += 2) {
        if (!make_pick(t, even, odd)) break;
        if (t + 1 < M && !make_pick(t + 1, odd, even)) break;
    }
    if (rank == 0 && warp == NW) {
#pragma unroll
        for (int k = 0; k < KW; ++k)
            if (lane + 32 * k < W) prm.fval[(int64_t)l * W + lane + 32 * k] = (long long)(f[k] >> 7) - (long long)kTrackedZero;
        // every pick but the last of a block takes the sample's own row off its gains (no other: as the cluster form counts)
        int blocks = 0;
#pragma unroll
        for (int k = 0; k < KW; ++k) blocks += __popc(__ballot_sync(0xffffffffu, lane + 32 * k < W && prm.quota[(int64_t)l * W + lane + 32 * k] > 0));
        if (lane == 0) atomicAdd(prm.stats + 15, (unsigned long long)(M - blocks));
    }
    lock_barrier(alone);                                   // (and nobody writes to a CTA that has gone)
    // class-local picks -> outputs (none where the loop stopped early: the words behind the last pick are whatever memory held)
    const bool stopped = __ldcg(prm.status) != 0;
    for (int t = (int)(rank * blockDim.x + threadIdx.x); t < M; t += (int)(C * blockDim.x)) {
        const uint32_t p = __ldcg(prm.picks + c.row0 + t);
        if (stopped) break;
        const int global = prm.perm[c.row0 + (p & 0xffff)];
        prm.assignment[global] = (int)(p >> 16);
        if (prm.order) prm.order[c.row0 + t] = global;
    }
}

typedef void (*LockKernel)(LockParams);
template <int KW>
static LockKernel pick_lockstep(int K)
{
    return K == 1 ? cut_lockstep_kernel<1, KW> : K == 2 ? cut_lockstep_kernel<2, KW> : K == 3 ? cut_lockstep_kernel<3, KW> : K <= 4 ? cut_lockstep_kernel<4, KW> : cut_lockstep_kernel<kLockColumns, KW>;
}

static LockKernel lock_kernel(const Sizes &sz, const LockPlan &plan)
{
    return sz.W <= 32 ? pick_lockstep<1>(plan.K) : sz.W <= 64 ? pick_lockstep<2>(plan.K) : pick_lockstep<4>(plan.K);
}

static cudaError_t allow_lockstep(const rcd_ctx *ctx, LockKernel kernel)
{
    const cudaError_t e = allow_shared(kernel, lock_shared(ctx->maxSmemOptin));
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

static cudaLaunchConfig_t lock_launch(const LockPlan &plan, int threads, size_t smem, int clusters, cudaLaunchAttribute *attr, cudaStream_t st)
{
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)plan.C;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * plan.C));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Whether the GPU can place a cluster of that many CTAs, with all the shared memory that a plan may ask for (a partition of a GPU may
// not: the launch would be refused).  Asked once per context and size.
static bool lock_clusters_fit(rcd_ctx *ctx, const Sizes &sz, const LockPlan &plan)
{
    int idx = 0;
    while ((1 << idx) < plan.C) ++idx;
    int &fits = ctx->lockClusters[idx];
    if (fits < 0) {
        const LockKernel kernel = lock_kernel(sz, plan);
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = lock_launch(plan, (kLockWarps + 1) * 32, (size_t)lock_shared(ctx->maxSmemOptin), 1, attr, nullptr);
        int active = 0;
        if (allow_lockstep(ctx, kernel) != cudaSuccess || cudaOccupancyMaxActiveClusters(&active, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            active = 0;
        }
        fits = active;
    }
    return fits > 0;
}

static bool plan_lockstep(rcd_ctx *ctx, const Sizes &sz, LockPlan &plan)
{
    if (!library_chooses(ctx->cfg)) return false;
    for (int most = kLockCtas;; most = plan.C / 2) {
        if (!lock_plan(ctx->smCount, ctx->maxSmemOptin, most, sz, plan)) return false;
        if (plan.C == 1 || lock_clusters_fit(ctx, sz, plan)) return true;
    }
}

bool cut_in_step(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, double otherCycles)
{
    LockPlan plan;
    if (!plan_lockstep(ctx, sz, plan)) return false;
    if (otherCycles <= 0) otherCycles = cut_chain_cycles(ctx->smCount, descHost);
    return cut_steps_cycles(ctx->smCount, ctx->maxSmemOptin, plan, descHost) <= otherCycles;
}

static rcd_status run_lockstep(rcd_ctx *ctx, const LockPlan &plan, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order, cudaStream_t st)
{
    LockParams prm;
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.base = (long long *)ws.cutBase;
    prm.top = ws.topGain;
    prm.fval = (long long *)ws.fval;
    prm.quota = ws.quota;
    prm.perm = ws.perm;
    prm.classOrder = ws.classOrder;
    prm.picks = (uint32_t *)ws.cand;
    prm.assignment = assignment;
    prm.order = order;
    prm.status = ctx->statusOwn;
    prm.stats = ws.phaseNs;
    prm.W = sz.W;
    prm.columns = plan.columns;
    prm.one = 1u;
    const LockKernel kernel = lock_kernel(sz, plan);
    RCD_CUDA(ctx, allow_lockstep(ctx, kernel));
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = lock_launch(plan, (plan.warps + 1) * 32, plan.smem, sz.L, attr, st);
    RCD_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, prm));
    ctx->kernelLaunches++;
    return RCD_OK;
}

rcd_status launch_cut_stopped_selftest(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order, cudaStream_t st)
{
    const int words = (int)(sz.maxM + 63) / 64;                          // of 32 columns, of each of two CTAs
    const LockPlan plan{2, 1, std::min(kLockWarps, words), words * 32, (size_t)sz.W * words * 32 * 8};
    return run_lockstep(ctx, plan, sz, ws, assignment, order, st);
}

// f(A_p) for every block from the definition: per row v the sums r_p(v) = sum_{a in A_p} S[v][a], then
// f_p += r_p(v) for every block p that v is not in.  int64 sums are exact; fp64 sums inside a row are
// accumulated with shared-memory atomics, so their last bits can differ from run to run.
template <typename SV>
__global__ void __launch_bounds__(256, 4) cut_objective_rows_kernel(const ClassDesc *__restrict__ desc, const SV *__restrict__ S,
                                                                   const int32_t *__restrict__ perm,
                                                                   const int32_t *__restrict__ assignment, int32_t W,
                                                                   int32_t maxBlocks,
                                                                   typename CutArith<SV>::FV *__restrict__ partial)
{
    using FV = typename CutArith<SV>::FV;
    using AT = typename std::conditional<std::is_integral<SV>::value, unsigned long long, double>::type;
    extern __shared__ unsigned char shraw[];
    AT *shSum = reinterpret_cast<AT *>(shraw);                  // [8 warps][W] block totals of this CTA's rows
    AT *shRow = shSum + (size_t)8 * W;                          // [8 warps][W] sums of the current row
    const int l = blockIdx.y;
    const ClassDesc c = desc[l];
    const int first = blockIdx.x * 64;
    if (first >= c.M) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    AT *sum = shSum + (size_t)warp * W, *cur = shRow + (size_t)warp * W;
    for (int p = lane; p < W; p += 32) sum[p] = 0;
    const int32_t *pl = perm + c.row0;
    for (int r = warp; r < 64; r += 8) {
        const int v = first + r;
        if (v >= c.M) break;
        for (int p = lane; p < W; p += 32) cur[p] = 0;
        __syncwarp();
        const SV *row = S + c.sOff + (int64_t)v * c.ld;
        for (int a = lane; a < c.M; a += 32) {
            const int p = assignment[pl[a]];
            if (p >= 0 && p < W) atomicAdd(&cur[p], (AT)(FV)row[a]);       // int64 wraps like two's complement
        }
        __syncwarp();
        const int mine = assignment[pl[v]];
        for (int p = lane; p < W; p += 32) if (p != mine) sum[p] += cur[p];
        __syncwarp();
    }
    __syncthreads();
    FV *out = partial + ((int64_t)l * maxBlocks + blockIdx.x) * W;
    for (int p = threadIdx.x; p < W; p += blockDim.x) {
        AT s = 0;
        for (int w = 0; w < 8; ++w) s += shSum[(size_t)w * W + p];
        out[p] = (FV)s;
    }
}

template <typename FV>
__global__ void cut_objective_reduce_kernel(const ClassDesc *__restrict__ desc, const FV *__restrict__ partial, int32_t L,
                                            int32_t W, int32_t maxBlocks, FV *__restrict__ partValues)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)L * W) return;
    const int l = (int)(idx / W), p = (int)(idx % W);
    const int nb = (desc[l].M + 63) / 64;
    FV s = 0;
    for (int b = 0; b < nb; ++b) s += partial[((int64_t)l * maxBlocks + b) * W + p];
    partValues[idx] = s;
}

template <typename FV>
__global__ void __launch_bounds__(256, 1) cut_objective_total_kernel(const FV *__restrict__ partValues, int64_t n, FV *__restrict__ total)
{
    __shared__ FV sh[256];
    FV s = 0;
    for (int64_t i = threadIdx.x; i < n; i += 256) s += partValues[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = sh[0];
}

template <typename SV>
static rcd_status run_cut(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order, cudaStream_t st)
{
    using FV = typename CutArith<SV>::FV;
    if (sz.W > kCutMaxBlocks) return fail(ctx, RCD_ERR_UNSUPPORTED, "graph cut: at most %d blocks", kCutMaxBlocks);
    CutParams<SV> prm;
    prm.desc = ws.desc;
    prm.S = (const SV *)ws.S;
    prm.tie = (FV *)ws.gains;
    prm.base = (FV *)ws.cutBase;
    prm.fval = (FV *)ws.fval;
    prm.quota = ws.quota;
    prm.pos = ws.pos;
    prm.perm = ws.perm;
    prm.assignment = assignment;
    prm.order = order;
    prm.status = ctx->statusOwn;
    prm.L = sz.L;
    prm.W = sz.W;
    cut_chain_kernel<SV><<<sz.L, kCutThreads, 0, st>>>(prm);
    ctx->kernelLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_cut(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, bool inStep, int32_t *assignment, int32_t *order, cudaStream_t st)
{
    if (sz.L == 0 || sz.maxM == 0) return RCD_OK;
    ctx->greedyForm = RCD_FORM_CUT_CHAIN;
    ctx->steps = sz.maxM;
    LockPlan plan;
    if (inStep && plan_lockstep(ctx, sz, plan)) {
        ctx->greedyForm = RCD_FORM_CUT_STEPS;
        ctx->phaseNsDev = ws.phaseNs;
        return run_lockstep(ctx, plan, sz, ws, assignment, order, st);
    }
    if (sz.floatArith) return run_cut<float>(ctx, sz, ws, assignment, order, st);
    return run_cut<int32_t>(ctx, sz, ws, assignment, order, st);
}

template <typename SV>
static rcd_status run_cut_objective(rcd_ctx *ctx, const Sizes &sz, const ClassDesc *descDev, const void *S, const int32_t *perm,
                                    const int32_t *assignment, void *partValues, void *total, void *scratch, cudaStream_t st)
{
    using FV = typename CutArith<SV>::FV;
    const int maxBlocks = (int)((sz.maxM + 63) / 64);
    const size_t smem = (size_t)16 * sz.W * 8;
    if ((int64_t)smem > whole_shared(ctx)) return fail(ctx, RCD_ERR_UNSUPPORTED, "W=%d too large for the cut objective kernel", sz.W);
    if (sz.L > 65535) return fail(ctx, RCD_ERR_UNSUPPORTED, "objective: more than 65535 classes");
    RCD_CUDA(ctx, allow_shared(cut_objective_rows_kernel<SV>, whole_shared(ctx)));
    if (maxBlocks > 0) {
        dim3 grid(maxBlocks, sz.L);
        cut_objective_rows_kernel<SV><<<grid, 256, smem, st>>>(descDev, (const SV *)S, perm, assignment, sz.W, maxBlocks, (FV *)scratch);
        ctx->kernelLaunches++;
    }
    const int64_t n = (int64_t)sz.L * sz.W;
    cut_objective_reduce_kernel<FV><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(descDev, (const FV *)scratch, sz.L, sz.W, maxBlocks, (FV *)partValues);
    cut_objective_total_kernel<FV><<<1, 256, 0, st>>>((const FV *)partValues, n, (FV *)total);
    ctx->kernelLaunches += 2;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_cut_objective(rcd_ctx *ctx, const Sizes &sz, const ClassDesc *descDev, const void *S, const int32_t *perm,
                                const int32_t *assignment, void *partValues, void *total, void *scratch, cudaStream_t st)
{
    if (sz.floatArith) return run_cut_objective<float>(ctx, sz, descDev, S, perm, assignment, partValues, total, scratch, st);
    return run_cut_objective<int32_t>(ctx, sz, descDev, S, perm, assignment, partValues, total, scratch, st);
}

}  // namespace rcd
