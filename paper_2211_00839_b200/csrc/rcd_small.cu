// The greedy loop of Algorithm 1 for classes whose similarity matrix fits the shared memory of one SM, one CTA per class: the form
// the library chooses for small classes, with the facility-location and (integers) the graph-cut objective.
//
// What bounds the alternative.  The cluster form (rcd_cluster.cu) hides trips to L2 behind the picks of other blocks; with small
// classes there is little to hide, and what remains is the hand-over between its leader and its teams, 1 us per pick and more.  Here a
// thread keeps one candidate, and all warps make every pick together, with two barriers:
//   the warps     post their best unassigned candidate for the block that is next;
//   a barrier     and everybody knows the pick: the warps list the columns it raised, each its own, while one more warp, the leader,
//                 chooses the next block (what does not depend on the pick is computed before the barrier);
//   a barrier     and the warps take the listed columns' rows of S off their candidates' gains.
// Gains and coverage are read and written by the one thread that owns the column, so only candidates and lists cross warps.
//
// What bounds it: the chain of a pick, 900 to 1100 cycles, of which 340 go into the candidates (two warp-wide maxima of 64 bits, 56 cycles
// each, and 25 of a barrier), as much into the row and its list, and 12 cycles per raised column once more than a few rise.  Whole calls, in us, the
// cluster form and this one: 2 classes of 200 int8 into 4 blocks 236 and 153 (138 with the class split in two launches); 10 of 160 into 32 blocks 332 and 215; 1000 of 100 into 8 blocks
// 896 and 294; 35 of 128 bf16 into 22 blocks 300 and 211; graph cut, 60 of 180 into 12 blocks 255 and 103.
//
// Results are those of the other forms bit for bit: gains are exact integers, decisions are made in the same order.
#include "rcd_exact.cuh"

#include <algorithm>

namespace rcd {

struct SmallParams {
    const ClassDesc *desc;
    const int32_t *S;
    const int32_t *perm;
    const int32_t *quota;
    long long *fval;           // [L][W]
    int32_t *assignment, *order;
    const int32_t *fixedExp;   // [L] floating-point similarities: their fixed-point scale (null: integers)
    const int32_t *classOrder;
    int32_t *status;
    unsigned long long *stats; // phase words
    int32_t W;
    int32_t ld;                // of a block's vectors in shared memory
    int32_t toFix;             // S holds floating-point dot products
    uint32_t one;              // the value 1, opaque to the compiler
    int32_t offCover, offGains, offList, offPicks;   // dynamic shared memory (S comes first)
};

namespace {

constexpr int kSmallWords = 8;            // of 32 samples at most
constexpr int kSmallBlocks = 128;

// A class's similarities to shared memory, as they are or rounded to fixed point (as fixed_point_kernel does).
__device__ __forceinline__ void load_similarities(int4 *to, const int4 *from, int n, bool toFix, int exponent)
{
    if (!toFix) {
#pragma unroll 4
        for (int i = threadIdx.x; i < n; i += blockDim.x) copy16(to + i, from + i);
        copies_commit();
        copies_wait<0>();
        return;
    }
    const float scale = ldexpf(1.f, exponent);
    constexpr int U = 8;
    for (int i0 = threadIdx.x; i0 < n; i0 += U * blockDim.x) {
        int4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = i0 + u * (int)blockDim.x < n ? ld_row_once(from + i0 + u * blockDim.x) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * (int)blockDim.x < n)
                to[i0 + u * blockDim.x] = make_int4(to_fixed(__int_as_float(x[u].x), scale), to_fixed(__int_as_float(x[u].y), scale),
                                                    to_fixed(__int_as_float(x[u].z), scale), to_fixed(__int_as_float(x[u].w), scale));
    }
}

// NW: warps with samples, a thread per sample; one more leads.  KW: blocks per lane of the leader.
template <int NW, int KW, bool kCut>
__global__ void __launch_bounds__((NW + 1) * 32) greedy_small_kernel(const __grid_constant__ SmallParams prm)
{
    extern __shared__ __align__(128) unsigned char shared[];
    __shared__ unsigned long long shBest[8];               // the warps' best candidates for the block that is next
    __shared__ int shCount[2];                             // columns that rose, for two picks in turn
    __shared__ int shFirst;                                // the first block
    __shared__ uint32_t shNext;                            // the leader's word: block that is next | 1 << 8: it is empty | 1 << 9: the last one is full
    const int l = prm.classOrder[blockIdx.x], W = prm.W;
    const ClassDesc c = prm.desc[l];
    const int M = c.M, v = threadIdx.x, lane = v & 31, warp = v >> 5;
    if (M == 0) {
        for (int p = v; p < W; p += (NW + 1) * 32) prm.fval[(int64_t)l * W + p] = 0;
        return;
    }
    const int exponent = prm.fixedExp ? prm.fixedExp[l] : 0;
    if (prm.fixedExp && exponent == kNotFixed) return;
    const int ld = c.ld, vs = min(v, ld - 1);              // (threads beyond the class work on its last column)
    int32_t *const S = reinterpret_cast<int32_t *>(shared);
    const int32_t *const col = S + vs;
    int32_t *const cover = reinterpret_cast<int32_t *>(shared + prm.offCover) + vs;                      // of block j: [j * prm.ld]
    unsigned long long *const gains = reinterpret_cast<unsigned long long *>(shared + prm.offGains) + vs;
    int4 *const list = reinterpret_cast<int4 *>(shared + prm.offList);                                   // columns that rose (and room for eight)
    uint32_t *const picks = reinterpret_cast<uint32_t *>(shared + prm.offPicks);

    load_similarities(reinterpret_cast<int4 *>(shared), reinterpret_cast<const int4 *>(prm.S + c.sOff), M * (ld >> 2), prm.toFix != 0, exponent);
    if (v < 8) shBest[v] = 0;
    if (v < 2) shCount[v] = 0;
    __syncthreads();

    // The gain for an empty block, the same for every block (S is symmetric: the row of a sample is its column).
    unsigned long long g0 = 0, bias = 0;
    if (warp < NW) {
        unsigned long long size = 0;
#pragma unroll 8
        for (int i = 0; i < M; ++i) {
            const int x = col[i * ld];
            g0 = add_wide(max(x, 0), prm.one, g0);
            if (kCut) size = add_wide(max(-x, 0), prm.one, size);
        }
        if (kCut) {
            const unsigned long long top = warp_max_u64(v < M ? g0 + size : 0ull);
            if (lane == 0) shBest[warp] = top;
            g0 = g0 - size - (long long)col[min(vs, M - 1) * ld];       // (no row beyond the class's: with one block less than that follows S)
        }
    }
    if (kCut) {
        // gains lie within three times the largest sum of |S| over a row, either way
        __syncthreads();
        bias = 3 * warp_max_u64(shBest[lane & 7]) + 1;
        g0 += bias;
        __syncthreads();
    }
    if (warp < NW) {
        bool taken = v >= M;
        unsigned long long g = g0;                         // of block j
        int j = 0, o = 0;                                  // (its coverage)
        for (int t = 0;; ++t) {
            // the warp's best unassigned candidate for block j
            const unsigned long long k = warp_max_u64(taken ? 0ull : make_key(g, v));
            if (lane == 0) shBest[warp] = k;
            __syncthreads();
            if (t == 0) j = shFirst;
            const int s = key_sample(warp_max_u64(shBest[lane & 7]));
            const int x = col[s * ld];
            taken = taken || v == s;
            if (!kCut) {
                // the sample's row against the block's coverage: what rises joins the list
                const bool up = x > o && v < M;
                const unsigned rose = __ballot_sync(0xffffffffu, up);
                if (rose) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&shCount[t & 1], __popc(rose));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(rose & ((1u << lane) - 1u));
                    if (up) list[at] = make_int4(v * ld, -o, x - o, 0);
                    o = max(x, o);
                }
            }
            __syncthreads();
            const uint32_t next = shNext;
            if (!(next >> 9 & 1)) {                        // (a full block needs no gains any more)
                if (kCut) {
                    // gain = column sum - twice the tie to the block: the sample's row is the tie's growth
                    g -= 2ll * x;
                } else {
                    const int n = *(volatile int *)&shCount[t & 1];
                    if (n == 1) {
                        const int4 e = list[0];
                        g -= (uint32_t)__viaddmin_s32_relu(col[e.x], e.y, e.z);
                    } else if (n > 0) {
                        // eight at a time, the next eight entries on their way (four losses, each below 2^30, add up in 32 bits)
                        int4 e[8];
                        int y[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) e[q] = list[q];
                        auto losses = [&](int q) {
                            return (uint32_t)__viaddmin_s32_relu(y[q], e[q].y, e[q].z) + (uint32_t)__viaddmin_s32_relu(y[q + 1], e[q + 1].y, e[q + 1].z) +
                                   (uint32_t)__viaddmin_s32_relu(y[q + 2], e[q + 2].y, e[q + 2].z) + (uint32_t)__viaddmin_s32_relu(y[q + 3], e[q + 3].y, e[q + 3].z);
                        };
                        int i = 0;
#pragma unroll 1
                        for (; i + 8 <= n; i += 8) {
#pragma unroll
                            for (int q = 0; q < 8; ++q) y[q] = col[e[q].x];
                            int4 next[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q) next[q] = list[i + 8 + q];
                            g -= losses(0);
                            g -= losses(4);
#pragma unroll
                            for (int q = 0; q < 8; ++q) e[q] = next[q];
                        }
                        if (i < n) {
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                y[q] = col[i + q < n ? e[q].x : 0];
                                e[q].z = i + q < n ? e[q].z : 0;
                            }
                            g -= losses(0);
                            if (i + 4 < n) g -= losses(4);
                        }
                    }
                }
                if (v < M) {
                    gains[j * prm.ld] = g;
                    if (!kCut) cover[j * prm.ld] = o;
                }
            }
            if (t + 1 == M) break;
            const int jn = (int)(next & 127);
            if (jn != j) {
                j = jn;
                if (next >> 8 & 1) {
                    g = g0;
                    o = 0;
                } else {
                    g = gains[j * prm.ld];
                    if (!kCut) o = cover[j * prm.ld];
                }
            }
        }
    } else {
        unsigned long long f[KW];                          // (value + kTrackedZero) << 7 | block
        int room[KW];
        uint32_t has[KW];                                  // blocks that are not empty
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            const int p = lane + 32 * k;
            f[k] = (kTrackedZero << 7) | (unsigned long long)p;
            room[k] = p < W ? prm.quota[(int64_t)l * W + p] : 0;
            has[k] = 0;
        }
        // the least value << 7 | block of those that have room, but for block `but` (~0: none)
        auto least_but = [&](int but) {
            unsigned long long m = ~0ull;
#pragma unroll
            for (int k = 0; k < KW; ++k) m = room[k] > 0 && lane + 32 * k != but ? umin(m, f[k]) : m;
            return ~warp_max_u64(~m);
        };
        unsigned long long least = least_but(-1);
        if (lane == 0) shFirst = (int)(least & 127);
        uint32_t rows = 0, corrected = 0;
        for (int t = 0; t < M; ++t) {
            // what does not depend on the pick
            const int j = (int)(least & 127);
            const unsigned long long others = least_but(j);
            int left = room[0];
#pragma unroll
            for (int k = 1; k < KW; ++k) left ^= (left ^ room[k]) & (j >> 5 == k ? ~0 : 0);
            const bool full = __shfl_sync(0xffffffffu, left, j & 31) == 1;
#pragma unroll
            for (int k = 0; k < KW; ++k) has[k] |= KW == 1 || j >> 5 == k ? 1u << (j & 31) : 0u;
            const int other = (int)(others & 127);
            uint32_t h = has[0];
#pragma unroll
            for (int k = 1; k < KW; ++k) h ^= (h ^ has[k]) & (other >> 5 == k ? ~0u : 0u);
            const uint32_t otherWord = (uint32_t)other | (h >> (other & 31) & 1 ? 0u : 1u << 8) | (full ? 1u << 9 : 0u);
            __syncthreads();
            const unsigned long long best = warp_max_u64(shBest[lane & 7]);
            const unsigned long long inc = ((best >> 16) - bias) << 7, now = full ? ~0ull : least + inc;
            least = umin(others, now);
            if (lane == 0) {
                shCount[(t + 1) & 1] = 0;
                shNext = others < now ? otherWord : (uint32_t)j | (full ? 1u << 9 : 0u);
                picks[t] = (uint32_t)key_sample(best) | (uint32_t)j << 16;
            }
            __syncthreads();
            if (least == ~0ull && t + 1 < M) {             // (cannot be: the quotas add up to M)
                if (lane == 0) atomicOr(prm.status, kDevNoCandidate);
                least = (unsigned long long)j;
            }
#pragma unroll
            for (int k = 0; k < KW; ++k) {
                f[k] += lane + 32 * k == j ? inc : 0ull;
                room[k] -= lane + 32 * k == j ? 1 : 0;
            }
            corrected += full ? 0 : 1;
            if (!kCut) rows += full ? 0 : *(volatile int *)&shCount[t & 1];
        }
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            const int p = lane + 32 * k;
            const long long value = (long long)(f[k] >> 7) - (long long)kTrackedZero;
            if (p < W) prm.fval[(int64_t)l * W + p] = prm.fixedExp ? __double_as_longlong(ldexp((double)value, -exponent)) : value;
        }
        if (lane == 0) {
            atomicAdd(prm.stats + 15, (unsigned long long)corrected);
            atomicAdd(prm.stats + 16, (unsigned long long)rows);
        }
    }
    // class-local picks -> outputs (the last of them was written before the last barrier)
    for (int t = v; t < M; t += (NW + 1) * 32) {
        const uint32_t p = picks[t];
        const int global = prm.perm[c.row0 + (p & 0xffff)];
        prm.assignment[global] = (int)(p >> 16);
        if (prm.order) prm.order[c.row0 + t] = global;
    }
}

typedef void (*SmallKernel)(SmallParams);
template <int KW, bool kCut>
static SmallKernel pick_words(int words)
{
    switch (words) {
    case 1: return greedy_small_kernel<1, KW, kCut>;
    case 2: return greedy_small_kernel<2, KW, kCut>;
    case 3: return greedy_small_kernel<3, KW, kCut>;
    case 4: return greedy_small_kernel<4, KW, kCut>;
    case 5: return greedy_small_kernel<5, KW, kCut>;
    case 6: return greedy_small_kernel<6, KW, kCut>;
    case 7: return greedy_small_kernel<7, KW, kCut>;
    default: return greedy_small_kernel<8, KW, kCut>;
    }
}
template <bool kCut>
static SmallKernel pick_small(int words, int W)
{
    return W <= 32 ? pick_words<1, kCut>(words) : W <= 64 ? pick_words<2, kCut>(words) : pick_words<4, kCut>(words);
}

}  // namespace

struct SmallPlan {
    int words;
    size_t smem;
    SmallParams prm;           // ld and the offsets are set
};

std::shared_ptr<SmallPlan> plan_greedy_small(rcd_ctx *ctx, const Sizes &sz)
{
    if (sz.W > kSmallBlocks || sz.maxM > kSmallWords * 32 || sz.maxM == 0 || (sz.graphCut && sz.floatArith)) return nullptr;
    SmallPlan plan{};
    SmallParams &prm = plan.prm;
    prm.ld = pad_row(sz.maxM);
    plan.words = (int)(sz.maxM + 31) / 32;
    size_t off = (size_t)sz.maxM * prm.ld * 4;
    auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 15) / 16 * 16; return (int32_t)at; };
    prm.offCover = take(sz.graphCut ? 0 : (size_t)sz.W * prm.ld * 4);
    prm.offGains = take((size_t)sz.W * prm.ld * 8);
    prm.offList = take(sz.graphCut ? 0 : ((size_t)plan.words * 32 + 8) * 16);
    prm.offPicks = take((size_t)sz.maxM * 4);
    plan.smem = off;
    if (off > (size_t)whole_shared(ctx)) return nullptr;
    return std::make_shared<SmallPlan>(plan);
}

rcd_status launch_greedy_small(rcd_ctx *ctx, SmallPlan &plan, const Sizes &sz, const Workspace &ws, bool toFix, int32_t *assignment, int32_t *order,
                               void *partValues, cudaStream_t st)
{
    SmallParams &prm = plan.prm;
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.perm = ws.perm;
    prm.quota = ws.quota;
    prm.fval = (long long *)(partValues ? partValues : ws.fval);
    prm.assignment = assignment;
    prm.order = order;
    prm.fixedExp = sz.floatArith ? ws.fixedExp : nullptr;
    prm.classOrder = ws.classOrder;
    prm.status = ctx->statusOwn;
    prm.stats = ws.phaseNs;
    prm.W = sz.W;
    prm.toFix = toFix ? 1 : 0;
    prm.one = 1u;
    const SmallKernel kernel = sz.graphCut ? pick_small<true>(plan.words, sz.W) : pick_small<false>(plan.words, sz.W);
    RCD_CUDA(ctx, allow_shared(kernel, whole_shared(ctx)));
    kernel<<<sz.L, (plan.words + 1) * 32, plan.smem, st>>>(prm);
    RCD_CUDA(ctx, cudaGetLastError());
    ctx->kernelLaunches++;
    return RCD_OK;
}

}  // namespace rcd
