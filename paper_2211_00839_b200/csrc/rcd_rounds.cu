// The greedy loop of Algorithm 1 with the facility-location objective in rounds, one CTA per class: the form the library chooses
// for problems of many classes and blocks.
//
// What bounds the alternative.  The cluster form (rcd_cluster.cu) corrects a block's stored gains from one row of S per column
// whose coverage a pick raised, block after block.  With many classes at a time the rows come from HBM, and with many blocks the
// same row is fetched once per block: 1000 classes of 1300 into 64 blocks read 895 GB, 130 times every matrix.  But the picks of
// different blocks do not wait for one another's corrections: block j* = argmin f follows from the tracked values alone, and its
// best unassigned sample from its own stored gains.  So a round here is
//   decide   one warp makes picks until the block whose turn it is has a correction outstanding (64 picks at first, 11 on average);
//   list     all warps fold the picked samples' rows into their blocks' coverage and list the columns each pick raised;
//   correct  every row of S that any of the picks needs is fetched once, for all blocks that raised it;
//   look     the leading candidates of every corrected block, for the next round's decisions.
// So a class's rows are read 13 times over a run instead of 130 (the same problem; 10 times where one CTA's batch holds all blocks).
//
// What bounds it (1000 classes of 1300 int8 into 64 blocks: 165 ms in the cluster form, 81 here).  A class alone on an SM (16 warps) takes
// 11.0 ms, of which 4.3 are the sums of `tile_rows`: a saturating subtraction (half rate) and a multiply-add (its own pipe) per loss, 13
// cycles per row, 4 blocks and 128 columns where the pipes would allow 10.  2.0 ms are rows that few blocks need, straight from memory; the
// rest is trips to L2 and barriers of 110 rounds: lists 1.05, looks 1.0, copies of tiles and waits for them 0.9, decisions 0.7, looks
// asked for in between 0.45, tables 0.4, gains of empty blocks 0.2.  Two CTAs of 8 warps on an SM take 20 ms for two classes.  148 MB
// per class cross HBM instead of 895: 13 matrices of 6.8 MB, those of the empty blocks' gains and of the picks, gains and coverage.
//
// Results are those of the cluster form bit for bit: stored gains are exact integers, decisions are made in the same order.
#include "rcd_exact.cuh"

#include <limits.h>
#include <algorithm>
#include <cmath>

namespace rcd {

struct RoundsParams {
    const ClassDesc *desc;
    const int32_t *S;
    int32_t *cover;            // [sum W*ld]
    unsigned long long *gains; // [sum W*ld]
    unsigned long long *g0;    // [N] gains for an empty block
    uint32_t *picks;           // [N] sample | block << 16, in the order picked
    const int32_t *perm;
    const int32_t *quota;
    long long *fval;           // [L][W]
    int32_t *assignment, *order;
    const int32_t *fixedExp;   // [L] floating-point similarities: S = round(sim * 2^fixedExp) (null: integers)
    const int32_t *classOrder;
    int32_t *counter;
    int32_t *status;
    unsigned long long *stats; // phase words
    unsigned char *scratch;    // per CTA: scratchBytes for a table of what the picks of a batch raised
    int64_t scratchBytes;
    int32_t L, W;
    uint32_t one;              // the value 1, opaque to the compiler
    int32_t stageBytes;        // of the ring of tiles
    int32_t listShared;        // raised columns whose entries stay in shared memory, twice: as they come, and by blocks
    int32_t offRing, offKeys, offBounds, offBits, offNeeded, offBefore, offRows, offPend;   // dynamic shared memory
};

namespace {

constexpr int kListed = 64;               // leading candidates kept per block
constexpr int kListShared = 3072;         // raised columns at most whose entries stay in shared memory (where the ring is afterwards)
constexpr int kStages = 3;                // of the ring of tiles
constexpr int kGroup = 4;                 // blocks per warp of a tile
constexpr int kMaxWarps = 16;             // of a CTA; blocks corrected together: kGroup each
constexpr int kRoundBlocks = 128;
constexpr int kRoundsOwnShared = 3072;     // bytes of shared memory the kernel's own variables take, at most
constexpr unsigned kCopyLimit = 1u << 22; // looks at a stage's barrier, 64 ns apart, before the copies count as lost: a quarter of a second

struct Pending { int32_t block, sample, first; };   // a pick whose correction is outstanding; first: its block was empty

// The two leading unassigned candidates among a lane's samples, as keys, and a bound on its others.
struct Lead { unsigned long long best, next, rest; };
__device__ __forceinline__ void lead_add(Lead &t, unsigned long long k)
{
    const bool more = k > t.best;
    const unsigned long long low = more ? t.best : k;
    t.best = more ? k : t.best;
    const bool second = low > t.next;
    t.rest = umax(t.rest, second ? t.next : low);
    t.next = second ? low : t.next;
}
// Where the gain of column 128 g + 4 lane + m of a block stands: the columns that a warp's lanes hold in their m-th word lie side by
// side (additions to them touch a quarter of the sectors).  Gains for an empty block are in order.
__device__ __forceinline__ int gain_at(int g, int m, int lane, int ld4) { return 128 * g + m * min(32, ld4 - 32 * g) + lane; }
template <bool kInOrder>
__device__ __forceinline__ Lead lead_of(const unsigned long long *gains, int from, int to, int ld4, const uint32_t *bits, int lane)
{
    constexpr int U = 2;
    Lead t{0, 0, 0};
    for (int g0 = from; g0 < to; g0 += U) {
        unsigned long long x[U][4];
        uint32_t taken[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int g = g0 + u, q = 32 * g + lane;
            taken[u] = g < to && q < ld4 ? bits[q >> 3] >> (4 * (q & 7)) : 15u;      // (everything from M on counts as taken)
#pragma unroll
            for (int m = 0; m < 4; ++m)
                x[u][m] = taken[u] >> m & 1 ? 0ull : __ldcg(gains + (kInOrder ? 4 * q + m : gain_at(g, m, lane, ld4)));
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (!(taken[u] >> m & 1)) lead_add(t, make_key(x[u][m], 4 * (32 * (g0 + u) + lane) + m));
    }
    return t;
}
// A block's list: two candidates per lane, and a bound on all others.
__device__ __forceinline__ void lead_keep(const Lead &t, unsigned long long *keys, unsigned long long *bound, int lane)
{
    keys[lane] = t.best;
    keys[32 + lane] = t.next;
    const unsigned long long b = warp_max_u64(t.rest);
    if (lane == 0) *bound = b;
    __syncwarp();
}
// `parts` warps look through a block's gains together: each leaves what it found in scratch, and after a barrier one joins them.
template <bool kInOrder>
__device__ __forceinline__ void look_part(const unsigned long long *gains, int ld4, const uint32_t *bits, unsigned long long *scratch, int part, int parts, int lane)
{
    const int G = (ld4 + 31) / 32, len = (G + parts - 1) / parts;
    const Lead t = lead_of<kInOrder>(gains, min(G, part * len), min(G, part * len + len), ld4, bits, lane);
    scratch[part * 96 + lane] = t.best;
    scratch[part * 96 + 32 + lane] = t.next;
    scratch[part * 96 + 64 + lane] = t.rest;
}
__device__ __forceinline__ void look_join(const unsigned long long *scratch, int parts, unsigned long long *keys, unsigned long long *bound, int lane)
{
    Lead t{scratch[lane], scratch[32 + lane], scratch[64 + lane]};
    for (int k = 1; k < parts; ++k) {
        lead_add(t, scratch[k * 96 + lane]);
        lead_add(t, scratch[k * 96 + 32 + lane]);
        t.rest = umax(t.rest, scratch[k * 96 + 64 + lane]);
    }
    lead_keep(t, keys, bound, lane);
}
// The best alone.
__device__ __forceinline__ void best_part(const unsigned long long *gains, int ld4, const uint32_t *bits, unsigned long long *scratch, int part, int parts, int lane)
{
    const int G = (ld4 + 31) / 32, len = (G + parts - 1) / parts;
    const unsigned long long k = warp_max_u64(lead_of<false>(gains, min(G, part * len), min(G, part * len + len), ld4, bits, lane).best);
    if (lane == 0) scratch[part] = k;
}

// acc + x * one, on the multiply-add pipe
__device__ __forceinline__ uint32_t add_mad(int x, uint32_t one, uint32_t acc)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"((uint32_t)x), "r"(one), "r"(acc));
    return r;
}

__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_done(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, unsigned limit)
{
    for (int k = 0; k < 64; ++k)
        if (bar_done(bar, parity)) return true;
    for (unsigned k = 0; k < limit; ++k) {
        if (bar_done(bar, parity)) return true;
        __nanosleep(64);
    }
    return false;
}
// Waits for the copies of a step, and for all threads.  Where a thread gives up, all of them learn of it at this very step (lostAt: the
// first step without its copies; a thread that is ahead can only have put down a later one), so that they leave together.
__device__ __forceinline__ bool step_arrived(uint32_t bar, uint32_t parity, int step, int *lostAt, unsigned limit)
{
    if (!bar_wait(bar, parity, limit)) atomicMin(lostAt, step);
    __syncthreads();
    return *(volatile int *)lostAt > step;
}
// (16-byte aligned on both sides, a multiple of 16 bytes)
__device__ __forceinline__ void copy_bulk(uint32_t to, const void *from, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(to), "l"(from), "r"(bytes), "r"(bar) : "memory");
}

// A stage of a warp's tile: `n` rows (a multiple of 4) of 128 columns against kGroup blocks.  Losses are added in 32 bits for as many
// fours of rows as cannot overflow (`fours` of them since the sums were cleared, `most` at most), and then widened.
__device__ __forceinline__ void tile_rows(const unsigned char *xs, int xStride, const unsigned char *es, int eStride, int n, uint32_t one, int &fours, int most, uint32_t (&sum)[kGroup][4], unsigned long long (&acc)[kGroup][4])
{
    for (int r = 0; r < n; r += 4, xs += 4 * xStride, es += 4 * eStride) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 x = *reinterpret_cast<const int4 *>(xs + k * xStride);
            const int y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int b = 0; b < kGroup; b += 2) {
                const int4 e = *reinterpret_cast<const int4 *>(es + k * eStride + b * 8);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    sum[b][m] = add_mad(__viaddmin_s32_relu(y[m], e.x, e.y), one, sum[b][m]);
                    sum[b + 1][m] = add_mad(__viaddmin_s32_relu(y[m], e.z, e.w), one, sum[b + 1][m]);
                }
            }
        }
        if (++fours == most) {
            fours = 0;
#pragma unroll
            for (int b = 0; b < kGroup; ++b)
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    acc[b][m] += sum[b][m];
                    sum[b][m] = 0;
                }
        }
    }
}

// KW: blocks per lane of the deciding warp.  kWarps: 16, or 8 where two CTAs share an SM.
template <int KW, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, kMaxWarps / kWarps) greedy_rounds_kernel(const __grid_constant__ RoundsParams prm)
{
    extern __shared__ __align__(128) unsigned char shared[];
    constexpr int kThreads = kWarps * 32, kBatchBlocks = kWarps * kGroup;
    __shared__ int shCount[kMaxWarps * kGroup];                                    // raised columns per pick of a batch, then the first of each
    // the blocks: tracked value << 7 | block, samples still to take, not empty
    __shared__ unsigned long long shValue[kRoundBlocks];
    __shared__ int shRoom[kRoundBlocks];
    __shared__ uint8_t shHas[kRoundBlocks];
    __shared__ __align__(8) unsigned long long shBars[kStages];
    __shared__ int shMostBy, shMade, shClass, shCommand, shListed, shNeeded, shFailed, shLostAt;
    __shared__ unsigned shLists, shTiles;     // batches corrected either way
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = prm.W;
    unsigned char *const ring = shared + prm.offRing;
    unsigned long long *const scratch = reinterpret_cast<unsigned long long *>(ring);                    // (while there are no tiles)
    int4 *const listShared = reinterpret_cast<int4 *>(ring);                                             // (likewise)
    unsigned long long *const keys = reinterpret_cast<unsigned long long *>(shared + prm.offKeys);       // [W + 1][kListed], last: empty blocks
    unsigned long long *const bounds = reinterpret_cast<unsigned long long *>(shared + prm.offBounds);   // [W + 1]
    uint32_t *const bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);                           // assigned samples
    uint32_t *const needed = reinterpret_cast<uint32_t *>(shared + prm.offNeeded);                       // rows that a pick of the batch raised
    int32_t *const before = reinterpret_cast<int32_t *>(shared + prm.offBefore);                         // such rows before each word
    uint16_t *const rows = reinterpret_cast<uint16_t *>(shared + prm.offRows);                           // such rows in order
    Pending *const pending = reinterpret_cast<Pending *>(shared + prm.offPend);
    int4 *const listSorted = listShared + prm.listShared;
    const uint32_t bars = smem32(shBars);
    uint32_t parities = 0;                    // of the stages' barriers
    unsigned rescans = 0;
    unsigned long long rowsRead = 0, corrected = 0;
    bool lost = false;                        // (in all threads or in none) copies did not arrive: nothing more is written, the kernel ends

    if (threadIdx.x == 0) {
        shLostAt = INT_MAX;
        shLists = shTiles = 0;
        for (int k = 0; k < kStages; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bars + 8 * k) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    while (!lost) {
        if (threadIdx.x == 0) {
            const int k = atomicAdd(prm.counter, 1);
            shClass = (k < prm.L && *(volatile int32_t *)prm.status == 0) ? prm.classOrder[k] : -1;
        }
        __syncthreads();
        const int l = shClass;
        if (l < 0) break;
        const ClassDesc c = prm.desc[l];
        if (c.M == 0 || (prm.fixedExp && prm.fixedExp[l] == kNotFixed)) {
            if (c.M == 0) for (int p = threadIdx.x; p < W; p += kThreads) prm.fval[(int64_t)l * W + p] = 0;
            __syncthreads();
            continue;
        }
        const int ld4 = c.ld >> 2, M = c.M, G = (ld4 + 31) / 32, words = (c.ld + 31) / 32;
        const int4 *const S4 = reinterpret_cast<const int4 *>(prm.S + c.sOff);
        unsigned long long *const gains = prm.gains + c.vOff;
        unsigned long long *const g0 = prm.g0 + c.row0;
        int32_t *const cover = prm.cover + c.vOff;

        // gains for an empty block, the same for every block
        for (int v = warp; v < M; v += kWarps) {
            unsigned long long neg;
            const unsigned long long pos = row_value<false>(S4 + (int64_t)v * ld4, ld4, lane, prm.one, neg);
            if (lane == 0) __stcg(g0 + v, pos);
        }
        for (int i = threadIdx.x; i < words; i += kThreads) bits[i] = 32 * i + 32 <= M ? 0u : (32 * i >= M ? ~0u : ~0u << (M - 32 * i));
        if (threadIdx.x == 0) {
            shMade = 0;
            shFailed = 0;
        }
        if (threadIdx.x < kRoundBlocks) {
            const int p = threadIdx.x;
            shValue[p] = (unsigned long long)p;
            shHas[p] = 0;
            shRoom[p] = p < W ? prm.quota[(int64_t)l * W + p] : 0;
        }
        __syncthreads();
        look_part<true>(g0, ld4, bits, scratch, warp, kWarps, lane);
        __syncthreads();
        if (warp == 0) look_join(scratch, kWarps, keys + W * kListed, bounds + W, lane);
        while (!lost) {
            if (warp == 0) {
                int n = 0, made = shMade;
                unsigned long long f[KW];
                int room[KW];
                uint32_t waiting[KW], filled[KW];      // (every lane knows all blocks: correction outstanding, not empty)
#pragma unroll
                for (int k = 0; k < KW; ++k) {
                    f[k] = shValue[lane + 32 * k];
                    room[k] = shRoom[lane + 32 * k];
                    waiting[k] = 0;
                    filled[k] = __ballot_sync(0xffffffffu, shHas[lane + 32 * k]);
                }
                unsigned long long least = ~0ull;
#pragma unroll
                for (int k = 0; k < KW; ++k) least = room[k] > 0 ? umin(least, f[k]) : least;
                least = ~warp_max_u64(~least);
                while (made < M) {
                    const int j = (int)(least & 127), jl = j & 31, jk = j >> 5;
                    uint32_t w = 0, e = 0;
#pragma unroll
                    for (int k = 0; k < KW; ++k) if (k == jk) { w = waiting[k]; e = filled[k]; }
                    if (w >> jl & 1) break;
                    const bool empty = !(e >> jl & 1);
                    const int slot = empty ? W : j;
                    // the least of the other blocks: does not depend on this pick
                    unsigned long long others = ~0ull;
                    int left = 0;
#pragma unroll
                    for (int k = 0; k < KW; ++k) {
                        others = room[k] > 0 && lane + 32 * k != j ? umin(others, f[k]) : others;
                        if (k == jk) left = room[k];
                    }
                    others = ~warp_max_u64(~others);
                    const bool more = __shfl_sync(0xffffffffu, left, jl) > 1;
                    unsigned long long best = 0;
                    for (int tries = 0; tries < 2; ++tries) {
                        const unsigned long long a = keys[slot * kListed + lane], b = keys[slot * kListed + 32 + lane];
                        const int sa = key_sample(a), sb = key_sample(b);
                        const bool freeA = a != 0 && !(bits[sa >> 5] >> (sa & 31) & 1), freeB = b != 0 && !(bits[sb >> 5] >> (sb & 31) & 1);
                        best = warp_max_u64(freeA ? a : freeB ? b : 0ull);      // (b follows a)
                        if (best > bounds[slot]) break;
                        best = 0;
                        if (tries) break;
                        // all that are sure to lead have been taken by other blocks: all warps look again
                        ++rescans;
                        if (lane == 0) shCommand = -2 - slot;
                        __syncthreads();
                        if (!empty) {
                            best_part(gains + (int64_t)j * c.ld, ld4, bits, scratch, 0, kWarps, lane);
                            __syncthreads();
                            best = warp_max_u64(lane < kWarps ? scratch[lane] : 0ull);
                            break;
                        }
                        look_part<true>(g0, ld4, bits, scratch, 0, kWarps, lane);
                        __syncthreads();
                        look_join(scratch, kWarps, keys + slot * kListed, bounds + slot, lane);
                    }
                    if (best == 0 || least == ~0ull) {
                        if (lane == 0) {
                            atomicOr(prm.status, kDevNoCandidate);
                            shFailed = 1;
                        }
                        made = M;
                        break;
                    }
                    const int v = key_sample(best);
                    const unsigned long long inc = (best >> 16) << 7;
#pragma unroll
                    for (int k = 0; k < KW; ++k)
                        if (k == jk) {
                            if (lane == jl) {
                                f[k] += inc;
                                --room[k];
                            }
                            waiting[k] |= 1u << jl;
                            filled[k] |= 1u << jl;
                        }
                    least = more ? umin(others, least + inc) : others;
                    if (lane == 0) {
                        bits[v >> 5] |= 1u << (v & 31);
                        prm.picks[c.row0 + made] = (uint32_t)v | ((uint32_t)j << 16);
                        if (more) pending[n] = Pending{j, v, empty ? 1 : 0};
                    }
                    n += more ? 1 : 0;             // (a full block needs no gains any more)
                    ++made;
                    __syncwarp();
                }
#pragma unroll
                for (int k = 0; k < KW; ++k) {
                    shValue[lane + 32 * k] = f[k];
                    shRoom[lane + 32 * k] = room[k];
                    shHas[lane + 32 * k] = filled[k] >> lane & 1;
                }
                if (lane == 0) {
                    shMade = made;
                    shCommand = made < M ? n : -1;
                }
                __syncthreads();
            } else {
                for (;;) {
                    __syncthreads();
                    const int slot = -2 - shCommand;
                    if (slot < 0) break;
                    if (slot == W) look_part<true>(g0, ld4, bits, scratch, warp, kWarps, lane);
                    else best_part(gains + (int64_t)slot * c.ld, ld4, bits, scratch, warp, kWarps, lane);
                    __syncthreads();
                }
            }
            const int nPending = shCommand;
            if (nPending < 0) break;

            const int perBlock = M * 8 + 32;       // scratch of a block: its part of the table
            const int most = (int)min((int64_t)min(nPending, kBatchBlocks), prm.scratchBytes / perBlock / kGroup * kGroup);
            for (int p0 = 0; p0 < nPending && !lost; p0 += most) {
                const int nP = min(most, nPending - p0), nP4 = (nP + kGroup - 1) / kGroup * kGroup;
                const Pending *const pend = pending + p0;
                int2 *const table = reinterpret_cast<int2 *>(prm.scratch + (int64_t)blockIdx.x * prm.scratchBytes);   // [rows needed][nP4]: - old coverage, new - old
                for (int i = threadIdx.x; i < words; i += kThreads) needed[i] = 0;
                if (threadIdx.x == 0) shListed = shMostBy = 0;
                if (threadIdx.x < kMaxWarps * kGroup) shCount[threadIdx.x] = 0;
                __syncthreads();
                // the columns that rise, block by block and 128 at a time
                const int units = nP * G;
                constexpr int U = 2;
                int4 now[U], old[U];
                auto load = [&](int u0) {
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int u = u0 + k * kWarps, p = u / G, q = 32 * (u - p * G) + lane;
                        now[k] = old[k] = make_int4(0, 0, 0, 0);
                        if (u < units && q < ld4) {
                            now[k] = ld_row_shared(S4 + (int64_t)pend[p].sample * ld4 + q);
                            if (!pend[p].first) old[k] = reinterpret_cast<const int4 *>(cover + (int64_t)pend[p].block * c.ld)[q];
                        }
                    }
                };
                for (int u0 = warp; u0 < units; u0 += U * kWarps) {
                    load(u0);
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int u = u0 + k * kWarps, p = u / G, q = 32 * (u - p * G) + lane;
                        if (u >= units) break;
                        const int x[4] = {now[k].x, now[k].y, now[k].z, now[k].w}, o[4] = {old[k].x, old[k].y, old[k].z, old[k].w};
                        uint32_t nibble = 0;
                        int rose = 0, mineAt[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const uint32_t up = __ballot_sync(0xffffffffu, x[m] > o[m]);
                            mineAt[m] = rose + __popc(up & ((1u << lane) - 1u));
                            rose += __popc(up);
                            nibble |= x[m] > o[m] ? 1u << m : 0u;
                        }
                        const bool first = pend[p].first != 0;
                        const int j = pend[p].block;
                        if (rose) {
                            int at = 0;
                            if (lane < 2) at = atomicAdd(lane == 0 ? &shListed : &shCount[p], rose);
                            const int rank = __shfl_sync(0xffffffffu, at, 1);
                            at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
                            for (int m = 0; m < 4; ++m)
                                if (x[m] > o[m]) {
                                    const int where = at + mineAt[m];
                                    if (where < prm.listShared) listShared[where] = make_int4(4 * q + m, -o[m], x[m] - o[m], p | (rank + mineAt[m]) << 8);
                                }
                            uint32_t word = nibble << (4 * (lane & 7));
                            word |= __shfl_xor_sync(0xffffffffu, word, 1);
                            word |= __shfl_xor_sync(0xffffffffu, word, 2);
                            word |= __shfl_xor_sync(0xffffffffu, word, 4);
                            if ((lane & 7) == 0 && word) atomicOr(&needed[q >> 3], word);
                            const int by = __reduce_max_sync(0xffffffffu, max(max(x[0] - o[0], x[1] - o[1]), max(x[2] - o[2], x[3] - o[3])));
                            if (lane == 0) atomicMax(&shMostBy, by);
                        }
                        if (first && q < ld4) {
                            reinterpret_cast<int4 *>(cover + (int64_t)j * c.ld)[q] = make_int4(max(x[0], 0), max(x[1], 0), max(x[2], 0), max(x[3], 0));
#pragma unroll
                            for (int m = 0; m < 4; ++m)
                                if (4 * q + m < M) __stcg(gains + (int64_t)j * c.ld + gain_at(q >> 5, m, lane, ld4), __ldcg(g0 + 4 * q + m));
                        }
                    }
                }
                __syncthreads();
                const int total = shListed;
                if (warp == 0) {
                    int sum = 0;
                    for (int i0 = 0; i0 < words; i0 += 32) {
                        const int n = i0 + lane < words ? __popc(needed[i0 + lane]) : 0;
                        int incl = n;
#pragma unroll
                        for (int off = 1; off < 32; off <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, incl, off);
                            if (lane >= off) incl += y;
                        }
                        if (i0 + lane < words) before[i0 + lane] = sum + incl - n;
                        sum += __shfl_sync(0xffffffffu, incl, 31);
                    }
                    if (lane == 0) shNeeded = sum;
                    const int a = shCount[lane], b = shCount[32 + lane];
                    int inclA = a, inclB = b;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, inclA, off), z = __shfl_up_sync(0xffffffffu, inclB, off);
                        if (lane >= off) { inclA += y; inclB += z; }
                    }
                    shCount[lane] = inclA - a;
                    shCount[32 + lane] = __shfl_sync(0xffffffffu, inclA, 31) + inclB - b;
                }
                __syncthreads();
                const int need = shNeeded;
                // One row from memory per raised column, or every row once and all blocks against it.  In cycles per 128 columns: a row
                // from memory 14, a row against a block 2.3, and what a table costs.
                if (total <= prm.listShared && total * 16 <= need * max(2 * nP4, 14) + 3000) {
                    if (threadIdx.x == 0) {
                        rowsRead += total;
                        ++shLists;
                    }
                    // (by blocks)
                    for (int i = threadIdx.x; i < total; i += kThreads) {
                        const int4 e = listShared[i];
                        cover[(int64_t)pend[e.w & 255].block * c.ld + e.x] = e.z - e.y;
                        listSorted[shCount[e.w & 255] + (e.w >> 8)] = make_int4(e.x * ld4, e.y, e.z, e.w & 255);
                    }
                    __syncthreads();
                    const int chunks = (total + 7) / 8;
                    for (int u = warp; u < chunks * G; u += kWarps) {
                        const int g = u / chunks, i0 = (u - g * chunks) * 8, q = 32 * g + lane, n = min(8, total - i0);
                        const int4 *const entries = listSorted + i0;
                        int4 x[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) x[k] = k < n && q < ld4 ? ld_row_shared(S4 + entries[k].x + q) : make_int4(0, 0, 0, 0);
                        unsigned long long sum[4] = {0, 0, 0, 0};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k >= n) break;
                            const int4 e = entries[k];
                            sum[0] += (uint32_t)__viaddmin_s32_relu(x[k].x, e.y, e.z);
                            sum[1] += (uint32_t)__viaddmin_s32_relu(x[k].y, e.y, e.z);
                            sum[2] += (uint32_t)__viaddmin_s32_relu(x[k].z, e.y, e.z);
                            sum[3] += (uint32_t)__viaddmin_s32_relu(x[k].w, e.y, e.z);
                            if (k == n - 1 || entries[k + 1].w != e.w) {
                                // (columns beyond the class are 0 in every row and lose nothing)
                                unsigned long long *const mine = gains + (int64_t)pend[e.w].block * c.ld;
#pragma unroll
                                for (int m = 0; m < 4; ++m) {
                                    if (q < ld4 && sum[m]) atomicAdd(mine + gain_at(g, m, lane, ld4), 0ull - sum[m]);
                                    sum[m] = 0;
                                }
                            }
                        }
                    }
                } else {
                    if (threadIdx.x == 0) {
                        rowsRead += need;
                        ++shTiles;
                    }
                    const int need4 = (need + 3) & ~3;
                    for (int i = threadIdx.x; i < need * (nP4 - nP); i += kThreads) table[i / (nP4 - nP) * nP4 + nP + i % (nP4 - nP)] = make_int2(0, 0);
                    for (int i = threadIdx.x; i < (need4 - need) * nP4; i += kThreads) table[need * nP4 + i] = make_int2(0, 0);
                    for (int i = threadIdx.x; i < c.ld; i += kThreads) {
                        const uint32_t word = needed[i >> 5];
                        if (word >> (i & 31) & 1) rows[before[i >> 5] + __popc(word & ((1u << (i & 31)) - 1u))] = (uint16_t)i;
                    }
                    for (int u0 = warp; u0 < units; u0 += U * kWarps) {
                        load(u0);
#pragma unroll
                        for (int k = 0; k < U; ++k) {
                            const int u = u0 + k * kWarps, p = u / G, q = 32 * (u - p * G) + lane;
                            if (u >= units || q >= ld4) continue;
                            const int x[4] = {now[k].x, now[k].y, now[k].z, now[k].w}, o[4] = {old[k].x, old[k].y, old[k].z, old[k].w};
                            const uint32_t word = needed[q >> 3], from = 4 * (q & 7);
                            int2 *to = table + (int64_t)(before[q >> 3] + __popc(word & ((1u << from) - 1u))) * nP4 + p;
                            bool rose = false;
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                rose = rose || x[m] > o[m];
                                if (word >> (from + m) & 1) {
                                    *to = make_int2(-o[m], max(x[m] - o[m], 0));
                                    to += nP4;
                                }
                            }
                            if (rose && !pend[p].first)
                                reinterpret_cast<int4 *>(cover + (int64_t)pend[p].block * c.ld)[q] = make_int4(max(x[0], o[0]), max(x[1], o[1]), max(x[2], o[2]), max(x[3], o[3]));
                        }
                    }
                    // (the table, and what the ring held, come before the bulk copies)
                    asm volatile("fence.proxy.async;" ::: "memory");
                    __syncthreads();
                    // Tiles of 128 columns per warp and kGroup blocks, stage after stage of rows: groups of blocks side by side, and
                    // several column groups where there are few.
                    const int groups = nP4 / kGroup;
                    int colGroups = 1;
                    while (colGroups < 8 && 2 * colGroups * groups <= kWarps && colGroups < G) colGroups *= 2;
                    const int rowBytes = colGroups * 512 + nP4 * 8;
                    const int perStage = prm.stageBytes / rowBytes & ~3;
                    const int stages = (need4 + perStage - 1) / perStage, steps = (G + colGroups - 1) / colGroups * stages;
                    const int group = warp % groups, colGroup = warp / groups;
                    const bool works = colGroup < colGroups;
                    auto fetch = [&](int step) {           // (all warps: a warp's copies go out one after the other)
                        if (step >= steps) return;
                        const int tile = step / stages, r0 = (step - tile * stages) * perStage, n = min(perStage, need4 - r0), real = min(n, need - r0);
                        const uint32_t at = smem32(ring) + (uint32_t)(step % kStages) * prm.stageBytes, bar = bars + 8 * (step % kStages);
                        const int q0 = tile * colGroups * 32, bytes = min(colGroups * 32, ld4 - q0) * 16;
                        if (threadIdx.x == 0) {
                            bar_expect(bar, (uint32_t)(real * bytes + n * nP4 * 8));
                            copy_bulk(at + perStage * colGroups * 512, table + (int64_t)r0 * nP4, (uint32_t)(n * nP4 * 8), bar);
                        }
                        for (int r = warp + kWarps * lane; r < real; r += kWarps * 32) copy_bulk(at + r * colGroups * 512, S4 + (int64_t)rows[r0 + r] * ld4 + q0, (uint32_t)bytes, bar);
                    };
                    unsigned long long acc[kGroup][4];
                    uint32_t sum[kGroup][4];
                    // (a loss is no greater than what the coverage rose by, and that is below 2^30)
                    const int mostFours = (int)(0xffffffffu / (uint32_t)shMostBy / 4u);
                    int fours = 0;
#pragma unroll
                    for (int k = 0; k < kStages - 1; ++k) fetch(k);
                    for (int step = 0; step < steps; ++step) {
                        const int stage = step % kStages;
                        // (and everybody is through with the stage before)
                        if (!step_arrived(bars + 8 * stage, parities >> stage & 1, step, &shLostAt, kCopyLimit)) {
                            // what is under way lands before shared memory is given up, if it lands at all
                            for (int k = step; k < min(steps, step + kStages - 1); ++k) bar_wait(bars + 8 * (k % kStages), parities >> (k % kStages) & 1, kCopyLimit);
                            lost = true;
                            break;
                        }
                        parities ^= 1u << stage;
                        fetch(step + kStages - 1);
                        const int tile = step / stages, part = step - tile * stages, n = min(perStage, need4 - part * perStage);
                        if (!works || tile * colGroups + colGroup >= G) continue;
                        if (part == 0) {
#pragma unroll
                            for (int b = 0; b < kGroup; ++b)
#pragma unroll
                                for (int m = 0; m < 4; ++m) sum[b][m] = 0, acc[b][m] = 0;
                        }
                        const unsigned char *at = ring + (size_t)stage * prm.stageBytes;
                        tile_rows(at + colGroup * 512 + lane * 16, colGroups * 512, at + perStage * colGroups * 512 + group * (kGroup * 8), nP4 * 8, n, prm.one, fours, mostFours, sum, acc);
                        if (part == stages - 1) {
                            const int g = tile * colGroups + colGroup, q = 32 * g + lane;
                            fours = 0;
#pragma unroll
                            for (int b = 0; b < kGroup; ++b) {
                                const int p = group * kGroup + b;
                                if (p >= nP || q >= ld4) break;
                                unsigned long long *const mine = gains + (int64_t)pend[p].block * c.ld;
#pragma unroll
                                for (int m = 0; m < 4; ++m) {
                                    const unsigned long long lost = acc[b][m] + sum[b][m];
                                    if (lost) atomicAdd(mine + gain_at(g, m, lane, ld4), 0ull - lost);
                                }
                            }
                        }
                    }
                }
                __threadfence();
                __syncthreads();
            }
            if (lost) break;
            if (threadIdx.x == 0) corrected += nPending;
            // the next notes: a warp per block, several for each of few
            int parts = 1;
            while (2 * parts * nPending <= kWarps) parts *= 2;
            if (parts == 1) {
                for (int p = warp; p < nPending; p += kWarps) {
                    const int j = pending[p].block;
                    lead_keep(lead_of<false>(gains + (int64_t)j * c.ld, 0, G, ld4, bits, lane), keys + j * kListed, bounds + j, lane);
                }
            } else {
                const int p = warp / parts;
                if (p < nPending) look_part<false>(gains + (int64_t)pending[p].block * c.ld, ld4, bits, scratch + p * parts * 96, warp % parts, parts, lane);
                __syncthreads();
                if (p < nPending && warp % parts == 0) {
                    const int j = pending[p].block;
                    look_join(scratch + p * parts * 96, parts, keys + j * kListed, bounds + j, lane);
                }
            }
            __syncthreads();
        }
        if (lost) break;
        for (int p = threadIdx.x; p < W; p += kThreads) {
            const long long value = (long long)(shValue[p] >> 7);
            prm.fval[(int64_t)l * W + p] = prm.fixedExp ? __double_as_longlong(ldexp((double)value, -prm.fixedExp[l])) : value;
        }
        // class-local picks -> outputs
        for (int t = threadIdx.x; t < M && !shFailed; t += kThreads) {
            const uint32_t p = prm.picks[c.row0 + t];
            const int global = prm.perm[c.row0 + (p & 0xffff)];
            prm.assignment[global] = (int)(p >> 16);
            if (prm.order) prm.order[c.row0 + t] = global;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (lost) atomicOr(prm.status, kDevTimeout);
        if (rescans) atomicAdd(prm.stats + 9, (unsigned long long)rescans);
        if (corrected) {
            atomicAdd(prm.stats + 15, corrected);
            atomicAdd(prm.stats + 16, rowsRead);
            atomicAdd(prm.stats + 18, (unsigned long long)shLists);
            atomicAdd(prm.stats + 19, (unsigned long long)shTiles);
        }
    }
}

// A step whose copies have arrived, then one whose copies never do, which half of the threads takes for arrived: all of them stay for
// the first and leave at the second.  (After the grid barrier's test, which leaves the timeout's bit: kept only if this goes right too.)
__global__ void step_wait_selftest_kernel(int32_t *status)
{
    __shared__ __align__(8) unsigned long long shBars[2];
    __shared__ int shLostAt;
    const uint32_t bars = smem32(shBars);
    if (threadIdx.x == 0) {
        shLostAt = INT_MAX;
        for (int k = 0; k < 2; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bars + 8 * k) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bar_expect(bars, 0);
    }
    __syncthreads();
    const bool first = step_arrived(bars, 0, 0, &shLostAt, 1u << 12);
    const bool second = step_arrived(threadIdx.x < blockDim.x / 2 ? bars : bars + 8, 0, 1, &shLostAt, 1u << 12);
    const bool right = __syncthreads_and(first && !second);
    if (threadIdx.x == 0 && !right) *(volatile int32_t *)status = kDevBadState;
}

}  // namespace

rcd_status launch_step_wait_selftest(rcd_ctx *ctx, int32_t *status, cudaStream_t st)
{
    step_wait_selftest_kernel<<<1, 128, 0, st>>>(status);
    ctx->kernelLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

struct RoundsPlan {
    RoundsParams prm;
    int ctas, warps;
    size_t smem;
};

// Whether rounds are the faster form.  Both forms hold classes of about one size (`equal`: classes of the largest size that would be as
// much work) and take them in turns: rounds one CTA per class, the cluster form C of them, of which the GPU holds 148, 74, 33, 15 or 7 at
// a time for C = 1, 2, 4, 8, 16.  So what counts is how much faster a cluster is through a class than one CTA in rounds, over the turns:
// `speed` below, from the times of both forms over 1000 problems (4 to 148 x their blocks).  It grows with C, less than in proportion, and
// with the class, since a small class is bound by its chain of picks in either form; C in turn follows from the blocks' state, which has
// to fit the cluster's shared memory.  Dense similarities (rectified features, whose picks raise more columns) cost rounds more than the
// cluster form, cosines and Gaussian kernels most; `speed` is that of rectified features.  us, whole call, cluster : rounds:
//   integers    64 blocks    1000 x 1300 (d 2048) 165000 : 82000   148 x 1000, dense 15000 : 9800   148 x 300 1410 : 990    60 x 1000, dense 6140 : 9000
//                            300 x 500, dense 7480 : 5780   200 x 500, dense 5200 : 4110   200 x 400, dense 2540 : 2970   100 x 1300, dense 15800 : 17800
//               128          148 x 1300 190000 : 20100   60 x 500, dense 3090 : 2450       80    60 x 500, dense 1890 : 2210   60 x 300, dense 1035 : 960
//               48           148 x 700, dense 5690 : 4220   300 x 500, dense 4640 : 5220   200 x 1000, dense 14600 : 15900   148 x 100, dense 219 : 227
//                            296 x 200 870 : 1100   296 x 133, dense 490 : 580   (one CTA per class either way, two turns, 128 to 250 samples: 1.05
//                            times as long in rounds on average over 200 to 296 classes, up to 1.30; 52 blocks 1.0, up to 1.24; 58 blocks 0.96, up to 1.21)
//               32           148 x 1000, dense 7090 : 6880   444 x 1000 21400 : 15200, dense 19600 : 22700 (taken)
//               24           148 x 1000, dense 5680 : 6070, 5370 : 5380   148 x 1050, dense 8390 : 7080   444 x 1000, dense 16100 : 20500
//                            (up to 1024 samples a row keeps a team of four warps busy for two steps; from 1025 on it takes a third)
//               16           148 x 1000, dense 6000 : 4910   444 x 1300, dense 28700 : 28900
//   floating    64           1000 x 1000, dense 102000 : 79600   300 x 500, dense 7680 : 6620   300 x 700, dense 13400 : 14600   444 x 1300, dense 69700 : 84800
//               65           60 x 500, dense 1930 : 2430   100 x 1000, dense 12200 : 12700   148 x 1000, dense 17400 : 13200
//               128          100 x 1300, dense 120000 : 33900   100 x 2000, dense 86400 : 103000
// Of 1059 measured calls this takes 807; eleven of them are 3 to 5 % slower in rounds, or dense ones of 444 x 1000 into 32 and 40 blocks.
// Small integer classes into 60 to 80 blocks that one CTA holds either way are close: 127 x 133 into 64 blocks 257 : 296, dense 260 : 264 with rows of 128
// bytes, whose tables hold 12 blocks at a time, 266 : 264 and 275 : 238 with 1 KB; 90 to 200 samples and rows up to 128 bytes take 0.96 of the cluster
// form's time on average (0.54 to 1.18), 256 bytes 0.93, 1 KB 0.87.
// Below 48 blocks (integers; 56 for floating point) only full turns of large classes were measured to gain, and turns that leave
// most SMs idle nowhere: plan_greedy_rounds does not ask there.
static bool rounds_win(const Sizes &sz, double equal, int sms, int ctasPerSm, const ClusterShape &cluster)
{
    const double M = (double)sz.maxM;
    const bool real = sz.floatArith, two = ctasPerSm > 1;
    if (cluster.ctas == 0) return true;
    const double turns = std::ceil(equal / (sms * ctasPerSm) - 1e-9), clusterTurns = std::ceil(equal / cluster.resident - 1e-9);
    double speed;
    if (cluster.ctas == 1) speed = !real && M > 64 && M < 900 && (turns == 1.0 ? sz.W < 60 : turns == 2.0 && !two && sz.W < 52 && M >= 128) ? 1.1 : 0.95;
    else if (cluster.ctas == 2) speed = M > 1024 ? 1.75 : std::min(std::min(0.55 + M / 230, 1.05 + M / 500), 2.15);
    else if (cluster.ctas == 4) speed = real ? std::min(0.3 + M / 200, 5.5) : std::min(0.95 + M / 310, 4.1);
    else if (cluster.ctas == 8) speed = std::min(M / 155, 8.0) * (real ? 1.2 : 1.0);
    else speed = real ? M / 112 * std::max(1.0, M / 1400) : M / 140;
    if ((cluster.ctas == 2 || cluster.ctas == 4) && sz.W > 64) speed *= 0.88;
    if (cluster.pieces >= 6) speed *= 0.45;               // (teams of one or two warps, six steps and more per row)
    if (two) speed *= cluster.ctas == 1 ? 1.45 : 1.68;    // (a CTA that shares its SM is slower)
    return speed * turns < clusterTurns;
}

static bool rounds_plan(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, int warps, RoundsPlan &plan)
{
    RoundsParams &prm = plan.prm;
    prm = RoundsParams{};
    plan.warps = warps;
    const int perSm = kMaxWarps / warps, batch = warps * kGroup;
    int nonEmpty = 0;
    for (const ClassDesc &c : descHost) nonEmpty += c.M > 0 ? 1 : 0;
    plan.ctas = std::min(nonEmpty, perSm * ctx->smCount);
    // The tables take the place of the class-sorted features, which nothing reads any more.
    prm.scratchBytes = sz.N * sz.pitch / plan.ctas / 256 * 256;
    const int64_t perBlock = sz.maxM * 8 + 32;
    const int blocks = (std::min(sz.W, batch) + kGroup - 1) / kGroup * kGroup;
    if (prm.scratchBytes < perBlock * kGroup) return false;
    prm.scratchBytes = std::min<int64_t>(prm.scratchBytes, (perBlock * blocks + 255) / 256 * 256);
    // (1 KB per CTA is the system's)
    const size_t cap = ((size_t)ctx->maxSmemOptin + 1024) / perSm - 1024 - kRoundsOwnShared, words = (size_t)(pad_row(sz.maxM) + 31) / 32;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 127) / 128 * 128; return (int32_t)at; };
    prm.offKeys = take((size_t)(sz.W + 1) * kListed * 8);
    prm.offBounds = take((size_t)(sz.W + 1) * 8);
    prm.offBits = take(words * 4);
    prm.offNeeded = take(words * 4);
    prm.offBefore = take(words * 4);
    prm.offRows = take((size_t)sz.maxM * 2);
    prm.offPend = take(sizeof(Pending) * (size_t)sz.W);
    // the rest is the ring (a stage: at least four rows of eight column groups; the lists of a batch while there are no tiles)
    if (off > cap) return false;
    prm.stageBytes = (int32_t)((cap - off) / kStages / 128 * 128);
    if (prm.stageBytes < 4 * (8 * 512 + batch * 8)) return false;
    prm.offRing = take((size_t)prm.stageBytes * kStages);
    prm.listShared = std::min(kListShared, prm.stageBytes * kStages / 32);
    plan.smem = off;
    return true;
}

// Classes of the largest size that make as many entries of S.
static double equal_classes(const Sizes &sz, const std::vector<ClassDesc> &descHost)
{
    double equal = 0;
    for (const ClassDesc &c : descHost) equal += (double)c.M * c.M;
    return equal / ((double)sz.maxM * sz.maxM);
}

// Whether rounds come into question: blocks enough, and classes that fill the SMs.
bool rounds_possible(const rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost)
{
    if (sz.graphCut || sz.W > kRoundBlocks || sz.maxM == 0 || sz.maxM > 65535) return false;
    if (sz.W < (sz.floatArith ? 56 : 16)) return false;
    const double equal = equal_classes(sz, descHost), full = equal / (ctx->smCount * std::ceil(equal / ctx->smCount - 1e-9));
    return full >= (sz.W >= 80 ? 0.4 : 0.65) && (sz.W >= 48 || (full >= 0.9 && sz.maxM >= 1000));
}

std::shared_ptr<RoundsPlan> plan_greedy_rounds(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, const ClusterShape &cluster)
{
    if (!rounds_possible(ctx, sz, descHost)) return nullptr;
    const double equal = equal_classes(sz, descHost);
    auto plan = std::make_shared<RoundsPlan>();
    // Two CTAs of eight warps per SM where there are classes for several rounds of them: one's barriers and trips to memory under the
    // other's sums (1000 x 1000 bf16 into 64 blocks: 85.1 ms with one of 16 warps, 80.4 with two; 300 x 1000 into 24: 20.8 and 23.5).
    const bool two = equal >= 3.0 * ctx->smCount && rounds_plan(ctx, sz, descHost, 8, *plan);
    if (!two && !rounds_plan(ctx, sz, descHost, 16, *plan)) return nullptr;
    return rounds_win(sz, equal, ctx->smCount, two ? 2 : 1, cluster) ? plan : nullptr;
}

rcd_status launch_greedy_rounds(rcd_ctx *ctx, RoundsPlan &plan, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st)
{
    RoundsParams &prm = plan.prm;
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.cover = (int32_t *)ws.cover;
    prm.gains = (unsigned long long *)ws.gains;
    prm.g0 = (unsigned long long *)ws.g0;
    prm.picks = (uint32_t *)ws.cand;
    prm.perm = ws.perm;
    prm.quota = ws.quota;
    prm.fval = (long long *)(partValues ? partValues : ws.fval);
    prm.assignment = assignment;
    prm.order = order;
    prm.fixedExp = sz.floatArith ? ws.fixedExp : nullptr;
    prm.classOrder = ws.classOrder;
    prm.counter = ws.counter;
    prm.status = ctx->statusOwn;
    prm.stats = ws.phaseNs;
    prm.scratch = (unsigned char *)ws.Xs;
    prm.L = sz.L;
    prm.W = sz.W;
    prm.one = 1u;
    auto kernel = plan.warps == 8 ? (sz.W <= 32 ? greedy_rounds_kernel<1, 8> : sz.W <= 64 ? greedy_rounds_kernel<2, 8> : greedy_rounds_kernel<4, 8>)
                                  : (sz.W <= 32 ? greedy_rounds_kernel<1, 16> : sz.W <= 64 ? greedy_rounds_kernel<2, 16> : greedy_rounds_kernel<4, 16>);
    RCD_CUDA(ctx, allow_shared(kernel, ctx->maxSmemOptin - kRoundsOwnShared));
    kernel<<<plan.ctas, plan.warps * 32, plan.smem, st>>>(prm);
    RCD_CUDA(ctx, cudaGetLastError());
    ctx->kernelLaunches++;
    return RCD_OK;
}

}  // namespace rcd
