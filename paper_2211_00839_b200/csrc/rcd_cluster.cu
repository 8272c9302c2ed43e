// The greedy loop of Algorithm 1 with the facility-location objective, one thread-block cluster per class: the form
// the library chooses by itself (the pass-based forms of rcd_greedy.cu serve explicit configurations).
//
// What bounds it.  A pick of block j depends on the previous pick of block j (its coverage and gains change), but on
// picks of OTHER blocks only through two things: the tracked values f (which block is next) and the set of unassigned
// samples.  Both are known the moment a pick is decided, because f grows by the gain of the chosen sample.  So picks of
// different blocks need not wait for each other's trips to memory:
//   leader  one warp per cluster decides pick after pick: j* = argmin f, then the best unassigned sample of j*'s list of
//           leading candidates (the "note" its team posted last), and tells j*'s team which sample it received;
//   teams   the cluster's other warps; every block belongs to one team, which keeps the block's coverage and stored
//           gains (in its CTA's shared memory when they fit), folds the sample in, brings the gains up to date and
//           posts the block's next candidates to the leader through distributed shared memory.
// With W blocks of similar size about W updates are in flight, and the loop takes (largest quota) x (one update)
// instead of M x (one update).
//
// Stored gains are always exact: a pick corrects those of its block from one row of S per column whose coverage it
// raised (S is symmetric).  All arithmetic is int64 on int32 similarities, hence independent of the order in which
// anything happens: results do not depend on timing.
#include "rcd_internal.h"

#include <limits.h>
#include <algorithm>

namespace rcd {

namespace {

constexpr int kMaxWarps = 16;             // team warps per CTA (one more warp leads in the cluster's first CTA)
constexpr int kRaisedPerWarp = 64;        // raised columns a team lists at a time, per warp
constexpr int kClusterBlocks = 128;       // blocks a cluster can lead (their notes sit in one CTA's shared memory)
constexpr int kEntries = 32;              // candidates per note
constexpr uint32_t kScanCmd = 0u;         // (a command's low word: 0 = look again, else sample + 1)
constexpr unsigned kPollLimit = 1u << 25;

struct Note {
    unsigned long long entry[kEntries];   // keys of exact candidates (0: none)
    unsigned long long bound[kMaxWarps];  // per team warp: no candidate outside the entries has a key above it
};

struct __align__(16) Raised {
    int32_t row;                          // a column whose coverage rose: its row of S, in 16-byte pieces from the class's first
    int32_t minusOld, by;                 // - old coverage, new - old
    int32_t pad_;
};

struct Team {
    unsigned long long best[kMaxWarps];
    int32_t count;                        // raised columns of the update in hand
    int32_t slot;                         // what warp 0 of the team decided to do next
    uint32_t what;
    int32_t pad_;
};

}  // namespace

struct ClusterParams {
    const ClassDesc *desc;
    const int32_t *S;
    int32_t *cover;            // [sum W*ld] used when the state of a CTA's blocks does not fit its shared memory
    long long *gains;
    long long *g0;             // [N] gains for an empty block
    uint32_t *picks;           // [N] sample | block << 16, in the order picked
    const int32_t *perm;
    const int32_t *quota;
    long long *fval;           // [L][W]
    int32_t *assignment, *order;
    const int32_t *classOrder;
    int32_t *counter;
    int32_t *status;
    unsigned long long *stats; // phase words
    int32_t L, W;
    int32_t warps;             // team warps per CTA
    int32_t teamWarps;         // T
    int32_t slots;             // blocks per CTA at most
    int32_t maxLd;
    uint32_t one;              // the value 1, opaque to the compiler
    // byte offsets into dynamic shared memory
    int32_t offTeams, offLists, offRows, offCmd, offSeen, offBits, offNotes, offBars, offCover, offGains;
};

namespace {
__device__ __forceinline__ uint32_t smem32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t remote(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, unsigned long long v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" :: "r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void st_remote32(uint32_t addr, uint32_t v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
// Asynchronous store to a CTA of the cluster; its 8 bytes count towards the phase of that CTA's mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, unsigned long long v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" :: "r"(addr), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed(uint32_t addr)      // (own shared memory)
{
    unsigned long long v;
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_fence() { asm volatile("fence.acq_rel.cluster;" ::: "memory"); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_done(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }

__device__ __forceinline__ void team_barrier(int team, int T)
{
    if (T == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" :: "r"(1 + team), "r"(T * 32) : "memory");
}

__device__ __forceinline__ int4 ld_row_once(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// acc + x on the multiply-add pipe (the maxima occupy the other one)
__device__ __forceinline__ unsigned long long add_wide(int x, uint32_t one, unsigned long long acc)
{
    unsigned long long r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"((uint32_t)x), "r"(one), "l"(acc));
    return r;
}

// Sum of a value below 2^43 per lane over the warp.
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x)
{
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)(x & 0xffffffu));
    const uint32_t hi = __reduce_add_sync(0xffffffffu, (uint32_t)(x >> 24));
    return ((unsigned long long)hi << 24) + lo;
}

// A gain and a sample as one key: greater gain first, lower sample among equals.  Gains stay below 2^47 (at most 2^16
// samples, similarities below 2^31).
__device__ __forceinline__ unsigned long long make_key(unsigned long long g, int v) { return (g << 16) | (unsigned long long)(65535 - v); }
__device__ __forceinline__ int key_sample(unsigned long long k) { return 65535 - (int)(k & 0xffffull); }

__device__ __forceinline__ unsigned long long umax(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned long long umin(unsigned long long a, unsigned long long b) { return a < b ? a : b; }

// sum_i max(0, S[v][i]) by one warp.
__device__ __forceinline__ unsigned long long row_value(const int4 *row, int ld4, int lane, uint32_t one)
{
    unsigned long long acc = 0;
    for (int q = lane; q < ld4; q += 8 * 32) {
        int4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = q + u * 32 < ld4 ? ld_row_once(row + q + u * 32) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            acc = add_wide(max(x[u].x, 0), one, acc);
            acc = add_wide(max(x[u].y, 0), one, acc);
            acc = add_wide(max(x[u].z, 0), one, acc);
            acc = add_wide(max(x[u].w, 0), one, acc);
        }
    }
    return warp_sum(acc);
}

// What a team knows while it works on a class.
struct TeamView {
    const int4 *S4;            // the class's similarity matrix
    int ld4;
    int warpIn, lane, T, team; // warp inside the team
    Team *tm;
    Raised *list;              // columns the update in hand raised
    int4 *rowBuf;              // row of sample bufV (each thread reads only the pieces it copied itself)
    int bufV;
    const uint32_t *bits;      // assigned samples (and everything from M on)
    uint32_t one;
};

// 16 bytes global -> shared without passing through registers
__device__ __forceinline__ void copy16(int4 *dst, const int4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem32(dst)), "l"(src) : "memory");
}

// Starts copying the team's pieces of row v into its row buffer.
__device__ __forceinline__ void fetch_row(TeamView &t, int v)
{
    const int4 *row = t.S4 + (int64_t)v * t.ld4;
    asm volatile("cp.async.wait_group 0;" ::: "memory");    // (an earlier fetch into the same buffer may be under way)
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) copy16(t.rowBuf + q, row + q);
    asm volatile("cp.async.commit_group;" ::: "memory");
    t.bufV = v;
}

// The block's leading candidates go to the leader: the bests of the team's 32 T threads merge into 32 candidates, and
// what they leave out is bounded.  Then the row of the first candidate is fetched: it is, as a rule, the sample the
// block receives next.
__device__ __forceinline__ void post_candidates(TeamView &t, const long long *gains, uint32_t noteAddr, uint32_t barAddr)
{
    const int T = t.T, lane = t.lane;
    unsigned long long e = 0, o = 0;
    for (int q = t.warpIn * 32 + lane; q < t.ld4; q += T * 32) {
        const uint32_t nib = t.bits[q >> 3] >> ((q & 7) * 4);
        const ulonglong2 a0 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q], a1 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q + 1];
        const unsigned long long g[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const unsigned long long k = (nib >> c & 1) ? 0ull : make_key(g[c], 4 * q + c);
            o = umax(o, umin(e, k));
            e = umax(e, k);
        }
    }
    for (int off = 1; off < T; off <<= 1) {
        const unsigned long long e2 = __shfl_xor_sync(0xffffffffu, e, off), o2 = __shfl_xor_sync(0xffffffffu, o, off);
        o = umax(umax(o, o2), umin(e, e2));
        e = umax(e, e2);
    }
    if ((lane & (T - 1)) == 0) st_async(noteAddr + (uint32_t)((t.warpIn * 32 + lane) / T) * 8, e, barAddr);
    o = warp_max_u64(o);
    if (lane == 0) st_async(noteAddr + (kEntries + t.warpIn) * 8, o, barAddr);
    unsigned long long top = warp_max_u64(e);
    if (T > 1) {
        if (lane == 0) t.tm->best[t.warpIn] = top;
        team_barrier(t.team, T);
        top = warp_max_u64(lane < T ? t.tm->best[lane] : 0ull);
    }
    if (top) fetch_row(t, key_sample(top));
}

// What a candidate loses for one raised column: min(max(x, old), new) - old, as one instruction.  Similarities stay
// within 2^30 either way, so x - old does not wrap.
__device__ __forceinline__ uint32_t loss(int x, const Raised &e) { return (uint32_t)__viaddmin_s32_relu(x, e.minusOld, e.by); }

// One batch of U raised columns applied to a thread's four columns q.
template <int U>
__device__ __forceinline__ void correct_batch(const int4 *base, const Raised *list, uint32_t one, unsigned long long (&d)[4])
{
    int4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = ld_row_once(base + list[u].row);
#pragma unroll
    for (int u = 0; u < U; u += 2) {
        const Raised a = list[u], b = list[u + 1];
        d[0] = add_wide(loss(x[u].x, a) + loss(x[u + 1].x, b), one, d[0]);       // (each below 2^31)
        d[1] = add_wide(loss(x[u].y, a) + loss(x[u + 1].y, b), one, d[1]);
        d[2] = add_wide(loss(x[u].z, a) + loss(x[u + 1].z, b), one, d[2]);
        d[3] = add_wide(loss(x[u].w, a) + loss(x[u + 1].w, b), one, d[3]);
    }
}

// A sample joins a block: its row is folded into the coverage and the stored gains follow, one row of S per column that
// rose (S is symmetric): g(v) falls by min(max(S[v][i], old), new) - old.  The list of raised columns has a fixed room;
// when more rise, the fold stops there and is taken up again after the correction.
__device__ __forceinline__ void take_sample(TeamView &t, int v, int4 *cov, long long *gains, unsigned &rows)
{
    const int first = t.warpIn * 32 + t.lane, step = t.T * 32;
    const int room = t.T * kRaisedPerWarp;
    if (t.bufV != v) fetch_row(t, v);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    for (;;) {
        for (int q = first; q < t.ld4; q += step) {
            const int4 r = t.rowBuf[q];
            const int4 m = cov[q];
            const int up = (r.x > m.x ? 1 : 0) | (r.y > m.y ? 2 : 0) | (r.z > m.z ? 4 : 0) | (r.w > m.w ? 8 : 0);
            if (up) {
                const int n = __popc(up);
                int at = atomicAdd(&t.tm->count, n);
                if (at + n <= room) {
                    const int row = 4 * q * t.ld4;
                    if (up & 1) t.list[at++] = Raised{row, -m.x, r.x - m.x, 0};
                    if (up & 2) t.list[at++] = Raised{row + t.ld4, -m.y, r.y - m.y, 0};
                    if (up & 4) t.list[at++] = Raised{row + 2 * t.ld4, -m.z, r.z - m.z, 0};
                    if (up & 8) t.list[at++] = Raised{row + 3 * t.ld4, -m.w, r.w - m.w, 0};
                    cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
                } else {
                    for (; at < room; ++at) t.list[at] = Raised{0, 0, 0, 0};     // (room that stays unused: no loss)
                }
            }
        }
        team_barrier(t.team, t.T);
        const int all = *(volatile int32_t *)&t.tm->count;
        const int n = min(all, room);
        rows += n;
        // the list is read in batches: entries without effect fill the last one
        if (first < 8 && n + first < room + 8) t.list[n + first] = Raised{0, 0, 0, 0};
        team_barrier(t.team, t.T);
        if (n > 0) {
            const bool own = n == 1 && t.list[0].row == v * t.ld4;           // (most picks: the sample itself is all that rose)
            for (int q = first; q < t.ld4; q += step) {
                unsigned long long d[4] = {0, 0, 0, 0};
                if (own) {
                    const int4 x = t.rowBuf[q];
                    const Raised e = t.list[0];
                    d[0] = loss(x.x, e); d[1] = loss(x.y, e); d[2] = loss(x.z, e); d[3] = loss(x.w, e);
                } else {
                    int e0 = 0;
                    for (; e0 + 4 < n; e0 += 8) correct_batch<8>(t.S4 + q, t.list + e0, t.one, d);
                    if (e0 + 2 < n) correct_batch<4>(t.S4 + q, t.list + e0, t.one, d);
                    else if (e0 < n) correct_batch<2>(t.S4 + q, t.list + e0, t.one, d);
                }
                if (d[0] | d[1] | d[2] | d[3]) {
                    ulonglong2 *p = reinterpret_cast<ulonglong2 *>(gains) + 2 * q;
                    ulonglong2 a = p[0], b = p[1];
                    a.x -= d[0]; a.y -= d[1]; b.x -= d[2]; b.y -= d[3];
                    p[0] = a; p[1] = b;
                }
            }
        }
        if (all <= room) break;
        team_barrier(t.team, t.T);
        if (first == 0) t.tm->count = 0;
        team_barrier(t.team, t.T);
    }
}

// The leader's loop over the picks of class c.  One warp; lane p % 32 keeps the value and the room of block p, and the
// parity of the mbarrier on which the block's notes arrive (they go on from class to class).
template <int KW>
__device__ void lead(const ClusterParams &prm, int l, const ClassDesc &c, unsigned char *shared, uint32_t C, uint32_t &parities)
{
    const int lane = threadIdx.x & 31, W = prm.W;
    const uint32_t noteBytes = (kEntries + prm.teamWarps) * 8;
    const uint32_t base = smem32(shared);
    volatile uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    const Note *notes = reinterpret_cast<const Note *>(shared + prm.offNotes);
    const uint32_t bars = base + prm.offBars;
    unsigned long long f[KW];
    int room[KW];
    uint32_t seq[KW];
    uint32_t awaited = 0;                  // bit k: block lane + 32 k owes a note
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        f[k] = 0;
        seq[k] = 0;
        room[k] = p < W ? prm.quota[(int64_t)l * W + p] : 0;
        if (room[k] > 0) {
            bar_expect(bars + p * 8, noteBytes);
            awaited |= 1u << k;
        }
    }
    __syncwarp();
    unsigned rescans = 0;
    bool ok = true;
    for (int t = 0; t < c.M && ok; ++t) {
        unsigned long long least = ~0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k)
            if (room[k] > 0) least = umin(least, (f[k] << 7) | (unsigned long long)(lane + 32 * k));
        least = ~warp_max_u64(~least);
        if (least == ~0ull) {
            if (lane == 0) atomicOr(prm.status, kDevNoCandidate);
            ok = false;
            break;
        }
        const int j = (int)(least & 127);
        const int jk = j >> 5, jl = j & 31;
        const uint32_t cmd = base + prm.offCmd + (uint32_t)(j / C) * 8;
        const uint32_t owner = (uint32_t)(j % C);
        unsigned long long best = 0;
        for (;;) {
            const uint32_t waits = __shfl_sync(0xffffffffu, awaited, jl) >> jk & 1;
            if (waits) {
                const uint32_t parity = __shfl_sync(0xffffffffu, parities, jl) >> jk & 1;
                unsigned spin = 0;
                while (!bar_done(bars + j * 8, parity) && ++spin < kPollLimit) { }
                if (spin >= kPollLimit) {
                    if (lane == 0) atomicOr(prm.status, kDevTimeout);
                    ok = false;
                    break;
                }
                if (lane == jl) { awaited &= ~(1u << jk); parities ^= 1u << jk; }
            }
            const unsigned long long k = notes[j].entry[lane];
            const unsigned long long bound = lane < prm.teamWarps ? notes[j].bound[lane] : 0ull;
            const int v = key_sample(k);
            const bool free = k != 0 && !(bits[v >> 5] >> (v & 31) & 1);
            best = warp_max_u64(free ? k : 0ull);
            if (best != 0 && __ballot_sync(0xffffffffu, bound >= best) == 0) break;
            // every candidate that is sure to lead has been taken by other blocks: look again
            ++rescans;
            cluster_fence();                               // (the team must see which samples are taken)
            if (lane == jl) {
                bar_expect(bars + j * 8, noteBytes);
                awaited |= 1u << jk;
#pragma unroll
                for (int q = 0; q < KW; ++q) if (q == jk) st_remote(remote(cmd, owner), ((unsigned long long)++seq[q] << 32) | kScanCmd);
            }
        }
        if (!ok) break;
        const int v = key_sample(best);
        const uint32_t word = bits[v >> 5] | (1u << (v & 31));
        __syncwarp();
        if (lane == 0) bits[v >> 5] = word;
        else if (lane < (int)C) st_remote32(remote(base + prm.offBits + (uint32_t)(v >> 5) * 4, lane), word);
        if (lane == jl) {
            const int left = [&] {
                int r = 0;
#pragma unroll
                for (int k = 0; k < KW; ++k) if (k == jk) { f[k] += best >> 16; r = --room[k]; }
                return r;
            }();
            if (left > 0) {                                // (a full block needs no gains any more)
                bar_expect(bars + j * 8, noteBytes);
                awaited |= 1u << jk;
#pragma unroll
                for (int k = 0; k < KW; ++k) if (k == jk) st_remote(remote(cmd, owner), ((unsigned long long)++seq[k] << 32) | (unsigned long long)(v + 1));
            }
        }
        if (lane == 0) prm.picks[c.row0 + t] = (uint32_t)v | ((uint32_t)j << 16);
        __syncwarp();
    }
    // notes still under way land before the class ends
    if (ok)
        for (int k = 0; k < KW; ++k)
            if (awaited >> k & 1) {
                unsigned spin = 0;
                while (!bar_done(bars + (lane + 32 * k) * 8, parities >> k & 1) && ++spin < kPollLimit) { }
                if (spin >= kPollLimit) atomicOr(prm.status, kDevTimeout);
                parities ^= 1u << k;
            }
    __syncwarp();
    if (lane < (int)C) st_remote(remote(base + prm.offCmd + (uint32_t)prm.slots * 8, lane), 1ull);
#pragma unroll
    for (int k = 0; k < KW; ++k)
        if (lane + 32 * k < W) prm.fval[(int64_t)l * W + lane + 32 * k] = (long long)f[k];
    if (lane == 0 && rescans) atomicAdd(prm.stats + 9, (unsigned long long)rescans);
}

template <int KW, bool kSmemState>
__global__ void __launch_bounds__((kMaxWarps + 1) * 32, 1) greedy_cluster_kernel(const __grid_constant__ ClusterParams prm)
{
    extern __shared__ __align__(128) unsigned char shared[];
    __shared__ int shClass[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rank = cluster_rank(), C = cluster_size();
    const int NW = prm.warps, T = prm.teamWarps, nTeams = NW / T;
    const uint32_t base = smem32(shared);
    uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    volatile unsigned long long *cmds = reinterpret_cast<volatile unsigned long long *>(shared + prm.offCmd);
    uint32_t *seen = reinterpret_cast<uint32_t *>(shared + prm.offSeen);
    const int W = prm.W;
    uint32_t parities = 0;

    if (rank == 0)
        for (int p = threadIdx.x; p < W; p += blockDim.x) bar_init(base + prm.offBars + p * 8, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");

    for (int turn = 0;; turn ^= 1) {
        if (rank == 0 && threadIdx.x == 0) {
            const int k = atomicAdd(prm.counter, 1);
            const int l = (k < prm.L && *(volatile int32_t *)prm.status == 0) ? prm.classOrder[k] : -1;
            for (uint32_t r = 0; r < C; ++r) st_remote32(remote(smem32(&shClass[turn]), r), (uint32_t)l);
        }
        cluster_barrier();
        const int l = *(volatile int *)&shClass[turn];
        if (l < 0) break;
        const ClassDesc c = prm.desc[l];
        if (c.M == 0) {
            if (rank == 0) for (int p = threadIdx.x; p < W; p += blockDim.x) prm.fval[(int64_t)l * W + p] = 0;
            continue;
        }
        const int ld4 = c.ld >> 2;
        const int4 *S4 = reinterpret_cast<const int4 *>(prm.S + c.sOff);

        // gains for an empty block, the same for every block: one row of S per sample, over all warps of the cluster
        if (warp < NW)
            for (int v = rank * NW + warp; v < c.M; v += C * NW) {
                const unsigned long long g = row_value(S4 + (int64_t)v * ld4, ld4, lane, prm.one);
                if (lane == 0) __stcg(prm.g0 + c.row0 + v, (long long)g);
            }
        for (int i = threadIdx.x; i < (c.ld + 31) / 32; i += blockDim.x)
            bits[i] = 32 * i + 32 <= c.M ? 0u : (32 * i >= c.M ? ~0u : ~0u << (c.M - 32 * i));
        for (int i = threadIdx.x; i <= prm.slots; i += blockDim.x) {
            cmds[i] = 0;
            if (i < prm.slots) seen[i] = 0;
        }
        cluster_barrier();

        if (warp == NW) {
            if (rank == 0) lead<KW>(prm, l, c, shared, C, parities);
        } else {
            const int team = warp / T;
            TeamView t;
            t.S4 = S4; t.ld4 = ld4;
            t.warpIn = warp - team * T; t.lane = lane; t.T = T; t.team = team;
            t.tm = reinterpret_cast<Team *>(shared + prm.offTeams) + team;
            t.list = reinterpret_cast<Raised *>(shared + prm.offLists) + team * (T * kRaisedPerWarp + 8);
            t.rowBuf = reinterpret_cast<int4 *>(shared + prm.offRows) + (size_t)team * (prm.maxLd >> 2);
            t.bufV = -1;
            t.bits = bits;
            t.one = prm.one;
            unsigned corrected = 0, rows = 0;
            auto cover_of = [&](int slot) -> int4 * {
                if (kSmemState) return reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)slot * (prm.maxLd >> 2);
                return reinterpret_cast<int4 *>(prm.cover + c.vOff) + (size_t)(slot * C + rank) * ld4;
            };
            auto gains_of = [&](int slot) -> long long * {
                if (kSmemState) return reinterpret_cast<long long *>(shared + prm.offGains) + (size_t)slot * prm.maxLd;
                return prm.gains + c.vOff + (size_t)(slot * C + rank) * c.ld;
            };
            const uint32_t notes0 = remote(base + prm.offNotes, 0);
            const uint32_t bars0 = remote(base + prm.offBars, 0);
            int mine = 0;
            for (int slot = team; slot < prm.slots; slot += nTeams) {
                const int j = slot * (int)C + (int)rank;
                if (j >= W) break;
                ++mine;
                if (prm.quota[(int64_t)l * W + j] == 0) continue;
                int4 *cov = cover_of(slot);
                long long *gains = gains_of(slot);
                for (int q = t.warpIn * 32 + lane; q < ld4; q += T * 32) {
                    cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
                    for (int u = 0; u < 4; ++u) gains[4 * q + u] = 4 * q + u < c.M ? __ldcg(prm.g0 + c.row0 + 4 * q + u) : 0;
                }
                post_candidates(t, gains, notes0 + j * (uint32_t)sizeof(Note), bars0 + j * 8);
            }
            for (;;) {
                if (t.warpIn == 0) {
                    // lane i watches the command of the team's i-th block, lane 31 the end of the class
                    const uint32_t at = base + prm.offCmd + (uint32_t)(lane == 31 ? prm.slots : team + lane * nTeams) * 8;
                    const uint32_t had = lane < mine ? seen[team + lane * nTeams] : 0u;
                    unsigned pending = 0;
                    unsigned long long cmd = 0;
                    for (unsigned spin = 0; spin < kPollLimit; ++spin) {
                        if (lane < mine || lane == 31) cmd = ld_relaxed(at);
                        pending = __ballot_sync(0xffffffffu, lane == 31 ? cmd != 0 : (lane < mine && (uint32_t)(cmd >> 32) != had));
                        if (pending) break;
                    }
                    if (pending == 0 && lane == 0) atomicOr(prm.status, kDevTimeout);
                    const int who = pending ? __ffs(pending) - 1 : 31;
                    if (lane == who) {
                        t.tm->count = 0;
                        t.tm->slot = who == 31 ? -1 : team + who * nTeams;
                        t.tm->what = (uint32_t)cmd;
                        if (who != 31) seen[team + who * nTeams] = (uint32_t)(cmd >> 32);
                        if ((uint32_t)cmd == kScanCmd) cluster_fence();
                    }
                }
                team_barrier(team, T);
                const int slot = *(volatile int32_t *)&t.tm->slot;
                if (slot < 0) break;
                const uint32_t what = *(volatile uint32_t *)&t.tm->what;
                const int j = slot * (int)C + (int)rank;
                int4 *cov = cover_of(slot);
                long long *gains = gains_of(slot);
                if (what != kScanCmd) {
                    ++corrected;
                    take_sample(t, (int)what - 1, cov, gains, rows);
                }
                post_candidates(t, gains, notes0 + j * (uint32_t)sizeof(Note), bars0 + j * 8);
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            if (lane == 0 && t.warpIn == 0 && corrected) {
                atomicAdd(prm.stats + 15, (unsigned long long)corrected);
                atomicAdd(prm.stats + 16, (unsigned long long)rows);
            }
        }
        cluster_barrier();
        // class-local picks -> outputs
        for (int t = rank * blockDim.x + threadIdx.x; t < c.M; t += C * blockDim.x) {
            const uint32_t p = __ldcg(prm.picks + c.row0 + t);
            const int global = prm.perm[c.row0 + (p & 0xffff)];
            prm.assignment[global] = (int)(p >> 16);
            if (prm.order) prm.order[c.row0 + t] = global;
        }
    }
}

}  // namespace

static int pow2_at_least(int x)
{
    int p = 1;
    while (p < x) p *= 2;
    return p;
}

template <int KW, bool kSmemState>
static rcd_status launch_cluster(rcd_ctx *ctx, const ClusterParams &prm, int C, int clusters, size_t smem, cudaStream_t st, bool query, int *active)
{
    auto kernel = greedy_cluster_kernel<KW, kSmemState>;
    RCD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    RCD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * C));
    cfg.blockDim = dim3((unsigned)((prm.warps + 1) * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (query) {
        RCD_CUDA(ctx, cudaOccupancyMaxActiveClusters(active, kernel, &cfg));
        return RCD_OK;
    }
    RCD_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, prm));
    ctx->kernelLaunches++;
    return RCD_OK;
}

// Whether the cluster form takes a problem: chosen by the library (no pass-based form or option asked for), samples of
// a class and blocks within the packed keys' range.
bool cluster_form_takes(const rcd_ctx *ctx, const Sizes &sz)
{
    const rcd_config &c = ctx->cfg;
    return c.greedy_path == 0 && c.profile < 2 && c.sweep_batch_max == 0 && c.sweep_mode == 0 && c.async_group == 0 && c.async_help_min == 0 &&
           c.threshold_from == 0 && c.threshold_hit_shift == 0 && c.lazy_mode == 0 && c.lazy_from == 0 && c.dense_ring == 0 &&
           c.incremental == 0 && c.incremental_max == 0 && sz.W <= kClusterBlocks && sz.maxM <= 65535 && !sz.graphCut && !sz.floatArith;
}

rcd_status launch_greedy_cluster(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                 int32_t *assignment, int32_t *order, cudaStream_t st)
{
    int nonEmpty = 0, maxLd = 8;
    std::vector<int32_t> bySize(descHost.size());
    for (size_t i = 0; i < bySize.size(); ++i) {
        bySize[i] = (int32_t)i;
        if (descHost[i].M > 0) ++nonEmpty;
        maxLd = std::max(maxLd, (int)descHost[i].ld);
    }
    std::stable_sort(bySize.begin(), bySize.end(), [&](int32_t a, int32_t b) { return descHost[(size_t)a].M > descHost[(size_t)b].M; });
    RCD_CUDA(ctx, cudaMemcpyAsync(ws.classOrder, bySize.data(), bySize.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    RCD_CUDA(ctx, cudaMemsetAsync(ws.nSweep, 0, 4 * sizeof(int32_t), st));
    RCD_CUDA(ctx, cudaMemsetAsync(ws.phaseNs, 0, kPhaseWords * sizeof(unsigned long long), st));

    ClusterParams prm{};
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.cover = (int32_t *)ws.cover;
    prm.gains = (long long *)ws.gains;
    prm.g0 = ws.g0;
    prm.picks = (uint32_t *)ws.cand;
    prm.perm = ws.perm;
    prm.quota = ws.quota;
    prm.fval = (long long *)ws.fval;
    prm.assignment = assignment;
    prm.order = order;
    prm.classOrder = ws.classOrder;
    prm.counter = ws.nSweep;
    prm.status = ws.status;
    prm.stats = ws.phaseNs;
    prm.L = sz.L;
    prm.W = sz.W;
    prm.maxLd = maxLd;
    prm.one = 1u;
    prm.warps = kMaxWarps;

    const size_t cap = (size_t)ctx->maxSmemOptin - 1024;
    auto layout = [&](int C, bool state) -> size_t {
        prm.slots = (sz.W + C - 1) / C;
        int teams = std::min(kMaxWarps, pow2_at_least(prm.slots));
        // no more warps per team than a row has work for
        teams = std::max(teams, kMaxWarps / std::min(kMaxWarps, pow2_at_least((maxLd / 4 + 15) / 16)));
        prm.teamWarps = kMaxWarps / teams;
        size_t off = 0;
        auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 15) / 16 * 16; return (int32_t)at; };
        prm.offTeams = take(sizeof(Team) * (size_t)teams);
        prm.offCmd = take(8 * (size_t)(prm.slots + 1));
        prm.offSeen = take(4 * (size_t)(prm.slots + 1));
        prm.offBits = take((size_t)(maxLd + 31) / 32 * 4);
        prm.offLists = take(sizeof(Raised) * (size_t)kMaxWarps * (kRaisedPerWarp + 8));
        prm.offRows = take((size_t)std::min(teams, prm.slots) * maxLd * 4);
        prm.offNotes = take(sizeof(Note) * (size_t)sz.W);
        prm.offBars = take(8 * (size_t)sz.W);
        prm.offCover = take(state ? (size_t)prm.slots * maxLd * 4 : 0);
        prm.offGains = take(state ? (size_t)prm.slots * maxLd * 8 : 0);
        return off;
    };
    // Cluster size: as many CTAs per class as there are blocks for and as all classes find room for at once; with more
    // classes than that, the fewest whose shared memory holds the state.
    const int most = std::min(16, pow2_at_least(sz.W));
    int C = 0;
    for (int i = 4; i >= 0; --i) {
        const int size = 1 << i;
        if (ctx->maxClusters[i] == 0) {
            layout(size, false);
            rcd_status rs = launch_cluster<4, true>(ctx, prm, size, 1, cap, st, true, &ctx->maxClusters[i]);
            if (rs != RCD_OK) return rs;
        }
        if (size <= most && ctx->maxClusters[i] >= nonEmpty && C == 0) C = size;
    }
    if (C == 0) {
        C = 1;
        while (C < most && layout(C, true) > cap) C *= 2;
        if (ctx->maxClusters[4] == 0 && C == 16) C = 8;
    }
    int idx = 0;
    while ((1 << idx) < C) ++idx;
    size_t smem = layout(C, true);
    const bool state = smem <= cap;
    if (!state) smem = layout(C, false);
    const int clusters = std::max(1, std::min(nonEmpty, ctx->maxClusters[idx]));
    const int kw = sz.W <= 32 ? 1 : (sz.W <= 64 ? 2 : 4);
    rcd_status rs;
    if (state) rs = kw == 1 ? launch_cluster<1, true>(ctx, prm, C, clusters, smem, st, false, nullptr)
                 : kw == 2 ? launch_cluster<2, true>(ctx, prm, C, clusters, smem, st, false, nullptr)
                           : launch_cluster<4, true>(ctx, prm, C, clusters, smem, st, false, nullptr);
    else rs = launch_cluster<4, false>(ctx, prm, C, clusters, smem, st, false, nullptr);
    if (rs != RCD_OK) return rs;
    ctx->steps = sz.maxM;
    ctx->phaseNsDev = ws.phaseNs;
    return RCD_OK;
}

}  // namespace rcd
