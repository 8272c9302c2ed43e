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
constexpr int kEntries = 16;              // candidates per note
constexpr uint32_t kScanCmd = 0u;         // a command's low word: look again;
constexpr uint32_t kStopCmd = ~0u;        //   the class is done;  anything else: sample + 1 joins the block
constexpr unsigned kPollLimit = 1u << 25;

// What a team tells the leader about a block: the key of its best candidate (0: none), and for the case that other
// blocks took that one: [1, 17) keys of leading candidates, [17, 17 + T) per team warp a key that no other exceeds.
struct Note {
    unsigned long long word[1 + kEntries + kMaxWarps];
};

struct __align__(16) Raised {
    int32_t row;                          // a column whose coverage rose: its row of S, in 16-byte pieces from the class's first
    int32_t minusOld, by;                 // - old coverage, new - old
    int32_t pad_;
};

struct Team {
    unsigned long long best[kMaxWarps];
    int32_t count[4];                     // lengths of its lists: foreseen samples (in turn), others
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
    const int32_t *fixedExp;   // [L] floating-point similarities: S = round(sim * 2^fixedExp) (null: integers)
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
    int32_t offTeams, offLists, offRows, offCmd, offBits, offNotes, offBars, offCover, offKeys;
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
    asm volatile("st.volatile.shared::cluster.u64 [%0], %1;" :: "r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void st_remote32(uint32_t addr, uint32_t v)
{
    asm volatile("st.volatile.shared::cluster.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
// Asynchronous store to a CTA of the cluster; its 8 bytes count towards the phase of that CTA's mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, unsigned long long v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" :: "r"(addr), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed(uint32_t addr)      // (own shared memory)
{
    unsigned long long v;
    asm volatile("ld.volatile.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
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
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
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

// key with a loss of l taken off its gain (one multiply-add)
__device__ __forceinline__ unsigned long long take_off(unsigned long long key, int l)
{
    unsigned long long r;
    asm("mad.wide.s32 %0, %1, -65536, %2;" : "=l"(r) : "r"(l), "l"(key));
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

// The team of a warp, and what it knows while it works on a class.
struct TeamView {
    const int4 *S4;            // the class's similarity matrix
    int ld4;
    int warpIn, lane, T, team; // warp inside the team
    Team *tm;
    Raised *list;              // columns the update in hand raised
    int4 *rowBuf;              // a sample's row (each thread reads only the pieces it copied itself)
    const uint32_t *bits;      // assigned samples (and everything from M on)
};

// 16 bytes global -> shared without passing through registers
__device__ __forceinline__ void copy16(int4 *dst, const int4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// Starts copying the team's pieces of row v into its row buffer.
__device__ __forceinline__ void fetch_row(const TeamView &t, int v)
{
    const int4 *row = t.S4 + (int64_t)v * t.ld4;
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) copy16(t.rowBuf + q, row + q);
    copies_commit();
}

// What a candidate loses for one raised column: min(max(x, old), new) - old, as one instruction.  Similarities stay
// below 2^30 either way, so x - old does not wrap, and two losses fit an int.
__device__ __forceinline__ int loss(int x, const Raised &e) { return __viaddmin_s32_relu(x, e.minusOld, e.by); }

__device__ __forceinline__ unsigned long long tile_max(uint32_t mask, unsigned long long k)
{
    const uint32_t hi = (uint32_t)(k >> 32), lo = (uint32_t)k;
    const uint32_t mhi = __reduce_max_sync(mask, hi);
    const uint32_t mlo = __reduce_max_sync(mask, hi == mhi ? lo : 0u);
    return ((unsigned long long)mhi << 32) | mlo;
}

// A warp's part of a note from its threads' best and second-best keys: entries (one per tile of 2 T lanes, at the tile's
// first lane), a bound on everything else, and the best of all.
struct Summary {
    unsigned long long entry, bound, top;
};
__device__ __forceinline__ Summary summarize(unsigned long long e, unsigned long long o, int T, int lane)
{
    Summary s;
    if (T <= 2) {
        for (int off = 1; off < 2 * T; off <<= 1) {
            const unsigned long long e2 = __shfl_xor_sync(0xffffffffu, e, off), o2 = __shfl_xor_sync(0xffffffffu, o, off);
            o = umax(umax(o, o2), umin(e, e2));
            e = umax(e, e2);
        }
        s.entry = e;
        s.bound = warp_max_u64(o);
    } else {
        const int tile = 2 * T;
        const uint32_t mask = tile == 32 ? 0xffffffffu : ((1u << tile) - 1u) << (lane & ~(tile - 1));
        s.entry = tile_max(mask, e);
        s.bound = warp_max_u64(e == s.entry ? o : e);
    }
    s.top = warp_max_u64(s.entry);
    return s;
}
__device__ __forceinline__ void post(const TeamView &t, const Summary &s, uint32_t noteAddr, uint32_t barAddr)
{
    const int tile = 2 * t.T;
    if ((t.lane & (tile - 1)) == 0) st_async(noteAddr + (uint32_t)(1 + (t.warpIn * 32 + t.lane) / tile) * 8, s.entry, barAddr);
    if (t.lane == 1) st_async(noteAddr + (uint32_t)(1 + kEntries + t.warpIn) * 8, s.bound, barAddr);
}

// Columns of one piece that rose join the list, as far as it has room.  Returns which did.
__device__ __forceinline__ int list_raised(const TeamView &t, int32_t *count, int q, const int4 &r, const int4 &m)
{
    int up = (r.x > m.x ? 1 : 0) | (r.y > m.y ? 2 : 0) | (r.z > m.z ? 4 : 0) | (r.w > m.w ? 8 : 0);
    if (up) {
        const int room = t.T * kRaisedPerWarp;
        int at = atomicAdd(count, __popc(up));
        const int row = 4 * q * t.ld4;
        const int took = min(room - at, __popc(up));
        if (took < __popc(up)) {                                          // the list is full: these wait for the next one
            for (int k = 0; k < took; ++k) t.list[at + k] = Raised{0, 0, 0, 0};
            return 0;
        }
        if (up & 1) t.list[at++] = Raised{row, -m.x, r.x - m.x, 0};
        if (up & 2) t.list[at++] = Raised{row + t.ld4, -m.y, r.y - m.y, 0};
        if (up & 4) t.list[at++] = Raised{row + 2 * t.ld4, -m.z, r.z - m.z, 0};
        if (up & 8) t.list[at++] = Raised{row + 3 * t.ld4, -m.w, r.w - m.w, 0};
    }
    return up;
}

// Takes the listed columns' losses off the keys (gain << 16 | tie-break) of one piece, U rows of S in flight.
template <int U>
__device__ __forceinline__ int correct_batch(const int4 *S4q, const Raised *list, int left, unsigned long long (&key)[4])
{
    int4 x[U];
    int changed = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = ld_row_once(S4q + list[min(u, left - 1)].row);
#pragma unroll
    for (int u = 0; u < U; u += 2) {
        const Raised a = list[min(u, left - 1)];
        Raised b = list[min(u + 1, left - 1)];
        if (u + 1 >= left) b.minusOld = b.by = 0;
        if (u < left) {
            const int l0 = loss(x[u].x, a) + loss(x[u + 1].x, b), l1 = loss(x[u].y, a) + loss(x[u + 1].y, b);
            const int l2 = loss(x[u].z, a) + loss(x[u + 1].z, b), l3 = loss(x[u].w, a) + loss(x[u + 1].w, b);
            changed |= l0 | l1 | l2 | l3;
            key[0] = take_off(key[0], l0);
            key[1] = take_off(key[1], l1);
            key[2] = take_off(key[2], l2);
            key[3] = take_off(key[3], l3);
        }
    }
    return changed;
}
__device__ __forceinline__ int correct_full(const int4 *S4q, const Raised *list, unsigned long long (&key)[4])
{
    int4 x[8];
    int changed = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = ld_row_once(S4q + list[u].row);
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
        const Raised a = list[u], b = list[u + 1];
        const int l0 = loss(x[u].x, a) + loss(x[u + 1].x, b), l1 = loss(x[u].y, a) + loss(x[u + 1].y, b);
        const int l2 = loss(x[u].z, a) + loss(x[u + 1].z, b), l3 = loss(x[u].w, a) + loss(x[u + 1].w, b);
        changed |= l0 | l1 | l2 | l3;
        key[0] = take_off(key[0], l0);
        key[1] = take_off(key[1], l1);
        key[2] = take_off(key[2], l2);
        key[3] = take_off(key[3], l3);
    }
    return changed;
}
__device__ __forceinline__ int correct(const TeamView &t, int n, int q, unsigned long long (&key)[4])
{
    const int4 *S4q = t.S4 + q;
    int changed = 0, e0 = 0;
    for (; e0 + 8 <= n; e0 += 8) changed |= correct_full(S4q, t.list + e0, key);
    if (e0 + 4 < n) changed |= correct_batch<8>(S4q, t.list + e0, n - e0, key);
    else if (e0 + 2 < n) changed |= correct_batch<4>(S4q, t.list + e0, n - e0, key);
    else if (e0 < n) changed |= correct_batch<2>(S4q, t.list + e0, n - e0, key);
    return changed;
}

// A thread's best and second-best key among its pieces of a block's stored gains.
__device__ __forceinline__ void scan_keys(const TeamView &t, const unsigned long long *keys, unsigned long long &e, unsigned long long &o)
{
    e = o = 0;
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) {
        const uint32_t nib = t.bits[q >> 3] >> ((q & 7) * 4);
        const ulonglong2 a0 = reinterpret_cast<const ulonglong2 *>(keys)[2 * q], a1 = reinterpret_cast<const ulonglong2 *>(keys)[2 * q + 1];
        const unsigned long long g[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned long long k = (nib >> u & 1) ? 0ull : g[u];
            o = umax(o, umin(e, k));
            e = umax(e, k);
        }
    }
}

// Applies the n listed columns to the thread's pieces of a block's keys.  Returns whether any moved.
__device__ __forceinline__ bool correct_keys(const TeamView &t, int n, unsigned long long *keys)
{
    bool moved = false;
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) {
        ulonglong2 *p = reinterpret_cast<ulonglong2 *>(keys) + 2 * q;
        ulonglong2 a = p[0], b = p[1];
        unsigned long long k[4] = {a.x, a.y, b.x, b.y};
        if (correct(t, n, q, k)) {
            moved = true;
            p[0] = make_ulonglong2(k[0], k[1]);
            p[1] = make_ulonglong2(k[2], k[3]);
        }
    }
    return moved;
}

// Folds a row into the coverage and corrects the keys, list by list.  The row: in the team's buffer (each thread's own
// pieces) or in S.
__device__ __forceinline__ void take_in_lists(const TeamView &t, const int4 *row, int4 *cov, unsigned long long *keys, unsigned &rows)
{
    const int tid = t.warpIn * 32 + t.lane, step = t.T * 32;
    const int room = t.T * kRaisedPerWarp;
    int32_t *count = &t.tm->count[2];
    for (;;) {
        team_barrier(t.team, t.T);                         // (the list's last readers are done)
        if (tid == 0) *count = 0;
        team_barrier(t.team, t.T);
        for (int q = tid; q < t.ld4; q += step) {
            const int4 r = row[q], m = cov[q];
            if (list_raised(t, count, q, r, m)) cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
        }
        team_barrier(t.team, t.T);
        const int all = *(volatile int32_t *)count;
        const int n = min(all, room);
        rows += n;
        if (n > 0) correct_keys(t, n, keys);
        if (all <= room) break;
    }
}

// Keys of an empty block and its coverage.
__device__ __forceinline__ void start_block(const ClusterParams &prm, const ClassDesc &c, const TeamView &t, int4 *cov, unsigned long long *keys)
{
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) {
        cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int v = 4 * q + u;
            keys[v] = v < c.M ? make_key((unsigned long long)__ldcg(prm.g0 + c.row0 + v), v) : 0ull;
        }
    }
}

// A team with one block.
__device__ __forceinline__ void team_of_one(const ClusterParams &prm, const ClassDesc &c, const TeamView &t, int4 *cov, unsigned long long *keys,
                                            uint32_t cmdAddr, uint32_t noteAddr, uint32_t barAddr, unsigned &corrected, unsigned &rows)
{
    const int T = t.T, tid = t.warpIn * 32 + t.lane, step = T * 32, lane = t.lane;
    const int room = T * kRaisedPerWarp;
    start_block(prm, c, t, cov, keys);
    if (tid == 0) t.tm->count[0] = t.tm->count[1] = 0;
    unsigned long long e = 0, o = 0;
    Summary sum{0, 0, 0};
    bool dirty = true;
    uint32_t had = 0;
    for (int par = 0;; par ^= 1) {
        // candidates: a thread looks again when its gains changed or its best has been assigned
        if (!dirty && e != 0) {
            const int s = key_sample(e);
            dirty = t.bits[s >> 5] >> (s & 31) & 1;
        }
        if (__any_sync(0xffffffffu, dirty)) {
            if (dirty) scan_keys(t, keys, e, o);
            __syncwarp();
            sum = summarize(e, o, T, lane);
            dirty = false;
            // (the warp's best may be the block's best some picks from now: its row comes to L2 meanwhile)
            if (T > 1 && sum.top) {
                const char *row = reinterpret_cast<const char *>(t.S4 + (int64_t)key_sample(sum.top) * t.ld4);
                for (int at = lane * 128; at < t.ld4 * 16; at += 32 * 128) asm volatile("prefetch.global.L2 [%0];" :: "l"(row + at));
            }
        }
        post(t, sum, noteAddr, barAddr);
        unsigned long long top = sum.top;
        if (T > 1) {
            if (lane == 0) t.tm->best[t.warpIn] = top;
            team_barrier(t.team, T);
            top = warp_max_u64(lane < T ? t.tm->best[lane] : 0ull);
        }
        if (tid == 0) st_async(noteAddr, top, barAddr);
        // until the command comes: the row of the best candidate, which is, as a rule, the sample the block receives
        // next, and the columns it would raise
        int v = top ? key_sample(top) : -1;
        int32_t *count = &t.tm->count[par];
        int all = 0;
        if (v >= 0) {
            fetch_row(t, v);
            copies_wait<0>();
            for (int q = tid; q < t.ld4; q += step) list_raised(t, count, q, t.rowBuf[q], cov[q]);
            team_barrier(t.team, T);
            all = *(volatile int32_t *)count;
        }
        if (tid == 0) t.tm->count[par ^ 1] = 0;
        unsigned long long cmd = 0;
        unsigned spin = 0;
        while ((uint32_t)((cmd = ld_relaxed(cmdAddr)) >> 32) == had && ++spin < kPollLimit) { }
        if (spin >= kPollLimit) {
            if (lane == 0) atomicOr(prm.status, kDevTimeout);
            break;
        }
        had = (uint32_t)(cmd >> 32);
        const uint32_t what = (uint32_t)cmd;
        if (what == kStopCmd) break;
        if (what == kScanCmd) {
            cluster_fence();
            dirty = true;
            continue;
        }
        ++corrected;
        if ((int)what - 1 != v || all > room) {
            // another sample than foreseen, or more raised columns than one list holds
            if ((int)what - 1 != v) {
                fetch_row(t, (int)what - 1);
                copies_wait<0>();
            }
            take_in_lists(t, t.rowBuf, cov, keys, rows);
            dirty = true;
            continue;
        }
        rows += all;
        const bool own = all == 1 && t.list[0].row == v * t.ld4;         // (most picks: the sample itself is all that rose)
        const Raised mine = t.list[0];
        for (int q = tid; q < t.ld4 && all > 0; q += step) {
            const int4 r = t.rowBuf[q], m = cov[q];
            if (r.x > m.x || r.y > m.y || r.z > m.z || r.w > m.w) cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
            if (own) {
                const int l0 = loss(r.x, mine), l1 = loss(r.y, mine), l2 = loss(r.z, mine), l3 = loss(r.w, mine);
                if (l0 | l1 | l2 | l3) {
                    dirty = true;
                    ulonglong2 *p = reinterpret_cast<ulonglong2 *>(keys) + 2 * q;
                    const ulonglong2 a = p[0], b = p[1];
                    p[0] = make_ulonglong2(take_off(a.x, l0), take_off(a.y, l1));
                    p[1] = make_ulonglong2(take_off(b.x, l2), take_off(b.y, l3));
                }
            }
        }
        if (!own && all > 0) dirty = correct_keys(t, all, keys);         // (the sample's own gain is 0 now)
    }
    copies_wait<0>();
}

// A one-warp team with several blocks: it serves whichever has a command.
template <typename Where>
__device__ __forceinline__ void team_of_many(const ClusterParams &prm, int l, const ClassDesc &c, const TeamView &t, int mine, uint32_t cmd0,
                                             int cmdStride, Where where, unsigned &corrected, unsigned &rows)
{
    const int lane = t.lane;
    int4 *cov;
    unsigned long long *keys;
    uint32_t noteAddr, barAddr;
    auto tell = [&] {
        unsigned long long e, o;
        scan_keys(t, keys, e, o);
        const Summary sum = summarize(e, o, 1, lane);
        post(t, sum, noteAddr, barAddr);
        if (lane == 0) st_async(noteAddr, sum.top, barAddr);
    };
    for (int i = 0; i < mine; ++i) {
        const int j = where(i, cov, keys, noteAddr, barAddr);
        start_block(prm, c, t, cov, keys);
        if (prm.quota[(int64_t)l * prm.W + j] > 0) tell();
    }
    // lane i watches the command of the team's i-th block
    const uint32_t at = cmd0 + (uint32_t)(min(lane, mine - 1) * cmdStride);
    uint32_t had = 0;
    for (;;) {
        unsigned long long cmd = 0;
        unsigned pending = 0, spin = 0;
        do {
            cmd = ld_relaxed(at);
            pending = __ballot_sync(0xffffffffu, lane < mine && (uint32_t)(cmd >> 32) != had);
        } while (pending == 0 && ++spin < kPollLimit);
        if (pending == 0) {
            if (lane == 0) atomicOr(prm.status, kDevTimeout);
            break;
        }
        const int who = __ffs(pending) - 1;
        const uint32_t what = __shfl_sync(0xffffffffu, (uint32_t)cmd, who);
        if (lane == who) had = (uint32_t)(cmd >> 32);
        if (what == kStopCmd) break;
        where(who, cov, keys, noteAddr, barAddr);
        if (what == kScanCmd) {
            cluster_fence();
        } else {
            ++corrected;
            take_in_lists(t, t.S4 + (int64_t)((int)what - 1) * t.ld4, cov, keys, rows);
        }
        __syncwarp();
        tell();
    }
}

// The leader's loop over the picks of class c.  One warp; lane p % 32 keeps the value and the room of block p, and the
// parity of the mbarrier on which the block's notes arrive (they go on from class to class).
template <int KW>
__device__ void lead(const ClusterParams &prm, int l, const ClassDesc &c, unsigned char *shared, uint32_t C, uint32_t &parities)
{
    const int lane = threadIdx.x & 31, W = prm.W, T = prm.teamWarps;
    const uint32_t noteBytes = (1 + kEntries + T) * 8;
    const uint32_t base = smem32(shared);
    volatile uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    const uint32_t myBits = remote(base + prm.offBits, (uint32_t)lane < C ? lane : 0);
    volatile const Note *notes = reinterpret_cast<const Note *>(shared + prm.offNotes);
    const uint32_t bars = base + prm.offBars;
    unsigned long long f[KW];              // value << 7 | block
    int room[KW];
    uint32_t seq[KW], cmdAddr[KW];
    uint32_t awaited = 0;                  // bit k: block lane + 32 k owes a note
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        f[k] = p;
        seq[k] = 0;
        room[k] = p < W ? prm.quota[(int64_t)l * W + p] : 0;
        cmdAddr[k] = remote(base + prm.offCmd + (uint32_t)((p < W ? p : 0) / C) * 8, (uint32_t)(p < W ? p : 0) % C);
        if (room[k] > 0) {
            bar_expect(bars + p * 8, noteBytes);
            awaited |= 1u << k;
        }
    }
    __syncwarp();
    unsigned rescans = 0;
    bool ok = true;
    for (int t = 0; t < c.M; ++t) {
        unsigned long long least = ~0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k) least = room[k] > 0 ? umin(least, f[k]) : least;
        least = ~warp_max_u64(~least);
        if (least == ~0ull) {
            if (lane == 0) atomicOr(prm.status, kDevNoCandidate);
            ok = false;
            break;
        }
        const int j = (int)(least & 127);
        const int jk = KW == 1 ? 0 : j >> 5, jl = j & 31;
        const uint32_t state = __shfl_sync(0xffffffffu, awaited | parities << 16, jl) >> jk;
        uint32_t waits = state & 1, parity = state >> 16 & 1;
        unsigned long long best = 0;
        for (;;) {
            if (waits) {
                unsigned spin = 0;
                while (!bar_done(bars + j * 8, parity) && ++spin < kPollLimit) { }
                if (spin >= kPollLimit) {
                    if (lane == 0) atomicOr(prm.status, kDevTimeout);
                    ok = false;
                    break;
                }
                parity ^= 1;
                if (lane == jl) { awaited &= ~(1u << jk); parities ^= 1u << jk; }
            }
            best = notes[j].word[0];
            {
                const int s = key_sample(best);
                if (best != 0 && !(bits[s >> 5] >> (s & 31) & 1)) break;
            }
            // the best one has been taken: the best of those left, if none that the note leaves out can lead
            const unsigned long long k = lane < kEntries + T ? notes[j].word[1 + lane] : 0ull;
            const int s = key_sample(k);
            const bool free = lane < kEntries && k != 0 && !(bits[s >> 5] >> (s & 31) & 1);
            best = warp_max_u64(free ? k : 0ull);
            if (best != 0 && __ballot_sync(0xffffffffu, lane >= kEntries && k >= best) == 0) break;
            // every candidate that is sure to lead has been taken by other blocks: look again
            ++rescans;
            waits = 1;
            cluster_fence();                               // (the team must see which samples are taken)
            if (lane == jl) {
                bar_expect(bars + j * 8, noteBytes);
                awaited |= 1u << jk;
#pragma unroll
                for (int q = 0; q < KW; ++q) if (q == jk) st_remote(cmdAddr[q], ((unsigned long long)++seq[q] << 32) | kScanCmd);
            }
        }
        if (!ok) break;
        const int v = key_sample(best);
        if (lane == jl) {
#pragma unroll
            for (int k = 0; k < KW; ++k)
                if (k == jk) {
                    f[k] += best >> 16 << 7;
                    if (--room[k] > 0) {                   // (a full block needs no gains any more)
                        bar_expect(bars + j * 8, noteBytes);
                        awaited |= 1u << k;
                        st_remote(cmdAddr[k], ((unsigned long long)++seq[k] << 32) | (unsigned long long)(v + 1));
                    }
                }
        }
        const uint32_t word = bits[v >> 5] | (1u << (v & 31));
        __syncwarp();
        if (lane == 0) {
            bits[v >> 5] = word;
            prm.picks[c.row0 + t] = (uint32_t)v | ((uint32_t)j << 16);
        } else if (lane < (int)C) {
            st_remote32(myBits + (uint32_t)(v >> 5) * 4, word);
        }
        __syncwarp();
    }
    // notes still under way land before the class ends; then every team is sent home
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        if (ok && (awaited >> k & 1)) {
            unsigned spin = 0;
            while (!bar_done(bars + p * 8, parities >> k & 1) && ++spin < kPollLimit) { }
            if (spin >= kPollLimit) atomicOr(prm.status, kDevTimeout);
            parities ^= 1u << k;
        }
        if (p < W) {
            st_remote(cmdAddr[k], ((unsigned long long)++seq[k] << 32) | kStopCmd);
            const long long value = (long long)(f[k] >> 7);
            prm.fval[(int64_t)l * W + p] = prm.fixedExp ? __double_as_longlong(ldexp((double)value, -prm.fixedExp[l])) : value;
        }
    }
    if (lane == 0 && rescans) atomicAdd(prm.stats + 9, (unsigned long long)rescans);
}

// kSmemState: coverage and stored gains fit the CTAs' shared memory.  kManyBlocks: teams of one warp with several blocks.
template <int KW, bool kSmemState, bool kManyBlocks>
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
        for (int i = threadIdx.x; i < prm.slots; i += blockDim.x) cmds[i] = 0;
        cluster_barrier();

        if (warp == NW) {
            if (rank == 0) lead<KW>(prm, l, c, shared, C, parities);
        } else {
            const int team = warp / T;
            TeamView t;
            t.S4 = S4; t.ld4 = ld4;
            t.warpIn = warp - team * T; t.lane = lane; t.T = T; t.team = team;
            t.tm = reinterpret_cast<Team *>(shared + prm.offTeams) + team;
            t.list = reinterpret_cast<Raised *>(shared + prm.offLists) + team * (T * kRaisedPerWarp + 1);
            t.rowBuf = reinterpret_cast<int4 *>(shared + prm.offRows) + (size_t)team * (prm.maxLd >> 2);
            t.bits = bits;
            unsigned corrected = 0, rows = 0;
            const uint32_t notes0 = remote(base + prm.offNotes, 0), bars0 = remote(base + prm.offBars, 0);
            // the i-th block of the team
            auto where = [&](int i, int4 *&cov, unsigned long long *&keys, uint32_t &noteAddr, uint32_t &barAddr) -> int {
                const int slot = team + i * nTeams, j = slot * (int)C + (int)rank;
                if (kSmemState) {
                    cov = reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)slot * (prm.maxLd >> 2);
                    keys = reinterpret_cast<unsigned long long *>(shared + prm.offKeys) + (size_t)slot * prm.maxLd;
                } else {
                    cov = reinterpret_cast<int4 *>(prm.cover + c.vOff) + (size_t)j * ld4;
                    keys = reinterpret_cast<unsigned long long *>(prm.gains + c.vOff) + (size_t)j * c.ld;
                }
                noteAddr = notes0 + j * (uint32_t)sizeof(Note);
                barAddr = bars0 + j * 8;
                return j;
            };
            int mine = 0;
            while (team + mine * nTeams < prm.slots && (team + mine * nTeams) * (int)C + (int)rank < W) ++mine;
            if (mine == 1 && !kManyBlocks) {
                int4 *cov;
                unsigned long long *keys;
                uint32_t noteAddr, barAddr;
                const int j = where(0, cov, keys, noteAddr, barAddr);
                if (prm.quota[(int64_t)l * W + j] > 0)
                    team_of_one(prm, c, t, cov, keys, base + prm.offCmd + team * 8, noteAddr, barAddr, corrected, rows);
            } else if (mine >= 1 && kManyBlocks) {
                team_of_many(prm, l, c, t, mine, base + prm.offCmd + team * 8, nTeams * 8, where, corrected, rows);
            }
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

// Floating-point similarities as fixed-point integers, so that sums of them are exact.  The largest similarity of a class
// is the largest squared norm (Cauchy-Schwarz), i.e. on the diagonal; it lands in [2^29, 2^30), which leaves every entry
// an absolute precision of 2^-30 of it: finer than the fp32 dot products themselves (2^-24 of the products they add up).
__global__ void __launch_bounds__(256, 8) fixed_exponent_kernel(const ClassDesc *__restrict__ desc, const float *__restrict__ S, int32_t *__restrict__ fixedExp)
{
    __shared__ float shMax[8];
    const ClassDesc c = desc[blockIdx.x];
    float m = 0.f;
    for (int v = threadIdx.x; v < c.M; v += 256) m = fmaxf(m, S[c.sOff + (int64_t)v * c.ld + v]);
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) shMax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = fmaxf(m, shMax[w]);
        int e = 0;
        if (m > 0.f && m <= 3.4e38f) frexpf(m, &e);         // m = x 2^e, x in [0.5, 1)
        fixedExp[blockIdx.x] = 30 - e;
    }
}
__global__ void __launch_bounds__(256, 8) fixed_point_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ fixedExp, float *__restrict__ S)
{
    const ClassDesc c = desc[blockIdx.y];
    const float scale = ldexpf(1.f, fixedExp[blockIdx.y]);
    float4 *p = reinterpret_cast<float4 *>(S + c.sOff);
    const int64_t n = (int64_t)c.M * (c.ld >> 2);
    constexpr int kMost = (1 << 30) - 1;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const float4 x = p[i];
        const int4 y = make_int4(min(max(__float2int_rn(x.x * scale), -kMost), kMost), min(max(__float2int_rn(x.y * scale), -kMost), kMost),
                                 min(max(__float2int_rn(x.z * scale), -kMost), kMost), min(max(__float2int_rn(x.w * scale), -kMost), kMost));
        reinterpret_cast<int4 *>(p)[i] = y;
    }
}

static int pow2_at_least(int x)
{
    int p = 1;
    while (p < x) p *= 2;
    return p;
}

typedef void (*ClusterKernel)(ClusterParams);

template <int KW>
static ClusterKernel pick_kernel(bool smemState, bool many)
{
    if (many) return smemState ? greedy_cluster_kernel<KW, true, true> : greedy_cluster_kernel<KW, false, true>;
    return smemState ? greedy_cluster_kernel<KW, true, false> : greedy_cluster_kernel<KW, false, false>;
}

static rcd_status launch_cluster(rcd_ctx *ctx, ClusterKernel kernel, const ClusterParams &prm, int C, int clusters, size_t smem, cudaStream_t st, int *active)
{
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
    if (active) {                                          // how many such clusters are resident at once
        RCD_CUDA(ctx, cudaOccupancyMaxActiveClusters(active, kernel, &cfg));
        return RCD_OK;
    }
    RCD_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, prm));
    ctx->kernelLaunches++;
    return RCD_OK;
}

// Whether the cluster form takes a problem: chosen by the library (no pass-based form or option asked for), samples of
// a class and blocks within the packed keys' range.
bool cluster_form_takes(const rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &)
{
    const rcd_config &c = ctx->cfg;
    return c.greedy_path == 0 && c.profile < 2 && c.sweep_batch_max == 0 && c.sweep_mode == 0 && c.async_group == 0 && c.async_help_min == 0 &&
           c.threshold_from == 0 && c.threshold_hit_shift == 0 && c.lazy_mode == 0 && c.lazy_from == 0 && c.dense_ring == 0 &&
           c.incremental == 0 && c.incremental_max == 0 && sz.W <= kClusterBlocks && sz.maxM <= 65535 && sz.d <= 65535 && !sz.graphCut && sz.L <= 65535 &&
           (sz.L <= ctx->smCount || sz.maxM <= 512);
}

rcd_status launch_greedy_cluster(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                 int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st)
{
    int nonEmpty = 0, maxLd = 8;
    for (const ClassDesc &c : descHost) {
        if (c.M > 0) ++nonEmpty;
        maxLd = std::max(maxLd, (int)c.ld);
    }

    ClusterParams prm{};
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.cover = (int32_t *)ws.cover;
    prm.gains = (long long *)ws.gains;
    prm.g0 = ws.g0;
    prm.picks = (uint32_t *)ws.cand;
    prm.perm = ws.perm;
    prm.quota = ws.quota;
    prm.fval = (long long *)(partValues ? partValues : ws.fval);
    prm.assignment = assignment;
    prm.order = order;
    prm.fixedExp = sz.floatArith ? ws.fixedExp : nullptr;
    if (sz.floatArith) {
        fixed_exponent_kernel<<<sz.L, 256, 0, st>>>(ws.desc, (const float *)ws.S, ws.fixedExp);
        const int64_t pieces = sz.maxM * (int64_t)(maxLd / 4);
        const dim3 grid((unsigned)std::min<int64_t>((pieces + 1023) / 1024, std::max(1, 16 * ctx->smCount / sz.L)), (unsigned)sz.L);
        fixed_point_kernel<<<grid, 256, 0, st>>>(ws.desc, ws.fixedExp, (float *)ws.S);
        ctx->kernelLaunches += 2;
        RCD_CUDA(ctx, cudaGetLastError());
    }
    prm.classOrder = ws.classOrder;
    prm.counter = ws.counter;
    prm.status = ctx->statusOwn;
    prm.stats = ws.phaseNs;
    prm.L = sz.L;
    prm.W = sz.W;
    prm.maxLd = maxLd;
    prm.one = 1u;
    prm.warps = kMaxWarps;

    const size_t cap = (size_t)ctx->maxSmemOptin - 1024;
    bool many = false;
    auto layout = [&](int C, bool state) -> size_t {
        prm.slots = (sz.W + C - 1) / C;
        // a team per block, of as many warps as a row has work for
        const int most = kMaxWarps / std::min(kMaxWarps, pow2_at_least(prm.slots));
        prm.teamWarps = std::min(most, pow2_at_least((maxLd / 4 + 31) / 32));
        many = prm.slots > kMaxWarps;
        const int teams = kMaxWarps / prm.teamWarps;
        size_t off = 0;
        auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 15) / 16 * 16; return (int32_t)at; };
        prm.offTeams = take(sizeof(Team) * (size_t)teams);
        prm.offCmd = take(8 * (size_t)prm.slots);
        prm.offBits = take((size_t)(maxLd + 31) / 32 * 4);
        prm.offLists = take(sizeof(Raised) * (size_t)(kMaxWarps * kRaisedPerWarp + teams));
        prm.offNotes = take(sizeof(Note) * (size_t)sz.W);
        prm.offBars = take(8 * (size_t)sz.W);
        prm.offRows = take(many ? 0 : (size_t)prm.slots * maxLd * 4);
        prm.offCover = take(state ? (size_t)prm.slots * maxLd * 4 : 0);
        prm.offKeys = take(state ? (size_t)prm.slots * maxLd * 8 : 0);
        return off;
    };
    // Cluster size: as many CTAs per class as there are blocks for and as all classes find room for at once; with more
    // classes than that, the fewest that keep the state on the chip.
    const int most = std::min(16, pow2_at_least(sz.W));
    int C = 0;
    for (int i = 4; i >= 0; --i) {
        const int size = 1 << i;
        if (ctx->maxClusters[i] == 0) {
            rcd_status rs = launch_cluster(ctx, pick_kernel<1>(true, false), prm, size, 1, cap, st, &ctx->maxClusters[i]);
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
    ClusterKernel kernel = sz.W <= 32 ? pick_kernel<1>(state, many) : sz.W <= 64 ? pick_kernel<2>(state, many) : pick_kernel<4>(state, many);
    const rcd_status rs = launch_cluster(ctx, kernel, prm, C, clusters, smem, st, nullptr);
    if (rs != RCD_OK) return rs;
    ctx->steps = sz.maxM;
    ctx->phaseNsDev = ws.phaseNs;
    return RCD_OK;
}

}  // namespace rcd
