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
#include <functional>

namespace rcd {

namespace {

constexpr int kMaxWarps = 16;             // team warps per CTA (one more warp leads in the cluster's first CTA)
constexpr int kMaxPieces = 5;             // pieces per thread of a team that keeps its block's gains in registers
constexpr int kRaisedPerWarp = 64;        // raised columns a team lists at a time, per warp
constexpr int kClusterBlocks = 128;       // blocks a cluster can lead (their notes sit in one CTA's shared memory)
constexpr int kEntries = 16;              // candidates per note
constexpr uint32_t kScanCmd = 0u;         // a command's low word: look again;
constexpr uint32_t kStopCmd = ~0u;        //   the class is done;  anything else: sample + 1 joins the block
constexpr unsigned kPollLimit = 1u << 25;
constexpr unsigned long long kZeroValue = 1ull << 55;   // (tracked values of the graph cut can be negative)

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
    int32_t rowPieces;         // 16-byte pieces of a team's row buffer
    unsigned long long *topGain;   // [L] zero at the start: largest gain for an empty block (graph cut: row sum of |S|)
    uint32_t one;              // the value 1, opaque to the compiler
    // byte offsets into dynamic shared memory
    int32_t offTeams, offLists, offRows, offCmd, offBits, offNotes, offBars, offCover, offGains;
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

// g - l (one multiply-add)
__device__ __forceinline__ unsigned long long take_off(unsigned long long g, int l)
{
    unsigned long long r;
    asm("mad.wide.s32 %0, %1, -1, %2;" : "=l"(r) : "r"(l), "l"(g));
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

// A row's contribution by one warp: sum_i max(0, S[v][i]), or for the graph cut sum_i S[v][i] and sum_i |S[v][i]|.
template <bool kCut>
__device__ __forceinline__ unsigned long long row_value(const int4 *row, int ld4, int lane, uint32_t one, unsigned long long &negative)
{
    unsigned long long acc = 0, neg = 0;
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
            if (kCut) {
                neg = add_wide(max(-x[u].x, 0), one, neg);
                neg = add_wide(max(-x[u].y, 0), one, neg);
                neg = add_wide(max(-x[u].z, 0), one, neg);
                neg = add_wide(max(-x[u].w, 0), one, neg);
            }
        }
    }
    negative = kCut ? warp_sum(neg) : 0ull;
    return warp_sum(acc);
}

// The team of a warp, and what it knows while it works on a class.
struct TeamView {
    const int4 *S4;            // the class's similarity matrix
    int ld4;
    int warpIn, lane, T, team; // warp inside the team
    Team *tm;
    Raised *list;              // columns the update in hand raised
    int4 *rowBuf;              // a sample's row, and the ring of correct_keys (each thread reads only the pieces it copied itself)
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

// The leading candidates among a thread's columns.  64-bit comparisons cost five instructions at half rate, so gains are
// compared by their leading 32 bits first (gain >> shift, with shift such that the block's largest gain fits) and, among
// equals, by their other bits and the sample number together: `shift` is at most 16.
struct Lead {
    uint32_t e, o;             // greatest and second-greatest gain >> shift (0: none, else + 1)
    uint32_t low;              // of those that have e: the greatest of (other bits of the gain << 16 | 65535 - sample)
};
__device__ __forceinline__ void lead_init(Lead &b) { b.e = b.o = b.low = 0; }
__device__ __forceinline__ uint32_t lead_part(unsigned long long g, int shift) { return (uint32_t)(g >> shift) + 1u; }
__device__ __forceinline__ uint32_t low_part(unsigned long long g, int shift, int v)
{
    return ((uint32_t)g & ((1u << shift) - 1u)) << 16 | (uint32_t)(65535 - v);
}
// (shift for gains up to g: gain >> shift stays below 2^31)
__device__ __forceinline__ int shift_for(unsigned long long g) { return max(0, 33 - __clzll((long long)g)); }

// A warp's part of a note: entries (one per tile of 2 T lanes, at the tile's first lane), a bound on every gain that is
// no entry, and the best of all, as keys.
struct Summary {
    unsigned long long entry, bound, top;
};
__device__ __forceinline__ unsigned long long key_of(uint32_t e, uint32_t low, int shift)
{
    if (e == 0) return 0ull;
    return ((((unsigned long long)(e - 1u)) << shift | (low >> 16)) << 16) | (low & 0xffffu);
}
__device__ __forceinline__ Summary summarize(Lead b, int shift, int T, int lane)
{
    Summary s;
    if (T <= 2) {
        for (int off = 1; off < 2 * T; off <<= 1) {
            const uint32_t e2 = __shfl_xor_sync(0xffffffffu, b.e, off), o2 = __shfl_xor_sync(0xffffffffu, b.o, off), l2 = __shfl_xor_sync(0xffffffffu, b.low, off);
            b.o = max(max(b.o, o2), min(b.e, e2));
            b.low = b.e > e2 ? b.low : (b.e < e2 ? l2 : max(b.low, l2));
            b.e = max(b.e, e2);
        }
        s.entry = key_of(b.e, b.low, shift);
        const uint32_t o = __reduce_max_sync(0xffffffffu, b.o);
        s.bound = o == 0 ? 0ull : key_of(o, (1u << shift) - 1u << 16 | 0xffffu, shift);
        const uint32_t m = __reduce_max_sync(0xffffffffu, b.e);
        s.top = key_of(m, __reduce_max_sync(0xffffffffu, b.e == m ? b.low : 0u), shift);
    } else {
        const int tile = 2 * T;
        const uint32_t mask = tile == 32 ? 0xffffffffu : ((1u << tile) - 1u) << (lane & ~(tile - 1));
        const uint32_t m = __reduce_max_sync(mask, b.e);
        const uint32_t low = __reduce_max_sync(mask, b.e == m ? b.low : 0u);
        s.entry = key_of(m, low, shift);
        const uint32_t o = __reduce_max_sync(0xffffffffu, b.e == m && b.low == low ? b.o : b.e);
        s.bound = o == 0 ? 0ull : key_of(o, (1u << shift) - 1u << 16 | 0xffffu, shift);
        s.top = s.entry;
        if (tile < 32) {
            const uint32_t m2 = __reduce_max_sync(0xffffffffu, b.e);
            s.top = key_of(m2, __reduce_max_sync(0xffffffffu, b.e == m2 ? b.low : 0u), shift);
        }
    }
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

// The n listed columns (an odd list is completed by an entry without effect) taken off the stored gains of a thread's
// pieces.  The rows of S travel through a ring of asynchronous copies in shared memory, each thread reading back only what
// it copied itself, two rows of one piece per step and kRing / 2 steps under way, across the ends of the list too: 80 KB
// in flight per SM cover the latency of L2 and HBM without holding registers.
constexpr int kRing = 10;
struct RowStream {
    int4 *ring;
    const int4 *S4;
    const Raised *list;
    int n, step, ld4;
    int fq, fe, fs, at;                                    // what is fetched next, and to which stage; the stage read next
    __device__ __forceinline__ void fetch()
    {
        if (fq < ld4) {
            copy16(ring + fs, S4 + (list[fe].row + fq));
            copy16(ring + fs + step, S4 + (list[fe + 1].row + fq));
            fe += 2;
            if (fe >= n) { fe = 0; fq += step; }
        }
        copies_commit();
        fs += 2 * step;
        if (fs == kRing * step) fs = 0;
    }
    __device__ __forceinline__ RowStream(const TeamView &t, int count)
    {
        const int first = t.warpIn * 32 + t.lane;
        step = t.T * 32;
        ring = t.rowBuf + first;
        S4 = t.S4; list = t.list; n = count; ld4 = t.ld4;
        fq = first; fe = 0; fs = 0; at = 0;
#pragma unroll 1
        for (int k = 0; k < kRing / 2 - 1; ++k) fetch();
    }
    // all n columns for the piece whose turn it is
    __device__ __forceinline__ int piece(unsigned long long (&g)[4])
    {
        int changed = 0;
#pragma unroll 1
        for (int e = 0; e < n; e += 2) {
            copies_wait<kRing / 2 - 2>();
            const int4 x = ring[at], y = ring[at + step];
            const Raised a = list[e], b = list[e + 1];
            at += 2 * step;
            if (at == kRing * step) at = 0;
            fetch();
            const int l0 = loss(x.x, a) + loss(y.x, b), l1 = loss(x.y, a) + loss(y.y, b);
            const int l2 = loss(x.z, a) + loss(y.z, b), l3 = loss(x.w, a) + loss(y.w, b);
            changed |= l0 | l1 | l2 | l3;
            g[0] = take_off(g[0], l0);
            g[1] = take_off(g[1], l1);
            g[2] = take_off(g[2], l2);
            g[3] = take_off(g[3], l3);
        }
        return changed;
    }
};

// Folds a sample's row into the coverage, list by list; `apply(n)` corrects the stored gains for the n listed columns.
template <typename Apply>
__device__ __forceinline__ void take_in_lists(const TeamView &t, int v, int4 *cov, unsigned &rows, Apply apply)
{
    const int tid = t.warpIn * 32 + t.lane, step = t.T * 32;
    const int room = t.T * kRaisedPerWarp;
    int32_t *count = &t.tm->count[2];
    const int4 *row = t.S4 + (int64_t)v * t.ld4;
    for (;;) {
        team_barrier(t.team, t.T);                         // (the list's last readers are done)
        if (tid == 0) *count = 0;
        team_barrier(t.team, t.T);
        for (int q = tid; q < t.ld4; q += step) {
            const int4 r = __ldg(row + q), m = cov[q];
            if (list_raised(t, count, q, r, m)) cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
        }
        team_barrier(t.team, t.T);
        const int all = *(volatile int32_t *)count;
        const int n = min(all, room);
        rows += n;
        if (tid == 0 && (n & 1)) t.list[n] = Raised{0, 0, 0, 0};
        team_barrier(t.team, t.T);
        if (n > 0) apply(n);
        if (all <= room) break;
    }
}

// A team with one block, its stored gains in registers: P pieces of four columns per thread.  Coverage in shared memory.
template <int P, bool kCut>
__device__ __forceinline__ void team_of_one(const ClusterParams &prm, const ClassDesc &c, const TeamView &t, int4 *cov, int shift, unsigned long long bias,
                                            uint32_t cmdAddr, uint32_t noteAddr, uint32_t barAddr, unsigned &corrected, unsigned &rows)
{
    const int T = t.T, tid = t.warpIn * 32 + t.lane, step = T * 32, lane = t.lane;
    const int room = T * kRaisedPerWarp;
    unsigned long long g[P][4];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int q = tid + p * step;
        if (!kCut && q < t.ld4) cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) g[p][u] = 4 * q + u < c.M ? (unsigned long long)__ldcg(prm.g0 + c.row0 + 4 * q + u) + bias : 0ull;
    }
    if (tid == 0) t.tm->count[0] = t.tm->count[1] = 0;
    Lead best;
    lead_init(best);
    Summary sum{0, 0, 0};
    bool dirty = true, newTop = false;
    uint32_t had = 0;
    for (int par = 0;; par ^= 1) {
        // candidates: a warp looks again when gains of its columns changed or one of its threads' best has been assigned
        if (!dirty && best.e) {
            const int s = 65535 - (int)(best.low & 0xffffu);
            dirty = t.bits[s >> 5] >> (s & 31) & 1;
        }
        if (__any_sync(0xffffffffu, dirty)) {
            lead_init(best);
            uint32_t nib[P];
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const int q = tid + p * step;
                nib[p] = q < t.ld4 ? t.bits[q >> 3] >> ((q & 7) * 4) : 15u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t k = (nib[p] >> u & 1) ? 0u : lead_part(g[p][u], shift);
                    best.o = max(best.o, min(best.e, k));
                    best.e = max(best.e, k);
                }
            }
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (lead_part(g[p][u], shift) == best.e && !(nib[p] >> u & 1)) best.low = max(best.low, low_part(g[p][u], shift, 4 * (tid + p * step) + u));
            const unsigned long long was = sum.top;
            sum = summarize(best, shift, T, lane);
            dirty = false;
            newTop = sum.top != was;
        }
        // the best of the team first: it is all the leader needs unless another block takes that sample
        unsigned long long top = sum.top;
        if (T > 1) {
            if (lane == 0) t.tm->best[t.warpIn] = top;
            team_barrier(t.team, T);
            top = warp_max_u64(lane < T ? t.tm->best[lane] : 0ull);
        }
        if (tid == 0) st_async(noteAddr, top, barAddr);
        post(t, sum, noteAddr, barAddr);
        // (the warp's best may be the block's best some picks from now: its row comes to L2 meanwhile)
        if (T > 1 && newTop && sum.top) {
            newTop = false;
            const char *row = reinterpret_cast<const char *>(t.S4 + (int64_t)key_sample(sum.top) * t.ld4);
            for (int at = lane * 128; at < t.ld4 * 16; at += 32 * 128) asm volatile("prefetch.global.L2 [%0];" :: "l"(row + at));
        }
        // until the command comes: the row of the best candidate, which is, as a rule, the sample the block receives
        // next, and the columns it would raise
        int v = top ? key_sample(top) : -1;
        int32_t *count = &t.tm->count[par];
        int all = 0;
        if (v >= 0) {
            fetch_row(t, v);
            copies_wait<0>();
            if (!kCut) {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const int q = tid + p * step;
                    if (q < t.ld4) list_raised(t, count, q, t.rowBuf[q], cov[q]);
                }
                team_barrier(t.team, T);
                all = *(volatile int32_t *)count;
                if (all & 1) {                             // (an entry without effect completes the last pair)
                    if (tid == 0 && all < room) t.list[all] = Raised{0, 0, 0, 0};
                    team_barrier(t.team, T);
                }
            }
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
        if (!kCut) shift = min(shift, shift_for(top >> 16));         // (gains only fall)
        if (kCut) {
            // gain = column sum - twice the tie to the block: the sample's row is the tie's growth
            const bool foreseen = (int)what - 1 == v;
            const int4 *row = t.S4 + (int64_t)((int)what - 1) * t.ld4;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const int q = tid + p * step;
                if (q < t.ld4) {
                    const int4 r = foreseen ? t.rowBuf[q] : __ldg(row + q);
                    g[p][0] = take_off(g[p][0], 2 * r.x);
                    g[p][1] = take_off(g[p][1], 2 * r.y);
                    g[p][2] = take_off(g[p][2], 2 * r.z);
                    g[p][3] = take_off(g[p][3], 2 * r.w);
                }
            }
            dirty = true;
            continue;
        }
        auto apply = [&](int n) {
            RowStream rs(t, n);
            int changed = 0;
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (tid + p * step < t.ld4) changed |= rs.piece(g[p]);
            copies_wait<0>();
            dirty = dirty || changed != 0;
        };
        if ((int)what - 1 != v || all > room) {
            // another sample than foreseen, or more raised columns than one list holds
            take_in_lists(t, (int)what - 1, cov, rows, apply);
            continue;
        }
        rows += all;
        if (all == 0) continue;
        const bool own = all == 1 && t.list[0].row == v * t.ld4;         // (most picks: the sample itself is all that rose)
        const Raised mine = t.list[0];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int q = tid + p * step;
            if (q < t.ld4) {
                const int4 r = t.rowBuf[q], m = cov[q];
                if (r.x > m.x || r.y > m.y || r.z > m.z || r.w > m.w) cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
                if (own) {
                    const int l0 = loss(r.x, mine), l1 = loss(r.y, mine), l2 = loss(r.z, mine), l3 = loss(r.w, mine);
                    if (l0 | l1 | l2 | l3) {
                        dirty = true;
                        g[p][0] = take_off(g[p][0], l0);
                        g[p][1] = take_off(g[p][1], l1);
                        g[p][2] = take_off(g[p][2], l2);
                        g[p][3] = take_off(g[p][3], l3);
                    }
                }
            }
        }
        if (!own) apply(all);
    }
    copies_wait<0>();
}

// A one-warp team with several blocks (coverage and gains in memory): it serves whichever has a command.
template <typename Where>
__device__ __forceinline__ void team_of_many(const ClusterParams &prm, int l, const ClassDesc &c, const TeamView &t, int mine, int shift, uint32_t cmd0,
                                             int cmdStride, Where where, unsigned &corrected, unsigned &rows)
{
    const int lane = t.lane;
    int4 *cov;
    unsigned long long *gains;
    uint32_t noteAddr, barAddr;
    auto tell = [&] {
        Lead best;
        lead_init(best);
        unsigned long long at = 0;
        for (int q = lane; q < t.ld4; q += 32) {
            const uint32_t nib = t.bits[q >> 3] >> ((q & 7) * 4);
            const ulonglong2 a0 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q], a1 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q + 1];
            const unsigned long long g[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t k = (nib >> u & 1) ? 0u : lead_part(g[u], shift);
                best.o = max(best.o, min(best.e, k));
                if (k >= best.e && k) {
                    const uint32_t low = low_part(g[u], shift, 4 * q + u);
                    best.low = k > best.e ? low : max(best.low, low);
                    best.e = k;
                }
            }
        }
        (void)at;
        const Summary sum = summarize(best, shift, 1, lane);
        post(t, sum, noteAddr, barAddr);
        if (lane == 0) st_async(noteAddr, sum.top, barAddr);
    };
    for (int i = 0; i < mine; ++i) {
        const int j = where(i, cov, gains, noteAddr, barAddr);
        for (int q = lane; q < t.ld4; q += 32) {
            cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) gains[4 * q + u] = 4 * q + u < c.M ? (unsigned long long)__ldcg(prm.g0 + c.row0 + 4 * q + u) : 0ull;
        }
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
        where(who, cov, gains, noteAddr, barAddr);
        if (what == kScanCmd) {
            cluster_fence();
        } else {
            ++corrected;
            take_in_lists(t, (int)what - 1, cov, rows, [&](int n) {
                RowStream rs(t, n);
#pragma unroll 1
                for (int q = lane; q < t.ld4; q += 32) {
                    ulonglong2 *p = reinterpret_cast<ulonglong2 *>(gains) + 2 * q;
                    const ulonglong2 k0 = p[0], k1 = p[1];
                    unsigned long long k[4] = {k0.x, k0.y, k1.x, k1.y};
                    if (rs.piece(k)) {
                        p[0] = make_ulonglong2(k[0], k[1]);
                        p[1] = make_ulonglong2(k[2], k[3]);
                    }
                }
                copies_wait<0>();
            });
        }
        __syncwarp();
        tell();
    }
}

// The leader's loop over the picks of class c.  One warp; lane p % 32 keeps the value and the room of block p, and the
// parity of the mbarrier on which the block's notes arrive (they go on from class to class).
template <int KW>
__device__ void lead(const ClusterParams &prm, int l, const ClassDesc &c, unsigned char *shared, uint32_t C, unsigned long long bias, uint32_t &parities)
{
    const int lane = threadIdx.x & 31, W = prm.W, T = prm.teamWarps;
    const uint32_t noteBytes = (1 + kEntries + T) * 8;
    const uint32_t base = smem32(shared);
    volatile uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    const uint32_t myBits = remote(base + prm.offBits, (uint32_t)lane < C ? lane : 0);
    volatile const Note *notes = reinterpret_cast<const Note *>(shared + prm.offNotes);
    const uint32_t bars = base + prm.offBars;
    unsigned long long f[KW];              // (value + kZeroValue) << 7 | block
    int room[KW];
    uint32_t seq[KW], cmdAddr[KW];
    uint32_t awaited = 0;                  // bit k: block lane + 32 k owes a note
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        f[k] = (kZeroValue << 7) | (unsigned long long)p;
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
    unsigned long long others = ~0ull, last = ~0ull;       // least of the blocks but the one picked last, and that one's
#pragma unroll
    for (int k = 0; k < KW; ++k) others = room[k] > 0 ? umin(others, f[k]) : others;
    others = ~warp_max_u64(~others);
    for (int t = 0; t < c.M; ++t) {
        const unsigned long long least = umin(others, last);
        if (least == ~0ull) {
            if (lane == 0) atomicOr(prm.status, kDevNoCandidate);
            ok = false;
            break;
        }
        const int j = (int)(least & 127);
        const int jk = KW == 1 ? 0 : j >> 5, jl = j & 31;
        const uint32_t state = __shfl_sync(0xffffffffu, awaited | parities << 16, jl) >> jk;
        uint32_t waits = state & 1, parity = state >> 16 & 1;
        // the least of the other blocks: known before this pick is made
        others = ~0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k) others = room[k] > 0 && lane + 32 * k != j ? umin(others, f[k]) : others;
        others = ~warp_max_u64(~others);
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
        last = least + (((best >> 16) - bias) << 7);
        int left = 0;
        if (lane == jl) {
#pragma unroll
            for (int k = 0; k < KW; ++k)
                if (k == jk) {
                    f[k] += ((best >> 16) - bias) << 7;
                    left = --room[k];
                    if (left > 0) {                   // (a full block needs no gains any more)
                        bar_expect(bars + j * 8, noteBytes);
                        awaited |= 1u << k;
                        st_remote(cmdAddr[k], ((unsigned long long)++seq[k] << 32) | (unsigned long long)(v + 1));
                    }
                }
        }
        if (__shfl_sync(0xffffffffu, left, jl) == 0) last = ~0ull;
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
            const long long value = (long long)(f[k] >> 7) - (long long)kZeroValue;
            prm.fval[(int64_t)l * W + p] = prm.fixedExp ? __double_as_longlong(ldexp((double)value, -prm.fixedExp[l])) : value;
        }
    }
    if (lane == 0 && rescans) atomicAdd(prm.stats + 9, (unsigned long long)rescans);
}

// P: pieces per thread of teams with one block; 0: teams of one warp with several blocks (kSmemState: which all fit the
// CTAs' shared memory).  kCut: graph-cut objective.
template <int KW, int P, bool kSmemState, bool kCut>
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
        if (warp < NW) {
            unsigned long long top = 0;
            for (int v = rank * NW + warp; v < c.M; v += C * NW) {
                unsigned long long neg;
                const unsigned long long pos = row_value<kCut>(S4 + (int64_t)v * ld4, ld4, lane, prm.one, neg);
                top = umax(top, pos + neg);
                if (lane == 0) __stcg(prm.g0 + c.row0 + v, (long long)(pos - neg) - (kCut ? (long long)prm.S[c.sOff + (int64_t)v * c.ld + v] : 0ll));
            }
            if (lane == 0 && top) atomicMax(prm.topGain + l, top);
        }
        for (int i = threadIdx.x; i < (c.ld + 31) / 32; i += blockDim.x)
            bits[i] = 32 * i + 32 <= c.M ? 0u : (32 * i >= c.M ? ~0u : ~0u << (c.M - 32 * i));
        for (int i = threadIdx.x; i < prm.slots; i += blockDim.x) cmds[i] = 0;
        cluster_barrier();
        // graph cut: gains lie within three times the largest sum of |S| over a row, either way
        const unsigned long long top = __ldcg(prm.topGain + l);
        const unsigned long long bias = kCut ? 3 * top + 1 : 0ull;
        const int shift = shift_for(bias + (kCut ? 3 : 1) * top);

        if (warp == NW) {
            if (rank == 0) lead<KW>(prm, l, c, shared, C, bias, parities);
        } else {
            const int team = warp / T;
            TeamView t;
            t.S4 = S4; t.ld4 = ld4;
            t.warpIn = warp - team * T; t.lane = lane; t.T = T; t.team = team;
            t.tm = reinterpret_cast<Team *>(shared + prm.offTeams) + team;
            t.list = reinterpret_cast<Raised *>(shared + prm.offLists) + team * (T * kRaisedPerWarp + 1);
            t.rowBuf = reinterpret_cast<int4 *>(shared + prm.offRows) + (size_t)team * prm.rowPieces;
            t.bits = bits;
            unsigned corrected = 0, rows = 0;
            const uint32_t notes0 = remote(base + prm.offNotes, 0), bars0 = remote(base + prm.offBars, 0);
            if (P > 0) {
                const int j = team * (int)C + (int)rank;
                if (team < prm.slots && j < W && prm.quota[(int64_t)l * W + j] > 0)
                    team_of_one<(P > 0 ? P : 1), kCut>(prm, c, t, reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)team * (prm.maxLd >> 2), shift, bias,
                                                       base + prm.offCmd + team * 8, notes0 + j * (uint32_t)sizeof(Note), bars0 + j * 8, corrected, rows);
            } else {
                // the i-th block of the team
                auto where = [&](int i, int4 *&cov, unsigned long long *&gains, uint32_t &noteAddr, uint32_t &barAddr) -> int {
                    const int slot = team + i * nTeams, j = slot * (int)C + (int)rank;
                    if (kSmemState) {
                        cov = reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)slot * (prm.maxLd >> 2);
                        gains = reinterpret_cast<unsigned long long *>(shared + prm.offGains) + (size_t)slot * prm.maxLd;
                    } else {
                        cov = reinterpret_cast<int4 *>(prm.cover + c.vOff) + (size_t)j * ld4;
                        gains = reinterpret_cast<unsigned long long *>(prm.gains + c.vOff) + (size_t)j * c.ld;
                    }
                    noteAddr = notes0 + j * (uint32_t)sizeof(Note);
                    barAddr = bars0 + j * 8;
                    return j;
                };
                int mine = 0;
                while (team + mine * nTeams < prm.slots && (team + mine * nTeams) * (int)C + (int)rank < W) ++mine;
                if (mine > 0) team_of_many(prm, l, c, t, mine, shift, base + prm.offCmd + team * 8, nTeams * 8, where, corrected, rows);
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

template <int KW, bool kCut>
static ClusterKernel pick_kernel(int P, bool smemState)
{
    if (P == 1) return greedy_cluster_kernel<KW, 1, true, kCut>;
    if (P == 2) return greedy_cluster_kernel<KW, 2, true, kCut>;
    if (P == 3) return greedy_cluster_kernel<KW, 3, true, kCut>;
    if (P > 0 && P <= 4) return greedy_cluster_kernel<KW, 4, true, kCut>;
    if (P > 0) return greedy_cluster_kernel<KW, kMaxPieces, true, kCut>;
    return smemState ? greedy_cluster_kernel<KW, 0, true, false> : greedy_cluster_kernel<KW, 0, false, false>;
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

// How a problem is laid out over clusters.
struct ClusterPlan {
    int C, clusters, P;        // CTAs per cluster, clusters, pieces per thread (0: several blocks per warp)
    bool smemState;
    size_t smem;
    ClusterParams prm;         // teamWarps, slots, maxLd, rowPieces and the offsets are set
};
static size_t cluster_layout(const Sizes &sz, int maxLd, int C, bool state, ClusterPlan &plan)
{
    ClusterParams &prm = plan.prm;
    prm.warps = kMaxWarps;
    prm.maxLd = maxLd;
    prm.slots = (sz.W + C - 1) / C;
    // a team per block, of as many warps as a row has work for
    const int most = kMaxWarps / std::min(kMaxWarps, pow2_at_least(prm.slots));
    prm.teamWarps = std::min(most, pow2_at_least((maxLd / 4 + 31) / 32));
    const int step = prm.teamWarps * 32, teams = kMaxWarps / prm.teamWarps;
    plan.P = prm.slots > kMaxWarps ? 0 : (maxLd / 4 + step - 1) / step;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 15) / 16 * 16; return (int32_t)at; };
    prm.offTeams = take(sizeof(Team) * (size_t)teams);
    prm.offCmd = take(8 * (size_t)prm.slots);
    prm.offBits = take((size_t)(maxLd + 31) / 32 * 4);
    prm.offLists = take(sizeof(Raised) * (size_t)(kMaxWarps * kRaisedPerWarp + teams));
    prm.offNotes = take(sizeof(Note) * (size_t)sz.W);
    prm.offBars = take(8 * (size_t)sz.W);
    prm.rowPieces = std::max(kRing, plan.P) * step;
    prm.offRows = take((size_t)std::min(teams, prm.slots) * prm.rowPieces * 16);
    prm.offCover = take(plan.P > 0 || state ? (size_t)prm.slots * maxLd * 4 : 0);
    prm.offGains = take(plan.P == 0 && state ? (size_t)prm.slots * maxLd * 8 : 0);
    return off;
}

// Whether the cluster form takes a problem, and how: chosen by the library (no pass-based form or option asked for),
// samples of a class and blocks within the packed keys' range, blocks that fit registers or shared memory.
static bool cluster_plan(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, ClusterPlan &plan)
{
    const rcd_config &c = ctx->cfg;
    if (c.greedy_path != 0 || c.profile >= 2 || c.sweep_batch_max != 0 || c.sweep_mode != 0 || c.async_group != 0 || c.async_help_min != 0 ||
        c.threshold_from != 0 || c.threshold_hit_shift != 0 || c.lazy_mode != 0 || c.lazy_from != 0 || c.dense_ring != 0 ||
        c.incremental != 0 || c.incremental_max != 0)
        return false;
    if (sz.W > kClusterBlocks || sz.maxM > 65535 || sz.d > 65535 || sz.L > 65535 || sz.maxM == 0) return false;
    if (sz.graphCut && (sz.floatArith || sz.maxM > 8192)) return false;
    int nonEmpty = 0, maxLd = 8;
    for (const ClassDesc &d : descHost) {
        if (d.M > 0) ++nonEmpty;
        maxLd = std::max(maxLd, (int)d.ld);
    }
    const size_t cap = (size_t)ctx->maxSmemOptin - 1024;
    plan.prm = ClusterParams{};
    for (int i = 0; i < 5; ++i)
        if (ctx->maxClusters[i] == 0) {
            plan.prm.warps = kMaxWarps;
            if (launch_cluster(ctx, pick_kernel<1, false>(3, true), plan.prm, 1 << i, 1, cap, nullptr, &ctx->maxClusters[i]) != RCD_OK) return false;
        }
    // Cluster size: the one whose clusters, drawing classes largest first, finish soonest by the estimate that a class of
    // M samples takes M (M / C + 300) (corrections, shared by the CTAs, and the chain of picks); blocks have to stay on
    // the chip.
    const int most = std::min(16, pow2_at_least(sz.W));
    std::vector<int> sizes;
    for (const ClassDesc &d : descHost) if (d.M > 0) sizes.push_back(d.M);
    std::sort(sizes.begin(), sizes.end(), std::greater<int>());
    double bestTime = 0;
    plan.C = 0;
    for (int i = 0; (1 << i) <= most; ++i) {
        const int C = 1 << i, n = ctx->maxClusters[i];
        if (n < 1) continue;
        const size_t smem = cluster_layout(sz, maxLd, C, true, plan);
        if (smem > cap || plan.P > kMaxPieces || (sz.graphCut && plan.P == 0)) continue;
        double time = 0;
        std::vector<double> busy((size_t)std::min<size_t>((size_t)n, sizes.size()), 0.0);      // (a heap of the clusters' finishing times)
        for (int M : sizes) {
            std::pop_heap(busy.begin(), busy.end(), std::greater<double>());
            busy.back() += (double)M * ((double)M / C + 300.0);
            time = std::max(time, busy.back());
            std::push_heap(busy.begin(), busy.end(), std::greater<double>());
        }
        if (plan.C == 0 || time < bestTime) { plan.C = C; bestTime = time; }
    }
    if (plan.C > 0) {
        plan.smem = cluster_layout(sz, maxLd, plan.C, true, plan);
        plan.smemState = true;
    } else {
        // several blocks per warp, in global memory
        plan.C = 1;
        plan.smem = cluster_layout(sz, maxLd, plan.C, false, plan);
        plan.smemState = false;
        if (plan.P > 0 || plan.smem > cap) return false;
    }
    if (sz.graphCut && plan.P == 0) return false;
    int idx = 0;
    while ((1 << idx) < plan.C) ++idx;
    if (ctx->maxClusters[idx] < 1) return false;
    plan.clusters = std::max(1, std::min(nonEmpty, ctx->maxClusters[idx]));
    return true;
}

// Runs the greedy loop if the cluster form takes the problem (*taken).  partValues (may be null) receives the tracked values.
rcd_status launch_greedy_cluster(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                 int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st, bool *taken)
{
    ClusterPlan plan;
    *taken = cluster_plan(ctx, sz, descHost, plan);
    if (!*taken) return RCD_OK;
    ClusterParams &prm = plan.prm;
    prm.desc = ws.desc;
    prm.S = (const int32_t *)ws.S;
    prm.cover = (int32_t *)ws.cover;
    prm.gains = (long long *)ws.gains;
    prm.g0 = ws.g0;
    prm.topGain = ws.topGain;
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
    prm.L = sz.L;
    prm.W = sz.W;
    prm.one = 1u;
    if (sz.floatArith) {
        fixed_exponent_kernel<<<sz.L, 256, 0, st>>>(ws.desc, (const float *)ws.S, ws.fixedExp);
        const int64_t pieces = sz.maxM * (int64_t)(prm.maxLd / 4);
        const dim3 grid((unsigned)std::min<int64_t>((pieces + 1023) / 1024, std::max(1, 16 * ctx->smCount / sz.L)), (unsigned)sz.L);
        fixed_point_kernel<<<grid, 256, 0, st>>>(ws.desc, ws.fixedExp, (float *)ws.S);
        ctx->kernelLaunches += 2;
        RCD_CUDA(ctx, cudaGetLastError());
    }
    ClusterKernel kernel = sz.graphCut ? (sz.W <= 32 ? pick_kernel<1, true>(plan.P, plan.smemState) : pick_kernel<4, true>(plan.P, plan.smemState))
                                       : (sz.W <= 32 ? pick_kernel<1, false>(plan.P, plan.smemState) : pick_kernel<4, false>(plan.P, plan.smemState));
    const rcd_status rs = launch_cluster(ctx, kernel, prm, plan.C, plan.clusters, plan.smem, st, nullptr);
    if (rs != RCD_OK) return rs;
    ctx->steps = sz.maxM;
    ctx->phaseNsDev = ws.phaseNs;
    return RCD_OK;
}

}  // namespace rcd
