// The greedy loop of Algorithm 1 with the facility-location objective, one thread-block cluster per class: the form
// the library chooses by itself, except where classes run in rounds (rcd_rounds.cu: enough classes to fill the SMs one by one,
// and many blocks).  The pass-based forms of rcd_greedy.cu serve explicit configurations.
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
#include "rcd_cut_plan.h"
#include "rcd_exact.cuh"

#include <limits.h>
#include <algorithm>
#include <functional>

namespace rcd {

namespace {

constexpr int kMaxWarps = 16;             // team warps per CTA; one more warp leads in the cluster's first CTA
// One block per CTA and long rows: a team of 15 warps, so that with the leader there are 16 and a thread may hold 128
// registers (17 warps get the share of 20: 96).
__host__ __device__ constexpr int team_warps(int T) { return T == 15 ? 15 : kMaxWarps; }
constexpr int kMaxPieces = 7;             // pieces per thread of a team that keeps its block's gains in registers
constexpr int kRaisedPerWarp = 64;        // raised columns a team lists at a time, per warp
constexpr int kClusterBlocks = 128;       // blocks a cluster can lead (their notes sit in one CTA's shared memory)
constexpr uint32_t kScanCmd = 0u;         // a command's low word: look again;
constexpr uint32_t kStopCmd = 0xfffffu;   //   the class is done;  anything else: sample + 1 joins the block
constexpr int kListers = 3;               // listing warps per CTA (17 warps would occupy the registers of 20 anyway)
constexpr unsigned kPollLimit = 1u << 28;

// Candidates a warp of a team of T contributes to a note: a power of two, at most 16 in all.
__host__ __device__ constexpr int entries_per_warp(int T) { return T <= 1 ? 16 : T <= 2 ? 8 : T <= 4 ? 4 : T <= 8 ? 2 : 1; }

// What the leader is told about a block (a note, words of 64 bits):
//   [0]            the key of its best candidate (0: none)
// and for the case that other blocks took that one (E = candidates per warp):
//   [1, 1 + TE)    keys of leading candidates
//   then T words   per team warp a key that no candidate left out exceeds
// and, where teams have several blocks, from a listing warp, some thousand cycles later (with many blocks the best candidates
// are often taken before the block's turn comes):
//   64 words       keys of leading candidates
//   1 word         a key that no candidate left out exceeds
//   1 word         number of the command that the list answers << 16 | number of the list, 0 while the list is being written
struct NoteLayout {
    int T;
    bool many;
    static constexpr int kList = 64;
    __host__ __device__ int entries() const { return T * entries_per_warp(T); }
    __host__ __device__ int list() const { return 1 + entries() + T; }
    __host__ __device__ int words() const { return list() + (many ? kList + 2 : 0); }
    __host__ __device__ uint32_t tracked() const { return (uint32_t)(1 + entries() + T) * 8; }   // bytes a new note brings
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
    int32_t teamWarps;         // T
    int32_t slots;             // blocks per CTA at most
    int32_t maxLd;
    int32_t rowPieces;         // 16-byte pieces of a team's row buffer
    unsigned long long *topGain;   // [L] zero at the start: largest gain for an empty block (graph cut: row sum of |S|)
    uint32_t one;              // the value 1, opaque to the compiler
    int32_t logC;
    // byte offsets into dynamic shared memory
    int32_t offTeams, offLists, offRows, offCmd, offBits, offNotes, offBars, offQueue, offTold, offListed, offFirsts, offCover, offGains;
    int32_t ring;              // command words per team (a power of two)
};

namespace {
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
// What the thread reads from the cluster's shared memory after this is not read before it.  Only that: a fence of both
// directions waits for the thread's own stores to other CTAs, and an acquire at cluster scope without the restriction drops the
// SM's L1 lines, which hold rows that several teams read (1000 classes of 1300 into 64 blocks: lists of candidates read with
// ld.acquire 166.8 ms, with this fence 165.0; 10 of 5000 with the graph cut, whose teams are told to look again often: their
// fence of both directions 9.58 ms, this one 8.84).
__device__ __forceinline__ void shared_acquire_fence() { asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory"); }
__device__ __forceinline__ uint32_t ld_acquire_block(uint32_t addr)          // (own shared memory, written by this CTA)
{
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// What the thread has written, or seen written, comes before what it writes after this.
__device__ __forceinline__ void release_fence() { asm volatile("fence.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
// (orders nothing by itself)
__device__ __forceinline__ bool bar_done(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
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

// g - l (one multiply-add)
__device__ __forceinline__ unsigned long long take_off(unsigned long long g, int l)
{
    unsigned long long r;
    asm("mad.wide.s32 %0, %1, -1, %2;" : "=l"(r) : "r"(l), "l"(g));
    return r;
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

// Starts copying the team's pieces of row v into its row buffer.
__device__ __forceinline__ void fetch_row(const TeamView &t, int v)
{
    const int4 *row = t.S4 + (int64_t)v * t.ld4;
    for (int q = t.warpIn * 32 + t.lane; q < t.ld4; q += t.T * 32) copy16(t.rowBuf + q, row + q);
    copies_commit();
}

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

// A warp's part of a note: entries (one per tile of 32 / E lanes, at the tile's first lane), a bound on every gain that is
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
    const int tile = 32 / entries_per_warp(T);
    if (tile <= 4) {
        for (int off = 1; off < tile; off <<= 1) {
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
__device__ __forceinline__ void post(const TeamView &t, int T, const Summary &s, uint32_t noteAddr, uint32_t barAddr)
{
    const int E = entries_per_warp(T), tile = 32 / E;
    if ((t.lane & (tile - 1)) == 0) st_async(noteAddr + (uint32_t)(1 + t.warpIn * E + t.lane / tile) * 8, s.entry, barAddr);
    if (t.lane == 1) st_async(noteAddr + (uint32_t)(1 + T * E + t.warpIn) * 8, s.bound, barAddr);
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

// Four listed columns taken off the stored gains of one piece.  Their losses (each below 2^30) add up in 32 bits, so that
// widening and subtracting is paid once for four.
__device__ __forceinline__ uint32_t apply_four(const int4 &x, const int4 &y, const int4 &z, const int4 &w, const Raised &a, const Raised &b,
                                               const Raised &c, const Raised &d, unsigned long long (&g)[4])
{
    const uint32_t l0 = (uint32_t)loss(x.x, a) + loss(y.x, b) + loss(z.x, c) + loss(w.x, d);
    const uint32_t l1 = (uint32_t)loss(x.y, a) + loss(y.y, b) + loss(z.y, c) + loss(w.y, d);
    const uint32_t l2 = (uint32_t)loss(x.z, a) + loss(y.z, b) + loss(z.z, c) + loss(w.z, d);
    const uint32_t l3 = (uint32_t)loss(x.w, a) + loss(y.w, b) + loss(z.w, c) + loss(w.w, d);
    g[0] -= l0;
    g[1] -= l1;
    g[2] -= l2;
    g[3] -= l3;
    return l0 | l1 | l2 | l3;
}
// (entry e of n, or one without effect)
__device__ __forceinline__ Raised entry_or_none(const Raised *list, int e, int n)
{
    Raised r = list[min(e, n - 1)];
    if (e >= n) r.minusOld = r.by = 0;
    return r;
}

// The n listed columns taken off one piece, rows straight to registers, up to sixteen in flight: sixteen warps of an SM then
// cover the trip to L2 or HBM (1000 classes of 1300 into 64 blocks, 148 SMs: 895 GB of rows in 162 ms, 0.85 of the copy
// bandwidth; 100 of 500 into 32 blocks, S in L2: 6.9 GB to the SMs in 1.39 ms).
__device__ __forceinline__ bool correct_piece(const int4 *S4q, const Raised *list, int n, unsigned long long (&g)[4])
{
    uint32_t changed = 0;
    int e = 0;
#pragma unroll 1
    for (; e + 16 <= n; e += 16) {
        int4 x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = ld_row_shared(S4q + list[e + u].row);
#pragma unroll
        for (int u = 0; u < 16; u += 4) changed |= apply_four(x[u], x[u + 1], x[u + 2], x[u + 3], list[e + u], list[e + u + 1], list[e + u + 2], list[e + u + 3], g);
    }
#pragma unroll 1
    for (; e + 8 <= n; e += 8) {
        int4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = ld_row_shared(S4q + list[e + u].row);
        changed |= apply_four(x[0], x[1], x[2], x[3], list[e], list[e + 1], list[e + 2], list[e + 3], g);
        changed |= apply_four(x[4], x[5], x[6], x[7], list[e + 4], list[e + 5], list[e + 6], list[e + 7], g);
    }
#pragma unroll 1
    for (; e < n; e += 4) {
        Raised r[4];
        int4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            r[u] = entry_or_none(list, e + u, n);
            x[u] = ld_row_shared(S4q + r[u].row);
        }
        changed |= apply_four(x[0], x[1], x[2], x[3], r[0], r[1], r[2], r[3], g);
    }
    return changed != 0;
}

// The same for a team that keeps its P pieces per thread in registers.  The rows travel through asynchronous copies in
// shared memory, each thread reading back only what it copied itself, so that loads in flight hold no registers.
// Up to three pieces: row by row over all pieces (a list entry and a row's address serve them all), eight rows of room,
// four under way while four are applied (10 classes of 5000 into 8 blocks, 80 SMs: 20.5 GB to the SMs in 7.5 ms, of which the
// first thousand picks of a class draw most).  More pieces, or less room: piece by piece through a ring of sixteen 16-byte
// slots per thread, twelve under way.
template <int P> struct RowRing { static constexpr bool byRow = P <= 3; };
constexpr int kRowStages = 8, kPieceStages = 16;
template <int P, int kT>
__device__ __forceinline__ void apply_list(const TeamView &t, int n, unsigned long long (&g)[P][4])
{
    const int first = t.warpIn * 32 + t.lane, step = (kT ? kT : t.T) * 32;
    int4 *const ring = t.rowBuf + first;
    const Raised *list = t.list;
    if constexpr (RowRing<P>::byRow) {
        const int stride = t.ld4;
        int fe = 0, fs = 0, at = 0;
        auto fetch = [&] {                                 // four rows
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (fe + u < n) {
                    const int4 *src = t.S4 + (list[fe + u].row + first);
#pragma unroll
                    for (int p = 0; p < P; ++p)
                        if (p * step + first < t.ld4) copy16(ring + fs + u * stride + p * step, src + p * step);
                }
            }
            copies_commit();
            fe += 4;
            fs = fs == 0 ? 4 * stride : 0;
        };
        fetch();
#pragma unroll 1
        for (int e = 0; e < n; e += 4) {
            fetch();
            copies_wait<1>();
            const int4 *x = ring + at;
            at = at == 0 ? 4 * stride : 0;
            Raised r[4];
            if (e + 4 <= n) {
#pragma unroll
                for (int u = 0; u < 4; ++u) r[u] = list[e + u];
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) r[u] = entry_or_none(list, e + u, n);
            }
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (p * step + first < t.ld4)
                    apply_four(x[p * step], x[p * step + stride], x[p * step + 2 * stride], x[p * step + 3 * stride], r[0], r[1], r[2], r[3], g[p]);
        }
    } else {
        int fq = first, fe = 0, fs = 0, at = 0;
        auto fetch = [&] {                                 // one piece of four rows
            if (fq < t.ld4) {
                const int4 *src = t.S4 + fq;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (fe + u < n) copy16(ring + (fs + u) * step, src + list[fe + u].row);
                fe += 4;
                if (fe >= n) { fe = 0; fq += step; }
            }
            copies_commit();
            fs += 4;
            if (fs == kPieceStages) fs = 0;
        };
        fetch();
        fetch();
        fetch();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (p * step + first < t.ld4) {
#pragma unroll 1
                for (int e = 0; e < n; e += 4) {
                    copies_wait<2>();
                    const int4 *x = ring + at * step;
                    at += 4;
                    if (at == kPieceStages) at = 0;
                    const int4 x0 = x[0], x1 = x[step], x2 = x[2 * step], x3 = x[3 * step];
                    fetch();
                    if (e + 4 <= n) {
                        apply_four(x0, x1, x2, x3, list[e], list[e + 1], list[e + 2], list[e + 3], g[p]);
                    } else {
                        Raised r[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) r[u] = entry_or_none(list, e + u, n);
                        apply_four(x0, x1, x2, x3, r[0], r[1], r[2], r[3], g[p]);
                    }
                }
            }
        }
    }
    copies_wait<0>();
}

// Folds a sample's row into the coverage, list by list; `apply(n)` corrects the stored gains for the n listed columns.
// `par`: which of two list lengths is in use (the other one is zero).
template <typename Apply>
__device__ __forceinline__ void take_in_lists(const TeamView &t, int v, int4 *cov, int32_t *counts, int &par, unsigned &rows, Apply apply)
{
    const int tid = t.warpIn * 32 + t.lane, step = t.T * 32;
    const int room = t.T * kRaisedPerWarp;
    const int4 *row = t.S4 + (int64_t)v * t.ld4;
    for (;;) {
        team_barrier(t.team, t.T);                         // (the list's last readers are done)
        int32_t *count = counts + par;
        for (int q = tid; q < t.ld4; q += step) {
            const int4 r = __ldg(row + q), m = cov[q];
            if (list_raised(t, count, q, r, m)) cov[q] = make_int4(max(r.x, m.x), max(r.y, m.y), max(r.z, m.z), max(r.w, m.w));
        }
        team_barrier(t.team, t.T);
        const int all = *(volatile int32_t *)count;
        par ^= 1;
        if (tid == 0) counts[par] = 0;
        const int n = min(all, room);
        rows += n;
        if (n > 0) apply(n);
        if (all <= room) break;
    }
}

// A team with one block, its stored gains in registers: P pieces of four columns per thread.  Coverage in shared memory.
// kT: warps per team (0: known at run time; a constant saves registers and address arithmetic).
template <int P, int kT, bool kCut>
__device__ __forceinline__ void team_of_one(const ClusterParams &prm, const ClassDesc &c, const TeamView &t, int4 *cov, int shift, unsigned long long bias,
                                            uint32_t cmdAddr, uint32_t noteAddr, uint32_t barAddr, unsigned &corrected, unsigned &rows)
{
    const int T = kT ? kT : t.T, tid = t.warpIn * 32 + t.lane, step = T * 32, lane = t.lane;
    const int room = T * kRaisedPerWarp;
    unsigned long long g[P][4];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int q = tid + p * step;
        if (!kCut && q < t.ld4) cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) g[p][u] = 4 * q + u < c.M ? (unsigned long long)__ldcg(prm.g0 + c.row0 + 4 * q + u) + bias : 0ull;
    }
    if (tid == 0) t.tm->count[0] = t.tm->count[1] = t.tm->count[2] = t.tm->count[3] = 0;
    int other = 0;
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
        post(t, T, sum, noteAddr, barAddr);
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
            shared_acquire_fence();
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
            // (nothing about candidates is kept meanwhile)
            lead_init(best);
            sum = Summary{0, 0, 0};
            dirty = true;
            apply_list<P, kT>(t, n, g);
        };
        if ((int)what - 1 != v || all > room) {
            // another sample than foreseen, or more raised columns than one list holds
            take_in_lists(t, (int)what - 1, cov, t.tm->count + 2, other, rows, apply);
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

// The leading candidates among a thread's pieces of a block's stored gains.
__device__ __forceinline__ Lead scan_gains(const uint32_t *bits, const unsigned long long *gains, int ld4, int first, int step, int shift)
{
    Lead best;
    lead_init(best);
    for (int q = first; q < ld4; q += step) {
        const uint32_t nib = bits[q >> 3] >> ((q & 7) * 4);
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
    return best;
}

// What a listing warp remembers of a block's list: per lane the two gains >> shift (+ 1) it listed, and whose they are.
struct Listed {
    uint32_t lead[NoteLayout::kList];
    uint16_t sample[NoteLayout::kList];
    uint32_t bound;
    uint32_t pad_;
};

// A listing warp serves the CTA's blocks first, first + step, ...  When a team has told the leader a block's best candidate
// (serial: number of the command that this answers), the warp lists the leading candidates, the two best of every lane;
// when other blocks have taken all but a few of those, it lists anew.
// From the moment a team writes its serial the stored gains are those of that command, until the leader has given the block
// another one -- and then it does not use lists of the earlier one any more, so a scan that ran into the next update
// does no harm.
template <typename Slot>
__device__ void list_candidates(const ClusterParams &prm, const uint32_t *bits, int ld4, int shift, uint32_t serials, Listed *listed, int first,
                                int step, int slots, const volatile uint32_t *ended, uint32_t turn, Slot where)
{
    const int lane = threadIdx.x & 31;
    const NoteLayout layout{prm.teamWarps, true};
    uint32_t had = 0, lists = 0;                           // lane i: of block first + i step: command listed last, and how often
    int turnOf = 0;
    const int mine = first < slots ? (slots - first + step - 1) / step : 0;
    for (unsigned spin = 0; spin < kPollLimit; ++spin) {
        if (*ended == turn) break;
        // a block told anew comes first; else a look at one block's list
        const uint32_t now = lane < mine ? ld_acquire_block(serials + (first + lane * step) * 4) : 0u;
        const unsigned m = __ballot_sync(0xffffffffu, now != had && now != 0);
        const bool fresh = m != 0;
        if (!fresh) turnOf = turnOf + 1 < mine ? turnOf + 1 : 0;
        const int i = fresh ? __ffs(m) - 1 : turnOf;
        const int slot = first + i * step;
        const uint32_t serial = __shfl_sync(0xffffffffu, now, i);
        if (mine == 0 || serial == 0) { __nanosleep(200); continue; }
        __syncwarp();                                      // (what the lane that read the serial sees, the warp sees)
        Listed &li = listed[slot];
        {
            if (!fresh) {
                // how many of the listed are left that are sure to lead?
                const uint32_t bound = li.bound;
                const int s0 = li.sample[lane], s1 = li.sample[32 + lane];
                const bool taken0 = *(volatile const uint32_t *)&bits[s0 >> 5] >> (s0 & 31) & 1, taken1 = *(volatile const uint32_t *)&bits[s1 >> 5] >> (s1 & 31) & 1;
                const unsigned sure = __popc(__ballot_sync(0xffffffffu, li.lead[lane] > bound && !taken0)) + __popc(__ballot_sync(0xffffffffu, li.lead[32 + lane] > bound && !taken1));
                const bool any = __any_sync(0xffffffffu, (li.lead[lane] && taken0) || (li.lead[32 + lane] && taken1));
                if (bound == 0 || sure > 2 || !any) {
                    __nanosleep(50);                       // (the teams need the issue slots)
                    continue;
                }
            }
            const unsigned long long *gains;
            const uint32_t listAddr = where(slot, gains) + (uint32_t)layout.list() * 8;
            if (lane == i) {
                st_remote(listAddr + (uint32_t)(NoteLayout::kList + 1) * 8, 0ull);
                lists = fresh ? 1 : lists + 1;
                had = serial;
            }
            uint32_t e = 0, f = 0, o = 0;                  // greatest, second and third gain >> shift (+ 1), and whose they are
            int ev = 0, fv = 0;
            for (int q = lane; q < ld4; q += 32) {
                const uint32_t nib = *(volatile const uint32_t *)&bits[q >> 3] >> ((q & 7) * 4);
                const ulonglong2 a0 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q], a1 = reinterpret_cast<const ulonglong2 *>(gains)[2 * q + 1];
                const unsigned long long g[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t k = (nib >> u & 1) ? 0u : lead_part(g[u], shift);
                    if (k > f) {
                        o = f;
                        if (k > e) { f = e; fv = ev; e = k; ev = 4 * q + u; }
                        else { f = k; fv = 4 * q + u; }
                    } else {
                        o = max(o, k);
                    }
                }
            }
            o = __reduce_max_sync(0xffffffffu, o);
            li.lead[lane] = e;
            li.lead[32 + lane] = f;
            li.sample[lane] = (uint16_t)ev;
            li.sample[32 + lane] = (uint16_t)fv;
            if (lane == 0) li.bound = o;
            // the list that was there is withdrawn before any word of the new one is written, and the new one complete
            // before its tag: the barrier hands every lane what the others stored, the fence after it orders that
            __syncwarp();
            release_fence();
            st_remote(listAddr + (uint32_t)lane * 8, e ? key_of(e, low_part(gains[ev], shift, ev), shift) : 0ull);
            st_remote(listAddr + (uint32_t)(32 + lane) * 8, f ? key_of(f, low_part(gains[fv], shift, fv), shift) : 0ull);
            if (lane == 0) st_remote(listAddr + (uint32_t)NoteLayout::kList * 8, o ? key_of(o, ((1u << shift) - 1u) << 16 | 0xffffu, shift) : 0ull);
            __syncwarp();
            release_fence();
            if (lane == i) st_remote(listAddr + (uint32_t)(NoteLayout::kList + 1) * 8, (unsigned long long)serial << 16 | (lists & 0xffffu));
            __syncwarp();
        }
    }
}

// A team with several blocks, coverage and stored gains in memory (shared memory where they fit).  Its commands come
// through a ring, in the order given.
template <bool kCut, typename Where>
__device__ __forceinline__ void team_of_many(const ClusterParams &prm, const ClassDesc &c, const TeamView &t, int mine, int shift,
                                             unsigned long long bias, uint32_t cmds, Where where, unsigned &corrected, unsigned &rows)
{
    const int lane = t.lane, T = t.T, tid = t.warpIn * 32 + lane, step = T * 32;
    int4 *cov;
    unsigned long long *gains;
    uint32_t noteAddr, barAddr;
    volatile uint32_t *told;
    uint32_t serial = 0;                                   // lane i: commands for block i so far
    // the block's best candidate goes to the leader, and the command it answers to the listing warps
    auto tell = [&](int i) {
        const Summary sum = summarize(scan_gains(t.bits, gains, t.ld4, tid, step, shift), shift, T, lane);
        unsigned long long top = sum.top;
        post(t, T, sum, noteAddr, barAddr);
        if (T > 1) {
            if (lane == 0) t.tm->best[t.warpIn] = top;
            team_barrier(t.team, T);
            if (t.warpIn == 0) top = warp_max_u64(lane < T ? t.tm->best[lane] : 0ull);
        }
        if (lane == i) ++serial;
        // (the whole team's gains are written: a barrier lies between them and here, in front of this call or above)
        if (t.warpIn == 0 && lane == i) {
            st_async(noteAddr, top, barAddr);
            __threadfence_block();
            *told = serial;
        }
    };
    if (tid == 0) t.tm->count[0] = t.tm->count[1] = 0;
    int par = 0;
    for (int i = 0; i < mine; ++i) {
        where(i, cov, gains, noteAddr, barAddr, told);
        for (int q = tid; q < t.ld4; q += step) {
            if (!kCut) cov[q] = make_int4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) gains[4 * q + u] = 4 * q + u < c.M ? (unsigned long long)__ldcg(prm.g0 + c.row0 + 4 * q + u) + bias : 0ull;
        }
    }
    team_barrier(t.team, T);
    for (uint32_t n = 1;; ++n) {
        const uint32_t at = cmds + ((n - 1) & (uint32_t)(prm.ring - 1)) * 8;
        unsigned long long cmd = 0;
        unsigned spin = 0;
        for (;;) {
            cmd = ld_relaxed(at);
            if ((uint32_t)(cmd >> 32) == n) break;
            if (++spin >= kPollLimit) break;
        }
        if (spin >= kPollLimit) {
            if (lane == 0) atomicOr(prm.status, kDevTimeout);
            break;
        }
        __syncwarp();
        const uint32_t what = (uint32_t)cmd & 0xfffffu;
        const int i = (int)((uint32_t)cmd >> 20);
        if (what == kStopCmd) break;
        where(i, cov, gains, noteAddr, barAddr, told);
        if (what == kScanCmd) {
            shared_acquire_fence();
            tell(i);
            continue;
        }
        ++corrected;
        if (kCut) {
            // gain = column sum - twice the tie to the block: the sample's row is the tie's growth
            const int4 *row = t.S4 + (int64_t)((int)what - 1) * t.ld4;
            for (int q = tid; q < t.ld4; q += step) {
                const int4 r = __ldg(row + q);
                ulonglong2 *p = reinterpret_cast<ulonglong2 *>(gains) + 2 * q;
                const ulonglong2 k0 = p[0], k1 = p[1];
                p[0] = make_ulonglong2(take_off(k0.x, 2 * r.x), take_off(k0.y, 2 * r.y));
                p[1] = make_ulonglong2(take_off(k1.x, 2 * r.z), take_off(k1.y, 2 * r.w));
            }
        } else {
            take_in_lists(t, (int)what - 1, cov, t.tm->count, par, rows, [&](int m) {
#pragma unroll 1
                for (int q = tid; q < t.ld4; q += step) {
                    ulonglong2 *p = reinterpret_cast<ulonglong2 *>(gains) + 2 * q;
                    const ulonglong2 k0 = p[0], k1 = p[1];
                    unsigned long long k[4] = {k0.x, k0.y, k1.x, k1.y};
                    if (correct_piece(t.S4 + q, t.list, m, k)) {
                        p[0] = make_ulonglong2(k[0], k[1]);
                        p[1] = make_ulonglong2(k[2], k[3]);
                    }
                }
            });
        }
        __syncwarp();
        tell(i);
    }
}

// The leader's loop over the picks of class c.  One warp; lane p % 32 keeps the value and the room of block p, and the
// parity of the mbarrier on which the block's notes arrive (they go on from class to class).  A pick is a chain of dependent
// latencies (shuffle, mbarrier, two shared-memory loads, the command); what does not depend on the pick
// (the least of the other blocks) is computed under them, and a block's state travels in one shuffle.
// kMany: every block's first sample comes from `firsts`, the greatest gains for an empty block in order (they are the same
// for all blocks, so notes would be overtaken by one another).
template <int KW, bool kMany>
__device__ void lead(const ClusterParams &prm, int l, const ClassDesc &c, unsigned char *shared, uint32_t C, int T, unsigned long long bias, uint32_t turn,
                     uint32_t &parities)
{
    const int lane = threadIdx.x & 31, W = prm.W;
    const NoteLayout layout{T, kMany};
    const uint32_t noteBytes = layout.tracked();
    const int nTeams = team_warps(T) / T;
    volatile uint32_t *queue = reinterpret_cast<uint32_t *>(shared + prm.offQueue);      // commands given to each team
    const uint32_t base = smem32(shared);
    volatile uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    const uint32_t myBits = remote(base + prm.offBits, (uint32_t)lane < C ? lane : 0);
    volatile const unsigned long long *notes = reinterpret_cast<const unsigned long long *>(shared + prm.offNotes);
    volatile const unsigned long long *firsts = reinterpret_cast<const unsigned long long *>(shared + prm.offFirsts);
    const uint32_t bars = base + prm.offBars, notesAt = base + prm.offNotes;
    unsigned long long f[KW];              // (value + kTrackedZero) << 7 | block
    int room[KW];
    uint32_t given[KW];                    // commands given to the block
    uint32_t cmdAddr[KW];
    uint32_t qWord[KW];                    // kMany: block's number in its team << 20 | its team's entry of queue
    // four bits for each k: the block owes a note; parity of its mbarrier; its next sample is its last; it is empty
    constexpr uint32_t kOwes = 1, kParity = 2, kLast = 4, kEmpty = 8;
    uint32_t state = 0;
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        f[k] = (kTrackedZero << 7) | (unsigned long long)p;
        given[k] = 0;
        room[k] = p < W ? prm.quota[(int64_t)l * W + p] : 0;
        const uint32_t owner = (uint32_t)(p < W ? p : 0) & (C - 1), slot = (uint32_t)(p < W ? p : 0) >> prm.logC;
        cmdAddr[k] = remote(base + prm.offCmd + slot % nTeams * prm.ring * 8, owner);
        qWord[k] = slot / nTeams << 20 | (owner * nTeams + slot % nTeams);
        uint32_t st = (parities >> k & 1 ? kParity : 0u) | (room[k] == 1 ? kLast : 0u);
        if (kMany) {
            st |= kEmpty;
        } else if (room[k] > 0) {
            bar_expect(bars + p * 8, noteBytes);
            st |= kOwes;
        }
        state |= st << (4 * k);
    }
    // (run by the lane that keeps block lane + 32 k)
    auto command = [&](int k, uint32_t what) {
#pragma unroll
        for (int i = 0; i < KW; ++i)
            if (i == k) {
                uint32_t n = ++given[i];
                if (kMany) {
                    n = queue[qWord[i] & 0xfffffu] + 1;
                    queue[qWord[i] & 0xfffffu] = n;
                    what |= qWord[i] & 0xfff00000u;
                }
                st_remote(cmdAddr[i] + ((n - 1) & (uint32_t)(prm.ring - 1)) * 8, ((unsigned long long)n << 32) | what);
            }
    };
    __syncwarp();
    unsigned rescans = 0;
    int nextFirst = 0;
    bool ok = true;
    unsigned long long others = ~0ull, last = ~0ull;       // least of the blocks but the one picked last, and that one's
#pragma unroll
    for (int k = 0; k < KW; ++k) others = room[k] > 0 ? umin(others, f[k]) : others;
    others = ~warp_max_u64(~others);
    uint32_t *picks = prm.picks + c.row0;
    for (int t = 0; t < c.M; ++t) {
        const unsigned long long least = umin(others, last);
        if (least == ~0ull) {
            if (lane == 0) atomicOr(prm.status, kDevNoCandidate);
            ok = false;
            break;
        }
        const int j = (int)(least & 127);
        const int jk = KW == 1 ? 0 : j >> 5, jl = j & 31;
        const uint32_t st = __shfl_sync(0xffffffffu, state, jl) >> (4 * jk);
        uint32_t parity = st & kParity;
        volatile const unsigned long long *note = notes + j * layout.words();
        auto await = [&]() -> bool {
            unsigned spin = 0;
            while (!bar_done(bars + j * 8, parity ? 1u : 0u) && ++spin < kPollLimit) { }
            parity ^= kParity;
            if (spin < kPollLimit) {
                shared_acquire_fence();                    // (the note)
                return true;
            }
            if (lane == 0) atomicOr(prm.status, kDevTimeout);
            return false;
        };
        if (st & kOwes) ok = await();
        if (!ok) break;
        unsigned long long best = kMany && (st & kEmpty) ? 0ull : note[0];
        // the least of the other blocks: does not depend on this pick
        others = ~0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k) others = room[k] > 0 && lane + 32 * k != j ? umin(others, f[k]) : others;
        others = ~warp_max_u64(~others);
        int v = key_sample(best);
        uint32_t word = bits[v >> 5];
        if (best == 0 || (word >> (v & 31) & 1)) {
            // the block's best candidate has been taken by another block, or the block is empty
            best = 0;
            if (kMany && (st & kEmpty)) {
                for (; nextFirst < W; ++nextFirst) {
                    const unsigned long long k = firsts[nextFirst];
                    const int s = key_sample(k);
                    if (k == 0) { nextFirst = W; break; }
                    if (!(bits[s >> 5] >> (s & 31) & 1)) { best = k; break; }
                }
            }
            uint32_t serial = 0;
            if (kMany) {
#pragma unroll
                for (int k = 0; k < KW; ++k) if (k == jk) serial = given[k];
                serial = __shfl_sync(0xffffffffu, serial, jl);
            }
            while (best == 0) {
                if (!kMany || serial > 0) {
                    // the best of the candidates left, if none that the note leaves out can lead
                    const unsigned long long k = lane < layout.entries() + T ? note[1 + lane] : 0ull;
                    const int s = key_sample(k);
                    const bool free = lane < layout.entries() && k != 0 && !(bits[s >> 5] >> (s & 31) & 1);
                    best = warp_max_u64(free ? k : 0ull);
                    if (__any_sync(0xffffffffu, lane >= layout.entries() && k >= best)) best = 0;
                }
                if (kMany && serial > 0 && best == 0) {
                    // the list, and its next edition when all that are sure to lead in this one have been taken
                    // (Tag, words, tag: the first fence keeps the words behind the tag, and with the second a word of the next
                    // edition comes with the withdrawal of this one.)
                    const uint32_t list = notesAt + (uint32_t)(j * layout.words() + layout.list()) * 8;
                    unsigned spin = 0, spent = 0;
                    while (best == 0 && ++spin < kPollLimit) {
                        const unsigned long long tag = ld_relaxed(list + (NoteLayout::kList + 1) * 8);
                        shared_acquire_fence();
                        const unsigned long long k = ld_relaxed(list + (uint32_t)lane * 8), k2 = ld_relaxed(list + (uint32_t)(32 + lane) * 8);
                        const unsigned long long bound = ld_relaxed(list + NoteLayout::kList * 8);
                        shared_acquire_fence();
                        const unsigned long long again = ld_relaxed(list + (NoteLayout::kList + 1) * 8);
                        if (!__all_sync(0xffffffffu, tag == again && (uint32_t)(tag >> 16) == serial && (tag & 0xffffu) == (__shfl_sync(0xffffffffu, (uint32_t)tag, 0) & 0xffffu))) continue;
                        const int s = key_sample(k), s2 = key_sample(k2);
                        const bool free = k != 0 && !(bits[s >> 5] >> (s & 31) & 1), free2 = k2 != 0 && !(bits[s2 >> 5] >> (s2 & 31) & 1);
                        best = warp_max_u64(umax(free ? k : 0ull, free2 ? k2 : 0ull));
                        if (bound >= best) {
                            best = 0;
                            if (++spent > 200) break;      // (equal gains: the team decides)
                        }
                    }
                    if (spin >= kPollLimit) {
                        if (lane == 0) atomicOr(prm.status, kDevTimeout);
                        ok = false;
                        break;
                    }
                }
                if (best) break;
                // every candidate that is sure to lead has been taken by other blocks: the team looks again
                ++rescans;
                release_fence();                           // (it must see which samples are taken)
                if (lane == jl) {
                    bar_expect(bars + j * 8, noteBytes);
                    command(jk, kScanCmd);
                }
                ++serial;
                ok = await();
                if (!ok) break;
                const unsigned long long k = note[0];
                const int s = key_sample(k);
                if (k != 0 && !(bits[s >> 5] >> (s & 31) & 1)) best = k;
            }
            if (!ok) break;
            v = key_sample(best);
            word = bits[v >> 5];
        }
        const unsigned long long inc = ((best >> 16) - bias) << 7;
        last = (st & kLast) ? ~0ull : least + inc;         // (a full block is out)
        word |= 1u << (v & 31);
        if (lane == jl) {
            if (!(st & kLast)) {                           // (and needs no gains any more)
                bar_expect(bars + j * 8, noteBytes);
                command(jk, (uint32_t)(v + 1));
            }
#pragma unroll
            for (int k = 0; k < KW; ++k)
                if (k == jk) {
                    f[k] += inc;
                    --room[k];
                    const uint32_t now = parity | (st & kLast ? 0u : kOwes) | (room[k] == 1 ? kLast : 0u);
                    state = (state & ~(15u << (4 * k))) | now << (4 * k);
                }
        }
        if (lane == 0) {
            bits[v >> 5] = word;
            picks[t] = (uint32_t)v | ((uint32_t)j << 16);
        }
        if (lane > 0 && lane < (int)C) st_remote32(myBits + (uint32_t)(v >> 5) * 4, word);
        __syncwarp();
    }
    // notes still under way land before the class ends; then every team is sent home
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int p = lane + 32 * k;
        uint32_t st = state >> (4 * k) & 15u;
        if (ok && (st & kOwes)) {
            unsigned spin = 0;
            while (!bar_done(bars + p * 8, st & kParity ? 1u : 0u) && ++spin < kPollLimit) { }
            if (spin >= kPollLimit) atomicOr(prm.status, kDevTimeout);
            st ^= kParity;
        }
        parities = (parities & ~(1u << k)) | (st & kParity ? 1u << k : 0u);
        if (p < W) {
            if (!kMany || p >> prm.logC < nTeams) command(k, kStopCmd);
            const long long value = (long long)(f[k] >> 7) - (long long)kTrackedZero;
            prm.fval[(int64_t)l * W + p] = prm.fixedExp ? __double_as_longlong(ldexp((double)value, -prm.fixedExp[l])) : value;
        }
    }
    if (kMany && lane < (int)C) st_remote32(remote(base + prm.offTold, lane), turn);
    if (lane == 0 && rescans) atomicAdd(prm.stats + 9, (unsigned long long)rescans);
}

// P: pieces per thread of teams with one block; 0: teams with several blocks (kSmemState: which all fit the
// CTAs' shared memory).  kCut: graph-cut objective.
template <int KW, int P, int kT, bool kSmemState, bool kCut>
__global__ void __launch_bounds__((P == 0 ? kMaxWarps + 1 + kListers : team_warps(kT) + 1) * 32, 1) greedy_cluster_kernel(const __grid_constant__ ClusterParams prm)
{
    extern __shared__ __align__(128) unsigned char shared[];
    __shared__ int shClass[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rank = cluster_rank(), C = cluster_size();
    constexpr int NW = team_warps(kT);
    const int T = kT ? kT : prm.teamWarps, nTeams = NW / T;
    const uint32_t base = smem32(shared);
    uint32_t *bits = reinterpret_cast<uint32_t *>(shared + prm.offBits);
    volatile unsigned long long *cmds = reinterpret_cast<volatile unsigned long long *>(shared + prm.offCmd);
    const int W = prm.W;
    uint32_t parities = 0;
    const NoteLayout layout{T, P == 0};
    uint32_t classes = 0;                                  // this cluster has drawn (classes left in floating point and empty ones too)

    // (for the listing warps: the number of the class that has ended last, 0 at first, then per block the command told last)
    volatile uint32_t *const ended = reinterpret_cast<uint32_t *>(shared + prm.offTold);
    volatile uint32_t *const told0 = ended + 4;
    if (P == 0 && threadIdx.x == 0) *ended = 0;
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
        ++classes;
        if (prm.fixedExp && prm.fixedExp[l] == kNotFixed) continue;
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
        for (int i = threadIdx.x; i < nTeams * prm.ring; i += blockDim.x) cmds[i] = 0;
        if (P == 0)
            for (int i = threadIdx.x; i < prm.slots; i += blockDim.x) told0[i] = 0;
        if (P == 0 && rank == 0) {
            for (int i = threadIdx.x; i < (int)C * nTeams; i += blockDim.x) reinterpret_cast<uint32_t *>(shared + prm.offQueue)[i] = 0;
            for (int i = threadIdx.x; i < W * layout.words(); i += blockDim.x) reinterpret_cast<unsigned long long *>(shared + prm.offNotes)[i] = 0;
        }
        cluster_barrier();
        if constexpr (P == 0) {
            // The greatest gains for an empty block in order: every sample's rank by counting, a share of the samples per CTA.
            if (rank == 0) for (int i = threadIdx.x; i < W; i += blockDim.x) reinterpret_cast<unsigned long long *>(shared + prm.offFirsts)[i] = 0;
            cluster_barrier();
            const uint32_t firsts0 = remote(base + prm.offFirsts, 0);
            const unsigned long long bias0 = kCut ? 3 * __ldcg(prm.topGain + l) + 1 : 0ull;
            auto key0 = [&](int v) { return make_key((unsigned long long)__ldcg(prm.g0 + c.row0 + v) + bias0, v); };
            for (int v = rank * (NW + 1 + kListers) + warp; v < c.M; v += C * (NW + 1 + kListers)) {
                const unsigned long long mine = key0(v);
                int above = 0;
                for (int u0 = 0; u0 < c.M && above < W; u0 += 256) {
                    int n = 0;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int w = u0 + u * 32 + lane;
                        n += w < c.M && key0(w) > mine ? 1 : 0;
                    }
                    above += __reduce_add_sync(0xffffffffu, n);
                }
                if (above < W && lane == 0) st_remote(firsts0 + above * 8, mine);
            }
            cluster_barrier();
        }
        // graph cut: gains lie within three times the largest sum of |S| over a row, either way
        const unsigned long long top = __ldcg(prm.topGain + l);
        const unsigned long long bias = kCut ? 3 * top + 1 : 0ull;
        const int shift = shift_for(bias + (kCut ? 3 : 1) * top);

        if (warp == NW) {
            if (rank == 0) lead<KW, P == 0>(prm, l, c, shared, C, T, bias, classes, parities);
        } else if (warp > NW) {
            list_candidates(prm, bits, ld4, shift, smem32((const void *)told0), reinterpret_cast<Listed *>(shared + prm.offListed), warp - NW - 1, kListers, prm.slots, ended, classes, [&](int slot, const unsigned long long *&gains) {
                const int j = slot * (int)C + (int)rank;
                if (kSmemState) gains = reinterpret_cast<const unsigned long long *>(shared + prm.offGains) + (size_t)slot * prm.maxLd;
                else gains = reinterpret_cast<const unsigned long long *>(prm.gains + c.vOff) + (size_t)j * c.ld;
                return remote(base + prm.offNotes, 0) + (uint32_t)(j * layout.words()) * 8;
            });
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
                if (team < prm.slots && team < nTeams && j < W && prm.quota[(int64_t)l * W + j] > 0)
                    team_of_one<(P > 0 ? P : 1), kT, kCut>(prm, c, t, reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)team * (prm.maxLd >> 2), shift, bias,
                                                       base + prm.offCmd + team * prm.ring * 8, notes0 + j * (uint32_t)layout.words() * 8, bars0 + j * 8, corrected, rows);
            } else {
                // the i-th block of the team
                auto where = [&](int i, int4 *&cov, unsigned long long *&gains, uint32_t &noteAddr, uint32_t &barAddr, volatile uint32_t *&told) {
                    const int slot = team + i * nTeams, j = slot * (int)C + (int)rank;
                    if (kSmemState) {
                        cov = reinterpret_cast<int4 *>(shared + prm.offCover) + (size_t)slot * (prm.maxLd >> 2);
                        gains = reinterpret_cast<unsigned long long *>(shared + prm.offGains) + (size_t)slot * prm.maxLd;
                    } else {
                        cov = reinterpret_cast<int4 *>(prm.cover + c.vOff) + (size_t)j * ld4;
                        gains = reinterpret_cast<unsigned long long *>(prm.gains + c.vOff) + (size_t)j * c.ld;
                    }
                    noteAddr = notes0 + j * (uint32_t)layout.words() * 8;
                    told = told0 + slot;
                    barAddr = bars0 + j * 8;
                };
                int mine = 0;
                while (team + mine * nTeams < prm.slots && (team + mine * nTeams) * (int)C + (int)rank < W) ++mine;
                if (mine > 0) team_of_many<kCut>(prm, c, t, mine, shift, bias, base + prm.offCmd + team * prm.ring * 8, where, corrected, rows);
            }
            if (lane == 0 && t.warpIn == 0 && corrected) {
                atomicAdd(prm.stats + 15, (unsigned long long)corrected);
                atomicAdd(prm.stats + 16, (unsigned long long)rows);
            }
        }
        cluster_barrier();
        // class-local picks -> outputs (none where the loop stopped early: the words behind the last pick are whatever memory held)
        const bool stopped = __ldcg(prm.status) != 0;
        for (int t = rank * blockDim.x + threadIdx.x; t < c.M; t += C * blockDim.x) {
            const uint32_t p = __ldcg(prm.picks + c.row0 + t);
            if (stopped) break;
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
// That holds for rows of about one norm (normalised features).  A class whose
// squared norms differ by more than a factor of 16, or are not finite, is left in floating point (kNotFixed) for
// launch_greedy_not_fixed.
__global__ void __launch_bounds__(256, 8) fixed_exponent_kernel(const ClassDesc *__restrict__ desc, const float *__restrict__ S, int32_t *__restrict__ fixedExp,
                                                               int32_t *__restrict__ sizesLeft, volatile int32_t *left)
{
    __shared__ float shMax[8], shMin[8];
    const ClassDesc c = desc[blockIdx.x];
    float m = 0.f, least = INFINITY;                       // (zero rows have similarity 0 with everything: exact at any scale)
    bool odd = false;
    for (int v = threadIdx.x; v < c.M; v += 256) {
        const float x = S[c.sOff + (int64_t)v * c.ld + v];
        odd = odd || !(x >= 0.f && x <= 1e30f);
        m = fmaxf(m, x);
        if (x > 0.f) least = fminf(least, x);
    }
    for (int off = 16; off > 0; off >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        least = fminf(least, __shfl_xor_sync(0xffffffffu, least, off));
    }
    if ((threadIdx.x & 31) == 0) { shMax[threadIdx.x >> 5] = m; shMin[threadIdx.x >> 5] = least; }
    odd = __syncthreads_or(odd);
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) { m = fmaxf(m, shMax[w]); least = fminf(least, shMin[w]); }
        int e = 0;
        if (m > 0.f && !odd) frexpf(m, &e);                // m = x 2^e, x in [0.5, 1)
        odd = odd || (m > 0.f && (m > 16.f * least || m < 1e-30f));
        fixedExp[blockIdx.x] = odd ? kNotFixed : 30 - e;
        sizesLeft[blockIdx.x] = odd ? c.M : 0;
        if (odd) *left = 1;                                // (the host's memory: read once the kernel is done)
    }
}
__global__ void __launch_bounds__(256, 8) fixed_point_kernel(const ClassDesc *__restrict__ desc, const int32_t *__restrict__ fixedExp, float *__restrict__ S)
{
    const ClassDesc c = desc[blockIdx.y];
    if (fixedExp[blockIdx.y] == kNotFixed) return;
    const float scale = ldexpf(1.f, fixedExp[blockIdx.y]);
    float4 *p = reinterpret_cast<float4 *>(S + c.sOff);
    const int64_t n = (int64_t)c.M * (c.ld >> 2);
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const float4 x = p[i];
        reinterpret_cast<int4 *>(p)[i] = make_int4(to_fixed(x.x, scale), to_fixed(x.y, scale), to_fixed(x.z, scale), to_fixed(x.w, scale));
    }
}

static int pow2_at_least(int x)
{
    int p = 1;
    while (p < x) p *= 2;
    return p;
}

typedef void (*ClusterKernel)(ClusterParams);

template <int KW, int kT, bool kCut>
static ClusterKernel pick_one(int P)
{
    switch (P) {
    case 1: return greedy_cluster_kernel<KW, 1, kT, true, kCut>;
    case 2: return greedy_cluster_kernel<KW, 2, kT, true, kCut>;
    case 3: return greedy_cluster_kernel<KW, 3, kT, true, kCut>;
    case 4: return greedy_cluster_kernel<KW, 4, kT, true, kCut>;
    case 5: return greedy_cluster_kernel<KW, 5, kT, true, kCut>;
    default: return greedy_cluster_kernel<KW, kMaxPieces, kT, true, kCut>;
    }
}
// (P = 0: teams with several blocks)
template <int KW, bool kCut>
static ClusterKernel pick_kernel(int P, int T, bool smemState)
{
    if (P == 0) return smemState ? greedy_cluster_kernel<KW, 0, 0, true, kCut> : greedy_cluster_kernel<KW, 0, 0, false, kCut>;
    if constexpr (KW == 1) {
        if (T == 15) return pick_one<KW, 15, kCut>(P);         // (one block per CTA: 16 at most)
        if constexpr (!kCut)
            if (T == 8) return pick_one<KW, 8, kCut>(P);
    }
    return pick_one<KW, 0, kCut>(P);
}

static rcd_status launch_cluster(rcd_ctx *ctx, ClusterKernel kernel, const ClusterParams &prm, int threads, int C, int clusters, size_t smem, cudaStream_t st, int *active)
{
    RCD_CUDA(ctx, allow_shared(kernel, whole_shared(ctx)));
    RCD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * C));
    cfg.blockDim = dim3((unsigned)threads);
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
    std::shared_ptr<RoundsPlan> rounds;   // not null: the classes run in rounds instead, one CTA each
    std::shared_ptr<SmallPlan> small;     // not null: one CTA each with the class's similarities in its shared memory
    double cutCycles = 0;      // graph cut: what the clusters are expected to take
    ClusterParams prm;         // teamWarps, slots, maxLd, rowPieces and the offsets are set
};
static size_t cluster_layout(const Sizes &sz, int maxLd, int C, bool state, size_t cap, ClusterPlan &plan)
{
    ClusterParams &prm = plan.prm;
    prm.maxLd = maxLd;
    prm.slots = (sz.W + C - 1) / C;
    prm.logC = 0;
    while ((1 << prm.logC) < C) ++prm.logC;
    const int ld4 = maxLd / 4;
    // A team per block, of as many warps as there are, or teams of several blocks: then a team has as many warps as a row
    // keeps busy (at least three fifths of their threads; measured on 300 to 1300 samples), half of that with more than 16
    // blocks to serve.
    const int rowWarps = (ld4 + 31) / 32;
    int one = std::min(kMaxWarps / std::min(kMaxWarps, pow2_at_least(prm.slots)), pow2_at_least(rowWarps));
    if (prm.slots == 1 && rowWarps > 8) one = 15;
    int busy = 1;
    for (int T = 2; T <= kMaxWarps; T *= 2)
        if (5 * ld4 >= 3 * 32 * T) busy = T;
    if (prm.slots > kMaxWarps && busy > 1) busy /= 2;
    const int onePieces = (ld4 + 32 * one - 1) / (32 * one);
    int pieces = onePieces;
    auto place = [&](bool many, bool state) -> size_t {
        prm.teamWarps = many ? busy : one;
        plan.P = many ? 0 : pieces;
        const int warps = many ? kMaxWarps : team_warps(prm.teamWarps);
        const int step = prm.teamWarps * 32, teams = warps / prm.teamWarps;
        const int perTeam = (prm.slots + teams - 1) / teams;
        prm.ring = many ? pow2_at_least(perTeam + 1) : 1;
        const NoteLayout note{prm.teamWarps, many};
        size_t off = 0;
        auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 15) / 16 * 16; return (int32_t)at; };
        prm.offTeams = take(sizeof(Team) * (size_t)teams);
        prm.offCmd = take(8 * (size_t)teams * prm.ring);
        prm.offBits = take((size_t)(maxLd + 31) / 32 * 4);
        prm.offLists = take(sizeof(Raised) * (size_t)(warps * kRaisedPerWarp + teams));
        prm.offNotes = take((size_t)note.words() * 8 * (size_t)sz.W);
        prm.offBars = take(8 * (size_t)sz.W);
        prm.offQueue = take(many ? 4 * (size_t)C * teams : 0);
        prm.offFirsts = take(many ? 8 * (size_t)sz.W : 0);
        prm.offListed = take(many ? sizeof(Listed) * (size_t)prm.slots : 0);
        prm.offTold = take(many ? 16 + 4 * (size_t)prm.slots : 0);
        // (a team's row buffer: the row of the sample foreseen, and the rows on their way through apply_list)
        prm.rowPieces = many ? 0 : (std::max(plan.P * step, plan.P <= 3 ? kRowStages * ld4 : kPieceStages * step) + 7) / 8 * 8;
        // (asynchronous 16-byte copies whose destination sits differently in its 32-byte sector than the source fetch two
        // sectors each: rows of S start on sectors, so the buffers do)
        off = (off + 127) / 128 * 128;
        prm.offRows = take((size_t)std::min(teams, prm.slots) * prm.rowPieces * 16);
        prm.offCover = take(!many || state ? (size_t)prm.slots * maxLd * 4 : 0);
        prm.offGains = take(many && state ? (size_t)prm.slots * maxLd * 8 : 0);
        plan.smemState = state;
        return off;
    };
    const bool oneFits = prm.slots <= kMaxWarps && onePieces <= kMaxPieces;
    const bool manyFits = (prm.slots + kMaxWarps / busy - 1) / (kMaxWarps / busy) <= 31;
    // (graph cut: the blocks' best candidates are mostly the same samples, so notes have to be kept fresh)
    if (oneFits && !(sz.graphCut && manyFits && prm.slots > 1) && (prm.slots == 1 || one >= 8 || (onePieces <= 3 && 2 * one >= busy) || !manyFits)) {
        const size_t need = place(false, true);
        if (need <= cap) return need;
    }
    if (manyFits) {
        const size_t need = place(true, true);
        if (need <= cap) return need;
    }
    if (oneFits) {
        size_t need = place(false, true);
        if (need <= cap) return need;
        if (plan.P == 3) {                                 // (less room: the four-piece kernel's ring)
            pieces = 4;
            need = place(false, true);
            if (need <= cap) return need;
        }
    }
    if (!state && manyFits) return place(true, false);     // (coverage and gains in global memory)
    return cap + 1;
}

// How a problem is laid out over clusters, if its blocks fit registers or shared memory.  resident: clusters at a time.
static bool cluster_shape(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, int nonEmpty, int maxLd, ClusterPlan &plan, int *resident)
{
    const size_t cap = (size_t)whole_shared(ctx);
    for (int i = 0; i < 5; ++i)
        if (ctx->maxClusters[i] < 0) {
            int active = 0;
            if (launch_cluster(ctx, pick_kernel<1, false>(3, 15, true), plan.prm, 16 * 32, 1 << i, 1, cap, nullptr, &active) != RCD_OK) return false;
            ctx->maxClusters[i] = active;
        }
    // Cluster size: the one whose clusters, drawing classes largest first, finish soonest by the estimate that a class of
    // M samples takes M (M / C + 300) (corrections, shared by the CTAs, and the chain of picks); blocks have to stay on
    // the chip.
    // (graph cut, small classes: an update is one row, so the time goes into stale notes, and several blocks per CTA with lists
    // of candidates do better than one: 2 classes of 400 into 8 blocks 791 us with 8 CTAs, 517 with 4, pass-free chain 583)
    const int most = std::min(sz.graphCut && sz.maxM <= 1536 ? 4 : 16, pow2_at_least(sz.W));
    std::vector<int> sizes;
    for (const ClassDesc &d : descHost) if (d.M > 0) sizes.push_back(d.M);
    std::sort(sizes.begin(), sizes.end(), std::greater<int>());
    std::vector<double> busy;
    double bestTime = 0;
    plan.C = 0;
    for (int i = 0; (1 << i) <= most; ++i) {
        const int C = 1 << i, n = ctx->maxClusters[i];
        if (n < 1) continue;
        if (cluster_layout(sz, maxLd, C, true, cap, plan) > cap) continue;
        const size_t held = std::min<size_t>((size_t)n, sizes.size());
        auto cost = [&](int M) { return (double)M * ((double)M / C + 300.0); };
        // (all clusters busy to the end: no sooner than that.  A call of many small classes waits for the host here, 874 of up to 253
        // samples 225 us without this)
        double work = 0;
        for (int M : sizes) work += cost(M);
        if (plan.C > 0 && work / (double)held * (1 - 1e-9) > bestTime) continue;
        double time = 0;
        busy.assign(held, 0.0);                            // a heap of the clusters' finishing times, the earliest first
        for (int M : sizes) {
            const double done = busy[0] + cost(M);
            time = std::max(time, done);
            size_t at = 0;
            for (size_t child; (child = 2 * at + 1) < held; at = child) {
                if (child + 1 < held && busy[child + 1] < busy[child]) ++child;
                if (busy[child] >= done) break;
                busy[at] = busy[child];
            }
            busy[at] = done;
        }
        if (plan.C == 0 || time < bestTime) { plan.C = C; bestTime = time; }
    }
    if (plan.C > 0) {
        plan.smem = cluster_layout(sz, maxLd, plan.C, true, cap, plan);
    } else {
        plan.C = std::min(8, most);
        plan.smem = cluster_layout(sz, maxLd, plan.C, false, cap, plan);
        if (plan.smem > cap) return false;
    }
    // Graph cut with many blocks per CTA: every pick makes most of the other blocks' notes stale, and the listing warps fall
    // behind the chain of one CTA per class (2 classes of 1000, 16 blocks per CTA: 2625 us against 1981; 2 of 3000 into 100
    // blocks 12.6 ms against 11.7; but 30 of 600, 15 blocks per CTA, 1124 against 1255).
    if (sz.graphCut && (sz.W > 64 || (sz.W + plan.C - 1) / plan.C > 15)) return false;
    int idx = 0;
    while ((1 << idx) < plan.C) ++idx;
    if (ctx->maxClusters[idx] < 1) return false;
    *resident = ctx->maxClusters[idx];
    plan.clusters = std::max(1, std::min(nonEmpty, *resident));
    return true;
}

// Whether the cluster form, the rounds or the form for small classes take a problem, and how: chosen by the library (no pass-based form or option asked for),
// samples of a class and blocks within the packed keys' range.
static bool cluster_plan(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, ClusterPlan &plan)
{
    if (!library_chooses(ctx->cfg)) return false;
    if (sz.W > kClusterBlocks || sz.maxM > 65535 || sz.d > 65535 || sz.L > 65535 || sz.maxM == 0) return false;
    if (sz.graphCut && (sz.floatArith || sz.maxM > 8192)) return false;
    int nonEmpty = 0, maxLd = 8, resident = 0;
    for (const ClassDesc &d : descHost) {
        if (d.M > 0) ++nonEmpty;
        maxLd = std::max(maxLd, (int)d.ld);
    }
    plan.prm = ClusterParams{};
    plan.prm.maxLd = maxLd;
    // (small classes whenever they fit: on mixtures of Gaussians 0.5 to 0.9 times the cluster form's time.  What a pick costs grows with the
    // columns it raises, which only the features tell: rectified ones 0.6 to 1.0 times, with 200 and more bf16 samples into 7 to 12 blocks
    // up to 1.1 for a few classes and 1.2 for one; independent normal ones, whose picks raise many, up
    // to 1.3 from 200 samples and 8 blocks on.  Rounds first: where those are faster than the cluster form was measured before, and they
    // stay)
    plan.small = plan_greedy_small(ctx, sz);
    if (plan.small && !rounds_possible(ctx, sz, descHost)) return true;
    const bool clusters = cluster_shape(ctx, sz, descHost, nonEmpty, maxLd, plan, &resident);
    plan.prm.maxLd = maxLd;
    if (sz.graphCut && clusters) plan.cutCycles = cut_cluster_cycles(plan.C, resident, sz.W, descHost);
    plan.rounds = plan_greedy_rounds(ctx, sz, descHost, clusters ? ClusterShape{plan.C, resident, plan.P} : ClusterShape{0, 0, 0});
    if (plan.rounds) plan.small = nullptr;
    return clusters || plan.rounds || plan.small;
}

std::shared_ptr<ClusterPlan> plan_greedy_cluster(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, bool *cutInStep)
{
    auto plan = std::make_shared<ClusterPlan>();
    if (!cluster_plan(ctx, sz, descHost, *plan)) plan = nullptr;
    *cutInStep = sz.graphCut && !(plan && plan->small) && cut_in_step(ctx, sz, descHost, plan ? plan->cutCycles : 0.0);
    return *cutInStep ? nullptr : plan;
}

// Runs the greedy loop.  partValues (may be null) receives the tracked values.
rcd_status launch_greedy_cluster(rcd_ctx *ctx, ClusterPlan &plan, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                 int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st)
{
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
    // Whether a class was left in floating point is known once the similarities are: the host waits for that under the loop's
    // kernel.  (A launch in every call that finds out by itself would have to bring as many CTAs as such classes need, all
    // resident at once, and so wait for whatever other streams run.)
    volatile int32_t *const left = ctx->hostStage + ctx->hostStageInts + kStageLeft;
    const bool toFix = sz.floatArith && ctx->cfg.similarity_kind != RCD_SIM_GAUSSIAN;     // (the Gaussian kernel writes fixed point itself)
    if (toFix) {
        // (a class may have to be left to the forms with passes: whether a call is refused is not to depend on its features)
        const rcd_status fits = check_coverage_fits(ctx, prm.maxLd);
        if (fits != RCD_OK) return fits;
        *left = 0;
        fixed_exponent_kernel<<<sz.L, 256, 0, st>>>(ws.desc, (const float *)ws.S, ws.fixedExp, ws.sizesLeft, left);
        RCD_CUDA(ctx, cudaEventRecord(ctx->evCounts, st));
        ctx->kernelLaunches++;
        if (!plan.small) {                                 // (that form rounds what it loads)
            const int64_t pieces = sz.maxM * (int64_t)(prm.maxLd / 4);
            const dim3 grid((unsigned)std::min<int64_t>((pieces + 1023) / 1024, std::max(1, 16 * ctx->smCount / sz.L)), (unsigned)sz.L);
            fixed_point_kernel<<<grid, 256, 0, st>>>(ws.desc, ws.fixedExp, (float *)ws.S);
            ctx->kernelLaunches++;
        }
        RCD_CUDA(ctx, cudaGetLastError());
    }
    if (plan.rounds) {
        const rcd_status rs = launch_greedy_rounds(ctx, *plan.rounds, sz, ws, assignment, order, partValues, st);
        if (rs != RCD_OK) return rs;
    } else if (plan.small) {
        const rcd_status rs = launch_greedy_small(ctx, *plan.small, sz, ws, toFix, assignment, order, partValues, st);
        if (rs != RCD_OK) return rs;
    } else {
        ClusterKernel kernel = sz.graphCut ? (sz.W <= 32 ? pick_kernel<1, true>(plan.P, prm.teamWarps, plan.smemState) : pick_kernel<4, true>(plan.P, prm.teamWarps, plan.smemState))
                                           : (sz.W <= 32 ? pick_kernel<1, false>(plan.P, prm.teamWarps, plan.smemState)
                                              : sz.W <= 64 ? pick_kernel<2, false>(plan.P, prm.teamWarps, plan.smemState) : pick_kernel<4, false>(plan.P, prm.teamWarps, plan.smemState));
        const rcd_status rs = launch_cluster(ctx, kernel, prm, (plan.P == 0 ? kMaxWarps + 1 + kListers : team_warps(prm.teamWarps) + 1) * 32, plan.C, plan.clusters, plan.smem, st, nullptr);
        if (rs != RCD_OK) return rs;
    }
    ctx->steps = sz.maxM;
    ctx->greedyForm = plan.rounds ? RCD_FORM_ROUNDS : plan.small ? RCD_FORM_SMALL : RCD_FORM_CLUSTER;
    ctx->phaseNsDev = ws.phaseNs;
    if (toFix) RCD_CUDA(ctx, cudaEventSynchronize(ctx->evCounts));
    if (toFix && *left) return launch_greedy_not_fixed(ctx, sz, ws, descHost, assignment, order, partValues, st);
    return RCD_OK;
}

}  // namespace rcd
