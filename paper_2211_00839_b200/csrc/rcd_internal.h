// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <algorithm>
#include <memory>
#include <string>
#include <vector>

#include "rcd.h"

namespace rcd {

constexpr int kMaxSweepBatch = 8;          // blocks refreshed by one dense pass over S
constexpr int kSparseMax = 64;             // blocks refreshed by one threshold pass over S
constexpr int kSweepThreads = 512;         // sweep CTA: 16 warps, one CTA per SM
constexpr int kSelectThreads = 512;        // pick/update CTA: one per class
constexpr int kLazyBlocks = 64;            // row skipping keeps a floor per block for classes of up to this many blocks
constexpr int kPhaseWords = 20;            // 64-bit counters a greedy launch keeps (phase clocks, barrier, pass statistics)
constexpr size_t kAlign = 256;

// Device-side status bits (OR-ed into the status word).
enum : int {
    kDevOk = 0,
    kDevBadLabel = 1,          // a label outside [0, L)
    kDevNoCandidate = 2,       // a class had samples left but no block could take one
    kDevBadState = 4,          // internal consistency check failed
    kDevTimeout = 8,           // a bounded wait inside a kernel ran out
};

// Hand-off word of one class between the CTA that makes its picks and the CTAs that sweep it (the
// asynchronous greedy kernel).  `epoch` is a sequence lock: even = sweep number epoch/2 is published
// and its parameters are stable, odd = the class belongs to its pick CTA (or is finished).
struct ClassSync {
    int32_t epoch;
    int32_t nGroups;   // row groups (tickets) of the published sweep
    int32_t done;      // row groups of the published sweep whose gains are written
    int32_t seq;       // order number of the published sweep (sweep number x L + class)
    int32_t pad_[2];   // (the word fills one 32-byte sector: the counters of two classes never share one)
    int32_t nR;        // of the published sweep: samples of the class still unassigned
    int32_t cfg;       //   blocks it refreshes | warps per row group << 8 | (1 = threshold pass) << 16
};
static_assert(sizeof(ClassSync) == 32, "one 32-byte sector per class");

// One class, as the kernels see it.  Built on the host once the class sizes are known.
struct ClassDesc {
    int32_t M;        // samples in the class
    int32_t ld;       // row pitch of S and of the per-block vectors, in elements (a multiple of 4; pad_row(M) inside rcd_partition)
    int32_t row0;     // first row of the class in class-sorted sample order
    int32_t pad_;
    int64_t sOff;     // element offset of S_l
    int64_t vOff;     // element offset of the class's [W][ld] arrays (coverage, gains)
};

// Where a kernel finds the descriptor of class l: a table in device memory, or (table == null)
// `L` classes of equal size laid out back to back.
struct DescSource {
    const ClassDesc *table;
    int32_t uniM, uniLd;
    __host__ __device__ ClassDesc get(int l) const
    {
        if (table) return table[l];
        ClassDesc c;
        c.M = uniM; c.ld = uniLd; c.row0 = l * uniM; c.pad_ = 0;
        c.sOff = (int64_t)l * uniM * uniLd; c.vOff = 0;
        return c;
    }
};

// The classes a similarity launch covers.
struct SimClasses {
    DescSource src;
    int32_t L;
    int64_t maxM;
    // tensor-core kernels: tiles that reach the diagonal or lie above it, listed class after class
    const int32_t *tilePrefixDev;   // [L+1] first tile index of every class (null: equal classes)
    int32_t uniTiles;               // tiles per class when the classes are equal
    int64_t upperTiles;             // tiles in all
    bool pairs;                     // tiles of 256 x 256 on pairs of SMs (see sim_pairs)
    bool clearStatus;               // the launch is a call of its own: its first CTA clears the status word (a memset in front of a
                                    // small call takes 2 us of 14)
};

// Pointers into the caller's workspace for one rcd_partition call.
struct Workspace {
    // grouping
    int32_t *counter;       // [4] zero when the call starts (classes drawn by the cluster form)
    unsigned long long *topGain;   // [L] zero when the call starts (cluster form)
    int32_t *counts;        // [L]
    int32_t *chunkHist;     // [nChunks][L]
    int32_t *perm;          // [N] class-sorted position -> dataset index
    void *Xs;               // [N][pitch] features in class-sorted order
    // per class
    ClassDesc *desc;        // [L]
    int32_t *tilePrefix;    // [L+1] first upper-triangle tile of every class (tensor-core similarity)
    void *S;                // similarity matrices
    void *gaussNorms;       // [N] squared norms of the class-sorted rows (int32 / float)
    double *gaussPartial;   // [L][ceil(maxM/64)] per-row-block sums of pairwise distances
    float *gaussSigma;      // [L] bandwidth of every class
    float *gaussScale;      // [L] 1 / (2 sigma^2)
    void *cutBase;          // [N] graph cut: column sum minus diagonal of every sample (int64 / double)
    void *cover;            // [sum W*ld] coverage vectors (int32 / float)
    void *gains;            // [sum W*ld] stored gains (int64 / float)
    void *fval;             // [L][W] tracked f (int64 / double)
    int32_t *cnt;           // [L][W]
    int32_t *quota;         // [L][W]
    uint8_t *valid;         // [L][W] 1 = stored gains of that block are current
    int32_t *cand;          // [N] unassigned samples of each class (class-local ids), compact
    int32_t *pos;           // [N] position of each sample in cand
    int32_t *nR;            // [L] unassigned count
    int32_t *jstar;         // [L] block chosen for the next pick (-1: none)
    int32_t *sweepN;        // [L] blocks to refresh in the next sweep (0: none)
    int32_t *sweepParts;    // [L][kSparseMax]
    int32_t *sweepMode;     // [L] dense / threshold pass
    void *thr;              // [sum ld] threshold vector of every class (int32 / float)
    unsigned long long *hitCount;   // [L]
    unsigned long long *sparseElems; // [L]
    int32_t *sparseFrom;    // [L]
    int32_t *sweepCS;       // [L] warps per row group in the next sweep
    int32_t *rowCtr;        // [L] ticket counter over row groups of the running sweep
    ClassSync *sync;        // [L] asynchronous kernel: hand-off words
    int32_t *tickets;       // [2N + L] asynchronous kernel: one ticket counter per (class, sweep number), never reused
    int32_t *sizesSorted;   // [L] class sizes, ascending
    int32_t *classOrder;    // [L] classes by descending size
    void *floorv;           // [L][kLazyBlocks] per block: every stored gain at or above it is exact (int64 / double)
    void *theta;            // [L][kLazyBlocks] per block: floor its next row-skipping pass will establish
    void *sweepTheta;       // [L][kLazyBlocks] floors of the blocks the class's next pass lists, in list order (int64 / fp32)
    int32_t *lazyStat;      // [L][4] row-skipping passes of the class, misses, members needed before rows are skipped
    long long *sweepF;      // [L][8] asynchronous kernel, int8 features: f of the first blocks in the sweep's list
    int32_t *sweepList;     // [3][L] classes that sweep in a step (three lists in rotation)
    int32_t *nSweep;        // [3] (+1 pad)
    unsigned long long *stepBytes;   // [2 maxM + 1] bytes the sweep of step t has to read
    unsigned long long *stepOps;     // [2 maxM + 1] element x block pairs of that sweep
    unsigned long long *phaseNs;     // [6] sweep-/pick-phase ns of the persistent kernel, barrier counter, threshold-pass hits / elements / max blocks
    long long *g0;          // [N] cluster form: gain of every sample for an empty block
    int32_t *fixedExp;      // [L] cluster form, floating-point similarities: S holds round(sim * 2^fixedExp), or kNotFixed
    int32_t *sizesLeft;     // [L] sizes of the classes marked kNotFixed, 0 for the others
    int32_t *status;        // [1]
    size_t bytes;           // total bytes laid out
};

// Words of rcd_ctx::statusOwn, and where the similarity kernel's tile tickets (zero between launches) begin.
constexpr int kStatusWords = 1024;
constexpr int kHistTicket = 32;            // label_hist_few_kernel's (zero between launches)
constexpr int kFirstTicket = 64;
// The staging buffer holds as many class sizes as a call may have, behind them the status words that come along, and last two words
// that the device writes: a class was left in floating point; the number of the last histogram whose sizes have arrived.
constexpr int kStageSpare = 1024, kStageLeft = kStageSpare - 1, kStageArrived = kStageSpare - 2;

// A class whose samples' norms lie too far apart for one fixed-point scale (see fixed_exponent_kernel).
constexpr int32_t kNotFixed = INT32_MIN;

struct Sizes {
    int64_t N, d;
    int32_t L, W;
    int64_t sElems;         // sum M_l * ld_l
    int64_t vElems;         // sum W * ld_l
    int64_t maxM;
    int32_t nChunks;
    int64_t pitch;          // bytes between rows of Xs
    bool floatArith;        // fp32 S / fp32 gains / double f (bf16 features, or the Gaussian kernel)
    bool graphCut;          // graph-cut objective: the gains array holds 8-byte ties
};

// Labels whose counters the class split keeps in shared memory: one per warp of a CTA and label, 192 KB.
constexpr int kMaxSharedLabels = 6000;
// Samples per chunk of the stable class split: small chunks while that is what fills the SMs, large ones where the table of
// chunks x labels, which is cleared and summed up on every call, would pass 64 MB (lists of 131072 samples over 20000 labels,
// 41 MB: 101 us, large chunks 126; over 100000, 205 MB: 923 us, large chunks 468).
inline int group_chunk(int64_t N, int64_t labels) { return N <= 131072 && (N + 255) / 256 * labels <= 1 << 24 ? 256 : 1024; }
// How a split goes about it: samples per chunk, threads per CTA, and whether every CTA adds up the numbers of all chunks by itself, which
// saves a memset, the launch of a scan and a copy.  With rows to gather (rows) up to 32 chunks and 4096 numbers (2 classes of 200: 148 -> 138
// us the whole call, 4 of 20 52 -> 40; with 9600 numbers, 300 classes of 27, the additions take longer than the scan, 79 us against 70).
// Lists alone have no rows to share out: their chunks are as large as gives an SM one, up to 16384 samples (1.3 million over 64 workers:
// 41 us with 1024 samples per chunk and a scan, 27 so; 80 samples 26 -> 20), and every CTA adds up where there are up to 1024 labels and
// 16384 numbers, with small chunks 8192: one warp finds where the labels begin (100 samples over 1024 labels 28 us, with the scan 32; over
// 2000 31 and 29, over 5000 63 and 31), and small CTAs take longer to add (4000 samples over 500 labels, 8000 numbers, 25.6 us, with the scan
// 27.8; over 1000 35 and 29; 20000 over 100 26.6 and 27.8, over 200 28.8 and 27.7).
struct GroupShape { int chunk, threads; bool few; };
inline GroupShape group_shape(int64_t N, int64_t labels, bool rows)
{
    GroupShape g{group_chunk(N, labels), 256, false};
    if (!rows && labels <= 1024 && N > 160 * 256) {
        g.chunk = (int)std::min<int64_t>((N + 144 * 1024 - 1) / (144 * 1024), 16) * 1024;
        g.threads = 1024;
    }
    const int64_t chunks = (N + g.chunk - 1) / g.chunk;
    g.few = N > 0 && labels <= kMaxSharedLabels && (rows ? chunks <= 32 && chunks * labels <= 4096
                                                                : chunks <= 144 && labels <= 1024 && chunks * labels <= (g.threads == 1024 ? 16384 : 8192));
    return g;
}
// Bytes between the class-sorted feature rows: whole 16-byte pieces, at least one 128-byte slab, so that every width can
// be loaded by the tensor-core kernel (the padding is zeros and adds nothing to a dot product).
inline int64_t row_pitch(int64_t rowBytes) { return rowBytes <= 128 ? 128 : (rowBytes + 15) / 16 * 16; }

inline size_t feat_bytes(rcd_feat_dtype t) { return t == RCD_FEAT_I8 ? 1 : 2; }
inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }
inline int32_t pad4(int64_t m) { return (int32_t)((m + 3) / 4 * 4); }
// Row pitch of S and of the per-block vectors inside rcd_partition / rcd_objective: a multiple of 8
// elements, so that every row starts on a 32-byte boundary (one memory sector): the 16-byte pieces that
// the sweeps copy then pair up into whole sectors.
inline int32_t pad_row(int64_t m) { return (int32_t)((m + 7) / 8 * 8); }

// Tiles the tensor-core similarity kernels compute for a class of M samples: those that reach the diagonal or lie above it, of
// 256 x 256 (pairs), or of 128 rows x 256 columns (row block tm with the column blocks from tm / 2 on).
inline int64_t sim_tiles(int64_t M, bool pairs)
{
    const int64_t rowBlocks = (M + 127) / 128, colBlocks = (M + 255) / 256;
    if (pairs) return colBlocks * (colBlocks + 1) / 2;
    int64_t n = 0;
    for (int64_t tm = 0; tm < rowBlocks; ++tm) n += colBlocks - tm / 2;
    return n;
}
// Units of work on pairs of SMs: tiles, as long as they fill rounds of one per pair; those left over are cut into 2, 4 or 8
// strips of columns, which share the last round out to more pairs (100 classes of 500 x 2048: 300 tiles on 74 pairs leave 4, a
// round of a quarter of a tile each instead of a whole one).
struct PairUnits { int whole, strips, count; };
__host__ __device__ inline PairUnits pair_units(int tiles, int pairs)
{
    PairUnits u;
    u.whole = tiles / pairs * pairs;
    u.strips = 1;
    while (u.strips < 8 && (tiles - u.whole) * u.strips * 2 <= pairs) u.strips *= 2;
    u.count = u.whole + (tiles - u.whole) * u.strips;
    return u;
}
// Whether pairs of SMs take a similarity launch: rows of at least 2 KB (40 classes of 1300 x 2048 bf16: 188 -> 170 us), or of
// 1 KB in classes of up to 1024 samples; in larger classes of such rows drawn tiles of half the size share the work out better
// (20 of 1300 x 1024 int8: 55 us, pairs 61), and below that writing S is the bound.  And where pairs need no more rounds, which
// take the same time: a tile a round, 0.7 of one for tiles in two strips, 0.5 for more (10 of 1025 x 2048: 2 rounds, 43 us;
// pairs 2.5 and 48).
inline bool sim_pairs(int64_t rowBytes, int64_t maxM, int64_t tiles, int64_t pairTiles, int sms)
{
    if (sms < 2 || maxM <= 128 || pairTiles > 0x7fffffffLL || (rowBytes < 2048 && (rowBytes < 1024 || maxM > 1024))) return false;
    const PairUnits u = pair_units((int)pairTiles, sms / 2);
    const double last = u.count == u.whole ? 0.0 : u.strips == 1 ? 1.0 : u.strips == 2 ? 0.7 : 0.5;
    return (double)(u.whole / (sms / 2)) + last <= (double)((tiles + sms - 1) / sms);
}

// The forms that find the next block by a warp-wide minimum keep a block's value as (value + kTrackedZero) << 7 | block in 64 bits, the
// topmost of which stays free: values have to lie below 2^55 either way.  Facility location does at any size these forms take (at most
// 65535 samples with entries below 2^31).  The graph cut's f(A) is a sum over |A| (M - |A|) <= M^2 / 4 entries of at most 2^14 d:
// what passes 2^55 (from 8193 samples of the largest width on, d = 131071, or 23171 of width 16384) is left to plain 64-bit integers.
// (Within that bound the gains fit the 48 bits of a key, too: three times a row's sum of |S| either way, up to 32768 samples.)
constexpr unsigned long long kTrackedZero = 1ull << 55;
inline bool cut_values_fit(int64_t maxM, int64_t d)
{
    return (unsigned __int128)maxM * (unsigned __int128)maxM / 4 * 16384 * (unsigned __int128)d < kTrackedZero;
}

// Lays the workspace out at `base` (may be null to measure).  Returns total bytes.
size_t layout_workspace(void *base, rcd_feat_dtype dtype, const Sizes &sz, Workspace *ws);

}  // namespace rcd

struct rcd_ctx {
    int device = 0;
    int smCount = 0;
    int maxSmemOptin = 0;
    bool cooperative = false;           // device supports cooperative launches
    rcd_config cfg{};
    std::string err;
    int32_t *hostStage = nullptr;       // pinned, counts / status read-back
    int32_t *statusOwn = nullptr;       // device status word for calls that take no workspace; from kFirstTicket on, tile tickets
    int32_t histTurn = 0;               // histograms of few numbers so far
    unsigned simReady = 0;              // tensor-core similarity kernels whose shared memory has been asked for, a bit each
    unsigned simTurn = 0;               // similarity launches so far: each takes the next ticket
    size_t hostStageInts = 0;
    unsigned char *hostBlob = nullptr;  // pinned, what a call's host side hands to its kernels
    size_t hostBlobBytes = 0;
    cudaEvent_t evBlob = nullptr;       // the last copy out of hostBlob
    cudaEvent_t evCounts = nullptr;     // the class sizes have arrived
    // profiling
    cudaEvent_t evPhase[5]{};           // start, after group, after similarity, after greedy, end
    bool phaseValid = false;
    std::vector<cudaEvent_t> evSweep;   // 2 per step
    int64_t sweepEventsUsed = 0;
    int64_t kernelLaunches = 0;
    int64_t tcLaunches = 0;
    int64_t steps = 0;
    int64_t greedyForm = 0;             // rcd_greedy_form of the last rcd_partition
    int64_t passes = 0;                 // entries of stepBytes / stepOps that count
    const unsigned long long *stepBytesDev = nullptr;
    const unsigned long long *stepOpsDev = nullptr;
    const unsigned long long *phaseNsDev = nullptr;
    const int32_t *statusDev = nullptr;
    int maxClusters[5] = {-1, -1, -1, -1, -1};   // clusters of 1, 2, 4, 8, 16 CTAs of the cluster form resident at once (-1: not asked yet)
    int lockClusters[5] = {-1, -1, -1, -1, -1};  // the same of the graph cut in step
};

namespace rcd {

// Whether the library chooses the form of the greedy loop: no pass-based form and none of their options asked for.
inline bool library_chooses(const rcd_config &c)
{
    return c.greedy_path == 0 && c.profile < 2 && c.sweep_batch_max == 0 && c.sweep_mode == 0 && c.async_group == 0 && c.async_help_min == 0 &&
           c.threshold_from == 0 && c.threshold_hit_shift == 0 && c.lazy_mode == 0 && c.lazy_from == 0 && c.dense_ring == 0 &&
           c.incremental == 0 && c.incremental_max == 0;
}

rcd_status fail(rcd_ctx *ctx, rcd_status st, const char *fmt, ...);
rcd_status cuda_fail(rcd_ctx *ctx, cudaError_t e, const char *what);

#define RCD_CUDA(ctx, call)                                            \
    do {                                                               \
        cudaError_t e__ = (call);                                      \
        if (e__ != cudaSuccess) return ::rcd::cuda_fail(ctx, e__, #call); \
    } while (0)

// Lets a kernel's launches take up to `most` bytes of dynamic shared memory: the most that any call may ask of it, which depends on the
// device alone.  The limit belongs to the function and so to all contexts and threads of the process: set to a call's own size, it can be
// lowered by another thread between this one's setting and its launch, which is then refused (lists for 1024 and 400 workers did that).
template <typename Kernel>
inline cudaError_t allow_shared(Kernel *kernel, int64_t most)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
// What a CTA with at most 1 KB of variables of its own in shared memory can be given besides.
inline int64_t whole_shared(const rcd_ctx *ctx) { return (int64_t)ctx->maxSmemOptin - 1024; }

// ---- launchers implemented in the .cu files (all asynchronous on `st`) ----

// class split
rcd_status launch_label_hist(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, int32_t *counts,
                             int32_t *status, int32_t *callStatus, cudaStream_t st);
rcd_status launch_label_hist_few(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, int32_t *counts, int32_t *status,
                                 int32_t *callStatus, int32_t *zeros, int64_t nZeros, int32_t *hostStatus, int32_t *hostCounts, cudaStream_t st);
rcd_status wait_few_counts(rcd_ctx *ctx, cudaStream_t st);
rcd_status launch_stable_split(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, const ClassDesc *descDev,
                               const int32_t *counts, int64_t *offsets, const int32_t *status, int32_t *perm,
                               const void *X, int64_t rowBytes, int64_t pitch, void *Xs, cudaStream_t st);

// similarity: S_l = Xs_l Xs_l^T for every class described by desc
rcd_status launch_similarity(rcd_ctx *ctx, const void *Xs, rcd_feat_dtype dtype, int64_t Ntot, int64_t d,
                             const SimClasses &cls, void *S, cudaStream_t st);

// In place of S, the coverage of every block: rows in block order within their class (blockOf[Ntot], -1: no block), cover[block][row]
// of a class at its vOff, zero at the start.  Tensor-core rows and cls.pairs false only.
rcd_status launch_similarity_maxima(rcd_ctx *ctx, const void *Xs, rcd_feat_dtype dtype, int64_t Ntot, int64_t d,
                                    const SimClasses &cls, const int32_t *blockOf, int32_t *cover, cudaStream_t st);

// Gaussian-kernel similarity: transforms the dot products in S in place, to fp32 or (fixedExp not null) to the fixed-point
// integers of the cluster form, whose scale it writes to fixedExp[l]
rcd_status launch_gaussian(rcd_ctx *ctx, const void *Xs, rcd_feat_dtype dtype, int64_t N, int64_t d, const SimClasses &cls,
                           void *S, void *norms, double *partial, float *sigma, float *scale, int32_t *fixedExp, cudaStream_t st);
size_t gaussian_scratch_bytes(int64_t N, int32_t L, int64_t maxM);

// greedy loop
rcd_status launch_greedy(rcd_ctx *ctx, rcd_feat_dtype dtype, const Sizes &sz, const Workspace &ws,
                         const std::vector<ClassDesc> &descHost, int32_t *assignment, int32_t *order,
                         cudaStream_t st);

// whether the forms with passes over S hold a class's coverage vector of one block in shared memory
rcd_status check_coverage_fits(rcd_ctx *ctx, int maxLd);

// the floating-point classes that the cluster form left (ws.fixedExp[l] == kNotFixed)
rcd_status launch_greedy_not_fixed(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                   int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st);

// greedy loop, one thread-block cluster per class: how it takes a problem (null: it does not), and the loop
struct ClusterPlan;
// (null: another form takes the problem; cutInStep: the graph cut in step does)
std::shared_ptr<ClusterPlan> plan_greedy_cluster(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, bool *cutInStep);
rcd_status launch_greedy_cluster(rcd_ctx *ctx, ClusterPlan &plan, const Sizes &sz, const Workspace &ws, const std::vector<ClassDesc> &descHost,
                                 int32_t *assignment, int32_t *order, void *partValues, cudaStream_t st);

// greedy loop in rounds, one CTA per class (null: it does not take the problem, or the cluster form would be faster)
struct RoundsPlan;
struct ClusterShape { int ctas, resident, pieces; };       // of the cluster form: CTAs per class (0: it does not take the problem), classes at a time, steps per row
std::shared_ptr<RoundsPlan> plan_greedy_rounds(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, const ClusterShape &cluster);
rcd_status launch_greedy_rounds(rcd_ctx *ctx, RoundsPlan &plan, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order,
                                void *partValues, cudaStream_t st);

bool rounds_possible(const rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost);

// greedy loop of small classes, one CTA per class with S in its shared memory (null: it does not take the problem; toFix: S holds
// floating-point dot products)
struct SmallPlan;
std::shared_ptr<SmallPlan> plan_greedy_small(rcd_ctx *ctx, const Sizes &sz);
rcd_status launch_greedy_small(rcd_ctx *ctx, SmallPlan &plan, const Sizes &sz, const Workspace &ws, bool toFix, int32_t *assignment, int32_t *order,
                               void *partValues, cudaStream_t st);

rcd_status launch_bounded_wait_selftest(rcd_ctx *ctx, unsigned *counter, int32_t *status, cudaStream_t st);
rcd_status launch_step_wait_selftest(rcd_ctx *ctx, int32_t *status, cudaStream_t st);

// graph-cut objective: the whole greedy loop, and f from an assignment (selftest: in step, on two CTAs, whatever the plan says)
rcd_status launch_cut_stopped_selftest(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, int32_t *assignment, int32_t *order, cudaStream_t st);
// (in step: integers, where that is faster than another form, which takes otherCycles; 0: one CTA per class)
bool cut_in_step(rcd_ctx *ctx, const Sizes &sz, const std::vector<ClassDesc> &descHost, double otherCycles);
rcd_status launch_cut(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, bool inStep, int32_t *assignment, int32_t *order, cudaStream_t st);
rcd_status launch_cut_objective(rcd_ctx *ctx, const Sizes &sz, const ClassDesc *descDev, const void *S, const int32_t *perm,
                                const int32_t *assignment, void *partValues, void *total, void *scratch, cudaStream_t st);

// objective from an assignment
// covered: the coverage is there already (launch_similarity_maxima), else it is taken from S
rcd_status launch_objective(rcd_ctx *ctx, rcd_feat_dtype dtype, const Sizes &sz, const Workspace &ws, const int32_t *assignment,
                            bool covered, void *partValues, void *total, cudaStream_t st);
// class-sorted positions in block order: ws.cand the dataset index, ws.pos the block (-1: none); ws.cover cleared
rcd_status launch_objective_order(rcd_ctx *ctx, const Sizes &sz, const Workspace &ws, const int32_t *assignment, cudaStream_t st);
// dst row r = row perm[r] of X, `pitch` bytes apart, zero-filled beyond rowBytes
rcd_status launch_gather_rows(rcd_ctx *ctx, const void *X, const int32_t *perm, int64_t N, int64_t rowBytes, int64_t pitch, void *dst, cudaStream_t st);


#ifdef __CUDACC__
// ---- warp-wide reductions of (value, index) pairs by 32-bit redux instead of shuffle ladders ----
// Order-preserving images in unsigned integers (a < b exactly when image(a) < image(b); -0.0 is taken as +0.0).
__device__ __forceinline__ unsigned long long ordered_u64(long long x) { return (unsigned long long)x ^ 0x8000000000000000ull; }
__device__ __forceinline__ unsigned long long ordered_u64(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x + 0.0);
    return b ^ ((b >> 63) ? ~0ull : 0x8000000000000000ull);
}
__device__ __forceinline__ unsigned ordered_u32(float x)
{
    const unsigned b = __float_as_uint(x + 0.0f);
    return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float from_ordered_u32(unsigned o) { return __uint_as_float(o ^ ((o >> 31) ? 0x80000000u : 0xffffffffu)); }

// Maximum of a 64-bit key over the warp (two 32-bit warp reductions: high words, then low words among the lanes that
// hold the greatest high word).
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long k)
{
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
    const unsigned mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
    return ((unsigned long long)mhi << 32) | mlo;
}
// Arg-maximum of (ordered image of the value, index) pairs over the warp: the greatest value, and among the lanes that
// hold it the lowest index; lanes without a candidate pass index INT_MAX.  Three warp-wide reductions.
__device__ __forceinline__ void warp_argmax_ordered(unsigned long long &ord, int &idx)
{
    const bool has = idx != 0x7fffffff;
    const unsigned hi = has ? (unsigned)(ord >> 32) : 0u, lo = has ? (unsigned)ord : 0u;
    const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
    const unsigned mlo = __reduce_max_sync(0xffffffffu, (has && hi == mhi) ? lo : 0u);
    const int mi = __reduce_min_sync(0xffffffffu, (has && hi == mhi && lo == mlo) ? idx : 0x7fffffff);
    ord = ((unsigned long long)mhi << 32) | mlo;
    idx = mi;
}
// The same for the least value (lowest index among equals).
__device__ __forceinline__ void warp_argmin_ordered(unsigned long long &ord, int &idx)
{
    unsigned long long inv = ~ord;
    warp_argmax_ordered(inv, idx);
    ord = ~inv;
}
__device__ __forceinline__ long long from_ordered_u64_ll(unsigned long long o) { return (long long)(o ^ 0x8000000000000000ull); }
__device__ __forceinline__ double from_ordered_u64_d(unsigned long long o)
{
    return __longlong_as_double((long long)(o ^ ((o >> 63) ? 0x8000000000000000ull : ~0ull)));
}
#endif

}  // namespace rcd
