// Class split (Algorithm 1: "Split the ground set V into L sets according to class labels"):
// label histogram, stable ranking of every sample inside its class, and the gather of the
// feature rows into class-sorted order.  Stable = inside a class the samples keep their
// dataset order, which is what fixes the lowest-index tie-breaks downstream.
#include "rcd_internal.h"

#include <algorithm>
#include <atomic>

namespace rcd {

// ---- stable split ---------------------------------------------------------------------------
// Chunks of consecutive samples (GroupShape says how large).  Three launches:
//   histogram  a CTA per chunk counts its labels in shared memory, writes chunkHist[chunk][label] and adds to counts[label];
//   scan       per label, exclusive running sum over the chunks, started at the class offset;
//   place      position = chunk base + rank inside the chunk; the CTA then copies its feature rows to their places.
// or two where few numbers come out: the histogram's last CTA hands the sizes to the host, and the placing CTAs add up for themselves.
// Up to kMaxSharedLabels labels the counters of a chunk sit in shared memory (a sample costs one shared-memory atomic
// and a few warp votes, against 1024 comparisons per sample and one global atomic before: 1.3 M samples over 64 labels
// 1155 -> 40 us, 27 in two launches).  More labels than that take the kernels at the end of this section.
constexpr int kGroupThreads = 256;
constexpr int kGroupWarps = kGroupThreads / 32;
// (histogram: a counter per label.  Placement: one per warp and label, with 32 warps up to 1024 labels (GroupShape), the labels' starts, and
// with rows the positions of up to 1024 samples)
static_assert(kMaxSharedLabels * 4 <= 48 * 1024, "a histogram's counters in the shared memory that every launch has");
static_assert((kGroupWarps + 1) * kMaxSharedLabels * 4 + 1024 * 4 <= 226 * 1024 && 33 * 1024 * 4 <= 226 * 1024, "counters in shared memory");

__global__ void __launch_bounds__(kGroupThreads) label_hist_kernel(const int32_t *__restrict__ labels, int64_t N, int32_t L, int32_t chunk,
                                                                  int32_t *__restrict__ chunkHist, int32_t *__restrict__ counts,
                                                                  int32_t *__restrict__ status, int32_t *__restrict__ callStatus)
{
    extern __shared__ int32_t shCount[];
    if (callStatus && blockIdx.x == 0 && threadIdx.x == 0) *callStatus = 0;       // (the word the later kernels report to)
    for (int l = threadIdx.x; l < L; l += kGroupThreads) shCount[l] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * chunk;
    const int n = (int)min((int64_t)chunk, N - base);
    bool bad = false;
    for (int i = threadIdx.x; i < n; i += kGroupThreads) {
        const int32_t lab = labels[base + i];
        if (lab < 0 || lab >= L) bad = true;
        else atomicAdd(&shCount[lab], 1);
    }
    if (bad) atomicOr(status, kDevBadLabel);
    __syncthreads();
    for (int l = threadIdx.x; l < L; l += kGroupThreads) {
        const int32_t c = shCount[l];
        chunkHist[(int64_t)blockIdx.x * L + l] = c;
        if (c) atomicAdd(&counts[l], c);
    }
}

// Adds the numbers of the first n chunks to sum[L] (shared memory): threads side by side take labels, and runs of chunks where labels are few.
__device__ __forceinline__ void add_chunks(const int32_t *chunkHist, int n, int32_t L, int32_t *sum)
{
    int parts = 1;
    while (2 * parts * L <= (int)blockDim.x) parts *= 2;
    const int per = (n + parts - 1) / parts;
    for (int i = threadIdx.x; i < parts * L; i += blockDim.x) {
        const int part = i / L, l = i - part * L;
        int32_t s = 0;
#pragma unroll 8
        for (int c = part * per; c < min(n, part * per + per); ++c) s += __ldcg(&chunkHist[(int64_t)c * L + l]);
        if (s) atomicAdd(&sum[l], s);
    }
}

// The same where few numbers come out (GroupShape::few): the CTA that is done last adds them up and writes the sizes and the verdict on the labels
// straight to the host's memory, so that neither a memset goes before this kernel nor a copy after it (4 of 52 us of the smallest calls).
// ticket: zero between launches (CTAs that are done, and from bit 16 on those that met a bad label).  zeros: words the later kernels
// want cleared.
__global__ void __launch_bounds__(1024) label_hist_few_kernel(const int32_t *__restrict__ labels, int64_t N, int32_t L, int32_t chunk,
                                                                      int32_t *__restrict__ chunkHist, int32_t *__restrict__ counts, int32_t *__restrict__ status,
                                                                      int32_t *__restrict__ callStatus, int32_t *__restrict__ zeros, int32_t nZeros,
                                                                      uint32_t *__restrict__ ticket, volatile int32_t *hostStatus, volatile int32_t *hostCounts,
                                                                      volatile int32_t *hostArrived, int32_t turn)
{
    extern __shared__ int32_t shCount[];
    __shared__ uint32_t shDone;
    if (blockIdx.x == 0) {
        if (callStatus && threadIdx.x == 0) *callStatus = 0;
        for (int i = threadIdx.x; i < nZeros; i += blockDim.x) zeros[i] = 0;
    }
    for (int l = threadIdx.x; l < L; l += blockDim.x) shCount[l] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * chunk;
    const int n = (int)min((int64_t)chunk, N - base);
    bool bad = false;
#pragma unroll 8
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int32_t lab = labels[base + i];
        if (lab < 0 || lab >= L) bad = true;
        else atomicAdd(&shCount[lab], 1);
    }
    bad = __syncthreads_or(bad);
    for (int l = threadIdx.x; l < L; l += blockDim.x) __stcg(&chunkHist[(int64_t)blockIdx.x * L + l], shCount[l]);
    if (gridDim.x > 1) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) shDone = atomicAdd(ticket, bad ? 0x10001u : 1u) + (bad ? 0x10001u : 1u);
        __syncthreads();
        if ((shDone & 0xffffu) != gridDim.x) return;
        __threadfence();
        bad = shDone >> 16 != 0;
        for (int l = threadIdx.x; l < L; l += blockDim.x) shCount[l] = 0;
        __syncthreads();
        add_chunks(chunkHist, (int)gridDim.x, L, shCount);
        __syncthreads();
    }
    for (int l = threadIdx.x; l < L; l += blockDim.x) {
        counts[l] = shCount[l];
        if (hostCounts) hostCounts[l] = shCount[l];
    }
    if (threadIdx.x == 0) {
        *status = bad ? kDevBadLabel : 0;
        *hostStatus = bad ? kDevBadLabel : 0;
        if (gridDim.x > 1) *ticket = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_system();                            // (for what the others wrote, too)
        *hostArrived = turn;
    }
}

// Exclusive sums over the chunks for 32 labels per CTA: thread (x, y) takes label x and the y-th of 32 runs of chunks.
// start: where label l begins (desc[l].row0), or null: after the counts of the labels below it.
__global__ void __launch_bounds__(1024) label_scan_kernel(int32_t *__restrict__ chunkHist, int32_t nChunks, int32_t L,
                                                         const ClassDesc *__restrict__ desc, const int32_t *__restrict__ counts,
                                                         int64_t *__restrict__ offsets, const int32_t *__restrict__ status)
{
    __shared__ int32_t shRun[32][33];
    __shared__ int32_t shStart[33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int l = blockIdx.x * 32 + x;
    const int per = (nChunks + 31) / 32;
    const int c0 = min(nChunks, y * per), c1 = min(nChunks, c0 + per);
    int32_t sum = 0;
    if (l < L)
        for (int c = c0; c < c1; ++c) sum += chunkHist[(int64_t)c * L + l];
    shRun[y][x] = sum;
    if (!desc) {
        // labels below this CTA's, by its first warp; then the 32 of its own
        if (y == 0) {
            int32_t below = 0;
            for (int i = x; i < (int)blockIdx.x * 32; i += 32) below += counts[i];
            below = __reduce_add_sync(0xffffffffu, below);
            int32_t run = l < L ? counts[l] : 0;
            const int32_t own = run;
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t up = __shfl_up_sync(0xffffffffu, run, off);
                if (x >= off) run += up;
            }
            shStart[x] = below + run - own;
            if (offsets && !(*status & kDevBadLabel)) {
                if (l < L) offsets[l] = below + run - own;
                if (l == L - 1) offsets[L] = below + run;
            }
        }
    } else if (y == 0) {
        shStart[x] = l < L ? desc[l].row0 : 0;
    }
    __syncthreads();
    if (y == 0) {
        int32_t run = shStart[x];
        for (int k = 0; k < 32; ++k) {
            const int32_t h = shRun[k][x];
            shRun[k][x] = run;
            run += h;
        }
    }
    __syncthreads();
    if (l < L) {
        int32_t run = shRun[y][x];
        for (int c = c0; c < c1; ++c) {
            const int64_t at = (int64_t)c * L + l;
            const int32_t h = chunkHist[at];
            chunkHist[at] = run;
            run += h;
        }
    }
}

// Copies one row of `bytes` to a row of `pitch` >= bytes (the rest zeros) by one warp.
__device__ __forceinline__ void copy_row(const uint8_t *__restrict__ src, uint8_t *__restrict__ dst, int64_t bytes, int64_t pitch, bool vec, int lane)
{
    if (vec) {
        const int4 *s = reinterpret_cast<const int4 *>(src);
        int4 *d = reinterpret_cast<int4 *>(dst);
        const int n = (int)(bytes >> 4), np = (int)(pitch >> 4);
        int i = lane;
        for (; i + 96 < n; i += 128) {
            const int4 a = __ldg(s + i), b = __ldg(s + i + 32), c = __ldg(s + i + 64), e = __ldg(s + i + 96);
            d[i] = a; d[i + 32] = b; d[i + 64] = c; d[i + 96] = e;
        }
        for (; i < np; i += 32) d[i] = i < n ? __ldg(s + i) : make_int4(0, 0, 0, 0);
    } else if (pitch % 16 == 0 && ((uintptr_t)dst) % 16 == 0) {
        // rows that start anywhere: 16 bytes of the copy from the five aligned words that hold them (only words with a byte of
        // the row in them are read).  Byte by byte a row of 2.7 KB took a warp 30 us.
        const uint32_t *s = reinterpret_cast<const uint32_t *>((uintptr_t)src & ~(uintptr_t)3);
        const int off = (int)((uintptr_t)src & 3), words = (int)((off + bytes + 3) >> 2), np = (int)(pitch >> 4);
        int4 *d = reinterpret_cast<int4 *>(dst);
#pragma unroll 2
        for (int i = lane; i < np; i += 32) {
            uint32_t w[5], o[4];
#pragma unroll
            for (int e = 0; e < 5; ++e) w[e] = 4 * i + e < words ? __ldg(s + 4 * i + e) : 0u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t left = bytes - 16 * (int64_t)i - 4 * e;            // bytes of the row from this word on
                const uint32_t x = __funnelshift_r(w[e], w[e + 1], 8 * off);
                o[e] = left >= 4 ? x : left <= 0 ? 0u : x & ((1u << (8 * (int)left)) - 1u);
            }
            d[i] = make_int4((int)o[0], (int)o[1], (int)o[2], (int)o[3]);
        }
    } else {
        for (int64_t i = lane; i < pitch; i += 32) dst[i] = i < bytes ? src[i] : (uint8_t)0;
    }
}

// The lanes with the same label, by its bits from the lowest up (`bits` ballots of 24 cycles that overlap; __match_any_sync takes 375).
__device__ __forceinline__ unsigned same_label(int lab, int bits)
{
    unsigned same = 0xffffffffu;
    for (int k = 0; k < bits; ++k) {
        const bool set = lab >> k & 1;
        const unsigned votes = __ballot_sync(0xffffffffu, set);
        same &= set ? votes : ~votes;
    }
    return same;
}

// kFew: no launch of label_scan_kernel before; chunkBase holds the chunks' own numbers, and every CTA adds up those before its own (null
// desc: counts says where the labels begin).  The number of threads and kFew are fixed at compile time, and five CTAs of 256 have to fit an
// SM: rows are copied by as many warps as there are.  One kernel for all of them, bounded by 1024 threads, took 64 registers instead of 48,
// and the split of 1.3 million rows of 2 KB over 1000 labels 1085 us (now 940), that of 81920 rows of 130 bytes over 4096 labels 186 (160),
// lists of 1.3 million samples over 5000 workers 156 (124).  (A run of 256 threads' samples has four per lane: counted all at once.)
template <int kThreads, bool kFew>
__global__ void __launch_bounds__(kThreads, kThreads == 1024 ? 1 : 5) label_place_kernel(const int32_t *__restrict__ labels, int64_t N, int32_t L, int32_t chunk,
                                                                   const int32_t *__restrict__ chunkBase, int32_t *__restrict__ perm,
                                                                   const uint8_t *__restrict__ X, int64_t rowBytes, int64_t pitch,
                                                                   uint8_t *__restrict__ Xs, const int32_t *__restrict__ status,
                                                                   const ClassDesc *__restrict__ desc, const int32_t *__restrict__ counts, int64_t *__restrict__ offsets)
{
    extern __shared__ int32_t shWarp[];                 // [warps][L] counters, then [chunk] positions
    if (status && (*status & kDevBadLabel)) return;
    constexpr int warps = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *mine = shWarp + (size_t)warp * L;
    int32_t *shPos = shWarp + (size_t)warps * L;
    const int64_t base = (int64_t)blockIdx.x * chunk;
    const int n = (int)min((int64_t)chunk, N - base);
    const int per = chunk / warps;                // a warp's run of consecutive samples (a multiple of 32)
    for (int l = lane; l < L; l += 32) mine[l] = 0;
    __syncwarp();
    const int i0 = warp * per, i1 = min(n, i0 + per);
#pragma unroll (kThreads == 1024 ? 8 : 4)
    for (int i = i0 + lane; i < i1; i += 32) atomicAdd(&mine[labels[base + i]], 1);
    __syncthreads();
    int32_t *const shStart = shWarp + (size_t)warps * L + (Xs ? chunk : 0);      // [L] where a label begins (kFew), then where the chunk's part of it does
    if (kFew && !desc) {
        if (warp == 0) {
            int32_t run = 0;
            for (int l0 = 0; l0 < L; l0 += 32) {
                const int32_t own = l0 + lane < L ? counts[l0 + lane] : 0;
                int32_t sum = own;
                for (int off = 1; off < 32; off <<= 1) {
                    const int32_t up = __shfl_up_sync(0xffffffffu, sum, off);
                    if (lane >= off) sum += up;
                }
                if (l0 + lane < L) {
                    shStart[l0 + lane] = run + sum - own;
                    if (offsets && blockIdx.x == 0 && blockIdx.y == 0) offsets[l0 + lane] = run + sum - own;
                }
                run += __shfl_sync(0xffffffffu, sum, 31);
            }
            if (offsets && blockIdx.x == 0 && blockIdx.y == 0 && lane == 0) offsets[L] = run;
        }
        __syncthreads();
    }
    if (kFew) {
        if (desc) {
            for (int l = threadIdx.x; l < L; l += kThreads) shStart[l] = desc[l].row0;
            __syncthreads();
        }
        add_chunks(chunkBase, (int)blockIdx.x, L, shStart);
        __syncthreads();
    }
    for (int l = threadIdx.x; l < L; l += kThreads) {
        int32_t run = kFew ? shStart[l] : chunkBase[(int64_t)blockIdx.x * L + l];
        for (int w = 0; w < warps; ++w) {
            const int32_t c = shWarp[(size_t)w * L + l];
            shWarp[(size_t)w * L + l] = run;
            run += c;
        }
    }
    __syncthreads();
    const int labelBits = 32 - __clz(L);                // (-1 for lanes without a sample differs from every label there)
    for (int i = i0; i < i1; i += 32) {
        const bool in = i + lane < i1;
        const int32_t lab = in ? labels[base + i + lane] : -1;
        const unsigned same = same_label(lab, labelBits);
        const int rank = __popc(same & ((1u << lane) - 1u));
        int32_t pos = 0;
        if (in) pos = mine[lab] + rank;
        __syncwarp();
        if (in && rank == 0) mine[lab] = pos + __popc(same);
        __syncwarp();
        if (in) {
            if (blockIdx.y == 0) perm[pos] = (int32_t)(base + i + lane);
            if (Xs) shPos[i + lane] = pos;
        }
    }
    if (!Xs) return;
    __syncthreads();
    const bool vec = rowBytes % 16 == 0 && pitch % 16 == 0 && ((uintptr_t)X) % 16 == 0 && ((uintptr_t)Xs) % 16 == 0;
    for (int i = warp + blockIdx.y * warps; i < n; i += warps * gridDim.y)
        copy_row(X + (base + i) * rowBytes, Xs + (int64_t)shPos[i] * pitch, rowBytes, pitch, vec, lane);
}

// ---- more labels than fit shared memory ------------------------------------------------------
__global__ void count_labels_kernel(const int32_t *__restrict__ labels, int64_t N, int32_t L,
                                    int32_t *__restrict__ counts, int32_t *__restrict__ status, int32_t *__restrict__ callStatus)
{
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    if (callStatus && blockIdx.x == 0 && threadIdx.x == 0) *callStatus = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
        int32_t lab = labels[i];
        if (lab < 0 || lab >= L) { bad = true; continue; }
        atomicAdd(&counts[lab], 1);
    }
    if (bad) atomicOr(status, kDevBadLabel);
}

__device__ __forceinline__ void chunk_rank(const int32_t *sh, int n, int t, int lab, int &rank, bool &last)
{
    rank = 0;
    last = true;
    for (int i = 0; i < n; ++i) {
        int other = sh[i];
        if (other == lab) {
            if (i < t) ++rank;
            if (i > t) last = false;
        }
    }
}

// hist: writes how many samples of the label the chunk holds (by the chunk's last sample of the label); else: places
template <bool kHist>
__global__ void __launch_bounds__(1024, 1) chunk_rank_kernel(const int32_t *__restrict__ labels, int64_t N, int32_t L, int32_t chunk,
                                                            int32_t *__restrict__ chunkHist, int32_t *__restrict__ perm, const int32_t *__restrict__ status)
{
    __shared__ int32_t sh[1024];
    if (!kHist && status && (*status & kDevBadLabel)) return;
    int64_t base = (int64_t)blockIdx.x * chunk;
    int n = (int)min((int64_t)chunk, N - base);
    int t = threadIdx.x;
    int lab = -1;
    if (t < n) lab = labels[base + t];
    sh[t] = lab;
    __syncthreads();
    if (t < n && lab >= 0 && lab < L) {
        int rank; bool last;
        chunk_rank(sh, n, t, lab, rank, last);
        const int64_t at = (int64_t)blockIdx.x * L + lab;
        if (!kHist) perm[chunkHist[at] + rank] = (int32_t)(base + t);
        else if (last) chunkHist[at] = rank + 1;
    }
}

// Rows of up to 512 bytes are moved eight at a time by a warp, which then reads eight indices at once and has a piece of a row on its way
// per lane (130000 rows of 64 bytes: 23.6 us a row at a time, 9.9 so).  Wider ones keep a warp busy by themselves.
constexpr int kGatherRows = 8, kNarrowRow = 512;
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint8_t *__restrict__ X, const int32_t *__restrict__ perm, int64_t N,
                                                          int64_t rowBytes, int64_t pitch, uint8_t *__restrict__ Xs)
{
    const int lane = threadIdx.x & 31;
    const bool vec = rowBytes % 16 == 0 && pitch % 16 == 0 && ((uintptr_t)X) % 16 == 0 && ((uintptr_t)Xs) % 16 == 0;
    if (vec && pitch <= kNarrowRow) {
        const int np = (int)(pitch >> 4), nx = (int)(rowBytes >> 4);
        for (int64_t r0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * kGatherRows; r0 < N; r0 += (int64_t)gridDim.x * 8 * kGatherRows) {
            const int pieces = (int)min((int64_t)kGatherRows, N - r0) * np;
            const int32_t mine = lane < kGatherRows && r0 + lane < N ? perm[r0 + lane] : 0;
            int4 *const to = reinterpret_cast<int4 *>(Xs + r0 * pitch);
#pragma unroll 4
            for (int q0 = 0; q0 < pieces; q0 += 32) {
                const int q = q0 + lane, row = q / np, piece = q - row * np;
                const int64_t from = __shfl_sync(0xffffffffu, mine, row & (kGatherRows - 1));
                if (q < pieces) to[q] = piece < nx ? __ldg(reinterpret_cast<const int4 *>(X + from * rowBytes) + piece) : make_int4(0, 0, 0, 0);
            }
        }
        return;
    }
    for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < N; r += (int64_t)gridDim.x * 8)
        copy_row(X + (int64_t)perm[r] * rowBytes, Xs + r * pitch, rowBytes, pitch, vec, lane);
}

static bool shared_labels(int32_t L) { return L <= kMaxSharedLabels; }

// Histogram of few numbers (GroupShape::few): the verdict on the labels and, unless null, the sizes arrive in pinned memory (wait_few_counts).
rcd_status launch_label_hist_few(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, int32_t *counts, int32_t *status,
                                 int32_t *callStatus, int32_t *zeros, int64_t nZeros, int32_t *hostStatus, int32_t *hostCounts, cudaStream_t st)
{
    const int chunk = shape.chunk;
    const size_t smem = (size_t)L * 4;
    label_hist_few_kernel<<<(unsigned)((N + chunk - 1) / chunk), shape.threads, smem, st>>>(labels, N, L, chunk, chunkHist, counts, status, callStatus, zeros, (int32_t)nZeros,
                                                                                     (uint32_t *)(ctx->statusOwn + kHistTicket), hostStatus, hostCounts,
                                                                                     ctx->hostStage + ctx->hostStageInts + kStageArrived, ++ctx->histTurn);
    ctx->kernelLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

// Waits for them: the kernel's last word is looked at directly, which is some microseconds sooner than an event behind the kernel.
rcd_status wait_few_counts(rcd_ctx *ctx, cudaStream_t st)
{
    volatile int32_t *const arrived = ctx->hostStage + ctx->hostStageInts + kStageArrived;
    for (unsigned k = 1; *arrived != ctx->histTurn; ++k)
        if (k % 65536 == 0) {                              // (a kernel that failed says nothing)
            const cudaError_t e = cudaStreamQuery(st);
            if (e == cudaSuccess && *arrived != ctx->histTurn) return fail(ctx, RCD_ERR_INTERNAL, "the class sizes did not arrive");
            if (e != cudaSuccess && e != cudaErrorNotReady) return cuda_fail(ctx, e, "waiting for the class sizes");
        }
    std::atomic_thread_fence(std::memory_order_acquire);
    return RCD_OK;
}

// Histogram of the labels: counts[L] (zeroed by the caller, like *status), and per chunk.
rcd_status launch_label_hist(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, int32_t *counts,
                             int32_t *status, int32_t *callStatus, cudaStream_t st)
{
    if (N == 0) {
        if (callStatus) RCD_CUDA(ctx, cudaMemsetAsync(callStatus, 0, sizeof(int32_t), st));
        return RCD_OK;
    }
    const int chunk = shape.chunk;
    const unsigned nChunks = (unsigned)((N + chunk - 1) / chunk);
    if (shared_labels(L)) {
        const size_t smem = (size_t)L * 4;
        label_hist_kernel<<<nChunks, kGroupThreads, smem, st>>>(labels, N, L, chunk, chunkHist, counts, status, callStatus);
        ctx->kernelLaunches++;
    } else {
        const unsigned blocks = (unsigned)std::min<int64_t>((N + 255) / 256, 4LL * ctx->smCount);
        count_labels_kernel<<<blocks, 256, 0, st>>>(labels, N, L, counts, status, callStatus);
        RCD_CUDA(ctx, cudaMemsetAsync(chunkHist, 0, (size_t)nChunks * L * sizeof(int32_t), st));
        chunk_rank_kernel<true><<<nChunks, 1024, 0, st>>>(labels, N, L, chunk, chunkHist, nullptr, nullptr);
        ctx->kernelLaunches += 2;
    }
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

rcd_status launch_gather_rows(rcd_ctx *ctx, const void *X, const int32_t *perm, int64_t N, int64_t rowBytes, int64_t pitch, void *dst, cudaStream_t st)
{
    if (N == 0) return RCD_OK;
    const unsigned blocks = (unsigned)std::min<int64_t>((N + 7) / 8, 32LL * ctx->smCount);
    gather_rows_kernel<<<blocks, 256, 0, st>>>((const uint8_t *)X, perm, N, rowBytes, pitch, (uint8_t *)dst);
    ctx->kernelLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

// Stable split after launch_label_hist: perm, and with X the rows in split order (Xs, `pitch` bytes apart, zero-filled
// beyond rowBytes).  desc null: label l starts after the counts of the labels below it; the starts go to offsets[L + 1].
rcd_status launch_stable_split(rcd_ctx *ctx, const int32_t *labels, int64_t N, int32_t L, const GroupShape &shape, int32_t *chunkHist, const ClassDesc *descDev,
                               const int32_t *counts, int64_t *offsets, const int32_t *status, int32_t *perm,
                               const void *X, int64_t rowBytes, int64_t pitch, void *Xs, cudaStream_t st)
{
    if (N == 0) {
        if (offsets) RCD_CUDA(ctx, cudaMemsetAsync(offsets, 0, (size_t)(L + 1) * sizeof(int64_t), st));
        return RCD_OK;
    }
    const int chunk = shape.chunk;
    const int nChunks = (int)((N + chunk - 1) / chunk);
    const bool few = shape.few;
    if (!few) {
        label_scan_kernel<<<(L + 31) / 32, 1024, 0, st>>>(chunkHist, nChunks, L, descDev, counts, offsets, status);
        ctx->kernelLaunches++;
    }
    if (shared_labels(L)) {
        const size_t smem = ((size_t)shape.threads / 32 * L + (Xs ? chunk : 0) + (few ? L : 0)) * 4;
        auto *const kernel = shape.threads == 1024 ? (few ? label_place_kernel<1024, true> : label_place_kernel<1024, false>)
                                                   : (few ? label_place_kernel<kGroupThreads, true> : label_place_kernel<kGroupThreads, false>);
        if (smem > 48 * 1024) RCD_CUDA(ctx, allow_shared(kernel, whole_shared(ctx)));
        // (few samples: several CTAs rank the same chunk and share its rows out, so that wide rows occupy more than a few SMs)
        const dim3 grid(nChunks, Xs ? std::max(1, std::min(16, 2 * ctx->smCount / nChunks)) : 1);
        kernel<<<grid, shape.threads, smem, st>>>(labels, N, L, chunk, chunkHist, perm, (const uint8_t *)X, rowBytes, pitch, (uint8_t *)Xs, status,
                                                  descDev, counts, few ? offsets : nullptr);
        ctx->kernelLaunches++;
    } else {
        chunk_rank_kernel<false><<<nChunks, 1024, 0, st>>>(labels, N, L, chunk, chunkHist, perm, status);
        ctx->kernelLaunches++;
        if (Xs) return launch_gather_rows(ctx, X, perm, N, rowBytes, pitch, Xs, st);
    }
    RCD_CUDA(ctx, cudaGetLastError());
    return RCD_OK;
}

}  // namespace rcd
