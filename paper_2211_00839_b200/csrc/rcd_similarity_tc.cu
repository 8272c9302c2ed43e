// Tensor-core similarity kernel for sm_100a:  S_l = X_l X_l^T  per class (Section 3.1: similarities
// from the feature vectors; int8 -> int32 exact, bf16 -> fp32).
//
// Persistent CTAs (one per SM) take tiles of 128 rows x 256 columns of every class, those that reach the
// diagonal or lie above it; S is symmetric, so each 128 x 128 block above the diagonal is computed once
// and written twice (itself and its mirror image), which halves the tensor work and the operand traffic
// (a tile whose left half lies below the diagonal computes its right half only).  The tile is twice as wide
// as it is high because the kernel is bound by operand traffic from L2 at 128 x 128 (512 bytes of operands
// per 32 768 multiply-adds and k-step): 128 x 256 moves 768 bytes per 65 536.  Both operands are rows of
// the class-sorted feature matrix (K-major), brought in 128-byte k-slabs by TMA (cp.async.bulk.tensor,
// 128-byte swizzle, out-of-range rows and columns filled with zeros) into a 4-stage shared-memory
// ring; one thread issues tcgen05.mma (kind::i8, or kind::f16 with bf16 inputs) into one of two
// 256-column accumulator buffers in tensor memory, so the next tile's MMAs run while eight warps read the
// previous accumulator back with tcgen05.ld, transpose 32 x 32 blocks through shared memory and
// write S with coalesced 128-bit stores (pad columns as zeros).
//
// Warp roles: 0 = TMA producer, 1 = TMEM allocation + MMA issue, 2..9 = epilogue (two warps per quarter of the
// tensor-memory lanes, one taking the even 32-column blocks of a tile and one the odd ones; the load of a warp's
// next block from tensor memory is in flight while it writes the current one).
// Every wait on an mbarrier is bounded: on expiry the CTA records kDevTimeout in the status
// word, stops issuing work, still waits (bounded) for the copies it has in flight, releases its
// tensor memory and returns.
#include "rcd_internal.h"

#include <cuda.h>

#include <algorithm>

namespace rcd {

namespace {

constexpr int kTileM = 128;
constexpr int kTileN = 256;
constexpr int kSlabBytes = 128;                         // k-slab per stage and operand row
constexpr int kStages = 4;
constexpr int kOperandBytes = kTileM * kSlabBytes;      // 16 KB: 128 rows of one k-slab
constexpr int kStageBytes = 3 * kOperandBytes;          // A (128 rows) + B (256 rows)
constexpr int kTileSlots = 2;                           // tiles between the producer, which draws them, and the other roles
constexpr int kEpiWarps = 8;                            // two per quarter of the TMEM lanes
constexpr int kTcThreads = 64 + 32 * kEpiWarps;
constexpr int kTmemCols = 512;                           // two accumulator buffers of 256 columns
constexpr uint32_t kSpinLimit = 1u << 22;               // polls of ~64 ns: a quarter of a second

struct TileCoord { int l, tm, sn, skip, n; };         // n: columns computed, from column sn * 256 + skip on
struct __align__(8) TileSlot {                          // a tile the producer has drawn
    TileCoord t;                                        // (t.l < 0: no more)
    ClassDesc c;
};

struct __align__(8) TcShared {
    uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t accFull[2];
    uint64_t accEmpty[2];
    uint64_t tileFull[kTileSlots];
    uint64_t tileEmpty[kTileSlots];
    TileSlot tile[kTileSlots];
    uint32_t tmemBase;
    int32_t abort;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (and raises the CTA's abort flag) when the limit is reached or
// another role has already given up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, TcShared *sh)
{
    for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
        if (mbar_test(bar, parity)) return true;
        if (spin > 64) {
            if (*(volatile int32_t *)&sh->abort) return false;
            __nanosleep(64);
        }
    }
    atomicExch(&sh->abort, 1);
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(smem_addr(dst)), "l"(map), "r"(c0), "r"(c1), "r"(smem_addr(bar)) : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 bytes apart,
// groups of 8 rows 1024 bytes apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3ffff) >> 4);             // start address, 16-byte units
    d |= (uint64_t)1 << 16;                             // leading byte offset (unused with 128-byte swizzle, K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                   // stride byte offset: next 8-row group
    d |= (uint64_t)1 << 46;                             // descriptor version for sm_100
    d |= (uint64_t)2 << 61;                             // layout type: 128-byte swizzle
    return d;
}

template <bool kInt8>
__device__ __forceinline__ void mma_issue(uint32_t tmemD, uint64_t descA, uint64_t descB, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (kInt8) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(tmemD), "l"(descA), "l"(descB), "r"(idesc), "r"(accumulate) : "memory");
    } else {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(tmemD), "l"(descA), "l"(descB), "r"(idesc), "r"(accumulate) : "memory");
    }
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void tmem_load_32cols(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr) : "memory");
}
// The registers of an earlier tmem_load_32cols hold their values only after this wait.
__device__ __forceinline__ void tmem_load_wait()
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_addr(bar)) : "memory");
}

// Tile idx of the launch -> (class, row block tm of 128 rows, column block sn of 256 columns).  The tiles of a class are
// those with sn >= tm / 2, which contain a 128 x 128 block on or above the diagonal.  skip = 128 when the left half of the
// tile lies below the diagonal (tm odd, sn = tm / 2): that half is the mirror image of a block another tile computes, so
// only the right half is computed.
__device__ __forceinline__ TileCoord decode_tile(const DescSource &src, const int32_t *__restrict__ prefix, int L, int uniTiles, int idx)
{
    TileCoord t;
    int local;
    if (prefix) {
        int lo = 0, hi = L;                              // prefix[lo] <= idx < prefix[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (prefix[mid] <= idx) lo = mid; else hi = mid;
        }
        t.l = lo;
        local = idx - prefix[lo];
    } else {
        t.l = idx / uniTiles;
        local = idx - t.l * uniTiles;
    }
    const ClassDesc c = src.get(t.l);
    const int colBlocks = (c.M + kTileN - 1) / kTileN;
    t.tm = 0;
    for (;;) {
        const int rowLen = colBlocks - t.tm / 2;
        if (local < rowLen) break;
        local -= rowLen;
        ++t.tm;
    }
    t.sn = t.tm / 2 + local;
    t.skip = (2 * t.sn < t.tm) ? kTileM : 0;
    // no further than the rows of S reach, pad columns included (in steps of 32 columns: the epilogue's block, and a
    // legal N of the MMA)
    t.n = min(kTileN - t.skip, (c.ld - (t.sn * kTileN + t.skip) + 31) & ~31);
    return t;
}

// An epilogue warp's column blocks (every other one of a tile's, from `half` on) -> S: the 32 rows from row0 on in 32 x 32
// blocks, transposed through shared memory, and the mirror image of those that are mirrored.  v: the first block, on its way.
template <typename Mirrored>
__device__ __forceinline__ void write_columns(uint32_t (*stage)[33], uint32_t *Sl, const ClassDesc &c, int row0, int colB, uint32_t tmemRow,
                                              int half, int nCb, uint32_t (&v)[32], Mirrored mirrored)
{
    const int lane = threadIdx.x & 31;
    const int cg = (lane & 7) * 4;                             // this lane's 4 columns of a 32-wide block
#pragma unroll 1
    for (int cb = half; cb < nCb; cb += kEpiWarps / 4) {
        tmem_load_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) stage[lane][j] = v[j];         // lane = row inside the quarter
        __syncwarp();
        // the next block of this warp travels from tensor memory while this one is written out
        if (cb + kEpiWarps / 4 < nCb) tmem_load_32cols(tmemRow + (uint32_t)((cb + kEpiWarps / 4) * 32), v);
        // block rows -> S[rowA + ..][colB + ..]: 8 lanes cover 32 columns with 128-bit stores, 4 rows per pass
        {
            const int col = colB + cb * 32 + cg;
#pragma unroll
            for (int pass = 0; pass < 8; ++pass) {
                const int r = pass * 4 + (lane >> 3);
                const int row = row0 + r;
                if (row < c.M && col < c.ld) {
                    uint4 o;
                    o.x = col + 0 < c.M ? stage[r][cg + 0] : 0u;
                    o.y = col + 1 < c.M ? stage[r][cg + 1] : 0u;
                    o.z = col + 2 < c.M ? stage[r][cg + 2] : 0u;
                    o.w = col + 3 < c.M ? stage[r][cg + 3] : 0u;
                    *reinterpret_cast<uint4 *>(Sl + (int64_t)row * c.ld + col) = o;
                }
            }
        }
        // the mirrored block -> S[colB + ..][rowA + ..] (blocks below the diagonal are never computed)
        if (mirrored(cb)) {
            const int col = row0 + cg;
#pragma unroll
            for (int pass = 0; pass < 8; ++pass) {
                const int jj = pass * 4 + (lane >> 3);
                const int row = colB + cb * 32 + jj;
                if (row < c.M && col < c.ld) {
                    uint4 o;
                    o.x = col + 0 < c.M ? stage[cg + 0][jj] : 0u;
                    o.y = col + 1 < c.M ? stage[cg + 1][jj] : 0u;
                    o.z = col + 2 < c.M ? stage[cg + 2][jj] : 0u;
                    o.w = col + 3 < c.M ? stage[cg + 3][jj] : 0u;
                    *reinterpret_cast<uint4 *>(Sl + (int64_t)row * c.ld + col) = o;
                }
            }
        }
        __syncwarp();
    }
}

// Where a tile's columns or rows belong, for the maxima: lane j holds the block of column (row) j of 32, -1: none.  The 32 are in block
// order, so that a run of equal blocks is one maximum; `starts` has a bit where a run starts behind the first.
__device__ __forceinline__ uint32_t run_starts(int block)
{
    const int before = __shfl_up_sync(0xffffffffu, block, 1);
    return __ballot_sync(0xffffffffu, (threadIdx.x & 31) > 0 && before != block);
}
// The greater of a maximum so far, not below zero, and an entry.  (fmaxf passes a NaN over, as a comparison does; positive floats
// order like their bit patterns.)
template <bool kInt8>
__device__ __forceinline__ uint32_t greater(uint32_t m, uint32_t x)
{
    if constexpr (kInt8) return (uint32_t)max((int32_t)m, (int32_t)x);
    else return __float_as_uint(fmaxf(__uint_as_float(m), __uint_as_float(x)));
}

constexpr int kFewRuns = 6;                                     // runs of 32 up to which each is gone through by itself

constexpr int kWarpCols = kTileN / 32 / (kEpiWarps / 4);       // column blocks of a tile that one epilogue warp takes

// An epilogue warp's column blocks of a tile of rows in block order -> the blocks' coverage: cover[b][i] = max(0, max over the columns
// of block b), row i per lane, and for blocks above the diagonal the same with rows and columns exchanged (through shared memory).  A
// maximum leaves the registers where the block changes: the rows' at the end of a run that may span the tile, the columns' once per
// 32 rows at least.  colBlock: the blocks of the warp's columns, looked up before the tile was ready.
// Bound by the operands' way from L2 and then by this epilogue's own instructions (10 classes of 5000 x 512 int8 into 8 blocks: 108 us,
// 93 with no epilogue at all, where 0.8 GB come at 8.9 TB/s; writing S took 200 us and reading it back 200 more).  A pass per run of columns as long as they are few; with
// more runs in 32 than kFewRuns a test per column is cheaper, four columns at a time from shared memory.  The code has to stay short:
// with that test unrolled for 32 columns in registers, and all of it for each of a warp's column blocks, a warp spent 37 % of its time
// waiting for instructions.  The whole call in us, through S : that code : as it is, by samples of a class per block (int8, 64 elements):
//   1000 classes of 400   2 samples 766 : 871 : 737   6  564 : 759 : 531   8  537 : 792 : 485   16  498 : 466 : 353   128  477 : 318 : 275
//   20 of 2500            4         385 : 385 : 363   6  334 : 386 : 318   8  312 : 439 : 279   16  287 : 238 : 210   625  264 : 151 : 128
// Runs gone through by themselves up to 3 : 4 : 6 : 8 in 32 (1000 x 400, 8 samples): 521 : 517 : 485 : 475; (4 samples) 638 : 611 : 609 : 620.
template <bool kInt8, typename Mirrored>
__device__ __forceinline__ void keep_maxima(uint32_t (*stage)[33], int32_t *cover, const ClassDesc &c, int row0, int colB, uint32_t tmemRow,
                                            int half, int nCb, uint32_t (&v)[32], int rowBlock, const int (&colBlock)[kWarpCols], Mirrored mirrored)
{
    const int lane = threadIdx.x & 31;
    uint4 *const block4 = reinterpret_cast<uint4 *>(stage);
    const uint32_t rowStarts = run_starts(rowBlock);
    auto join = [&](int block, int i, uint32_t m) {
        if (block >= 0 && i < c.M && (int32_t)m > 0) atomicMax(cover + (int64_t)block * c.ld + i, (int32_t)m);
    };
    uint32_t m = 0;
    int block = -1;
#pragma unroll 1
    for (int k = 0; k < kWarpCols; ++k) {
        const int cb = half + k * (kEpiWarps / 4), col0 = colB + cb * 32;
        if (cb >= nCb) break;
        int mine = colBlock[0];
#pragma unroll
        for (int x = 1; x < kWarpCols; ++x) mine = k == x ? colBlock[x] : mine;
        const uint32_t colStarts = run_starts(mine);
        const int firstBlock = __shfl_sync(0xffffffffu, mine, 0);
        const bool mirror = mirrored(cb);
        tmem_load_wait();
        if (firstBlock != block) {
            join(block, row0 + lane, m);
            m = 0;
            block = firstBlock;
        }
        if (colStarts == 0) {                              // one block, as almost always where blocks are large
            uint32_t part[4] = {m, 0, 0, 0};
#pragma unroll
            for (int j = 0; j < 32; ++j) part[j & 3] = greater<kInt8>(part[j & 3], v[j]);
            m = greater<kInt8>(greater<kInt8>(part[0], part[1]), greater<kInt8>(part[2], part[3]));
        } else if (__popc(colStarts) < kFewRuns) {
            for (uint32_t left = colStarts | 1u; left; left &= left - 1) {
                const uint32_t later = left & (left - 1), run = (later & (0u - later)) - (left & (0u - left));   // the run's columns
                const int of = __shfl_sync(0xffffffffu, mine, __ffs((int)left) - 1);
                if (of != block) {
                    join(block, row0 + lane, m);
                    m = 0;
                    block = of;
                }
                uint32_t part[4] = {m, 0, 0, 0};
#pragma unroll
                for (int j = 0; j < 32; ++j) part[j & 3] = greater<kInt8>(part[j & 3], run >> j & 1 ? v[j] : 0u);
                m = greater<kInt8>(greater<kInt8>(part[0], part[1]), greater<kInt8>(part[2], part[3]));
            }
        }
        // (16-byte pieces, each row's turned by the row's number: neither side meets a bank twice)
        const bool manyRuns = __popc(colStarts) >= kFewRuns;
        if (mirror || manyRuns) {
#pragma unroll
            for (int g = 0; g < 8; ++g) block4[lane * 8 + (g ^ (lane & 7))] = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
        }
        if (manyRuns) {
#pragma unroll 1
            for (int g = 0; g < 8; ++g) {
                const uint4 x = block4[lane * 8 + (g ^ (lane & 7))];   // (the lane's own)
                const uint32_t y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (colStarts >> (4 * g + j) & 1) {
                        join(block, row0 + lane, m);
                        m = 0;
                        block = __shfl_sync(0xffffffffu, mine, 4 * g + j);
                    }
                    m = greater<kInt8>(m, y[j]);
                }
            }
        }
        __syncwarp();
        if (cb + kEpiWarps / 4 < nCb) tmem_load_32cols(tmemRow + (uint32_t)((cb + kEpiWarps / 4) * 32), v);
        if (mirror) {
            if (__popc(rowStarts) < kFewRuns) {
                for (uint32_t left = rowStarts | 1u; left; left &= left - 1) {
                    const uint32_t later = left & (left - 1);
                    const int from = __ffs((int)left) - 1, to = later ? __ffs((int)later) - 1 : 32;
                    // four columns per lane, every fourth row; then the four lanes of a piece
                    uint4 n = make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int k8 = 0; k8 < 8; ++k8) {
                        const int r = 4 * k8 + (lane >> 3);
                        const uint4 x = block4[r * 8 + ((lane & 7) ^ (r & 7))];
                        const bool in = r >= from && r < to;
                        n.x = greater<kInt8>(n.x, in ? x.x : 0u);
                        n.y = greater<kInt8>(n.y, in ? x.y : 0u);
                        n.z = greater<kInt8>(n.z, in ? x.z : 0u);
                        n.w = greater<kInt8>(n.w, in ? x.w : 0u);
                    }
#pragma unroll
                    for (int off = 8; off < 32; off <<= 1) {
                        n.x = greater<kInt8>(n.x, __shfl_xor_sync(0xffffffffu, n.x, off));
                        n.y = greater<kInt8>(n.y, __shfl_xor_sync(0xffffffffu, n.y, off));
                        n.z = greater<kInt8>(n.z, __shfl_xor_sync(0xffffffffu, n.z, off));
                        n.w = greater<kInt8>(n.w, __shfl_xor_sync(0xffffffffu, n.w, off));
                    }
                    join(__shfl_sync(0xffffffffu, rowBlock, from), col0 + 4 * (lane & 7) + (lane >> 3),
                         lane < 16 ? (lane < 8 ? n.x : n.y) : (lane < 24 ? n.z : n.w));
                }
            } else {
                uint32_t n = 0;
                int run = __shfl_sync(0xffffffffu, rowBlock, 0);
#pragma unroll 4
                for (int r = 0; r < 32; ++r) {
                    if (rowStarts >> r & 1) {
                        join(run, col0 + lane, n);
                        n = 0;
                        run = __shfl_sync(0xffffffffu, rowBlock, r);
                    }
                    n = greater<kInt8>(n, reinterpret_cast<const uint32_t *>(block4)[r * 32 + (((lane >> 2) ^ (r & 7)) << 2 | (lane & 3))]);
                }
                join(run, col0 + lane, n);
            }
        }
        __syncwarp();
    }
    join(block, row0 + lane, m);
}

// kMaxima: rows are in block order within their class (blockOf), and instead of S the blocks' coverage is written.
template <bool kInt8, bool kMaxima>
__global__ void __launch_bounds__(kTcThreads, 1) sim_tc_kernel(const __grid_constant__ CUtensorMap map, DescSource src, int32_t L,
                                                              const int32_t *__restrict__ tilePrefix, int32_t uniTiles,
                                                              int32_t *ticket, int32_t totalTiles, int32_t numSlabs, uint32_t *__restrict__ S,
                                                              const int32_t *__restrict__ blockOf, int32_t *cover, int32_t *status, bool clearStatus)
{
    extern __shared__ unsigned char smemRaw[];
    // operand stages need 1024-byte alignment for the 128-byte swizzle pattern
    unsigned char *tiles = reinterpret_cast<unsigned char *>(((uintptr_t)smemRaw + 1023) & ~(uintptr_t)1023);
    __shared__ TcShared sh;
    __shared__ __align__(16) uint32_t stage32[kEpiWarps][32][33];             // per epilogue warp: one 32 x 32 block, padded

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (clearStatus && blockIdx.x == 0 && threadIdx.x == 0) *(volatile int32_t *)status = 0;    // (no wait runs out for a quarter of a second)

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&sh.accFull[b], 1); mbar_init(&sh.accEmpty[b], kEpiWarps); }
        for (int k = 0; k < kTileSlots; ++k) { mbar_init(&sh.tileFull[k], 1); mbar_init(&sh.tileEmpty[k], 1 + kEpiWarps); }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_addr(&sh.tmemBase)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmemBase = sh.tmemBase;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t it = 0;                             // k-slabs issued so far, over all tiles
            bool ok = true;
            int idx = blockIdx.x;
            // the next tile: every gridDim.x-th, or drawn from the launch's ticket, which whoever draws last puts back to zero
            auto draw = [&]() { return ticket ? atomicAdd(ticket, 1) : idx; };
            auto tile_of = [&](int k) {
                if (ticket && k == totalTiles - 1) atomicExch(ticket, 0);
                return k + (int)gridDim.x < totalTiles ? k + (int)gridDim.x : -1;
            };
            for (uint32_t nt = 0; ok; ++nt) {
                const int slot = nt % kTileSlots;
                if (!mbar_wait(&sh.tileEmpty[slot], ((nt / kTileSlots) & 1) ^ 1, &sh)) break;
                if (idx < 0) {
                    sh.tile[slot].t.l = -1;
                    mbar_arrive(&sh.tileFull[slot]);
                    break;
                }
                int next = -1;
                // (once for all roles: a search in the prefixes and a walk along the row blocks, which the epilogue would wait for
                // tile by tile)
                const TileCoord t = decode_tile(src, tilePrefix, L, uniTiles, idx);
                const ClassDesc c = src.get(t.l);
                sh.tile[slot].t = t;
                sh.tile[slot].c = c;
                mbar_arrive(&sh.tileFull[slot]);
                const int rowA = c.row0 + t.tm * kTileM, rowB = c.row0 + t.sn * kTileN + t.skip;
                const int halves = (t.n + kTileM - 1) / kTileM;         // 128-row pieces of B to bring in: 2, or 1
                const bool shared = t.sn == t.tm / 2;                   // on the diagonal the first of them is A
                for (int kb = 0; kb < numSlabs; ++kb, ++it) {
                    if (kb == max(numSlabs - kStages, 0)) next = draw();       // (looked at behind the last slab)
                    const int s = it % kStages;
                    if (!mbar_wait(&sh.empty[s], ((it / kStages) & 1) ^ 1, &sh)) { ok = false; break; }
                    unsigned char *a = tiles + (size_t)s * kStageBytes;
                    mbar_expect_tx(&sh.full[s], ((shared ? 0 : 1) + halves) * kOperandBytes);
                    const int k0 = kb * (kInt8 ? kSlabBytes : kSlabBytes / 2);         // element coordinate
                    if (!shared) tma_load_2d(a, &map, k0, rowA, &sh.full[s]);
                    for (int h = 0; h < halves; ++h) tma_load_2d(a + (1 + h) * kOperandBytes, &map, k0, rowB + h * kTileM, &sh.full[s]);
                }
                if (next < 0) next = draw();
                idx = tile_of(next);
            }
            while (idx >= 0) idx = tile_of(draw());       // (given up: the tickets still have to run out)
            // after an abort: let the copies already issued land before the CTA leaves
            if (*(volatile int32_t *)&sh.abort) {
                for (uint32_t k = (it > (uint32_t)kStages ? it - kStages : 0); k < it; ++k) {
                    const int s = k % kStages;
                    for (uint32_t spin = 0; spin < kSpinLimit && !mbar_test(&sh.full[s], (k / kStages) & 1); ++spin) __nanosleep(64);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            // instruction descriptor: D format, A/B format, K-major operands, N and M of the tile
            const uint32_t idescBase = (kInt8 ? (2u << 4) | (1u << 7) | (1u << 10)   // S32 accumulate, S8 x S8
                                              : (1u << 4) | (1u << 7) | (1u << 10))  // F32 accumulate, BF16 x BF16
                                       | ((uint32_t)(kTileM >> 4) << 24);
            uint32_t it = 0, nt = 0;
            bool ok = true;
            for (; ok; ++nt) {
                const int slot = nt % kTileSlots;
                if (!mbar_wait(&sh.tileFull[slot], (nt / kTileSlots) & 1, &sh)) break;
                const TileCoord t = sh.tile[slot].t;
                mbar_arrive(&sh.tileEmpty[slot]);
                if (t.l < 0) break;
                const uint32_t idesc = idescBase | ((uint32_t)(t.n >> 3) << 17);   // N = 256, less for a half tile or at the class's edge
                const uint32_t buf = nt & 1;
                // the epilogue must have drained this accumulator buffer (two tiles ago)
                if (!mbar_wait(&sh.accEmpty[buf], ((nt >> 1) & 1) ^ 1, &sh)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tmemD = tmemBase + buf * kTileN;
                for (int kb = 0; kb < numSlabs; ++kb, ++it) {
                    const int s = it % kStages;
                    if (!mbar_wait(&sh.full[s], (it / kStages) & 1, &sh)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t aAddr = smem_addr(tiles + (size_t)s * kStageBytes);
                    const uint64_t descA = make_smem_desc(t.sn == t.tm / 2 ? aAddr + kOperandBytes : aAddr);
                    const uint64_t descB = make_smem_desc(aAddr + kOperandBytes);
#pragma unroll
                    for (int k = 0; k < kSlabBytes / 32; ++k)          // one MMA consumes 32 bytes of k per row
                        mma_issue<kInt8>(tmemD, descA + (uint64_t)(2 * k), descB + (uint64_t)(2 * k), idesc, (kb > 0 || k > 0) ? 1u : 0u);
                    mma_commit(&sh.empty[s]);                          // frees the stage when those MMAs retire
                }
                mma_commit(&sh.accFull[buf]);                          // accumulator complete (or abandoned)
            }
        }
    } else {
        // ---------------- epilogue: TMEM -> registers -> shared (transpose) -> global ----------------
        const int q = warp & 3;                                        // TMEM lane quarter this warp may read
        const int ew = warp - 2;
        const int half = ew >> 2;                                      // which column blocks of the tile: even or odd
        uint32_t nt = 0;
        for (;; ++nt) {
            const int slot = nt % kTileSlots;
            if (!mbar_wait(&sh.tileFull[slot], (nt / kTileSlots) & 1, &sh)) break;
            const TileCoord t = sh.tile[slot].t;
            const ClassDesc c = sh.tile[slot].c;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.tileEmpty[slot]);
            if (t.l < 0) break;
            const int rowA = t.tm * kTileM, colB = t.sn * kTileN + t.skip;   // class-local: first row, first column computed
            const uint32_t buf = nt & 1;
            [[maybe_unused]] int rowBlock = -1, colBlock[kWarpCols];
            if constexpr (kMaxima) {
                const int32_t *const of = blockOf + c.row0;
                if (rowA + q * 32 + lane < c.M) rowBlock = of[rowA + q * 32 + lane];
#pragma unroll
                for (int k = 0; k < kWarpCols; ++k) {
                    const int col = colB + (half + k * (kEpiWarps / 4)) * 32 + lane;
                    colBlock[k] = col < c.M ? of[col] : -1;
                }
            }
            if (!mbar_wait(&sh.accFull[buf], (nt >> 1) & 1, &sh)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (*(volatile int32_t *)&sh.abort) break;
            [[maybe_unused]] uint32_t *Sl = S + c.sOff;
            const int nCb = t.n / 32;
            const uint32_t tmemRow = tmemBase + buf * kTileN + ((uint32_t)(q * 32) << 16);
            uint32_t v[32];
            if (half < nCb) tmem_load_32cols(tmemRow + (uint32_t)(half * 32), v);
            // a 128 x 128 block lies on the diagonal (stored once) or above it (stored twice: itself and its mirror image)
            auto mirrored = [&](int cb) { return (colB + cb * 32) / kTileM != t.tm; };
            if constexpr (kMaxima) keep_maxima<kInt8>(stage32[ew], cover + c.vOff, c, rowA + q * 32, colB, tmemRow, half, nCb, v, rowBlock, colBlock, mirrored);
            else write_columns(stage32[ew], Sl, c, rowA + q * 32, colB, tmemRow, half, nCb, v, mirrored);
            // hand the accumulator buffer back to the MMA warp
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.accEmpty[buf]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmemBase), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && sh.abort && status) atomicOr(status, kDevTimeout);
}

// ---------------------------------------------------------------------------------------------
// Long rows: a pair of SMs per 256 x 256 tile (cta_group::2).  Each CTA holds 128 of the tile's rows (A and the accumulator)
// and half of its columns (B), so every operand row comes in once: 32 KB per SM and k-slab, 16 on the diagonal, where both
// operands are the same rows, against 48 and 32 above.  CTA 0 issues the MMAs of both.  Tiles on the diagonal are computed
// whole and stored as they are, the others stored twice.  Bound by the tensor cores: their pipe is active 60 % of the time an SM
// has work.  100 classes of 500 x 2048 bf16: 78.7 us, the 128 x 256 kernel above 85.0 (both under the profiler; 67 GFLOP, at
// least 40 us; writing S and reading X, 47).
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = 2 * kOperandBytes;
constexpr int kPairTile = 256;

struct __align__(8) PairShared {
    uint64_t full[kPairStages];                         // CTA 0's: both CTAs' copies of a slab have landed
    uint64_t empty[kPairStages];
    uint64_t accFull[2];
    uint64_t accEmpty[2];                               // CTA 0's: the epilogue warps of both CTAs have read the accumulator
    uint32_t tmemBase;
    int32_t abort;
};

__device__ __forceinline__ uint32_t leader_addr(const void *p)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_addr(p)));
    return a;
}
__device__ __forceinline__ bool pair_wait(uint64_t *bar, uint32_t parity, PairShared *sh)
{
    for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
        if (ok) return true;
        if (spin > 64) {
            if (*(volatile int32_t *)&sh->abort) return false;
            __nanosleep(64);
        }
    }
    atomicExch(&sh->abort, 1);
    return false;
}
__device__ __forceinline__ void pair_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint32_t leaderBar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(smem_addr(dst)), "l"(map), "r"(c0), "r"(c1), "r"(leaderBar) : "memory");
}
template <bool kInt8>
__device__ __forceinline__ void pair_mma(uint32_t tmemD, uint64_t descA, uint64_t descB, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (kInt8) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(tmemD), "l"(descA), "l"(descB), "r"(idesc), "r"(accumulate) : "memory");
    } else {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(tmemD), "l"(descA), "l"(descB), "r"(idesc), "r"(accumulate) : "memory");
    }
}
// arrives at the barrier of this offset in both CTAs
__device__ __forceinline__ void pair_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(smem_addr(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Unit -> class, row block of 256, first column and columns computed; column blocks run from the row block on.
struct PairTile { int l, tb, col, n; bool diag, shared; };      // diag: stored once; shared: A's rows are B's
__device__ __forceinline__ PairTile decode_pair_tile(const DescSource &src, const int32_t *__restrict__ prefix, int L, int uniTiles,
                                                     const PairUnits &units, int unit)
{
    PairTile t;
    int local, idx = unit, strip = 0;
    const bool cut = unit >= units.whole && units.strips > 1;
    if (cut) {
        idx = units.whole + (unit - units.whole) / units.strips;
        strip = (unit - units.whole) % units.strips;
    }
    if (prefix) {
        int lo = 0, hi = L;                              // prefix[lo] <= idx < prefix[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (prefix[mid] <= idx) lo = mid; else hi = mid;
        }
        t.l = lo;
        local = idx - prefix[lo];
    } else {
        t.l = idx / uniTiles;
        local = idx - t.l * uniTiles;
    }
    const ClassDesc c = src.get(t.l);
    const int blocks = (c.M + kPairTile - 1) / kPairTile;
    for (t.tb = 0; local >= blocks - t.tb; ++t.tb) local -= blocks - t.tb;
    const int width = cut ? kPairTile / units.strips : kPairTile;
    t.diag = local == 0;
    t.shared = t.diag && !cut;                           // (each CTA's 128 rows are its half of the columns too)
    t.col = (t.tb + local) * kPairTile + strip * width;
    t.n = t.shared ? kPairTile : max(32, min(width, (c.ld - t.col + 31) & ~31));
    return t;
}

template <bool kInt8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1) sim_pair_kernel(
    const __grid_constant__ CUtensorMap map, DescSource src, int32_t L, const int32_t *__restrict__ tilePrefix, int32_t uniTiles,
    int32_t totalTiles, int32_t kernelPairs, int32_t numSlabs, uint32_t *__restrict__ S, int32_t *status, bool clearStatus)
{
    extern __shared__ unsigned char smemRaw[];
    unsigned char *tiles = reinterpret_cast<unsigned char *>(((uintptr_t)smemRaw + 1023) & ~(uintptr_t)1023);
    __shared__ PairShared sh;
    __shared__ uint32_t stage32[kEpiWarps][32][33];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (clearStatus && blockIdx.x == 0 && threadIdx.x == 0) *(volatile int32_t *)status = 0;    // (no wait runs out for a quarter of a second)
    const int rank = blockIdx.x & 1;                     // (clusters are consecutive pairs of blocks)
    const int firstUnit = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const PairUnits units = pair_units(totalTiles, kernelPairs);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPairStages; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&sh.accFull[b], 1); mbar_init(&sh.accEmpty[b], 2 * kEpiWarps); }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_addr(&sh.tmemBase)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_barrier();                                   // the other CTA's barriers exist
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmemBase = sh.tmemBase;

    if (warp == 0) {
        // ---------------- TMA producer: this CTA's half of both operands ----------------
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int idx = firstUnit; idx < units.count && ok; idx += pairs) {
                const PairTile t = decode_pair_tile(src, tilePrefix, L, uniTiles, units, idx);
                const ClassDesc c = src.get(t.l);
                const int rowA = c.row0 + t.tb * kPairTile + rank * kTileM, rowB = c.row0 + t.col + rank * (t.n / 2);
                for (int kb = 0; kb < numSlabs; ++kb, ++it) {
                    const int s = it % kPairStages;
                    if (!pair_wait(&sh.empty[s], ((it / kPairStages) & 1) ^ 1, &sh)) { ok = false; break; }
                    unsigned char *a = tiles + (size_t)s * kPairStageBytes;
                    if (rank == 0) mbar_expect_tx(&sh.full[s], 2 * (t.shared ? 1 : 2) * kOperandBytes);
                    const uint32_t bar = leader_addr(&sh.full[s]);
                    const int k0 = kb * (kInt8 ? kSlabBytes : kSlabBytes / 2);
                    pair_load_2d(a, &map, k0, rowA, bar);
                    if (!t.shared) pair_load_2d(a + kOperandBytes, &map, k0, rowB, bar);
                }
            }
            // after an abort: let the copies already issued land (they report to CTA 0, so by time: some 2 ms)
            if (*(volatile int32_t *)&sh.abort)
                for (uint32_t spin = 0; spin < (1u << 15); ++spin) __nanosleep(64);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: CTA 0, for both ----------------
        if (lane == 0 && rank == 0) {
            const uint32_t idescBase = (kInt8 ? (2u << 4) | (1u << 7) | (1u << 10) : (1u << 4) | (1u << 7) | (1u << 10)) | ((uint32_t)(kPairTile >> 4) << 24);
            uint32_t it = 0, nt = 0;
            bool ok = true;
            for (int idx = firstUnit; idx < units.count && ok; idx += pairs, ++nt) {
                const PairTile t = decode_pair_tile(src, tilePrefix, L, uniTiles, units, idx);
                const uint32_t idesc = idescBase | ((uint32_t)(t.n >> 3) << 17);
                const uint32_t buf = nt & 1;
                if (!pair_wait(&sh.accEmpty[buf], ((nt >> 1) & 1) ^ 1, &sh)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tmemD = tmemBase + buf * kPairTile;
                for (int kb = 0; kb < numSlabs; ++kb, ++it) {
                    const int s = it % kPairStages;
                    if (!pair_wait(&sh.full[s], (it / kPairStages) & 1, &sh)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t aAddr = smem_addr(tiles + (size_t)s * kPairStageBytes);
                    const uint64_t descA = make_smem_desc(aAddr);
                    const uint64_t descB = make_smem_desc(t.shared ? aAddr : aAddr + kOperandBytes);
#pragma unroll
                    for (int k = 0; k < kSlabBytes / 32; ++k)
                        pair_mma<kInt8>(tmemD, descA + (uint64_t)(2 * k), descB + (uint64_t)(2 * k), idesc, (kb > 0 || k > 0) ? 1u : 0u);
                    pair_commit(&sh.empty[s]);
                }
                pair_commit(&sh.accFull[buf]);
            }
        }
    } else {
        // ---------------- epilogue: this CTA's 128 rows ----------------
        const int q = warp & 3, ew = warp - 2, half = ew >> 2;
        uint32_t nt = 0;
        for (int idx = firstUnit; idx < units.count; idx += pairs, ++nt) {
            const PairTile t = decode_pair_tile(src, tilePrefix, L, uniTiles, units, idx);
            const ClassDesc c = src.get(t.l);
            const uint32_t buf = nt & 1;
            if (!pair_wait(&sh.accFull[buf], (nt >> 1) & 1, &sh)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (*(volatile int32_t *)&sh.abort) break;
            const int row0 = t.tb * kPairTile + rank * kTileM + q * 32;
            const int nCb = row0 < c.M ? t.n / 32 : 0;
            const uint32_t tmemRow = tmemBase + buf * kPairTile + ((uint32_t)(q * 32) << 16);
            uint32_t v[32];
            if (half < nCb) tmem_load_32cols(tmemRow + (uint32_t)(half * 32), v);
            write_columns(stage32[ew], S + c.sOff, c, row0, t.col, tmemRow, half, nCb, v, [&](int) { return !t.diag; });
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(leader_addr(&sh.accEmpty[buf])) : "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_barrier();                                   // nothing of the other CTA is on its way here any more
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmemBase), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && sh.abort && status) atomicOr(status, kDevTimeout);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

}  // namespace

rcd_status launch_similarity_tc(rcd_ctx *ctx, const void *Xs, rcd_feat_dtype dtype, int64_t Ntot, int64_t d,
                                const SimClasses &cls, void *S, const int32_t *blockOf, int32_t *cover, cudaStream_t st, bool *handled)
{
    *handled = false;
    const int64_t rowBytes = d * (int64_t)feat_bytes(dtype);
    // TMA needs 16-byte row pitch and base; a row shorter than one 128-byte slab goes to the generic kernel
    if (rowBytes % 16 != 0 || rowBytes < kSlabBytes || ((uintptr_t)Xs) % 16 != 0 || ((uintptr_t)S) % 16 != 0) return RCD_OK;
    if (cls.L == 0 || cls.maxM == 0 || Ntot == 0) { *handled = true; return RCD_OK; }
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return fail(ctx, RCD_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");

    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)Ntot};
    const cuuint64_t strides[1] = {(cuuint64_t)rowBytes};
    const cuuint32_t box[2] = {(cuuint32_t)(dtype == RCD_FEAT_I8 ? kSlabBytes : kSlabBytes / 2), (cuuint32_t)kTileM};
    const cuuint32_t estr[2] = {1, 1};
    CUresult cr = encode(&map, dtype == RCD_FEAT_I8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                         const_cast<void *>(Xs), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) return fail(ctx, RCD_ERR_CUDA, "cuTensorMapEncodeTiled failed with %d", (int)cr);

    const int numSlabs = (int)((rowBytes + kSlabBytes - 1) / kSlabBytes);
    const size_t smem = (size_t)kStages * kStageBytes + 1024;
    if (cls.upperTiles <= 0 || cls.upperTiles > 0x7fffffffLL) return RCD_OK;
    const int totalTiles = (int)cls.upperTiles;
    const int grid = totalTiles < ctx->smCount ? totalTiles : ctx->smCount;
    int32_t *status = const_cast<int32_t *>(ctx->statusDev);
    const bool isInt8 = dtype == RCD_FEAT_I8;
    // (shared memory beyond 48 KB is asked for once per context and kernel, not on every call)
    auto allow = [&](auto *kernel, int bit, size_t bytes) {
        if (ctx->simReady >> bit & 1) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess) ctx->simReady |= 1u << bit;
        return e;
    };
    if (cls.pairs) {
        const size_t pairSmem = (size_t)kPairStages * kPairStageBytes + 1024;
        const int pairs = std::max(1, ctx->smCount / 2);
        const int pairGrid = 2 * std::min(pairs, pair_units(totalTiles, pairs).count);
        auto *kernel = isInt8 ? sim_pair_kernel<true> : sim_pair_kernel<false>;
        RCD_CUDA(ctx, allow(kernel, isInt8 ? 3 : 2, pairSmem));
        kernel<<<pairGrid, kTcThreads, pairSmem, st>>>(map, cls.src, cls.L, cls.tilePrefixDev, cls.uniTiles, totalTiles, pairs,
                                                       numSlabs, (uint32_t *)S, status, cls.clearStatus);
    } else {
        // Tiles are drawn, since they are not equally long and an uneven share leaves most SMs idle at the end: 10 classes of
        // 5000 x 256 int8 217 -> 177 us, 50 of 1300 x 192 bf16 112 -> 99, 100 of 500 x 512 bf16 47 -> 44.  Not so for short
        // rows in classes of at most 8 tiles (500 samples: 6): every gridDim.x-th is as even then, and a CTA has to draw such
        // tiles up to three ahead of their turn (200 of 257 x 256 int8: 29 -> 34 us).  A ticket of its own for every launch
        // that can be under way at once: calls may overlap on several streams.
        int32_t *ticket = totalTiles <= 8LL * cls.L && numSlabs < 8 ? nullptr : ctx->statusOwn + kFirstTicket + ctx->simTurn++ % (kStatusWords - kFirstTicket);
        auto *kernel = blockOf ? (isInt8 ? sim_tc_kernel<true, true> : sim_tc_kernel<false, true>)
                               : (isInt8 ? sim_tc_kernel<true, false> : sim_tc_kernel<false, false>);
        RCD_CUDA(ctx, allow(kernel, (isInt8 ? 1 : 0) + (blockOf ? 4 : 0), smem));
        kernel<<<grid, kTcThreads, smem, st>>>(map, cls.src, cls.L, cls.tilePrefixDev, cls.uniTiles, ticket, totalTiles,
                                               numSlabs, (uint32_t *)S, blockOf, cover, status, cls.clearStatus);
    }
    ctx->kernelLaunches++;
    ctx->tcLaunches++;
    RCD_CUDA(ctx, cudaGetLastError());
    *handled = true;
    return RCD_OK;
}

}  // namespace rcd
