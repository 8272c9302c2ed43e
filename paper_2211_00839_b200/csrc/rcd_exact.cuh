// What the forms of the greedy loop with exact stored gains (rcd_cluster.cu, rcd_rounds.cu, rcd_small.cu) have in common: keys, losses, and
// the loads of rows of S.
#pragma once

#include "rcd_internal.h"

namespace rcd {
namespace {

struct __align__(16) Raised {
    int32_t row;                          // a column whose coverage rose: its row of S, in 16-byte pieces from the class's first
    int32_t minusOld, by;                 // - old coverage, new - old
    int32_t pad_;
};

__device__ __forceinline__ uint32_t smem32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int4 ld_row_shared(const int4 *p)       // (other teams of the CTA read the same rows: L1 may serve them)
{
    int4 v;
    asm volatile("ld.global.nc.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
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

// What a candidate loses for one raised column: min(max(x, old), new) - old, as one instruction.  Similarities stay
// below 2^30 either way, so x - old does not wrap, and two losses fit an int.
__device__ __forceinline__ int loss(int x, const Raised &e) { return __viaddmin_s32_relu(x, e.minusOld, e.by); }

// A floating-point similarity as a fixed-point integer below 2^30.
__device__ __forceinline__ int to_fixed(float x, float scale) { return min(max(__float2int_rn(x * scale), -((1 << 30) - 1)), (1 << 30) - 1); }

// 16 bytes global -> shared without passing through registers
__device__ __forceinline__ void copy16(int4 *dst, const int4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

}  // namespace
}  // namespace rcd
