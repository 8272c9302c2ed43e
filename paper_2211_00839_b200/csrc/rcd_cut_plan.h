// How the integer graph cut in step (rcd_cut.cu) is laid out: CTAs per class, columns per thread.  Host code only.
#pragma once

#include <algorithm>
#include <cmath>

#include "rcd_internal.h"

namespace rcd {

constexpr int kLockWarps = 8;             // with columns, at most
constexpr int kLockColumns = 8;           // of a thread, at most
constexpr int kLockBlocks = 128;
constexpr int kLockCtas = 16;

struct LockPlan { int C, K, warps, columns; size_t smem; };

inline int64_t lock_shared(int maxSmemOptin) { return (int64_t)maxSmemOptin - 8192; }

// Whether the classes run in step, and on how many CTAs each (mostCtas at most): those with which they are through soonest.  A pick takes
// 1600 cycles with one CTA, 1700 with several, and 260 more for every column of a thread (measured on 250 to 5000 samples); clusters keep
// within a GPC.
// Not with few blocks and classes, whose picks wait for the sample's row, while the cluster form foresees it (3 or 30 classes of 700 to
// 2500: 0.6 to 0.9 times as fast with 2 and 4 blocks, 1.0 to 1.7 times with 8, 1.1 to 2.7 with more; 200 classes: 1.2 to 3 times, but 0.96
// for 1300 samples into 2 blocks), and not where short classes come one to an SM and have to come again (200 of 400 into 50 blocks in one
// CTA each 1014 us, the cluster form 874).
inline bool lock_plan(int smCount, int maxSmemOptin, int mostCtas, const Sizes &sz, LockPlan &plan)
{
    if (sz.W > kLockBlocks || sz.maxM == 0 || sz.maxM > 65535 || sz.floatArith || !cut_values_fit(sz.maxM, sz.d)) return false;
    if (sz.W < 6 && sz.maxM <= 8192 && (sz.L <= 64 || (sz.W < 4 && sz.maxM >= 1024))) return false;
    double best = 0;
    plan.C = 0;
    bool again = false;
    for (int C = 1; C <= mostCtas; C *= 2) {
        LockPlan p;
        p.C = C;
        const int share = (int)((sz.maxM + C - 1) / C), words = (share + 31) / 32;
        p.K = (words + kLockWarps - 1) / kLockWarps;
        if (p.K > 4) p.K = kLockColumns;
        p.warps = std::min(kLockWarps, (words + p.K - 1) / p.K);
        p.columns = words * 32;
        p.smem = (size_t)sz.W * p.columns * 8;
        if (words > kLockWarps * kLockColumns || (int64_t)p.smem > lock_shared(maxSmemOptin) || (C > 1 && share < 128)) continue;
        const int perSm = (int)std::max<size_t>(1, std::min<size_t>(6, (size_t)maxSmemOptin / (p.smem + 4096)));
        const double resident = std::max(1.0, C == 1 ? (double)smCount * perSm : C == 16 ? (double)(smCount / 20) : std::floor(0.9 * smCount / C));
        const double turns = std::max(1.0, std::ceil(sz.L / resident - 1e-9));
        const double time = turns * ((C == 1 ? 1570.0 : 1700.0) + 260.0 * p.K);
        if (plan.C == 0 || time < best) {
            plan = p;
            best = time;
            again = turns > 1 && perSm == 1 && sz.maxM < 512;
        }
    }
    return plan.C > 0 && !again;
}

}  // namespace rcd
