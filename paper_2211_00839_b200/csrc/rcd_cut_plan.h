// How the integer graph cut in step (rcd_cut.cu) is laid out: CTAs per class, columns per thread.  Host code only.
#pragma once

#include <algorithm>
#include <cmath>
#include <functional>
#include <vector>

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

// When the last of the classes is through, if `at` of them run at a time and the largest start first (cost: of a class of M samples).
template <typename Cost>
inline double cut_finish(const std::vector<ClassDesc> &classes, int at, Cost cost)
{
    std::vector<double> costs;
    bool equal = true;
    for (const ClassDesc &c : classes)
        if (c.M > 0) {
            costs.push_back(cost((double)c.M));
            equal = equal && costs.back() == costs[0];
        }
    if (costs.empty()) return 0;
    at = std::max(at, 1);
    if (equal) return costs[0] * (double)((costs.size() + at - 1) / at);
    std::sort(costs.begin(), costs.end(), std::greater<double>());
    std::vector<double> busy(std::min<size_t>((size_t)at, costs.size()), 0.0);      // a heap, the earliest first
    for (double c : costs) {
        std::pop_heap(busy.begin(), busy.end(), std::greater<double>());
        busy.back() += c;
        std::push_heap(busy.begin(), busy.end(), std::greater<double>());
    }
    return *std::max_element(busy.begin(), busy.end());
}

// What the forms of the graph cut take, in cycles: in step, in clusters of C CTAs of which `resident` run at a time, and in one CTA per
// class (two to an SM).  Fitted to 660 random problems of 260 to 6000 samples, 1 to 300 classes, a third of them of uneven sizes, 2 to
// 128 blocks: a tenth off on average (the chain a fifth).  With 330 more: of some 720 that run in step two are slower than without that form
// (5 and 13 %), and six that would be faster are left to another (by 6 to 20 %); by the largest class alone those of many classes and
// blocks took up to 2.8 times as long (208 of 1383 into 111 blocks 20.7 ms in step, 7.4 in the chain), uneven ones up to 1.5 times (83 of up to 1051 into 6 2467 us,
// in clusters 1644), equal ones up to 1.3 times (70 of 1941 into 7 4791 us, in clusters 3780).
inline double cut_steps_cycles(int smCount, int maxSmemOptin, const LockPlan &plan, const std::vector<ClassDesc> &classes)
{
    // CTAs that share an SM slow one another down a little, and so do the many of the largest clusters
    const int perSm = (int)std::max<size_t>(1, std::min<size_t>(6, (size_t)maxSmemOptin / (plan.smem + 4096)));
    const int resident = plan.C == 1 ? smCount * perSm : plan.C == 16 ? smCount / 20 * perSm : (int)(0.9 * smCount * perSm / plan.C);
    double samples = 0, largest = 1;
    for (const ClassDesc &c : classes) {
        samples += c.M;
        largest = std::max(largest, (double)c.M);
    }
    const double share = std::min((double)perSm, std::max(1.0, std::ceil(samples / largest * plan.C / smCount - 1e-9)));
    const double pick = (plan.C == 1 ? 1600.0 : plan.C == 16 ? 1800.0 : 1400.0) + 400.0 * plan.K;
    return cut_finish(classes, resident, [&](double M) { return M * pick; }) * (1.0 + 0.15 * (share - 1.0));
}
inline double cut_cluster_cycles(int C, int resident, int W, const std::vector<ClassDesc> &classes)
{
    const double pick = 1200.0 + 300.0 * std::log2((double)W);
    return cut_finish(classes, resident, [&](double M) { return M * (pick + 2.0 * M / C + 0.0003 * (M / C) * (M / C)); });
}
inline double cut_chain_cycles(int smCount, const std::vector<ClassDesc> &classes)
{
    int64_t some = 0;
    for (const ClassDesc &c : classes) some += c.M > 0 ? 1 : 0;
    return cut_finish(classes, some <= smCount ? smCount : 2 * smCount, [&](double M) { return M * (2000.0 + 3.0 * M); }) * (some <= smCount ? 1.0 : 1.4);
}

}  // namespace rcd
