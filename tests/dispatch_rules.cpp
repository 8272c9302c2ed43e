// Answers questions about the library's dispatch rules (test_dispatch_rules.py), one per line of standard input.
#include <iostream>
#include <string>

#include "rcd_cut_plan.h"

int main()
{
    std::string what;
    while (std::cin >> what) {
        if (what == "cut_values") {
            int64_t M, d;
            std::cin >> M >> d;
            std::cout << rcd::cut_values_fit(M, d) << "\n";
        } else if (what == "cut_plan") {
            int sms, shared, most;
            rcd::Sizes sz{};
            std::cin >> sms >> shared >> most >> sz.L >> sz.maxM >> sz.d >> sz.W;
            rcd::LockPlan p{};
            if (rcd::lock_plan(sms, shared, most, sz, p)) std::cout << p.C << " " << p.K << " " << p.warps << " " << p.columns << " " << p.smem << "\n";
            else std::cout << "0 0 0 0 0\n";
        } else if (what == "cut_cycles") {                 // in step (0: not), in clusters of C CTAs, in a CTA per class
            int W, C, resident, L, M;
            std::cin >> W >> C >> resident >> L;
            std::vector<rcd::ClassDesc> classes;
            rcd::Sizes sz{};
            for (int l = 0; l < L; ++l) {
                std::cin >> M;
                classes.push_back(rcd::ClassDesc{M, 0, 0, 0, 0, 0});
                sz.maxM = std::max<int64_t>(sz.maxM, M);
            }
            sz.L = L; sz.W = W; sz.d = 64;
            rcd::LockPlan p{};
            const bool taken = rcd::lock_plan(148, 232448, 16, sz, p);
            std::cout << (int64_t)(taken ? rcd::cut_steps_cycles(148, 232448, p, classes) : 0) << " "
                      << (int64_t)rcd::cut_cluster_cycles(C, resident, W, classes) << " " << (int64_t)rcd::cut_chain_cycles(148, classes) << "\n";
        } else {
            return 1;
        }
    }
    return 0;
}
