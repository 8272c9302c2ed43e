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
        } else {
            return 1;
        }
    }
    return 0;
}
