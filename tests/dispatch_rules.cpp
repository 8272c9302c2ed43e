// Answers questions about the library's dispatch rules (test_dispatch_rules.py), one per line of standard input.
#include <iostream>
#include <string>

#include "rcd_internal.h"

int main()
{
    std::string what;
    while (std::cin >> what) {
        if (what == "cut_values") {
            int64_t M, d;
            std::cin >> M >> d;
            std::cout << rcd::cut_values_fit(M, d) << "\n";
        } else {
            return 1;
        }
    }
    return 0;
}
