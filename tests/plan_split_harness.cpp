// Prints plans_in_turn (csrc/geometry.cpp) for each line of stdin: "threads n",
// then n numbers of active DOFs in descending order.  Test infrastructure;
// built by tests/test_plan_split.py.
#include <cstdio>

#include "../paper_1307_2666_gb300/csrc/geometry.h"

int main() {
    int threads, n;
    while (std::scanf("%d %d", &threads, &n) == 2) {
        std::vector<int64_t> a(n);
        for (auto& v : a) {
            long long t;
            if (std::scanf("%lld", &t) != 1) return 2;
            v = t;
        }
        std::printf("%d\n", hif::plans_in_turn(a, threads));
    }
    return 0;
}
