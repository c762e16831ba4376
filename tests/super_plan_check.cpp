// The calls whose tensor-core products have bounded waits (super_plan.h), against
// the lists of superblocks that the Sylvester solve works through: its levels
// are the superblock anti-diagonals from the bottom-left one, and every one
// after the first has sums.  Prints "ok <shapes checked>".
#include <cstdio>
#include <set>

#include "super_plan.h"

using namespace signtri;

int main()
{
    long long shapes = 0;
    for (int m = 1; m <= 520; m++)
        for (int p = 1; p <= 520; p++, shapes++) {
            std::set<int> levels;
            for (int a = 0; a * kSuperEdge < m; a++)
                for (int b = 0; b * kSuperEdge < p; b++) levels.insert((m - 1) / kSuperEdge - a + b);
            const bool sums = levels.size() > 1;
            if (sylvester_products(m, p) != sums || ps_products(m, p, 0) != sums || !ps_products(m, p, 1)) {
                std::printf("FAIL %d x %d\n", m, p);
                return 1;
            }
        }
    if (sylvester_products(0, 300) || sylvester_products(300, 0)) return 1;
    std::printf("ok %lld\n", shapes);
    return 0;
}
