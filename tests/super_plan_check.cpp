// The calls whose tensor-core products have bounded waits (super_plan.h), against
// the lists of superblocks that the Sylvester solve works through: its levels
// are the superblock anti-diagonals from the bottom-left one, and every one
// after the first has sums.  And where the products' operands lie: the tiles of
// a form fill its bytes, each once, and hold every K-block that a product reads.
// Prints "ok <shapes checked>".
#include <cstdio>
#include <set>
#include <vector>

#include "super_plan.h"

using namespace signtri;

static bool fills(const rns::Layout &l, int panels)
{
    std::vector<char> seen(l.before(panels) * rns::kMods, 0);
    size_t count = 0;
    for (int P = 0; P < panels; P++)
        for (int m = 0; m < rns::kMods; m++)
            for (int kb = l.first(P); kb < l.first(P) + l.count(P); kb++, count++) {
                const size_t t = l.tile(P, m, kb);
                if (t >= seen.size() || seen[t]++) return false;
                if (m + 1 < rns::kMods && l.tile(P, m + 1, kb) != t + l.count(P)) return false;
            }
    return count == seen.size();
}

static bool holds(const rns::Layout &l, int P, const SuperSpan &k)
{
    if (k.e1 > k.e0 && (k.e0 < k.k0 || k.e1 > k.k1)) return false;
    return k.k1 <= k.k0 || (k.k0 >= l.first(P) && k.k1 <= l.first(P) + l.count(P));
}

int main()
{
    using namespace rns;
    for (int nr = 1; nr <= 24; nr++)
        for (int nc = 1; nc <= 24; nc++) {
            const Layout fm{kUpperRows, 2 * nr}, fn{kUpperCols, 2 * nc}, vr{kFull, 2 * nc}, vc{kFull, 2 * nr};
            if (!fills(fm, nr) || !fills(fn, nc) || !fills(vr, nr) || !fills(vc, nc)) return 1;
            for (int A = 0; A < nr; A++)
                for (int B = 0; B < nc; B++) {
                    const SuperSpan a = span_vn(false, A, B), b = span_mv(false, 2 * nr, A, B);
                    if (!holds(vr, A, a) || !holds(fn, B, a) || !holds(fm, A, b) || !holds(vc, B, b)) return 1;
                }
            if (nr != nc) continue;
            const Layout ur{kUpperRows, 2 * nr}, uc{kUpperCols, 2 * nr};
            for (int A = 0; A < nr; A++)
                for (int B = A + 1; B < nr; B++) {
                    const SuperSpan a = span_vn(true, A, B), b = span_mv(true, 2 * nr, A, B), c = span_uu(A, B);
                    if (!holds(ur, A, a) || !holds(fn, B, a) || !holds(fm, A, b) || !holds(uc, B, b) ||
                        !holds(ur, A, c) || !holds(uc, B, c))
                        return 1;
                }
        }
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
