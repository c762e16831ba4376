// Checks of level_split.h on the host: for every anti-diagonal the CTAs'
// ranges cover the K-blocks once and in order, none of a tile's partials is
// left unwritten (every CTA between a tile's first and last owns part of it),
// split_owner names the CTA whose range holds a K-block, and the slab numbers
// c + I stay below level_slabs.
#include <cstdio>

#include "level_split.h"

using namespace signtri::lvl;

static int check(int nb, int e, int stride, long long slabs)
{
    const Split s = make_split(nb - e, e, far_leaves(nb, e));
    if (split_start(s, 0) != 0 || split_start(s, s.G) != s.W) return 1;
    for (int c = 0; c < s.G; c++) {
        const long long len = split_start(s, c + 1) - split_start(s, c);
        if (len < 0 || (len == 0 && !(s.lam == 0 && c < s.L))) return 2;
    }
    int c = 0;
    for (long long x = 0; x < s.W; x += stride) {
        while (split_start(s, c + 1) <= x) c++;
        if (split_owner(s, x) != c) return 3;
        if (c + x / s.cpt >= slabs) return 4;
    }
    return 0;
}

int main()
{
    int n = 0;
    for (int nb = 2; nb <= 1024; nb = nb < 170 ? nb + 1 : nb + 61) {
        const long long slabs = (long long)level_slabs(nb * LB);
        for (int e = 1; e < nb; e += nb < 170 ? 1 : 7) {
            const int r = check(nb, e, nb < 100 ? 1 : 13, slabs);
            if (r) {
                printf("nb %d e %d: check %d\n", nb, e, r);
                return 1;
            }
            n++;
        }
    }
    printf("ok %d anti-diagonals\n", n);
    return 0;
}
