// Reads of the sweeps' log by apply_rotations_kernel, replayed on the host: logs of
// sweeps whose windows shrink, the last of them ending at the log's end, taken
// in runs of up to eight sweeps of one window as the kernel takes them.  Every
// read has to lie in its own sweep's record, and every rotation has to be read
// once.  Prints "ok <reads>".
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>

#include "apply_window.h"

using namespace signtri;

int main()
{
    std::mt19937 rng(5);
    long long reads = 0;
    for (int trial = 0; trial < 400; trial++) {
        struct Rec { int l, i; long long off; };
        std::vector<Rec> log;
        long long end = 0;
        int l = 0, i = 20 + (int)(rng() % 300);
        while (i > l + 1 && log.size() < 200) {
            const int nbul = 1 + (int)(rng() % 10);
            for (int b = 0; b < nbul; b++, end += i - l) log.push_back({l, i, end});
            i -= (int)(rng() % 40);                       // deflations at the window's end
            if (rng() % 3 == 0) l += (int)(rng() % 3);   // and at its start
        }
        std::vector<int> seen(end, 0);
        const int logged = (int)log.size();
        for (int w = 0; w < logged;) {
            int nb = 0;
            while (nb < 8 && w + nb < logged && log[w + nb].l == log[w].l && log[w + nb].i == log[w].i) nb++;
            const int L = log[w].i - log[w].l, steps = L + 2 + 2 * (nb - 1);
            for (int g = 0; g < 8; g++) {
                const Rec &r = log[std::min(w + g, logged - 1)];
                for (int t = -2 * g; t < steps - 2 * g + 2; t++) {   // u of the first load .. of the last one ahead
                    if (!apply_reads(g, nb, t, L)) continue;
                    const long long at = r.off + t - 1;
                    if (at < r.off || at >= r.off + (r.i - r.l) || at >= end) {
                        std::printf("FAIL trial %d: group %d of %d reads %lld beyond its sweep\n", trial, g, nb, at);
                        return 1;
                    }
                    seen[at]++;
                    reads++;
                }
            }
            w += nb;
        }
        if (std::count(seen.begin(), seen.end(), 1) != end) {
            std::printf("FAIL trial %d: a rotation not read once\n", trial);
            return 1;
        }
    }
    std::printf("ok %lld\n", reads);
    return 0;
}
