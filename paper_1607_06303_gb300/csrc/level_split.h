// level_split.h -- how one launch of ph_level.cuh shares its work: the early
// sums of a block anti-diagonal cut over the launch's CTAs.  Compiled for the
// device and the host; the tests compile it on its own.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define SGT_HD __host__ __device__
#else
#define SGT_HD
#endif

namespace signtri {
namespace lvl {

constexpr int LB = 16;   // block order

// Anti-diagonal e has tiles (nb - e of them in one matrix) of e + 1 K-blocks
// (K = I .. J), W in all, numbered tile by tile.  The launch has G CTAs, of which the first L solve
// a leaf first, worth about kLeafBlocks K-blocks of float64 work.  CTA c sums
// the K-blocks [start(c), start(c + 1)), the leaf CTAs fewer, so that all end
// together; when that leaves them fewer than kFarShare, they sum nothing and
// the others share W evenly, in ranges of about kFarShare at least (a tile's
// leaf adds its partials one after another, 128 cycles each).  One CTA (or as
// many as the leaves need) per SM: its sixteen warps keep the float64 pipes
// busy, and a leaf that shares them takes longer.  With more than kManyLeaves
// leaves (batches) every SM solves several in turn whatever the placement,
// and the sums go to kManyFar CTAs behind them.  The cut depends on sizes only, so results do not depend on the GPU.
constexpr int kSms = 152;
constexpr int kLeafBlocks = 5;
constexpr int kFarShare = 4;
constexpr int kManyLeaves = 4 * kSms;
constexpr int kManyFar = 16 * kSms;

struct Split {
    long long W;   // K-blocks
    int cpt;       // K-blocks per tile
    int L;         // CTAs that solve a leaf first
    int G;         // CTAs
    int lam;       // K-blocks a leaf counts for; 0: leaf CTAs sum nothing
};

SGT_HD constexpr Split make_split(int tiles, int e, int leaves)
{
    const int cpt = e + 1;
    Split s{(long long)tiles * cpt, cpt, leaves, kSms, kLeafBlocks};
    if (leaves > kManyLeaves) s.G = leaves + kManyFar;
    else while (s.G < leaves + kSms / 8) s.G += kSms;
    if (leaves > kManyLeaves || s.W + (long long)kLeafBlocks * leaves < (long long)(kLeafBlocks + kFarShare) * s.G) {
        long long g = s.G - leaves;
        const long long most = (long long)tiles * ((cpt + kFarShare - 1) / kFarShare);
        if (g > most) g = most;
        s.G = leaves + (int)g;
        s.lam = 0;
    }
    return s;
}

SGT_HD inline long long split_start(const Split &s, int c)
{
    if (s.lam) return c * (s.W + (long long)s.lam * s.L) / s.G - (long long)s.lam * (c < s.L ? c : s.L);
    return c <= s.L ? 0 : (c - s.L) * s.W / (s.G - s.L);
}

// the CTA that sums K-block x
SGT_HD inline int split_owner(const Split &s, long long x)
{
    int c;
    if (!s.lam) {
        c = s.L + (int)(x * (s.G - s.L) / s.W);
    } else {
        const long long V = s.W + (long long)s.lam * s.L;   // K-blocks and leaves together
        const long long xl = s.L * V / s.G - (long long)s.lam * s.L;   // start of the CTAs without a leaf
        c = x >= xl ? (int)((x + (long long)s.lam * s.L) * s.G / V) : (int)(x * s.G / (V - (long long)s.lam * s.G));
    }
    if (c >= s.G) c = s.G - 1;
    while (c > 0 && split_start(s, c) > x) c--;
    while (split_start(s, c + 1) <= x) c++;
    return c;
}

// leaf CTAs in the launch that forms the early sums of anti-diagonal e
SGT_HD constexpr int far_leaves(int nb, int e) { return e >= 2 ? nb - e + 1 : 0; }

// Slabs one anti-diagonal needs at most (CTA c's partial for tile I goes to
// slab c + I, so a tile's partials are consecutive); two sets are in use.
constexpr size_t level_slabs(int n)
{
    const int nb = (n + LB - 1) / LB;
    int most = 0;
    for (int e = 1; e < nb; e++) {
        const int g = make_split(nb - e, e, far_leaves(nb, e)).G + nb - e;
        if (g > most) most = g;
    }
    return (size_t)most;
}

// The same for any set of at most `tiles` tiles and `leaves` leaves.
SGT_HD constexpr size_t slabs_bound(long long tiles, long long leaves)
{
    return (size_t)(tiles + leaves + kManyFar + 2 * kSms);
}

}  // namespace lvl
}  // namespace signtri
