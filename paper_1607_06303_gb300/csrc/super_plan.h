// super_plan.h -- what the superblocks' products (ph_super.cu, rns.cu) read and
// where it lies, and which calls run products of superblocks or of slices,
// whose waits have a bound and whose error word has then to be read.  Plain C++: compiled for the device code and, on its own, by the tests.
#pragma once

#include <cstddef>

#include "level_split.h"

namespace signtri {

constexpr int kSuperEdge = 128;   // superblock edge
inline int super_panels(int n) { return (n + kSuperEdge - 1) / kSuperEdge; }

// The Sylvester solve of an m x p unknown sums over other superblocks as soon as
// there are two of them.
inline bool sylvester_products(int m, int p) { return m > 0 && p > 0 && super_panels(m) + super_panels(p) > 2; }

// Parlett-Sylvester: that solve's products, and with swaps those of the
// back-transform (and of the blocked reorder).
inline bool ps_products(int npos, int nneg, long long swaps) { return swaps > 0 || sylvester_products(npos, nneg); }

namespace rns {

constexpr int kMods = 18;   // residues per entry (rns.cuh)

// The residues of a matrix cut into panels of 128 rows (a row form: rows of
// M) or of 128 columns (a column form: columns of M), K-contiguous, in tiles
// (panel, modulus, K-block) already in the 128-byte swizzle the MMA descriptor
// names.  An upper triangular M has K-blocks 2 P on in row panel P, 2 P + 1 and
// before in column panel P, and room for these only.
enum Shape { kFull = 0, kUpperRows = 1, kUpperCols = 2 };
struct Layout {
    int shape, nkb;   // nkb: K-blocks of a full panel
    SGT_HD constexpr int first(int P) const { return shape == kUpperRows ? 2 * P : 0; }
    SGT_HD constexpr int count(int P) const { return shape == kUpperRows ? nkb - 2 * P : shape == kUpperCols ? 2 * P + 2 : nkb; }
    // K-blocks of the panels before P
    SGT_HD constexpr size_t before(int P) const
    {
        const size_t p = (size_t)P;
        return shape == kUpperRows ? p * nkb - p * (P - 1) : shape == kUpperCols ? p * (P + 1) : p * nkb;
    }
    // the tile (P, modulus m, K-block kb); the next modulus's lies count(P) tiles on
    SGT_HD constexpr size_t tile(int P, int m, int kb) const
    {
        return before(P) * kMods + (size_t)m * count(P) + (kb - first(P));
    }
};

}  // namespace rns

// The K-blocks of one product of superblock (A, B), [k0, k1), of which [e0, e1) hold
// none of the level before and may be summed beside it: of V, that level solves
// the superblocks (A, B - 1) and (A + 1, B).
struct SuperSpan {
    int k0, k1, e0, e1;
};
// triangular V: from the diagonal superblock of the row and to that of the column,
// whose strictly upper parts are known; else over all of V's nkbr K-blocks of rows
// and every column before B.
SGT_HD constexpr SuperSpan span_vn(bool triangular, int A, int B)
{
    const int k0 = triangular ? 2 * A : 0;
    return {k0, 2 * B, k0, 2 * (B - 1)};
}
SGT_HD constexpr SuperSpan span_mv(bool triangular, int nkbr, int A, int B)
{
    const int k1 = triangular ? 2 * (B + 1) : nkbr;
    return {2 * (A + 1), k1, 2 * (A + 2), k1};
}
SGT_HD constexpr SuperSpan span_uu(int A, int B) { return {2 * (A + 1), 2 * B, 2 * (A + 2), 2 * (B - 1)}; }

}  // namespace signtri
