// rns.cuh -- float64 products on the tensor cores through residues (rns.cu).
#pragma once

#include <cuda_bf16.h>

#include "internal.cuh"
#include "super_plan.h"

namespace signtri {
namespace rns {

// Pairwise coprime moduli; their product is 2^140.4.  (With the first 16 of
// them, 2^125.3, operands keep 55 bits at K = 8192 and their rounding is as large
// as that of float64 sums on ungraded data: no room for data that spreads.)
constexpr int kModulus[kMods] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193, 191, 181};
constexpr int kPanel = 128;                    // rows of a panel, and edge of a product tile
constexpr int kTileElems = kPanel * 64;        // one panel's K-block of 64, one modulus: 16 KB of bf16

// Bits kept of each operand entry below its row's (column's) power-of-two
// scale: sums of K products then stay below half the moduli's product.  62 up to
// K = 32768 (an entry's 53 bits whole down to 2^-9 of the scale), 61 up to
// 131072; no more than 62, so that a rounded entry fits 63 bits and its sign.
constexpr int operand_bits(int K)
{
    int lg = 0;
    while (lg < 30 && (1 << lg) < K) lg++;
    const int b = (139 - lg) / 2;
    return b < 62 ? b : 62;
}

constexpr size_t form_tile_bytes(const Layout &l, int panels) { return l.before(panels) * kMods * kTileElems * 2; }

// One 128 x 128 product: panel pa of source number `src`'s A form times panel pb of
// its B form over K-blocks [kb0, kb1), of which [e0, e1) may be summed ahead.
struct Tile {
    int src, pa, pb, kb0, kb1, e0, e1;
};
// grownA[pa], grownB[pb] (where not null): the panel has been converted anew
// since the K-blocks [e0, e1) were summed, so that sum is of no use.
struct Source {
    const __nv_bfloat16 *A, *B;
    Layout la, lb;
    const int *grownA, *grownB;
};

// Residues of tiles [0, ntiles) of d_tiles, `per` consecutive tiles sharing
// panels, in [tile][modulus][row][column], int8.
//   early: the K-blocks [e0, e1) alone, into `ahead`;
//   else:  all K-blocks, the ones in `ahead` (where not null) from there,
//          already multiplied by the modulus's cofactor inverse, into out.
signtri_status gemm(const Source *d_src, const Tile *d_tiles, int ntiles, int per, bool early, int8_t *ahead,
                    int8_t *out, int *d_err, int cls, cudaStream_t st);

}  // namespace rns
}  // namespace signtri
