// super_plan.h -- which calls run products of superblocks (ph_super.cu) or of
// slices, whose waits have a bound and whose error word has then to be read.
// Plain C++: compiled for the device code and, on its own, by the tests.
#pragma once

namespace signtri {

constexpr int kSuperEdge = 128;   // superblock edge
inline int super_panels(int n) { return (n + kSuperEdge - 1) / kSuperEdge; }

// The Sylvester solve of an m x p unknown sums over other superblocks as soon as
// there are two of them.
inline bool sylvester_products(int m, int p) { return m > 0 && p > 0 && super_panels(m) + super_panels(p) > 2; }

// Parlett-Sylvester: that solve's products, and with swaps those of the
// back-transform (and of the blocked reorder).
inline bool ps_products(int npos, int nneg, long long swaps) { return swaps > 0 || sylvester_products(npos, nneg); }

}  // namespace signtri
