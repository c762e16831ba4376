// apply_window.h -- the rotations that apply_rotations_kernel (schur.cu) reads from
// the sweeps' log.  Compiled for the device and the host; the tests compile it
// on its own.
#pragma once

#ifdef __CUDACC__
#define SGT_APPLY_HD __host__ __device__ __forceinline__
#else
#define SGT_APPLY_HD inline
#endif

namespace signtri {

// Group g of four lanes takes sweep g of nb sweeps of one window, L rotations each;
// its step u = t - 2 g is a rotation for u = 1 .. L.  The groups beyond nb
// hold records of other windows, which may have fewer rotations left in the log:
// they read none.
SGT_APPLY_HD bool apply_reads(int g, int nb, int u, int L) { return g < nb && u >= 1 && u <= L; }

}  // namespace signtri
