// complex.cu -- sign(T) of a complex upper triangular T, and the complex
// Schur route S = Q sign(T) Q^H (Section 1; Algorithm 3's first step takes a
// complex Schur form A = Q T Q^*).
//
// u_ii = sign(Re t_ii) (the sign function is defined off the imaginary axis,
// Section 1); for i < j, entry (i, j) of TU = UT (Eq. 1) or of U^2 = I
// (Eq. 2), exactly as for real T:
//   signs differ: u_ij = t_ij (u_ii - u_jj) / (t_ii - t_jj)
//                        + [sum_{i<k<j} (u_ik t_kj - t_ik u_kj)] / (t_ii - t_jj)
//   signs agree:  u_ij = -[sum_{i<k<j} u_ik u_kj] / (u_ii + u_jj)
// in complex float64 arithmetic, blocked as the real float64 path: blocks of
// 16, one launch per block anti-diagonal (ph_level.cuh, on double2 entries),
// bound by the float64 pipes.  (Entry by entry, one launch per element
// anti-diagonal, n = 1000 took 21 ms; blocked 3.3 ms.)
//
// The route's products W = U Q^H and S = Q W are complex: each is four real
// emulated-float64 tensor-core products of the real and imaginary planes
// (slices.cu), combined by small kernels.
//
// Layout: complex matrices are interleaved (re, im) float64 pairs,
// column-major, leading dimensions counted in complex elements (LAPACK's
// COMPLEX*16).
#include <algorithm>
#include <climits>

#include "internal.cuh"
#include "ph_level.cuh"

namespace signtri {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a / b by Smith's algorithm (R. L. Smith, CACM 5(8), 1962): scale by the
// larger of |Re b|, |Im b| so that no intermediate overflows needlessly
__device__ __forceinline__ double2 cdiv(double2 a, double2 b)
{
    if (fabs(b.x) >= fabs(b.y)) {
        const double r = b.y / b.x, den = b.x + b.y * r;
        return make_double2((a.x + a.y * r) / den, (a.y - a.x * r) / den);
    }
    const double r = b.x / b.y, den = b.x * r + b.y;
    return make_double2((a.x * r + a.y) / den, (a.y * r - a.x) / den);
}

// Diagonal check (first bad index: 4 i + status, as the real scan); strictly
// lower part of U zeroed.
__global__ void complex_init_kernel(int n, const double2 *__restrict__ T, int ldt, double2 *__restrict__ U, int ldu,
                                    int *__restrict__ bad)
{
    const int j = blockIdx.x;
    if (threadIdx.x == 0) {
        const double2 tjj = T[(size_t)j + (size_t)j * ldt];
        int key = INT_MAX;
        if (!isfinite(tjj.x) || !isfinite(tjj.y)) key = 4 * j + SIGNTRI_ERR_NONFINITE;
        else if (tjj.x == 0.0) key = 4 * j + SIGNTRI_ERR_ZERO_EIGENVALUE;
        if (key != INT_MAX) atomicMin(bad, key);
    }
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) SGT_AT(U, ldu, i, j) = make_double2(0.0, 0.0);
}

// Diagonal blocks of 16, by anti-diagonal: the products of all the
// anti-diagonal's terms spread over the threads, then each entry's sum and
// quotient by a thread of its own; the quotients that need no sum at the start.
__global__ void __launch_bounds__(lvl::LT)
complex_diag_kernel(int n, const double2 *__restrict__ T, int ldt, double2 *__restrict__ U, int ldu)
{
    using namespace lvl;
    __shared__ double2 Ts[BLK], Us[BLK], Pr[BLK], Q1[BLK];
    const int r0 = blockIdx.x * LB, bs = min(LB, n - r0);
    const int lo = threadIdx.x % LB, hi = threadIdx.x / LB, at = lo + hi * LD;
    const bool in = lo <= hi && hi < bs;
    const double2 zero = make_double2(0.0, 0.0);
    const double2 t = in ? SGT_AT(T, ldt, r0 + lo, r0 + hi) : zero;
    Ts[at] = t;
    Us[at] = lo == hi ? make_double2(t.x > 0.0 ? 1.0 : -1.0, 0.0) : zero;
    __syncthreads();
    {
        const double ui = Us[lo * (LD + 1)].x, uj = Us[hi * (LD + 1)].x;
        if (in && lo < hi && ui + uj == 0.0)
            Q1[at] = cdiv(scaled(t, ui - uj), csub(Ts[lo * (LD + 1)], Ts[hi * (LD + 1)]));
    }
    for (int d = 1; d < bs; d++) {
        const int terms = d - 1;
        if (terms > 0 && threadIdx.x < (bs - d) * terms) {   // at most 8 * 7 of them
            const int i = threadIdx.x / terms, k = i + 1 + threadIdx.x % terms, j = i + d;
            const bool opp = Us[i * (LD + 1)].x != Us[j * (LD + 1)].x;
            const double2 ik = Us[i + k * LD], kj = Us[k + j * LD];
            Pr[i * LD + (k - i - 1)] = opp ? csub(cmul(ik, Ts[k + j * LD]), cmul(Ts[i + k * LD], kj)) : cmul(ik, kj);
        }
        __syncthreads();
        if (threadIdx.x < bs - d) {
            const int i = threadIdx.x, j = i + d;
            double2 s = zero;
            for (int k = 0; k < terms; k++) s = cadd(s, Pr[i * LD + k]);
            const double uii = Us[i * (LD + 1)].x, ujj = Us[j * (LD + 1)].x;
            if (uii + ujj == 0.0)
                Us[i + j * LD] = cadd(Q1[i + j * LD], cdiv(s, csub(Ts[i * (LD + 1)], Ts[j * (LD + 1)])));
            else
                Us[i + j * LD] = scaled(s, -0.5 * uii);   // -s / (+-2)
        }
        __syncthreads();
    }
    if (in) SGT_AT(U, ldu, r0 + lo, r0 + hi) = Us[at];
}

// Real and imaginary planes of an n x n complex matrix (ld in complex
// elements); conj = 1 stores -Im.
__global__ void split_planes_kernel(int n, const double2 *__restrict__ M, int ldm, double *__restrict__ re,
                                    double *__restrict__ im)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double2 v = M[(size_t)i + (size_t)j * ldm];
        re[(size_t)i + (size_t)j * n] = v.x;
        im[(size_t)i + (size_t)j * n] = v.y;
    }
}

// out = a + sa * b (n x n planes, ld n)
__global__ void combine_kernel(int n, const double *__restrict__ a, const double *__restrict__ b, double sa,
                               double *__restrict__ out)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < (size_t)n * n) out[idx] = a[idx] + sa * b[idx];
}

// S = re + i im, interleaved, ld in complex elements
__global__ void join_planes_kernel(int n, const double *__restrict__ re, const double *__restrict__ im,
                                   double2 *__restrict__ S, int lds)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        S[(size_t)i + (size_t)j * lds] = make_double2(re[(size_t)i + (size_t)j * n], im[(size_t)i + (size_t)j * n]);
}

}  // namespace

size_t complex_workspace_bytes(int n)
{
    if (n <= 0) return 0;
    return lvl::level_workspace_bytes<double2>(n) + sizeof(int) + 256;
}

signtri_status complex_sign_run(int n, const double *T, int ldt, double *U, int ldu, Arena &ws, int *bad_index,
                                cudaStream_t st)
{
    if (n <= 0) return SIGNTRI_OK;
    auto *bad = static_cast<int *>(ws.take(sizeof(int)));
    if (!bad) return SIGNTRI_ERR_NO_WORKSPACE;
    const auto *Tc = reinterpret_cast<const double2 *>(T);
    auto *Uc = reinterpret_cast<double2 *>(U);
    const int big = INT_MAX;
    SGT_CUDA_TRY(cudaMemcpyAsync(bad, &big, sizeof(int), cudaMemcpyHostToDevice, st));
    {
        ProfScope ps(SIGNTRI_KC_SCAN, st);
        complex_init_kernel<<<n, kThreads, 0, st>>>(n, Tc, ldt, Uc, ldu, bad);
        SGT_LAUNCH_CHECK();
    }
    int key = INT_MAX;
    SGT_CUDA_TRY(cudaMemcpyAsync(&key, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
    SGT_CUDA_TRY(cudaStreamSynchronize(st));
    if (key != INT_MAX) {
        if (bad_index) *bad_index = key / 4;
        return (signtri_status)(key % 4);
    }
    {
        ProfScope ps(SIGNTRI_KC_DIAG_LEAF, st);
        complex_diag_kernel<<<(n + lvl::LB - 1) / lvl::LB, lvl::LT, 0, st>>>(n, Tc, ldt, Uc, ldu);
        SGT_LAUNCH_CHECK();
    }
    return lvl::launch_levels<false>(n, Tc, ldt, Uc, ldu, ws, st);
}

size_t complex_schur_workspace_bytes(int n)
{
    if (n <= 0) return 0;
    const size_t nn = (size_t)n * n * sizeof(double) + 256;
    return std::max(complex_workspace_bytes(n), 8 * nn + emulated_product_workspace_bytes(n, n, n));
}

signtri_status complex_schur_run(int n, const double *Q, int ldq, const double *T, int ldt, double *S, int lds,
                                 Arena &ws, int *d_err, int *bad_index, cudaStream_t st)
{
    if (n <= 0) return SIGNTRI_OK;
    // U = sign(T) into S (complex, ld lds), then the products by planes
    const size_t mark0 = ws.used;
    signtri_status rs = complex_sign_run(n, T, ldt, S, lds, ws, bad_index, st);
    if (rs != SIGNTRI_OK) return rs;
    ws.used = mark0;
    const size_t nn = (size_t)n * n;
    double *P[8];
    for (double *&p : P) {
        p = static_cast<double *>(ws.take(nn * sizeof(double)));
        if (!p) return SIGNTRI_ERR_NO_WORKSPACE;
    }
    double *Qr = P[0], *Qi = P[1], *Ur = P[2], *Ui = P[3], *Wr = P[4], *Wi = P[5], *X1 = P[6], *X2 = P[7];
    const size_t mark = ws.used;
    const unsigned cblocks = (unsigned)((nn + kThreads - 1) / kThreads);
    {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        split_planes_kernel<<<n, kThreads, 0, st>>>(n, reinterpret_cast<const double2 *>(Q), ldq, Qr, Qi);
        SGT_LAUNCH_CHECK();
        split_planes_kernel<<<n, kThreads, 0, st>>>(n, reinterpret_cast<const double2 *>(S), lds, Ur, Ui);
        SGT_LAUNCH_CHECK();
    }
    auto prod = [&](const double *A, const double *B, bool transB, double *C) -> signtri_status {
        ws.used = mark;
        return emulated_product(n, n, n, A, n, B, n, transB, C, n, false, SIGNTRI_KC_GEMM_F64, ws, d_err, st);
    };
    auto comb = [&](const double *a, const double *b, double sa, double *out) -> signtri_status {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        combine_kernel<<<cblocks, kThreads, 0, st>>>(n, a, b, sa, out);
        SGT_LAUNCH_CHECK();
        return SIGNTRI_OK;
    };
    // W = U Q^H: Wr = Ur Qr^T + Ui Qi^T, Wi = Ui Qr^T - Ur Qi^T
    if ((rs = prod(Ur, Qr, true, X1)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Ui, Qi, true, X2)) != SIGNTRI_OK) return rs;
    if ((rs = comb(X1, X2, 1.0, Wr)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Ui, Qr, true, X1)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Ur, Qi, true, X2)) != SIGNTRI_OK) return rs;
    if ((rs = comb(X1, X2, -1.0, Wi)) != SIGNTRI_OK) return rs;
    // S = Q W: Sr = Qr Wr - Qi Wi, Si = Qr Wi + Qi Wr (the U planes are free now)
    if ((rs = prod(Qr, Wr, false, X1)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Qi, Wi, false, X2)) != SIGNTRI_OK) return rs;
    if ((rs = comb(X1, X2, -1.0, Ur)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Qr, Wi, false, X1)) != SIGNTRI_OK) return rs;
    if ((rs = prod(Qi, Wr, false, X2)) != SIGNTRI_OK) return rs;
    if ((rs = comb(X1, X2, 1.0, Ui)) != SIGNTRI_OK) return rs;
    {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        join_planes_kernel<<<n, kThreads, 0, st>>>(n, Ur, Ui, reinterpret_cast<double2 *>(S), lds);
        SGT_LAUNCH_CHECK();
    }
    return SIGNTRI_OK;
}

}  // namespace signtri
