// schur.cu -- the complex Schur decomposition A = Q T Q^H of a general real A
// on the GPU: the first step of the paper's route to sign(A) = Q sign(T) Q^H
// for a general matrix (Section 1; Algorithm 3 starts from a complex Schur
// form).
//
// Two textbook stages (Golub and Van Loan, Matrix Computations, 4th ed.,
// Sections 7.4-7.5):
//  1. Householder reduction to upper Hessenberg form H = Q0^T A Q0, float64.
//     For column k a reflector P = I - tau v v^T (v_0 = 1) maps A[k+1:, k]
//     onto beta e_1; it is applied from the left to the columns right of k
//     and from the right to the rows of A.  Where A fits in a cluster's shared
//     memory one kernel runs all columns (hess_cluster_kernel), else four
//     launches a column; Q0's rows take the kept reflectors one by one in
//     form_q_kernel, beside the second stage.
//  2. Implicitly shifted QR iteration on H in complex float64.  A complex
//     shift needs no double-shift pairing, so every sweep over the active
//     window [l, i] is a chain of plane rotations: the first from
//     (h_ll - sigma, h_{l+1,l}), each later one zeroing the bulge
//     h_{k+1,k-1}; each rotation G acts on rows k, k+1 of H over all columns
//     and G^H on columns k, k+1 over the rows that hold nonzeros (so H
//     becomes all of T, not just its diagonal) and on Q's columns.  Up to ten
//     sweeps follow one another three rows apart, shifted by the eigenvalues
//     of the window's trailing block (by those of its trailing 2 x 2 where a
//     window is small or does not converge), with one ad hoc shift every tenth
//     time without a deflation; h_{k,k-1} is negligible, and set to 0, when
//     |h_{k,k-1}| <= eps (|h_{k-1,k-1}| + |h_kk|) (|z| = |Re z| + |Im z|).
//     Deflation takes the window's last row when its subdiagonal entry is
//     negligible.  The rotations of a sweep depend on one another (each reads
//     what the one before wrote), so one cluster of 16 CTAs (8 where the
//     device cannot place 16) runs the sweeps with a cluster barrier per step
//     of all its bulges, applying each rotation to the active window only
//     (schur_qr_kernel says how the work is split); a launch runs sweeps
//     until a rotation budget is spent and logs them, then a kernel on the
//     other SMs applies the logged rotations to the columns right of each
//     sweep's window and to Q, on a second stream while the next launch
//     runs, and the host relaunches until the window is empty.
//     The chain of steps bounds the stage: ~0.3 n^2 of ~3,300 cycles each
//     (n = 200: 21 of 29 ms; two bulges at a time took 1.0 n^2 of 6,000).
//
// Layout: A real column-major; Q, T complex interleaved (re, im) float64
// pairs, column-major, leading dimensions counted in complex elements.
#include <algorithm>
#include <cfloat>
#include <climits>

#include <cooperative_groups.h>

#include "apply_window.h"
#include "df_arith.cuh"
#include "internal.cuh"

namespace signtri {

namespace {

constexpr int kThreads = 256;
constexpr int kQrThreads = 256;
constexpr int kMaxSweepsPerEigenvalue = 100;
// rotations per launch of the QR kernel (then a sweep's end); the last launch's
// are applied alone, so fewer to a launch are better until the launches count
// (n = 64, 200, 400, ms: 2^11 6.31, 29.96, 110.5; 2^13 6.40, 29.75, 108.0; 2^15
// 7.08, 30.5)
constexpr long long kRotationBudget = 1LL << 13;
// rotations (and sweeps) a launch's log holds: two sweeps of a full window
// always fit
inline size_t rotation_room(int n) { return ((size_t)1 << 15) + 2 * (size_t)n + 2; }

#define SGT_A(M, ld, i, j) (M)[(size_t)(i) + (size_t)(j) * (size_t)(ld)]

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double cabs1(double2 a) { return fabs(a.x) + fabs(a.y); }
// The rotation G = [c s; -conj(s) c] (c real >= 0, c^2 + |s|^2 = 1) with
// G [x; y] = [r; 0]: c = |x| / nrm, s = (x / |x|) conj(y) / nrm,
// nrm^2 = |x|^2 + |y|^2.  x and y are first scaled by the power of two that
// brings their largest component into [1, 2) (exact), so the squares
// neither overflow nor lose range (below 2^-1000 the scale stops at 2^1000);
// then two reciprocal square roots and
// products (the rotation sits on the QR sweep's serial chain, where each
// float64 division or hypot costs a long dependent sequence).
__device__ __forceinline__ void make_rotation(double2 x, double2 y, double &c, double2 &s)
{
    const double my = fmax(fabs(y.x), fabs(y.y));
    if (my == 0.0) {
        c = 1.0;
        s = make_double2(0.0, 0.0);
        return;
    }
    const double m = fmax(my, fmax(fabs(x.x), fabs(x.y)));
    const double sc = ldexp(1.0, -max(ilogb(m), -1000));   // 2^1000 at most (m subnormal)
    const double2 xs = make_double2(x.x * sc, x.y * sc), ys = make_double2(y.x * sc, y.y * sc);
    const double ax2 = fma(xs.x, xs.x, xs.y * xs.y), ay2 = fma(ys.x, ys.x, ys.y * ys.y);
    if (ax2 == 0.0) {
        const double r = rsqrt(ay2);
        c = 0.0;
        s = make_double2(ys.x * r, -ys.y * r);
        return;
    }
    const double inv_n = rsqrt(ax2 + ay2), inv_ax = rsqrt(ax2);
    c = ax2 * inv_ax * inv_n;
    const double2 t = cmul(xs, cconj(ys));
    const double f = inv_ax * inv_n;
    s = make_double2(t.x * f, t.y * f);
}

// (a, b) of rows k, k+1 in one column -> G (a, b)
__device__ __forceinline__ void rot_rows(double c, double2 s, double2 &a, double2 &b)
{
    const double2 sa = cmul(s, b), sb = cmul(cconj(s), a);
    const double2 na = make_double2(c * a.x + sa.x, c * a.y + sa.y);
    const double2 nb = make_double2(c * b.x - sb.x, c * b.y - sb.y);
    a = na;
    b = nb;
}
// (a, b) of columns k, k+1 in one row -> (a, b) G^H
__device__ __forceinline__ void rot_cols(double c, double2 s, double2 &a, double2 &b)
{
    const double2 sa = cmul(cconj(s), b), sb = cmul(s, a);
    const double2 na = make_double2(c * a.x + sa.x, c * a.y + sa.y);
    const double2 nb = make_double2(c * b.x - sb.x, c * b.y - sb.y);
    a = na;
    b = nb;
}

// ------------------------------------------------------------- Hessenberg --

// First non-finite entry (its column) of A, into *bad (atomicMin).
__global__ void finite_check_kernel(int n, const double *__restrict__ A, int lda, int *__restrict__ bad)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (!isfinite(SGT_A(A, lda, i, j))) atomicMin(bad, j);
}

// H = A (a working copy)
__global__ void hess_init_kernel(int n, const double *__restrict__ A, int lda, double *__restrict__ H)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x) SGT_A(H, n, i, j) = SGT_A(A, lda, i, j);
}

__device__ __forceinline__ double block_sum(double x, double *red)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    const int w = threadIdx.x / 32, nw = blockDim.x / 32;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = x;
    __syncthreads();
    double s = 0.0;
    for (int k = 0; k < nw; k++) s += red[k];   // same order in every thread
    return s;
}

__device__ __forceinline__ double block_max(double x, double *red)
{
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
    const int w = threadIdx.x / 32, nw = blockDim.x / 32;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = x;
    __syncthreads();
    double s = 0.0;
    for (int k = 0; k < nw; k++) s = fmax(s, red[k]);
    return s;
}

// The reflector of column k: x = H[k+1:, k] (m = n - k - 1 entries),
// alpha = x_0, beta = -sign(alpha) ||x||, tau = (beta - alpha) / beta,
// v = x / (alpha - beta) with v_0 = 1; column k becomes (beta, 0, ...).
// tau = 0 (P = I) when x_1.. are all zero.  One CTA.
__global__ void house_kernel(int n, int k, double *__restrict__ H, double *__restrict__ v, double *__restrict__ tau)
{
    __shared__ double red[32];
    const int m = n - k - 1;
    double *x = &SGT_A(H, n, k + 1, k);
    double mx = 0.0;
    for (int i = 1 + threadIdx.x; i < m; i += blockDim.x) mx = fmax(mx, fabs(x[i]));
    mx = block_max(mx, red);
    if (mx == 0.0) {
        for (int i = threadIdx.x; i < m; i += blockDim.x) v[i] = (i == 0) ? 1.0 : 0.0;
        if (threadIdx.x == 0) *tau = 0.0;
        return;
    }
    // ||x_1..|| scaled by its largest magnitude (no overflow or underflow)
    double ss = 0.0;
    for (int i = 1 + threadIdx.x; i < m; i += blockDim.x) {
        const double t = x[i] / mx;
        ss = fma(t, t, ss);
    }
    ss = block_sum(ss, red);
    const double xnorm = mx * sqrt(ss);
    const double alpha = x[0];
    const double beta = -copysign(hypot(alpha, xnorm), alpha);
    const double scal = 1.0 / (alpha - beta);
    for (int i = threadIdx.x; i < m; i += blockDim.x) v[i] = (i == 0) ? 1.0 : x[i] * scal;
    __syncthreads();   // every x[i] read before column k is overwritten
    for (int i = threadIdx.x; i < m; i += blockDim.x) x[i] = (i == 0) ? beta : 0.0;
    if (threadIdx.x == 0) *tau = (beta - alpha) / beta;
}

// H[k+1:, j] -= tau v (v^T H[k+1:, j]) for the columns j > k: one CTA each.
__global__ void house_left_kernel(int n, int k, double *__restrict__ H, const double *__restrict__ v,
                                  const double *__restrict__ tau)
{
    __shared__ double red[32];
    const double t = *tau;
    if (t == 0.0) return;
    const int j = k + 1 + blockIdx.x;
    const int m = n - k - 1;
    double *col = &SGT_A(H, n, k + 1, j);
    double w = 0.0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) w = fma(v[i], col[i], w);
    w = block_sum(w, red) * t;
    for (int i = threadIdx.x; i < m; i += blockDim.x) col[i] = fma(-v[i], w, col[i]);
}

// The right application H[r, k+1:] -= tau (H[r, k+1:] v) v^T in two
// launches: y_r = tau H[r, k+1:] v with 32 rows per CTA (lane = row, so each column's 32 entries are one
// coalesced read) and the columns split over the 8 warps, then the rank-1
// update with a CTA per column.
constexpr int kGemvWarps = 8;
__global__ void __launch_bounds__(32 * kGemvWarps)
house_gemv_kernel(int n, int k, const double *__restrict__ H, const double *__restrict__ v,
                  const double *__restrict__ tau, double *__restrict__ y)
{
    __shared__ double part[kGemvWarps][32];
    const double t = *tau;
    if (t == 0.0) return;
    const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
    const int g = blockIdx.x * 32 + lane;
    const int m = n - k - 1;
    double acc = 0.0;
    if (g < n)
        for (int j = w; j < m; j += kGemvWarps) acc = fma(SGT_A(H, n, g, k + 1 + j), v[j], acc);
    part[w][lane] = acc;
    __syncthreads();
    if (w == 0 && g < n) {
        double sum = 0.0;
        for (int q = 0; q < kGemvWarps; q++) sum += part[q][lane];
        y[g] = t * sum;
    }
}

__global__ void house_rank1_kernel(int n, int k, double *__restrict__ H, const double *__restrict__ v,
                                   const double *__restrict__ tau, const double *__restrict__ y)
{
    if (*tau == 0.0) return;
    const int j = k + 1 + blockIdx.x;
    const double vj = v[blockIdx.x];
    for (int g = threadIdx.x; g < n; g += blockDim.x) SGT_A(H, n, g, j) = fma(-y[g], vj, SGT_A(H, n, g, j));
}

// The whole reduction in one cluster of CL CTAs with H in their shared
// memory (column j in CTA j % CL), where it fits (n up to 654 for 16 CTAs):
// per column the launches above took ~52 us at n = 200, most of it their
// starts and ends; here it is three cluster barriers and the float64 chains
// between them (~1 ms for all columns instead of 10.3).  Step k: the owner
// of column k forms the reflector (scaled by the power of two of its largest
// entry); every CTA fetches v, applies the reflector to its columns from the
// left (a warp per column) and sums its columns' share of H v; the shares
// are added by rows (16 lanes a row, a lane per CTA) and sent to every CTA,
// which updates its columns from the right.  v goes to V's column k (rows
// k+1..), tau to taus[k]; T = H, complex.
constexpr int kHessThreads = 512;
inline size_t hess_smem(int n, int cl) { return ((size_t)((n + cl - 1) / cl) * n + 3 * (size_t)n) * sizeof(double); }
constexpr size_t kHessSmemMax = 225 * 1024;

template <int CL>
__global__ void __launch_bounds__(kHessThreads)
hess_cluster_kernel(int n, const double *__restrict__ A, int lda, double2 *__restrict__ T, int ldt,
                    double *__restrict__ V, double *__restrict__ taus)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ double hess_sh[];
    constexpr int kWarps = kHessThreads / 32;
    __shared__ double red[kWarps], out[3];   // out: 1 / (alpha - beta), tau, beta (scaled)
    __shared__ int redi[kWarps];
    __shared__ double tau_own;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, me = (int)cl.block_rank();
    const int cols = (n + CL - 1) / CL;
    double *Hc = hess_sh, *v = Hc + (size_t)cols * n, *ypart = v + n, *y = ypart + n;
    for (int c = 0; me + c * CL < n; c++)
        for (int i = tid; i < n; i += kHessThreads) Hc[(size_t)c * n + i] = SGT_A(A, lda, i, me + c * CL);
    __syncthreads();
    for (int k = 0; k + 2 < n; k++) {
        const int owner = k % CL;
        if (me == owner) {
            double *x = Hc + (size_t)(k / CL) * n;
            int em = -1000, nz = 0;
            for (int i = k + 1 + tid; i < n; i += kHessThreads) {
                em = max(em, ((__double2hiint(x[i]) >> 20) & 0x7ff) - 1023);
                nz |= i > k + 1 && x[i] != 0.0;
            }
            em = __reduce_max_sync(0xffffffffu, em);
            if (lane == 0) redi[warp] = em;
            nz = __syncthreads_or(nz);
            if (nz) {
                em = min(__reduce_max_sync(0xffffffffu, redi[lane % kWarps]), 1000);
                const double sc = __hiloint2double((1023 - em) << 20, 0);
                double ss = 0.0;
                for (int i = k + 1 + tid; i < n; i += kHessThreads) {
                    const double t = x[i] * sc;
                    ss = fma(t, t, ss);
                }
                for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if (lane == 0) red[warp] = ss;
                __syncthreads();
                if (warp == 0) {
                    ss = lane < kWarps ? red[lane] : 0.0;
                    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                    const double alpha = x[k + 1] * sc;
                    const double beta = -copysign(sqrt(ss), alpha);
                    // lane 0: 1 / (alpha - beta); lane 1: (beta - alpha) / beta
                    const double d = lane ? beta : alpha - beta;
                    const double q = (lane ? beta - alpha : 1.0) / d;
                    if (lane < 2) out[lane] = q;
                    if (lane == 2) out[2] = beta * __hiloint2double((1023 + em) << 20, 0);
                }
                __syncthreads();
                const double scal = out[0];
                const double tau = out[1], beta = out[2];
                for (int i = k + 1 + tid; i < n; i += kHessThreads) {
                    const double vi = i == k + 1 ? 1.0 : x[i] * sc * scal;
                    v[i] = vi;
                    SGT_A(V, n, i, k) = vi;
                    x[i] = i == k + 1 ? beta : 0.0;
                }
                if (tid == 0) {
                    tau_own = tau;
                    taus[k] = tau;
                }
            } else if (tid == 0) {
                tau_own = 0.0;
                taus[k] = 0.0;
            }
        }
        cl.sync();
        const double tau = *cl.map_shared_rank(&tau_own, owner);
        if (me != owner) {
            const double *vo = cl.map_shared_rank(v, owner);
            for (int i = k + 1 + tid; i < n; i += kHessThreads) v[i] = vo[i];
        }
        if (tau == 0.0) continue;   // the same in every CTA
        __syncthreads();
        const int c0 = (k + 1 - me + CL - 1) / CL;   // the first of this CTA's columns right of k
        const int first = c0 > 0 ? c0 : 0;
        for (int c = first + warp; me + c * CL < n; c += kWarps) {
            double *x = Hc + (size_t)c * n;
            double w = 0.0;
            for (int i = k + 1 + lane; i < n; i += 32) w = fma(v[i], x[i], w);
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            w *= tau;
            for (int i = k + 1 + lane; i < n; i += 32) x[i] = fma(-v[i], w, x[i]);
        }
        __syncthreads();
        for (int r = tid; r < n; r += kHessThreads) {
            double a = 0.0;
            for (int c = first; me + c * CL < n; c++) a = fma(Hc[(size_t)c * n + r], v[me + c * CL], a);
            ypart[r] = a;
        }
        cl.sync();
        for (int r0 = me * (kHessThreads / CL); r0 < n; r0 += kHessThreads) {
            const int r = r0 + tid / CL, q = tid % CL;
            double a = r < n ? cl.map_shared_rank(ypart, q)[r] : 0.0;
            for (int o = CL / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (r < n) cl.map_shared_rank(y, q)[r] = tau * a;
        }
        cl.sync();
        for (int r = tid; r < n; r += kHessThreads) {
            const double yr = y[r];
            for (int c = first; me + c * CL < n; c++) {
                double &h = Hc[(size_t)c * n + r];
                h = fma(-yr, v[me + c * CL], h);
            }
        }
        __syncthreads();
    }
    for (int c = 0; me + c * CL < n; c++) {
        const int j = me + c * CL;
        for (int i = tid; i < n; i += kHessThreads)
            SGT_A(T, ldt, i, j) = make_double2(i <= j + 1 ? Hc[(size_t)c * n + i] : 0.0, 0.0);
    }
    cl.sync();   // no CTA leaves while another reads its shared memory
}

// Q = P_0 P_1 .. P_{n-3}, complex: a row of Q takes every reflector from the
// right by itself, so a warp per row runs through them without a barrier (lane
// owns the columns lane + 32 t), the row in shared memory or, above kQRowsMax,
// in `rows` (n x n).
constexpr int kFormWarps = 4;
constexpr int kQRowsMax = 5120;

__global__ void __launch_bounds__(32 * kFormWarps)
form_q_kernel(int n, const double *__restrict__ V, const double *__restrict__ taus, double *rows,
              double2 *__restrict__ Q, int ldq)
{
    extern __shared__ double form_sh[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = blockIdx.x * kFormWarps + warp;
    if (r >= n) return;
    double *q = n <= kQRowsMax ? form_sh + (size_t)warp * n : rows + (size_t)r * n;
    for (int i = lane; i < n; i += 32) q[i] = i == r ? 1.0 : 0.0;
    for (int k = 0; k + 2 < n; k++) {
        const double t = taus[k];
        if (t == 0.0) continue;
        const double *vk = V + (size_t)k * n;
        const int i0 = ((k + 1) & ~31) + lane;
        double w = 0.0;
        for (int i = i0; i < n; i += 32)
            if (i > k) w = fma(q[i], vk[i], w);
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        w *= t;
        for (int i = i0; i < n; i += 32)
            if (i > k) q[i] = fma(-w, vk[i], q[i]);
    }
    for (int i = lane; i < n; i += 32) SGT_A(Q, ldq, r, i) = make_double2(q[i], 0.0);
}

// complex T = H with its entries below the subdiagonal exactly 0
__global__ void to_complex_kernel(int n, const double *__restrict__ H, double2 *__restrict__ T, int ldt)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        SGT_A(T, ldt, i, j) = make_double2(i <= j + 1 ? SGT_A(H, n, i, j) : 0.0, 0.0);
}

// ---------------------------------------------------------- QR iteration --

struct QrState {
    int ihi;          // last row of the active window (-1: all converged)
    int its;          // sweeps since the last deflation
    int status;       // 0 running, 1 converged, 2 no convergence
    long long sweeps;
    long long rotations;
};

// A sweep of the last launch: its window [l, i] and where its i - l
// rotations start in the rotation log.
struct SweepRec {
    int l, i;
    long long off;
};

__global__ void qr_state_init_kernel(int n, QrState *st)
{
    st->ihi = n - 1;
    st->its = 0;
    st->status = 0;
    st->sweeps = 0;
    st->rotations = 0;
}

// One cluster of CL CTAs runs the sweeps, up to kMaxBulges bulges at a time,
// each started 3 steps behind the one before it: mathematically single-shift
// sweeps one after the other (the rotations of a front sweep that touch a
// rear bulge's rows and columns are all done before it gets there, and the
// later ones act on disjoint rows and columns), in 1 / kMaxBulges of the
// dependent steps.  Three bulges and more take the eigenvalues of the
// window's trailing block of as many rows as shifts (small_eigs, single
// precision: a shift only steers the convergence, to a factor ~1e-7 a sweep),
// two the eigenvalues of the trailing 2 x 2 in float64, which is also what a
// window goes back to after 6 sweeps without a deflation (a graded block's
// small eigenvalues are lost in single precision).
// A step is bounded by latencies.  A float64 instruction takes ~74 cycles and
// a warp has one in flight, an SM starts one every 16-20 cycles, so the kernel
// is laid out around the float64 instructions of its longest chain:
//  * a chief warp per bulge (kChiefs per CTA, in CTAs 0..kChiefCtas-1) runs
//    that chase's serial part: the 2 x 2 block at (k, k) and row k+2 of
//    columns k, k+1, where the next rotation's inputs (h_{k+1,k}, h_{k+2,k})
//    are formed, one real output per lane (8 lanes for G's action on the
//    block's two columns, 12 for G^H's on its three rows, 3 float64
//    instructions each), kept in registers from step to step; then the next
//    rotation (one reciprocal square root), stored into every CTA's shared
//    memory (two slots per bulge, alternating).  The one entry of the next
//    block that another thread writes, h_{k+1,k+2} (row op of column k+2),
//    comes through shared memory, and so do h_{k+2,k+2} and h_{k+3,k+2},
//    which the bulge in front wrote one and zero steps before (as its block's
//    corner and as the entry left of its block).
//  * a helper warp per bulge forms the entry left of the block (h_{k,k-1},
//    zeroing the old bulge), logs the rotation, and fetches from T what no
//    bulge in front hands on (for the front chase, and for the others once the
//    chase in front has ended), off the chief's chain.
//  * the other CTAs do the rest of every rotation: a warp takes 32 columns of
//    rows k, k+1 or 32 rows of columns k, k+1 of one bulge (whole warps of
//    one kind: mixed ones ran each kind's loads and arithmetic in turn), and
//    a few warps the 2 x 2 blocks at a rear bulge's rows and a front bulge's
//    columns, which take the rear rotation from the left and the front one
//    from the right.
// One cluster barrier per step; no entry is written by one thread while
// another reads it.  CTA 0 alone takes every decision (deflation, shifts,
// stop) and broadcasts it, so all CTAs run the same barriers.  Where T fits in
// the cluster's shared memory (kLocal, n up to 448 at 16 CTAs) its columns lie
// there, column j in CTA j % CL, for the launch's time: a read takes ~440 cycles
// instead of ~900 and the fence before a barrier ~500 instead of ~1,000.  Else T
// is read with L2-only loads (another CTA may have written it since).  The rotations'
// action on the columns right of the window (rows there are never read by a
// later sweep: the window only shrinks) and on Q is left to
// apply_rotations_kernel, which runs on other SMs alongside the next launch:
// this kernel logs each sweep and its rotations instead (a rear sweep after
// the one in front of it).
inline size_t qr_smem(int n, int cl) { return (size_t)((n + cl - 1) / cl) * (n | 1) * sizeof(double2); }
constexpr size_t kQrSmemMax = 200 * 1024;
// (8 bulges measured 30.3 ms for the sign of a general matrix at n = 200, 10
// 29.9, 12 29.6; at n = 400 111, 104 and 112)
constexpr int kMaxBulges = 10;
constexpr int kCross = kMaxBulges * (kMaxBulges - 1) / 2;   // pairs of bulges
constexpr int kCrossWarps = (kCross + 3) / 4;               // eight lanes per pair
enum { kActSweep = 0, kActStop = 2 };


// make_rotation for a chief warp, lane-parallel.  v: in every lane the
// operands of one product sum p q + u w, by lane & 3 of 0 |x|^2, 1 |y|^2,
// 2 Re x conj(y), 3 Im x conj(y).  With f = (|x|^2 (|x|^2 + |y|^2))^(-1/2):
// c = |x|^2 f, s = x conj(y) f, every lane's product its own output, passed
// by shuffles.  Only where x's and y's exponents lie in [-200, 200], so that
// no product leaves the normal range; else make_rotation.
__device__ __forceinline__ void make_rotation_warp(double p, double q, double u, double w, int lane, double &c,
                                                   double2 &s)
{
    const int em = max(exp_field(p), exp_field(u));   // lane 0: x's exponent, lane 1: y's
    const unsigned fine = __ballot_sync(0xffffffffu, em <= 200 && em >= -200);
    if ((fine & 3u) != 3u) {
        const double2 x = make_double2(__shfl_sync(0xffffffffu, p, 0), __shfl_sync(0xffffffffu, u, 0));
        const double2 y = make_double2(__shfl_sync(0xffffffffu, p, 1), __shfl_sync(0xffffffffu, u, 1));
        make_rotation(x, y, c, s);
        return;
    }
    const double val = fma(p, q, u * w);
    const double ax2 = __shfl_sync(0xffffffffu, val, 0), ay2 = __shfl_sync(0xffffffffu, val, 1);
    const double out = val * rsqrt_normal(ax2 * (ax2 + ay2));
    c = __shfl_sync(0xffffffffu, out, 0);
    s = make_double2(__shfl_sync(0xffffffffu, out, 2), __shfl_sync(0xffffffffu, out, 3));
}

// One real output of G or G^H acting on a pair, in one of the chief warp's
// lanes: out = c alpha + beta gamma + delta epsilon (3 float64 instructions).
__device__ __forceinline__ double pair_part(double c, double alpha, double beta, double gamma, double delta,
                                            double epsilon)
{
    return fma(c, alpha, fma(beta, gamma, delta * epsilon));
}

// The eigenvalues of [a b; c d]: with x = (a - d) / 2 and y = sqrt(x^2 + bc)
// signed so that |x + y| is the larger, the one nearer d is d - bc / (x + y)
// (Wilkinson's shift), the other a + d minus it.  Scaled by a power of two to
// entries of at most 2; roots and quotients by reciprocal square roots (a
// division or hypot is a long chain of float64 latencies).
__device__ __forceinline__ void wilkinson(double2 a, double2 b, double2 c, double2 d, double2 &near, double2 &other)
{
    int em = max(max(exp_field(a.x), exp_field(a.y)), max(exp_field(b.x), exp_field(b.y)));
    em = max(em, max(max(exp_field(c.x), exp_field(c.y)), max(exp_field(d.x), exp_field(d.y))));
    em = min(max(em, -1000), 1000);
    const double sc = __hiloint2double((1023 - em) << 20, 0);
    const double2 x = make_double2(0.5 * (a.x * sc - d.x * sc), 0.5 * (a.y * sc - d.y * sc));
    const double2 bc = cmul(make_double2(b.x * sc, b.y * sc), make_double2(c.x * sc, c.y * sc));
    const double2 xx = cmul(x, x);
    const double2 z = make_double2(xx.x + bc.x, xx.y + bc.y);
    // y = sqrt(z): with t = (|z| + |Re z|) / 2, sqrt(t) is the larger part,
    // Im z / (2 sqrt(t)) the other
    constexpr double kTiny = 0x1p-900;
    double2 y = make_double2(0.0, 0.0);
    const double z2 = fma(z.x, z.x, z.y * z.y);
    const double t = 0.5 * ((z2 > kTiny ? z2 * rsqrt(z2) : 0.0) + fabs(z.x));
    if (t > kTiny) {
        const double r = rsqrt(t), big = t * r, small = 0.5 * z.y * r;
        y = z.x >= 0.0 ? make_double2(big, small) : make_double2(fabs(small), copysign(big, z.y));
    }
    if (x.x * y.x + x.y * y.y < 0.0) y = make_double2(-y.x, -y.y);
    const double2 xy = make_double2(x.x + y.x, x.y + y.y);
    const double d2 = fma(xy.x, xy.x, xy.y * xy.y);
    near = d;
    if (d2 > kTiny) {
        const double r = rsqrt(d2), rr = r * r;
        const double2 q = cmul(bc, make_double2(xy.x * rr, -xy.y * rr));
        const double un = __hiloint2double((1023 + em) << 20, 0);
        near = make_double2(d.x - q.x * un, d.y - q.y * un);
    }
    other = make_double2(a.x + d.x - near.x, a.y + d.y - near.y);
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// A warp's eigenvalues of the m x m Hessenberg block h (entries of at most
// 2), in single precision: single-shift QR sweeps over the block's own
// window, a lane per column and then per row.  eig[q] is where the diagonal
// entry q converged; after 8 sweeps without a deflation the diagonal is taken
// as it stands (these are shifts: any value is valid).
__device__ void small_eigs(float2 (*h)[kMaxBulges + 1], int m, int lane, float2 *eig)
{
    int i = m - 1, its = 0;
    while (i >= 0) {
        bool small = false;
        if (lane >= 1 && lane <= i) {
            const float2 s = h[lane][lane - 1], u = h[lane - 1][lane - 1], v = h[lane][lane];
            small = fabsf(s.x) + fabsf(s.y) <= 1e-6f * (fabsf(u.x) + fabsf(u.y) + fabsf(v.x) + fabsf(v.y));
        }
        const unsigned mask = __ballot_sync(0xffffffffu, small);
        const int l = mask ? 31 - __clz((int)mask) : 0;
        if (l == i || its >= 8) {
            if (lane == 0) eig[i] = h[i][i];
            i--;
            if (its < 8) its = 0;
            continue;
        }
        const float2 a = h[i - 1][i - 1], b = h[i - 1][i], c = h[i][i - 1], d = h[i][i];
        const float2 x = make_float2(0.5f * (a.x - d.x), 0.5f * (a.y - d.y));
        const float2 bc = cmulf(b, c), xx = cmulf(x, x);
        const float2 z = make_float2(xx.x + bc.x, xx.y + bc.y);
        const float t = 0.5f * (sqrtf(z.x * z.x + z.y * z.y) + fabsf(z.x));
        float2 y = make_float2(0.0f, 0.0f);
        if (t > 0.0f) {
            const float r = rsqrtf(t), big = t * r, sm = 0.5f * z.y * r;
            y = z.x >= 0.0f ? make_float2(big, sm) : make_float2(fabsf(sm), copysignf(big, z.y));
        }
        if (x.x * y.x + x.y * y.y < 0.0f) y = make_float2(-y.x, -y.y);
        const float2 xy = make_float2(x.x + y.x, x.y + y.y);
        const float d2 = xy.x * xy.x + xy.y * xy.y;
        float2 sh = d;
        if (d2 > 0.0f) {
            const float2 q = cmulf(bc, make_float2(xy.x / d2, -xy.y / d2));
            sh = make_float2(d.x - q.x, d.y - q.y);
        }
        if (l == i - 1) {
            if (lane == 0) {
                eig[i] = sh;
                eig[i - 1] = make_float2(a.x + d.x - sh.x, a.y + d.y - sh.y);
            }
            i -= 2;
            its = 0;
            continue;
        }
        its++;
        for (int k = l; k < i; k++) {
            float2 p = h[k][max(k - 1, l)], q = h[k + 1][max(k - 1, l)];
            if (k == l) p = make_float2(p.x - sh.x, p.y - sh.y);
            const float p2 = p.x * p.x + p.y * p.y, q2 = q.x * q.x + q.y * q.y;
            float cc = 1.0f;
            float2 s = make_float2(0.0f, 0.0f);
            if (q2 > 1e-30f) {
                const float in = rsqrtf(p2 + q2);
                if (p2 > 1e-30f) {
                    const float ip = rsqrtf(p2);
                    cc = p2 * ip * in;
                    s = cmulf(p, make_float2(q.x, -q.y));
                    s = make_float2(s.x * ip * in, s.y * ip * in);
                } else {
                    cc = 0.0f;
                    s = make_float2(q.x * in, -q.y * in);
                }
            }
            __syncwarp();
            if (lane >= max(k - 1, l) && lane <= i) {
                const float2 u = h[k][lane], v = h[k + 1][lane];
                const float2 sv = cmulf(s, v), su = cmulf(make_float2(s.x, -s.y), u);
                h[k][lane] = make_float2(cc * u.x + sv.x, cc * u.y + sv.y);
                h[k + 1][lane] = make_float2(cc * v.x - su.x, cc * v.y - su.y);
            }
            __syncwarp();
            if (lane >= l && lane <= min(k + 2, i)) {
                const float2 u = h[lane][k], v = h[lane][k + 1];
                const float2 sv = cmulf(make_float2(s.x, -s.y), v), su = cmulf(s, u);
                h[lane][k] = make_float2(cc * u.x + sv.x, cc * u.y + sv.y);
                h[lane][k + 1] = make_float2(cc * v.x - su.x, cc * v.y - su.y);
            }
            __syncwarp();
        }
    }
    __syncwarp();
}

// The cluster barrier of a step: the warps that stored something order it
// before their arrival by a fence, the others do not wait for any memory
// (arriving with release semantics in every thread measured 850-1500 cycles
// at 16 CTAs, this 120 without stores, ~650 with stores to shared memory and
// ~1000 with stores to global memory).
__device__ __forceinline__ void step_barrier(bool wrote)
{
    if (wrote) asm volatile("fence.acq_rel.cluster;" ::: "memory");
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int CL, bool kLocal>
__global__ void __launch_bounds__(kQrThreads)
schur_qr_kernel(int n, double2 *__restrict__ T, int ldt, QrState *__restrict__ st, long long budget, long long room,
                SweepRec *__restrict__ sweeplog, double *__restrict__ rclog, double2 *__restrict__ rslog,
                int *__restrict__ nlogged)
{
    namespace cg = cooperative_groups;
    // Chief warps (and as many helpers) of a chief CTA: they share its float64
    // pipe, and the fewer they are, the fewer CTAs do the rest (kLocal, n = 200:
    // four 31.4 ms, three 30.2, two 30.1; n = 400: 109.8, 110.8, 113.8; from
    // global memory, n = 1000: 1,054, 1,096, 1,133)
    constexpr int kChiefs = kLocal ? 3 : 4, kChiefCtas = (kMaxBulges + kChiefs - 1) / kChiefs;
    constexpr int kWorkers = CL - kChiefCtas, kWarps = kQrThreads / 32, kWorkerWarps = kWorkers * kWarps;
    static_assert(kWorkers > 0 && kWarps >= 2 * kChiefs && kWorkerWarps >= kCrossWarps + kMaxBulges, "roles");
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ double2 tsm[];                      // kLocal: columns crank, crank + CL, .. of T
    __shared__ int redi[kWarps];
    __shared__ double rc[kMaxBulges][2];
    __shared__ double2 rs[kMaxBulges][2];
    __shared__ double2 bslot[kMaxBulges][2];              // h_{k+1,k+2} after a step, in the bulge's chief CTA
    __shared__ double inp[kMaxBulges][2][4];              // a rotation's inputs x, y, for the helper
    __shared__ double2 handF[kMaxBulges][4], handH[kMaxBulges][2];   // h_{k+2,k+2} a step ahead, h_{k+3,k+2} (four and two slots)
    __shared__ double2 sig[kMaxBulges];                   // the bulges' shifts
    __shared__ float2 blk[kMaxBulges][kMaxBulges + 1], eig[kMaxBulges];
    __shared__ int ctl[4];                                // action, l, i, bulges (CTA 0's decision)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int crank = (int)cl.block_rank();
    const int my = crank * kChiefs + warp % kChiefs;      // the bulge of a chief or helper warp
    const bool chief_cta = crank < kChiefCtas;
    const bool chief = chief_cta && warp < kChiefs && my < kMaxBulges;
    const bool helper = chief_cta && warp >= kChiefs && warp < 2 * kChiefs && my < kMaxBulges;
    const bool chief0 = crank == 0 && warp == 0;
    // a worker's warp number: consecutive ones alternate CTAs; the last
    // kCrossWarps take the pairs of bulges, eight lanes a pair
    const int w = warp * kWorkers + (crank - kChiefCtas);
    const bool crosser = !chief_cta && w >= kWorkerWarps - kCrossWarps;
    int pa = 0, pb = 0;                                   // this lane's pair: pa in front of pb
    if (crosser) {
        const int pair = (w - (kWorkerWarps - kCrossWarps)) * 4 + (lane >> 3);
        if (pair < kCross) {
            pb = 1;
            while (pair >= pb * (pb + 1) / 2) pb++;
            pa = pair - pb * (pb - 1) / 2;
        }
    }
    int i = st->ihi, its = st->its, status = st->status;
    const int lds = n | 1, ihi = i;
    auto entry = [&](int r, int c) -> double2 * {
        if constexpr (kLocal) return cl.map_shared_rank(tsm, c % CL) + (c / CL) * lds + r;
        else return &SGT_A(T, ldt, r, c);
    };
    auto ld = [&](const double2 *q) -> double2 {
        if constexpr (kLocal) return *q;
        else return __ldcg(q);
    };
    if constexpr (kLocal) {
        // the columns up to the window's last one: those right of it may be at
        // work in apply_rotations_kernel
        for (int c = crank; c <= ihi; c += CL)
            for (int r = tid; r < n; r += kQrThreads) tsm[(c / CL) * lds + r] = SGT_A(T, ldt, r, c);
        cl.sync();
    }
    long long logged = 0, rot = 0;
    const double eps = DBL_EPSILON;
    const double tiny = DBL_MIN * ((double)n / DBL_EPSILON);
    const double2 zero = make_double2(0.0, 0.0);
    const int part = lane & 3;
    const bool odd = part & 1, hi = part >= 2, col1 = (lane >> 2) & 1;
    const int row = min(lane >> 2, 2);
    // A chief warp's registers.  Lane 4 col + part forms the real output part
    // (0 top.x, 1 top.y, 2 bottom.x, 3 bottom.y) of G on the block's column
    // col ((A, E) or (B, F), the block (A B; E F) at (k, k)): al, ga, ep are
    // its operands in pair_part; ho, he are h_{k+2,k+1}'s part `odd` and the
    // other one; the step's rotation.
    double al = 0.0, ga = 0.0, ep = 0.0, ho = 0.0, he = 0.0, c_cur = 1.0;
    double2 s_cur = zero;
    auto as_double = [](double2 *q) { return reinterpret_cast<double *>(q); };
    const int po = odd ? 1 : 0, pe = odd ? 0 : 1;
    auto put_rotation = [&](int b, int slot) {
        // lanes 0..CL-1 of a chief warp store into CTA `lane`
        if (lane < CL) {
            *cl.map_shared_rank(&rc[b][slot], lane) = c_cur;
            *cl.map_shared_rank(&rs[b][slot], lane) = s_cur;
        }
    };
    // a chase's first block and rotation, at (l, l) with the shift sg
    auto start_chase = [&](int b, int slot, int l, int last, double2 sg) {
        const double2 top = ld(entry(l, l + (col1 ? 1 : 0)));
        const double2 bot = ld(entry(l + 1, l + (col1 ? 1 : 0)));
        const double2 A = ld(entry(l, l)), E = ld(entry(l + 1, l));
        if (b == 0) {
            const double2 H = (l + 2 <= last) ? ld(entry(l + 2, l + 1)) : zero;
            const double2 F = (l + 2 <= last) ? ld(entry(l + 2, l + 2)) : zero;
            if (lane == 0) handF[0][3] = F;
            ho = odd ? H.y : H.x;
            he = odd ? H.x : H.y;
        }
        const double2 u1 = hi ? bot : top, v1 = hi ? top : bot;
        al = odd ? u1.y : u1.x;
        ga = odd ? v1.y : v1.x;
        ep = odd ? v1.x : v1.y;
        const double2 X = make_double2(A.x - sg.x, A.y - sg.y);
        const double2 v = part == 1 ? E : X, u = part == 0 ? X : E;
        // parts 0, 1: v.x v.x + v.y v.y; 2: X.x E.x + X.y E.y; 3: X.y E.x - X.x E.y
        make_rotation_warp(part == 3 ? X.y : v.x, part < 2 ? v.x : u.x, part == 3 ? -X.x : v.y, part < 2 ? v.y : u.y,
                           lane, c_cur, s_cur);
        put_rotation(b, slot);
    };
    for (;;) {
        if (crank == 0) {
            int l;
            for (;;) {
                // l: the largest k in [1, i] whose h_{k,k-1} is negligible, else 0
                int lk = 0;
                for (int k = 1 + tid; k <= i; k += kQrThreads) {
                    const double sub = cabs1(ld(entry(k, k - 1)));
                    const double ref = cabs1(ld(entry(k - 1, k - 1))) + cabs1(ld(entry(k, k)));
                    if (sub <= fmax(eps * ref, tiny)) lk = k;
                }
                lk = __reduce_max_sync(0xffffffffu, lk);
                if (lane == 0) redi[warp] = lk;
                __syncthreads();
                l = __reduce_max_sync(0xffffffffu, lane < kWarps ? redi[lane] : 0);
                __syncthreads();
                if (status != 0 || i <= 0 || l < i) break;
                // the window's last row has converged
                if (tid == 0) *entry(i, i - 1) = zero;
                i--;
                its = 0;
            }
            if (chief0) {
                int act = kActSweep, nbul = 1;
                if (status != 0 || i <= 0) {
                    act = kActStop;
                    if (status == 0) {
                        status = 1;
                        i = -1;
                    }
                } else if (rot >= budget || (rot > 0 && rot + (long long)kMaxBulges * (i - l) > room)) {
                    act = kActStop;
                } else if (its >= kMaxSweepsPerEigenvalue) {
                    act = kActStop;
                    status = 2;
                } else {
                    if (l > 0 && lane == 0) *entry(l, l - 1) = zero;
                    const int sw_its = its + 1;
                    double2 sigma;
                    if (sw_its % 10 == 0) {
                        // ad hoc shift, one bulge: off the window's top
                        // (sweeps 10, 30, ..) or bottom corner (20, 40, ..)
                        // by 3/4 of a subdiagonal entry's real part
                        const bool top = (sw_its / 10) % 2 == 1;
                        const double2 d = top ? ld(entry(l, l)) : ld(entry(i, i));
                        const double e = top ? ld(entry(l + 1, l)).x : ld(entry(i, i - 1)).x;
                        sigma = make_double2(d.x + 0.75 * fabs(e), d.y);
                    } else {
                        // a bulge per three rows; two where the log has no
                        // room for more
                        if (i - l >= 3) nbul = sw_its > 6 ? 2 : min(kMaxBulges, max(2, (i - l + 1) / 3));
                        if ((long long)nbul * (i - l) > room) nbul = min(nbul, 2);
                        if (nbul <= 2) {
                            double2 other;
                            wilkinson(ld(entry(i - 1, i - 1)), ld(entry(i - 1, i)),
                                      ld(entry(i, i - 1)), ld(entry(i, i)), sigma, other);
                            if (lane < kChiefCtas) *cl.map_shared_rank(&sig[1], lane) = other;
                        } else {
                            const int r0 = i - nbul + 1;
                            int em = -1000;
                            for (int t = lane; t < nbul * nbul; t += 32) {
                                const int r = t % nbul, q = t / nbul;
                                if (r > q + 1) continue;
                                const double2 v = ld(entry(r0 + r, r0 + q));
                                em = max(em, max(exp_field(v.x), exp_field(v.y)));
                            }
                            em = min(__reduce_max_sync(0xffffffffu, em), 1000);
                            const double sc = __hiloint2double((1023 - em) << 20, 0);
                            for (int t = lane; t < nbul * nbul; t += 32) {
                                const int r = t % nbul, q = t / nbul;
                                const double2 v = r > q + 1 ? zero : ld(entry(r0 + r, r0 + q));
                                blk[r][q] = make_float2((float)(v.x * sc), (float)(v.y * sc));
                            }
                            __syncwarp();
                            small_eigs(blk, nbul, lane, eig);
                            // the last row's eigenvalue goes first
                            const double un = __hiloint2double((1023 + em) << 20, 0);
                            if (lane < nbul) {
                                const float2 v = eig[nbul - 1 - lane];
                                const double2 sg = make_double2(v.x * un, v.y * un);
                                for (int r = 0; r < kChiefCtas; r++) *cl.map_shared_rank(&sig[lane], r) = sg;
                            }
                            const float2 v0 = eig[nbul - 1];
                            sigma = make_double2(v0.x * un, v0.y * un);
                        }
                    }
                    start_chase(0, 0, l, i, sigma);
                    if (lane < nbul) sweeplog[logged + lane] = SweepRec{l, i, rot + (long long)lane * (i - l)};
                }
                if (lane < CL) {
                    int *rem = cl.map_shared_rank(ctl, lane);
                    rem[0] = act;
                    rem[1] = l;
                    rem[2] = i;
                    rem[3] = nbul;
                }
            }
        }
        cl.sync();
        const int act = ctl[0], l = ctl[1], nbul = ctl[3];
        i = ctl[2];
        if (act == kActStop) break;
        its++;
        const int L = i - l, S = L + 3 * (nbul - 1);
        // this worker warp's bulge, its first piece of 32 there and the stride
        const int wq = (kWorkerWarps - kCrossWarps) / nbul;
        const int wb = w % nbul;
        const bool worker = !chief_cta && w < wq * nbul;
        for (int s = 0; s < S; s++) {
            bool wrote = false;   // this warp has stores for the others to see
            if (worker) {
                const int k = l + s - 3 * wb;
                if (s >= 3 * wb && s < L + 3 * wb) {
                    const double c0 = rc[wb][s & 1];
                    const double2 s0 = rs[wb][s & 1];
                    const int rw = (i - k - 1 + 31) >> 5, cw = (k + 31) >> 5;
                    wrote = true;
                    for (int q = w / nbul; q < rw + cw; q += wq) {
                        if (q < rw) {
                            // rows k, k+1 at column j, but for the columns of
                            // the bulges in front, k + 3 t and k + 3 t + 1
                            const int d = 2 + (q << 5) + lane, j = k + d, t = d / 3;
                            const bool cross = d >= 3 && t <= wb && d - 3 * t < 2 && s < L + 3 * (wb - t);
                            if (j <= i && !cross) {
                                double2 a = ld(entry(k, j)), b = ld(entry(k + 1, j));
                                rot_rows(c0, s0, a, b);
                                *entry(k, j) = a;
                                *entry(k + 1, j) = b;
                                if (d == 2) *cl.map_shared_rank(&bslot[wb][(s + 1) & 1], wb / kChiefs) = b;
                            }
                        } else {
                            // columns k, k+1 at row r < k, but for the rows of
                            // the bulges behind, k - 3 t and k - 3 t + 1
                            const int r = ((q - rw) << 5) + lane, g = k - r + 1, t = g / 3;
                            const bool cross = t >= 1 && t <= nbul - 1 - wb && g - 3 * t < 2 && k - 3 * t >= l;
                            if (r < k && !cross) {
                                double2 a = ld(entry(r, k)), b = ld(entry(r, k + 1));
                                rot_cols(c0, s0, a, b);
                                *entry(r, k) = a;
                                *entry(r, k + 1) = b;
                            }
                        }
                    }
                }
            } else if (crosser) {
                // lane 4 f + part of a pair's eight: column k0 + f through the
                // rear rotation, then row k1 + f through the front one, an
                // output each (as in the chief's block)
                const int k0 = l + s - 3 * pa, k1 = l + s - 3 * pb, f = (lane >> 2) & 1;
                const bool on = pb > pa && pb < nbul && s >= 3 * pb && s < L + 3 * pa;
                wrote = __any_sync(0xffffffffu, on);
                if (wrote) {
                    double2 a = zero, b = zero, sr = zero, sc = zero;
                    double cr = 1.0, cc = 1.0;
                    if (on) {
                        a = ld(entry(k1, k0 + f));
                        b = ld(entry(k1 + 1, k0 + f));
                        cr = rc[pb][s & 1];
                        sr = rs[pb][s & 1];
                        cc = rc[pa][s & 1];
                        sc = rs[pa][s & 1];
                    }
                    const double2 u = hi ? b : a, v = hi ? a : b;
                    const double r1 = pair_part(cr, odd ? u.y : u.x, hi ? -sr.x : sr.x, odd ? v.y : v.x,
                                                odd ? sr.y : -sr.y, odd ? v.x : v.y);
                    // row f: part of its entry in column k0 (lanes 2 f + .. of
                    // the pair) and in column k0 + 1 (4 lanes on)
                    const int at = (lane & 24) + 2 * f + po + (hi ? 0 : 4);
                    const double g2 = __shfl_sync(0xffffffffu, r1, at), e2 = __shfl_sync(0xffffffffu, r1, at ^ 1);
                    const double a2 = __shfl_sync(0xffffffffu, r1, at ^ 4);
                    const double r2 = pair_part(cc, a2, hi ? -sc.x : sc.x, g2, odd ? -sc.y : sc.y, e2);
                    if (on) as_double(entry(k1 + f, k0 + (part >> 1)))[part & 1] = r2;
                }
            } else if (chief && my < nbul) {
                const int b = my, kb = l + s - 3 * b;
                if (b > 0 && s == 3 * b - 1) {
                    // this chase starts next step at (l, l): entries final
                    // since the last step (h_{l+2,l+1} comes after this step,
                    // from the bulge in front)
                    start_chase(b, (s + 1) & 1, l, i, sig[b]);
                    wrote = true;
                } else if (s >= 3 * b && s < L + 3 * b) {
                    const double c = c_cur;
                    const double2 sn = s_cur;
                    wrote = true;
                    // G on the block's columns
                    const double bx = hi ? -sn.x : sn.x, dy = odd ? sn.y : -sn.y;
                    const double r1 = pair_part(c, al, bx, ga, dy, ep);
                    // G^H on the rows k, k+1, k+2: lane 4 row + part gives part
                    // (0 p.x, 1 p.y, 2 q.x, 3 q.y) of row (p, q): the block's
                    // two rows after G, and (0, h_{k+2,k+1})
                    const int sp = (2 * row + po + (hi ? 0 : 4)) & 31;
                    double g2 = __shfl_sync(0xffffffffu, r1, sp), e2 = __shfl_sync(0xffffffffu, r1, sp ^ 1);
                    double a2 = __shfl_sync(0xffffffffu, r1, sp ^ 4);
                    if (row == 2) {
                        a2 = hi ? ho : 0.0;
                        g2 = hi ? 0.0 : ho;
                        e2 = hi ? 0.0 : he;
                    }
                    const double r2 = pair_part(c, a2, bx, g2, -dy, e2);
                    if (kb + 2 <= i) {
                        // the next rotation zeroes the bulge h_{k+2,k} (lanes 8, 9)
                        // against h_{k+1,k} (lanes 4, 5)
                        const double p = __shfl_sync(0xffffffffu, r2, part == 1 ? 8 : (part == 3 ? 5 : 4));
                        const double q = __shfl_sync(0xffffffffu, r2, part == 0 ? 4 : 8);
                        double u = __shfl_sync(0xffffffffu, r2, part == 1 ? 9 : (part == 3 ? 4 : 5));
                        const double v = __shfl_sync(0xffffffffu, r2, part == 0 ? 5 : 9);
                        if (part == 3) u = -u;
                        // what r2 holds already goes out before the rotation is
                        // formed, so that the barrier does not wait for it
                        if (lane < 12) as_double(entry(kb + (lane >> 2), kb + (part >> 1)))[part & 1] = r2;
                        if (lane == 4 || lane == 5 || lane == 8 || lane == 9)
                            inp[b][(s + 1) & 1][(lane & 1) | (lane >> 2 & 2)] = r2;
                        // the block's corner h_kk, for the bulge behind
                        if (lane < 2 && b + 1 < nbul)
                            as_double(cl.map_shared_rank(&handF[b + 1][s & 3], (b + 1) / kChiefs))[lane] = r2;
                        make_rotation_warp(p, q, u, v, lane, c_cur, s_cur);
                        put_rotation(b, (s + 1) & 1);
                        // the next block's first column, (h_{k+1,k+1}, h_{k+2,k+1})
                        // (lanes 6, 7 and 10, 11); its second one after the barrier
                        al = __shfl_sync(0xffffffffu, r2, (hi ? 10 : 6) + po);
                        ga = __shfl_sync(0xffffffffu, r2, (hi ? 6 : 10) + po);
                        ep = __shfl_sync(0xffffffffu, r2, (hi ? 6 : 10) + pe);
                    } else {
                        if (lane < 8) as_double(entry(kb + (lane >> 2), kb + (part >> 1)))[part & 1] = r2;
                        if (lane < 2 && b + 1 < nbul)
                            as_double(cl.map_shared_rank(&handF[b + 1][s & 3], (b + 1) / kChiefs))[lane] = r2;
                    }
                }
            } else if (helper && my < nbul) {
                const int b = my, kb = l + s - 3 * b;
                if (s >= 3 * b && s < L + 3 * b) {
                    const double c = rc[b][s & 1];
                    const double2 sn = rs[b][s & 1];
                    wrote = true;
                    if (lane == 0) {
                        const long long at = rot + (long long)b * L + (kb - l);
                        rclog[at] = c;
                        rslog[at] = sn;
                    }
                    if (kb > l && lane < 4) {
                        // h_{k,k-1} = c x + s y (the entry the rotation keeps,
                        // lanes 0, 1), h_{k+1,k-1} = 0 (the bulge it zeroes)
                        const double *xy = inp[b][s & 1];
                        const double rz = pair_part(c, odd ? xy[1] : xy[0], sn.x, odd ? xy[3] : xy[2],
                                                    odd ? sn.y : -sn.y, odd ? xy[2] : xy[3]);
                        reinterpret_cast<double *>(entry(kb + (hi ? 1 : 0), kb - 1))[odd ? 1 : 0] =
                            hi ? 0.0 : rz;
                        if (lane < 2 && b + 1 < nbul)
                            as_double(cl.map_shared_rank(&handH[b + 1][s & 1], (b + 1) / kChiefs))[lane] = rz;
                    }
                    if ((b == 0 || s >= L + 3 * (b - 1)) && kb + 3 <= i && lane >= 4 && lane < 6) {
                        // the front chase, or the one in front has ended (its
                        // last entries, a step old)
                        if (lane == 4)
                            handF[b][s & 3] = ld(entry(kb + 3, kb + 3));
                        else
                            handH[b][s & 1] = ld(entry(kb + 3, kb + 2));
                    }
                }
            }
            step_barrier(wrote);
            if (chief && my < nbul) {
                const int b = my;
                const bool on = s >= 3 * b && s < L + 3 * b;
                if (on && col1) {
                    // the block's second column for the next step:
                    // (h_{k+1,k+2}, h_{k+2,k+2})
                    const double *bs = as_double(&bslot[b][(s + 1) & 1]), *hf = as_double(&handF[b][(s - 1) & 3]);
                    al = (hi ? hf : bs)[po];
                    ga = (hi ? bs : hf)[po];
                    ep = (hi ? bs : hf)[pe];
                }
                if (on || s == 3 * b - 1) {
                    // h_{k+3,k+2} (h_{l+2,l+1} before the first step)
                    const double *hh = as_double(&handH[b][s & 1]);
                    ho = hh[po];
                    he = hh[pe];
                }
            }
        }
        rot += (long long)nbul * L;
        logged += nbul;
    }
    if constexpr (kLocal) {   // every CTA's stores are in: the barrier of the decision to stop
        for (int c = crank; c <= ihi; c += CL)
            for (int r = tid; r < n; r += kQrThreads) SGT_A(T, ldt, r, c) = tsm[(c / CL) * lds + r];
    }
    if (chief0 && lane == 0) {
        st->ihi = i;
        st->its = its;
        st->status = status;
        *nlogged = (int)logged;
        st->sweeps += logged;
        st->rotations += rot;
    }
}

// The logged sweeps' rotations where schur_qr_kernel left them out: unit u
// < n is column u of T, which takes the row rotations of every sweep whose
// window ends above it (u > i), down the column with the carried row; unit
// u >= n is row u - n of Q, which takes every sweep's column rotations along
// the row.  In log order, so each entry sees its rotations in the order of
// the QR iteration.  The chain of rotations along a line bounds this kernel,
// so a warp per line runs up to eight consecutive sweeps of one window in a
// wavefront: group g of four lanes takes sweep g two steps behind group g - 1,
// whose finished entry it gets by shuffles; group 0 reads the line, the last
// one writes it.  Each lane computes one real output of a rotation (3 float64
// instructions, 24 lanes' rotations in one).  The next steps' rotations and
// entries are loaded two steps ahead.
__global__ void __launch_bounds__(kThreads)
apply_rotations_kernel(int n, double2 *T, int ldt, double2 *Q, int ldq, const int *__restrict__ nlogged,
                       const SweepRec *__restrict__ sweeplog, const double *__restrict__ rclog,
                       const double2 *__restrict__ rslog)
{
    const int unit = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (unit >= 2 * n) return;   // a warp's lanes leave together
    const int g = lane >> 2, part = lane & 3, base = lane & 28;
    const bool odd = part & 1, hi = part >= 2;
    const bool isT = unit < n;
    // entry k of the unit's line: T(k, j) (stride 1) or Q(r, k) (stride ldq)
    double2 *line = isT ? &SGT_A(T, ldt, 0, unit) : &SGT_A(Q, ldq, unit - n, 0);
    const size_t stride = isT ? 1 : (size_t)ldq;
    const int logged = *nlogged;
    const double2 zero = make_double2(0.0, 0.0);
    for (int w = 0; w < logged;) {
        const int mine = min(w + g, logged - 1);
        const SweepRec sr = sweeplog[mine], s0 = {__shfl_sync(0xffffffffu, sr.l, 0), __shfl_sync(0xffffffffu, sr.i, 0), 0};
        const unsigned same = __ballot_sync(0xffffffffu, w + g < logged && sr.l == s0.l && sr.i == s0.i);
        const int nb = __ffs((int)~same) == 0 ? 8 : (__ffs((int)~same) - 1) >> 2;   // sweeps of this window in a row
        w += nb;
        if (isT && unit <= s0.i) continue;
        const int l = s0.l, L = s0.i - s0.l;
        // step t of group g: u = t - 2 g; u = 0 takes the entry l over, u in
        // [1, L] is rotation l + u - 1, u = L + 1 passes the last entry on
        auto load_c = [&](int u) { return apply_reads(g, nb, u, L) ? rclog[sr.off + u - 1] : 1.0; };
        auto load_s = [&](int u) { return apply_reads(g, nb, u, L) ? rslog[sr.off + u - 1] : zero; };
        auto load_e = [&](int t) { return g == 0 && t <= L ? line[(size_t)(l + t) * stride] : zero; };
        double r = 0.0;
        double c0 = load_c(-2 * g), c1 = load_c(1 - 2 * g);
        double2 q0 = load_s(-2 * g), q1 = load_s(1 - 2 * g);
        double2 e0 = load_e(0), e1 = load_e(1);
        const int steps = L + 2 + 2 * (nb - 1);
        for (int t = 0; t < steps; t++) {
            const int u = t - 2 * g;
            const double c = c0;
            const double2 s = q0, e = e0;
            c0 = c1;
            q0 = q1;
            e0 = e1;
            c1 = load_c(u + 2);
            q1 = load_s(u + 2);
            e1 = load_e(t + 2);
            // the carried entry a (this group's parts 2, 3) and the incoming b
            // (parts 0, 1 of the group in front), each as its part `odd` and
            // the other one
            const double ao = __shfl_sync(0xffffffffu, r, base + 2 + (odd ? 1 : 0));
            const double ae = __shfl_sync(0xffffffffu, r, base + 2 + (odd ? 0 : 1));
            double bo = __shfl_sync(0xffffffffu, r, (base + 28 + (odd ? 1 : 0)) & 31);
            double be = __shfl_sync(0xffffffffu, r, (base + 28 + (odd ? 0 : 1)) & 31);
            if (g == 0) {
                bo = odd ? e.y : e.x;
                be = odd ? e.x : e.y;
            }
            // G (T's rows) or G^H (Q's columns) on (a, b): lane part gives
            // part 0 a'.x, 1 a'.y, 2 b'.x, 3 b'.y
            const double sy = isT == odd ? s.y : -s.y;
            const double v = pair_part(c, hi ? bo : ao, hi ? -s.x : s.x, hi ? ao : bo, sy, hi ? ae : be);
            r = u >= 1 && u <= L ? v : (hi ? bo : ao);
            if (g == nb - 1 && u >= 1 && u <= L + 1 && !hi)
                reinterpret_cast<double *>(&line[(size_t)(l + u - 1) * stride])[part] = r;
        }
        __syncwarp();   // the next window's reads of entries other lanes wrote
    }
}

// T's strictly lower part -> 0 (what remains there is at most negligible)
__global__ void clear_lower_kernel(int n, double2 *__restrict__ T, int ldt)
{
    const int j = blockIdx.x;
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) SGT_A(T, ldt, i, j) = make_double2(0.0, 0.0);
}

__global__ void real_part_kernel(int n, const double2 *__restrict__ Sc, double *__restrict__ S, int lds)
{
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x) SGT_A(S, lds, i, j) = SGT_A(Sc, n, i, j).x;
}

}  // namespace

namespace {

// The cluster of the QR sweeps and of the reduction to Hessenberg form: 16
// CTAs (a non-portable size: the float64 pipes of the CTAs bound the work
// beside the chains) where the device can place such a cluster of both
// kernels, else 8.
cudaLaunchConfig_t cluster_config(int cl, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute *at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

bool places_16(const void *kernel, int threads, size_t smem)
{
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = cluster_config(16, threads, smem, nullptr, at);
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= 1)
        return true;
    cudaGetLastError();
    return false;
}

int cluster_size()
{
    return places_16((const void *)schur_qr_kernel<16, false>, kQrThreads, 0) &&
                   places_16((const void *)schur_qr_kernel<16, true>, kQrThreads, kQrSmemMax) &&
                   places_16((const void *)hess_cluster_kernel<16>, kHessThreads, kHessSmemMax)
               ? 16
               : 8;
}

cudaError_t launch_hess(int cl, int n, const double *A, int lda, double2 *T, int ldt, double *V, double *taus,
                        cudaStream_t stream)
{
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = cluster_config(cl, kHessThreads, hess_smem(n, cl), stream, at);
    if (cl == 16) return cudaLaunchKernelEx(&cfg, hess_cluster_kernel<16>, n, A, lda, T, ldt, V, taus);
    const cudaError_t e = cudaFuncSetAttribute(hess_cluster_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kHessSmemMax);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, hess_cluster_kernel<8>, n, A, lda, T, ldt, V, taus) : e;
}

cudaError_t launch_qr(int cl, int n, double2 *T, int ldt, QrState *st, SweepRec *sweeplog, double *rclog, double2 *rslog,
                      int *nlogged, cudaStream_t stream)
{
    const size_t smem = qr_smem(n, cl);
    const bool local = smem <= kQrSmemMax;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = cluster_config(cl, kQrThreads, local ? smem : 0, stream, at);
    auto go = [&](auto *kernel) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)cfg.dynamicSmemBytes);
        return e != cudaSuccess ? e
                                : cudaLaunchKernelEx(&cfg, kernel, n, T, ldt, st, kRotationBudget,
                                                     (long long)rotation_room(n), sweeplog, rclog, rslog, nlogged);
    };
    if (cl == 16) return local ? go(schur_qr_kernel<16, true>) : go(schur_qr_kernel<16, false>);
    return local ? go(schur_qr_kernel<8, true>) : go(schur_qr_kernel<8, false>);
}

}  // namespace

size_t schur_workspace_bytes(int n)
{
    if (n <= 0) return 0;
    // eleven takes, each rounded up to 256 bytes; two logs of one launch each
    const size_t nn = (size_t)n * n;
    const size_t nlog = rotation_room(n);
    return 2 * nn * sizeof(double) + 3 * (size_t)n * sizeof(double) + sizeof(double) + sizeof(int) + sizeof(QrState) +
           2 * nlog * (sizeof(SweepRec) + sizeof(double) + sizeof(double2)) + 2 * sizeof(int) + 11 * 256;
}

signtri_status schur_run(int n, const double *A, int lda, double *Q, int ldq, double *T, int ldt, Arena &ws,
                         int *bad_index, long long counts_out[2], cudaStream_t st)
{
    if (n <= 0) return SIGNTRI_OK;
    const size_t nn = (size_t)n * n;
    auto *H = static_cast<double *>(ws.take(nn * sizeof(double)));
    auto *V = static_cast<double *>(ws.take(nn * sizeof(double)));   // the reflectors, column k in rows k+1..
    auto *taus = static_cast<double *>(ws.take((size_t)n * sizeof(double)));
    auto *y = static_cast<double *>(ws.take((size_t)2 * n * sizeof(double)));
    auto *bad = static_cast<int *>(ws.take(sizeof(int)));
    auto *qs = static_cast<QrState *>(ws.take(sizeof(QrState)));
    // a launch's log has room for nlog rotations, and as many sweeps: the kernel
    // starts a multi-sweep only where all of its bulges' fit, with two bulges
    // where the window has more than they leave room for (two sweeps of a full
    // window, 2 (n - 1), always fit); launches alternate between two logs
    const size_t nlog = rotation_room(n);
    auto *sweeplog = static_cast<SweepRec *>(ws.take(2 * nlog * sizeof(SweepRec)));
    auto *rclog = static_cast<double *>(ws.take(2 * nlog * sizeof(double)));
    auto *rslog = static_cast<double2 *>(ws.take(2 * nlog * sizeof(double2)));
    auto *nlogged = static_cast<int *>(ws.take(2 * sizeof(int)));
    if (!H || !V || !taus || !y || !bad || !qs || !sweeplog || !rclog || !rslog || !nlogged)
        return SIGNTRI_ERR_NO_WORKSPACE;
    const int big = INT_MAX;
    SGT_CUDA_TRY(cudaMemcpyAsync(bad, &big, sizeof(int), cudaMemcpyHostToDevice, st));
    {
        ProfScope ps(SIGNTRI_KC_SCAN, st);
        finite_check_kernel<<<n, kThreads, 0, st>>>(n, A, lda, bad);
        SGT_LAUNCH_CHECK();
    }
    int first_bad = INT_MAX;
    SGT_CUDA_TRY(cudaMemcpyAsync(&first_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
    SGT_CUDA_TRY(cudaStreamSynchronize(st));
    if (first_bad != INT_MAX) {
        if (bad_index) *bad_index = first_bad;
        return SIGNTRI_ERR_NONFINITE;
    }
    auto *Tc = reinterpret_cast<double2 *>(T);
    auto *Qc = reinterpret_cast<double2 *>(Q);
    const int cl = cluster_size();
    if (hess_smem(n, cl) <= kHessSmemMax) {
        ProfScope ps(SIGNTRI_KC_HESSENBERG, st);
        SGT_CUDA_TRY(launch_hess(cl, n, A, lda, Tc, ldt, V, taus, st));
    } else {
        {
            ProfScope ps(SIGNTRI_KC_FILL, st);
            hess_init_kernel<<<n, kThreads, 0, st>>>(n, A, lda, H);
            SGT_LAUNCH_CHECK();
        }
        for (int k = 0; k + 2 < n; k++) {
            ProfScope ps(SIGNTRI_KC_HESSENBERG, st, true, false);
            prof_count(SIGNTRI_KC_HESSENBERG, 4);
            double *v = V + (size_t)k * n + k + 1, *tau = taus + k;
            house_kernel<<<1, 1024, 0, st>>>(n, k, H, v, tau);
            SGT_LAUNCH_CHECK();
            house_left_kernel<<<n - k - 1, kThreads, 0, st>>>(n, k, H, v, tau);
            SGT_LAUNCH_CHECK();
            house_gemv_kernel<<<(n + 31) / 32, 32 * kGemvWarps, 0, st>>>(n, k, H, v, tau, y);
            SGT_LAUNCH_CHECK();
            house_rank1_kernel<<<n - k - 1, kThreads, 0, st>>>(n, k, H, v, tau, y);
            SGT_LAUNCH_CHECK();
        }
        ProfScope ps(SIGNTRI_KC_FILL, st);
        to_complex_kernel<<<n, kThreads, 0, st>>>(n, H, Tc, ldt);
        SGT_LAUNCH_CHECK();
    }
    {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        qr_state_init_kernel<<<1, 1, 0, st>>>(n, qs);
        SGT_LAUNCH_CHECK();
    }
    // Relaunch until converged; a bound on the launches for safety (each
    // launch runs at least one sweep or one deflation while status is 0).
    // Launch m's rotations are applied on a second stream while launch m + 1
    // runs: the two touch disjoint entries (launch m + 1 stays in the
    // columns up to its window's last row i, which is where launch m ended;
    // the applies act on columns right of each logged sweep's window, which
    // ended at i or further down, and alone on Q), and launch m + 2 writes
    // launch m's log only after its apply.
    // Each launch's applies are issued after the next QR launch, so that the
    // cluster finds its SMs free (a QR CTA takes a whole SM's registers).
    CallStream ap;
    SGT_CUDA_TRY(ap.init());
    // Q's reflectors on the second stream as well, while the sweeps begin
    SGT_CUDA_TRY(cudaEventRecord(ap.ready[0], st));
    SGT_CUDA_TRY(cudaStreamWaitEvent(ap.s, ap.ready[0], 0));
    auto form_q = [&]() -> signtri_status {
        const size_t smem = n <= kQRowsMax ? (size_t)kFormWarps * n * sizeof(double) : 0;
        SGT_CUDA_TRY(cudaFuncSetAttribute(form_q_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(kFormWarps * kQRowsMax * sizeof(double))));
        ProfScope ps(SIGNTRI_KC_HESSENBERG, ap.s);
        form_q_kernel<<<(n + kFormWarps - 1) / kFormWarps, 32 * kFormWarps, smem, ap.s>>>(n, V, taus, H, Qc, ldq);
        SGT_LAUNCH_CHECK();
        return SIGNTRI_OK;
    };
    auto apply = [&](int p) -> signtri_status {
        const size_t lo = p * nlog;
        SGT_CUDA_TRY(cudaStreamWaitEvent(ap.s, ap.ready[p], 0));
        {
            ProfScope ps(SIGNTRI_KC_SCHUR, ap.s);
            apply_rotations_kernel<<<(int)((64LL * n + kThreads - 1) / kThreads), kThreads, 0, ap.s>>>(
                n, Tc, ldt, Qc, ldq, nlogged + p, sweeplog + lo, rclog + lo, rslog + lo);
            SGT_LAUNCH_CHECK();
        }
        SGT_CUDA_TRY(cudaEventRecord(ap.done[p], ap.s));
        return SIGNTRI_OK;
    };
    QrState h{};
    const long long max_launches = 4LL * n * kMaxSweepsPerEigenvalue + 16;
    for (long long it = 0;; it++) {
        if (it >= max_launches) return SIGNTRI_ERR_NO_CONVERGENCE;
        const int p = (int)(it & 1);
        const size_t lo = p * nlog;
        if (it >= 2) SGT_CUDA_TRY(cudaStreamWaitEvent(st, ap.done[p], 0));
        {
            ProfScope ps(SIGNTRI_KC_SCHUR, st);
            SGT_CUDA_TRY(launch_qr(cl, n, Tc, ldt, qs, sweeplog + lo, rclog + lo, rslog + lo, nlogged + p, st));
        }
        SGT_CUDA_TRY(cudaEventRecord(ap.ready[p], st));
        if (it == 0) {
            const signtri_status rq = form_q();
            if (rq != SIGNTRI_OK) return rq;
        } else {
            const signtri_status ra = apply(1 - p);
            if (ra != SIGNTRI_OK) return ra;
        }
        SGT_CUDA_TRY(cudaMemcpyAsync(&h, qs, sizeof(QrState), cudaMemcpyDeviceToHost, st));
        SGT_CUDA_TRY(cudaStreamSynchronize(st));
        if (h.status == 2) return SIGNTRI_ERR_NO_CONVERGENCE;
        if (h.status == 1) {
            const signtri_status ra = apply(p);
            if (ra != SIGNTRI_OK) return ra;
            break;
        }
    }
    SGT_CUDA_TRY(cudaStreamSynchronize(ap.s));
    if (counts_out) {
        counts_out[0] = h.sweeps;
        counts_out[1] = h.rotations;
    }
    {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        clear_lower_kernel<<<n, kThreads, 0, st>>>(n, Tc, ldt);
        SGT_LAUNCH_CHECK();
    }
    return SIGNTRI_OK;
}

size_t sign_general_workspace_bytes(int n)
{
    if (n <= 0) return 0;
    const size_t cnn = (size_t)n * n * sizeof(double2) + 256;
    return 3 * cnn + std::max(schur_workspace_bytes(n), complex_schur_workspace_bytes(n));
}

signtri_status sign_general_run(int n, const double *A, int lda, double *S, int lds, Arena &ws, int *d_err,
                                int *bad_index, long long counts_out[2], cudaStream_t st)
{
    if (n <= 0) return SIGNTRI_OK;
    const size_t cnn = (size_t)n * n * sizeof(double2);
    auto *Qc = static_cast<double *>(ws.take(cnn));
    auto *Tc = static_cast<double *>(ws.take(cnn));
    auto *Sc = static_cast<double *>(ws.take(cnn));
    if (!Qc || !Tc || !Sc) return SIGNTRI_ERR_NO_WORKSPACE;
    const size_t mark = ws.used;
    signtri_status rs = schur_run(n, A, lda, Qc, n, Tc, n, ws, bad_index, counts_out, st);
    if (rs != SIGNTRI_OK) return rs;
    ws.used = mark;
    rs = complex_schur_run(n, Qc, n, Tc, n, Sc, n, ws, d_err, bad_index, st);
    if (rs != SIGNTRI_OK) return rs;
    {
        ProfScope ps(SIGNTRI_KC_FILL, st);
        real_part_kernel<<<n, kThreads, 0, st>>>(n, reinterpret_cast<const double2 *>(Sc), S, lds);
        SGT_LAUNCH_CHECK();
    }
    return SIGNTRI_OK;
}

}  // namespace signtri
