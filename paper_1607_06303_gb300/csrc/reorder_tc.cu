// reorder_tc.cu -- blocked reorder by sign for Parlett-Sylvester (Section 2,
// Section 3; Section 4.1's blocking applied to the swaps).
//
// The same stable partition as the odd-even rounds of ps_fp64.cu, done by
// windows (reorder_schedule.h, schedule_window_sweeps): in each sweep every
// window W = [a, a + w) (w <= 128) that still holds a negative above a
// positive is partitioned on its own by adjacent Givens swaps.  One CTA per
// window keeps the diagonal block T[W, W] in shared memory, runs the swaps as
// odd-even rounds there (each rotation as in ps_fp64.cu: G's first column the
// eigenvector of the entry moving up, the 2 x 2 diagonal block swapped
// exactly) and logs them; four CTAs a window then form its orthogonal factor
// Z_W = G_1 G_2 ... by applying the logged rotations to the identity.  The rest of
// T and Q receive the window's rotations at once, as products:
//   T[W, right of W] <- Z_W^T T[W, right of W]
//   T[above W, W]    <- T[above W, W] Z_W
//   Q[:, W]          <- Q[:, W] Z_W
// (left and right factors commute, so all row products of a sweep come
// first, then all column products).  GB300 has no fast float64 product, so
// these run on the tensor cores as emulated-float64 products of exact 8-bit
// slices (tc_gemm.cu), written straight back into T and Q: each product
// reads the slices, snapshots taken before it, never the matrix it writes.
#include <algorithm>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "df_arith.cuh"
#include "exact_slices.cuh"
#include "internal.cuh"
#include "reorder_schedule.h"
#include "tc_gemm.cuh"

namespace signtri {

namespace {

constexpr int kWin = 128;                  // window width (two 64-row panels)
constexpr int kWinLD = kWin + 1;
constexpr int kMaxRot = (kWin / 2) * (kWin / 2);   // swaps of a window at most
constexpr int kWinThreads = 512;
// Exact slices of 8 bits, 6 of them (48 bits, the 21 pairs with s + t <= 5):
// a window product's K range is one window (128 <= 256), so every fp32 unit
// sum of products below 2^16 stays exact, and 8-bit slices take a quarter
// fewer pairs, and so a quarter fewer epilogue drains, than 7-bit ones.
constexpr int kSlices = 6;
constexpr int kBits = 8;

// The rotations of a window's rounds, read by window_factor_kernel: round
// r's are [off[r], off[r + 1]), each (c, s) as double-float pairs and its
// first position k.
struct WindowLog {
    float4 rot[kMaxRot];   // c hi, c lo, s hi, s lo
    short k[kMaxRot];
    int off[2 * kWin + 8];
    int rounds;
};

// Shared memory of a window's sort: its block as double-float planes (hi, lo)
size_t window_smem_bytes() { return 2 * (size_t)kWin * kWinLD * sizeof(float); }

// One window per CTA: stable partition of T[W, W] by swaps, the rotations
// logged for window_factor_kernel.
// GB300's float64 rate is about 1/64 of its fp32 rate, and a window is one
// SM's work, so the rotations are applied in double-float (df_arith.cuh:
// about 2^-47 per operation) to the block held as hi/lo planes; the
// diagonal stays float64 (swapped exactly) and each rotation's (c, s) is
// computed in float64 from it and the coupling, one thread per pair (one
// reciprocal square root: hypot and two divisions were ~3,000 of a round's
// ~6,000 cycles).
// The rounds form a chain: a round's rotations need the couplings that the
// round before leaves.  So two chief warps (a thread per pair of the next
// round) apply the few rotations that change those couplings, find the next
// round's pairs and form its rotations, while the other warps apply the rest
// of the round; one barrier a round.
constexpr int kChiefThreads = 64;

__global__ void __launch_bounds__(kWinThreads)
window_sort_kernel(double *__restrict__ Tr, int ldt, const int2 *__restrict__ wins, WindowLog *__restrict__ logs)
{
    extern __shared__ float wsm[];
    float *Bh = wsm, *Bl = Bh + kWin * kWinLD;               // Bh/Bl[i + j * kWinLD]: T[a + i, a + j], i < j
    // of the round at work and the next one, by the round's parity: the
    // diagonal, each pair's rotation and first position, the pair (its index
    // in the round) holding a position or -1, the pairs
    __shared__ double dg[2][kWin + 2];
    __shared__ float4 rot[2][kWin / 2];
    __shared__ short first[2][kWin / 2], pm[2][kWin + 2];
    __shared__ int wc[2][2], cnt[2];
    const int a = wins[blockIdx.x].x, w = wins[blockIdx.x].y;
    WindowLog *log = logs + blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int idx = tid; idx < kWin * kWin; idx += kWinThreads) {
        const int i = idx % kWin, j = idx / kWin;
        const double v = (i < j && j < w) ? SGT_AT(Tr, ldt, a + i, a + j) : 0.0;
        split_df(v, Bh[i + j * kWinLD], Bl[i + j * kWinLD]);
        if (i == j) dg[1][i] = (j < w) ? SGT_AT(Tr, ldt, a + i, a + i) : 1.0;
    }
    if (tid < 2) {
        dg[tid][kWin] = dg[tid][kWin + 1] = 1.0;
        cnt[tid] = 0;
    }
    for (int i = tid; i < kWin + 2; i += kWinThreads) pm[0][i] = pm[1][i] = -1;
    __syncthreads();
    int r = -1, base = 0;   // round -1 has no pairs; the chiefs find round 0's
    for (;; r++) {
        const int cur = r & 1, nxt = cur ^ 1;
        const int P = cnt[cur];
        if (tid < kChiefThreads) {
            // the next round's pair slot (k, k + 1); of this round, the pair A
            // = (k - 1, k) and the pair C = (k + 1, k + 2)
            const int k = 2 * tid + nxt;
            const int eA = k > 0 ? pm[cur][k] : -1, eC = k + 1 < kWin ? pm[cur][k + 1] : -1;
            float bh = 0.f, bl = 0.f;   // the coupling (k, k + 1) after this round
            if (k + 1 < w) {
                const int at = k + (k + 1) * kWinLD;
                bh = Bh[at];
                bl = Bl[at];
                float uh = 0.f, ul = 0.f;   // row k - 1 of column k + 1
                if (eA >= 0) {
                    const float4 g = rot[cur][eA];
                    const float ph = Bh[at - 1], pl = Bl[at - 1];
                    df_rot(g.x, g.y, ph, pl, g.z, g.w, bh, bl, uh, ul);        // c u + s v
                    df_rot(-g.z, -g.w, ph, pl, g.x, g.y, bh, bl, bh, bl);      // -s u + c v
                }
                if (eC >= 0) {
                    const float4 g2 = rot[cur][eC];
                    const int at2 = at + kWinLD;
                    float qh = Bh[at2], ql = Bl[at2];   // row k of column k + 2
                    if (eA >= 0) {
                        const float4 g = rot[cur][eA];
                        const float ph = Bh[at2 - 1], pl = Bl[at2 - 1];
                        float th, tl;
                        df_rot(g.x, g.y, ph, pl, g.z, g.w, qh, ql, th, tl);
                        df_rot(-g.z, -g.w, ph, pl, g.x, g.y, qh, ql, qh, ql);
                        float xh, xl;
                        df_rot(g2.x, g2.y, uh, ul, g2.z, g2.w, th, tl, xh, xl);            // u c + v s
                        df_rot(-g2.z, -g2.w, uh, ul, g2.x, g2.y, th, tl, Bh[at2 - 1], Bl[at2 - 1]);   // -u s + v c
                        uh = xh;
                        ul = xl;
                    }
                    const float vh = bh, vl = bl;
                    df_rot(g2.x, g2.y, vh, vl, g2.z, g2.w, qh, ql, bh, bl);
                    df_rot(-g2.z, -g2.w, vh, vl, g2.x, g2.y, qh, ql, Bh[at2], Bl[at2]);
                }
                if (eA >= 0) {
                    Bh[at - 1] = uh;
                    Bl[at - 1] = ul;
                }
                if (eA >= 0 || eC >= 0) {
                    Bh[at] = bh;
                    Bl[at] = bl;
                }
            }
            // the diagonal after the round's swaps (exact)
            const double d0 = eA >= 0 ? dg[cur][k - 1] : dg[cur][k];
            const double d1 = eC >= 0 ? dg[cur][k + 2] : dg[cur][k + 1];
            dg[nxt][k] = d0;
            dg[nxt][k + 1] = d1;
            if (nxt == 1 && tid == 0) {
                dg[1][0] = eA >= 0 ? dg[0][1] : dg[0][0];
                pm[1][0] = -1;
            }
            const bool on = k + 1 < w && !(d0 > 0.0) && d1 > 0.0;
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            if (lane == 0) wc[nxt][warp] = __popc(bal);
            asm volatile("bar.sync 1, %0;" ::"n"(kChiefThreads) : "memory");
            const int pos = (warp ? wc[nxt][0] : 0) + __popc(bal & ((1u << lane) - 1u));
            const int total = wc[nxt][0] + wc[nxt][1];
            pm[nxt][k] = pm[nxt][k + 1] = on ? (short)pos : (short)-1;
            if (tid == 0) {
                cnt[nxt] = total;
                log->off[r + 1] = base;
            }
            if (on) {
                // G's first column is the eigenvector of the entry moving up:
                // (bb, d) / |(bb, d)|
                const double bb = df_to_double(bh, bl), d = d1 - d0;
                const int em = max(exp_field(bb), exp_field(d));
                double c, s;
                if (em > -500 && em < 500) {
                    const double rh = rsqrt_normal(fma(bb, bb, d * d));
                    c = bb * rh;
                    s = d * rh;
                } else {
                    const double h = hypot(bb, d);
                    c = bb / h;
                    s = d / h;
                }
                float4 g;
                split_df(c, g.x, g.y);
                split_df(s, g.z, g.w);
                rot[nxt][pos] = g;
                first[nxt][pos] = (short)k;
                log->rot[base + pos] = g;
                log->k[base + pos] = (short)k;
            }
            base += total;
        } else {
            // the rest of round r, four warps' items a pair e = (k, k + 1),
            // one per position x: x right of the pair -- G^T on rows k, k+1 of
            // column x, and, where x is in a pair itself, that pair's G on
            // columns x, x+1 (the two columns in neighbouring lanes); x left
            // of the pair and in none -- G on columns k, k+1 of row x.  What
            // touches the couplings next to the pair is the chiefs'.
            for (int task = warp - kChiefThreads / 32; task < 4 * P; task += (kWinThreads - kChiefThreads) / 32) {
                const int k = first[cur][task >> 2];
                const int x = (((task & 3) << 5) + lane + cur) & (kWin - 1);
                const int q = pm[cur][x];
                const bool right = x < w && (q < 0 ? x >= k + 3 : first[cur][q] >= k + 4);
                const bool left = q < 0 && x <= k - 2;
                const float4 g = rot[cur][task >> 2];
                const int i0 = right ? k + x * kWinLD : x + k * kWinLD, i1 = i0 + (right ? 1 : kWinLD);
                float uh = 0.f, ul = 0.f, vh = 0.f, vl = 0.f, sh, sl, th, tl;
                if (right || left) {
                    uh = Bh[i0];
                    ul = Bl[i0];
                    vh = Bh[i1];
                    vl = Bl[i1];
                }
                df_rot(g.x, g.y, uh, ul, g.z, g.w, vh, vl, sh, sl);        // c u + s v
                df_rot(-g.z, -g.w, uh, ul, g.x, g.y, vh, vl, th, tl);      // -s u + c v
                const bool both = right && q >= 0;
                if (__any_sync(0xffffffffu, both)) {
                    const float osh = __shfl_xor_sync(0xffffffffu, sh, 1), osl = __shfl_xor_sync(0xffffffffu, sl, 1);
                    const float oth = __shfl_xor_sync(0xffffffffu, th, 1), otl = __shfl_xor_sync(0xffffffffu, tl, 1);
                    if (both) {
                        // first column u c + v s, second -u s + v c
                        float4 g2 = rot[cur][q];
                        if (lane & 1) {
                            g2.z = -g2.z;
                            g2.w = -g2.w;
                        }
                        df_rot(g2.x, g2.y, sh, sl, g2.z, g2.w, osh, osl, sh, sl);
                        df_rot(g2.x, g2.y, th, tl, g2.z, g2.w, oth, otl, th, tl);
                    }
                }
                if (right || left) {
                    Bh[i0] = sh;
                    Bl[i0] = sl;
                    Bh[i1] = th;
                    Bl[i1] = tl;
                }
            }
        }
        __syncthreads();
        // two rounds in a row without a swap end the sort (at most w + 1 rounds)
        if ((r >= 0 && P == 0 && cnt[nxt] == 0) || r >= 2 * kWin) break;
    }
    // round r + 1 is the last one logged, and empty
    if (tid == 0) {
        log->off[r + 2] = base;
        log->rounds = r + 2;
    }
    const double *dl = dg[(r & 1) ^ 1];
    for (int idx = tid; idx < kWin * kWin; idx += kWinThreads) {
        const int i = idx % kWin, j = idx / kWin;
        if (j < w && i < j) SGT_AT(Tr, ldt, a + i, a + j) = df_to_double(Bh[i + j * kWinLD], Bl[i + j * kWinLD]);
        else if (j < w && i == j) SGT_AT(Tr, ldt, a + i, a + i) = dl[i];
    }
}

// The window's orthogonal factor Z_W = I G_1 G_2 ... as the exact column
// slices the products read -- ZC[s][a + j][a + i] = slice s of Z_W[i][j]
// under the column's power-of-two scale sZ[a + j] (rp rows of pitch kp per
// slice).  Entries of ZC outside the windows' blocks are never read (the
// products' K ranges stay inside the window).  A row of Z takes every
// rotation by itself, so a cluster of kFactorCtas CTAs takes 32 rows each (a
// sweep has n / 128 windows, far fewer than SMs): a warp per pair of a round,
// a row per lane; the columns' maxima meet in shared memory.
constexpr int kFactorCtas = kWin / 32;
constexpr int kFactorLD = 33;

constexpr size_t kFactorAlone = 200 * 1024;   // where there are SMs enough, a CTA to each
size_t factor_smem_bytes()
{
    return (size_t)kMaxRot * (sizeof(float4) + sizeof(short)) + 2 * (size_t)kWin * kFactorLD * sizeof(float);
}

__global__ void __cluster_dims__(kFactorCtas, 1, 1) __launch_bounds__(kWinThreads)
window_factor_kernel(const int2 *__restrict__ wins, const WindowLog *__restrict__ logs, __nv_bfloat16 *__restrict__ ZC,
                     float *__restrict__ sZ, int rp, int kp)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ float4 fsm[];
    float4 *rot = fsm;
    float *Zh = reinterpret_cast<float *>(rot + kMaxRot), *Zl = Zh + kWin * kFactorLD;   // [i + j * kFactorLD]
    short *first = reinterpret_cast<short *>(Zl + kWin * kFactorLD);
    __shared__ int off[2 * kWin + 8], cexp[kWin];
    __shared__ float cmax[kWin];
    const int win = blockIdx.x / kFactorCtas, a = wins[win].x, w = wins[win].y;
    const int part = (int)cl.block_rank(), row0 = 32 * part;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const WindowLog *log = logs + win;
    const int rounds = log->rounds, nlog = log->off[rounds];
    for (int r = tid; r <= rounds; r += kWinThreads) off[r] = log->off[r];
    for (int e = tid; e < nlog; e += kWinThreads) {
        rot[e] = log->rot[e];
        first[e] = log->k[e];
    }
    for (int idx = tid; idx < 32 * kWin; idx += kWinThreads) {
        const int i = idx & 31, j = idx >> 5;
        Zh[i + j * kFactorLD] = (row0 + i == j) ? 1.f : 0.f;
        Zl[i + j * kFactorLD] = 0.f;
    }
    __syncthreads();
    // round by round (a round's rotations act on disjoint columns)
    for (int r = 0; r < rounds; r++) {
        for (int e = off[r] + warp; e < off[r + 1]; e += kWinThreads / 32) {
            const float4 g = rot[e];
            const int i0 = lane + first[e] * kFactorLD, i1 = i0 + kFactorLD;
            const float uh = Zh[i0], ul = Zl[i0], vh = Zh[i1], vl = Zl[i1];
            df_rot(g.x, g.y, uh, ul, g.z, g.w, vh, vl, Zh[i0], Zl[i0]);
            df_rot(-g.z, -g.w, uh, ul, g.x, g.y, vh, vl, Zh[i1], Zl[i1]);
        }
        __syncthreads();
    }
    // per column of Z: the power-of-two scale above its largest entry (an
    // orthogonal column: between 1 / sqrt(w) and 1; |hi + lo| < 2^e whenever
    // |hi| < 2^e, lo being at most half an ulp of hi), then its exact slices
    for (int j = warp; j < w; j += kWinThreads / 32) {
        float mx = row0 + lane < w ? fabsf(Zh[lane + j * kFactorLD]) : 0.f;
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) cmax[j] = mx;
    }
    cl.sync();
    for (int j = tid; j < w; j += kWinThreads) {
        float mx = 0.f;
        for (int q = 0; q < kFactorCtas; q++) mx = fmaxf(mx, cl.map_shared_rank(cmax, q)[j]);
        int e = 0;
        frexpf(mx, &e);
        cexp[j] = e;
        if (part == 0) sZ[a + j] = ldexpf(1.f, e);
    }
    cl.sync();   // also: no CTA leaves while another reads its maxima
    for (int idx = tid; idx < 32 * w; idx += kWinThreads) {
        const int i = idx & 31, j = idx >> 5;
        if (row0 + i >= w) continue;
        float q[kSlices];
        exact_slices<kSlices>(df_to_double(Zh[i + j * kFactorLD], Zl[i + j * kFactorLD]), cexp[j], kSlices, kBits, q);
#pragma unroll
        for (int sl = 0; sl < kSlices; sl++)
            ZC[((size_t)sl * rp + a + j) * kp + a + row0 + i] = __float2bfloat16_rn(q[sl]);
    }
}

// The slices the products of one sweep read, for the active 64-blocks of K
// only (kbl: the sweep's window blocks, ascending).  Three kinds of lines:
//   kColsT: column j of T, K = rows kk < j (row products: tiles kb < jb);
//   kRowsT: row r of T, K = columns kk > r (column products: tiles rb < kb,
//           plus the zero rows [np, np + 64));
//   kRowsQ: row r of Q, K = every active column.
// Every entry a tile holds is then strictly upper for T.  The scale of a line
// is the power of two above its largest entry in the tiles it reads (1 for
// none); lines outside every tile are not outputs of the sweep's products.
constexpr int kColsT = 0, kRowsT = 1, kRowsQ = 2;

template <int MODE>
__device__ __forceinline__ bool tile_used(int kb, int lb, int zero_lb)
{
    if (MODE == kColsT) return lb > kb;
    if (MODE == kRowsT) return lb < kb || lb == zero_lb;
    return true;
}

template <int MODE>
__global__ void __launch_bounds__(256)
masked_absmax_kernel(int n, const double *__restrict__ M, int ldm, const int *__restrict__ kbl, int zero_lb,
                     unsigned long long *__restrict__ mx)
{
    const int kb = kbl[blockIdx.x], lb = blockIdx.y;
    if (!tile_used<MODE>(kb, lb, zero_lb) || lb == zero_lb) return;
    const int k0 = kb * 64, l0 = lb * 64;
    if (MODE == kColsT) {
        // a warp per column: two rows per lane, reduced by shuffles
        const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
        for (int c = wp; c < 64; c += 8) {
            const int j = l0 + c;
            unsigned long long v = 0;   // maxima on the bits of |x| (integer pipes)
            if (j < n) {
                if (k0 + lane < n) v = abs_bits(SGT_AT(M, ldm, k0 + lane, j));
                if (k0 + lane + 32 < n) v = max(v, abs_bits(SGT_AT(M, ldm, k0 + lane + 32, j)));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == 0 && v > 0) atomicMax(&mx[j], v);
        }
    } else {
        // a thread per row and quarter of the columns, then the quarters reduced
        __shared__ unsigned long long part[4][64];
        const int t = threadIdx.x & 63, q = threadIdx.x >> 6, r = l0 + t;
        unsigned long long v = 0;
        if (r < n)
            for (int c = q * 16; c < q * 16 + 16; c++)
                if (k0 + c < n) v = max(v, abs_bits(SGT_AT(M, ldm, r, k0 + c)));
        part[q][t] = v;
        __syncthreads();
        if (threadIdx.x < 64) {
            v = max(max(part[0][t], part[1][t]), max(part[2][t], part[3][t]));
            if (v > 0) atomicMax(&mx[r], v);
        }
    }
}

__device__ __forceinline__ int line_exp(const unsigned long long *mx, int line, int n)
{
    if (line >= n) return 0;
    const unsigned long long m = mx[line];
    return m ? max(frexp_exp_of_bits(m), -120) : 0;
}

// Exact slices (kSlices of kBits bits) of the used tiles, K-contiguous lines of
// pitch kp, rp lines per slice; the line scales go to `scale` (written once
// per line, by the CTA of the first (kColsT, kRowsQ) or last (kRowsT) block).
template <int MODE>
__global__ void __launch_bounds__(256)
masked_slices_kernel(int n, const double *__restrict__ M, int ldm, const int *__restrict__ kbl, int zero_lb,
                     const unsigned long long *__restrict__ mx, __nv_bfloat16 *__restrict__ out, float *__restrict__ scale,
                     int rp, int kp)
{
    const int kb = kbl[blockIdx.x], lb = blockIdx.y;
    if (!tile_used<MODE>(kb, lb, zero_lb)) return;
    const int k0 = kb * 64, l0 = lb * 64;
    const bool zero = lb == zero_lb;
    const bool writes_scale = !zero && (int)blockIdx.x == (MODE == kRowsT ? (int)gridDim.x - 1 : 0);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    if (MODE == kColsT) {
        // column j's K run is contiguous in M: lane reads rows k0 + 2 lane, + 1
        for (int c = wp; c < 64; c += 8) {
            const int j = l0 + c, kk = k0 + 2 * lane;
            double v0 = 0.0, v1 = 0.0;
            if (j < n) {
                if (kk < n) v0 = SGT_AT(M, ldm, kk, j);
                if (kk + 1 < n) v1 = SGT_AT(M, ldm, kk + 1, j);
            }
            const int e = line_exp(mx, j, n);
            float q0[kSlices], q1[kSlices];
            exact_slices<kSlices>(v0, e, kSlices, kBits, q0);
            exact_slices<kSlices>(v1, e, kSlices, kBits, q1);
#pragma unroll
            for (int sl = 0; sl < kSlices; sl++)
                *reinterpret_cast<__nv_bfloat162 *>(&out[((size_t)sl * rp + j) * kp + kk]) =
                    __floats2bfloat162_rn(q0[sl], q1[sl]);
            if (writes_scale && lane == 0 && j < n) scale[j] = ldexpf(1.f, e);
        }
    } else {
        // rows: transposed through shared memory (tile[kk][r])
        __shared__ double tile[64][65];
        for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
            const int t = idx & 63, c = idx >> 6, r = l0 + t, kk = k0 + c;
            tile[c][t] = (!zero && r < n && kk < n) ? SGT_AT(M, ldm, r, kk) : 0.0;
        }
        __syncthreads();
        for (int t = wp; t < 64; t += 8) {
            const int r = l0 + t, kk = k0 + 2 * lane;
            const int e = zero ? 0 : line_exp(mx, r, n);
            float q0[kSlices], q1[kSlices];
            exact_slices<kSlices>(tile[2 * lane][t], e, kSlices, kBits, q0);
            exact_slices<kSlices>(tile[2 * lane + 1][t], e, kSlices, kBits, q1);
#pragma unroll
            for (int sl = 0; sl < kSlices; sl++)
                *reinterpret_cast<__nv_bfloat162 *>(&out[((size_t)sl * rp + r) * kp + kk]) =
                    __floats2bfloat162_rn(q0[sl], q1[sl]);
            if (writes_scale && lane == 0 && r < n) scale[r] = ldexpf(1.f, e);
        }
    }
}

}  // namespace

size_t reorder_blocked_workspace_bytes(int n)
{
    if (n <= 0) return 0;
    const size_t rp = (size_t)pad64(n) + 64, kp = (size_t)pad64(n);
    size_t b = 4 * (kSlices * rp * kp * 2 + 256);                    // slices: Z, T (two forms), Q
    b += 4 * (rp * sizeof(float) + 256) + 3 * rp * 8 + 256;           // scales, line maxima
    b += sizeof(TcPairs) + 256;
    // the window and job lists of every sweep go to memory of their own
    return b;
}

signtri_status reorder_blocked_run(int n, const double *T, int ldt, double *Tr, int ldtr, double *Q, int ldq,
                                   long long *swaps_out, Arena &ws, int *d_err, cudaStream_t st)
{
    if (n <= 0) return SIGNTRI_OK;
    const int np = pad64(n), rp = np + 64, kp = np, zero = np;   // rows [np, np + 64) of every slice array are zero
    auto slices = [&]() { return static_cast<__nv_bfloat16 *>(ws.take((size_t)kSlices * rp * kp * 2)); };
    __nv_bfloat16 *ZC = slices(), *TC = slices(), *TR = slices(), *QR = slices();
    float *sZ = static_cast<float *>(ws.take(rp * sizeof(float)));
    float *sTc = static_cast<float *>(ws.take(rp * sizeof(float)));
    float *sTr = static_cast<float *>(ws.take(rp * sizeof(float)));
    float *sQ = static_cast<float *>(ws.take(rp * sizeof(float)));
    auto *mx = static_cast<unsigned long long *>(ws.take(3 * (size_t)rp * sizeof(unsigned long long)));
    auto *d_pairs = static_cast<TcPairs *>(ws.take(sizeof(TcPairs)));
    if (!ZC || !TC || !TR || !QR || !sZ || !sTc || !sTr || !sQ || !mx || !d_pairs) return SIGNTRI_ERR_NO_WORKSPACE;
    signtri_status rs = copy_upper_identity(n, T, ldt, Tr, ldtr, Q, ldq, st);   // T~ = upper part of T, Q = I
    if (rs != SIGNTRI_OK) return rs;
    std::vector<double> diag(n);
    SGT_CUDA_TRY(cudaMemcpy2DAsync(diag.data(), sizeof(double), T, ((size_t)ldt + 1) * sizeof(double), sizeof(double),
                                   n, cudaMemcpyDeviceToHost, st));
    SGT_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<std::vector<int2>> sweeps;
    long long swaps = 0;
    schedule_window_sweeps(diag, kWin, sweeps, swaps);
    if (swaps_out) *swaps_out = swaps;
    if (swaps == 0) return SIGNTRI_OK;
    // every sweep's windows and the jobs of its three products, built here
    // and uploaded once
    auto job = [](int rt, int rb, int cl, int cr, int kb0, int kb1) {
        TcJob j;
        j.rt = rt; j.rb = rb; j.cl = cl; j.cr = cr; j.kb0 = kb0; j.kb1 = kb1; j.slot = 0; j.pad = 0;
        return j;
    };
    std::vector<int2> wins_all;
    std::vector<TcJob> jobs_all;
    std::vector<int> kbl_all;   // each sweep's window 64-blocks, ascending
    struct Sweep { int w0, nw; int j[4]; double kb[3]; int k0, nk; };
    std::vector<Sweep> plan;
    for (const std::vector<int2> &sw : sweeps) {
        if (sw.empty()) continue;
        Sweep p{(int)wins_all.size(), (int)sw.size(), {0, 0, 0, 0}, {0, 0, 0}, (int)kbl_all.size(), 0};
        wins_all.insert(wins_all.end(), sw.begin(), sw.end());
        for (const int2 &win : sw)
            for (int kb = win.x / 64; kb <= (win.x + win.y - 1) / 64; kb++) kbl_all.push_back(kb);
        p.nk = (int)kbl_all.size() - p.k0;
        for (int phase = 0; phase < 3; phase++) {
            p.j[phase] = (int)jobs_all.size();
            for (const int2 &win : sw) {
                const int a = win.x, e = win.x + win.y, kb0 = a / 64, kb1 = (e + 63) / 64;
                const int second = win.y > 64 ? a + 64 : zero;
                if (phase == 0) {
                    // rows: T[W, c..c+128) <- Z^T T[W, c..c+128) for the columns right of W
                    for (int c = e; c < n; c += 128) jobs_all.push_back(job(a, second, c, c + 64 < n ? c + 64 : zero, kb0, kb1));
                } else {
                    // columns: T[r..r+128, W] <- T[r..r+128, W] Z above W; Q[r..r+128, W] <- Q[..] Z for all rows
                    const int rows = phase == 1 ? a : n;
                    for (int r = 0; r < rows; r += 128)
                        jobs_all.push_back(job(r, r + 64 < rows ? r + 64 : zero, a, second, kb0, kb1));
                }
            }
            for (int q = p.j[phase]; q < (int)jobs_all.size(); q++) p.kb[phase] += 4.0 * (jobs_all[q].kb1 - jobs_all[q].kb0);
        }
        p.j[3] = (int)jobs_all.size();
        plan.push_back(p);
    }
    int2 *d_wins = nullptr;
    TcJob *d_jobs = nullptr;
    int *d_kbl = nullptr;
    if (cudaMalloc(&d_wins, std::max<size_t>(wins_all.size(), 1) * sizeof(int2)) != cudaSuccess ||
        cudaMalloc(&d_jobs, std::max<size_t>(jobs_all.size(), 1) * sizeof(TcJob)) != cudaSuccess ||
        cudaMalloc(&d_kbl, std::max<size_t>(kbl_all.size(), 1) * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(d_wins);
        cudaFree(d_jobs);
        return SIGNTRI_ERR_NO_WORKSPACE;
    }
    CallStream side;
    auto body = [&]() -> signtri_status {
        SGT_CUDA_TRY(side.init());
        SGT_CUDA_TRY(cudaMemcpyAsync(d_wins, wins_all.data(), wins_all.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
        SGT_CUDA_TRY(cudaMemcpyAsync(d_jobs, jobs_all.data(), jobs_all.size() * sizeof(TcJob), cudaMemcpyHostToDevice, st));
        SGT_CUDA_TRY(cudaMemcpyAsync(d_kbl, kbl_all.data(), kbl_all.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        const TcPairs pairs = ozaki_pairs_impl(kSlices, kBits);
        SGT_CUDA_TRY(cudaMemcpyAsync(d_pairs, &pairs, sizeof(TcPairs), cudaMemcpyHostToDevice, st));
        // the zero rows past the matrix, read by the half-empty jobs
        SGT_CUDA_TRY(cudaMemsetAsync(ZC, 0, (size_t)kSlices * rp * kp * 2, st));
        const size_t smem = window_smem_bytes();
        SGT_CUDA_TRY(cudaFuncSetAttribute(window_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        SGT_CUDA_TRY(cudaFuncSetAttribute(window_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kFactorAlone));
        // the windows' rotation logs lie in T's column slices, which each
        // sweep writes after its factors are formed (rp x kp >= 128 x 64, and
        // a sweep has at most n / 128 + 2 windows)
        size_t nw_max = 0;
        for (const Sweep &p : plan) nw_max = std::max(nw_max, (size_t)p.nw);
        if (nw_max * sizeof(WindowLog) > (size_t)kSlices * rp * kp * 2) return SIGNTRI_ERR_NO_WORKSPACE;
        const TcSource srcZ{ZC, kSlices, rp, kp, kp, sZ}, srcTc{TC, kSlices, rp, kp, kp, sTc};
        const TcSource srcTr{TR, kSlices, rp, kp, kp, sTr}, srcQ{QR, kSlices, rp, kp, kp, sQ};
        const TcQuadOut toT{{Tr, Tr, Tr, Tr}, ldtr, n, n, 0}, toQ{{Q, Q, Q, Q}, ldq, n, n, 0};
        const double fl = tc_flops(pairs.n, 1, 1);
        auto product = [&](const Sweep &p, int phase, const TcSource &top, const TcSource &left,
                           const TcQuadOut &out, cudaStream_t st) -> signtri_status {
            const int cnt = p.j[phase + 1] - p.j[phase];
            if (cnt == 0) return SIGNTRI_OK;
            return tc_blocksums(top, top, left, left, d_jobs + p.j[phase], cnt, pairs, d_pairs, kExactChunkKb8, nullptr,
                                out, d_err, SIGNTRI_KC_GIVENS, st, fl * p.kb[phase]);
        };
        const int zero_lb = np / 64;
        unsigned long long *mxTc = mx, *mxTr = mx + rp, *mxQ = mx + 2 * (size_t)rp;
        // scales and slices of the active K blocks of one kind of line
        auto convert = [&](int mode, const Sweep &p, const double *M, int ldm, unsigned long long *m,
                           __nv_bfloat16 *out, float *scale, cudaStream_t st) -> signtri_status {
            ProfScope ps(SIGNTRI_KC_CONVERT, st);
            const dim3 grid(p.nk, rp / 64);
            const int *kbl = d_kbl + p.k0;
            if (mode == kColsT) {
                masked_absmax_kernel<kColsT><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m);
                masked_slices_kernel<kColsT><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m, out, scale, rp, kp);
            } else if (mode == kRowsT) {
                masked_absmax_kernel<kRowsT><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m);
                masked_slices_kernel<kRowsT><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m, out, scale, rp, kp);
            } else {
                masked_absmax_kernel<kRowsQ><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m);
                masked_slices_kernel<kRowsQ><<<grid, 256, 0, st>>>(n, M, ldm, kbl, zero_lb, m, out, scale, rp, kp);
            }
            SGT_LAUNCH_CHECK();
            return SIGNTRI_OK;
        };
        signtri_status r2;
        // A sweep's sort needs T alone, and few SMs: so Q's slices and product
        // run on a second stream beside the next sweep's sort; its factors,
        // which replace Z, wait for them.  (At n = 3001 and 42 sweeps: 28.4 ms
        // in one stream, 25.2 with Q's part beside T's products, 22.6 so.)
        auto q_part = [&](const Sweep &p) -> signtri_status {
            SGT_CUDA_TRY(cudaStreamWaitEvent(side.s, side.ready[0], 0));
            SGT_CUDA_TRY(cudaMemsetAsync(mxQ, 0, (size_t)rp * sizeof(unsigned long long), side.s));
            signtri_status r3 = convert(kRowsQ, p, Q, ldq, mxQ, QR, sQ, side.s);
            if (r3 == SIGNTRI_OK) r3 = product(p, 2, srcQ, srcZ, toQ, side.s);
            if (r3 != SIGNTRI_OK) return r3;
            SGT_CUDA_TRY(cudaEventRecord(side.done[0], side.s));
            SGT_CUDA_TRY(cudaStreamWaitEvent(st, side.done[0], 0));
            return SIGNTRI_OK;
        };
        auto *logs = reinterpret_cast<WindowLog *>(TC);   // where T's column slices follow
        const Sweep *before = nullptr;
        for (const Sweep &p : plan) {
            SGT_CUDA_TRY(cudaMemsetAsync(mx, 0, 2 * (size_t)rp * sizeof(unsigned long long), st));
            {
                ProfScope ps(SIGNTRI_KC_GIVENS, st);
                window_sort_kernel<<<p.nw, kWinThreads, smem, st>>>(Tr, ldtr, d_wins + p.w0, logs);
                SGT_LAUNCH_CHECK();
            }
            if (before && (r2 = q_part(*before)) != SIGNTRI_OK) return r2;
            {
                ProfScope ps(SIGNTRI_KC_GIVENS, st);
                window_factor_kernel<<<p.nw * kFactorCtas, kWinThreads,
                                       p.nw * kFactorCtas <= 152 ? kFactorAlone : factor_smem_bytes(), st>>>(
                    d_wins + p.w0, logs, ZC, sZ, rp, kp);
                SGT_LAUNCH_CHECK();
            }
            if ((r2 = convert(kColsT, p, Tr, ldtr, mxTc, TC, sTc, st)) != SIGNTRI_OK) return r2;
            if ((r2 = product(p, 0, srcZ, srcTc, toT, st)) != SIGNTRI_OK) return r2;     // rows of T
            if ((r2 = convert(kRowsT, p, Tr, ldtr, mxTr, TR, sTr, st)) != SIGNTRI_OK) return r2;
            if ((r2 = product(p, 1, srcTr, srcZ, toT, st)) != SIGNTRI_OK) return r2;     // columns of T
            SGT_CUDA_TRY(cudaEventRecord(side.ready[0], st));
            before = &p;
        }
        if (before && (r2 = q_part(*before)) != SIGNTRI_OK) return r2;   // columns of Q
        // the host lists stay alive until the copies above are done; so do the
        // device lists until the last product
        SGT_CUDA_TRY(cudaStreamSynchronize(st));
        return SIGNTRI_OK;
    };
    rs = body();
    if (rs != SIGNTRI_OK) {
        cudaStreamSynchronize(st);
        if (side.s) cudaStreamSynchronize(side.s);
    }
    cudaFree(d_wins);
    cudaFree(d_jobs);
    cudaFree(d_kbl);
    return rs;
}

}  // namespace signtri
