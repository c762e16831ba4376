// mixed.cu -- Parlett-Higham with tensor-core block sums and float64
// refinement of both defining equations.
//
// 1. Low-precision solve.  The block anti-diagonal schedule of the float64
//    path (Algorithms 4-6 reordered, blocks of 64), with the block sums
//      X_IJ = sum_K U_IK T_KJ - T_IK U_KJ,   Y_IJ = sum_K U_IK U_KJ
//    formed on the tensor cores (tc_gemm.cu) from 16-bit splits of U and T:
//    one bf16 term (BF16 variant), a three-term bf16 split hi + mid + lo with
//    the six products of s + t <= 2 (about fp32 accuracy, the "FP32"
//    variant), or a two-term fp16 split hi + lo with the three products of
//    s + t <= 1 (about 2^-21; T, U and the correction scaled by powers of two
//    into fp16's range, the FP16 variant); in-block recurrences (Algorithm 6,
//    1x1 case) in fp32, a 64-row tile solved by 4 x 4 micro-blocks.
// 2. Refinement.  With U = U0 + E and E strictly upper triangular, UT = TU
//    and U^2 = I become, entry by entry (i < j):
//      signs differ: (t_ii - t_jj) e_ij = -Rc_ij + sum_{i<k<j} (e_ik t_kj - t_ik e_kj)
//      signs equal:  (u_ii + u_jj) e_ij = -Rs_ij - sum_{i<k<j} (u0_ik e_kj + e_ik u0_kj)
//    (the second dropping e_ik e_kj), with the residuals Rc = T U0 - U0 T and
//    Rs = U0^2 - I.  These are the Parlett-Higham recurrences with U replaced
//    by E, so E is computed by the same schedule (block sums X^E = E T - T E,
//    Y^E = U0 E + E U0 on the tensor cores, recurrences in fp32).  Newton's
//    iteration X <- X(3I - X^2)/2 alone would only drive U^2 = I and cannot
//    correct the entries fixed by UT = TU, hence both equations.
//    Entry (i, j) uses Rc_ij when the signs differ and Rs_ij when they agree
//    (the same choice as Algorithm 3), so the residual that drives the first
//    correction forms only that one (Section 5.3's economy applied to the
//    residual products); acceptance always rests on both residuals over all
//    entries (an ill-conditioned problem can meet its own recurrences long
//    before the other equation).  The residuals
//    come from exact 7-bit integer slices of the strictly upper parts of T and
//    U0 (seven slices, 28 pairs over K-chunks of 1024: emulated float64
//    products, about 2^-45 relative to |T||U| -- the slices are scaled per
//    row and column of the strictly upper parts, whose entries are of similar
//    magnitude, the diagonals being taken apart; 8-bit slices would need 21
//    pairs but K-chunks of 256, and the fourfold epilogue work costs more than
//    the pairs save) plus the
//    diagonal terms in float64:
//      Rc_ij = (N_T N_U - N_U N_T)_ij + t_ii u_ij + t_ij u_jj - u_ii t_ij - u_ij t_jj
//      Rs_ij = (N_U N_U)_ij + u_ii u_ij + u_ij u_jj.
//    For the products the indices are gathered per superblock of kSuper
//    consecutive indices, positives first, each sign class padded to whole
//    64-blocks: every 64 x 64 output block then has one sign class in its rows
//    and one in its columns, and a tensor-core job computes four such blocks
//    that all need the same product (Y = N_U N_U, or one of the two parts of
//    X).  Block upper triangular structure survives at superblock level, so a
//    job's K range lies within its superblocks, trimmed to where its rows and
//    columns can have nonzero terms (the rest are structural zeros).
//    The full residuals use the original layout and four-quadrant jobs
//    [N_T I.; N_U I.] x [N_U .J | N_T .J].  Stop when ||Rc||_F / (||T||_F
//    ||U||_F) and ||Rs||_F / ||U||_F^2 are both below the tolerance; fall back
//    to the float64 path when a step does not reduce the larger of the two by
//    a factor 10, or after the step limit.
// 3. Memory traffic.  The sweeps stream each tile's operand panels once per
//    anti-diagonal (bf16 slices stored as contiguous 64 x 64 tiles).  Launches
//    that read the same panels run side by side on side streams with matched
//    CTA splits, so the second read comes from L2: the correction's X^E and
//    Y^E (shared E panels), and the initial sweep's look-ahead pairs, where an
//    anti-diagonal's tiles sum the next one's interior K-blocks (shared row
//    panels) and a short completion launch adds the four K-blocks left.
#include <algorithm>
#include <utility>
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "df_arith.cuh"
#include "internal.cuh"
#include "gathered_layout.h"
#include "sweep_schedule.h"
#include "tc_gemm.cuh"

namespace signtri {

namespace {

constexpr int MB = 64;
static_assert(MB == kSweepTile, "the sweep work lists and the kernels share the tile size");

constexpr int kOzakiSlices = 7;   // exact slices of kOzakiBits bits: 49 bits, 28 pairs
constexpr int kOzakiBits = 7;
constexpr int kSuper = 1024;   // superblock of the gathered residual layout

__device__ __forceinline__ float fsgn(double t) { return t > 0.0 ? 1.f : -1.f; }

// One term of a rounding split: the 16-bit rounding of x (bf16, or fp16 when
// f16), x left holding the remainder (exact in fp32).
__device__ __forceinline__ unsigned short split_term(float &x, bool f16)
{
    if (f16) {
        const __half h = __float2half_rn(x);
        x -= __half2float(h);
        return __half_as_ushort(h);
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    x -= __bfloat162float(h);
    return __bfloat16_as_ushort(h);
}

// Four consecutive entries, S terms each, slice s at dst + s * sstride.
__device__ __forceinline__ void split_store4(float4 r, int S, bool f16, __nv_bfloat16 *dst, size_t sstride)
{
    for (int s = 0; s < S; s++) {
        const unsigned a = split_term(r.x, f16), b = split_term(r.y, f16);
        const unsigned c = split_term(r.z, f16), d = split_term(r.w, f16);
        *reinterpret_cast<uint2 *>(dst + s * sstride) = make_uint2(a | (b << 16), c | (d << 16));
    }
}

// --------------------------------------------------------------- leaves ---

constexpr int kLeafThreads = 256;
constexpr int kMicro = 4;            // micro-block edge of the in-tile solve: one thread's entries
constexpr int kMicros = MB / kMicro; // micro-blocks per tile edge
constexpr int kTri = kMicros * (kMicros + 1) / 2;   // micro-blocks of an upper triangular tile
// words from one micro-block to the next in shared memory: eight consecutive
// ones lie in different banks for 16-byte reads
constexpr int kMicroPitch = kMicro * kMicro + 4;
// What a launch of no more leaves than SMs asks for, so that each gets one (left to
// itself the scheduler pairs some beside empty SMs: 27 us a launch all the same
// alone, n = 3001 8.65 -> 7.82 ms, n = 16384 188.5 -> 184.4).
constexpr size_t kLeafAlone = 200 * 1024;
constexpr size_t kLeafSmem = (size_t)(4 * kTri + kMicros * kMicros) * kMicroPitch * sizeof(float);

// Number of micro-block (r, c), r <= c, of an upper triangular tile, row by row.
__host__ __device__ constexpr int tri_index(int r, int c) { return r * kMicros - r * (r - 1) / 2 + c - r; }

// Per-sign operators of the in-block recurrences.  Entry (p, q) of a tile
// (I, J) is fixed by
//   signs differ:  v_pq (t_pp - t_qq) = c_pq + sum_k v_pk T_kq - sum_k T_pk v_kq
//   signs agree:   v_pq (s_p + s_q)   = c_pq - sum_k v_pk A_kq - sum_k A_pk v_kq
// (k over the tile's own rows and columns; A = U in the initial solve, U0 in
// the correction).  So the column part is - sum_k M^{s_q}_pk v_kq, where row
// r of M^+ is A's row r if s_r = +, else T's, and M^- the other way round,
// and the row part is + sum_k v_pk N^{s_p}_kq, where column c of N^+ is -A's
// column c if s_c = +, else +T's, and N^- the other way round.  Per diagonal
// block I, fp32, zero on and below the diagonal (the diagonal terms of T sit
// in the divisor t_pp - t_qq), the micro-blocks of the upper triangle one
// after another (tri_index), M's row by row, N's column by column:
//   OPS[(4 I + 0) 16 kTri ..]  M^+      OPS[(4 I + 1) 16 kTri ..]  M^-
//   OPS[(4 I + 2) 16 kTri ..]  N^+      OPS[(4 I + 3) 16 kTri ..]  N^-
// and DIAG[i] = (float) t_ii (0 beyond n).
__global__ void leaf_ops_kernel(int n, const double *__restrict__ T, int ldt, const double *__restrict__ A, int lda,
                                float *__restrict__ OPS, float *__restrict__ DIAG)
{
    constexpr int E = kMicro * kMicro;
    const int r0 = blockIdx.x * MB;
    __shared__ float sg[MB];
    for (int i = threadIdx.x; i < MB; i += blockDim.x) {
        const bool in = r0 + i < n;
        const double t = in ? SGT_AT(T, ldt, r0 + i, r0 + i) : 0.0;
        sg[i] = (in && t > 0.0) ? 1.f : -1.f;
        DIAG[r0 + i] = (float)t;
    }
    __syncthreads();
    float *mp = OPS + (size_t)(4 * blockIdx.x) * E * kTri;
    for (int idx = threadIdx.x; idx < MB * MB; idx += blockDim.x) {
        const int i = idx % MB, j = idx / MB;   // element (i, j) of the block, i fastest
        if (i / kMicro > j / kMicro) continue;
        const bool in = r0 + j < n && i < j;
        const float t = in ? (float)SGT_AT(T, ldt, r0 + i, r0 + j) : 0.f;
        const float a = in ? (float)SGT_AT(A, lda, r0 + i, r0 + j) : 0.f;
        // M: row i picks by the sign of i; N: column j by the sign of j
        const int mb = tri_index(i / kMicro, j / kMicro) * E;
        const int rm = mb + i % kMicro * kMicro + j % kMicro, cm = mb + j % kMicro * kMicro + i % kMicro;
        mp[0 * E * kTri + rm] = sg[i] > 0.f ? a : t;
        mp[1 * E * kTri + rm] = sg[i] > 0.f ? t : a;
        mp[2 * E * kTri + cm] = sg[j] > 0.f ? -a : t;
        mp[3 * E * kTri + cm] = sg[j] > 0.f ? t : -a;
    }
}

// The seeds of anti-diagonal d's tiles (blockIdx.x): per entry the block sums
// (their K range includes the diagonal blocks K = I and K = J, so they already
// hold the in-block products of the known blocks: U_II T_IJ - T_IJ U_JJ for
// opposite signs in mode 0, E_II T_IJ - T_IJ E_JJ and E_II U0_IJ + U0_IJ E_JJ in
// mode 1; terms with the unknown V_IJ vanish, its slices being still zero),
// float2 (hi, lo) partials summed in fp32 over the slots, and the base terms;
// micro-block by micro-block as the leaf's threads own them, column by column.
// A launch of its own: up to 16 slots of 64 to 96 KB a tile took one leaf CTA
// up to 40 us to read, sixteen CTAs a few.
template <int MODE>
__global__ void __launch_bounds__(kLeafThreads)
leaf_seed_kernel(int n, const double *__restrict__ T, int ldt, const float *__restrict__ DIAG,
                 const double *__restrict__ Rc, const double *__restrict__ Rs, int ldr, int d,
                 const int2 *__restrict__ tslot, const int2 *__restrict__ tslot2, const double *PA,
                 const double *PB, float *__restrict__ SEED)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the leaves may load their operators
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int I = blockIdx.x, J = I + d;
    const int e = blockIdx.y * kLeafThreads + threadIdx.x, p = e % MB, q = e / MB;
    const int gi = I * MB + p, gj = J * MB + q;
    const int2 ts = tslot[I];
    const int2 ts2 = (MODE == 0 && tslot2) ? tslot2[I] : make_int2(0, 0);
    const bool sp = DIAG[gi] > 0.f, sq = gj >= n || DIAG[gj] > 0.f, opp = sp != sq;
    const double own = gj >= n ? 0.0
                       : MODE == 0 ? (opp ? SGT_AT(T, ldt, gi, gj) : 0.0)
                                   : SGT_AT(opp ? Rc : Rs, ldr, gi, gj);
    const float2 *PA2 = reinterpret_cast<const float2 *>(PA), *PB2 = reinterpret_cast<const float2 *>(PB);
    float acc = 0.f;
#pragma unroll 4
    for (int s = 0; s < ts.y + ts2.y; s++) {
        // mode 0: slots of PA, then (look-ahead pairing) slots of PB.  Signs
        // differ: TL - BR of PA (X); agree: TR (Y, mode 0) or TL + BR of PB (Y^E)
        const bool second = s >= ts.y;
        const size_t at = (size_t)(second ? ts2.x + s - ts.y : ts.x + s) * 16384 + e;
        const float2 *P0 = (second ? PB2 : PA2) + at;
        const float2 *src = opp ? P0 : (MODE == 0 ? P0 + 4096 : PB2 + at);
        const float2 l1 = src[0];
        float2 l2 = make_float2(0.f, 0.f);
        if (MODE == 1 || opp) l2 = src[3 * 4096];
        const float sg = opp ? -1.f : 1.f;
        acc += (l1.x + sg * l2.x) + (l1.y + sg * l2.y);
    }
    const float b = (float)own;
    float c = opp ? acc : -acc;
    if (MODE == 0) c += opp ? b * (sp ? 2.f : -2.f) : 0.f;
    else c -= b;
    if (gj >= n) c = 0.f;
    SEED[(size_t)I * MB * MB + ((p / kMicro * kMicros + q / kMicro) * kMicro + q % kMicro) * kMicro + p % kMicro] = c;
}

// MODE 0: V = U (initial solve).  MODE 1: V = E (correction), with Rc, Rs.
// Each of the 256 threads owns a 4 x 4 micro-block of the tile: its seeds (base
// terms and block sums) wait in shared memory where its V will be, the in-tile
// terms gather in registers.  Phase ph = 0 .. 30
// solves the micro-blocks with 15 - mr + mc = ph, each by its thread (they
// depend on those below and to the left only), and, after one barrier, every
// later micro-block of the same rows or columns takes the phase's terms as
// 4 x 4 x 4 products: 31 barriers and short register chains, where 16 x 16
// sub-blocks solved by one warp each took 7 phases of 31 steps of shuffles
// (100 thousand cycles a tile, 73 of them in the solve).
// Shared memory (fp32): the operators of block I (M^+, M^-) and of block J
// (N^+, N^-) and the solved V, micro-block by micro-block (V's columns of four).
template <int MODE>
__global__ void __launch_bounds__(kLeafThreads, 2)
mixed_leaf_kernel(int n, double *__restrict__ V, int ldv, const float *__restrict__ OPS, const float *__restrict__ DIAG,
                  int d, const float *SEED, __nv_bfloat16 *__restrict__ Vr, __nv_bfloat16 *__restrict__ Vc,
                  int S, int nbk, float sigma)
{
    constexpr int E = kMicro * kMicro, PT = kMicroPitch;
    static_assert(kLeafThreads == kMicros * kMicros, "one micro-block per thread");
    extern __shared__ float4 fsm4[];
    float *Mp = reinterpret_cast<float *>(fsm4), *Mm = Mp + kTri * PT, *Np = Mm + kTri * PT, *Nm = Np + kTri * PT;
    float *Vs = Nm + kTri * PT;
    const int I = blockIdx.x, J = I + d;
    const int r0 = I * MB, c0 = J * MB;
    const int bj = min(MB, n - c0);
    // a warp's micro-blocks: 8 rows of 4, so that its rows' and its columns'
    // terms both come in few of the phases
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mr = (warp >> 2) * 8 + (lane >> 2), mc = (warp & 3) * 4 + (lane & 3), own = mr * kMicros + mc;
    auto four = [](const float *x) { return *reinterpret_cast<const float4 *>(x); };
    // the operators, all loads in flight before the first store
    {
        const float4 *sm = reinterpret_cast<const float4 *>(OPS + (size_t)(4 * I) * E * kTri);
        const float4 *sn = reinterpret_cast<const float4 *>(OPS + (size_t)(4 * J + 2) * E * kTri);
        constexpr int N4 = 2 * E * kTri / 4, V4 = (N4 + kLeafThreads - 1) / kLeafThreads;
        float4 vm[V4], vn[V4];
#pragma unroll
        for (int i = 0; i < V4; i++) {
            const int x = threadIdx.x + i * kLeafThreads;
            if (x < N4) {
                vm[i] = sm[x];
                vn[i] = sn[x];
            }
        }
#pragma unroll
        for (int i = 0; i < V4; i++) {
            const int x = threadIdx.x + i * kLeafThreads;
            if (x < N4) {
                *reinterpret_cast<float4 *>(Mp + x / kMicro * PT + x % kMicro * kMicro) = vm[i];
                *reinterpret_cast<float4 *>(Np + x / kMicro * PT + x % kMicro * kMicro) = vn[i];
            }
        }
    }
    bool sp[4], sq[4];         // signs of the rows and columns (beyond n: +)
    float c[4][4], rd[4][4];   // [row][column]: pending values, reciprocal divisors t_pp - t_qq or s_p + s_q
    {
        const float4 a = four(DIAG + r0 + kMicro * mr), b = four(DIAG + c0 + kMicro * mc);
        const float dp[4] = {a.x, a.y, a.z, a.w}, dq[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            sp[i] = dp[i] > 0.f;
            sq[i] = kMicro * mc + i >= bj || dq[i] > 0.f;
        }
#pragma unroll
        for (int p = 0; p < 4; p++)
#pragma unroll
            for (int q = 0; q < 4; q++)
                rd[p][q] = __fdividef(1.f, sp[p] != sq[q] ? dp[p] - dq[q] : (sp[p] ? 2.f : -2.f));
    }
    // (SEED is written by the launch before: a restricted pointer's loads could
    // be moved above the wait)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 4; q++) {
        *reinterpret_cast<float4 *>(Vs + own * PT + q * kMicro) =
            four(SEED + (size_t)I * MB * MB + (own * kMicro + q) * kMicro);
        c[0][q] = c[1][q] = c[2][q] = c[3][q] = 0.f;
    }
    __syncthreads();

    const int mine = kMicros - 1 - mr + mc;
    for (int ph = 0; ph < 2 * kMicros - 1; ph++) {
        if (ph == mine) {
            // the micro-block's own recurrence (Algorithm 6, 1x1 case), column by
            // column from the bottom row up; the term solved last is added last
            const int dm = tri_index(mr, mr) * PT, dn = tri_index(mc, mc) * PT;
            float4 mp[3], mm[3], np[4], nm[4];
#pragma unroll
            for (int i = 0; i < 3; i++) {
                mp[i] = four(Mp + dm + i * kMicro);
                mm[i] = four(Mm + dm + i * kMicro);
                np[i + 1] = four(Np + dn + (i + 1) * kMicro);
                nm[i + 1] = four(Nm + dn + (i + 1) * kMicro);
            }
            auto el = [](const float4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; };
#pragma unroll
            for (int q = 0; q < 4; q++) {
                float *vq = Vs + own * PT + q * kMicro;
                const float4 seed = four(vq);
#pragma unroll
                for (int p = 3; p >= 0; p--) {
                    float x = c[p][q] + el(seed, p);
#pragma unroll
                    for (int k = 0; k < q; k++) x = fmaf(c[p][k], sp[p] ? el(np[q], k) : el(nm[q], k), x);
#pragma unroll
                    for (int k = 3; k > p; k--) x = fmaf(sq[q] ? -el(mp[p], k) : -el(mm[p], k), c[k][q], x);
                    c[p][q] = x * rd[p][q];
                }
                *reinterpret_cast<float4 *>(vq) = make_float4(c[0][q], c[1][q], c[2][q], c[3][q]);
            }
        }
        __syncthreads();
        if (ph < mine) {
            // the micro-blocks solved now in the same rows (K, to the left) and in
            // the same columns (L, below)
            const int K = ph - (kMicros - 1) + mr, L = kMicros - 1 + mc - ph;
            if (K >= 0) {
                const float *v = Vs + (mr * kMicros + K) * PT;
                const int o = tri_index(K, mc) * PT;
                const float4 v0 = four(v), v1 = four(v + 4), v2 = four(v + 8), v3 = four(v + 12);
                const float w[4][4] = {{v0.x, v1.x, v2.x, v3.x}, {v0.y, v1.y, v2.y, v3.y},
                                       {v0.z, v1.z, v2.z, v3.z}, {v0.w, v1.w, v2.w, v3.w}};
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float4 a = four(Np + o + q * kMicro), b = four(Nm + o + q * kMicro);
#pragma unroll
                    for (int p = 0; p < 4; p++) {
                        c[p][q] = fmaf(w[p][0], sp[p] ? a.x : b.x, c[p][q]);
                        c[p][q] = fmaf(w[p][1], sp[p] ? a.y : b.y, c[p][q]);
                        c[p][q] = fmaf(w[p][2], sp[p] ? a.z : b.z, c[p][q]);
                        c[p][q] = fmaf(w[p][3], sp[p] ? a.w : b.w, c[p][q]);
                    }
                }
            }
            if (L < kMicros) {
                const float *v = Vs + (L * kMicros + mc) * PT;
                const int o = tri_index(mr, L) * PT;
                float4 w[4];
#pragma unroll
                for (int q = 0; q < 4; q++) w[q] = four(v + q * kMicro);
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    const float4 a = four(Mp + o + p * kMicro), b = four(Mm + o + p * kMicro);
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        c[p][q] = fmaf(sq[q] ? -a.x : -b.x, w[q].x, c[p][q]);
                        c[p][q] = fmaf(sq[q] ? -a.y : -b.y, w[q].y, c[p][q]);
                        c[p][q] = fmaf(sq[q] ? -a.z : -b.z, w[q].z, c[p][q]);
                        c[p][q] = fmaf(sq[q] ? -a.w : -b.w, w[q].w, c[p][q]);
                    }
                }
            }
        }
    }
    // (the last phase's barrier was passed after its values were stored)

    // V (float64) and its 16-bit splits in the blocked slice layout: row
    // slices tile (I, J) of Vr[s] (row-major), column slices tile (J, I) of
    // Vc[s] (V^T, row-major).  The split runs in fp32, of V (bf16 terms) or
    // of sigma V (fp16 terms, sigma a power of two): each remainder is exact
    const bool f16 = sigma > 0.f;
    const float sc = f16 ? sigma : 1.f;
    const size_t tr = ((size_t)I * nbk + J) * MB * MB, tc = ((size_t)J * nbk + I) * MB * MB;
    const size_t sstride = (size_t)nbk * nbk * MB * MB;
    // four consecutive entries per thread and store
    for (int idx = threadIdx.x; idx < MB * MB / 4; idx += kLeafThreads) {
        const int m = idx % kMicros, q = idx / kMicros;   // rows 4 m .., column q
        if (q < bj) {
            const float4 r = four(Vs + (m * kMicros + q / kMicro) * PT + q % kMicro * kMicro);
            double *vo = &SGT_AT(V, ldv, r0 + kMicro * m, c0 + q);
            vo[0] = f32_to_f64_bits(r.x);
            vo[1] = f32_to_f64_bits(r.y);
            vo[2] = f32_to_f64_bits(r.z);
            vo[3] = f32_to_f64_bits(r.w);
            split_store4(make_float4(r.x * sc, r.y * sc, r.z * sc, r.w * sc), S, f16, Vc + tc + q * MB + kMicro * m, sstride);
        }
    }
    for (int idx = threadIdx.x; idx < MB * MB / 4; idx += kLeafThreads) {
        const int m = idx % kMicros, pr = idx / kMicros;   // row pr, columns 4 m .. (beyond n: 0)
        if (kMicro * m < bj) {
            const float *v = Vs + (pr / kMicro * kMicros + m) * PT + pr % kMicro;
            split_store4(make_float4(v[0] * sc, v[4] * sc, v[8] * sc, v[12] * sc), S, f16, Vr + tr + pr * MB + kMicro * m, sstride);
        }
    }
}

// Correction on the diagonal blocks: the recurrences above restricted to one
// block, by anti-diagonal, float64, each entry's terms split over four
// neighbouring lanes (a chain of dependent float64 operations takes 74 cycles
// for each: one lane an entry took 0.5 ms).
__global__ void __launch_bounds__(kLeafThreads)
corr_diag_leaf_kernel(int n, const double *__restrict__ T, int ldt, const double *__restrict__ U0, int ldu0,
                      const double *__restrict__ Rc, const double *__restrict__ Rs, int ldr, double *__restrict__ E,
                      int lde)
{
    constexpr int LD = MB + 1;
    static_assert(kLeafThreads == 4 * MB, "four lanes per entry of an anti-diagonal");
    extern __shared__ double dsm[];
    double *Ts = dsm;
    double *Us = Ts + MB * LD;
    double *Es = Us + MB * LD;   // -Rc or -Rs until the entry is solved
    const int r0 = blockIdx.x * MB;
    const int bs = min(MB, n - r0);
    for (int idx = threadIdx.x; idx < bs * bs; idx += kLeafThreads) {
        const int i = idx % bs, j = idx / bs;
        Ts[i + j * LD] = (i <= j) ? SGT_AT(T, ldt, r0 + i, r0 + j) : 0.0;
        Us[i + j * LD] = (i <= j) ? SGT_AT(U0, ldu0, r0 + i, r0 + j) : 0.0;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < bs * bs; idx += kLeafThreads) {
        const int i = idx % bs, j = idx / bs;
        const bool opp = (__double2hiint(Ts[i + i * LD]) ^ __double2hiint(Ts[j + j * LD])) < 0;
        Es[i + j * LD] = i < j ? -SGT_AT(opp ? Rc : Rs, ldr, r0 + i, r0 + j) : 0.0;
    }
    __syncthreads();
    const int i = threadIdx.x / 4, part = threadIdx.x % 4;
    for (int dd = 1; dd < bs; dd++) {
        const int j = i + dd;
        const bool live = j < bs;
        double s = 0.0;
        bool opp = false;
        if (live) {
            opp = (__double2hiint(Ts[i + i * LD]) ^ __double2hiint(Ts[j + j * LD])) < 0;
            // signs differ: e t - t e; agree: - u e - e u
            const double *M = opp ? Ts : Us;
            for (int k = i + 1 + part; k < j; k += 4) {
                s = fma(-M[i + k * LD], Es[k + j * LD], s);
                s = fma(opp ? Es[i + k * LD] : -Es[i + k * LD], M[k + j * LD], s);
            }
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (live && part == 0) {
            s += Es[i + j * LD];
            const Divisor<double> dv = divisor_recip(Ts[i + i * LD] - Ts[j + j * LD]);
            Es[i + j * LD] = opp ? s * dv.r * power_of_2(dv.ex) : s * copysign(0.5, Ts[i + i * LD]);
        }
        __syncthreads();
    }
    for (int idx = threadIdx.x; idx < bs * bs; idx += kLeafThreads) {
        const int i2 = idx % bs, j2 = idx / bs;
        if (i2 < j2) SGT_AT(E, lde, r0 + i2, r0 + j2) = Es[i2 + j2 * LD];
    }
}

// ------------------------------------------------------------- residual ---

// Residual of entry (i < j) into R (column-major n x n): Rc_ij when the signs
// of i and j differ, Rs_ij when they agree, from the gathered products
// (RA: Y at equal-sign positions, N_T N_U at opposite-sign ones; RB: N_U N_T)
// plus the diagonal terms.  Only the strictly upper part of R is written: the
// correction reads nothing else.  Squared Frobenius norms of the used Rc and
// Rs entries, of T and of U into norms[0..3].  Bound by the float64 pipes (10
// instructions an entry; 15 with the diagonal terms written out).
__global__ void needed_finalize_kernel(int n, const double *__restrict__ T, int ldt, const double *__restrict__ U,
                                       int ldu, const int *__restrict__ gmap, const double *__restrict__ RA,
                                         const double *__restrict__ RB, int ldg, double *__restrict__ R,
                                         double *__restrict__ norms)
{
    const int j = blockIdx.x;
    double nc = 0.0, ns = 0.0, nt = 0.0, nu = 0.0;
    const double tjj = SGT_AT(T, ldt, j, j), ujj = SGT_AT(U, ldu, j, j);
    const double two = 2.0 * ujj;
    const size_t gj = (size_t)gmap[j] * ldg;
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
        const double tii = SGT_AT(T, ldt, i, i);
        const double tij = SGT_AT(T, ldt, i, j), uij = SGT_AT(U, ldu, i, j);
        const size_t g = (size_t)gmap[i] + gj;
        const bool opp = (__double2hiint(tii) ^ __double2hiint(tjj)) < 0;
        // u_ii = +-1 and u_jj = +-1: u_ii u_ij + u_ij u_jj = 2 u_jj u_ij where they
        // agree, t_ij u_jj - u_ii t_ij = 2 u_jj t_ij where they differ
        double r = fma(two, opp ? tij : uij, RA[g]);
        if (opp) r += fma(tii, uij, -(uij * tjj)) - RB[g];
        nc = fma(r, opp ? r : 0.0, nc);
        ns = fma(r, opp ? 0.0 : r, ns);
        nt += tij * tij;
        nu += uij * uij;
        SGT_AT(R, n, i, j) = r;
    }
    if (threadIdx.x == 0) {
        nt += tjj * tjj;
        nu += ujj * ujj;
    }
    __shared__ double red[4][256];
    red[0][threadIdx.x] = nc; red[1][threadIdx.x] = ns; red[2][threadIdx.x] = nt; red[3][threadIdx.x] = nu;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off)
            for (int c = 0; c < 4; c++) red[c][threadIdx.x] += red[c][threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int c = 0; c < 4; c++) atomicAdd(&norms[c], red[c][0]);
}

// Full residuals, in place: Ptu -> Rc, Puu -> Rs (i < j; other entries 0),
// and the squared Frobenius norms of Rc, Rs (all entries), T, U into
// norms[0..3].
__global__ void residual_finalize_kernel(int n, const double *__restrict__ T, int ldt, const double *__restrict__ U,
                                         int ldu, double *__restrict__ Ptu, const double *__restrict__ Put,
                                         double *__restrict__ Puu, int ldp, double *__restrict__ norms)
{
    const int j = blockIdx.x;
    double nc = 0.0, ns = 0.0, nt = 0.0, nu = 0.0;
    const double tjj = SGT_AT(T, ldt, j, j), ujj = SGT_AT(U, ldu, j, j);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double rc = 0.0, rs = 0.0;
        if (i < j) {
            const double tii = SGT_AT(T, ldt, i, i), uii = SGT_AT(U, ldu, i, i);
            const double tij = SGT_AT(T, ldt, i, j), uij = SGT_AT(U, ldu, i, j);
            rc = SGT_AT(Ptu, ldp, i, j) - SGT_AT(Put, ldp, i, j) + (tii * uij - uij * tjj) + (tij * ujj - uii * tij);
            rs = SGT_AT(Puu, ldp, i, j) + uii * uij + uij * ujj;
            nt += tij * tij;
            nu += uij * uij;
        } else if (i == j) {
            nt += tjj * tjj;
            nu += ujj * ujj;
        }
        SGT_AT(Ptu, ldp, i, j) = rc;
        SGT_AT(Puu, ldp, i, j) = rs;
        nc += rc * rc;
        ns += rs * rs;
    }
    __shared__ double red[4][256];
    red[0][threadIdx.x] = nc; red[1][threadIdx.x] = ns; red[2][threadIdx.x] = nt; red[3][threadIdx.x] = nu;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off)
            for (int c = 0; c < 4; c++) red[c][threadIdx.x] += red[c][threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int c = 0; c < 4; c++) atomicAdd(&norms[c], red[c][0]);
}

// sign flags of the diagonal (1 = positive)
__global__ void diag_sign_kernel(int n, const double *__restrict__ T, int ldt, unsigned char *__restrict__ pos)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pos[i] = SGT_AT(T, ldt, i, i) > 0.0 ? 1 : 0;
}

// U += E on the strictly upper part; ||E||_F^2 into norms[4].
__global__ void apply_correction_kernel(int n, double *__restrict__ U, int ldu, const double *__restrict__ E, int lde,
                                        double *__restrict__ norms)
{
    const int j = blockIdx.x;
    double ne = 0.0;
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
        const double e = SGT_AT(E, lde, i, j);
        SGT_AT(U, ldu, i, j) += e;
        ne += e * e;
    }
    __shared__ double red[256];
    red[threadIdx.x] = ne;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(&norms[4], red[0]);
}

// Rounding-split slices of the strictly upper part of the diagonal blocks
// of V (U after the float64 diagonal leaves, E after the corrections'
// diagonal leaves), in the blocked layout the leaves write: tile (I, I) of
// Vr[s] (row-major) and of Vc[s] (transposed).  bf16 terms of V (split in
// float64), or fp16 terms of sigma V (sigma > 0, split in fp32: two terms
// keep 22 bits).  One CTA per block.
__global__ void diag_slices_kernel(int n, const double *__restrict__ V, int ldv, __nv_bfloat16 *__restrict__ Vr,
                                   __nv_bfloat16 *__restrict__ Vc, int S, int nbk, float sigma)
{
    const int I = blockIdx.x, r0 = I * MB;
    const int bs = min(MB, n - r0);
    const size_t t = ((size_t)I * nbk + I) * MB * MB, sstride = (size_t)nbk * nbk * MB * MB;
    for (int idx = threadIdx.x; idx < bs * bs; idx += blockDim.x) {
        const int i = idx % bs, j = idx / bs;
        double r = (i < j) ? SGT_AT(V, ldv, r0 + i, r0 + j) : 0.0;
        if (sigma > 0.f) {
            float x = (float)(r * (double)sigma);
            for (int s = 0; s < S; s++) {
                const unsigned short h = split_term(x, true);
                Vr[s * sstride + t + i * MB + j] = __ushort_as_bfloat16(h);
                Vc[s * sstride + t + j * MB + i] = __ushort_as_bfloat16(h);
            }
            continue;
        }
        for (int s = 0; s < S; s++) {
            const __nv_bfloat16 h = __double2bfloat16(r);
            Vr[s * sstride + t + i * MB + j] = h;
            Vc[s * sstride + t + j * MB + i] = h;
            r -= (double)__bfloat162float(h);
        }
    }
}

// Rounding-split slices (of the fp32 value, as the leaves split: bf16 terms,
// or fp16 terms of sigma M when sigma > 0) of the strictly upper part of the
// n x n matrix M in the blocked layout: tile (I, K) of R[s] (row-major) and
// tile (K, I) of C[s] (transposed) for every block K >= I; the blocks below
// are never read and not written.
__global__ void blocked_split_kernel(int n, const double *__restrict__ M, int ldm, int S, int nbk,
                                     __nv_bfloat16 *__restrict__ R, __nv_bfloat16 *__restrict__ C, float sigma)
{
    __shared__ float tile[MB][MB + 1];   // [column][row]
    const int K = blockIdx.x, I = blockIdx.y;
    if (K < I) return;
    const bool f16 = sigma > 0.f;
    const double sc = f16 ? (double)sigma : 1.0;
    const size_t sstride = (size_t)nbk * nbk * MB * MB;
    const size_t tr = ((size_t)I * nbk + K) * MB * MB, tc = ((size_t)K * nbk + I) * MB * MB;
    for (int idx = threadIdx.x; idx < MB * MB; idx += blockDim.x) {
        const int r = idx % MB, k = idx / MB;
        const int gi = I * MB + r, gk = K * MB + k;
        const float v = (gi < gk && gk < n) ? (float)(SGT_AT(M, ldm, gi, gk) * sc) : 0.f;
        tile[k][r] = v;
        float x = v;
        for (int s = 0; s < S; s++) C[s * sstride + tc + k * MB + r] = __ushort_as_bfloat16(split_term(x, f16));
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < MB * MB; idx += blockDim.x) {
        const int k = idx % MB, r = idx / MB;
        float x = tile[k][r];
        for (int s = 0; s < S; s++) R[s * sstride + tr + r * MB + k] = __ushort_as_bfloat16(split_term(x, f16));
    }
}

// Largest |entry| of the strictly upper parts of the 64 x 64 diagonal blocks
// of the n x n matrix M, as the bits of a non-negative float (ordered like
// the values) max-ed into *out.
__global__ void absmax_diag_blocks_kernel(int n, const double *__restrict__ M, int ldm, unsigned *__restrict__ out)
{
    float m = 0.f;
    const long long total = (long long)((n + MB - 1) / MB) * MB * MB;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(e / (MB * MB)), w = (int)(e % (MB * MB));
        const int i = b * MB + w % MB, j = b * MB + w / MB;
        if (i < j && j < n) m = fmaxf(m, fabsf(f64_to_f32_trunc(SGT_AT(M, ldm, i, j))));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// Largest of `count` non-negative float64 values held as their bits (the
// per-row maxima the exact slices' scales come from), as float bits max-ed
// into *out.
__global__ void max_of_maxima_kernel(int count, const unsigned long long *__restrict__ bits, unsigned *__restrict__ out)
{
    float m = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        m = fmaxf(m, (float)__longlong_as_double((long long)bits[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// Largest first-order correction term |e_ij| ~ |Rc_ij| / |t_ii - t_jj|
// (signs differ) or |Rs_ij| / 2 (signs agree) over the strictly upper
// entries, max-ed into *out as float bits (see absmax_diag_blocks_kernel).
// D: t_ii in fp32.  One column per CTA step: coalesced reads of R and D.
__global__ void corr_magnitude_kernel(int n, const float *__restrict__ D, const double *__restrict__ Rc,
                                      const double *__restrict__ Rs, int ldr, unsigned *__restrict__ out)
{
    float m = 0.f;
    for (int j = blockIdx.x; j < n; j += gridDim.x) {
        const float tj = D[j];
        for (int i = threadIdx.x; i < j; i += blockDim.x) {
            const float ti = D[i];
            // fp32 magnitudes truncated from the bits (no float64 conversion)
            const float v = ((ti > 0.f) != (tj > 0.f)) ? fabsf(f64_to_f32_trunc(SGT_AT(Rc, ldr, i, j))) / fabsf(ti - tj)
                                                       : 0.5f * fabsf(f64_to_f32_trunc(SGT_AT(Rs, ldr, i, j)));
            m = fmaxf(m, v);
        }
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

__global__ void fill_float_kernel(int count, float v, float *__restrict__ p)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) p[i] = v;
}

// ---------------------------------------------------------- probe check ---
// Acceptance test by random probes: for Z (n x kProbes) with independent +-1
// entries, E ||R Z||_F^2 = kProbes ||R||_F^2 for any R, so
// ||R Z||_F / sqrt(kProbes) estimates ||R||_F.  R Z = T (U Z) - U (T Z) and
// U (U Z) - Z are formed with the emulated-float64 products of the full
// residual (n x n by n x kProbes), about 2^-45 |T||U| entrywise.
constexpr int kProbes = 128;

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x)
{
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}

// Z[i + j n] = +-1 (bit of a counter hash), its one bf16 column slice
// Zc[j][i] = +-64 with column scale 2 (+-1 = 2 * 64 * 2^-7 exactly), zero
// padding up to np.
__global__ void probe_kernel(int n, int np, unsigned long long seed, double *__restrict__ Z,
                             __nv_bfloat16 *__restrict__ Zc, float *__restrict__ zscale)
{
    const int j = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
        float z = 0.f;
        if (i < n) {
            z = (splitmix64(seed ^ ((unsigned long long)j << 32 ^ (unsigned long long)i)) >> 63) ? -1.f : 1.f;
            Z[(size_t)i + (size_t)j * n] = (double)z;
        }
        Zc[(size_t)j * np + i] = __float2bfloat16_rn(64.f * z);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) zscale[j] = 2.f;
}

// W = Pa + Pb + diag(M) Y  (n x kProbes, column-major, ld n)
__global__ void probe_combine_kernel(int n, const double *__restrict__ Pa, const double *__restrict__ Pb,
                                     const double *__restrict__ M, int ldm, const double *__restrict__ Y,
                                     double *__restrict__ W)
{
    const int j = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const size_t e = (size_t)i + (size_t)j * n;
        W[e] = Pa[e] + Pb[e] + SGT_AT(M, ldm, i, i) * Y[e];
    }
}

// R_c Z = N_T W1 + diag(T) W1 - N_U W2 - diag(U) W2 and R_s Z = N_U W1 +
// diag(U) W1 - Z, squared norms into norms[0], norms[1] (each product as two
// K halves a, b).
__global__ void probe_residual_kernel(int n, const double *__restrict__ T, int ldt, const double *__restrict__ U,
                                      int ldu, const double *__restrict__ Z, const double *__restrict__ W1,
                                      const double *__restrict__ W2, const double *__restrict__ P1a,
                                      const double *__restrict__ P1b, const double *__restrict__ P2a,
                                      const double *__restrict__ P2b, const double *__restrict__ P3a,
                                      const double *__restrict__ P3b, double *__restrict__ norms)
{
    const int j = blockIdx.y;
    double nc = 0.0, ns = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const size_t e = (size_t)i + (size_t)j * n;
        const double tii = SGT_AT(T, ldt, i, i), uii = SGT_AT(U, ldu, i, i);
        const double rc = (P1a[e] + P1b[e]) + tii * W1[e] - (P2a[e] + P2b[e]) - uii * W2[e];
        const double rs = (P3a[e] + P3b[e]) + uii * W1[e] - Z[e];
        nc += rc * rc;
        ns += rs * rs;
    }
    __shared__ double red[2][256];
    red[0][threadIdx.x] = nc;
    red[1][threadIdx.x] = ns;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) {
            red[0][threadIdx.x] += red[0][threadIdx.x + off];
            red[1][threadIdx.x] += red[1][threadIdx.x + off];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd(&norms[0], red[0][0]);
        atomicAdd(&norms[1], red[1][0]);
    }
}

__global__ void zero_kernel(size_t count, double *__restrict__ p)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        p[i] = 0.0;
}

// ------------------------------------------------------------ host side ---

// A schedule's device copy (job list, per-CTA job ranges, per-tile slots).
struct DevSchedule {
    TcJob *jobs = nullptr;
    int *cta_off = nullptr;
    int2 *tslot = nullptr;
};

struct MixedCtx {
    int n, np, S;
    // fp16 split (S = 2): T, U and E are split as sT T, sU U, sE E (powers of
    // two), and the products' rows and columns scaled back by invT, invU,
    // invE (np + 64 entries, constant); sT = sU = sE = 0 for the bf16 splits
    bool f16;
    float sT, sU, sE;
    float *invT, *invU, *invE;
    unsigned *amax;             // float bits of a maximum the fp16 scales come from
    cudaStream_t st;
    int *d_err;
    Schedule sc, sc2;           // initial sweep; correction (two launches side by side)
    DevSchedule ds, ds2;
    Schedule scA, scB, scC;     // initial sweep's look-ahead pairs: lead, look-ahead, completion
    DevSchedule dsA, dsB, dsC;
    cudaStream_t side;          // second stream of the correction launches (null: one stream)
    cudaEvent_t ev_fork, ev_join;
    TcPairs pairs_split, pairs_oz;
    TcPairs *d_pairs_split, *d_pairs_oz;
    // bf16 splits (S slices) of T and of the unknowns, row and column forms,
    // blocked layout (each 64 x 64 tile contiguous)
    __nv_bfloat16 *Tr, *Tc, *Ur, *Uc, *Er, *Ec;
    float *SEED;                // the leaves' seeds of one anti-diagonal
    float *OPS, *DIAG;          // per-sign fp32 operators of the diagonal blocks for the leaves, fp32 diagonal
    // exact slices of the strictly upper parts of T and U in the gathered
    // layout (residual products): ng gathered positions, rows_g allocated
    // (the last 64 all zero), pitch rows_g
    int ng, rows_g;
    int *gmap, *ginv;           // original -> gathered, gathered -> original (-1 padding)
    int *sbbase;                // gathered start of each superblock (nsb + 1 entries)
    unsigned char *pos;         // diagonal sign flags
    __nv_bfloat16 *NTgr, *NTgc;         // T, gathered layout
    __nv_bfloat16 *NTr, *NTc;           // T, original layout
    __nv_bfloat16 *NUr, *NUc;           // U, either layout (sized for the gathered one)
    float *sTr, *sTc, *sUr, *sUc;       // scales, original indices
    float *gTr, *gTc, *gUr, *gUc;       // scales, gathered
    unsigned long long *tmpmax, *tmpmax2;
    double *PA, *PB;            // block-sum partials
    double *E;                  // correction
    // residual products: gathered RA, RB or full-layout Ptu -> Rc, Put (same
    // memory); R = Rs (full) or the per-entry residual (needed form)
    double *RA, *RB, *R;
    const double *res_c, *res_s;   // what the last residual left for the correction
    double *norms, *norms_host; // [0] Rc^2 [1] Rs^2 [2] T^2 [3] U^2 [4] E^2
    // probe check: Z, its slice and scale, W1 = U Z, W2 = T Z and their
    // slices and scales, the product halves, the jobs (row pairs x K halves)
    double *Z, *W1, *W2, *Pp;
    __nv_bfloat16 *Zc, *W1c, *W2c;
    float *zscale, *w1scale, *w2scale;
    TcJob *d_probe_jobs;
    int n_probe_jobs;
    double probe_kb;
    TcPairs pairs_z;            // (s, 0): Z has one slice
    TcPairs *d_pairs_z;
    double nT2, nU2;            // squared norms of T and U from the last needed residual
    TcJob *d_full_jobs;         // full residual: 2 x 2 block jobs
    int n_full_jobs;
    double full_kb;             // sum over full jobs of used quadrants x K-blocks
    TcJob *d_res_jobs;          // needed residual: equal-sign jobs, then opposite-sign jobs
    int n_res_same, n_res_opp;
    double res_kb_same, res_kb_opp;   // sum over jobs of used quadrants x K-blocks
};

// Gathered size bound: each superblock pads two sign classes to 64.
int gathered_bound(int n) { return pad64(n) + 128 * ((n + kSuper - 1) / kSuper); }

size_t bytes_for(int n, int S)
{
    const size_t np = (size_t)pad64(n);
    const size_t nb = np / MB;
    size_t b = 0;
    b += 6 * (size_t)S * np * np * 2 + 6 * 256;                       // split slices
    const size_t ngr = (size_t)gathered_bound(n) + 64;
    b += 4 * (size_t)kOzakiSlices * ngr * ngr * 2 + 4 * 256;           // exact slices: T gathered, U
    b += 2 * (size_t)kOzakiSlices * (np + 64) * np * 2 + 2 * 256;      // exact slices: T original
    b += 4 * (np + 64) * 4 + 2 * (np + 64) * 8 + 7 * 256;               // scales, tmp
    b += 4 * ngr * 4 + 4 * 256 + 2 * ngr * 4 + np + 3 * 256;            // gathered scales, maps, signs
    b += ((size_t)(n + kSuper - 1) / kSuper + 1) * 4 + 256;             // superblock starts
    b += 2 * ngr * ngr * 8 + 2 * 256;                                   // RA, RB
    const size_t maxjobs = (size_t)kSweepCtas + 2 * nb + 8;
    b += 2 * maxjobs * 16384 * 8 + 2 * 256;                             // partials
    b += 2 * (size_t)n * n * 8 + 2 * 256;                               // E, R (= Rs)
    b += 64 + 256;                                                      // norms
    b += ph_fp64_workspace_bytes(n, 16) + 512;                         // diagonal blocks' partial sums
    // leaf operators, seeds, diagonal
    b += nb * (4 * kMicro * kMicro * kTri + MB * MB + MB) * sizeof(float) + 3 * 256;
    b += 3 * (np + 64) * sizeof(float) + 64 + 4 * 256;                  // fp16 split scales, max slot
    const size_t pairs_max = ngr / 128 + 2 * (size_t)((n + kSuper - 1) / kSuper) + 2;
    b += pairs_max * pairs_max * sizeof(TcJob) + 256;                   // needed-residual jobs
    const size_t nbp = (nb + 1) / 2;
    b += nbp * (nbp + 1) / 2 * sizeof(TcJob) + 256;                     // full-residual jobs
    b += 5 * (nb * (size_t)(kSweepCtas + 2 * nb) * sizeof(TcJob) + 256); // wavefront jobs (bound), 5 schedules
    b += 5 * (nb * (size_t)(kSweepCtas + 1) * sizeof(int) + 256);         // per-CTA job ranges
    b += 5 * ((size_t)nb * nb * sizeof(int2) + 256);                      // per-tile partial slots
    b += 3 * sizeof(TcPairs) + 768;
    b += 13 * (size_t)n * kProbes * 8 + 4 * 256;                       // probe Z, W1, W2, product halves
    b += (1 + 2 * (size_t)kOzakiSlices) * kProbes * np * 2 + 3 * 256;  // their slices
    b += 3 * kProbes * 4 + (2 * nbp + 2) * sizeof(TcJob) + 4 * 256;     // scales, probe jobs
    return b;
}

template <typename P>
P *take(Arena &ws, size_t count)
{
    return static_cast<P *>(ws.take(count * sizeof(P)));
}

// 2^(target - floor(log2 m)) for m > 0: scales m into [2^target, 2^(target+1)).
float pow2_scale(float m, int target)
{
    int e = 0;
    std::frexp(m, &e);   // m = f 2^e, f in [0.5, 1)
    return std::ldexp(1.f, std::max(-120, std::min(120, target - (e - 1))));
}

// Reads back the float max-ed into c.amax (the host waits for it).
signtri_status read_amax(MixedCtx &c, float &m)
{
    unsigned bits = 0;
    SGT_CUDA_TRY(cudaMemcpyAsync(&bits, c.amax, sizeof(unsigned), cudaMemcpyDeviceToHost, c.st));
    SGT_CUDA_TRY(cudaStreamSynchronize(c.st));
    std::memcpy(&m, &bits, sizeof(float));
    return SIGNTRI_OK;
}

// Largest |entry| of the strictly upper parts of M's diagonal blocks into m.
signtri_status diag_blocks_absmax(MixedCtx &c, const double *M, int ldm, float &m)
{
    SGT_CUDA_TRY(cudaMemsetAsync(c.amax, 0, sizeof(unsigned), c.st));
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, c.st);
        absmax_diag_blocks_kernel<<<152, 256, 0, c.st>>>(c.n, M, ldm, c.amax);
        SGT_LAUNCH_CHECK();
    }
    return read_amax(c, m);
}

// Largest of the per-row maxima in c.tmpmax (np + 64 entries) into m.
signtri_status row_maxima_max(MixedCtx &c, float &m)
{
    SGT_CUDA_TRY(cudaMemsetAsync(c.amax, 0, sizeof(unsigned), c.st));
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, c.st);
        max_of_maxima_kernel<<<32, 256, 0, c.st>>>(c.np + 64, c.tmpmax, c.amax);
        SGT_LAUNCH_CHECK();
    }
    return read_amax(c, m);
}

// inv[0 .. np + 64) = 1 / sigma: the engine's row / column scales of a product
// whose operand was split as sigma M
signtri_status fill_inverse(MixedCtx &c, float *inv, float sigma)
{
    ProfScope ps(SIGNTRI_KC_FILL, c.st);
    fill_float_kernel<<<8, 256, 0, c.st>>>(c.np + 64, 1.f / sigma, inv);
    SGT_LAUNCH_CHECK();
    return SIGNTRI_OK;
}

// Blocked-layout rounding splits of the strictly upper part of M (row and
// column forms) for the sweeps.
signtri_status split_full(MixedCtx &c, const double *M, int ldm, __nv_bfloat16 *R, __nv_bfloat16 *C, float sigma)
{
    if (c.S > 8) return SIGNTRI_ERR_BAD_ARG;
    const int nbk = c.np / MB;
    ProfScope ps(SIGNTRI_KC_CONVERT, c.st);
    blocked_split_kernel<<<dim3(nbk, nbk), 256, 0, c.st>>>(c.n, M, ldm, c.S, nbk, R, C, sigma);
    SGT_LAUNCH_CHECK();
    return SIGNTRI_OK;
}

// One low-precision sweep: MODE 0 solves for U (into V = U), MODE 1 for E.
template <int MODE>
signtri_status sweep(MixedCtx &c, const double *T, int ldt, double *V, int ldv, __nv_bfloat16 *Vr,
                     __nv_bfloat16 *Vc, const double *U0, int ldu0)
{
    const int n = c.n, nb = c.sc.nb;
    const size_t leaf_smem = kLeafSmem;
    SGT_CUDA_TRY(cudaFuncSetAttribute(mixed_leaf_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kLeafAlone));
    SGT_CUDA_TRY(cudaFuncSetAttribute(mixed_leaf_kernel<MODE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      cudaSharedmemCarveoutMaxShared));   // two leaves per SM
    {
        // the leaves' per-sign fp32 operators of the diagonal blocks, built
        // from T and the known blocks the same-sign recurrences use (U in
        // mode 0, U0 in mode 1)
        ProfScope ps(MODE == 0 ? SIGNTRI_KC_OFFDIAG_LEAF_F32 : SIGNTRI_KC_CORRECTION, c.st);
        leaf_ops_kernel<<<nb, 256, 0, c.st>>>(n, T, ldt, MODE == 0 ? V : U0, MODE == 0 ? ldv : ldu0, c.OPS, c.DIAG);
        SGT_LAUNCH_CHECK();
    }
    // slices in the blocked layout: every 64 x 64 tile one contiguous 8 KB run
    // fp16 splits carry their scales: the engine scales the products back
    const int h = c.f16 ? 1 : 0;
    const float *iT = c.f16 ? c.invT : nullptr, *iU = c.f16 ? c.invU : nullptr;
    const float *iV = c.f16 ? (MODE == 0 ? c.invU : c.invE) : nullptr;
    const TcSource srcT_r{c.Tr, c.S, c.np, c.np, c.np, iT, 1, h}, srcT_c{c.Tc, c.S, c.np, c.np, c.np, iT, 1, h};
    const TcSource srcV_r{Vr, c.S, c.np, c.np, c.np, iV, 1, h}, srcV_c{Vc, c.S, c.np, c.np, c.np, iV, 1, h};
    const TcSource srcU_r{c.Ur, c.S, c.np, c.np, c.np, iU, 1, h}, srcU_c{c.Uc, c.S, c.np, c.np, c.np, iU, 1, h};
    const TcQuadOut slots{{nullptr, nullptr, nullptr, nullptr}, 0, 0, 0};
    // K-blocks per tensor-core unit: with several unit-weight slice pairs the
    // engine keeps every slice of a K-block resident and accumulates all pairs
    // into one unit, so 2 K-blocks keep each fp32 accumulation short; a single
    // pair takes long units
    const int chunk = c.pairs_split.n > 1 ? 2 : 16;
    // the correction's two launches per anti-diagonal run side by side on
    // their own half-width schedule when a second stream is available; so do
    // the initial sweep's look-ahead pairs
    const bool pair = (MODE == 1) && c.side != nullptr;
    const bool look = (MODE == 0) && c.side != nullptr;
    const Schedule &sc = pair ? c.sc2 : c.sc;
    const DevSchedule &ds = pair ? c.ds2 : c.ds;
    const TcJob *d_jobs = ds.jobs;
    const int *d_coff = ds.cta_off;
    const int2 *d_tslot = ds.tslot;
    const double kb_bytes = (double)c.S * MB * MB * 2;   // one 64-row panel of S bf16 slices, one K-block
    auto fork = [&]() -> signtri_status {
        SGT_CUDA_TRY(cudaEventRecord(c.ev_fork, c.st));
        SGT_CUDA_TRY(cudaStreamWaitEvent(c.side, c.ev_fork, 0));
        return SIGNTRI_OK;
    };
    auto join = [&]() -> signtri_status {
        SGT_CUDA_TRY(cudaEventRecord(c.ev_join, c.side));
        SGT_CUDA_TRY(cudaStreamWaitEvent(c.st, c.ev_join, 0));
        return SIGNTRI_OK;
    };
    for (int d = 1; d < nb; d++) {
        const int ntiles = nb - d;
        const long long sum_kb = (long long)ntiles * (d + 1);
        const int2 *leaf_slots = d_tslot + sc.tile_begin[d];
        const int2 *leaf_slots2 = nullptr;
        signtri_status rs;
        if (MODE == 0 && look && look_lead(d, nb)) {
            // lead: anti-diagonal d in full beside the look-ahead sums of d + 1
            const Schedule &A = c.scA, &B = c.scB;
            const int e = d + 1, ne = nb - e;
            const long long look_kb = (long long)ne * (d - 2);
            ProfScope pg(SIGNTRI_KC_BLOCK_SUMS_TC, c.st, true, false);
            const int cls = SIGNTRI_KC_BLOCK_SUMS_TC | kProfUntimed;
            if ((rs = fork()) != SIGNTRI_OK) return rs;
            rs = tc_blocksums(srcV_r, srcT_r, srcT_c, srcV_c, c.dsA.jobs + A.job_off[d], A.job_off[d + 1] - A.job_off[d],
                              c.pairs_split, c.d_pairs_split, chunk, c.PA, slots, c.d_err, cls | kTcFollows, c.st,
                              tc_flops(c.pairs_split.n, sum_kb, 3), c.dsA.cta_off + A.cta_begin[d], A.nctas[d]);
            if (rs == SIGNTRI_OK)
                rs = tc_blocksums(srcV_r, srcT_r, srcT_c, srcV_c, c.dsB.jobs + B.job_off[e],
                                  B.job_off[e + 1] - B.job_off[e], c.pairs_split, c.d_pairs_split, chunk, c.PB, slots,
                                  c.d_err, cls, c.side, tc_flops(c.pairs_split.n, look_kb, 3),
                                  c.dsB.cta_off + B.cta_begin[e], B.nctas[e]);
            // join even after a failed launch: nothing on the side stream outlives the call
            const signtri_status rj = join();
            if (rs != SIGNTRI_OK) return rs;
            if (rj != SIGNTRI_OK) return rj;
            // the look-ahead reads its row panels from L2: only its column panels are new
            prof_add_bytes(SIGNTRI_KC_BLOCK_SUMS_TC, (4.0 * sum_kb + 2.0 * look_kb) * kb_bytes);
            leaf_slots = c.dsA.tslot + A.tile_begin[d];
        } else if (MODE == 0 && look && look_follow(d, nb)) {
            // follow: the four K-blocks per tile the look-ahead left, then the
            // leaves sum both slot sets
            const Schedule &B = c.scB, &C = c.scC;
            rs = tc_blocksums(srcV_r, srcT_r, srcT_c, srcV_c, c.dsC.jobs + C.job_off[d], C.job_off[d + 1] - C.job_off[d],
                              c.pairs_split, c.d_pairs_split, chunk, c.PA, slots, c.d_err,
                              SIGNTRI_KC_BLOCK_SUMS_TC | kTcFollows, c.st, tc_flops(c.pairs_split.n, 4LL * ntiles, 3), c.dsC.cta_off + C.cta_begin[d],
                              C.nctas[d]);
            if (rs != SIGNTRI_OK) return rs;
            prof_add_bytes(SIGNTRI_KC_BLOCK_SUMS_TC, 4.0 * 4.0 * ntiles * kb_bytes);
            leaf_slots = c.dsC.tslot + C.tile_begin[d];
            leaf_slots2 = c.dsB.tslot + B.tile_begin[d];
        } else {
            const int njobs = sc.job_off[d + 1] - sc.job_off[d];
            const TcJob *jobs = d_jobs + sc.job_off[d];
            const int *coff = d_coff + sc.cta_begin[d];
            const int G = sc.nctas[d];
            if (njobs > 0) {
                if (MODE == 0) {
                    // [U_I.; T_I.] x [T_.J | U_.J]: TL = U T, TR = U U, BR = T U
                    rs = tc_blocksums(srcV_r, srcT_r, srcT_c, srcV_c, jobs, njobs, c.pairs_split, c.d_pairs_split,
                                      chunk, c.PA, slots, c.d_err, SIGNTRI_KC_BLOCK_SUMS_TC | kTcFollows, c.st,
                                      tc_flops(c.pairs_split.n, sum_kb, 3), coff, G);
                    if (rs != SIGNTRI_OK) return rs;
                    prof_add_bytes(SIGNTRI_KC_BLOCK_SUMS_TC, 4.0 * sum_kb * kb_bytes);
                } else {
                    // X^E: [E_I.; T_I.] x [T_.J | E_.J]: TL = E T, BR = T E, and
                    // Y^E: [U0_I.; E_I.] x [E_.J | U0_.J]: TL = U0 E, BR = E U0.  Side by side
                    // (same split, CTA c of each on the same tiles and K-blocks at the
                    // same time) they read the E panels once: six panels for both.
                    ProfScope pg(SIGNTRI_KC_BLOCK_SUMS_TC, c.st, pair, false);
                    const int cls = pair ? (SIGNTRI_KC_BLOCK_SUMS_TC | kProfUntimed) : SIGNTRI_KC_BLOCK_SUMS_TC;
                    cudaStream_t sy = c.st;
                    if (pair) {
                        if ((rs = fork()) != SIGNTRI_OK) return rs;
                        sy = c.side;
                    }
                    rs = tc_blocksums(srcV_r, srcT_r, srcT_c, srcV_c, jobs, njobs, c.pairs_split, c.d_pairs_split,
                                      chunk, c.PA, slots, c.d_err, cls | kTcFollows, c.st, tc_flops(c.pairs_split.n, sum_kb, 2),
                                      coff, G);
                    if (rs == SIGNTRI_OK)
                        rs = tc_blocksums(srcU_r, srcV_r, srcV_c, srcU_c, jobs, njobs, c.pairs_split,
                                          c.d_pairs_split, chunk, c.PB, slots, c.d_err, cls, sy,
                                          tc_flops(c.pairs_split.n, sum_kb, 2), coff, G);
                    const signtri_status rj = pair ? join() : SIGNTRI_OK;   // also after a failed launch
                    if (rs != SIGNTRI_OK) return rs;
                    if (rj != SIGNTRI_OK) return rj;
                    prof_add_bytes(SIGNTRI_KC_BLOCK_SUMS_TC, (pair ? 6.0 : 8.0) * sum_kb * kb_bytes);
                }
            }
        }
        ProfScope ps(MODE == 0 ? SIGNTRI_KC_OFFDIAG_LEAF_F32 : SIGNTRI_KC_CORRECTION, c.st);
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ntiles, MB * MB / kLeafThreads);
        cfg.blockDim = dim3(kLeafThreads);
        cfg.stream = c.st;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        SGT_CUDA_TRY(cudaLaunchKernelEx(&cfg, leaf_seed_kernel<MODE>, n, T, ldt, (const float *)c.DIAG,
                                        (const double *)c.res_c, (const double *)c.res_s, n, d, leaf_slots, leaf_slots2,
                                        (const double *)c.PA, (const double *)c.PB, c.SEED));
        cfg.gridDim = dim3(ntiles);
        cfg.dynamicSmemBytes = ntiles <= 152 ? kLeafAlone : leaf_smem;
        SGT_CUDA_TRY(cudaLaunchKernelEx(&cfg, mixed_leaf_kernel<MODE>, n, V, ldv, (const float *)c.OPS,
                                        (const float *)c.DIAG, d, (const float *)c.SEED, Vr, Vc, c.S, nb,
                                        c.f16 ? (MODE == 0 ? c.sU : c.sE) : 0.f));
        SGT_LAUNCH_CHECK();
    }
    return SIGNTRI_OK;
}

// The gathered layout and the residual job lists, from the diagonal signs
// (one small device-to-host read): per superblock of kSuper indices the
// positives in order, padded to 64, then the negatives; output jobs pair two
// row blocks of one class and superblock with two column blocks of one class
// and superblock (a lone block pairs with the zero block at ng).
signtri_status setup_gathered(MixedCtx &c, const double *T, int ldt)
{
    const int n = c.n;
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, c.st);
        diag_sign_kernel<<<(n + 255) / 256, 256, 0, c.st>>>(n, T, ldt, c.pos);
        SGT_LAUNCH_CHECK();
    }
    std::vector<unsigned char> pos(n);
    SGT_CUDA_TRY(cudaMemcpyAsync(pos.data(), c.pos, n, cudaMemcpyDeviceToHost, c.st));
    SGT_CUDA_TRY(cudaStreamSynchronize(c.st));
    GatheredLayout L;
    build_gathered_layout(n, pos.data(), kSuper, L);
    c.ng = L.ng;
    c.rows_g = L.rows_g;
    if (c.rows_g > gathered_bound(n) + 64) return SIGNTRI_ERR_NO_WORKSPACE;
    c.n_res_same = L.n_same;
    c.n_res_opp = L.n_opp;
    c.res_kb_same = L.kb_same;
    c.res_kb_opp = L.kb_opp;
    if (!L.jobs.empty())
        SGT_CUDA_TRY(cudaMemcpyAsync(c.d_res_jobs, L.jobs.data(), L.jobs.size() * sizeof(TcJob),
                                     cudaMemcpyHostToDevice, c.st));
    SGT_CUDA_TRY(cudaMemcpyAsync(c.gmap, L.gmap.data(), (size_t)n * sizeof(int), cudaMemcpyHostToDevice, c.st));
    SGT_CUDA_TRY(cudaMemcpyAsync(c.sbbase, L.base.data(), L.base.size() * sizeof(int), cudaMemcpyHostToDevice,
                                 c.st));
    SGT_CUDA_TRY(cudaMemcpyAsync(c.ginv, L.ginv.data(), (size_t)c.rows_g * sizeof(int), cudaMemcpyHostToDevice, c.st));
    // the host tables are pageable and local
    SGT_CUDA_TRY(cudaStreamSynchronize(c.st));
    return SIGNTRI_OK;
}

// Exact slices of the strictly upper part of M (T or U) in the gathered layout
// (scales sR, sC computed here unless `scaled`).
signtri_status gathered_slices_of(MixedCtx &c, const double *M, int ldm, __nv_bfloat16 *R, __nv_bfloat16 *C,
                                  float *sR, float *sC, float *gR, float *gC, bool scaled = false)
{
    signtri_status rs;
    if (!scaled &&
        (rs = make_scales_both(c.n, M, ldm, 1, c.np + 64, c.tmpmax, c.tmpmax2, sR, sC, c.st)) != SIGNTRI_OK)
        return rs;
    return make_gathered_slices(c.n, M, ldm, c.ginv, c.gmap, c.sbbase, kSuper, c.ng, kOzakiSlices, kOzakiBits, sR,
                                sC, gR, gC, R, C, c.rows_g, c.rows_g, c.st);
}

// Exact slices of the strictly upper part of M in the original layout (scales
// computed here unless `scaled`).
signtri_status exact_slices_of(MixedCtx &c, const double *M, int ldm, __nv_bfloat16 *R, __nv_bfloat16 *C, float *sR,
                               float *sC, bool scaled = false, bool cols = true)
{
    signtri_status rs;
    if (!scaled &&
        (rs = make_scales_both(c.n, M, ldm, 1, c.np + 64, c.tmpmax, c.tmpmax2, sR, sC, c.st)) != SIGNTRI_OK)
        return rs;
    // the probe and full-residual jobs pair 64-blocks (2i, 2i+1): they never
    // read row slices left of a row's even block or column slices past a
    // column's block pair
    if ((rs = make_row_slices(c.n, c.n, M, ldm, 1, kOzakiSlices, kOzakiBits, sR, R, c.np + 64, c.np, c.st, 1)) !=
        SIGNTRI_OK)
        return rs;
    if (!cols) return SIGNTRI_OK;
    return make_col_slices(c.n, c.n, M, ldm, 1, kOzakiSlices, kOzakiBits, sC, C, c.np + 64, c.np, c.st, 1);
}

signtri_status read_norms(MixedCtx &c)
{
    SGT_CUDA_TRY(cudaMemcpyAsync(c.norms_host, c.norms, 8 * sizeof(double), cudaMemcpyDeviceToHost, c.st));
    SGT_CUDA_TRY(cudaStreamSynchronize(c.st));
    return SIGNTRI_OK;
}

// Needed residual of U (Rc or Rs per entry) into c.R and its norms: three
// tensor-core launches over the gathered layout, each job's four quadrants
// all used -- equal-sign blocks  Y = N_U N_U  (into RA),
// opposite-sign blocks  N_T N_U  (into RA) and  N_U N_T  (into RB) -- then
// the float64 finalize in the original layout.
signtri_status residual_needed(MixedCtx &c, const double *T, int ldt, const double *U, int ldu)
{
    signtri_status rs = gathered_slices_of(c, U, ldu, c.NUr, c.NUc, c.sUr, c.sUc, c.gUr, c.gUc);
    if (rs != SIGNTRI_OK) return rs;
    const int R = c.rows_g, K = c.ng, ld = c.rows_g;
    const TcSource uR{c.NUr, kOzakiSlices, R, K, ld, c.gUr}, uC{c.NUc, kOzakiSlices, R, K, ld, c.gUc};
    const TcSource tR{c.NTgr, kOzakiSlices, R, K, ld, c.gTr}, tC{c.NTgc, kOzakiSlices, R, K, ld, c.gTc};
    const TcQuadOut qa{{c.RA, c.RA, c.RA, c.RA}, c.ng, c.ng, c.ng};
    const TcQuadOut qb{{c.RB, c.RB, c.RB, c.RB}, c.ng, c.ng, c.ng};
    const TcJob *same = c.d_res_jobs, *opp = c.d_res_jobs + c.n_res_same;
    const double fl_same = tc_flops(c.pairs_oz.n, 1, 1) * c.res_kb_same;
    const double fl_opp = tc_flops(c.pairs_oz.n, 1, 1) * c.res_kb_opp;
    rs = tc_blocksums(uR, uR, uC, uC, same, c.n_res_same, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qa, c.d_err,
                      SIGNTRI_KC_RESIDUAL, c.st, fl_same);
    if (rs != SIGNTRI_OK) return rs;
    rs = tc_blocksums(tR, tR, uC, uC, opp, c.n_res_opp, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qa, c.d_err,
                      SIGNTRI_KC_RESIDUAL, c.st, fl_opp);
    if (rs != SIGNTRI_OK) return rs;
    rs = tc_blocksums(uR, uR, tC, tC, opp, c.n_res_opp, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qb, c.d_err,
                      SIGNTRI_KC_RESIDUAL, c.st, fl_opp);
    if (rs != SIGNTRI_OK) return rs;
    SGT_CUDA_TRY(cudaMemsetAsync(c.norms, 0, 8 * sizeof(double), c.st));
    {
        ProfScope ps(SIGNTRI_KC_RESIDUAL_SUM, c.st);
        needed_finalize_kernel<<<c.n, 256, 0, c.st>>>(c.n, T, ldt, U, ldu, c.gmap, c.RA, c.RB, c.ng, c.R, c.norms);
        SGT_LAUNCH_CHECK();
    }
    c.res_c = c.R;
    c.res_s = c.R;
    if ((rs = read_norms(c)) != SIGNTRI_OK) return rs;
    c.nT2 = c.norms_host[2];
    c.nU2 = c.norms_host[3];
    return SIGNTRI_OK;
}

// Both residuals of U over all entries (Rc into RA's memory, Rs into R) and
// their norms.  Original layout; each job pairs row blocks (2i, 2i+1) with
// column blocks (2j, 2j+1), j >= i, over K-blocks [2i, 2j+2) (terms outside
// an output block's own range are structural zeros), and three launches use
// all four quadrants: N_U N_U (into Rs), N_T N_U (into Ptu) and N_U N_T
// (into Put).  A lone last block pairs with the zero block at row np.
signtri_status residual_full(MixedCtx &c, const double *T, int ldt, const double *U, int ldu)
{
    signtri_status rs = exact_slices_of(c, U, ldu, c.NUr, c.NUc, c.sUr, c.sUc);
    if (rs != SIGNTRI_OK) return rs;
    const int R = c.np + 64;
    const TcSource uR{c.NUr, kOzakiSlices, R, c.np, c.np, c.sUr}, uC{c.NUc, kOzakiSlices, R, c.np, c.np, c.sUc};
    const TcSource tR{c.NTr, kOzakiSlices, R, c.np, c.np, c.sTr}, tC{c.NTc, kOzakiSlices, R, c.np, c.np, c.sTc};
    double *Ptu = c.RA, *Put = c.RB, *Rs = c.R;
    const TcQuadOut qs{{Rs, Rs, Rs, Rs}, c.n, c.n, c.n};
    const TcQuadOut qtu{{Ptu, Ptu, Ptu, Ptu}, c.n, c.n, c.n};
    const TcQuadOut qut{{Put, Put, Put, Put}, c.n, c.n, c.n};
    const double fl = tc_flops(c.pairs_oz.n, 1, 1) * c.full_kb;
    rs = tc_blocksums(uR, uR, uC, uC, c.d_full_jobs, c.n_full_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qs, c.d_err,
                      SIGNTRI_KC_RESIDUAL, c.st, fl);
    if (rs != SIGNTRI_OK) return rs;
    rs = tc_blocksums(tR, tR, uC, uC, c.d_full_jobs, c.n_full_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qtu,
                      c.d_err, SIGNTRI_KC_RESIDUAL, c.st, fl);
    if (rs != SIGNTRI_OK) return rs;
    rs = tc_blocksums(uR, uR, tC, tC, c.d_full_jobs, c.n_full_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7, nullptr, qut,
                      c.d_err, SIGNTRI_KC_RESIDUAL, c.st, fl);
    if (rs != SIGNTRI_OK) return rs;
    SGT_CUDA_TRY(cudaMemsetAsync(c.norms, 0, 8 * sizeof(double), c.st));
    {
        ProfScope ps(SIGNTRI_KC_RESIDUAL_SUM, c.st);
        residual_finalize_kernel<<<c.n, 256, 0, c.st>>>(c.n, T, ldt, U, ldu, Ptu, Put, Rs, c.n, c.norms);
        SGT_LAUNCH_CHECK();
    }
    c.res_c = Ptu;
    c.res_s = Rs;
    if ((rs = read_norms(c)) != SIGNTRI_OK) return rs;
    c.nT2 = c.norms_host[2];
    c.nU2 = c.norms_host[3];
    return SIGNTRI_OK;
}

// Probe estimate of both residuals of U over all entries, into
// c.norms_host[0], [1] (squared, scaled to ||R||_F^2), with [2], [3] the
// squared norms of T and of U from the last needed residual (U moved by the
// correction only, ~1e-8 relative: immaterial for the test).
// Products n x n by n x kProbes, jobs = row pairs x two K halves (longest
// first), each half into its own buffer.
signtri_status probe_check(MixedCtx &c, const double *T, int ldt, const double *U, int ldu, unsigned long long seed)
{
    const int n = c.n, np = c.np;
    signtri_status rs;
    if ((rs = make_scales(n, n, U, ldu, 1, true, np + 64, c.tmpmax, c.sUr, c.st)) != SIGNTRI_OK) return rs;
    if ((rs = make_row_slices(n, n, U, ldu, 1, kOzakiSlices, kOzakiBits, c.sUr, c.NUr, np + 64, np, c.st, 1)) !=
        SIGNTRI_OK)
        return rs;
    const size_t blk = (size_t)n * kProbes;
    double *P[10];
    for (int i = 0; i < 10; i++) P[i] = c.Pp + i * blk;
    {
        ProfScope ps(SIGNTRI_KC_RESIDUAL_SUM, c.st);
        probe_kernel<<<dim3(std::min((np + 255) / 256, 64), kProbes), 256, 0, c.st>>>(n, np, seed, c.Z, c.Zc,
                                                                                      c.zscale);
        SGT_LAUNCH_CHECK();
    }
    const int R = np + 64;
    const TcSource uR{c.NUr, kOzakiSlices, R, np, np, c.sUr}, tR{c.NTr, kOzakiSlices, R, np, np, c.sTr};
    const TcSource zC{c.Zc, 1, kProbes, np, np, c.zscale};
    const TcSource w1C{c.W1c, kOzakiSlices, kProbes, np, np, c.w1scale}, w2C{c.W2c, kOzakiSlices, kProbes, np, np,
                                                                              c.w2scale};
    auto out = [&](double *m) { return TcQuadOut{{m, m, m, m}, n, n, kProbes, blk}; };
    const double flz = tc_flops(c.pairs_z.n, 1, 1) * c.probe_kb, flw = tc_flops(c.pairs_oz.n, 1, 1) * c.probe_kb;
    // W1 = U Z, W2 = T Z (Z: one slice, pairs (s, 0))
    if ((rs = tc_blocksums(uR, uR, zC, zC, c.d_probe_jobs, c.n_probe_jobs, c.pairs_z, c.d_pairs_z, kExactChunkKb7,
                           nullptr, out(P[0]), c.d_err, SIGNTRI_KC_RESIDUAL, c.st, flz)) != SIGNTRI_OK)
        return rs;
    if ((rs = tc_blocksums(tR, tR, zC, zC, c.d_probe_jobs, c.n_probe_jobs, c.pairs_z, c.d_pairs_z, kExactChunkKb7,
                           nullptr, out(P[2]), c.d_err, SIGNTRI_KC_RESIDUAL, c.st, flz)) != SIGNTRI_OK)
        return rs;
    {
        ProfScope ps(SIGNTRI_KC_RESIDUAL_SUM, c.st);
        const dim3 g(std::min((n + 255) / 256, 64), kProbes);
        probe_combine_kernel<<<g, 256, 0, c.st>>>(n, P[0], P[1], U, ldu, c.Z, c.W1);
        SGT_LAUNCH_CHECK();
        probe_combine_kernel<<<g, 256, 0, c.st>>>(n, P[2], P[3], T, ldt, c.Z, c.W2);
        SGT_LAUNCH_CHECK();
    }
    if ((rs = make_scales(n, kProbes, c.W1, n, 0, false, kProbes, c.tmpmax, c.w1scale, c.st)) != SIGNTRI_OK)
        return rs;
    if ((rs = make_scales(n, kProbes, c.W2, n, 0, false, kProbes, c.tmpmax, c.w2scale, c.st)) != SIGNTRI_OK)
        return rs;
    if ((rs = make_col_slices(n, kProbes, c.W1, n, 0, kOzakiSlices, kOzakiBits, c.w1scale, c.W1c, kProbes, np,
                              c.st)) != SIGNTRI_OK)
        return rs;
    if ((rs = make_col_slices(n, kProbes, c.W2, n, 0, kOzakiSlices, kOzakiBits, c.w2scale, c.W2c, kProbes, np,
                              c.st)) != SIGNTRI_OK)
        return rs;
    // N_T W1, N_U W2, N_U W1
    if ((rs = tc_blocksums(tR, tR, w1C, w1C, c.d_probe_jobs, c.n_probe_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7,
                           nullptr, out(P[4]), c.d_err, SIGNTRI_KC_RESIDUAL, c.st, flw)) != SIGNTRI_OK)
        return rs;
    if ((rs = tc_blocksums(uR, uR, w2C, w2C, c.d_probe_jobs, c.n_probe_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7,
                           nullptr, out(P[6]), c.d_err, SIGNTRI_KC_RESIDUAL, c.st, flw)) != SIGNTRI_OK)
        return rs;
    if ((rs = tc_blocksums(uR, uR, w1C, w1C, c.d_probe_jobs, c.n_probe_jobs, c.pairs_oz, c.d_pairs_oz, kExactChunkKb7,
                           nullptr, out(P[8]), c.d_err, SIGNTRI_KC_RESIDUAL, c.st, flw)) != SIGNTRI_OK)
        return rs;
    SGT_CUDA_TRY(cudaMemsetAsync(c.norms, 0, 2 * sizeof(double), c.st));
    {
        ProfScope ps(SIGNTRI_KC_RESIDUAL_SUM, c.st);
        probe_residual_kernel<<<dim3(std::min((n + 255) / 256, 64), kProbes), 256, 0, c.st>>>(
            n, T, ldt, U, ldu, c.Z, c.W1, c.W2, P[4], P[5], P[6], P[7], P[8], P[9], c.norms);
        SGT_LAUNCH_CHECK();
    }
    SGT_CUDA_TRY(cudaMemcpyAsync(c.norms_host, c.norms, 2 * sizeof(double), cudaMemcpyDeviceToHost, c.st));
    SGT_CUDA_TRY(cudaStreamSynchronize(c.st));
    c.norms_host[0] /= kProbes;
    c.norms_host[1] /= kProbes;
    c.norms_host[2] = c.nT2;
    c.norms_host[3] = c.nU2;
    return SIGNTRI_OK;
}

}  // namespace

// The correction's second stream and its fork / join events, one set per
// device, created on first use (the library's calls are serialized).
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};
SideStream g_side[64];

signtri_status side_stream(MixedCtx &c)
{
    c.side = nullptr;
    int dev = 0;
    SGT_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return SIGNTRI_OK;
    SideStream &g = g_side[dev];
    // a piece is stored only once created, so a call after a failed attempt
    // creates what is still missing; the side stream is used only with both
    // of its events
    if (!g.s) {
        cudaStream_t s = nullptr;
        SGT_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        g.s = s;
    }
    if (!g.fork) {
        cudaEvent_t e = nullptr;
        SGT_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        g.fork = e;
    }
    if (!g.join) {
        cudaEvent_t e = nullptr;
        SGT_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        g.join = e;
    }
    c.side = g.s;
    c.ev_fork = g.fork;
    c.ev_join = g.join;
    return SIGNTRI_OK;
}

size_t mixed_workspace_bytes(int n, int S) { return n > 0 ? bytes_for(n, S) + (64 << 10) : 0; }

signtri_status mixed_run(int n, const double *T, int ldt, double *U, int ldu, int S, const MixedParams &prm,
                         MixedReport &rep, Arena &ws, int *d_err, double *norms_host, cudaStream_t st)
{
    MixedCtx c{};
    c.n = n;
    c.np = pad64(n);
    c.f16 = S < 0;   // a negative S asks for the fp16 split of -S terms
    if (S < 0) S = -S;
    c.S = S;
    c.st = st;
    c.d_err = d_err;
    build_schedule(n, kSweepCtas, c.sc);
    build_schedule(n, kSweepCtas / 2, c.sc2);
    build_look_schedules(n, kSweepCtas / 2, c.scA, c.scB, c.scC);
    const int nb = c.sc.nb;
    const size_t np = c.np;
    const size_t split_elems = (size_t)S * np * np;
    const size_t ngr = (size_t)gathered_bound(n) + 64, oz_elems = (size_t)kOzakiSlices * ngr * ngr;
    c.Tr = take<__nv_bfloat16>(ws, split_elems); c.Tc = take<__nv_bfloat16>(ws, split_elems);
    c.Ur = take<__nv_bfloat16>(ws, split_elems); c.Uc = take<__nv_bfloat16>(ws, split_elems);
    c.Er = take<__nv_bfloat16>(ws, split_elems); c.Ec = take<__nv_bfloat16>(ws, split_elems);
    const size_t oz_orig = (size_t)kOzakiSlices * (np + 64) * np;
    c.NTgr = take<__nv_bfloat16>(ws, oz_elems); c.NTgc = take<__nv_bfloat16>(ws, oz_elems);
    c.NTr = take<__nv_bfloat16>(ws, oz_orig); c.NTc = take<__nv_bfloat16>(ws, oz_orig);
    c.NUr = take<__nv_bfloat16>(ws, oz_elems); c.NUc = take<__nv_bfloat16>(ws, oz_elems);
    // original-index scales and their max buffer cover the zero block too
    c.sTr = take<float>(ws, np + 64); c.sTc = take<float>(ws, np + 64);
    c.sUr = take<float>(ws, np + 64); c.sUc = take<float>(ws, np + 64);
    c.gTr = take<float>(ws, ngr); c.gTc = take<float>(ws, ngr); c.gUr = take<float>(ws, ngr); c.gUc = take<float>(ws, ngr);
    c.gmap = take<int>(ws, ngr); c.ginv = take<int>(ws, ngr); c.pos = take<unsigned char>(ws, np);
    c.sbbase = take<int>(ws, (size_t)(n + kSuper - 1) / kSuper + 1);
    c.tmpmax = take<unsigned long long>(ws, np + 64);
    c.tmpmax2 = take<unsigned long long>(ws, np + 64);
    const size_t maxjobs = (size_t)std::max({c.sc.max_jobs, c.scA.max_jobs, c.scB.max_jobs, c.scC.max_jobs, 1});
    c.PA = take<double>(ws, maxjobs * 16384); c.PB = take<double>(ws, maxjobs * 16384);
    c.E = take<double>(ws, (size_t)n * n); c.R = take<double>(ws, (size_t)n * n);
    c.OPS = take<float>(ws, (size_t)4 * nb * kMicro * kMicro * kTri);
    c.SEED = take<float>(ws, (size_t)nb * MB * MB);
    c.DIAG = take<float>(ws, (size_t)nb * MB);
    c.invT = take<float>(ws, np + 64); c.invU = take<float>(ws, np + 64); c.invE = take<float>(ws, np + 64);
    c.amax = take<unsigned>(ws, 16);
    if (!c.invT || !c.invU || !c.invE || !c.amax) return SIGNTRI_ERR_NO_WORKSPACE;
    const int nbp = (nb + 1) / 2;
    c.n_full_jobs = nbp * (nbp + 1) / 2;
    c.d_full_jobs = take<TcJob>(ws, (size_t)c.n_full_jobs);
    c.RA = take<double>(ws, ngr * ngr); c.RB = take<double>(ws, ngr * ngr);
    c.norms = take<double>(ws, 8);
    const size_t pairs_max = ngr / 128 + 2 * (size_t)((n + kSuper - 1) / kSuper) + 2;
    c.d_res_jobs = take<TcJob>(ws, pairs_max * pairs_max);
    for (auto pr : {std::make_pair(&c.sc, &c.ds), std::make_pair(&c.sc2, &c.ds2), std::make_pair(&c.scA, &c.dsA),
                    std::make_pair(&c.scB, &c.dsB), std::make_pair(&c.scC, &c.dsC)}) {
        pr.second->jobs = take<TcJob>(ws, std::max<size_t>(pr.first->jobs.size(), 1));
        pr.second->cta_off = take<int>(ws, std::max<size_t>(pr.first->cta_off.size(), 1));
        pr.second->tslot = take<int2>(ws, std::max<size_t>(pr.first->tslot.size(), 1));
        if (!pr.second->jobs || !pr.second->cta_off || !pr.second->tslot) return SIGNTRI_ERR_NO_WORKSPACE;
    }
    c.d_pairs_split = take<TcPairs>(ws, 1);
    c.d_pairs_oz = take<TcPairs>(ws, 1);
    c.d_pairs_z = take<TcPairs>(ws, 1);
    {
        const size_t blk = (size_t)n * kProbes;
        c.Z = take<double>(ws, blk); c.W1 = take<double>(ws, blk); c.W2 = take<double>(ws, blk);
        c.Pp = take<double>(ws, 10 * blk);
        c.Zc = take<__nv_bfloat16>(ws, (size_t)kProbes * np);
        c.W1c = take<__nv_bfloat16>(ws, (size_t)kOzakiSlices * kProbes * np);
        c.W2c = take<__nv_bfloat16>(ws, (size_t)kOzakiSlices * kProbes * np);
        c.zscale = take<float>(ws, kProbes); c.w1scale = take<float>(ws, kProbes); c.w2scale = take<float>(ws, kProbes);
        c.d_probe_jobs = take<TcJob>(ws, (size_t)2 * nbp + 2);
        if (!c.Z || !c.W1 || !c.W2 || !c.Pp || !c.Zc || !c.W1c || !c.W2c || !c.zscale || !c.w1scale || !c.w2scale ||
            !c.d_probe_jobs || !c.d_pairs_z)
            return SIGNTRI_ERR_NO_WORKSPACE;
    }
    c.norms_host = norms_host;
    if (!c.Tr || !c.Tc || !c.Ur || !c.Uc || !c.Er || !c.Ec || !c.NTgr || !c.NTgc || !c.NTr || !c.NTc || !c.NUr ||
        !c.NUc || !c.d_full_jobs || !c.sTr ||
        !c.sTc || !c.sUr || !c.sUc || !c.gTr || !c.gTc || !c.gUr || !c.gUc || !c.gmap || !c.ginv || !c.pos ||
        !c.tmpmax || !c.tmpmax2 || !c.PA || !c.PB || !c.E || !c.R || !c.RA || !c.RB || !c.norms || !c.d_res_jobs ||
        !c.d_pairs_split || !c.d_pairs_oz || !c.OPS || !c.SEED || !c.DIAG || !c.sbbase)
        return SIGNTRI_ERR_NO_WORKSPACE;
    c.pairs_split = split_pairs(S);
    c.pairs_oz = ozaki_pairs_impl(kOzakiSlices, kOzakiBits);
    // probe products with Z (one slice): pairs (s, 0)
    std::memset(&c.pairs_z, 0, sizeof(c.pairs_z));
    for (int sl = 0; sl < kOzakiSlices; sl++) {
        c.pairs_z.s[sl] = sl;
        c.pairs_z.t[sl] = 0;
        c.pairs_z.w[sl] = ldexpf(1.0f, -kOzakiBits * (sl + 2));
    }
    c.pairs_z.n = kOzakiSlices;
    SGT_CUDA_TRY(cudaMemcpyAsync(c.d_pairs_z, &c.pairs_z, sizeof(TcPairs), cudaMemcpyHostToDevice, st));
    {
        // probe jobs: row pairs (2I, 2I+1) x K halves of [2I, nb), longest first
        std::vector<TcJob> pj;
        double kb = 0.0;
        for (int I = 0; I < nbp; I++)
            for (int h = 0; h < 2; h++) {
                const int k0 = 2 * I, mid = (k0 + nb + 1) / 2;
                TcJob j;
                j.rt = 2 * I * MB; j.rb = 2 * I + 1 < nb ? (2 * I + 1) * MB : (int)np;
                j.cl = 0; j.cr = 64;
                j.kb0 = h ? mid : k0; j.kb1 = h ? nb : mid; j.slot = h; j.pad = 0;
                kb += (double)((j.rb != (int)np) + 1) * 2 * std::max(0, j.kb1 - j.kb0);
                pj.push_back(j);
            }
        std::stable_sort(pj.begin(), pj.end(),
                         [](const TcJob &x, const TcJob &y) { return x.kb1 - x.kb0 > y.kb1 - y.kb0; });
        c.n_probe_jobs = (int)pj.size();
        c.probe_kb = kb;
        SGT_CUDA_TRY(cudaMemcpyAsync(c.d_probe_jobs, pj.data(), pj.size() * sizeof(TcJob), cudaMemcpyHostToDevice,
                                     st));
        SGT_CUDA_TRY(cudaStreamSynchronize(st));
    }
    for (auto pr : {std::make_pair(&c.sc, &c.ds), std::make_pair(&c.sc2, &c.ds2), std::make_pair(&c.scA, &c.dsA),
                    std::make_pair(&c.scB, &c.dsB), std::make_pair(&c.scC, &c.dsC)}) {
        if (!pr.first->jobs.empty())
            SGT_CUDA_TRY(cudaMemcpyAsync(pr.second->jobs, pr.first->jobs.data(), pr.first->jobs.size() * sizeof(TcJob),
                                         cudaMemcpyHostToDevice, st));
        if (!pr.first->cta_off.empty())
            SGT_CUDA_TRY(cudaMemcpyAsync(pr.second->cta_off, pr.first->cta_off.data(),
                                         pr.first->cta_off.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        if (!pr.first->tslot.empty())
            SGT_CUDA_TRY(cudaMemcpyAsync(pr.second->tslot, pr.first->tslot.data(),
                                         pr.first->tslot.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
    }
    {
        const signtri_status ss = side_stream(c);
        if (ss != SIGNTRI_OK) return ss;
    }
    SGT_CUDA_TRY(cudaMemcpyAsync(c.d_pairs_split, &c.pairs_split, sizeof(TcPairs), cudaMemcpyHostToDevice, st));
    SGT_CUDA_TRY(cudaMemcpyAsync(c.d_pairs_oz, &c.pairs_oz, sizeof(TcPairs), cudaMemcpyHostToDevice, st));
    {
        // full-residual jobs in 8 x 8 groups of block pairs: the CTAs resident
        // together share row and column panels in L2
        std::vector<TcJob> rj;
        rj.reserve(c.n_full_jobs);
        double kb = 0.0;
        constexpr int G = 8;
        const int zero = (int)np;   // the zero block
        for (int I0 = 0; I0 < nbp; I0 += G)
            for (int J0 = I0 / G * G; J0 < nbp; J0 += G)
                for (int I = I0; I < std::min(I0 + G, nbp); I++)
                    for (int J = std::max(J0, I); J < std::min(J0 + G, nbp); J++) {
                        TcJob j;
                        j.rt = 2 * I * MB; j.rb = 2 * I + 1 < nb ? (2 * I + 1) * MB : zero;
                        j.cl = 2 * J * MB; j.cr = 2 * J + 1 < nb ? (2 * J + 1) * MB : zero;
                        j.kb0 = 2 * I; j.kb1 = std::min(2 * J + 2, nb); j.slot = 0; j.pad = 0;
                        kb += (double)((j.rb != zero) + 1) * ((j.cr != zero) + 1) * (j.kb1 - j.kb0);
                        rj.push_back(j);
                    }
        c.full_kb = kb;
        SGT_CUDA_TRY(cudaMemcpyAsync(c.d_full_jobs, rj.data(), rj.size() * sizeof(TcJob), cudaMemcpyHostToDevice,
                                     st));
        SGT_CUDA_TRY(cudaStreamSynchronize(st));
    }
    signtri_status rs0 = setup_gathered(c, T, ldt);
    if (rs0 != SIGNTRI_OK) return rs0;
    // slices start from zero (padding and the not-yet-computed blocks)
    SGT_CUDA_TRY(cudaMemsetAsync(c.Ur, 0, split_elems * 2, st));
    SGT_CUDA_TRY(cudaMemsetAsync(c.Uc, 0, split_elems * 2, st));
    SGT_CUDA_TRY(cudaMemsetAsync(c.Er, 0, split_elems * 2, st));
    SGT_CUDA_TRY(cudaMemsetAsync(c.Ec, 0, split_elems * 2, st));
    signtri_status rs;
    if ((rs = gathered_slices_of(c, T, ldt, c.NTgr, c.NTgc, c.sTr, c.sTc, c.gTr, c.gTc)) != SIGNTRI_OK) return rs;
    if (c.f16) {
        // T's largest strictly upper entry (from the row maxima the exact
        // slices' scales were just taken from) to 2^13 .. 2^14 (fp16 stops
        // at 65504)
        float m = 0.f;
        if ((rs = row_maxima_max(c, m)) != SIGNTRI_OK) return rs;
        c.sT = m > 0.f ? pow2_scale(m, 13) : 1.f;
        if ((rs = fill_inverse(c, c.invT, c.sT)) != SIGNTRI_OK) return rs;
    }
    if ((rs = split_full(c, T, ldt, c.Tr, c.Tc, c.f16 ? c.sT : 0.f)) != SIGNTRI_OK) return rs;
    // T's scales serve both layouts; the probe check reads only T's row
    // slices, the full residual also its column slices
    if ((rs = exact_slices_of(c, T, ldt, c.NTr, c.NTc, c.sTr, c.sTc, true, prm.verify_full != 0)) != SIGNTRI_OK)
        return rs;

    // 1. low-precision solve: diagonal blocks in float64, the rest by sweep
    // the diagonal 64 x 64 blocks, by leaves of 16 (block anti-diagonals 0 .. 3,
    // what they hold beyond the blocks to be overwritten)
    {
        const size_t mark = ws.used;
        if ((rs = ph_fp64_near_run(n, T, ldt, U, ldu, MB / 16 - 1, ws, st)) != SIGNTRI_OK) return rs;
        ws.used = mark;
    }
    if (c.f16) {
        // U's scale from its diagonal blocks, largest entry to 2^12 .. 2^13:
        // room for off-diagonal entries up to 8x larger
        float m = 0.f;
        if ((rs = diag_blocks_absmax(c, U, ldu, m)) != SIGNTRI_OK) return rs;
        c.sU = m > 0.f ? pow2_scale(m, 12) : c.sT;
        if ((rs = fill_inverse(c, c.invU, c.sU)) != SIGNTRI_OK) return rs;
    }
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, st);
        diag_slices_kernel<<<nb, 256, 0, st>>>(n, U, ldu, c.Ur, c.Uc, S, nb, c.f16 ? c.sU : 0.f);
        SGT_LAUNCH_CHECK();
    }
    if ((rs = sweep<0>(c, T, ldt, U, ldu, c.Ur, c.Uc, nullptr, 0)) != SIGNTRI_OK) return rs;

    // 2. refinement.  Corrections are driven by the needed residuals (Rc at
    // opposite-sign entries, Rs at equal-sign ones); acceptance rests on both
    // residuals over all entries: the full products (verify_full) or their
    // probe estimate.
    double prev = 1e300;
    rep.steps = 0;
    rep.fallback = 0;
    auto verify = [&](int step) -> signtri_status {
        return prm.verify_full ? residual_full(c, T, ldt, U, ldu)
                               : probe_check(c, T, ldt, U, ldu, 0x5eedull * 1315423911ull + (unsigned long long)step);
    };
    auto worst_of = [&]() {
        const double *h = c.norms_host;
        const double nT = std::sqrt(h[2]), nU = std::sqrt(h[3]);
        rep.resid_commute = std::sqrt(h[0]) / (nT * nU);
        rep.resid_involution = std::sqrt(h[1]) / (nU * nU);
        return std::max(rep.resid_commute, rep.resid_involution);
    };
    for (int step = 0;; step++) {
        bool verified = step > 0;
        if ((rs = verified ? verify(step) : residual_needed(c, T, ldt, U, ldu)) != SIGNTRI_OK) return rs;
        double worst = worst_of();
        if (!verified && worst <= prm.tol) {
            // needed residuals already small: check both equations
            if ((rs = verify(step)) != SIGNTRI_OK) return rs;
            verified = true;
            worst = worst_of();
        }
        if (step == 0) rep.resid0 = worst;
        if (!(worst == worst)) { rep.fallback = 1; return SIGNTRI_OK; }   // NaN
        if (verified && worst <= prm.tol) return SIGNTRI_OK;
        if (step >= prm.max_steps || (step > 0 && worst > prev / prm.min_contraction)) {
            rep.fallback = 1;
            return SIGNTRI_OK;
        }
        prev = worst;
        // the correction reads Rc / Rs entrywise: the full residual left them;
        // after a probe test (or a confirmed step 0) form the needed ones
        if (verified && !prm.verify_full && (rs = residual_needed(c, T, ldt, U, ldu)) != SIGNTRI_OK) return rs;
        // E: zero, diagonal blocks in float64, off-diagonal blocks by sweep
        {
            ProfScope ps(SIGNTRI_KC_FILL, st);
            zero_kernel<<<1024, 256, 0, st>>>((size_t)n * n, c.E);
            SGT_LAUNCH_CHECK();
        }
        SGT_CUDA_TRY(cudaMemsetAsync(c.Er, 0, split_elems * 2, st));
        SGT_CUDA_TRY(cudaMemsetAsync(c.Ec, 0, split_elems * 2, st));
        // U0's slices: after the initial sweep they are already in Ur / Uc
        // (off-diagonal blocks from the leaves, diagonal blocks from
        // diag_slices_kernel); after a correction U has moved
        if (step > 0 && (rs = split_full(c, U, ldu, c.Ur, c.Uc, c.f16 ? c.sU : 0.f)) != SIGNTRI_OK) return rs;
        {
            const size_t dsm = 3 * (size_t)MB * (MB + 1) * sizeof(double);
            SGT_CUDA_TRY(cudaFuncSetAttribute(corr_diag_leaf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)dsm));
            ProfScope ps(SIGNTRI_KC_CORRECTION, st);
            corr_diag_leaf_kernel<<<nb, kLeafThreads, dsm, st>>>(n, T, ldt, U, ldu, c.res_c, c.res_s, n, c.E, n);
            SGT_LAUNCH_CHECK();
        }
        if (c.f16) {
            // the correction's scale from its first-order terms, Rc_ij /
            // (t_ii - t_jj) or Rs_ij / 2 (its diagonal blocks are no guide,
            // U0's being float64-exact), largest to 2^10 .. 2^11: room for
            // entries of E up to 32x larger
            float m = 0.f;
            SGT_CUDA_TRY(cudaMemsetAsync(c.amax, 0, sizeof(unsigned), st));
            {
                ProfScope ps(SIGNTRI_KC_CONVERT, st);
                // c.DIAG: t_ii in fp32, from the initial sweep (same T)
                corr_magnitude_kernel<<<1216, 256, 0, st>>>(n, c.DIAG, c.res_c, c.res_s, n, c.amax);
                SGT_LAUNCH_CHECK();
            }
            if ((rs = read_amax(c, m)) != SIGNTRI_OK) return rs;
            c.sE = m > 0.f ? pow2_scale(m, 10) : c.sU;
            if ((rs = fill_inverse(c, c.invE, c.sE)) != SIGNTRI_OK) return rs;
        }
        {
            ProfScope ps(SIGNTRI_KC_CONVERT, st);
            diag_slices_kernel<<<nb, 256, 0, st>>>(n, c.E, n, c.Er, c.Ec, S, nb, c.f16 ? c.sE : 0.f);
            SGT_LAUNCH_CHECK();
        }
        if ((rs = sweep<1>(c, T, ldt, c.E, n, c.Er, c.Ec, U, ldu)) != SIGNTRI_OK) return rs;
        {
            ProfScope ps(SIGNTRI_KC_CORRECTION, st);
            apply_correction_kernel<<<n, 256, 0, st>>>(n, U, ldu, c.E, n, c.norms);
            SGT_LAUNCH_CHECK();
        }
        rep.steps = step + 1;
    }
}

}  // namespace signtri
