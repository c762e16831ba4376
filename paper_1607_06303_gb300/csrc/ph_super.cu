// ph_super.cu -- large float64 Parlett-Higham: superblocks of 128, their block
// sums as residue products on the tensor cores.
//
// The equations of ph_level.cuh with the off-diagonal part cut into
// superblocks (A, B) of 128 x 128, solved by superblock anti-diagonal
// D = B - A.  For each D:
//   1. rns::gemm: UT = U_A. T_.B and TU = T_A. U_.B over the superblocks
//      K = A .. B whose entries are known (the strictly upper parts of the
//      diagonal superblocks among them), and UU = U_A. U_.B over A < K < B, as
//      residues (rns.cu: rounding the operands to 53 or more bits of their
//      row's or column's largest is the only error);
//   2. 15 launches of wave_kernel: the superblocks' 16 x 16 blocks by block
//      anti-diagonal, from the bottom-left corner, in float64: per entry the
//      residue sum its signs ask for, UT - TU or - UU, and the terms that hold
//      entries of the superblock itself,
//        - sum_{k > p, k in A} m_pk v_kq + sum_{k < q, k in B} v_pk n_kq;
//   3. the new superblocks of U join the row and column forms.
// The float64 work that stays on the SMs' float64 pipes falls from n^3 / 3 or
// more to about 64 n^2 multiply-adds and the leaves'.
//
// Scales: T's rows and columns by their largest entry.  U's are not known in
// advance: a row starts with two bits of headroom over its first superblock
// and is converted anew, with two bits again, when a later superblock outgrows
// them.  Data that does not suit one scale per row (most of a superblock's
// entries below 2^-24 of their row's or column's largest) or is not finite
// sets a flag, and the caller runs the plain float64 path instead.
#include <algorithm>
#include <climits>

#include "internal.cuh"
#include "ph_level.cuh"
#include "rns.cuh"

namespace signtri {
namespace sup {

using lvl::BLK;
using lvl::LB;
using lvl::LD;
using lvl::LT;

constexpr int SP = rns::kPanel;   // superblock edge
constexpr int SB = SP / LB;       // blocks of 16 per edge
constexpr int kThreads = 256;
constexpr int kNoExp = INT_MIN / 2;
constexpr int kHeadroom = 2;
constexpr int kMinExp = -900;     // keeps 2^(bits - exp) a normal number
constexpr int kWideBits = 24;

namespace {

// ---- scales and residues ----------------------------------------------------

__device__ __forceinline__ int exponent_above(double x)   // |x| < 2^result
{
    return ((__double2hiint(x) >> 20) & 0x7ff) - 1022;
}

// A matrix read as rows x cols, or only its strictly upper part.
struct Mat {
    const double *M;
    int ld, rows, cols;
    bool strict;
    __device__ __forceinline__ double operator()(int i, int j) const
    {
        return i < rows && j < cols && (!strict || i < j) ? SGT_AT(M, ld, i, j) : 0.0;
    }
};

// Largest exponents of the rows and columns of superblock (A, B), in shared
// memory; returns with the block synchronised.
__device__ __forceinline__ void superblock_exps(const Mat &M, int A, int B, int *rmax, int *cmax)
{
    if (threadIdx.x < SP) rmax[threadIdx.x] = cmax[threadIdx.x] = kNoExp;
    __syncthreads();
    const int i = threadIdx.x % SP, h = threadIdx.x / SP;
    int rm = kNoExp;
    for (int j = h; j < SP; j += kThreads / SP) {
        const double x = M(A * SP + i, B * SP + j);
        const int e = x != 0.0 ? exponent_above(x) : kNoExp;
        rm = max(rm, e);
        const int cm = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0) atomicMax(&cmax[j], cm);
    }
    atomicMax(&rmax[i], rm);
    __syncthreads();
}

// The exponents of M's superblocks (the diagonal ones only, or all).
__global__ void __launch_bounds__(kThreads)
fixed_exps_kernel(const __grid_constant__ Mat M, bool diagonal_only, int *__restrict__ rexp,
                  int *__restrict__ cexp, int *__restrict__ flags)
{
    const int A = blockIdx.x, B = diagonal_only ? A : blockIdx.y;
    if (A > B) return;
    __shared__ int rmax[SP], cmax[SP];
    superblock_exps(M, A, B, rmax, cmax);
    if (threadIdx.x < SP) {
        if (rexp) atomicMax(&rexp[A * SP + threadIdx.x], rmax[threadIdx.x]);
        if (cexp) atomicMax(&cexp[B * SP + threadIdx.x], cmax[threadIdx.x]);
        if (rmax[threadIdx.x] > 1024) atomicOr(flags, 1);
    }
}

// The exponents of the new superblocks (a0 + t, b0 + t) that outgrow their row or
// column, and which panels to convert anew.  rnew, cnew: the new superblocks'
// largest, gathered by the leaves that solved them and reset here.
__global__ void __launch_bounds__(SP)
grow_exps_kernel(int a0, int b0, int *__restrict__ rnew, int *__restrict__ cnew, int *__restrict__ rexp, int *__restrict__ cexp,
                 int *__restrict__ rgrown, int *__restrict__ cgrown, int *__restrict__ flags)
{
    const int A = a0 + blockIdx.x, B = b0 + blockIdx.x;
    const int r = A * SP + threadIdx.x, c = B * SP + threadIdx.x;
    const int er = rnew[r], ec = cnew[c];
    rnew[r] = kNoExp;
    cnew[c] = kNoExp;
    if (er > 1024) atomicOr(flags, 1);
    const bool rg = er > rexp[r], cg = ec > cexp[c];
    if (rg) rexp[r] = er + kHeadroom;
    if (cg) cexp[c] = ec + kHeadroom;
    const int ra = __syncthreads_or(rg), ca = __syncthreads_or(cg);
    if (threadIdx.x == 0) { rgrown[A] = ra; cgrown[B] = ca; }
}

struct ConvConst {
    float c[rns::kMods][5];   // 2^(14 d) mod m, within m / 2 of 0
    float m[rns::kMods], rm[rns::kMods];
};
constexpr ConvConst make_conv_const()
{
    ConvConst k{};
    for (int i = 0; i < rns::kMods; i++) {
        const int m = rns::kModulus[i];
        k.m[i] = (float)m;
        k.rm[i] = 1.f / (float)m;
        int p = 1 % m;
        for (int d = 0; d < 5; d++) {
            k.c[i][d] = (float)(p > m / 2 ? p - m : p);
            p = p * (16384 % m) % m;
        }
    }
    return k;
}
__constant__ ConvConst c_conv = make_conv_const();

// Residues of one 128 x 128 superblock of M into panel P's K-blocks 2 K, 2 K + 1.  rows: P holds rows, K counts columns; else P
// holds columns and K counts rows.  Part `part` of kConvParts of it.
constexpr int kConvParts = SP * SP / 8 / kThreads;
__device__ __forceinline__ void convert_superblock(const Mat &M, int bits, bool rows,
                                                   int P, int K, int part, const int *__restrict__ exps,
                                                   __nv_bfloat16 *__restrict__ tiles, int nkb, int *flags)
{
    int small = 0, some = 0;
    const int it = part * kThreads + threadIdx.x;
    {
        // line `i` of the panel, 8 entries along K from 8 ch; the threads of a
        // warp run along the matrix's columns, which are contiguous
        const int i = rows ? it % SP : it / (SP / 8), ch = rows ? it / SP : it % (SP / 8);
        const int g = P * SP + i;
        const int e = max(exps[g], kMinExp);
        const double sc = __hiloint2double((1023 + bits - e) << 20, 0);
        float dig[8][5];
#pragma unroll
        for (int t = 0; t < 8; t++) {
            const int k = K * SP + ch * 8 + t;
            const double x = rows ? M(g, k) : M(k, g);
            if (x != 0.0) {
                some++;
                small += exponent_above(x) < e - kWideBits;
            }
            // bits <= 56: five balanced digits of 14 bits
            long long v = __double2ll_rn(x * sc);
#pragma unroll
            for (int d = 0; d < 5; d++) {
                const int r = ((int)(v & 16383) ^ 8192) - 8192;
                dig[t][d] = (float)r;
                v = (v - r) >> 14;
            }
        }
        const int kb = 2 * K + ch / 8, c8 = ch & 7;
        __nv_bfloat16 *dst = tiles + ((size_t)P * rns::kMods * nkb + kb) * rns::kTileElems + i * 64 + ((c8 ^ (i & 7)) * 8);
        for (int m = 0; m < rns::kMods; m++) {
            const float mm = c_conv.m[m], rm = c_conv.rm[m];
            float y[8];
#pragma unroll
            for (int t = 0; t < 8; t++) {
                float s = dig[t][0];
#pragma unroll
                for (int d = 1; d < 5; d++) s = __fmaf_rn(dig[t][d], c_conv.c[m][d], s);
                const float q = __fsub_rn(__fmaf_rn(s, rm, 12582912.f), 12582912.f);
                y[t] = __fmaf_rn(-q, mm, s);
            }
            uint4 w;
            unsigned *wp = &w.x;
#pragma unroll
            for (int t = 0; t < 4; t++) {
                const __nv_bfloat162 b = __floats2bfloat162_rn(y[2 * t], y[2 * t + 1]);
                wp[t] = *reinterpret_cast<const unsigned *>(&b);
            }
            *reinterpret_cast<uint4 *>(dst + (size_t)m * nkb * rns::kTileElems) = w;
        }
    }
    some = __syncthreads_count(2 * small > some);   // threads most of whose entries are far below their scale
    if (threadIdx.x == 0 && some > kThreads / 2) atomicOr(flags, 2);
}

// All superblocks above the diagonal ones of a triangular M, both forms (rt,
// ct; null: not wanted) and their parts (blockIdx.z).
__global__ void __launch_bounds__(kThreads)
convert_fixed_kernel(const __grid_constant__ Mat M, int bits, const int *__restrict__ rexp,
                     const int *__restrict__ cexp, __nv_bfloat16 *__restrict__ rt, __nv_bfloat16 *__restrict__ ct,
                     int nkb, bool with_diagonal, int *__restrict__ flags)
{
    const int A = blockIdx.x, B = blockIdx.y, part = blockIdx.z / 2;
    if (A > B || (A == B && !with_diagonal)) return;
    if (blockIdx.z % 2 == 0) {
        if (rt) convert_superblock(M, bits, true, A, B, part, rexp, rt, nkb, flags);
    } else {
        if (ct) convert_superblock(M, bits, false, B, A, part, cexp, ct, nkb, flags);
    }
}

// The new superblocks (A, B) = (a0 + t, b0 + t), and the whole of a panel whose
// scale grew: of row panel A the superblocks before B (down to low, or to the
// diagonal when low < 0), of column panel B those below A (up to high, or to
// the diagonal).
__global__ void __launch_bounds__(kThreads)
convert_new_kernel(const __grid_constant__ Mat M, int bits, int a0, int b0, int low, int high,
                   const int *__restrict__ rexp, const int *__restrict__ cexp, const int *__restrict__ rgrown,
                   const int *__restrict__ cgrown, __nv_bfloat16 *__restrict__ rt, int nkbr,
                   __nv_bfloat16 *__restrict__ ct, int nkbc, int *__restrict__ flags)
{
    const int A = a0 + blockIdx.x, B = b0 + blockIdx.x, y = blockIdx.y, part = blockIdx.z / 2;
    if (blockIdx.z % 2 == 0) {
        if (B - y >= (low < 0 ? A : low) && (y == 0 || rgrown[A]))
            convert_superblock(M, bits, true, A, B - y, part, rexp, rt, nkbr, flags);
    } else {
        if (A + y <= (high < 0 ? B : high) && (y == 0 || cgrown[B]))
            convert_superblock(M, bits, false, B, A + y, part, cexp, ct, nkbc, flags);
    }
}

// ---- products ----------------------------------------------------------------

// The products of every superblock, D by D: UT, TU, UU.
__global__ void tiles_kernel(int ns, rns::Tile *__restrict__ tiles)
{
    const int D = blockIdx.x + 1;
    // superblocks of smaller D: sum_{d < D} (ns - d)
    const size_t base = (size_t)(D - 1) * ns - (size_t)(D - 1) * D / 2;
    for (int A = threadIdx.x; A < ns - D; A += blockDim.x) {
        const int B = A + D;
        rns::Tile *t = tiles + 3 * (base + A);
        t[0] = {0, A, B, 2 * A, 2 * B};
        t[1] = {1, A, B, 2 * (A + 1), 2 * (B + 1)};
        t[2] = {2, A, B, 2 * (A + 1), 2 * B};
    }
}

// The products of A X - X B's superblocks, step by step (superblocks (a, b),
// a = nr - 1 - s + b): X B and A X.
__global__ void sylvester_tiles_kernel(int nr, int nc, rns::Tile *__restrict__ tiles)
{
    const int s = blockIdx.x;
    int base = 0;
    for (int u = 0; u < s; u++) base += min(nc - 1, u) - max(0, u - (nr - 1)) + 1;
    const int b0 = max(0, s - (nr - 1)), b1 = min(nc - 1, s);
    for (int b = b0 + threadIdx.x; b <= b1; b += blockDim.x) {
        const int a = nr - 1 - s + b;
        rns::Tile *t = tiles + 2 * (base + b - b0);
        t[0] = {0, a, b, 0, 2 * b};
        t[1] = {1, a, b, 2 * (a + 1), 2 * nr};
    }
}

struct CrtConst {
    unsigned w[rns::kMods][3];   // floor(2^96 / m), 32-bit limbs
    int m[rns::kMods];
    double P;                    // the moduli's product
};
constexpr CrtConst make_crt_const()
{
    CrtConst k{};
    k.P = 1.0;
    for (int i = 0; i < rns::kMods; i++) {
        const unsigned long long m = (unsigned long long)rns::kModulus[i];
        k.m[i] = (int)m;
        k.P *= (double)m;
        unsigned long long r = 1;   // long division of 2^96
        for (int l = 2; l >= 0; l--) {
            const unsigned long long cur = r << 32;
            k.w[i][l] = (unsigned)(cur / m);
            r = cur % m;
        }
    }
    return k;
}
__constant__ CrtConst c_crt = make_crt_const();

// The product an entry's residues stand for (16 bytes, 16 KB apart).
__device__ __forceinline__ double crt(const int8_t *__restrict__ y)
{
    unsigned long long a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
    for (int m = 0; m < rns::kMods; m++) {
        int r = y[(size_t)m * SP * SP];
        r += r < 0 ? c_crt.m[m] : 0;
        a0 += (unsigned long long)(unsigned)r * c_crt.w[m][0];
        a1 += (unsigned long long)(unsigned)r * c_crt.w[m][1];
        a2 += (unsigned long long)(unsigned)r * c_crt.w[m][2];
    }
    a1 += a0 >> 32;
    const unsigned long long hi = (a2 << 32) + a1;   // top 64 of 96 bits; whole multiples of P drop out
    return (__ll2double_rn((long long)hi) * 0x1p-64 + (double)(unsigned)a0 * 0x1p-96) * c_crt.P;
}

// ---- the superblocks' own solve -----------------------------------------------

// Superblock t of a launch: rows A = a0 + t of the row set, columns B = b0 + t
// of the column set.  M = RT / RU and N = CT / CU are the sets' diagonal
// superblocks (RU, CU null: every entry takes RT, CT).  The sums over the other superblocks come as residues, three
// products to a tile: VN = sum v n (its row and column exponents er0, ec0), MV
// = sum m v (er1, ec1), and, where the signs agree, UU (er0, ec1).  The new
// entries' exponents go to rnew, cnew.
struct Wave {
    const double *RT, *RU, *CT, *CU, *C0;
    double *V;
    const int8_t *res;
    const int *er0, *ec0, *er1, *ec1;
    int *rnew, *cnew;
    int ldrt, ldru, ldct, ldcu, ldc0, ldv;
    int rows, cols, a0, b0, tiles, bits;
    int products;      // a tile's products in res: 3, or 2 without UU; 0: no sums
    double own;        // an entry's own term is own (u_pp - u_qq) C0
};

// The residue sums of entry (i, j) of superblock t, in row panel A and column
// panel B.
__device__ __forceinline__ double residue_sum(const Wave &w, int t, int i, int j, bool opp)
{
    if (w.products == 0) return 0.0;
    const int8_t *y = w.res + (size_t)t * w.products * rns::kMods * SP * SP + i * SP + j;
    const int r = (w.a0 + t) * SP + i, c = (w.b0 + t) * SP + j;
    if (!opp)
        return -scalbn(crt(y + (size_t)2 * rns::kMods * SP * SP), max(w.er0[r], kMinExp) + max(w.ec1[c], kMinExp) - 2 * w.bits);
    return scalbn(crt(y), max(w.er0[r], kMinExp) + max(w.ec0[c], kMinExp) - 2 * w.bits) -
           scalbn(crt(y + (size_t)rns::kMods * SP * SP), max(w.er1[r], kMinExp) + max(w.ec1[c], kMinExp) - 2 * w.bits);
}

// Blocks (i, j) of a superblock at step l = 7 - i + j.
__host__ __device__ constexpr int wave_blocks(int l) { return l < 0 || l > 2 * SB - 2 ? 0 : (l < SB ? l + 1 : 2 * SB - 1 - l); }
// Their sums over finished blocks more than one away are cut in three.
constexpr int kParts = 3;

struct WaveBlock {
    int t, jj, I, J, c, r;   // tile, place in the step, global blocks, finished blocks below and to the left
};
__device__ __forceinline__ WaveBlock wave_block(const Wave &w, int b, int l)
{
    WaveBlock k;
    const int cnt = wave_blocks(l);
    k.t = b / cnt;
    k.jj = b % cnt;
    const int j = max(0, l - (SB - 1)) + k.jj, i = SB - 1 - (l - j);
    const int A = w.a0 + k.t, B = w.b0 + k.t;
    k.I = A * SB + i;
    k.J = B * SB + j;
    const int nbr = min(SB, (w.rows + LB - 1) / LB - A * SB);   // row blocks the panel has
    k.c = nbr - 1 - i;
    k.r = j;
    return k;
}
// finished blocks beyond the near two, and how many each part takes
__device__ __forceinline__ int far_count(const WaveBlock &k) { return max(k.c - 1, 0) + max(k.r - 1, 0); }
__device__ __forceinline__ int far_per(int f) { return (f + kParts - 1) / kParts; }

union WaveSmem {
    struct {
        double TI[BLK], UI[BLK], TJ[BLK], UJ[BLK];
        double T1[BLK], U1[BLK], T2[BLK], U2[BLK], X1[BLK], X2[BLK];
        double C[BLK], V[BLK];
        double urow[LB], ucol[LB];
    } leaf;
    struct {
        double OT[2][BLK], OU[2][BLK], X[2][BLK];
    } far;
};

__device__ __forceinline__ double at_or_zero(const double *__restrict__ M, int ld, int i, int j, int ni, int nj)
{
    return i < ni && j < nj ? SGT_AT(M, ld, i, j) : 0.0;
}

__device__ __forceinline__ void wave_far(const Wave &w, int b, int l, double *__restrict__ slabs, WaveSmem &sm)
{
    const WaveBlock k = wave_block(w, b / kParts, l);
    const int part = b % kParts;
    const int r0 = k.I * LB, c0 = k.J * LB;
    if (r0 >= w.rows || c0 >= w.cols) return;
    const int f = far_count(k), per = far_per(f), x0 = part * per, x1 = min(f, x0 + per);
    if (x0 >= x1) return;
    const int ncol = max(k.c - 1, 0);
    const int lo = threadIdx.x % LB, hi = threadIdx.x / LB, at = lo + hi * LD;
    double ot, ou = 0.0, xv;
    auto fetch = [&](int x) {
        if (x < ncol) {   // column part: M of (I, K), V of (K, J)
            const int kb = r0 + (2 + x) * LB;
            ot = at_or_zero(w.RT, w.ldrt, r0 + lo, kb + hi, w.rows, w.rows);
            if (w.RU) ou = at_or_zero(w.RU, w.ldru, r0 + lo, kb + hi, w.rows, w.rows);
            xv = at_or_zero(w.V, w.ldv, kb + lo, c0 + hi, w.rows, w.cols);
        } else {          // row part: V of (I, K), N of (K, J)
            const int kb = c0 - (2 + x - ncol) * LB;
            ot = at_or_zero(w.CT, w.ldct, kb + lo, c0 + hi, w.cols, w.cols);
            if (w.CU) ou = at_or_zero(w.CU, w.ldcu, kb + lo, c0 + hi, w.cols, w.cols);
            xv = at_or_zero(w.V, w.ldv, r0 + lo, kb + hi, w.rows, w.cols);
        }
    };
    fetch(x0);
    const int p = lo, q = hi;
    bool opp = true;
    if (w.RU) opp = SGT_AT(w.RU, w.ldru, min(r0 + p, w.rows - 1), min(r0 + p, w.rows - 1)) +
                    SGT_AT(w.CU, w.ldcu, min(c0 + q, w.cols - 1), min(c0 + q, w.cols - 1)) == 0.0;
    const unsigned long long flip = opp ? 0ull : 0x8000000000000000ull;
    double acc = 0.0;
    for (int x = x0, buf = 0; x < x1; x++, buf ^= 1) {
        sm.far.OT[buf][at] = ot;
        sm.far.OU[buf][at] = ou;
        sm.far.X[buf][at] = xv;
        __syncthreads();
        const bool col = x < ncol;
        if (x + 1 < x1) fetch(x + 1);
        const double *O = opp ? sm.far.OT[buf] : sm.far.OU[buf], *X = sm.far.X[buf];
        if (col) {
#pragma unroll 8
            for (int i = 0; i < LB; i++) acc = fma(-O[p + i * LD], X[i + q * LD], acc);
        } else {
#pragma unroll 8
            for (int i = 0; i < LB; i++) acc = fma(lvl::flip_sign(X[p + i * LD], flip), O[i + q * LD], acc);
        }
    }
    slabs[(((size_t)k.t * SB + k.jj) * kParts + part) * LT + p + q * LB] = acc;
}

__device__ __forceinline__ void wave_leaf(const Wave &w, int b, int l, bool first, const double *__restrict__ slabs,
                                          WaveSmem &sm)
{
    auto &s = sm.leaf;
    const WaveBlock k = wave_block(w, b, l);
    const int r0 = k.I * LB, c0 = k.J * LB;
    if (r0 >= w.rows || c0 >= w.cols) {
        // every CTA waits, so that a launch of absent blocks only does not end
        // before the launch before it
        lvl::dependency_wait();
        return;
    }
    const int lo = threadIdx.x % LB, hi = threadIdx.x / LB, at = lo + hi * LD;
    const bool up = lo <= hi, hasU = w.RU != nullptr;
    if (first) lvl::dependency_wait();   // the residues come from the launch before
    const bool inr = r0 + lo < w.rows, inc = c0 + hi < w.cols, in = inr && inc;
    const double *RT = w.RT, *RU = hasU ? w.RU : w.RT, *CT = w.CT, *CU = hasU ? w.CU : w.CT;
    const int ldru = hasU ? w.ldru : w.ldrt, ldcu = hasU ? w.ldcu : w.ldct;
    // the diagonal superblocks' parts and the entries' own terms do not depend
    // on the launch before
    s.TI[at] = up ? at_or_zero(RT, w.ldrt, r0 + lo, r0 + hi, w.rows, w.rows) : 0.0;
    s.TJ[at] = up ? at_or_zero(CT, w.ldct, c0 + lo, c0 + hi, w.cols, w.cols) : 0.0;
    s.UI[at] = hasU && up ? at_or_zero(RU, ldru, r0 + lo, r0 + hi, w.rows, w.rows) : 0.0;
    s.UJ[at] = hasU && up ? at_or_zero(CU, ldcu, c0 + lo, c0 + hi, w.cols, w.cols) : 0.0;
    if (k.c > 0) {
        s.T1[at] = at_or_zero(RT, w.ldrt, r0 + lo, r0 + LB + hi, w.rows, w.rows);
        s.U1[at] = hasU ? at_or_zero(RU, ldru, r0 + lo, r0 + LB + hi, w.rows, w.rows) : 0.0;
    }
    if (k.r > 0) {
        s.T2[at] = at_or_zero(CT, w.ldct, c0 - LB + lo, c0 + hi, w.cols, w.cols);
        s.U2[at] = hasU ? at_or_zero(CU, ldcu, c0 - LB + lo, c0 + hi, w.cols, w.cols) : 0.0;
    }
    const double own = in ? SGT_AT(w.C0, w.ldc0, r0 + lo, c0 + hi) : 0.0;
    if (threadIdx.x < LB) {
        const int i = threadIdx.x;
        s.urow[i] = hasU && r0 + i < w.rows ? SGT_AT(RU, ldru, r0 + i, r0 + i) : 1.0;
        s.ucol[i] = hasU && c0 + i < w.cols ? SGT_AT(CU, ldcu, c0 + i, c0 + i) : -1.0;
    }
    int p, q;
    lvl::entry_of(threadIdx.x, p, q);
    const int step = LB - 1 - p + q;
    __syncthreads();
    const double upp = s.urow[p], uqq = s.ucol[q];
    const bool opp = upp + uqq == 0.0;
    const bool live = r0 + p < w.rows && c0 + q < w.cols;
    const double rinv = !live ? 0.0 : opp ? 1.0 / (s.TI[p + p * LD] - s.TJ[q + q * LD]) : 0.5 * upp;
    const unsigned long long flip = opp ? 0ull : 0x8000000000000000ull;
    const double *M = opp ? s.TI : s.UI, *N = opp ? s.TJ : s.UJ;
    const double *M1 = opp ? s.T1 : s.U1, *N2 = opp ? s.T2 : s.U2;
    // here a thread takes entry (hi, lo): residues lie row by row
    s.C[hi + lo * LD] = residue_sum(w, k.t, (k.I % SB) * LB + hi, (k.J % SB) * LB + lo, s.urow[hi] + s.ucol[lo] == 0.0);
    __syncthreads();

    lvl::dependency_wait();
    lvl::dependency_release();
    const int f = far_count(k), per = far_per(f), nslab = f > 0 ? (f + per - 1) / per : 0;
    const double *sl = slabs + ((size_t)k.t * SB + k.jj) * kParts * LT + threadIdx.x;
    double x1 = 0.0, x2 = 0.0, v[kParts];
    if (k.c > 0) x1 = at_or_zero(w.V, w.ldv, r0 + LB + lo, c0 + hi, w.rows, w.cols);
    if (k.r > 0 && inr) x2 = SGT_AT(w.V, w.ldv, r0 + lo, c0 - LB + hi);
#pragma unroll
    for (int t = 0; t < kParts; t++) v[t] = t < nslab ? sl[(size_t)t * LT] : 0.0;
    double sum = s.C[at];
#pragma unroll
    for (int t = 0; t < kParts; t++)
        if (t < nslab) sum += v[t];
    s.X1[at] = x1;
    s.X2[at] = x2;
    const double ui = s.urow[lo], uj = s.ucol[hi];
    s.C[at] = sum;
    s.V[at] = ui + uj == 0.0 ? own * (w.own * (ui - uj)) : 0.0;
    __syncthreads();
    double acc = s.C[p + q * LD];
    const double base = s.V[p + q * LD];
    if (k.c > 0) {
#pragma unroll 8
        for (int i = 0; i < LB; i++) acc = fma(-M1[p + i * LD], s.X1[i + q * LD], acc);
    }
    if (k.r > 0) {
#pragma unroll 8
        for (int i = 0; i < LB; i++) acc = fma(lvl::flip_sign(s.X2[p + i * LD], flip), N2[i + q * LD], acc);
    }
    lvl::solve16(acc, base, rinv, flip, M, N, s.V, p, q, step);
    const double x = in ? s.V[at] : 0.0;
    if (in) SGT_AT(w.V, w.ldv, r0 + lo, c0 + hi) = x;
    // a warp holds 16 rows of two columns
    const int e = x != 0.0 ? exponent_above(x) : kNoExp;
    const int er = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    int ec = e;
#pragma unroll
    for (int o = 1; o < LB; o <<= 1) ec = max(ec, __shfl_xor_sync(0xffffffffu, ec, o));
    if ((threadIdx.x & 31) < LB && inr) atomicMax(&w.rnew[r0 + lo], er);
    if (lo == 0 && inc) atomicMax(&w.cnew[c0 + hi], ec);
}

// Step l of every superblock of the launch: its leaves, and beside them the
// sums of step l + 1 over finished blocks that this step does not change.
__global__ void __launch_bounds__(kThreads)
wave_kernel(const __grid_constant__ Wave w, int l, bool first, const double *__restrict__ in, double *__restrict__ out)
{
    __shared__ WaveSmem sm;
    const int leaves = w.tiles * wave_blocks(l), b = blockIdx.x;
    if (b < leaves) {
        wave_leaf(w, b, l, first, in, sm);
    } else {
        lvl::dependency_wait();
        lvl::dependency_release();
        wave_far(w, b - leaves, l + 1, out, sm);
    }
}

signtri_status run_wave(const Wave &w, double *slab0, double *slab1, int cls, cudaStream_t st)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    double *slab[2] = {slab0, slab1};
    // the steps that hold blocks (a ragged panel has fewer rows or columns of
    // them; the first superblock has the most)
    const int nbr = std::min(SB, (w.rows + LB - 1) / LB - w.a0 * SB), nbc = std::min(SB, (w.cols + LB - 1) / LB - w.b0 * SB);
    const int l0 = SB - nbr, l1 = SB - 1 + nbc;
    for (int l = l0; l < l1; l++) {
        cfg.gridDim = dim3(w.tiles * (wave_blocks(l) + kParts * wave_blocks(l + 1)));
        ProfScope ps(cls, st);
        SGT_CUDA_TRY(cudaLaunchKernelEx(&cfg, wave_kernel, w, l, l == l0, (const double *)slab[l & 1], slab[(l + 1) & 1]));
    }
    return SIGNTRI_OK;
}
size_t wave_slab_bytes(int tiles) { return (size_t)tiles * SB * kParts * LT * sizeof(double); }

}  // namespace
}  // namespace sup

// ---- the whole solve ------------------------------------------------------------

size_t ph_super_workspace_bytes(int n)
{
    using namespace sup;
    const int ns = (n + SP - 1) / SP;
    const size_t form = rns::form_tile_bytes(ns, 2 * ns);
    return 4 * (form + 256) + 6 * ((size_t)ns * SP * sizeof(int) + 256) + 2 * ((size_t)ns * sizeof(int) + 256) +
           (size_t)ns * (ns - 1) / 2 * 3 * sizeof(rns::Tile) + 256 + (size_t)(ns - 1) * 3 * rns::kMods * SP * SP + 256 +
           2 * (wave_slab_bytes(ns - 1) + 256) + 256 +
           lvl::level_workspace_bytes<double>(n);
}

// flags_host (pinned): nonzero on return when the data did not suit one scale
// per row and the plain path has to run; waits for the stream.
signtri_status ph_super_run(int n, const double *T, int ldt, double *U, int ldu, Arena &ws, int *d_err,
                            int *flags_host, cudaStream_t st)
{
    using namespace sup;
    const int ns = (n + SP - 1) / SP, nkb = 2 * ns, bits = rns::operand_bits(ns * SP);
    auto take = [&](size_t b) { return ws.take(b); };
    __nv_bfloat16 *form[4];   // T rows, T columns, U rows, U columns
    int *exps[6];             // of the same, and the newest superblocks' of U
    for (auto *&f : form) f = static_cast<__nv_bfloat16 *>(take(rns::form_tile_bytes(ns, nkb)));
    for (auto *&e : exps) e = static_cast<int *>(take((size_t)ns * SP * sizeof(int)));
    int *rgrown = static_cast<int *>(take((size_t)ns * sizeof(int)));
    int *cgrown = static_cast<int *>(take((size_t)ns * sizeof(int)));
    auto *tiles = static_cast<rns::Tile *>(take((size_t)ns * (ns - 1) / 2 * 3 * sizeof(rns::Tile)));
    auto *res = static_cast<int8_t *>(take((size_t)(ns - 1) * 3 * rns::kMods * SP * SP));
    auto *slab0 = static_cast<double *>(take(wave_slab_bytes(ns - 1)));
    auto *slab1 = static_cast<double *>(take(wave_slab_bytes(ns - 1)));
    int *flags = static_cast<int *>(take(sizeof(int)));
    if (!flags) return SIGNTRI_ERR_NO_WORKSPACE;
    const Mat Tm{T, ldt, n, n, true}, Um{U, ldu, n, n, true};
    // the diagonal superblocks
    signtri_status rs = ph_fp64_near_run(n, T, ldt, U, ldu, SB - 1, ws, st);
    if (rs != SIGNTRI_OK) return rs;
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, st);
        for (auto *e : exps) SGT_CUDA_TRY(cudaMemsetAsync(e, 0xc0, (size_t)ns * SP * sizeof(int), st));   // below every exponent
        SGT_CUDA_TRY(cudaMemsetAsync(flags, 0, sizeof(int), st));
        tiles_kernel<<<ns - 1, 128, 0, st>>>(ns, tiles);
        SGT_LAUNCH_CHECK();
        fixed_exps_kernel<<<dim3(ns, ns), kThreads, 0, st>>>(Tm, false, exps[0], exps[1], flags);
        SGT_LAUNCH_CHECK();
        convert_fixed_kernel<<<dim3(ns, ns, 2 * kConvParts), kThreads, 0, st>>>(Tm, bits, exps[0], exps[1], form[0],
                                                                                form[1], nkb, false, flags);
        SGT_LAUNCH_CHECK();
        fixed_exps_kernel<<<ns, kThreads, 0, st>>>(Um, true, exps[4], exps[5], flags);
        SGT_LAUNCH_CHECK();
    }
    auto join = [&](int D) -> signtri_status {
        ProfScope ps(SIGNTRI_KC_CONVERT, st);
        grow_exps_kernel<<<ns - D, SP, 0, st>>>(0, D, exps[4], exps[5], exps[2], exps[3], rgrown, cgrown, flags);
        SGT_LAUNCH_CHECK();
        convert_new_kernel<<<dim3(ns - D, D + 1, 2 * kConvParts), kThreads, 0, st>>>(
            Um, bits, 0, D, -1, -1, exps[2], exps[3], rgrown, cgrown, form[2], nkb, form[3], nkb, flags);
        SGT_LAUNCH_CHECK();
        return SIGNTRI_OK;
    };
    if ((rs = join(0)) != SIGNTRI_OK) return rs;
    const rns::Sources src{{{form[2], form[1], nkb, nkb}, {form[0], form[3], nkb, nkb}, {form[2], form[3], nkb, nkb}}};
    size_t at = 0;
    for (int D = 1; D < ns; D++) {
        const int nt = ns - D;
        rs = rns::gemm(src, tiles + 3 * at, 3 * nt, 3, res, d_err, SIGNTRI_KC_BLOCK_SUMS_F64, st);
        if (rs != SIGNTRI_OK) return rs;
        at += nt;
        const Wave w{T, U, T, U, T, U, res, exps[2], exps[1], exps[0], exps[3], exps[4], exps[5], ldt, ldu, ldt, ldu, ldt, ldu,
                     n, n, 0, D, nt, bits, 3, 1.0};
        if ((rs = run_wave(w, slab0, slab1, SIGNTRI_KC_OFFDIAG_LEAF, st)) != SIGNTRI_OK) return rs;
        if (D + 1 < ns && (rs = join(D)) != SIGNTRI_OK) return rs;
    }
    SGT_CUDA_TRY(cudaMemcpyAsync(flags_host, flags, sizeof(int), cudaMemcpyDeviceToHost, st));
    SGT_CUDA_TRY(cudaStreamSynchronize(st));
    return SIGNTRI_OK;
}

// ---- A X - X B = C -----------------------------------------------------------------

static size_t sylvester_super_bytes(int nr, int nc, int nt)
{
    using namespace sup;
    size_t b = 2 * (wave_slab_bytes(nt) + 256) + 3 * ((size_t)(nr + nc) * SP * sizeof(int) + 512) + 256;
    if (nr + nc > 2)
        b += rns::form_tile_bytes(nr, 2 * nr) + rns::form_tile_bytes(nc, 2 * nc) + rns::form_tile_bytes(nr, 2 * nc) +
             rns::form_tile_bytes(nc, 2 * nr) + (size_t)nr * nc * 2 * sizeof(rns::Tile) +
             (size_t)nt * 2 * rns::kMods * SP * SP + (size_t)(nr + nc) * sizeof(int) + 8 * 256;
    return b;
}

size_t sylvester_super_workspace_bytes(int m, int p)
{
    if (m <= 0 || p <= 0) return 0;
    const int nr = (m + sup::SP - 1) / sup::SP, nc = (p + sup::SP - 1) / sup::SP;
    return sylvester_super_bytes(nr, nc, std::min(nr, nc));
}

// for every m + p = n: the forms take 2 (nr + nc)^2 tiles of K-blocks
size_t sylvester_super_workspace_bound(int n)
{
    const int k = (n + sup::SP - 1) / sup::SP + 1;
    return sylvester_super_bytes(k, 1, k / 2 + 1) + (size_t)k * k / 2 * sizeof(rns::Tile);
}

// X of A X - X B = cscale C by superblocks of 128 from the bottom-left one,
// as ph_super_run: the terms between superblocks as residue products, those
// inside one by wave_kernel.  flags_host (pinned) as there; one superblock
// needs no products, sets no flag and returns without waiting.
signtri_status sylvester_super_run(int m, int p, const double *A, int lda, const double *B, int ldb, const double *C,
                                   int ldc, double cscale, double *X, int ldx, Arena &ws, int *d_err, int *flags_host,
                                   cudaStream_t st)
{
    using namespace sup;
    const int nr = (m + SP - 1) / SP, nc = (p + SP - 1) / SP, nt = std::min(nr, nc);
    const int bits = rns::operand_bits(std::max(nr, nc) * SP);
    const bool products = nr + nc > 2;
    auto take = [&](size_t b) { return ws.take(b); };
    auto *slab0 = static_cast<double *>(take(wave_slab_bytes(nt)));
    auto *slab1 = static_cast<double *>(take(wave_slab_bytes(nt)));
    // exponents: A's rows, B's columns, X's rows and columns, and of X's newest
    int *ea = static_cast<int *>(take((size_t)nr * SP * sizeof(int))), *eb = static_cast<int *>(take((size_t)nc * SP * sizeof(int)));
    int *er = static_cast<int *>(take((size_t)nr * SP * sizeof(int))), *ec = static_cast<int *>(take((size_t)nc * SP * sizeof(int)));
    int *rnew = static_cast<int *>(take((size_t)nr * SP * sizeof(int))), *cnew = static_cast<int *>(take((size_t)nc * SP * sizeof(int)));
    int *flags = static_cast<int *>(take(sizeof(int)));
    if (!flags) return SIGNTRI_ERR_NO_WORKSPACE;
    *flags_host = 0;
    const Mat Am{A, lda, m, m, true}, Bm{B, ldb, p, p, true}, Xm{X, ldx, m, p, false};
    __nv_bfloat16 *fa = nullptr, *fb = nullptr, *fr = nullptr, *fc = nullptr;
    rns::Tile *tiles = nullptr;
    int8_t *res = nullptr;
    int *rgrown = nullptr, *cgrown = nullptr;
    {
        ProfScope ps(SIGNTRI_KC_CONVERT, st);
        for (int *e : {ea, er, rnew}) SGT_CUDA_TRY(cudaMemsetAsync(e, 0xc0, (size_t)nr * SP * sizeof(int), st));
        for (int *e : {eb, ec, cnew}) SGT_CUDA_TRY(cudaMemsetAsync(e, 0xc0, (size_t)nc * SP * sizeof(int), st));
        if (products) {
            fa = static_cast<__nv_bfloat16 *>(take(rns::form_tile_bytes(nr, 2 * nr)));
            fb = static_cast<__nv_bfloat16 *>(take(rns::form_tile_bytes(nc, 2 * nc)));
            fr = static_cast<__nv_bfloat16 *>(take(rns::form_tile_bytes(nr, 2 * nc)));
            fc = static_cast<__nv_bfloat16 *>(take(rns::form_tile_bytes(nc, 2 * nr)));
            tiles = static_cast<rns::Tile *>(take((size_t)nr * nc * 2 * sizeof(rns::Tile)));
            res = static_cast<int8_t *>(take((size_t)nt * 2 * rns::kMods * SP * SP));
            rgrown = static_cast<int *>(take((size_t)nr * sizeof(int)));
            cgrown = static_cast<int *>(take((size_t)nc * sizeof(int)));
            if (!cgrown) return SIGNTRI_ERR_NO_WORKSPACE;
            SGT_CUDA_TRY(cudaMemsetAsync(flags, 0, sizeof(int), st));
            sylvester_tiles_kernel<<<nr + nc - 1, 128, 0, st>>>(nr, nc, tiles);
            SGT_LAUNCH_CHECK();
            fixed_exps_kernel<<<dim3(nr, nr), kThreads, 0, st>>>(Am, false, ea, nullptr, flags);
            SGT_LAUNCH_CHECK();
            fixed_exps_kernel<<<dim3(nc, nc), kThreads, 0, st>>>(Bm, false, nullptr, eb, flags);
            SGT_LAUNCH_CHECK();
            convert_fixed_kernel<<<dim3(nr, nr, 2 * kConvParts), kThreads, 0, st>>>(Am, bits, ea, nullptr, fa, nullptr,
                                                                                    2 * nr, false, flags);
            SGT_LAUNCH_CHECK();
            convert_fixed_kernel<<<dim3(nc, nc, 2 * kConvParts), kThreads, 0, st>>>(Bm, bits, nullptr, eb, nullptr, fb,
                                                                                    2 * nc, false, flags);
            SGT_LAUNCH_CHECK();
        }
    }
    const rns::Sources src{{{fr, fb, 2 * nc, 2 * nc}, {fa, fc, 2 * nr, 2 * nr}, {}}};
    size_t at = 0;
    for (int s = 0; s < nr + nc - 1; s++) {
        const int b0 = std::max(0, s - (nr - 1)), cnt = std::min(nc - 1, s) - b0 + 1, a0 = nr - 1 - s + b0;
        signtri_status rs = SIGNTRI_OK;
        if (s > 0 && (rs = rns::gemm(src, tiles + 2 * at, 2 * cnt, 2, res, d_err, SIGNTRI_KC_SYLV_SUMS, st)) != SIGNTRI_OK)
            return rs;
        at += cnt;
        const Wave w{A, nullptr, B, nullptr, C, X, res, er, eb, ea, ec, rnew, cnew, lda, 0, ldb, 0, ldc, ldx,
                     m, p, a0, b0, cnt, bits, s > 0 ? 2 : 0, 0.5 * cscale};
        if ((rs = run_wave(w, slab0, slab1, SIGNTRI_KC_SYLV_LEAF, st)) != SIGNTRI_OK) return rs;
        if (s + 1 == nr + nc - 1) break;
        ProfScope ps(SIGNTRI_KC_CONVERT, st);
        grow_exps_kernel<<<cnt, SP, 0, st>>>(a0, b0, rnew, cnew, er, ec, rgrown, cgrown, flags);
        SGT_LAUNCH_CHECK();
        convert_new_kernel<<<dim3(cnt, std::max(b0 + cnt, nr - a0), 2 * kConvParts), kThreads, 0, st>>>(
            Xm, bits, a0, b0, 0, nr - 1, er, ec, rgrown, cgrown, fr, 2 * nc, fc, 2 * nr, flags);
        SGT_LAUNCH_CHECK();
    }
    if (!products) return SIGNTRI_OK;
    SGT_CUDA_TRY(cudaMemcpyAsync(flags_host, flags, sizeof(int), cudaMemcpyDeviceToHost, st));
    SGT_CUDA_TRY(cudaStreamSynchronize(st));
    return SIGNTRI_OK;
}

}  // namespace signtri
