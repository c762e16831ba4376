// ph_super.cu -- large float64 Parlett-Higham: superblocks of 128, their block
// sums as residue products on the tensor cores.
//
// The equations of ph_level.cuh with the off-diagonal part cut into
// superblocks (A, B) of 128 x 128, solved by superblock anti-diagonal
// D = B - A.  For each D:
//   1. rns::gemm: UT = U_A. T_.B and TU = T_A. U_.B over the superblocks
//      K = A .. B whose entries are known (the strictly upper parts of the
//      diagonal superblocks among them), and UU = U_A. U_.B over A < K < B, as
//      residues (rns.cu: rounding the operands to 62 bits below their row's or
//      column's scale is the only error), all but the superblocks
//      of level D - 1 on a second stream beside that level's waves;
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
// them.
//
// Whether one scale per row and column suits the data is tested on the results.
// With an operand's entries rounded to 2^-(bits + 1) of their scale R (of the row)
// or C (of the column), a sum over k of u_ik t_kj is off by about
//   E = 2^-(bits + 1) R C sqrt(|t_.j / C|^2 + |u_i. / R|^2),
// whatever the entries; the squared norms are gathered with the forms.  A leaf
// compares E with 2^-53 of what its sums and own terms came to, u_ij (t_ii - t_jj)
// or 2 u_ij: half a unit in the last place, less than a float64 sum's own
// roundings.  Where more than a quarter of a leaf's entries exceed that (or data
// is not finite), a flag is set and the caller runs the plain float64 path.
// Similar matrices D^-1 T D lose the same bits in every entry, so the test sees
// any such grading, in whatever order; single entries that came out small by
// cancellation stay below a quarter.  On ungraded data E is 2^-4 of the limit; D of two levels
// passes up to about 2^5 between them (n = 1792).
//
// The kernels work on lists of superblocks of any number of problems (a batch
// shares its launches), and on A X - X B = C as well, where every entry is of
// the first kind and rows and columns belong to different matrices.
#include <algorithm>
#include <climits>
#include <vector>

#include "df_arith.cuh"
#include "internal.cuh"
#include "ph_level.cuh"
#include "rns.cuh"
#include "super_plan.h"

namespace signtri {
namespace sup {

using lvl::BLK;
using lvl::LB;
using lvl::LD;
using lvl::LT;

constexpr int SP = kSuperEdge;
static_assert(SP == rns::kPanel, "a superblock is a product tile");
constexpr int SB = SP / LB;       // blocks of 16 per edge
constexpr int kThreads = 256;
constexpr int kNoExp = INT_MIN / 2;
constexpr int kHeadroom = 2;
constexpr int kMinExp = -900;     // keeps 2^(bits - exp) a normal number
constexpr int kNormBits = 14;     // squared norms count 2^-14
// A rounded entry is below 2^bits: a 53-bit significand moved up by 10 at most,
// in a signed 64-bit integer, and five balanced digits of 14 bits.
static_assert(rns::operand_bits(1) <= 62, "53 + 10 bits with the sign, and 5 x 14 - 1");
// An entry's E may be 2^slack times 2^-53 of its sum: for X, whose plain path sums
// in double-float (48 bits), more.
constexpr int kSylvSlack = 4;
// Where a level's products are summed ahead, beside the wave before: in runs of
// kAheadLevels levels with sums or more, beside waves of at most kAheadTiles
// superblocks.  Wider waves fill the float64 pipes and lose by the company (a
// batch of 300, hundreds of superblocks a level: 44.2 ms, with every level
// ahead 46.3); limits of 24, 40, 64 and 128 measure 36.6, 36.0, 36.3 and 36.3
// ms at n = 8192.
constexpr size_t kAheadTiles = 64;
constexpr int kAheadLevels = 4;
// A run of one problem ends kTellLevels levels after a flag was set, where it has
// kTellMin or more (the host lets no more than so many run ahead of it).
constexpr int kTellLevels = 3, kTellMin = 8;

namespace {

// One problem: V (U of sign(T), or X) over a set of rows and a set of columns
// with the operators m of the rows' (RT, RU) and n of the columns' (CT, CU) own
// triangular matrices; RU, CU null: every entry takes RT, CT.
struct Problem {
    const double *RT, *RU, *CT, *CU, *C0;
    double *V;
    int ldrt, ldru, ldct, ldcu, ldc0, ldv;
    int rows, cols;
    double own2;                                // an entry's own term is own2 (u_pp - u_qq) / 2 C0
    int bits, slack;
    bool triangular;                            // V strictly upper, rows and columns the same
    int *er0, *ec0, *er1, *ec1;                 // exponents: V's rows, CT's columns, RT's rows, V's columns
    unsigned *nr0, *nc0, *nr1, *nc1;            // squared norms of the converted part under these scales, in 2^-kNormBits
    int *rnew, *cnew;                           // of V's newest superblocks
    int *rgrown, *cgrown;                       // panels whose exponents grew
    __nv_bfloat16 *vr, *vc, *fm, *fn;           // row and column forms of V, row form of RT, column form of CT
    rns::Layout lvr, lvc, lfm, lfn;             // their layouts
    int nkbr, nkbc;                             // K-blocks over the rows (vc, fm) and over the columns (vr, fn)
    int *flags;
    int *told;                                  // null, or the host's copy of "a flag is set"
};

struct Super {   // superblock (A, B) of problem k
    int k, A, B;
};

// ---- scales and residues ----------------------------------------------------

__device__ __forceinline__ int exponent_above(double x)   // |x| < 2^result
{
    return ((__double2hiint(x) >> 20) & 0x7ff) - 1022;
}

// The problem is one for the plain path: 1 not finite, 2 not suited by one scale.
__device__ __forceinline__ void raise(const Problem &p, int why)
{
    atomicOr(p.flags, why);
    if (p.told) *static_cast<volatile int *>(p.told) = 1;
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

// What a pass reads: the rows' operators by rows, the columns' by columns, or V
// by both.
enum { kRowOps = 0, kColOps = 1, kV = 2 };
__device__ __forceinline__ Mat matrix_of(const Problem &p, int what)
{
    if (what == kRowOps) return {p.RT, p.ldrt, p.rows, p.rows, true};
    if (what == kColOps) return {p.CT, p.ldct, p.cols, p.cols, true};
    return {p.V, p.ldv, p.rows, p.cols, p.triangular};
}

// Every exponent of a problem below any that an entry has (a CTA per problem: six
// memsets each took 1.7 ms of a batch with 100 of them).
__global__ void __launch_bounds__(kThreads)
init_exps_kernel(const Problem *__restrict__ probs)
{
    const Problem p = probs[blockIdx.x];
    for (int i = threadIdx.x; i < p.nkbr / 2 * SP; i += kThreads) {
        p.er0[i] = p.er1[i] = p.rnew[i] = kNoExp;
        p.nr0[i] = p.nr1[i] = 0;
    }
    for (int i = threadIdx.x; i < p.nkbc / 2 * SP; i += kThreads) {
        p.ec0[i] = p.ec1[i] = p.cnew[i] = kNoExp;
        p.nc0[i] = p.nc1[i] = 0;
    }
}

// The largest exponents of the superblocks' rows (kRowOps), columns (kColOps)
// or both (kV, into rnew and cnew).
__global__ void __launch_bounds__(kThreads)
exps_kernel(const Problem *__restrict__ probs, const Super *__restrict__ list, int what)
{
    const Super t = list[blockIdx.x];
    const Problem p = probs[t.k];
    const Mat M = matrix_of(p, what);
    __shared__ int rmax[SP], cmax[SP];
    if (threadIdx.x < SP) rmax[threadIdx.x] = cmax[threadIdx.x] = kNoExp;
    __syncthreads();
    const int i = threadIdx.x % SP, h = threadIdx.x / SP;
    int rm = kNoExp;
    for (int j = h; j < SP; j += kThreads / SP) {
        const double x = M(t.A * SP + i, t.B * SP + j);
        const int e = x != 0.0 ? exponent_above(x) : kNoExp;
        rm = max(rm, e);
        const int cm = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0) atomicMax(&cmax[j], cm);
    }
    atomicMax(&rmax[i], rm);
    __syncthreads();
    if (threadIdx.x < SP) {
        int *re = what == kRowOps ? p.er1 : p.rnew, *ce = what == kColOps ? p.ec0 : p.cnew;
        if (what != kColOps) atomicMax(&re[t.A * SP + i], rmax[i]);
        if (what != kRowOps) atomicMax(&ce[t.B * SP + i], cmax[i]);
        if (rmax[i] > 1024) raise(p, 1);
    }
}

// The exponents of V's new superblocks that outgrow their row or column, and
// which panels to convert anew.  rnew, cnew: the new superblocks' largest,
// gathered by the leaves that solved them and reset here.
__global__ void __launch_bounds__(SP)
grow_exps_kernel(const Problem *__restrict__ probs, const Super *__restrict__ list)
{
    const Super t = list[blockIdx.x];
    const Problem p = probs[t.k];
    const int r = t.A * SP + threadIdx.x, c = t.B * SP + threadIdx.x;
    const int er = p.rnew[r], ec = p.cnew[c];
    p.rnew[r] = kNoExp;
    p.cnew[c] = kNoExp;
    if (er > 1024) raise(p, 1);
    const bool rg = er > p.er0[r], cg = ec > p.ec1[c];
    if (rg) p.er0[r] = er + kHeadroom;
    if (cg) p.ec1[c] = ec + kHeadroom;
    const int ra = __syncthreads_or(rg), ca = __syncthreads_or(cg);
    // all of a grown panel is converted anew, and its norms with it
    if (ra) p.nr0[r] = 0;
    if (ca) p.nc1[c] = 0;
    if (threadIdx.x == 0) { p.rgrown[t.A] = ra; p.cgrown[t.B] = ca; }
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

// Residues of one 128 x 128 superblock of M into panel P's K-blocks 2 K, 2 K + 1.
// rows: P holds rows, K counts columns; else P holds columns and K counts rows.
// Part `part` of kConvParts of it.
constexpr int kConvParts = SP * SP / 8 / kThreads;
__device__ __forceinline__ void convert_superblock(const Mat &M, int bits, bool rows,
                                                   int P, int K, int part, const int *__restrict__ exps,
                                                   unsigned *norms, __nv_bfloat16 *__restrict__ tiles,
                                                   const rns::Layout &form)
{
    const int it = part * kThreads + threadIdx.x;
    {
        // line `i` of the panel, 8 entries along K from 8 ch: eight threads write
        // a line's 128 bytes of a tile (a line each wrote half sectors: 4x
        // slower); along rows, four lines' entries of a column make a sector
        const int i = rows ? it / 8 % SP : it / (SP / 8), ch = rows ? it % 8 + it / (8 * SP) * 8 : it % (SP / 8);
        const int g = P * SP + i;
        const int e = max(exps[g], kMinExp);
        float dig[8][5];
        unsigned norm = 0;
#pragma unroll
        for (int t = 0; t < 8; t++) {
            const int k = K * SP + ch * 8 + t;
            const long long x = __double_as_longlong(rows ? M(g, k) : M(k, g));
            // |x| 2^(bits - e), rounded, by integer operations (the float64 pipe
            // is 1 / 64 of the others): the significand moved by the exponents'
            // difference; subnormal numbers lie below every scale's last bit
            const int ex = (int)(x >> 52) & 0x7ff;
            const int sh = (e - bits) - (ex - 1075);
            long long v = ex ? (x & 0xfffffffffffffll) | 0x10000000000000ll : 0;
            v = sh <= 0 ? v << min(-sh, 10) : sh < 63 ? (v + (1ll << (sh - 1))) >> sh : 0;
            // its square, rounded up
            const unsigned h = (unsigned)(v >> (bits - 12)) + 1;
            norm += v ? (h * h >> (24 - kNormBits)) + 1 : 0;
            if (x < 0) v = -v;
            // five balanced digits of 14 bits
#pragma unroll
            for (int d = 0; d < 5; d++) {
                const int r = ((int)(v & 16383) ^ 8192) - 8192;
                dig[t][d] = (float)r;
                v = (v - r) >> 14;
            }
        }
        const int kb = 2 * K + ch / 8, c8 = ch & 7;
        __nv_bfloat16 *dst = tiles + form.tile(P, 0, kb) * rns::kTileElems + i * 64 + ((c8 ^ (i & 7)) * 8);
        const size_t next = (size_t)form.count(P) * rns::kTileElems;
#pragma unroll 4
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
            *reinterpret_cast<uint4 *>(dst + (size_t)m * next) = w;
        }
        // (whole numbers: the sum does not depend on its order)
        const int lanes = rows ? 8 : SP / 8;
        for (int o = 1; o < lanes; o <<= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
        if (it % lanes == 0 && norm) atomicAdd(&norms[g], norm);
    }
}

// The operators' superblocks: row form of the rows' (kRowOps), column form of
// the columns' (kColOps).  blockIdx.y: the parts.
__global__ void __launch_bounds__(kThreads)
convert_ops_kernel(const Problem *__restrict__ probs, const Super *__restrict__ list, int what)
{
    const Super t = list[blockIdx.x];
    const Problem p = probs[t.k];
    if (what == kRowOps)
        convert_superblock(matrix_of(p, what), p.bits, true, t.A, t.B, blockIdx.y, p.er1, p.nr1, p.fm, p.lfm);
    else
        convert_superblock(matrix_of(p, what), p.bits, false, t.B, t.A, blockIdx.y, p.ec0, p.nc0, p.fn, p.lfn);
}

// V's new superblocks (A, B), and the whole of a panel whose scale grew: of row
// panel A the superblocks before B, of column panel B those below A, as far
// as the panels hold any.  blockIdx.z: form and part.
__global__ void __launch_bounds__(kThreads)
convert_new_kernel(const Problem *__restrict__ probs, const Super *__restrict__ list)
{
    const Super t = list[blockIdx.x];
    const Problem p = probs[t.k];
    const Mat M = matrix_of(p, kV);
    const int part = blockIdx.z / 2;
    if (blockIdx.z % 2 == 0) {
        const int count = 1 + (p.rgrown[t.A] ? t.B - (p.triangular ? t.A : 0) : 0);
        for (int y = blockIdx.y; y < count; y += gridDim.y)
            convert_superblock(M, p.bits, true, t.A, t.B - y, part, p.er0, p.nr0, p.vr, p.lvr);
    } else {
        const int count = 1 + (p.cgrown[t.B] ? (p.triangular ? t.B : p.nkbr / 2 - 1) - t.A : 0);
        for (int y = blockIdx.y; y < count; y += gridDim.y)
            convert_superblock(M, p.bits, false, t.B, t.A + y, part, p.ec1, p.nc1, p.vc, p.lvc);
    }
}

// ---- products ----------------------------------------------------------------

// Every superblock's products: V N over the finished blocks of its row, M V over
// those of its column, and, for sign(T), U U.
__global__ void tiles_kernel(const Problem *__restrict__ probs, const Super *__restrict__ list, int count, int products,
                             rns::Tile *__restrict__ tiles)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const Super t = list[i];
    const Problem &p = probs[t.k];
    rns::Tile *o = tiles + (size_t)products * i;
    auto tile = [&](int which, const SuperSpan &k) { return rns::Tile{3 * t.k + which, t.A, t.B, k.k0, k.k1, k.e0, k.e1}; };
    o[0] = tile(0, span_vn(p.triangular, t.A, t.B));
    o[1] = tile(1, span_mv(p.triangular, p.nkbr, t.A, t.B));
    if (products == 3) o[2] = tile(2, span_uu(t.A, t.B));
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

// An unsigned integer of 32 bits as float64, by the bits and one addition: the
// conversion instructions and the additions share the SM's one float64 pipe, which
// the leaves fill.
__device__ __forceinline__ double from_u32(unsigned x) { return __hiloint2double(0x43300000, (int)x) - 0x1p52; }

// 2^k times the product an entry's residues stand for (kMods bytes, 16 KB apart).
// 96 bits of its quotient by the moduli's product: off by 2^-68 R C.
__device__ __forceinline__ double crt(const int8_t *y, int k)
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
    // (signed) hi + a0 / 2^32: the upper half as 2^84 + 2^32 (h + 2^31), the lower
    // as 2^52 + l, their excess taken off exactly
    const double top = __hiloint2double(0x45300000, (int)((unsigned)(hi >> 32) ^ 0x80000000u)) - (0x1p84 + 0x1p63 + 0x1p52);
    const double x = fma(from_u32((unsigned)a0), 0x1p-32, top + __hiloint2double(0x43300000, (int)(unsigned)hi));
    // times P 2^(k - 64): exact but for one rounding, the power of two in P's exponent
    const int e = (__double2hiint(c_crt.P) >> 20) + k - 64;
    if (e < 1 || e > 2046 - 64) return scalbn(x * (c_crt.P * 0x1p-64), k);
    return x * __hiloint2double(__double2hiint(c_crt.P) + ((k - 64) << 20), __double2loint(c_crt.P));
}

// ---- the superblocks' own solve -----------------------------------------------

// A launch: its superblocks, their residues (products to a superblock; 0: no
// sums) and the problems they belong to.
struct Wave {
    const Problem *probs;
    const Super *list;
    const int8_t *res;
    int tiles, products;
};

// The exponent above sqrt(a + b), squared norms in 2^-kNormBits.
__device__ __forceinline__ int norm_exp(unsigned a, unsigned b)
{
    const unsigned long long s = (unsigned long long)a + b;
    return (65 - __clzll((long long)s) - kNormBits) >> 1;
}

// The residue sums of entry (i, j) of superblock t; off: the exponent of their
// error E (far below any where there is none).
__device__ __forceinline__ double residue_sum(const Wave &w, const Problem &pr, const Super &s, int t, int i, int j,
                                              bool opp, int &off)
{
    off = -4000;
    if (w.products == 0) return 0.0;
    const int8_t *y = w.res + (size_t)t * w.products * rns::kMods * SP * SP + i * SP + j;
    const int r = s.A * SP + i, c = s.B * SP + j, b2 = 2 * pr.bits;
    // both kinds of entry take their first sum in one pass: UT, or UU
    const int er0 = max(pr.er0[r], kMinExp), ec1 = max(pr.ec1[c], kMinExp);
    const int first = er0 + (opp ? max(pr.ec0[c], kMinExp) : ec1);
    const unsigned nr0 = pr.nr0[r], nc = opp ? pr.nc0[c] : pr.nc1[c];
    const double v = crt(opp ? y : y + (size_t)2 * rns::kMods * SP * SP, first - b2);
    // (of neighbouring superblocks A, B there are no products U U)
    if (nr0 && nc && (opp || s.B > s.A + 1)) off = first + norm_exp(nr0, nc) - pr.bits - 1;
    if (!opp) return -v;
    const int second = max(pr.er1[r], kMinExp) + ec1;
    const unsigned nr1 = pr.nr1[r], nc1 = pr.nc1[c];
    if (nr1 && nc1) off = max(off, second + norm_exp(nr1, nc1) - pr.bits - 1);
    return v - crt(y + (size_t)rns::kMods * SP * SP, second - b2);
}

// Blocks (i, j) of a superblock at step l = 7 - i + j.
__host__ __device__ constexpr int wave_blocks(int l) { return l < 0 || l > 2 * SB - 2 ? 0 : (l < SB ? l + 1 : 2 * SB - 1 - l); }
// Their sums over finished blocks more than one away are cut in two, each as
// long as a leaf or shorter and fewer CTAs to share the SMs with the leaves (one,
// two, three, four: Sylvester equation of a sorted diagonal, n = 8192, 16.1, 14.9,
// 16.0, 16.8 ms; Schur pair n = 2000 4.80, 4.58, 4.77, 4.92; sign(T) n = 8192 38.1,
// 36.3, 36.3, 36.3; batch of 300 44.6, 44.2, 44.8, 45.3).
constexpr int kParts = 2;

struct WaveBlock {
    int t, jj, I, J, c, r;   // tile, place in the step, global blocks, finished blocks below and to the left
    Super s;
    Problem p;
};
__device__ __forceinline__ WaveBlock wave_block(const Wave &w, int b, int l)
{
    WaveBlock k;
    const int cnt = wave_blocks(l);
    k.t = b / cnt;
    k.jj = b % cnt;
    k.s = w.list[k.t];
    k.p = w.probs[k.s.k];
    const int j = max(0, l - (SB - 1)) + k.jj, i = SB - 1 - (l - j);
    k.I = k.s.A * SB + i;
    k.J = k.s.B * SB + j;
    const int nbr = min(SB, (k.p.rows + LB - 1) / LB - k.s.A * SB);   // row blocks the panel has
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
        short off[BLK];                     // residue_sum's errors
    } leaf;
    struct {
        double OT[2][BLK], OU[2][BLK], X[2][BLK];
    } far;
};

__device__ __forceinline__ double at_or_zero(const double *M, int ld, int i, int j, int ni, int nj)
{
    return i < ni && j < nj ? SGT_AT(M, ld, i, j) : 0.0;
}

__device__ __forceinline__ void wave_far(const Wave &wv, int b, int l, double *slabs, WaveSmem &sm)
{
    const WaveBlock k = wave_block(wv, b / kParts, l);
    const Problem &w = k.p;
    const int part = b % kParts;
    lvl::dependency_wait();
    lvl::dependency_release();
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
    if (w.RU) opp = lvl::signs_differ(SGT_AT(w.RU, w.ldru, min(r0 + p, w.rows - 1), min(r0 + p, w.rows - 1)),
                                      SGT_AT(w.CU, w.ldcu, min(c0 + q, w.cols - 1), min(c0 + q, w.cols - 1)));
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

__device__ __forceinline__ void wave_leaf(const Wave &wv, int b, int l, bool first, const double *slabs,
                                          WaveSmem &sm)
{
    auto &s = sm.leaf;
    const WaveBlock k = wave_block(wv, b, l);
    const Problem &w = k.p;
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
    const bool opp = lvl::signs_differ(upp, uqq);
    const bool live = r0 + p < w.rows && c0 + q < w.cols;
    const double dif = s.TI[p + p * LD] - s.TJ[q + q * LD];
    Divisor<double> dv = !live ? Divisor<double>{0.0, 0}
                               : opp ? divisor_recip(dif) : Divisor<double>{copysign(0.5, upp), 0};
    const unsigned long long flip = opp ? 0ull : 0x8000000000000000ull;
    const double *M = opp ? s.TI : s.UI, *N = opp ? s.TJ : s.UJ;
    const double *M1 = opp ? s.T1 : s.U1, *N2 = opp ? s.T2 : s.U2;
    // here a thread takes entry (hi, lo): residues lie row by row
    int off;
    s.C[hi + lo * LD] = residue_sum(wv, w, k.s, k.t, (k.I % SB) * LB + hi, (k.J % SB) * LB + lo,
                                    lvl::signs_differ(s.urow[hi], s.ucol[lo]), off);
    s.off[hi + lo * LD] = (short)off;
    // own (u_ii - u_jj) = +-2 own
    s.V[at] = lvl::signs_differ(s.urow[lo], s.ucol[hi]) ? lvl::flip_sign(own, (unsigned long long)__double_as_longlong(s.urow[lo]) & 0x8000000000000000ull) * w.own2 : 0.0;
    __syncthreads();
    const double quot = opp && live ? lvl::quotient(s.V[p + q * LD], dif, dv) : 0.0;
    const bool far = __any_sync(0xffffffffu, dv.ex != 0);

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
    s.C[at] = sum;
    __syncthreads();
    double acc = 0.0;
    if (k.c > 0) {
#pragma unroll 8
        for (int i = 0; i < LB; i++) acc = fma(-M1[p + i * LD], s.X1[i + q * LD], acc);
    }
    if (k.r > 0) {
#pragma unroll 8
        for (int i = 0; i < LB; i++) acc = fma(lvl::flip_sign(s.X2[p + i * LD], flip), N2[i + q * LD], acc);
    }
    if (far && opp && live) dv.ex = divisor_shift(exponent_field(s.TI[p + p * LD] - s.TJ[q + q * LD]));
    lvl::solve16<false>(s.C[p + q * LD] + acc, quot, dv, far, flip, M, N, s.V, p, q, step);
    const double x = in ? s.V[at] : 0.0;
    if (in) SGT_AT(w.V, w.ldv, r0 + lo, c0 + hi) = x;
    // a warp holds 16 rows of two columns
    const bool some = (__double2hiint(x) << 1 | __double2loint(x)) != 0;   // x != 0, by the bits
    const int e = some ? exponent_above(x) : kNoExp;
    const int er = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    int ec = e;
#pragma unroll
    for (int o = 1; o < LB; o <<= 1) ec = max(ec, __shfl_xor_sync(0xffffffffu, ec, o));
    if ((threadIdx.x & 31) < LB && inr) atomicMax(&w.rnew[r0 + lo], er);
    if (lo == 0 && inc) atomicMax(&w.cnew[c0 + hi], ec);
    if (wv.products == 0) return;
    // what the sums and the own term came to: x (t_ii - t_jj) or 2 x
    const int ev = e + (lvl::signs_differ(s.urow[lo], s.ucol[hi]) ? exponent_above(s.TI[lo * (LD + 1)] - s.TJ[hi * (LD + 1)]) - 1 : 1);
    const int over = __syncthreads_count(some && s.off[at] > ev - 53 + w.slack);
    if (threadIdx.x == 0 && 4 * over > min(LB, w.rows - r0) * min(LB, w.cols - c0)) raise(w, 2);
}

// Step l of every superblock of the launch: its leaves, and beside them the
// sums of step l + 1 over finished blocks that this step does not change.
__global__ void __launch_bounds__(kThreads)
wave_kernel(const __grid_constant__ Wave w, int l, bool first, const double *in, double *out)
{
    __shared__ WaveSmem sm;
    const int leaves = w.tiles * wave_blocks(l), b = blockIdx.x;
    if (b < leaves) {
        wave_leaf(w, b, l, first, in, sm);
    } else {
        wave_far(w, b - leaves, l + 1, out, sm);
    }
}

// Shared memory a launch of G CTAs asks for beside its own: where there are
// few, an SM's divided by the CTAs an SM gets, so that they spread evenly (the
// scheduler puts four on an SM and leaves others empty, and a leaf that shares its
// float64 pipe waits for it); 66 KB at two an SM leaves one beside the residue
// products' CTA.  Measured with none / this, ms: Sylvester equation of a sorted
// diagonal, n = 8192, 17.1 / 14.9; Schur pair n = 2000 4.85 / 4.58; sign(T)
// n = 8192 36.2 / 36.3; four an SM (G up to 608) no better than none.
int wave_spread(int G)
{
    const int per = (G + lvl::kSms - 1) / lvl::kSms;
    return (per == 1 ? 190 : per == 2 ? 66 : per == 3 ? 45 : 0) * 1024;
}

// l0, l1: the first and one past the last step that hold blocks.
signtri_status run_wave(const Wave &w, int l0, int l1, double *slab0, double *slab1, int cls, cudaStream_t st)
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
    SGT_CUDA_TRY(cudaFuncSetAttribute(wave_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, wave_spread(1)));
    for (int l = l0; l < l1; l++) {
        cfg.gridDim = dim3(w.tiles * (wave_blocks(l) + kParts * wave_blocks(l + 1)));
        cfg.dynamicSmemBytes = wave_spread((int)cfg.gridDim.x);
        ProfScope ps(cls, st);
        SGT_CUDA_TRY(cudaLaunchKernelEx(&cfg, wave_kernel, w, l, l == l0, (const double *)slab[l & 1], slab[(l + 1) & 1]));
    }
    return SIGNTRI_OK;
}
size_t wave_slab_bytes(size_t tiles) { return tiles * SB * kParts * LT * sizeof(double); }

// ---- host side -------------------------------------------------------------------

int panels_of(int n) { return super_panels(n); }

// What a run of `levels` of superblocks works in besides its problems' own.
size_t run_bytes(size_t problems, size_t superblocks, size_t ops, size_t widest, int products)
{
    return problems * (sizeof(Problem) + 3 * sizeof(rns::Source) + sizeof(int)) + (superblocks + ops) * sizeof(Super) +
           superblocks * products * sizeof(rns::Tile) + 3 * widest * products * rns::kMods * SP * SP +
           2 * wave_slab_bytes(widest) + 12 * 256;
}
// A problem's exponents, norms and growth marks, and its forms.
size_t problem_bytes(int nr, int nc)
{
    return 5 * ((size_t)(nr + nc) * SP * sizeof(int) + 512) + (size_t)(nr + nc) * sizeof(int) + 512;
}
struct Forms {
    rns::Layout fm, fn, vr, vc;
    Forms(int nr, int nc, bool triangular)
        : fm{rns::kUpperRows, 2 * nr}, fn{rns::kUpperCols, 2 * nc},
          vr{triangular ? rns::kUpperRows : rns::kFull, 2 * nc}, vc{triangular ? rns::kUpperCols : rns::kFull, 2 * nr}
    {
    }
    size_t bytes(int nr, int nc) const
    {
        return rns::form_tile_bytes(fm, nr) + rns::form_tile_bytes(fn, nc) + rns::form_tile_bytes(vr, nr) +
               rns::form_tile_bytes(vc, nc) + 4 * 256;
    }
};

// A set of problems whose superblocks are solved level by level, every level's
// in the same launches.
struct Run {
    std::vector<Problem> probs;
    std::vector<Super> list;        // level by level
    std::vector<size_t> off{0};     // where the levels start
    std::vector<Super> row_ops, col_ops, diagonal;
    int products = 3;
    int sums_from = 0;              // the first level with sums
    int cls_sums, cls_leaf;

    bool reserve(Arena &ws, Problem &p, int nr, int nc, bool forms)
    {
        auto ints = [&](size_t n) { return static_cast<int *>(ws.take(n * sizeof(int))); };
        p.er0 = ints((size_t)nr * SP);
        p.er1 = ints((size_t)nr * SP);
        p.rnew = ints((size_t)nr * SP);
        p.ec0 = ints((size_t)nc * SP);
        p.ec1 = ints((size_t)nc * SP);
        p.cnew = ints((size_t)nc * SP);
        p.nr0 = reinterpret_cast<unsigned *>(ints((size_t)nr * SP));
        p.nr1 = reinterpret_cast<unsigned *>(ints((size_t)nr * SP));
        p.nc0 = reinterpret_cast<unsigned *>(ints((size_t)nc * SP));
        p.nc1 = reinterpret_cast<unsigned *>(ints((size_t)nc * SP));
        p.rgrown = ints(nr);
        p.cgrown = ints(nc);
        p.nkbr = 2 * nr;
        p.nkbc = 2 * nc;
        if (!forms) return p.cgrown != nullptr;
        const Forms l(nr, nc, p.triangular);
        auto form = [&](const rns::Layout &f, int panels) {
            return static_cast<__nv_bfloat16 *>(ws.take(rns::form_tile_bytes(f, panels)));
        };
        p.lfm = l.fm;
        p.lfn = l.fn;
        p.lvr = l.vr;
        p.lvc = l.vc;
        p.fm = form(l.fm, nr);
        p.fn = form(l.fn, nc);
        p.vr = form(l.vr, nr);
        p.vc = form(l.vc, nc);
        return p.vc != nullptr;
    }

    // flags (host, one per problem): nonzero where the data did not suit one
    // scale per row.  Where products run, waits for the stream and reads the
    // error word of their waits.  told: null, or (one problem) a pinned word the
    // kernels can write
    signtri_status run(Arena &ws, int *d_err, int *flags, int *told, cudaStream_t st)
    {
        const int np = (int)probs.size(), levels = (int)off.size() - 1;
        size_t widest = 0;
        for (int l = 0; l < levels; l++) widest = std::max(widest, off[l + 1] - off[l]);
        auto *d_probs = static_cast<Problem *>(ws.take(np * sizeof(Problem)));
        auto *d_src = static_cast<rns::Source *>(ws.take(3 * (size_t)np * sizeof(rns::Source)));
        auto *d_flags = static_cast<int *>(ws.take(np * sizeof(int)));
        std::vector<Super> all = list;
        for (auto *v : {&row_ops, &col_ops, &diagonal}) all.insert(all.end(), v->begin(), v->end());
        auto *d_list = static_cast<Super *>(ws.take(all.size() * sizeof(Super)));
        auto *tiles = static_cast<rns::Tile *>(ws.take(list.size() * products * sizeof(rns::Tile)));
        auto *res = static_cast<int8_t *>(ws.take(widest * products * rns::kMods * SP * SP));
        int8_t *ahead[2];
        for (int8_t *&h : ahead) h = static_cast<int8_t *>(ws.take(widest * products * rns::kMods * SP * SP));
        auto *slab0 = static_cast<double *>(ws.take(wave_slab_bytes(widest)));
        auto *slab1 = static_cast<double *>(ws.take(wave_slab_bytes(widest)));
        if (!slab1) return SIGNTRI_ERR_NO_WORKSPACE;
        std::vector<rns::Source> src(3 * (size_t)np);
        for (int k = 0; k < np; k++) {
            Problem &p = probs[k];
            p.flags = d_flags + k;
            p.told = told;
            src[3 * k] = {p.vr, p.fn, p.lvr, p.lfn, p.rgrown, nullptr};
            src[3 * k + 1] = {p.fm, p.vc, p.lfm, p.lvc, nullptr, p.cgrown};
            src[3 * k + 2] = {p.vr, p.vc, p.lvr, p.lvc, p.rgrown, p.cgrown};
        }
        SGT_CUDA_TRY(cudaMemcpyAsync(d_probs, probs.data(), np * sizeof(Problem), cudaMemcpyHostToDevice, st));
        SGT_CUDA_TRY(cudaMemcpyAsync(d_src, src.data(), src.size() * sizeof(rns::Source), cudaMemcpyHostToDevice, st));
        SGT_CUDA_TRY(cudaMemcpyAsync(d_list, all.data(), all.size() * sizeof(Super), cudaMemcpyHostToDevice, st));
        SGT_CUDA_TRY(cudaMemsetAsync(d_flags, 0, np * sizeof(int), st));
        const bool sums = levels > sums_from;
        {
            ProfScope ps(SIGNTRI_KC_CONVERT, st);
            init_exps_kernel<<<np, kThreads, 0, st>>>(d_probs);
            SGT_LAUNCH_CHECK();
            if (sums) {
                tiles_kernel<<<(unsigned)((list.size() + 255) / 256), 256, 0, st>>>(d_probs, d_list, (int)list.size(),
                                                                                    products, tiles);
                SGT_LAUNCH_CHECK();
                const Super *rl = d_list + list.size(), *cl = rl + row_ops.size();
                for (int what : {kRowOps, kColOps}) {
                    const Super *l = what == kRowOps ? rl : cl;
                    const unsigned n = (unsigned)(what == kRowOps ? row_ops.size() : col_ops.size());
                    exps_kernel<<<n, kThreads, 0, st>>>(d_probs, l, what);
                    SGT_LAUNCH_CHECK();
                    convert_ops_kernel<<<dim3(n, kConvParts), kThreads, 0, st>>>(d_probs, l, what);
                    SGT_LAUNCH_CHECK();
                }
            }
        }
        // V's superblocks [l, l + n) join its forms
        auto join = [&](const Super *l, size_t n, int longest) -> signtri_status {
            ProfScope ps(SIGNTRI_KC_CONVERT, st);
            grow_exps_kernel<<<(unsigned)n, SP, 0, st>>>(d_probs, l);
            SGT_LAUNCH_CHECK();
            convert_new_kernel<<<dim3((unsigned)n, std::min(longest, 8), 2 * kConvParts), kThreads, 0, st>>>(d_probs, l);
            SGT_LAUNCH_CHECK();
            return SIGNTRI_OK;
        };
        signtri_status rs = SIGNTRI_OK;
        if (sums && !diagonal.empty()) {
            const Super *l = d_list + all.size() - diagonal.size();
            exps_kernel<<<(unsigned)diagonal.size(), kThreads, 0, st>>>(d_probs, l, kV);
            SGT_LAUNCH_CHECK();
            if ((rs = join(l, diagonal.size(), 1)) != SIGNTRI_OK) return rs;
        }
        // The products stream their operands from memory, the waves wait on
        // float64 chains: so, beside a level's wave, the next level's products
        // sum on a second stream what that wave does not change, and only the
        // K-blocks of two superblocks are left between the waves (n = 8192:
        // 37.9 -> 36.3 ms; Sylvester equation of a sorted diagonal 17.8 -> 14.9).
        CallStream side;
        bool summed_ahead = false;
        const bool overlap = levels - sums_from >= kAheadLevels;
        if (overlap) SGT_CUDA_TRY(side.init());
        const bool tell = told && levels >= kTellMin;
        CallEvents behind;   // the last levels' ends
        if (tell) {
            *told = 0;
            SGT_CUDA_TRY(behind.init(kTellLevels));
        }
        for (int l = 0; l < levels; l++) {
            if (tell && l >= kTellLevels) {
                SGT_CUDA_TRY(cudaEventSynchronize(behind.e[l % kTellLevels]));
                if (*static_cast<volatile int *>(told)) break;
            }
            const size_t n = off[l + 1] - off[l];
            const Super *at = d_list + off[l];
            const bool with_sums = l >= sums_from;
            if (with_sums) {
                const bool have = summed_ahead;
                summed_ahead = false;
                if (have) SGT_CUDA_TRY(cudaStreamWaitEvent(st, side.done[l & 1], 0));
                rs = rns::gemm(d_src, tiles + products * off[l], (int)(products * n), products, false,
                               have ? ahead[l & 1] : nullptr, res, d_err, cls_sums, st);
                if (rs != SIGNTRI_OK) return rs;
            }
            if (overlap && l + 1 < levels && l + 1 >= sums_from + 2 && n <= kAheadTiles) {
                summed_ahead = true;
                SGT_CUDA_TRY(cudaEventRecord(side.ready[l & 1], st));
                SGT_CUDA_TRY(cudaStreamWaitEvent(side.s, side.ready[l & 1], 0));
                rs = rns::gemm(d_src, tiles + products * off[l + 1], (int)(products * (off[l + 2] - off[l + 1])), products,
                               true, ahead[(l + 1) & 1], nullptr, d_err, cls_sums, side.s);
                if (rs != SIGNTRI_OK) return rs;
                SGT_CUDA_TRY(cudaEventRecord(side.done[(l + 1) & 1], side.s));
            }
            // the steps that hold blocks: ragged panels have fewer rows or columns
            int nbr = 0, nbc = 0;
            for (size_t i = off[l]; i < off[l + 1]; i++) {
                const Problem &p = probs[list[i].k];
                nbr = std::max(nbr, std::min(SB, (p.rows + LB - 1) / LB - list[i].A * SB));
                nbc = std::max(nbc, std::min(SB, (p.cols + LB - 1) / LB - list[i].B * SB));
            }
            const Wave w{d_probs, at, res, (int)n, with_sums ? products : 0};
            if ((rs = run_wave(w, SB - nbr, SB - 1 + nbc, slab0, slab1, cls_leaf, st)) != SIGNTRI_OK) return rs;
            if (l + 1 < levels && (rs = join(at, n, l + 2)) != SIGNTRI_OK) return rs;
            if (tell) SGT_CUDA_TRY(cudaEventRecord(behind.e[l % kTellLevels], st));
        }
        if (!sums) {   // nothing that could have set a flag
            for (int k = 0; k < np; k++) flags[k] = 0;
            return SIGNTRI_OK;
        }
        int err = 0;
        SGT_CUDA_TRY(cudaMemcpyAsync(flags, d_flags, np * sizeof(int), cudaMemcpyDeviceToHost, st));
        if (overlap) SGT_CUDA_TRY(cudaStreamSynchronize(side.s));   // products beside the last wave
        SGT_CUDA_TRY(cudaMemcpyAsync(&err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
        SGT_CUDA_TRY(cudaStreamSynchronize(st));
        return err ? SIGNTRI_ERR_TIMEOUT : SIGNTRI_OK;
    }
};

}  // namespace
}  // namespace sup

// ---- sign(T) ------------------------------------------------------------------------

size_t ph_super_workspace_bytes(int count, const int *n)
{
    using namespace sup;
    size_t b = 0, superblocks = 0, ops = 0, widest = 0;
    for (int k = 0; k < count; k++) {
        const size_t ns = panels_of(n[k]);
        b += problem_bytes((int)ns, (int)ns) + Forms((int)ns, (int)ns, true).bytes((int)ns, (int)ns);
        superblocks += ns * (ns - 1) / 2;
        ops += ns * (ns + 1) + ns;
        widest += ns - 1;
    }
    return b + run_bytes(count, superblocks, ops, widest, 3);
}

signtri_status ph_super_run(int count, const BatchDesc *mats, Arena &ws, int *d_err, int *flags, int *told,
                            cudaStream_t st)
{
    using namespace sup;
    Run r;
    r.cls_sums = SIGNTRI_KC_BLOCK_SUMS_F64;
    r.cls_leaf = SIGNTRI_KC_OFFDIAG_LEAF;
    int most = 0;
    for (int k = 0; k < count; k++) {
        const BatchDesc &m = mats[k];
        const int ns = panels_of(m.n);
        most = std::max(most, ns);
        Problem p{};
        p.RT = p.CT = p.C0 = m.T;
        p.RU = p.CU = m.U;
        p.V = m.U;
        p.ldrt = p.ldct = p.ldc0 = m.ldt;
        p.ldru = p.ldcu = p.ldv = m.ldu;
        p.rows = p.cols = m.n;
        p.own2 = 2.0;
        p.bits = rns::operand_bits(ns * SP);
        p.triangular = true;
        if (!r.reserve(ws, p, ns, ns, true)) return SIGNTRI_ERR_NO_WORKSPACE;
        r.probs.push_back(p);
        for (int A = 0; A < ns; A++) {
            r.diagonal.push_back({k, A, A});
            for (int B = A; B < ns; B++) r.row_ops.push_back({k, A, B});
        }
    }
    r.col_ops = r.row_ops;
    for (int D = 1; D < most; D++) {
        for (int k = 0; k < count; k++)
            for (int A = 0; A + D < panels_of(mats[k].n); A++) r.list.push_back({k, A, A + D});
        r.off.push_back(r.list.size());
    }
    return r.run(ws, d_err, flags, count == 1 ? told : nullptr, st);
}

// ---- A X - X B = C ----------------------------------------------------------------

static size_t sylvester_super_bytes(int nr, int nc, int nt)
{
    using namespace sup;
    return problem_bytes(nr, nc) + run_bytes(1, (size_t)nr * nc, ((size_t)nr * (nr + 1) + (size_t)nc * (nc + 1)) / 2, nt, 2);
}

size_t sylvester_super_workspace_bytes(int m, int p)
{
    if (m <= 0 || p <= 0) return 0;
    const int nr = sup::panels_of(m), nc = sup::panels_of(p);
    return sylvester_super_bytes(nr, nc, std::min(nr, nc)) + (nr + nc > 2 ? sup::Forms(nr, nc, false).bytes(nr, nc) : 0);
}

// for every m + p = n, with k panels in all: the forms hold nr (nr + 1) + nc (nc + 1) + 4 nr nc
// K-blocks, most at nr = nc
size_t sylvester_super_workspace_bound(int n)
{
    const int k = sup::panels_of(n) + 1, h = (k + 1) / 2;
    return sylvester_super_bytes(k, 1, k / 2 + 1) + sup::Forms(h, h, false).bytes(h, h) +
           (size_t)k * k / 2 * (2 * sizeof(rns::Tile) + sizeof(sup::Super));
}

signtri_status sylvester_super_run(int m, int p, const double *A, int lda, const double *B, int ldb, const double *C,
                                   int ldc, double cscale, double *X, int ldx, Arena &ws, int *d_err, int *flags,
                                   int *told, cudaStream_t st)
{
    using namespace sup;
    const int nr = panels_of(m), nc = panels_of(p);
    Run r;
    r.cls_sums = SIGNTRI_KC_SYLV_SUMS;
    r.cls_leaf = SIGNTRI_KC_SYLV_LEAF;
    r.products = 2;
    r.sums_from = 1;
    Problem q{};
    q.RT = A;
    q.CT = B;
    q.C0 = C;
    q.V = X;
    q.ldrt = lda;
    q.ldct = ldb;
    q.ldc0 = ldc;
    q.ldv = ldx;
    q.rows = m;
    q.cols = p;
    q.own2 = cscale;   // (rows and columns stand for u = 1 and -1)
    q.bits = rns::operand_bits(std::max(nr, nc) * SP);
    q.slack = kSylvSlack;
    if (!r.reserve(ws, q, nr, nc, nr + nc > 2)) return SIGNTRI_ERR_NO_WORKSPACE;
    r.probs.push_back(q);
    for (int a = 0; a < nr; a++)
        for (int b = a; b < nr; b++) r.row_ops.push_back({0, a, b});
    for (int a = 0; a < nc; a++)
        for (int b = a; b < nc; b++) r.col_ops.push_back({0, a, b});
    for (int s = 0; s < nr + nc - 1; s++) {   // from the bottom-left superblock
        for (int b = std::max(0, s - (nr - 1)); b <= std::min(nc - 1, s); b++) r.list.push_back({0, nr - 1 - s + b, b});
        r.off.push_back(r.list.size());
    }
    return r.run(ws, d_err, flags, told, st);
}

}  // namespace signtri
