// ph_level.cuh -- one launch per block anti-diagonal: the float64
// Parlett-Higham leaves of blocks of 16 and, beside them in the same launch,
// the block sums of the next anti-diagonal.  Used by the single-matrix
// (ph_fp64.cu), batched (batched.cu) and general-phi (funm.cu) paths.
//
// Entry (p, q) of block (I, J), J = I + d, is fixed by (Algorithm 6, 1x1 case)
//   signs differ: (t_pp - t_qq) v_pq = t_pq (u_pp - u_qq) + sum_k (u_pk t_kq - t_pk u_kq)
//   signs agree:  (u_pp + u_qq) v_pq = - sum_k u_pk u_kq
// with k running over every index strictly between p and q.  Only the terms
//   - m_pk u_kq  for k in block I + 1     (u_kq: anti-diagonal d - 1)
//   + u_pk n_kq  for k in block J - 1     (u_pk: anti-diagonal d - 1)
// and those inside blocks I and J that hold v itself need the anti-diagonal
// just before; all others ("early" terms) need d - 2 or less, or the diagonal
// blocks.  (m = t, n = t where the signs differ; m = u, n = -u where they
// agree.)  So launch d runs two kinds of CTAs that do not depend on each
// other:
//   leaf CTAs, one per block of anti-diagonal d: add the early sums (partial
//     slabs of launch d - 1), the two near blocks, and solve the block;
//   far CTAs: the early sums of anti-diagonal d + 1.
// One launch per anti-diagonal instead of two, and the block sums hide behind
// the leaves, which bound small problems: a leaf is a chain of 31 dependent
// steps of float64 arithmetic, whose pipe takes one warp instruction per 64
// cycles and sub-partition on GB300.  Launches are programmatic dependents:
// a leaf loads its operands and forms its reciprocals before it waits for the
// launch before it.
//
// Inside a leaf one thread owns one entry.  A solved entry is pushed at once
// into the later entries that need it (one multiply-add for the row, one for
// the column), so a step's critical path is three multiply-adds and a barrier,
// whatever the length of the entry's sum; threads are numbered
// along the block's anti-diagonals, so whole warps fall idle as the solve
// proceeds and leave the float64 pipe to the others.
#pragma once

#include <algorithm>

#include "df_arith.cuh"
#include "internal.cuh"
#include "level_split.h"
#include "ph_bodies.cuh"

namespace signtri {
namespace lvl {

constexpr int LT = LB * LB;     // threads of a leaf, and of each half of a far CTA: one per entry
constexpr int kLevelThreads = 2 * LT;
constexpr int LD = LB + 1;      // shared-memory pitch of a block
constexpr int BLK = LB * LD;    // doubles per staged block

// What a launch before may still be writing when a kernel starts (U, the slabs)
// is passed without __restrict__: a restricted pointer's loads may be moved
// above the wait.
// Wait for the launch this one programmatically depends on (all of it, with
// its writes visible); let the next launch start its independent part.
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- arithmetic of real (double) and complex (double2) entries ------------
__device__ __forceinline__ double mac(double a, double b, double c) { return fma(a, b, c); }     // c + a b
__device__ __forceinline__ double nmac(double a, double b, double c) { return fma(-a, b, c); }   // c - a b
__device__ __forceinline__ double2 mac(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 nmac(double2 a, double2 b, double2 c)
{
    return make_double2(fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double flip_sign(double a, unsigned long long m)
{
    return __longlong_as_double(__double_as_longlong(a) ^ m);
}
__device__ __forceinline__ double2 flip_sign(double2 a, unsigned long long m)
{
    return make_double2(flip_sign(a.x, m), flip_sign(a.y, m));
}
__device__ __forceinline__ double re(double a) { return a; }
__device__ __forceinline__ double re(double2 a) { return a.x; }
__device__ __forceinline__ double scaled(double a, double r) { return a * r; }
__device__ __forceinline__ double2 scaled(double2 a, double r) { return make_double2(a.x * r, a.y * r); }
template <class S>
__device__ __forceinline__ S real_value(double r);
template <>
__device__ __forceinline__ double real_value<double>(double r) { return r; }
template <>
__device__ __forceinline__ double2 real_value<double2>(double r) { return make_double2(r, 0.0); }
__device__ __forceinline__ double sub(double a, double b) { return a - b; }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ bool finite(double a) { return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool finite(double2 a) { return finite(a.x) && finite(a.y); }
// complex 1 / d by R. L. Smith's algorithm (CACM 5(8), 1962)
__device__ __forceinline__ Divisor<double2> divisor(double2 d)
{
    const int ex = divisor_shift(max((__double2hiint(d.x) >> 20) & 0x7ff, (__double2hiint(d.y) >> 20) & 0x7ff));
    if (ex) d = scaled(d, power_of_2(ex));
    const double x = d.x, y = d.y;
    if (fabs(x) >= fabs(y)) {
        const double r = y / x, den = fma(y, r, x);
        return {make_double2(1.0 / den, -r / den), ex};
    }
    const double r = x / y, den = fma(x, r, y);
    return {make_double2(r / den, -1.0 / den), ex};
}
using signtri::divisor;
// c + a b with one rounding of c's size (mac of complex entries has two)
__device__ __forceinline__ double mac_once(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 mac_once(double2 a, double2 b, double2 c)
{
    return add(make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x)), c);
}
// base / d + sum / d, the first quotient given
template <class S>
__device__ __forceinline__ S add_quotient(S sum, const Divisor<S> &dv, S quot)
{
    if (dv.ex == 0) return mac_once(sum, dv.r, quot);
    return add(scaled(mac(sum, dv.r, real_value<S>(0.0)), power_of_2(dv.ex)), quot);
}
// base / d: the product with 1 / d and one step of iterative refinement, as
// accurate as a division
template <class S>
__device__ __forceinline__ S quotient(S base, S d, const Divisor<S> &dv)
{
    const S zero = real_value<S>(0.0);
    S x = add_quotient(base, dv, zero);
    if (dv.ex == 0 && finite(x)) x = mac_once(nmac(d, x, base), dv.r, x);
    return x;
}

// barrier of one half of a CTA
__device__ __forceinline__ void half_sync(int half)
{
    asm volatile("bar.sync %0, %1;" ::"r"(half + 1), "n"(LT) : "memory");
}

// the position of set bit number r of a 16-bit mask
__device__ __forceinline__ int nth_bit(unsigned mask, int r)
{
    for (int i = 0; i < r; i++) mask &= mask - 1;
    return __ffs(mask) - 1;
}

template <class S>
union alignas(16) Smem {
    struct {
        S AU[2][LB * LB], AT[2][LB * LB];   // [buffer][k * 16 + row]
        S BU[2][BLK], BT[2][BLK];           // [buffer][column * 17 + k]
    } far[2];                                    // per half of the CTA
    struct {
        S TI[BLK], UI[BLK], TJ[BLK], UJ[BLK];       // diagonal blocks, [row + column * 17]
        S T1[BLK], U1[BLK], T2[BLK], U2[BLK];       // blocks (I, I+1) and (J-1, J)
        S X1[BLK], X2[BLK];                         // U of blocks (I+1, J) and (I, J-1)
        S C[BLK], V[BLK];
        S urow[LB], ucol[LB];
    } leaf;
};

// Shared memory a CTA of a launch of G asks for: an SM's, divided by the CTAs
// an SM gets, so that they spread evenly (left to itself the scheduler puts
// 152 CTAs on 123 SMs, and a leaf that shares its SM takes twice as long).
// Small launches ask for less, so that they start beside the one before and
// have their operands loaded when it ends.
constexpr int kSmallLaunch = 64;
template <class S>
constexpr int level_smem(int G)
{
    const int per = (G + kSms - 1) / kSms;
    const int b = (227 - per) / per * 1024;
    return G > kSmallLaunch && b > (int)sizeof(Smem<S>) ? b : (int)sizeof(Smem<S>);
}
template <class S>
constexpr size_t level_workspace_bytes(int n)
{
    return level_slabs(n) == 0 ? 0 : 2 * (level_slabs(n) * LT * sizeof(S) + 256);
}

// Early sums of tile (I, J) over the K-blocks [kb0, kb1) of I .. J, written to
// slab (entry (p, q) at p + 16 q): where the signs differ
//   sum u_pk t_kq over K = I (k > p) and I < K <= J - 2, minus
//   sum t_pk u_kq over I + 2 <= K < J and K = J (k < q);
// where they agree sum u_pk u_kq over I + 2 <= K <= J - 2.  general: every
// entry takes the first form.  Entries are dealt to threads by kind (rows and
// columns gathered by sign), so a warp issues one multiply-add a term or two,
// not both kinds for every entry; at most one warp of a half holds both, and
// the second half deals them in reverse, so that every sub-partition gets
// both kinds.  The two halves of the CTA take every other K-block, each at
// its own pace (one fills the float64 pipes while the other waits at its
// barrier), and add up at the end; the next K-block is in flight in registers
// while one is summed.
template <bool general, class S>
__device__ __forceinline__ void far_sums(int n, const S *__restrict__ T, int ldt, const S *U,
                                         int ldu, int I, int J, int kb0, int kb1, S *slab,
                                         Smem<S> &sm)
{
    const int r0 = I * LB, c0 = J * LB;
    const int bj = min(LB, n - c0);
    const int half = threadIdx.x / LT, tid = threadIdx.x % LT;
    const int lo = tid % LB, hi = tid / LB, lane = tid & 31;
    S au, at, bu, bt;
    auto fetch = [&](int kb) {
        const bool useUT = kb == I || kb <= J - 2, useTU = kb == J || kb >= I + 2;
        const int k0 = kb * LB;
        au = at = bu = bt = real_value<S>(0.0);
        // A: rows of block I (lo = row), B: columns of block J (hi = column);
        // only the last block of all can be ragged
        if (useUT) {
            au = SGT_AT(U, ldu, r0 + lo, k0 + hi);
            if (hi < bj) bt = SGT_AT(T, ldt, k0 + lo, c0 + hi);
        }
        if (useTU) {
            if (kb < J || hi < bj) at = SGT_AT(T, ldt, r0 + lo, k0 + hi);
            if (hi < bj && (kb < J || lo < bj)) bu = SGT_AT(U, ldu, k0 + lo, c0 + hi);
        }
    };
    if (kb0 + half < kb1) fetch(kb0 + half);
    int p = lo, q = hi;
    bool opp = true;
    if (!general) {
        const int g = (lane < LB) ? r0 + lane : c0 + lane - LB;
        const unsigned pos = __ballot_sync(0xffffffffu, g < n && re(SGT_AT(T, ldt, g < n ? g : 0, g < n ? g : 0)) > 0.0);
        const unsigned rm = pos & 0xffffu, cm = pos >> 16;
        const int rp = __popc(rm), cp = __popc(cm), rn = LB - rp, cn = LB - cp;
        int t = half ? LT - 1 - tid : tid;
        unsigned rset, cset;
        int len;
        if (t < rp * cp) { rset = rm; cset = cm; len = rp; opp = false; }
        else if ((t -= rp * cp) < rn * cn) { rset = ~rm; cset = ~cm; len = rn; opp = false; }
        else if ((t -= rn * cn) < rp * cn) { rset = rm; cset = ~cm; len = rp; }
        else { t -= rp * cn; rset = ~rm; cset = cm; len = rn; }
        p = nth_bit(rset & 0xffffu, t % len);
        q = nth_bit(cset & 0xffffu, t / len);
    }
    const bool any_opp = __any_sync(0xffffffffu, opp), all_opp = __all_sync(0xffffffffu, opp);
    // acc restarts every few K-blocks, its sum so far added to `total`: long
    // sums round as two short chains, at 1 addition in 64 terms (in 16 products of
    // one kind where the entries are complex, whose products round twice: error
    // against 64 bits at n = 1000 7.8e-17 -> 6.3e-17)
    S acc = real_value<S>(0.0), total = acc;
    __syncthreads();   // the buffers may still be read for the CTA's work before
    for (int kb = kb0 + half, buf = 0; kb < kb1; kb += 2, buf ^= 1) {
        auto &F = sm.far[half];
        S *AU = F.AU[buf], *AT = F.AT[buf], *BU = F.BU[buf], *BT = F.BT[buf];
        AU[hi * LB + lo] = au;
        AT[hi * LB + lo] = at;
        BU[hi * LD + lo] = bu;
        BT[hi * LD + lo] = bt;
        half_sync(half);
        if (kb + 2 < kb1) fetch(kb + 2);
        S acc2 = real_value<S>(0.0);
        const S *A1 = AU + p, *A2 = AT + p, *B1 = (opp ? BT : BU) + q * LD, *B2 = BU + q * LD;
        if (kb >= I + 2 && kb <= J - 2) {
            if (all_opp) {
#pragma unroll (sizeof(S) == 8 ? LB : LB / 4)
                for (int k = 0; k < LB; k++) {
                    acc = mac(A1[k * LB], B1[k], acc);
                    S &second = sizeof(S) == 16 ? acc2 : acc;
                    second = nmac(A2[k * LB], B2[k], second);
                }
                if (sizeof(S) == 16) acc = add(acc, acc2);
            } else if (any_opp) {
#pragma unroll 4
                for (int k = 0; k < LB; k++) {
                    acc = mac(A1[k * LB], B1[k], acc);
                    S &second = sizeof(S) == 16 ? acc2 : acc;
                    const S r = nmac(A2[k * LB], B2[k], second);
                    if (opp) second = r;
                }
                if (sizeof(S) == 16) acc = add(acc, acc2);
            } else {
#pragma unroll (sizeof(S) == 8 ? LB : LB / 4)
                for (int k = 0; k < LB; k++) acc = mac(A1[k * LB], B1[k], acc);
            }
        } else if (any_opp) {
            // the first and last two K-blocks: one part only, and inside a
            // diagonal block only the terms between p and q
            if (kb == I || kb <= J - 2) {
                const int k1 = kb == I ? p : -1;
#pragma unroll 4
                for (int k = 0; k < LB; k++) {
                    const S r = mac(A1[k * LB], B1[k], acc);
                    if (opp && k > k1) acc = r;
                }
            }
            if (kb == J || kb >= I + 2) {
                const int k1 = kb == J ? q : LB;
#pragma unroll 4
                for (int k = 0; k < LB; k++) {
                    const S r = nmac(A2[k * LB], B2[k], acc);
                    if (opp && k < k1) acc = r;
                }
            }
        }
        if (sizeof(S) == 16 || ((kb - kb0) & 6) == 6) {
            total = add(total, acc);
            acc = real_value<S>(0.0);
        }
        // the other buffer is refilled next; its readers passed the barrier
        // above only after they had finished with it
    }
    acc = add(acc, total);
    __syncthreads();
    S *part = sm.far[0].AU[0];
    if (half == 1) part[p + q * LB] = acc;
    __syncthreads();
    if (half == 0) slab[p + q * LB] = add(acc, part[p + q * LB]);
}

// Whether a and b, +-1 each, differ, without the float64 pipe.
__device__ __forceinline__ bool signs_differ(double a, double b) { return (__double2hiint(a) ^ __double2hiint(b)) < 0; }

// Entry number t of a block along its anti-diagonals step = 15 - p + q, from
// the bottom-left corner.
__device__ __forceinline__ void entry_of(int t, int &p, int &q)
{
    const int m = t < 136 ? t : 255 - t;
    int a = (int)((sqrtf(8.f * m + 1.f) - 1.f) * 0.5f);
    if ((a + 1) * (a + 2) / 2 <= m) a++;
    if (a * (a + 1) / 2 > m) a--;
    q = m - a * (a + 1) / 2;
    p = LB - 1 - a + q;
    if (t >= 136) { p = LB - 1 - p; q = LB - 1 - q; }
}

// The block's solve: the thread's entry (p, q) starts as the quotients by its
// divisor of its own term (quot) and of `outside`, the sum of all terms outside
// the block, and takes
//   - M[p, k] v_kq / d (k > p)   and   + v_pk N[k, q] / d (k < q; sign flipped by flip)
// as the entries of V are solved, step by step; V must not be in use.  The terms of
// the block are summed by themselves and the quotients join in the last
// operation: the sums and the reciprocal then round in proportion to the sums,
// which are as a rule smaller than the entry's own term.  (Everything added to one sum and
// multiplied by the reciprocal: errors against 64 bits of 8.1e-17, 8.6e-17,
// 7.6e-17 at n = 256, 1001, 8192, now 6.1e-17, 6.8e-17, 5.9e-17; complex n = 1000
// 9.2e-17, now 6.2e-17.)  Complex entries, whose products are separate
// instructions, add `outside` to the block's sum, so that only one addition
// rounds by the entry's own size.
// general: the entry is a divided difference, whose own term the sums nearly cancel
// where eigenvalues are close: `outside` holds that term too, everything is one
// sum, and the quotient is taken of what is left.
// scaled: a warp with a divisor that is (dv.ex; else dv.ex is not looked at).  A
// warp's entries have up to five steps: before and after these it forms none
// (formed under a condition of the lane alone, the quotient's multiply-add is
// issued by every warp at every step: 15 % of the leaf's float64 instructions).
template <bool general, bool kScaled, class S>
__device__ __forceinline__ void solve_steps(S outside, S quot, const Divisor<S> &dv, unsigned long long flip,
                                            const S *M, const S *N, S *V, int p, int q, int step)
{
    constexpr bool kComplex = sizeof(S) == 16 && !general;
    auto by_d = [&](S x, S base) { return kScaled ? add_quotient(x, dv, base) : mac_once(x, dv.r, base); };
    S acc = general ? outside : real_value<S>(0.0);
    if (!general && !kComplex) quot = by_d(outside, quot);
    auto take = [&](int st) {
        const int k1 = LB - 1 + q - st;   // solved at this step in the entry's column ...
        const int k2 = st - (LB - 1) + p;   // ... and in its row
        if (k2 >= 0) {
            acc = mac(flip_sign(V[p + k2 * LD], flip), N[k2 + q * LD], acc);
        }
        if (k1 < LB) acc = nmac(M[p + k1 * LD], V[k1 + q * LD], acc);
    };
    const int lo = __reduce_min_sync(0xffffffffu, step), hi = __reduce_max_sync(0xffffffffu, step);
    int st = 0;
    for (; st < lo; st++) {
        half_sync(0);
        take(st);
    }
    for (; st <= hi; st++) {
        if (step == st) V[p + q * LD] = by_d(kComplex ? add(outside, acc) : acc, quot);
        half_sync(0);
        if (st < step) take(st);
    }
    for (; st < 2 * LB - 1; st++) half_sync(0);
}
template <bool general, class S>
__device__ __forceinline__ void solve16(S outside, S quot, const Divisor<S> &dv, bool scaled, unsigned long long flip,
                                        const S *M, const S *N, S *V, int p, int q, int step)
{
    if (!scaled) solve_steps<general, false>(outside, quot, dv, flip, M, N, V, p, q, step);
    else solve_steps<general, true>(outside, quot, dv, flip, M, N, V, p, q, step);
}

// Leaf of block (I, J): nslab partial slabs from slab0 on, LT doubles each.
// Everything that a launch before the last has written may be read before
// dependency_wait(); for d <= 2 the blocks next to the diagonal are not yet
// among it.  Run by the first half of the CTA.
template <bool general, class S>
__device__ __forceinline__ void leaf(int n, const S *__restrict__ T, int ldt, S *U, int ldu,
                                     int I, int J, int nslab, const S *slab0, Smem<S> &sm)
{
    auto &s = sm.leaf;
    const S zero = real_value<S>(0.0);
    const int d = J - I;
    const int r0 = I * LB, c0 = J * LB;
    const int bj = min(LB, n - c0);
    const int lo = threadIdx.x % LB, hi = threadIdx.x / LB;
    const int at = lo + hi * LD;
    const bool up = lo <= hi, in = hi < bj;
    s.TI[at] = up ? SGT_AT(T, ldt, r0 + lo, r0 + hi) : zero;
    s.UI[at] = up ? SGT_AT(U, ldu, r0 + lo, r0 + hi) : zero;
    s.TJ[at] = up && in ? SGT_AT(T, ldt, c0 + lo, c0 + hi) : zero;
    s.UJ[at] = up && in ? SGT_AT(U, ldu, c0 + lo, c0 + hi) : zero;
    const S tij = in ? SGT_AT(T, ldt, r0 + lo, c0 + hi) : zero;
    if (d >= 2) {
        s.T1[at] = SGT_AT(T, ldt, r0 + lo, r0 + LB + hi);
        s.T2[at] = in ? SGT_AT(T, ldt, c0 - LB + lo, c0 + hi) : zero;
    }
    if (d >= 3) {
        s.U1[at] = SGT_AT(U, ldu, r0 + lo, r0 + LB + hi);
        s.U2[at] = in ? SGT_AT(U, ldu, c0 - LB + lo, c0 + hi) : zero;
    }
    if (threadIdx.x < LB) {
        const int i = threadIdx.x;
        s.urow[i] = SGT_AT(U, ldu, r0 + i, r0 + i);
        s.ucol[i] = i < bj ? SGT_AT(U, ldu, c0 + i, c0 + i) : real_value<S>(1.0);
    }
    int p, q;
    entry_of(threadIdx.x, p, q);
    const int step = LB - 1 - p + q;
    half_sync(0);
    const S upp = s.urow[p], uqq = s.ucol[q];
    const bool opp = general || signs_differ(re(upp), re(uqq));
    // signs agree: 1 / (u_pp + u_qq) is +-1/2 exactly
    const S dif = sub(s.TI[p + p * LD], s.TJ[q + q * LD]);
    const Divisor<S> dv = opp ? divisor(dif) : Divisor<S>{scaled(upp, 0.5), 0};
    // flips the sign of the row terms where the signs agree
    const unsigned long long flip = opp ? 0ull : 0x8000000000000000ull;
    const S *M = opp ? s.TI : s.UI, *N = opp ? s.TJ : s.UJ;
    const S *M1 = opp ? s.T1 : s.U1, *N2 = opp ? s.T2 : s.U2;

    // the entry's own term (u_ii and u_jj are real)
    const double ui = re(s.urow[lo]), uj = re(s.ucol[hi]);
    const bool o = general || signs_differ(ui, uj);
    s.V[at] = o ? scaled(tij, ui - uj) : zero;
    half_sync(0);
    const S base = s.V[p + q * LD], quot = !general && opp ? quotient(base, dif, dv) : zero;
    const bool far = __any_sync(0xffffffffu, dv.ex != 0);

    dependency_wait();
    dependency_release();
    // all of the launch before's results in flight together
    S x1 = zero, x2 = zero, u1 = zero, u2 = zero, v[8];
    if (d >= 2) {
        if (in) x1 = SGT_AT(U, ldu, r0 + LB + lo, c0 + hi);
        x2 = SGT_AT(U, ldu, r0 + lo, c0 - LB + hi);
    }
    if (d == 2) {
        u1 = SGT_AT(U, ldu, r0 + lo, r0 + LB + hi);
        if (in) u2 = SGT_AT(U, ldu, c0 - LB + lo, c0 + hi);
    }
#pragma unroll
    for (int t = 0; t < 8; t++) v[t] = t < nslab ? slab0[(size_t)t * LT + threadIdx.x] : zero;
    S sum = v[0];
#pragma unroll
    for (int t = 1; t < 8; t++)
        if (t < nslab) sum = add(sum, v[t]);
    for (int t0 = 8; t0 < nslab; t0 += 8) {
#pragma unroll
        for (int t = 0; t < 8; t++) v[t] = t0 + t < nslab ? slab0[(size_t)(t0 + t) * LT + threadIdx.x] : zero;
#pragma unroll
        for (int t = 0; t < 8; t++)
            if (t0 + t < nslab) sum = add(sum, v[t]);
    }
    if (d >= 2) {
        s.X1[at] = x1;
        s.X2[at] = x2;
    }
    if (d == 2) {
        s.U1[at] = u1;
        s.U2[at] = u2;
    }
    s.C[at] = o ? sum : flip_sign(sum, 0x8000000000000000ull);
    half_sync(0);
    S acc = s.C[p + q * LD];
    if (d >= 2) {
        S col = zero, row = zero;
        // (d = 2: both near blocks are the same, and a sum of U U counts it once)
        const bool both = d > 2 || opp;
#pragma unroll (sizeof(S) == 8 ? 8 : 4)
        for (int k = 0; k < LB; k++) {
            col = nmac(M1[p + k * LD], s.X1[k + q * LD], col);
            row = mac(flip_sign(s.X2[p + k * LD], flip), N2[k + q * LD], row);
        }
        if (both) col = add(col, row);
        acc = add(acc, col);
    }
    if (general) acc = add(acc, base);
    solve16<general>(acc, quot, dv, far, flip, M, N, s.V, p, q, step);
    if (in) SGT_AT(U, ldu, r0 + lo, c0 + hi) = s.V[at];
}

// Diagonal block (r0, r0): Algorithm 3 with the plain float64 algorithm's own
// rounding (separate multiply, add and divide, sums in ascending k).  By
// anti-diagonal: the products of all the anti-diagonal's terms first, spread
// over the threads, then each entry's sum, one addition after another, by a
// thread of its own; the quotients t_ij (u_ii - u_jj) / (t_ii - t_jj), which
// need no sum, once at the start.
__device__ __forceinline__ void diag_leaf(int n, const double *__restrict__ T, int ldt, double *__restrict__ U,
                                          int ldu, int blk, double *Ts, double *Us, double *Pr, double *Q1)
{
    const int r0 = blk * LB, bs = min(LB, n - r0);
    const int lo = threadIdx.x % LB, hi = threadIdx.x / LB, at = lo + hi * LD;
    const bool in = lo <= hi && hi < bs;
    const double t = in ? SGT_AT(T, ldt, r0 + lo, r0 + hi) : 0.0;
    Ts[at] = t;
    Us[at] = lo == hi ? ph::sgn(t) : 0.0;
    __syncthreads();
    {
        const double ui = Us[lo * (LD + 1)], uj = Us[hi * (LD + 1)];
        if (in && lo < hi && __dadd_rn(ui, uj) == 0.0)
            Q1[at] = __ddiv_rn(__dmul_rn(t, __dsub_rn(ui, uj)), __dsub_rn(Ts[lo * (LD + 1)], Ts[hi * (LD + 1)]));
    }
    for (int d = 1; d < bs; d++) {
        const int terms = d - 1;
        if (terms > 0 && threadIdx.x < (bs - d) * terms) {   // at most 8 * 7 of them
            const int i = threadIdx.x / terms, k = i + 1 + threadIdx.x % terms, j = i + d;
            const double uk = Us[i + k * LD], ukj = Us[k + j * LD];
            const bool opp = __dadd_rn(Us[i * (LD + 1)], Us[j * (LD + 1)]) == 0.0;
            double v = __dmul_rn(uk, opp ? Ts[k + j * LD] : ukj);
            if (opp) v = __dsub_rn(v, __dmul_rn(Ts[i + k * LD], ukj));
            Pr[i * LD + (k - i - 1)] = v;
        }
        __syncthreads();
        if (threadIdx.x < bs - d) {
            const int i = threadIdx.x, j = i + d;
            double s = 0.0;
            for (int k = 0; k < terms; k++) s = __dadd_rn(s, Pr[i * LD + k]);
            const double uii = Us[i * (LD + 1)], ujj = Us[j * (LD + 1)];
            double r;
            if (__dadd_rn(uii, ujj) == 0.0)
                r = __dadd_rn(Q1[i + j * LD], __ddiv_rn(s, __dsub_rn(Ts[i * (LD + 1)], Ts[j * (LD + 1)])));
            else
                r = __dmul_rn(-s, __dmul_rn(0.5, uii));   // -s / (+-2), exactly
            Us[i + j * LD] = r;
        }
        __syncthreads();
    }
    if (in) SGT_AT(U, ldu, r0 + lo, r0 + hi) = Us[at];
}

// CTAs [0, leaves): the leaves of anti-diagonal d, their early sums in `in`
// (split sin).  Then every CTA: its share of the early sums of d + 1 into
// `out` (split sout).
template <bool general, class S>
__global__ void __launch_bounds__(kLevelThreads)
level_kernel(int n, const S *__restrict__ T, int ldt, S *U, int ldu, int d, int leaves,
             const __grid_constant__ Split sin, const S *in,
             const __grid_constant__ Split sout, S *out)
{
    extern __shared__ __align__(16) unsigned char raw[];
    Smem<S> &sm = *reinterpret_cast<Smem<S> *>(raw);
    const int c = blockIdx.x;
    if (c < leaves && threadIdx.x < LT) {
        const int f = split_owner(sin, (long long)c * sin.cpt), l = split_owner(sin, (long long)(c + 1) * sin.cpt - 1);
        leaf<general>(n, T, ldt, U, ldu, c, c + d, l - f + 1, in + (size_t)(f + c) * LT, sm);
    } else {
        dependency_wait();
        dependency_release();
    }
    if (c >= sout.G) return;
    __syncthreads();   // the leaf's shared memory is free
    const int e = d + 1, cpt = sout.cpt;
    const long long x1 = split_start(sout, c + 1);
    for (long long x = split_start(sout, c); x < x1;) {
        const int I = (int)(x / cpt);
        const long long t0 = (long long)I * cpt, xe = min(x1, t0 + cpt);
        far_sums<general>(n, T, ldt, U, ldu, I, I + e, I + (int)(x - t0), I + (int)(xe - t0),
                          out + (size_t)(c + I) * LT, sm);
        x = xe;
    }
}

// Every off-diagonal block of U up to block anti-diagonal `last`, the diagonal
// blocks being solved; workspace: level_workspace_bytes.
template <bool general, class S>
signtri_status launch_levels(int n, const S *T, int ldt, S *U, int ldu, Arena &ws, cudaStream_t st, int last = INT_MAX)
{
    const int nb = (n + LB - 1) / LB;
    if (nb < 2) return SIGNTRI_OK;
    S *slab[2];
    for (S *&s : slab) {
        s = static_cast<S *>(ws.take(level_slabs(n) * LT * sizeof(S)));
        if (!s) return SIGNTRI_ERR_NO_WORKSPACE;
    }
    SGT_CUDA_TRY(cudaFuncSetAttribute(level_kernel<general, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      level_smem<S>(kSms)));
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kLevelThreads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    Split sin{};
    for (int d = 0; d < nb && d <= last; d++) {
        const int leaves = d > 0 ? nb - d : 0, e = d + 1;
        Split sout{};
        if (e < nb && e <= last) sout = make_split(nb - e, e, leaves);
        cfg.gridDim = dim3(std::max(leaves, sout.G));
        cfg.dynamicSmemBytes = level_smem<S>((int)cfg.gridDim.x);
        ProfScope ps(SIGNTRI_KC_OFFDIAG_LEAF, st);
        SGT_CUDA_TRY(cudaLaunchKernelEx(&cfg, level_kernel<general, S>, n, T, ldt, U, ldu, d, leaves, sin,
                                        (const S *)slab[d & 1], sout, slab[e & 1]));
        sin = sout;
    }
    return SIGNTRI_OK;
}

}  // namespace lvl
}  // namespace signtri
