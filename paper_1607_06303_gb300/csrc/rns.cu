// rns.cu -- float64 products on the tensor cores through residues.
//
// GB300 multiplies float64 at 1.2 TFLOP/s and bf16 at 1.9 PFLOP/s.  A product
// of integers is formed here modulo 18 pairwise coprime numbers up to 256
// (the residue number system; Garner, "The residue number system", IRE Trans.
// EC-8, 1959; for matrix products Ozaki, Uchino and Imamura, "Ozaki scheme
// II", 2025): residues between -128 and 128 are exact in bf16, and a sum of
// 960 of their products is an integer below 2^24, exact in the tensor
// cores' fp32 accumulators.  Entries are first rounded to integers of 62
// bits under a power-of-two scale per row of the left operand and per column
// of the right; the integer product, below half the moduli's product, comes
// back from its residues by the Chinese remainder theorem.  So the only error
// is that of rounding the entries to 2^-63 of their scale; the sums are exact.
//
// 18 products instead of the 36 of eight 7-bit slices, and independent ones:
// a 128 x 128 tile is 18 tasks, so a few tiles already fill the GPU.
//
// rns_gemm_kernel: persistent CTAs; a task is one (tile, modulus).  Warp 0
// loads K-blocks of 64 of both panels, 16 KB each, stored in the swizzled
// layout so that a plain bulk copy brings them, into a ring of 4; one thread
// of warp 1 issues M = N = 128 MMAs into 4 TMEM buffers, one per up to 15
// K-blocks; 8 warps drain them, reduce modulo m and add.  Bound by the
// operands' bytes (32 KB per K-block and 2 x 128^2 x 64 operations).
#include <algorithm>

#include "rns.cuh"
#include "tc_ptx.cuh"

namespace signtri {
namespace rns {

namespace {

constexpr int kStages = 4;      // leaves shared memory for the kernels this one runs beside
constexpr int kStageBytes = 32768;
constexpr int kThreads = 320;   // and at most 102 registers each: room for two CTAs of the waves beside it
constexpr int kBufs = 4;
// CTAs of an early launch, which runs beside another kernel: half the SMs keep
// up with memory (n = 8192 in all: 152 CTAs 40.2 ms, 100 37.4, 84 37.1, 76 36.3,
// 64 37.5, 48 43.8)
constexpr int kEarlyCtas = 76;
constexpr int kChunkKb = 15;    // 960 products of residues of at most 129: below 2^24
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256;

// kind::f16, D fp32, A and B bf16, K-major, N = M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

constexpr int inv_mod(int a, int m)
{
    a %= m;
    for (int x = 1; x < m; x++)
        if (a * x % m == 1) return x;
    return 0;
}
// the inverse of P / m_i modulo m_i
constexpr int cofactor_inverse(int i)
{
    int r = 1;
    for (int j = 0; j < kMods; j++)
        if (j != i) r = r * (kModulus[j] % kModulus[i]) % kModulus[i];
    return inv_mod(r, kModulus[i]);
}
struct GemmConst {
    float m[kMods], rm[kMods], inv[kMods];
};
constexpr GemmConst make_gemm_const()
{
    GemmConst c{};
    for (int i = 0; i < kMods; i++) {
        c.m[i] = (float)kModulus[i];
        c.rm[i] = 1.f / (float)kModulus[i];
        c.inv[i] = (float)cofactor_inverse(i);
    }
    return c;
}
__constant__ GemmConst c_gemm = make_gemm_const();

// x - m rint(x / m) for integers |x| <= 2^24: within m / 2 of 0 (the
// quotient's rounding can only move a tie)
__device__ __forceinline__ float reduce(float x, float m, float rm)
{
    const float q = __fsub_rn(__fmaf_rn(x, rm, 12582912.f), 12582912.f);
    return __fmaf_rn(-q, m, x);
}

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint64_t *bar, uint32_t bytes)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Bounded wait without the abort flag, for draining.
__device__ __forceinline__ void mbar_drain(uint64_t *bar, uint32_t parity)
{
    const uint32_t a = smem_u32(bar);
    const long long t0 = clock64();
    while (clock64() - t0 < kWaitCycles) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) break;
    }
}

// The K-blocks of a task: n0 from a0 on, then the rest from a1 on.
struct Span {
    int a0, n0, a1, n;
    bool ahead;   // the others are summed already
    __device__ __forceinline__ int operator[](int i) const { return i < n0 ? a0 + i : a1 + i - n0; }
};
__device__ __forceinline__ Span span_of(const Tile &t, const Source &s, bool early, bool ahead)
{
    const int n = max(t.e1 - t.e0, 0);
    if (early) return {t.e0, n, 0, n, false};
    if (!ahead || n == 0 || (s.grownA && s.grownA[t.pa]) || (s.grownB && s.grownB[t.pb])) {
        const int all = max(t.kb1 - t.kb0, 0);
        return {t.kb0, all, 0, all, false};
    }
    return {t.kb0, t.e0 - t.kb0, t.e1, t.e0 - t.kb0 + t.kb1 - t.e1, true};
}

struct Task {
    int tile, mod;
};
__device__ __forceinline__ Task task_of(int id, int per)
{
    return {id / (per * kMods) * per + id % per, id / per % kMods};
}

__global__ void __launch_bounds__(kThreads, 2)
rns_gemm_kernel(const Source *__restrict__ src, const Tile *__restrict__ tiles, int ntasks, int per, bool early,
                const int8_t *__restrict__ ahead, int8_t *__restrict__ out, int *__restrict__ err)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes);
    uint64_t *empty = full + kStages;
    uint64_t *tfull = empty + kStages;
    uint64_t *tempty = tfull + kBufs;
    uint64_t *done_bar = tempty + kBufs;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(done_bar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < kBufs; b++) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 8); }
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_holder))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = *tmem_holder;

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            long long issued = 0;
            bool ok = true;
            for (int id = blockIdx.x; id < ntasks && ok; id += gridDim.x) {
                const Task k = task_of(id, per);
                const Tile t = tiles[k.tile];
                const Source s = src[t.src];
                const __nv_bfloat16 *a = s.A + s.la.tile(t.pa, k.mod, 0) * kTileElems;
                const __nv_bfloat16 *b = s.B + s.lb.tile(t.pb, k.mod, 0) * kTileElems;
                const Span ks = span_of(t, s, early, ahead != nullptr);
                for (int i = 0; i < ks.n; i++) {
                    const int kb = ks[i];
                    if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
                    unsigned char *base = smem + stage * kStageBytes;
                    mbar_expect_tx(&full[stage], kStageBytes);
                    bulk_load(base, a + (size_t)kb * kTileElems, &full[stage], kStageBytes / 2);
                    bulk_load(base + kStageBytes / 2, b + (size_t)kb * kTileElems, &full[stage], kStageBytes / 2);
                    issued++;
                    if (++stage == kStages) { stage = 0; phase ^= 1; }
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(err, 1);
                // drain: wait (bounded) for the loads of the last stages issued
                const long long tail = issued < kStages ? issued : kStages;
                for (long long i = 0; i < tail; i++) {
                    if (stage == 0) { stage = kStages - 1; phase ^= 1; } else stage--;
                    mbar_drain(&full[stage], phase);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int stage = 0, g = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int id = blockIdx.x; id < ntasks && ok; id += gridDim.x) {
                const Tile t = tiles[task_of(id, per).tile];
                const Span ks = span_of(t, src[t.src], early, ahead != nullptr);
                for (int kc = 0; kc < ks.n && ok; kc += kChunkKb, g++) {
                    const int buf = g % kBufs;
                    if (!mbar_wait(&tempty[buf], (uint32_t)((g / kBufs) & 1) ^ 1, abort_flag)) { ok = false; break; }
                    fence_after();
                    const uint32_t d = tmem_base + (uint32_t)(buf * 128);
                    const int ke = min(kc + kChunkKb, ks.n);
                    for (int kb = kc; kb < ke; kb++) {
                        if (!mbar_wait(&full[stage], phase, abort_flag)) { ok = false; break; }
                        fence_after();
                        unsigned char *base = smem + stage * kStageBytes;
                        const uint64_t ad = smem_desc(base), bd = smem_desc(base + kStageBytes / 2);
#pragma unroll
                        for (int k = 0; k < 4; k++)
                            mma_bf16(d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), kIdesc,
                                     (kb > kc || k > 0) ? 1u : 0u);
                        mma_commit(&empty[stage]);
                        if (++stage == kStages) { stage = 0; phase ^= 1; }
                    }
                    if (!ok) break;
                    mma_commit(&tfull[buf]);
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(err, 1);
            }
            // arrives once every MMA issued by this thread has completed
            mma_commit(done_bar);
        }
    } else {
        const int q = warp & 3;                 // TMEM lane quadrant this warp may read
        const int cg = (warp - 2) >> 2;         // 64-column group 0, 1
        const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(cg * 64);
        bool ok = true;
        int g = 0;
        for (int id = blockIdx.x; id < ntasks && ok; id += gridDim.x) {
            const Task k = task_of(id, per);
            const Tile t = tiles[k.tile];
            const float m = c_gemm.m[k.mod], rm = c_gemm.rm[k.mod], inv = c_gemm.inv[k.mod];
            const Span ks = span_of(t, src[t.src], early, ahead != nullptr);
            if (early && ks.n == 0) continue;
            const size_t at = (((size_t)k.tile * kMods + k.mod) * kPanel + 32 * q + lane) * kPanel + 64 * cg;
            float acc[64];
            if (ks.ahead) {
                const char4 *h = reinterpret_cast<const char4 *>(ahead + at);
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const char4 c = h[i];
                    acc[4 * i] = (float)(signed char)c.x;
                    acc[4 * i + 1] = (float)(signed char)c.y;
                    acc[4 * i + 2] = (float)(signed char)c.z;
                    acc[4 * i + 3] = (float)(signed char)c.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 64; i++) acc[i] = 0.f;
            }
            for (int kc = 0; kc < ks.n && ok; kc += kChunkKb, g++) {
                const int buf = g % kBufs;
                if (!mbar_wait(&tfull[buf], (uint32_t)((g / kBufs) & 1), abort_flag)) { ok = false; break; }
                fence_after();
#pragma unroll
                for (int cc = 0; cc < 64; cc += 16) {
                    uint32_t r[16];
                    tmem_ld16_nowait(lane_base + (uint32_t)(buf * 128 + cc), r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 16; i++) acc[cc + i] += reduce(__uint_as_float(r[i]), m, rm);
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[buf]);
            }
            if (!ok) break;
            int4 v[4];
            int *w = reinterpret_cast<int *>(v);
#pragma unroll
            for (int i = 0; i < 64; i += 4) {
                unsigned x = 0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    float y = reduce(acc[i + j], m, rm);
                    if (!early) y = reduce(__fmul_rn(y, inv), m, rm);
                    x |= ((unsigned)(int)y & 0xffu) << (8 * j);
                }
                w[i / 4] = (int)x;
            }
            int4 *o = reinterpret_cast<int4 *>(out + at);
#pragma unroll
            for (int i = 0; i < 4; i++) o[i] = v[i];
        }
        if (!ok) {
            *abort_flag = 1;
            atomicExch(err, 1);
        }
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        mbar_drain(done_bar, 0);   // completes once, when all MMAs of this CTA have finished
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

}  // namespace

signtri_status gemm(const Source *d_src, const Tile *d_tiles, int ntiles, int per, bool early, int8_t *ahead,
                    int8_t *out, int *d_err, int cls, cudaStream_t st)
{
    if (ntiles <= 0) return SIGNTRI_OK;
    SGT_CUDA_TRY(cudaFuncSetAttribute(rns_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
    const int ntasks = ntiles * kMods;
    ProfScope ps(cls, st);
    rns_gemm_kernel<<<std::min(ntasks, early ? kEarlyCtas : 152), kThreads, kSmemBytes, st>>>(
        d_src, d_tiles, ntasks, per, early, early ? nullptr : ahead, early ? ahead : out, d_err);
    SGT_LAUNCH_CHECK();
    return SIGNTRI_OK;
}

}  // namespace rns
}  // namespace signtri
