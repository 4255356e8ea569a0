// FP64-accurate GEMM on the BF16 tensor cores of sm_103a (tcgen05), by exact
// integer slicing (the error-free splitting scheme of Ozaki, Ogita, Oishi and
// Rump, 2012).
//
//   C = alpha * op(A) * diag(kscale) * op(B) + beta * Cin        (FP64 data)
//
// 1. Every row i of op(A) is scaled by 2^{-e_i} and every column j of op(B)
//    by 2^{-f_j} (exact) so that all entries lie in (-1, 1).
// 2. Each scaled entry x is rounded to F = round(x 2^56) (error <= 2^-57)
//    and F is cut into S = 8 integer digits of 7 bits, balanced base 128:
//      x ~ sum_t d_t 2^{-7t},  |d_1| <= 128,  |d_t| <= 64 (t > 1);
//    the d_t are exact in BF16.  (Integer work only: FP64 arithmetic is a
//    slow pipe on this part.)
// 3. For every level L = a + b (2 <= L <= S+1) the slice products
//    sum_{a+b=L} D^A_a D^B_b are integers; one term is at most
//    2^14 + max(0, L-3) 2^12 (two products with a slice d_1, the rest 2^12).
//    Over a 512-term stretch of k the levels L <= 7 stay at or below 2^24, so
//    the tensor cores' FP32 accumulation of them is exact.  Levels 8 and 9 can
//    pass 2^24 only when the (1, L-1) and (L-1, 1) products are near 2^13,
//    i.e. when the entries are near their row/column maxima; their rounding
//    (at most 512 units at weight 2^{-7L}) is then below 2^-55 of
//    sum_p |a_ip b_pj|.  Each level has its own accumulator in tensor memory
//    (8 levels x 64 columns = all 512).
// 4. Every 512 terms of k the eight level sums are scaled by 2^{-7L} (exact)
//    and added into a float-pair (TwoSum) accumulator per output; at the end
//    C = alpha 2^{e_i + f_j} (hi + lo) + beta Cin in FP64.
// Products with a + b > S + 1 (36 of 64 kept) are dropped.  Level L = a + b
// carries weight 2^{-7L} and its terms are at most 2^12 (2^14 with a d_1 slice),
// so the first dropped level (L = 10, seven products) contributes up to about
// 7 * 2^12 * 2^-70 ~ 2^-55 of the row/column maxima per term, and the levels
// beyond it less: the dropped part is ~2^-55 relative to sum_p |a_ip||b_pj| in
// the worst case (the measured error is 0.9-1.7e-15 of that sum).
//
// Kernel layout: one CTA of 18 warps per 128 x 64 output tile, warp-specialised:
// warp 16 streams the 8 A-slice tiles (128 x 16 BF16) and 8 B-slice tiles
// (64 x 16) of one k block, stored pre-tiled and pre-swizzled (32-byte swizzle)
// by the slicing pass, as two contiguous bulk copies into a 4-stage mbarrier ring; warp 17 issues 12
// tcgen05.mma kind::f16 (M=128, N=64..256, K=16) per stage, which cover the 36
// slice products, into 8 accumulators of 64 TMEM columns and frees each stage
// with tcgen05.commit; warps 0-15 flush the accumulators every 512 terms
// (warp w reads TMEM lanes 32 (w % 4) .. and 16 columns per level, so four
// warps per SM sub-partition hide the TwoSum latency) while the producer keeps
// prefetching, then signal the MMA warp that the accumulators are free.
// Every pipeline mbarrier wait is bounded by the caller's limit (error flag,
// then the kernel waits -- under a fixed, longer bound -- for its own bulk
// copies and MMAs in flight, frees TMEM and returns).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "mbar.cuh"
#include "pssd_internal.h"

namespace pssd {

namespace {

constexpr int OZ_S = 8;                    // slices
constexpr int OZ_LEVELS = OZ_S;            // levels L = 2 .. S+1
constexpr int OZ_BM = 128, OZ_BN = 64, OZ_BK = 16;   // BK in BF16 elements = 32 bytes = one MMA K
constexpr int OZ_STAGES = 4;
constexpr int OZ_CHUNK_STAGES = 32;        // flush every 32 x 16 = 512 terms of k
constexpr int OZ_A_TILE = OZ_BM * OZ_BK * 2;          // 4 KB
constexpr int OZ_B_TILE = OZ_BN * OZ_BK * 2;          // 2 KB
constexpr int OZ_STAGE_BYTES = OZ_S * (OZ_A_TILE + OZ_B_TILE);   // 48 KB
constexpr int OZ_SMEM_BYTES = OZ_STAGES * OZ_STAGE_BYTES + 1024 + 256;
constexpr unsigned long long OZ_WAIT_LIMIT = 1ull << 26;   // default pipeline bound and the drain bound
constexpr int OZ_TMEM_COLS = 512;
constexpr int OZ_FLUSH_WARPS = 16;         // warp w: TMEM lanes 32 (w % 4) .., columns 16 (w / 4) ..
constexpr int OZ_FCOLS = OZ_BN / (OZ_FLUSH_WARPS / 4);   // 16 output columns per flush thread
constexpr int OZ_PRODUCER_WARP = OZ_FLUSH_WARPS, OZ_MMA_WARP = OZ_FLUSH_WARPS + 1;
constexpr int OZ_THREADS = 32 * (OZ_FLUSH_WARPS + 2);
constexpr int OZ_GROUP_M = 8;              // row blocks per group of the tile order

struct OzArgs {
    // slices, tiled: block (z, row tile, k block) = 8 slices x tile rows x 16 k,
    // 32-byte-swizzled rows, contiguous (32 KB for A, 16 KB for B): one copy per operand and k
    // block (with one copy per slice, 16 in all, a 4096^3 product took 3.32 ms instead of 2.73)
    const __nv_bfloat16 *sa, *sb;
    int kblocks;                           // k_pad / 16
    int m, n, k, batch, m_pad, n_pad;
    int triA, triB, lowerC;
    const int *ea, *eb;                    // exponents per row of op(A) (batch*m_pad), per column of op(B)
    double *C; long long ldc, sC;
    const double *Cin; long long ldcin, sCin;
    double alpha, beta;
    int alpha_e, alpha_e_valid, alpha_neg;   // alpha = (-1)^neg 2^alpha_e when valid
    int *err;
    unsigned long long wait_limit;         // polls per pipeline wait before giving up
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"((unsigned long long)src), "r"(bytes), "r"(bar)
        : "memory");
}

// K-major operand, 32-byte swizzle: rows of 32 bytes, 8-row groups 256 bytes apart
__device__ __forceinline__ unsigned long long smem_desc_sw32(uint32_t addr)
{
    unsigned long long d = 0;
    d |= (unsigned long long)((addr >> 4) & 0x3FFF);
    d |= (unsigned long long)(16 >> 4) << 16;
    d |= (unsigned long long)(256 >> 4) << 32;
    d |= 1ull << 46;
    d |= 6ull << 61;                       // 32-byte swizzle
    return d;
}

// kind::f16, D = F32, A = B = BF16, both K-major, M = 128, N = 64 .. 256
__host__ __device__ constexpr uint32_t oz_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_BM >> 4) << 24);
}

// one product of stacked slices; the descriptors' low words and their common high word
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t dhi, uint32_t idesc,
                                         uint32_t acc, uint32_t pred)
{
    asm volatile(
        "{\n.reg .pred p, q;\n.reg .b64 da, db;\n"
        "setp.ne.b32 p, %5, 0;\nsetp.ne.b32 q, %6, 0;\n"
        "mov.b64 da, {%1, %3};\nmov.b64 db, {%2, %3};\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n}\n" ::"r"(tmem_d),
        "r"(alo), "r"(blo), "r"(dhi), "r"(idesc), "r"(acc), "r"(pred));
}

__device__ __forceinline__ void mma_commit_if(uint32_t bar, uint32_t pred)
{
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
        "r"(pred)
        : "memory");
}

// 1 in one lane of a converged warp
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t e;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
    return e;
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t *r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// float-pair accumulation (TwoSum, then renormalisation)
__device__ __forceinline__ void df_add(float &hi, float &lo, float x)
{
    float s = __fadd_rn(hi, x);
    float bp = __fsub_rn(s, hi);
    float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    float l = __fadd_rn(lo, e);
    float s2 = __fadd_rn(s, l);              // Fast2Sum renormalisation (|s| >= |l|)
    lo = __fsub_rn(l, __fsub_rn(s2, s));
    hi = s2;
}

// f 2^E as a double from the bit fields (exact); false when f is not a normal
// float or the result leaves the normal double range
__device__ __forceinline__ bool f2d_scaled(float f, int E, double &out)
{
    const uint32_t u = __float_as_uint(f);
    if ((u & 0x7FFFFFFFu) == 0) { out = 0.0; return true; }
    const int ef = (int)((u >> 23) & 0xFF);
    if (ef == 0 || ef == 255) return false;
    const int ed = ef - 127 + 1023 + E;
    if (ed < 1 || ed > 2046) return false;
    const unsigned long long b = ((unsigned long long)(u >> 31) << 63) | ((unsigned long long)ed << 52) |
                                 ((unsigned long long)(u & 0x7FFFFFu) << 29);
    out = __longlong_as_double((long long)b);
    return true;
}

__global__ void __launch_bounds__(OZ_THREADS, 1) oz_gemm_kernel(const __grid_constant__ OzArgs g)
{
    // grouped tile order: runs of OZ_GROUP_M row blocks sweep the column blocks
    // together, so the CTAs resident at one time share their A and B tiles in L2
    const int mt = (g.m + OZ_BM - 1) / OZ_BM, nt = (g.n + OZ_BN - 1) / OZ_BN;
    const int pid = blockIdx.x, per_group = OZ_GROUP_M * nt;
    const int first_m = (pid / per_group) * OZ_GROUP_M, gm = min(mt - first_m, OZ_GROUP_M);
    const int tm = first_m + (pid % per_group) % gm, tn = (pid % per_group) / gm;
    const int i0 = tm * OZ_BM, j0 = tn * OZ_BN, z = blockIdx.z;
    if (i0 >= g.m || j0 >= g.n) return;
    if (g.lowerC && j0 > i0 + OZ_BM - 1) return;

    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned long long *bars = (unsigned long long *)(smem + OZ_STAGES * OZ_STAGE_BYTES);
    // bars[0..ST): full, [ST..2ST): empty, [2ST]: chunk done (MMA -> flush), [2ST+1]: accumulators free
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * OZ_STAGES + 4);
    __shared__ int s_abort, s_issued;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    int kbeg = 0, kend = g.k;
    if (g.triA == TRI_LOWER) kend = min(kend, i0 + OZ_BM);
    if (g.triA == TRI_UPPER) kbeg = max(kbeg, i0);
    if (g.triB == TRI_LOWER) kbeg = max(kbeg, j0);
    if (g.triB == TRI_UPPER) kend = min(kend, j0 + OZ_BN);
    const int kb0 = kbeg / OZ_BK;
    const int nkb = (kend > kbeg) ? (kend + OZ_BK - 1) / OZ_BK - kb0 : 0;
    const int nchunks = (nkb + OZ_CHUNK_STAGES - 1) / OZ_CHUNK_STAGES;
    const uint32_t b_full = smem_u32(&bars[0]), b_empty = smem_u32(&bars[OZ_STAGES]);
    const uint32_t b_done = smem_u32(&bars[2 * OZ_STAGES]), b_free = smem_u32(&bars[2 * OZ_STAGES + 1]);
    const uint32_t b_drain = smem_u32(&bars[2 * OZ_STAGES + 2]);   // MMA drain after an abort

    if (tid == 0) {
        s_abort = 0;
        s_issued = 0;
        for (int s = 0; s < OZ_STAGES; ++s) {
            mbar_init(b_full + 8 * s, 1);
            mbar_init(b_empty + 8 * s, 1);
        }
        mbar_init(b_done, 1);
        mbar_init(b_free, 32 * OZ_FLUSH_WARPS);
        mbar_init(b_drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(OZ_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;

    if (warp == OZ_PRODUCER_WARP) {
        // ---------------- bulk-copy producer ----------------
        if (lane == 0) {
            const __nv_bfloat16 *srca = g.sa + (((long long)z * (g.m_pad / OZ_BM) + tm) * g.kblocks + kb0) *
                                                   (OZ_S * OZ_BM * OZ_BK);
            const __nv_bfloat16 *srcb = g.sb + (((long long)z * (g.n_pad / OZ_BN) + tn) * g.kblocks + kb0) *
                                                   (OZ_S * OZ_BN * OZ_BK);
            for (int q = 0; q < nkb; ++q) {
                const int s = q % OZ_STAGES;
                if (q >= OZ_STAGES &&
                    !mbar_wait(b_empty + 8 * s, (uint32_t)(((q / OZ_STAGES) - 1) & 1), g.wait_limit)) {
                    s_abort = 1; atomicExch(g.err, 1); break;
                }
                if (s_abort) break;
                const uint32_t st = smem_u32(smem + s * OZ_STAGE_BYTES);
                mbar_expect_tx(b_full + 8 * s, OZ_STAGE_BYTES);
                bulk_load(st, srca + (long long)q * (OZ_S * OZ_BM * OZ_BK), OZ_S * OZ_A_TILE, b_full + 8 * s);
                bulk_load(st + OZ_S * OZ_A_TILE, srcb + (long long)q * (OZ_S * OZ_BN * OZ_BK), OZ_S * OZ_B_TILE,
                          b_full + 8 * s);
                s_issued = q + 1;
            }
        }
    } else if (warp == OZ_MMA_WARP) {
        // ---------------- MMA issuer ----------------
        // The warp runs converged and one elected lane issues, so that the operands stay in
        // uniform registers: from a lane in a branch of its own a k block took 1500 clocks to
        // issue, more than its 36 products (1152).
        const uint32_t leader = elect_one();
        const uint32_t dhi = (uint32_t)(smem_desc_sw32(0) >> 32), dlo0 = (uint32_t)smem_desc_sw32(smem_u32(smem));
        bool ok = true;
        int s = 0;
        uint32_t phase = 0;
        for (int c = 0; c < nchunks && ok; ++c) {
            if (c > 0 && !mbar_wait(b_free, (uint32_t)((c - 1) & 1), g.wait_limit)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int q0 = c * OZ_CHUNK_STAGES, q1 = min(nkb, q0 + OZ_CHUNK_STAGES);
#pragma unroll 1
            for (int q = q0; q < q1; ++q) {
                if (!mbar_wait(b_full + 8 * s, phase, g.wait_limit)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t dlo = dlo0 + (uint32_t)(s * (OZ_STAGE_BYTES >> 4));
                const uint32_t fresh = q == q0 ? 0u : 1u;   // a = 1 reaches every level first
                // A slice a against B slices b = 1 .. S+1-a stacked along N: the product
                // (a, b) belongs to level a+b-2, whose accumulator starts at column
                // 64 (a+b-2), so slices b..b+3 form one N <= 256 MMA into consecutive levels.
#pragma unroll
                for (int a = 1; a <= OZ_S; ++a) {
#pragma unroll
                    for (int b0 = 1; b0 <= OZ_S + 1 - a; b0 += 4) {
                        const int nb = min(4, OZ_S + 2 - a - b0);
                        mma_bf16(tmem + (uint32_t)((a + b0 - 2) * OZ_BN), dlo + (uint32_t)((a - 1) * OZ_A_TILE >> 4),
                                 dlo + (uint32_t)((OZ_S * OZ_A_TILE + (b0 - 1) * OZ_B_TILE) >> 4), dhi,
                                 oz_idesc(nb * OZ_BN), a == 1 ? fresh : 1u, leader);
                    }
                }
                mma_commit_if(b_empty + 8 * s, leader);
                if (++s == OZ_STAGES) { s = 0; phase ^= 1; }
            }
            if (ok) mma_commit_if(b_done, leader);
        }
        if (!ok && leader) { s_abort = 1; atomicExch(g.err, 2); }
        // Every MMA issued has retired before TMEM and the stages go away, whatever
        // the other roles did (a flush warp that gave up no longer waits for them).
        mma_commit_if(b_drain, leader);
        mbar_wait(b_drain, 0u, OZ_WAIT_LIMIT);
    } else {
        // ---------------- flush warps: lanes 32 (w % 4) .., columns c0 .. c0 + 15 ----------------
        const int quad = warp & 3, c0 = (warp >> 2) * OZ_FCOLS;
        float hi[OZ_FCOLS], lo[OZ_FCOLS];
#pragma unroll
        for (int q = 0; q < OZ_FCOLS; ++q) { hi[q] = 0.f; lo[q] = 0.f; }
        bool ok = true;
        for (int c = 0; c < nchunks; ++c) {
            if (!mbar_wait(b_done, (uint32_t)(c & 1), g.wait_limit)) { ok = false; atomicExch(g.err, 4); break; }
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int L = 0; L < OZ_LEVELS; ++L) {
                const float sc = __int_as_float((127 - 7 * (L + 2)) << 23);   // 2^{-7(L+2)}
                uint32_t r[OZ_FCOLS];
                tmem_ld16_nowait(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(L * OZ_BN + c0), r);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int q = 0; q < OZ_FCOLS; ++q) df_add(hi[q], lo[q], __fmul_rn(__uint_as_float(r[q]), sc));
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            mbar_arrive(b_free);
        }
        const int i = i0 + quad * 32 + lane;
        if (ok && !s_abort && i < g.m) {
            double *C = g.C + (long long)z * g.sC;
            const double *Cin = g.Cin ? g.Cin + (long long)z * g.sCin : nullptr;
            // exponents of all-zero rows / columns are very negative; their pairs are 0
            const int ei = max(g.ea[z * g.m_pad + i], -4000) + g.alpha_e;
            const double *eCin = Cin ? Cin + (long long)i * g.ldcin : nullptr;
            double *eC = C + (long long)i * g.ldc;
#pragma unroll
            for (int q = 0; q < OZ_FCOLS; ++q) {
                const int j = j0 + c0 + q;
                if (j >= g.n || (g.lowerC && j > i)) continue;
                const int E = ei + max(g.eb[z * g.n_pad + j], -4000);
                double dh, dl, v;
                if (f2d_scaled(hi[q], E, dh) && f2d_scaled(lo[q], E, dl)) {
                    v = dh + dl;                  // a power-of-two alpha is folded into E and the sign
                    if (g.alpha_neg) v = -v;
                    if (!g.alpha_e_valid) v *= g.alpha;
                } else {
                    v = ldexp((double)hi[q] + (double)lo[q], E - g.alpha_e) * g.alpha;
                }
                if (g.beta != 0.0) v = fma(g.beta, eCin[j], v);
                eC[j] = v;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (s_abort && tid == 32 * OZ_PRODUCER_WARP) {   // producer lane: let the last copies issued land
        for (int q = max(0, s_issued - OZ_STAGES); q < s_issued; ++q)
            mbar_wait(b_full + 8 * (q % OZ_STAGES), (uint32_t)((q / OZ_STAGES) & 1), OZ_WAIT_LIMIT);
    }
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS));
}

// ---------------------------------------------------------------------------
// operand preparation
//   logical operand X(r, p), r < rows, p < k:  trans ? src[p][r] : src[r][p],
//   structural zeros (tri, in (r, p) terms) forced to 0, optional ks[p] scaling
// ---------------------------------------------------------------------------
// frexp exponent of v (v = f 2^e, 0.5 <= |f| < 1) from the IEEE-754 fields;
// a very small value for zero
__device__ __forceinline__ int oz_frexp_exp(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int bexp = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = b & ((1ull << 52) - 1);
    if (bexp != 0) return bexp - 1022;
    if (m == 0) return INT_MIN / 2;
    return -1010 - __clzll((long long)m);      // subnormal: leading bit of m at 63 - clz
}

// round(v 2^{56-e}) as an integer, for |v| < 2^e: |result| <= 2^56, error <= 1/2
__device__ __forceinline__ long long oz_fixed56(double v, int e)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    int bexp = (int)((b >> 52) & 0x7FF);
    unsigned long long m = b & ((1ull << 52) - 1);
    if (bexp == 0) { if (m == 0 || e < -1100) return 0; bexp = 1; }
    else m |= 1ull << 52;
    const int sh = (bexp - 1075) - e + 56;    // v = m 2^{bexp-1075};  m 2^sh < 2^56
    unsigned long long f;
    if (sh >= 0) f = m << sh;
    else if (sh > -64) f = (m >> (-sh)) + ((m >> (-sh - 1)) & 1ull);
    else f = 0;
    return (b >> 63) ? -(long long)f : (long long)f;
}

// float bit pattern of a small integer d (|d| <= 256) through the float 2^23 + 128: the
// integer add lands d in the last mantissa bits and one float subtraction (exact, Sterbenz)
// leaves float(d); its upper 16 bits are the BF16 pattern of d, exactly, since d has at most
// 9 significant bits.  Full-rate integer and FP32 instructions instead of two conversions.
__device__ __forceinline__ uint32_t oz_small_int_bits(int d)
{
    return __float_as_uint(__int_as_float(0x4B000080 + d) - 8388736.0f);
}

// the eight balanced base-128 digits of F (|F| <= 2^56) as float bit patterns, most
// significant first: d_8 .. d_2 in [-64, 63], the rest d_1 (|d_1| <= 128).  F = hi 2^28 + lo
// with lo in [0, 2^28): the four low digits come from lo in 32-bit arithmetic (leaving a carry
// of 0 or 1, added to hi), the other four from hi -- the same digits as extracting from F.
__device__ __forceinline__ void oz_digits(long long F, uint32_t *bits)
{
    int lo = (int)(F & 0x0FFFFFFFLL);
    int hi = (int)(F >> 28);
#pragma unroll
    for (int t = OZ_S; t >= OZ_S - 3; --t) {
        const int c = ((lo + 64) & 127) - 64;
        lo = (lo - c) >> 7;
        bits[t - 1] = oz_small_int_bits(c);
    }
    hi += lo;
#pragma unroll
    for (int t = OZ_S - 4; t >= 2; --t) {
        const int c = ((hi + 64) & 127) - 64;
        hi = (hi - c) >> 7;
        bits[t - 1] = oz_small_int_bits(c);
    }
    bits[0] = oz_small_int_bits(hi);
}

// One operand of the preparation: op(X) is rows x k (trans: op(X)[r][p] = X[p][r]), with
// structural zeros (tri), an optional inner scaling ks[p], rows padded to rows_pad.
struct OzOperand {
    const double *X; long long ld, sb; int trans, rows, tri; const double *ks;
    int rows_pad, tile_rows; int *e; __nv_bfloat16 *out;
};

// Exponents and slices of both operands in one launch; blocks [0, nA) serve A, the rest B.  A
// CTA has a band of 16 rows of op(X) and all of k: it reads the band for the rows' largest
// magnitudes, then again -- 128 KB at k = 1024, from L2 -- for the digits.  A warp covers the 16
// rows of one k block (16 columns); a lane has eight consecutive columns of one row, and each of
// its slices is one 16-byte store, 512 contiguous bytes per warp.  With trans = 0 the two lanes
// of a row read 128 contiguous bytes between them, with trans = 1 half a warp reads 16
// consecutive doubles of a memory row: no transposition through shared memory.  Bound by HBM:
// 8 B read and 16 B written per element (4096^2, both operands: 200 us in one launch; three
// launches took 303 us: a fill, an exponent pass over the matrix, the slices).
// F = round(x 2^{56-e}) is cut into balanced base-128 digits: x 2^{-e} = sum_t d_t 2^{-7t} +
// O(2^-57).  In shared memory the GEMM expects 32-byte rows whose 16-byte halves are swapped where bit 2 of the row
// is set (the 32-byte swizzle), so they are written that way.
__global__ void __launch_bounds__(256) oz_prepare_kernel(OzOperand a, OzOperand b, int k, int k_pad, int nA)
{
    __shared__ int top[8][16];
    const bool isA = (int)blockIdx.x < nA;
    const OzOperand &o = isA ? a : b;
    const int z = blockIdx.z, r0 = (isA ? (int)blockIdx.x : (int)blockIdx.x - nA) * 16;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // rows next to each other in memory go to lanes next to each other
    const int rl = o.trans ? lane & 15 : lane >> 1, half = o.trans ? lane >> 4 : lane & 1;
    const int r = r0 + rl, kblocks = k_pad / 16;
    const double *X = o.X + (long long)z * o.sb;
    const long long ld = o.ld;
    const bool live = r < o.rows;
    // columns of this row that are not structurally zero
    const int plo = o.tri == TRI_UPPER ? r : 0, phi = o.tri == TRI_LOWER ? min(k, r + 1) : k;
    // k blocks that hold any of the band's columns
    const int kb_lo = o.tri == TRI_UPPER ? min(r0 / 16, kblocks) : 0;
    const int kb_hi = o.tri == TRI_LOWER ? min(kblocks, r0 / 16 + 1) : kblocks;
    const bool quads = !o.trans && (ld & 1) == 0 && ((uintptr_t)X & 15) == 0;
    auto load = [&](int kb, double *v) {
        const int p0 = kb * 16 + half * 8;
        const bool whole = live && p0 >= plo && p0 + 8 <= phi;
        if (whole && quads) {
            const double2 *x = reinterpret_cast<const double2 *>(X + (long long)r * ld + p0);
#pragma unroll
            for (int q = 0; q < 4; ++q) { const double2 t = x[q]; v[2 * q] = t.x; v[2 * q + 1] = t.y; }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int p = p0 + q;
                const bool in = whole || (live && p >= plo && p < phi);
                v[q] = in ? (o.trans ? X[(long long)p * ld + r] : X[(long long)r * ld + p]) : 0.0;
            }
        }
        if (o.ks) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (p0 + q < k) v[q] *= o.ks[p0 + q];
        }
    };
    int mx = INT_MIN / 2;
    for (int kb = kb_lo + warp; kb < kb_hi; kb += 8) {
        double v[8];
        load(kb, v);
        int h = 0;                                     // largest high word of a magnitude: orders them by exponent
#pragma unroll
        for (int q = 0; q < 8; ++q) h = max(h, __double2hiint(v[q]) & 0x7FFFFFFF);
        if (h >= 0x00100000) {
            mx = max(mx, (h >> 20) - 1022);
        } else {                                       // zeros and subnormal numbers only
#pragma unroll
            for (int q = 0; q < 8; ++q) mx = max(mx, oz_frexp_exp(v[q]));
        }
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o.trans ? 16 : 1));
    if (half == 0) top[warp][rl] = mx;
    __syncthreads();
    int ex = top[0][rl];
#pragma unroll
    for (int w = 1; w < 8; ++w) ex = max(ex, top[w][rl]);
    if (warp == 0 && half == 0) o.e[(long long)z * o.rows_pad + r] = ex;
    if (!live || ex <= -2000) ex = -4000;
    // row tiles read the k range of their own triangle rounded out to their height: blocks
    // within 256 rows of it are written as zeros, those beyond are never read
    const int w_lo = o.tri == TRI_UPPER ? max(0, min(kblocks, r0 / 16) - 16) : 0;
    const int w_hi = o.tri == TRI_LOWER ? min(kblocks, r0 / 16 + 17) : kblocks;
    __nv_bfloat16 *tile = o.out + ((long long)z * (o.rows_pad / o.tile_rows) + r / o.tile_rows) * kblocks * (OZ_S * o.tile_rows * 16) +
                          (r % o.tile_rows) * 16 + ((half ^ (r >> 2)) & 1) * 8;
    for (int kb = w_lo + warp; kb < w_hi; kb += 8) {
        double v[8];
        long long f[8];
        uint32_t w[OZ_S][4];
        load(kb, v);
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = (ex > -2000) ? oz_fixed56(v[q], ex) : 0;
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            uint32_t ba[OZ_S], bb[OZ_S];
            oz_digits(f[q], ba);
            oz_digits(f[q + 1], bb);
#pragma unroll
            for (int t = 0; t < OZ_S; ++t) w[t][q >> 1] = __byte_perm(ba[t], bb[t], 0x7632);   // two upper halves
        }
        __nv_bfloat16 *dst = tile + (long long)kb * (OZ_S * o.tile_rows * 16);
#pragma unroll
        for (int t = 0; t < OZ_S; ++t)
            *reinterpret_cast<uint4 *>(dst + t * o.tile_rows * 16) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
    }
}

}  // namespace

namespace {
struct OzLayout {
    int kp, mp, np;                        // k, rows of A, rows of B padded
    __nv_bfloat16 *sa, *sb;
    int *ea, *eb;
};
OzLayout oz_layout(const GemmArgs &g, void *ws)
{
    OzLayout L;
    L.kp = (g.k + 15) / 16 * 16;
    L.mp = (g.m + OZ_BM - 1) / OZ_BM * OZ_BM; L.np = (g.n + OZ_BN - 1) / OZ_BN * OZ_BN;
    unsigned char *base = (unsigned char *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    L.sa = (__nv_bfloat16 *)base;
    L.sb = L.sa + (size_t)OZ_S * L.mp * L.kp * g.batch;
    L.ea = (int *)(L.sb + (size_t)OZ_S * L.np * L.kp * g.batch);
    L.eb = L.ea + (size_t)L.mp * g.batch;
    return L;
}
}  // namespace

size_t oz_gemm_workspace_bytes(const GemmArgs &g)
{
    const long long kp = (g.k + 15) / 16 * 16;
    const long long mp = (g.m + OZ_BM - 1) / OZ_BM * OZ_BM, np = (g.n + OZ_BN - 1) / OZ_BN * OZ_BN;
    return (size_t)(OZ_S * (mp + np) * kp * g.batch) * 2 + (size_t)(mp + np) * g.batch * sizeof(int) + 2048;
}

// operand preparation: exponents and slices of op(A) and op(B) into ws
int oz_gemm_prepare(const GemmArgs &g, void *ws, cudaStream_t s)
{
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return 0;
    const OzLayout L = oz_layout(g, ws);
    const int triB = g.triB == TRI_LOWER ? TRI_UPPER : (g.triB == TRI_UPPER ? TRI_LOWER : TRI_NONE);
    // op(A) rows are memory rows unless A is transposed; op(B) columns are memory rows when B is transposed
    OzOperand oa{(const double *)g.A, g.lda, g.sA, g.ta, g.m, g.triA, (const double *)g.kscale, L.mp, OZ_BM, L.ea, L.sa};
    OzOperand ob{(const double *)g.B, g.ldb, g.sB, g.tb ? 0 : 1, g.n, triB, nullptr, L.np, OZ_BN, L.eb, L.sb};
    const int nA = L.mp / 16, nB = L.np / 16;
    oz_prepare_kernel<<<dim3(nA + nB, 1, g.batch), 256, 0, s>>>(oa, ob, g.k, L.kp, nA); count_launch();
    return 0;
}

// the tensor-core product on operands prepared by oz_gemm_prepare(g, ws)
int oz_gemm_run(const GemmArgs &g, void *ws, int *err, cudaStream_t s)
{
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return 0;
    const OzLayout L = oz_layout(g, ws);
    OzArgs a;
    a.sa = L.sa; a.sb = L.sb; a.kblocks = L.kp / 16;
    a.m = g.m; a.n = g.n; a.k = g.k; a.batch = g.batch; a.m_pad = L.mp; a.n_pad = L.np;
    a.triA = g.triA; a.triB = g.triB; a.lowerC = g.lowerC;
    a.ea = L.ea; a.eb = L.eb;
    a.C = (double *)g.C; a.ldc = g.ldc; a.sC = g.sC;
    a.Cin = (const double *)g.Cin; a.ldcin = g.ldcin; a.sCin = g.sCin;
    a.alpha = g.alpha; a.beta = g.beta; a.err = err;
    a.wait_limit = g.wait_limit > 0 ? (unsigned long long)g.wait_limit : OZ_WAIT_LIMIT;
    {
        int ex = 0;
        const double fr = std::frexp(std::fabs(g.alpha), &ex);
        a.alpha_e_valid = (fr == 0.5) ? 1 : 0;            // |alpha| = 2^(ex-1)
        a.alpha_e = a.alpha_e_valid ? ex - 1 : 0;
        a.alpha_neg = (a.alpha_e_valid && g.alpha < 0) ? 1 : 0;
    }
    const int tiles = ((g.n + OZ_BN - 1) / OZ_BN) * ((g.m + OZ_BM - 1) / OZ_BM);
    if (!ensure_dynamic_smem((const void *)oz_gemm_kernel, OZ_SMEM_BYTES)) return -2;
    oz_gemm_kernel<<<dim3(tiles, 1, g.batch), OZ_THREADS, OZ_SMEM_BYTES, s>>>(a);
    count_launch();
    return 0;
}

// estimate of the slice engine's time in microseconds: the two launches, prologue and epilogue,
// then 1 us for each k block of the tiles a busiest SM takes in turn (preparation included)
double oz_gemm_time_us(const GemmArgs &g)
{
    const double mt = (g.m + OZ_BM - 1) / OZ_BM, nt = (g.n + OZ_BN - 1) / OZ_BN;
    return 11.0 + std::ceil((g.lowerC ? 0.5 : 1.0) * mt * nt * g.batch / 152.0) * (g.k / OZ_BK);
}

int oz_gemm_launch(const GemmArgs &g, void *ws, int *err, cudaStream_t s)
{
    int st = oz_gemm_prepare(g, ws, s);
    return st ? st : oz_gemm_run(g, ws, err, s);
}

}  // namespace pssd
