// FP32-accurate GEMM on the 5th-generation tensor cores of sm_103a (tcgen05).
//
//   C = alpha * op(A) * diag(kscale) * op(B) + beta * Cin        (FP32 data)
//
// with the same operand conventions as gemm_kernel (triangular operands,
// lower-only output, batch).  Each FP32 operand x is split once, in an HBM
// pass that also applies the triangular masks, the inner scaling and the
// transposition to K-major order, into x = hi + lo with hi = tf32(x) and
// lo = x - hi; the product is accumulated in FP32 in tensor memory as
//     A_lo B_hi + A_hi B_lo + A_hi B_hi      (3xTF32, ~FP32 accuracy).
//
// Kernel layout (one CTA of 10 warps per 128 x BN output tile, BN = 64, 128 or 256):
//   * the split pass writes, for every (row tile, 16-term k block), the hi
//     and lo parts as one contiguous block already in the 64-byte-swizzled
//     order the MMA descriptors read (A: 2 x 128 rows x 64 bytes = 16 KB,
//     B: 2 x BN rows x 64 bytes);
//   * warp 8 streams one k block per stage with two cp.async.bulk copies into
//     a ring of 96 KB (4, 3 or 2 stages) with full/empty mbarriers;
//   * warp 9 issues per stage 2 (K = 8) x 3 tcgen05.mma kind::tf32 (M = 128,
//     N = BN) into one FP32 accumulator of BN TMEM columns and frees each
//     stage with tcgen05.commit;
//   * warps 0-7 wait for the final commit and write C (warp w: TMEM lanes
//     32 (w % 4) .., i.e. tile rows, and columns BN/2 (w / 4) ..), through the
//     ring: written from the accumulator's lanes a store touches 32 rows.
// Two CTAs share an SM, so that one's epilogue and first copies run under the
// other's products.  A large product is bound by shared memory, 96 bytes of
// operand reads and 64 of copies for every 128 clocks of products at BN = 256.
// Every pipeline mbarrier wait is bounded by the caller's limit: on timeout the
// kernel sets *err, skips the remaining work, waits (under a fixed, longer
// bound) for its own bulk copies and MMAs in flight, frees its TMEM and returns.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "mbar.cuh"
#include "pssd_internal.h"

namespace pssd {

namespace {

constexpr int TC_BM = 128, TC_BN_MAX = 256, TC_BK = 16;   // BK in FP32 elements = 64 bytes per row
constexpr int TC_A_BYTES = 2 * TC_BM * TC_BK * 4;      // hi + lo, 16 KB
__host__ __device__ constexpr int tc_b_bytes(int bn) { return 2 * bn * TC_BK * 4; }
__host__ __device__ constexpr int tc_smem_bytes(int bn, int stages)
{
    return stages * (TC_A_BYTES + tc_b_bytes(bn)) + 1024 /* alignment */ + 256 /* barriers */;
}
constexpr unsigned long long TC_WAIT_LIMIT = 1ull << 26;   // default pipeline bound and the drain bound
constexpr int TC_EPI_WARPS = 8;                        // warp w: lanes 32 (w % 4) .., columns BN/2 (w / 4) ..
constexpr int TC_PRODUCER_WARP = TC_EPI_WARPS, TC_MMA_WARP = TC_EPI_WARPS + 1;
constexpr int TC_THREADS = 32 * (TC_EPI_WARPS + 2);
constexpr int TC_GROUP_M = 8;                          // row blocks per group of the tile order

struct TcArgs {
    const float *a, *b;                        // tiled split operands (see the split kernel)
    int kblocks;                               // k_pad / 16
    int m, n, k, batch;
    int m_pad, n_pad;
    int triA, triB, lowerC;
    float *C; long long ldc, sC;
    const float *Cin; long long ldcin, sCin;
    float alpha, beta;
    int *err;
    unsigned long long wait_limit;             // polls per pipeline wait before giving up
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"((unsigned long long)src), "r"(bytes), "r"(bar)
        : "memory");
}

// shared-memory matrix descriptor: K-major operand, 64-byte swizzle, 8-row
// groups 512 bytes apart (SBO), version 1 (sm_100 family)
__device__ __forceinline__ unsigned long long smem_desc(uint32_t addr)
{
    unsigned long long d = 0;
    d |= (unsigned long long)((addr >> 4) & 0x3FFF);          // start address
    d |= (unsigned long long)(16 >> 4) << 16;                  // leading byte offset (unused, swizzled K-major)
    d |= (unsigned long long)(512 >> 4) << 32;                 // stride byte offset
    d |= 1ull << 46;                                           // descriptor version
    d |= 4ull << 61;                                           // 64-byte swizzle
    return d;
}

// instruction descriptor: kind::tf32, D = F32, A = B = TF32, both K-major, M = 128, N = bn
__host__ __device__ constexpr uint32_t tc_idesc(int bn)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, unsigned long long a, unsigned long long b,
                                         uint32_t idesc, uint32_t acc, uint32_t pred)
{
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(pred));
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

// waits for the loads in flight; r, which one of them fills, is not read before
__device__ __forceinline__ void tmem_wait16(uint32_t *r)
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

template <int BN, int STAGES, int CTAS>
__global__ void __launch_bounds__(TC_THREADS, CTAS) tc_gemm_kernel(const __grid_constant__ TcArgs g)
{
    constexpr int TC_BN = BN, TC_STAGES = STAGES, TC_B_BYTES = tc_b_bytes(BN), TC_TMEM_COLS = BN;
    constexpr int TC_STAGE_BYTES = TC_A_BYTES + TC_B_BYTES;
    constexpr int TC_ECOLS = TC_BN / (TC_EPI_WARPS / 4);
    static_assert(TC_EPI_WARPS * 32 * 33 * 4 <= TC_STAGES * TC_STAGE_BYTES, "the epilogue's blocks go into the ring");
    // grouped tile order: runs of TC_GROUP_M row blocks sweep the column blocks together
    const int mt = (g.m + TC_BM - 1) / TC_BM, nt = (g.n + TC_BN - 1) / TC_BN;
    const int pid = blockIdx.x, per_group = TC_GROUP_M * nt;
    const int first_m = (pid / per_group) * TC_GROUP_M, gm = min(mt - first_m, TC_GROUP_M);
    const int tm = first_m + (pid % per_group) % gm, tn = (pid % per_group) / gm;
    const int i0 = tm * TC_BM, j0 = tn * TC_BN, z = blockIdx.z;
    if (i0 >= g.m || j0 >= g.n) return;
    if (g.lowerC && j0 > i0 + TC_BM - 1) return;

    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned long long *bars = (unsigned long long *)(smem + TC_STAGES * TC_STAGE_BYTES);
    // bars[0..ST): full, [ST..2ST): empty, [2ST]: accumulator done
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * TC_STAGES + 2);
    __shared__ int s_abort, s_issued;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // k range that can contribute to this tile (structural zeros skipped)
    int kbeg = 0, kend = g.k;
    if (g.triA == TRI_LOWER) kend = min(kend, i0 + TC_BM);
    if (g.triA == TRI_UPPER) kbeg = max(kbeg, i0);
    if (g.triB == TRI_LOWER) kbeg = max(kbeg, j0);
    if (g.triB == TRI_UPPER) kend = min(kend, j0 + TC_BN);
    const int kb0 = kbeg / TC_BK;
    const int nkb = (kend > kbeg) ? (kend + TC_BK - 1) / TC_BK - kb0 : 0;
    const uint32_t b_full = smem_u32(&bars[0]), b_empty = smem_u32(&bars[TC_STAGES]);
    const uint32_t b_done = smem_u32(&bars[2 * TC_STAGES]);
    const uint32_t b_drain = smem_u32(&bars[2 * TC_STAGES + 1]);   // MMA drain after an abort

    if (tid == 0) {
        s_abort = 0;
        s_issued = 0;
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(b_full + 8 * s, 1);
            mbar_init(b_empty + 8 * s, 1);
        }
        mbar_init(b_done, 1);
        mbar_init(b_drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;

    if (warp == TC_PRODUCER_WARP) {
        // ---------------- bulk-copy producer ----------------
        if (lane == 0) {
            const float *srca = g.a + (((long long)z * (g.m_pad / TC_BM) + tm) * g.kblocks + kb0) * (TC_A_BYTES / 4);
            const float *srcb = g.b + (((long long)z * (g.n_pad / TC_BN) + tn) * g.kblocks + kb0) * (TC_B_BYTES / 4);
            for (int q = 0; q < nkb; ++q) {
                const int s = q % TC_STAGES;
                if (q >= TC_STAGES && !mbar_wait(b_empty + 8 * s, (uint32_t)(((q / TC_STAGES) - 1) & 1), g.wait_limit)) {
                    s_abort = 1; atomicExch(g.err, 1); break;
                }
                if (s_abort) break;
                const uint32_t st = smem_u32(smem + s * TC_STAGE_BYTES);
                mbar_expect_tx(b_full + 8 * s, TC_STAGE_BYTES);
                bulk_load(st, srca + (long long)q * (TC_A_BYTES / 4), TC_A_BYTES, b_full + 8 * s);
                bulk_load(st + TC_A_BYTES, srcb + (long long)q * (TC_B_BYTES / 4), TC_B_BYTES, b_full + 8 * s);
                s_issued = q + 1;
            }
        }
    } else if (warp == TC_MMA_WARP) {
        // ---------------- MMA issuer ----------------
        // The warp runs converged and one elected lane issues: the operands stay in uniform
        // registers, and six products of 128 clocks a stage are not held up by their issue.
        const uint32_t leader = elect_one(), idesc = tc_idesc(BN);
        bool ok = true;
        int s = 0;
        uint32_t phase = 0;
#pragma unroll 1
        for (int q = 0; q < nkb; ++q) {
            if (!mbar_wait(b_full + 8 * s, phase, g.wait_limit)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t st = smem_u32(smem) + s * TC_STAGE_BYTES;
            const uint32_t ah = st, al = st + TC_A_BYTES / 2;
            const uint32_t bh = st + TC_A_BYTES, bl = st + TC_A_BYTES + TC_B_BYTES / 2;
#pragma unroll
            for (int kk = 0; kk < TC_BK / 8; ++kk) {           // K = 8 TF32 = 32 bytes per instruction
                const uint32_t off = kk * 32;
                mma_tf32(tmem, smem_desc(al + off), smem_desc(bh + off), idesc, (q > 0 || kk > 0) ? 1u : 0u, leader);
                mma_tf32(tmem, smem_desc(ah + off), smem_desc(bl + off), idesc, 1u, leader);
                mma_tf32(tmem, smem_desc(ah + off), smem_desc(bh + off), idesc, 1u, leader);
            }
            mma_commit_if(b_empty + 8 * s, leader);            // stage s is free when these MMAs retire
            if (++s == TC_STAGES) { s = 0; phase ^= 1; }
        }
        if (nkb > 0) {
            if (ok) mma_commit_if(b_done, leader);
            else if (leader) { s_abort = 1; atomicExch(g.err, 2); }
        }
        // Every MMA issued has retired before TMEM and the stages go away, whatever
        // the other roles did (an epilogue warp that gave up no longer waits for them).
        mma_commit_if(b_drain, leader);
        mbar_wait(b_drain, 0u, TC_WAIT_LIMIT);
    } else {
        // ---------------- epilogue warps: 32 rows, BN / 2 columns in blocks of 32 ----------------
        // A thread reads one row of the accumulator; the block goes through the ring (free:
        // every product has retired) so that a store covers 128 bytes of one row instead of
        // 4 bytes of 32 rows (the products of a 12288 split: 151 ms so, 129 through the ring).
        const int quad = warp & 3, c0 = (warp >> 2) * TC_ECOLS, r0 = i0 + quad * 32;
        bool have = nkb > 0;
        if (have && !mbar_wait(b_done, 0u, g.wait_limit)) { have = false; atomicExch(g.err, 3); }
        have = __all_sync(0xffffffffu, have);
        asm volatile("tcgen05.fence::after_thread_sync;");
        float *T = reinterpret_cast<float *>(smem) + warp * (32 * 33);
        if (have || nkb == 0) {   // nkb == 0: the product is zero and C = beta Cin; a failed wait writes nothing
#pragma unroll 1
            for (int cc = 0; cc < TC_ECOLS; cc += 32) {
                const int jb = j0 + c0 + cc, j = jb + lane;
                if (r0 >= g.m || jb >= g.n || (g.lowerC && jb > r0 + 31)) break;
                if (have) {
                    uint32_t ra[16], rb[16];
                    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(c0 + cc);
                    tmem_ld16_nowait(taddr, ra);
                    tmem_ld16_nowait(taddr + 16, rb);
                    tmem_wait16(ra);
                    tmem_wait16(rb);
                    __syncwarp();                              // the block before has been read
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        T[lane * 33 + q] = __uint_as_float(ra[q]);
                        T[lane * 33 + 16 + q] = __uint_as_float(rb[q]);
                    }
                    __syncwarp();
                }
                float *C = g.C + (long long)z * g.sC + j;
                const float *Cin = g.beta != 0.f ? g.Cin + (long long)z * g.sCin + j : nullptr;
                constexpr int NB = 8;                          // rows in flight of beta Cin
#pragma unroll 1
                for (int p = 0; p < 32; p += NB) {
                    float cv[NB];
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const int row = r0 + p + u;
                        const bool in = row < g.m && j < g.n && !(g.lowerC && j > row);
                        cv[u] = Cin && in ? Cin[(long long)row * g.ldcin] : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const int row = r0 + p + u;
                        if (row >= g.m || j >= g.n || (g.lowerC && j > row)) continue;
                        const float v = have ? T[(p + u) * 33 + lane] : 0.f;
                        C[(long long)row * g.ldc] = Cin ? __fmaf_rn(g.alpha, v, __fmul_rn(g.beta, cv[u]))
                                                        : __fmul_rn(g.alpha, v);
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (s_abort && tid == 32 * TC_PRODUCER_WARP) {   // producer lane: let the last copies issued land
        for (int q = max(0, s_issued - TC_STAGES); q < s_issued; ++q)
            mbar_wait(b_full + 8 * (q % TC_STAGES), (uint32_t)((q / TC_STAGES) & 1), TC_WAIT_LIMIT);
    }
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS));
}

// ---------------------------------------------------------------------------
// operand preparation: masked, scaled, K-major, split into tf32 hi + lo
//   logical operand row r < rows, column p < k:
//   src = trans ? X[z][p][r] : X[z][r][p]; structural zeros (tri) forced to 0
// tri: relation of (r, p) that is structurally nonzero:
//   TRI_LOWER: p <= r,  TRI_UPPER: p >= r  (for A: op(A)[i][p]);
//   for B the caller passes the relation in terms of (j, p) of op(B)[p][j]:
//   op(B) lower (p >= j) -> TRI_UPPER here, op(B) upper (p <= j) -> TRI_LOWER
// Output, tiled for the GEMM's bulk copies: block
//   ((z * rows_pad / tile_rows + r / tile_rows) * (k_pad / 16) + p / 16)
// of 2 * tile_rows * 16 floats holds the hi part (rows rr = r % tile_rows,
// 16 floats each) then the lo part; inside a 64-byte row the 16-byte chunk
// (p % 16) / 4 is stored at chunk ((p % 16) / 4) ^ ((rr / 2) % 4) (the
// 64-byte shared-memory swizzle the MMA descriptors expect).
// ---------------------------------------------------------------------------
// One operand: op(X) is rows x k (trans: op(X)[r][p] = X[p][r]), tri and ks as above.
struct TcOperand {
    const float *X; long long ld, sb; int trans, rows, rows_pad, tile_rows, tri; const float *ks; float *out;
};

// both operands in one launch: grid rows [0, nA) serve A, the rest B
__global__ void __launch_bounds__(256) tf32_split_kernel(TcOperand a, TcOperand b, int k, int k_pad, int nA)
{
    const bool isA = (int)blockIdx.y < nA;
    const TcOperand &op = isA ? a : b;
    const float *X = op.X, *ks = op.ks;
    const long long ld = op.ld, sb = op.sb;
    const int trans = op.trans, rows = op.rows, rows_pad = op.rows_pad, tile_rows = op.tile_rows, tri = op.tri;
    float *out = op.out;
    __shared__ float T[32][33];
    const int z = blockIdx.z;
    const int r0 = (isA ? (int)blockIdx.y : (int)blockIdx.y - nA) * 32, p0 = blockIdx.x * 32;
    // A row tile's k range ends (begins) at the end (start) of its triangle: blocks beyond are never
    // read (R^{-T} R^{-1}, 4 of order 1024: 36 us, 23 without them).
    const int t0 = r0 / tile_rows * tile_rows;
    if ((tri == TRI_LOWER && p0 >= t0 + tile_rows) || (tri == TRI_UPPER && p0 + 32 <= t0)) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
    X += (long long)z * sb;
    // load the 32 x 32 block in the orientation that is contiguous in memory
    for (int yy = ty; yy < 32; yy += 8) {
        float v = 0.f;
        if (trans) {   // memory rows are p, contiguous r
            int p = p0 + yy, r = r0 + tx;
            if (p < k && r < rows) v = X[(long long)p * ld + r];
            T[tx][yy] = v;   // T[r][p]
        } else {
            int r = r0 + yy, p = p0 + tx;
            if (r < rows && p < k) v = X[(long long)r * ld + p];
            T[yy][tx] = v;
        }
    }
    __syncthreads();
    // each thread: one row of the tile and four consecutive k -- one 16-byte chunk of the
    // swizzled layout -- written as one 16-byte store for the hi parts and one for the lo parts
    const int kblocks = k_pad / 16, tiles = rows_pad / tile_rows;
    const int yy = threadIdx.x >> 3, q4 = (threadIdx.x & 7) * 4;
    const int r = r0 + yy, pq = p0 + q4;
    if (r >= rows_pad || pq >= k_pad) return;      // k_pad is a multiple of 16: the four p all fit
    float hv[4], lv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int p = pq + t;
        float v = (r < rows && p < k) ? T[yy][q4 + t] : 0.f;
        if (tri == TRI_LOWER && p > r) v = 0.f;
        if (tri == TRI_UPPER && p < r) v = 0.f;
        if (ks && p < k) v *= ks[p];
        uint32_t u;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(v));
        hv[t] = __uint_as_float(u);
        lv[t] = v - hv[t];
    }
    const int rr = r % tile_rows, kk = pq & 15;
    const long long blk = ((long long)z * tiles + r / tile_rows) * kblocks + (pq >> 4);
    float *o = out + blk * (2 * tile_rows * 16) + rr * 16 + ((((kk >> 2) ^ (rr >> 1)) & 3) << 2);
    *reinterpret_cast<float4 *>(o) = make_float4(hv[0], hv[1], hv[2], hv[3]);
    *reinterpret_cast<float4 *>(o + tile_rows * 16) = make_float4(lv[0], lv[1], lv[2], lv[3]);
}

}  // namespace

size_t tc_gemm_workspace_bytes(const GemmArgs &g)
{
    const long long kp = (g.k + 15) / 16 * 16;
    const long long mp = (g.m + TC_BM - 1) / TC_BM * TC_BM, np = (g.n + TC_BN_MAX - 1) / TC_BN_MAX * TC_BN_MAX;
    return (size_t)(2 * (mp + np) * kp * g.batch) * sizeof(float) + 1024;
}

namespace {
struct TcTile { int bn; int (*launch)(const TcArgs &, cudaStream_t); };

template <int BN, int STAGES, int CTAS>
int tc_launch_tile(const TcArgs &a, cudaStream_t s)
{
    const auto kernel = tc_gemm_kernel<BN, STAGES, CTAS>;
    if (!ensure_dynamic_smem((const void *)kernel, tc_smem_bytes(BN, STAGES))) return -2;
    const dim3 grid(((a.n + BN - 1) / BN) * ((a.m + TC_BM - 1) / TC_BM), 1, a.batch);
    kernel<<<grid, TC_THREADS, tc_smem_bytes(BN, STAGES), s>>>(a); count_launch();
    return 0;
}

// The tile width that takes the least time, counted in rounds of two CTAs an SM.  A CTA's round
// costs 91 (64 columns), 128 or 241 (256) -- the measured times of k = 2048 products of many
// rounds: 344, 276 and 263 us for 4 x 2048^3.  Wide tiles read A less often, narrow ones fill the
// chip with a small product: 4 x 500^3 18, 24, 38 us (34 with one CTA an SM and four stages);
// 4 x 1024^3 61, 47, 72; 6144^3 2006, 1458, 1366.  With a triangular operand the work differs from
// tile to tile, there are no rounds, and 256 columns compute more of what is zero: 304 us with
// 128, 351 with 256 for R^{-T} R^{-1} of order 6144.
TcTile tc_tile(const GemmArgs &g)
{
    static const struct { TcTile tile; long long cost; } t[] = {
        {{64, tc_launch_tile<64, 4, 2>}, 91}, {{128, tc_launch_tile<128, 3, 2>}, 128}, {{256, tc_launch_tile<256, 2, 2>}, 241}};
    const long long slots = 2 * 152, mt = (g.m + TC_BM - 1) / TC_BM;
    const bool tri = g.triA != TRI_NONE || g.triB != TRI_NONE;
    TcTile best = t[0].tile;
    long long least = LLONG_MAX;
    for (const auto &x : t) {
        if (tri && x.tile.bn == 256) break;
        const long long nt = (g.n + x.tile.bn - 1) / x.tile.bn;
        long long tiles = g.lowerC ? 0 : mt * nt;
        for (long long i = 0; g.lowerC && i < mt; ++i)
            tiles += std::min(nt, (i * TC_BM + TC_BM - 1) / x.tile.bn + 1);
        const long long c = (tiles * g.batch + slots - 1) / slots * x.cost;
        if (c < least) { least = c; best = x.tile; }
    }
    return best;
}

void tc_layout(const GemmArgs &g, void *ws, int bn, int &kp, int &mp, int &np, float *&ta, float *&tb)
{
    kp = (g.k + 15) / 16 * 16;
    mp = (g.m + TC_BM - 1) / TC_BM * TC_BM; np = (g.n + bn - 1) / bn * bn;
    float *base = (float *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    ta = base; tb = ta + (size_t)2 * mp * kp * g.batch;
}
}  // namespace

// operand preparation: masked, scaled, K-major tf32 hi/lo tiles of op(A), op(B) into ws
int tc_gemm_prepare(const GemmArgs &g, void *ws, cudaStream_t s)
{
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return 0;
    const int bn = tc_tile(g).bn;
    int kp, mp, np; float *ta, *tb;
    tc_layout(g, ws, bn, kp, mp, np, ta, tb);
    // A: rows i of op(A); B: rows j of op(B)^T (op(B)[p][j] = B[p][j] or B[j][p]); both K-major
    const int triB = g.triB == TRI_LOWER ? TRI_UPPER : (g.triB == TRI_UPPER ? TRI_LOWER : TRI_NONE);
    const TcOperand oa{(const float *)g.A, g.lda, g.sA, g.ta, g.m, mp, TC_BM, g.triA, (const float *)g.kscale, ta};
    const TcOperand ob{(const float *)g.B, g.ldb, g.sB, g.tb ? 0 : 1, g.n, np, bn, triB, nullptr, tb};
    const int nA = mp / 32, nB = np / 32;
    tf32_split_kernel<<<dim3((kp + 31) / 32, nA + nB, g.batch), 256, 0, s>>>(oa, ob, g.k, kp, nA); count_launch();
    return 0;
}

// the tensor-core product on operands prepared by tc_gemm_prepare(g, ws); err: device int (0 on entry)
int tc_gemm_run(const GemmArgs &g, void *ws, int *err, cudaStream_t s)
{
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return 0;
    const TcTile t = tc_tile(g);
    int kp, mp, np; float *ta, *tb;
    tc_layout(g, ws, t.bn, kp, mp, np, ta, tb);
    TcArgs a;
    a.a = ta; a.b = tb; a.kblocks = kp / 16;
    a.m = g.m; a.n = g.n; a.k = g.k; a.batch = g.batch; a.m_pad = mp; a.n_pad = np;
    a.triA = g.triA; a.triB = g.triB; a.lowerC = g.lowerC;
    a.C = (float *)g.C; a.ldc = g.ldc; a.sC = g.sC;
    a.Cin = (const float *)g.Cin; a.ldcin = g.ldcin; a.sCin = g.sCin;
    a.alpha = (float)g.alpha; a.beta = (float)g.beta;
    a.err = err;
    a.wait_limit = g.wait_limit > 0 ? (unsigned long long)g.wait_limit : TC_WAIT_LIMIT;
    return t.launch(a, s);
}

// ws: device workspace of tc_gemm_workspace_bytes(g) bytes; err: device int (0 on entry)
int tc_gemm_launch(const GemmArgs &g, void *ws, int *err, cudaStream_t s)
{
    int st = tc_gemm_prepare(g, ws, s);
    return st ? st : tc_gemm_run(g, ws, err, s);
}

}  // namespace pssd
