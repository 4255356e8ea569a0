// FP64 kernels of libpssd (sm_103a).
//
// On GB300 the FP64 pipe retires 2 DFMA per clock per SM (about 1.1 TFLOP/s
// for the chip), so every FP64 contraction here is bound by the DFMA issue
// rate, not by memory (dgemm_kernel below).
// The HBM-bound passes (symmetrisation, mirror, shift, combine, norms) use
// 32x32 shared-memory transposes so that both the row and the column access
// are coalesced.
#include <algorithm>
#include <mutex>
#include <set>
#include <utility>

#include "mbar.cuh"
#include "pssd_internal.h"

#include <math.h>

#include <type_traits>

namespace pssd {

std::atomic<long long> g_launches{0};
std::atomic<long long> g_phase_launches[PH_COUNT];
thread_local int g_phase = PH_OTHER;

bool ensure_dynamic_smem(const void *func, int bytes)
{
    static std::mutex mu;
    static std::set<std::pair<int, const void *>> done;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, func})) return true;
    if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    done.insert({dev, func});
    return true;
}


// --------------------------------------------------------------------------
// GEMM with triangular operands, lower-only output and inner scaling, in
// two arithmetic modes on the FP32 pipe (FP64 storage on the DFMA pipe:
// dgemm_kernel below):
//   GM_F32  FP32 storage, FFMA accumulation
//   GM_DF   FP64 storage, FP64 emulated on the FP32 pipe: each operand is
//           split into a pair of floats (hi = fl32(x), lo = fl32(x - hi)), the
//           product hi*hi is made error-free with an FMA, the cross terms are
//           added in FP32, the running sum is a float pair updated by TwoSum
//           (Knuth) and flushed into an FP64 accumulator every 128 k-steps.
//           The operands arrive already split (split_pairs, one HBM pass),
//           so the FP64 pipe -- 1/64 of the FP32 rate on GB300 -- only sees
//           the flushes.  Relative error per 128-term block ~2^-46.
// --------------------------------------------------------------------------
constexpr int GBK = 16;                              // tile of Q x Q outputs a thread, 16 x 16 threads

template <class T>
__device__ __forceinline__ T load_op(const T *P, long long ld, int trans, int r, int c)
{
    return trans ? P[(long long)c * ld + r] : P[(long long)r * ld + c];
}

template <int MODE, int Q>
__global__ void __launch_bounds__(256) gemm_kernel(GemmArgs g)
{
    using T = typename std::conditional<MODE == GM_F32, float, double>::type;
    constexpr int GBM = 16 * Q, GBN = 16 * Q;
    const int z = blockIdx.z;
    const int i0 = blockIdx.y * GBM, j0 = blockIdx.x * GBN;
    if (i0 >= g.m || j0 >= g.n) return;
    if (g.lowerC && j0 > i0 + GBM - 1) return;   // tile strictly above the diagonal

    const T *A = (const T *)g.A + (long long)z * g.sA;
    const T *B = (const T *)g.B + (long long)z * g.sB;
    const T *ks = (const T *)g.kscale;
    // GM_DF: float pairs split beforehand
    const float *Ah = (const float *)g.A + (long long)z * g.sA, *Al = (const float *)g.Alo + (long long)z * g.sA;
    const float *Bh = (const float *)g.B + (long long)z * g.sB, *Bl = (const float *)g.Blo + (long long)z * g.sB;
    int kbeg = 0, kend = g.k;
    if (g.triA == TRI_LOWER) kend = min(kend, i0 + GBM);   // op(A)[i][p] = 0 for p > i
    if (g.triA == TRI_UPPER) kbeg = max(kbeg, i0);         // op(A)[i][p] = 0 for p < i
    if (g.triB == TRI_LOWER) kbeg = max(kbeg, j0);         // op(B)[p][j] = 0 for p < j
    if (g.triB == TRI_UPPER) kend = min(kend, j0 + GBN);   // op(B)[p][j] = 0 for p > j

    using S = float;
    __shared__ S As[GBK][GBM + 1], Bs[GBK][GBN + 1];
    __shared__ float Asl[MODE == GM_DF ? GBK : 1][GBM + 1], Bsl[MODE == GM_DF ? GBK : 1][GBN + 1];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    T acc[Q][Q];
    float ah_[Q][Q], al_[Q][Q];   // DF running float pair (unused otherwise)
#pragma unroll
    for (int a = 0; a < Q; ++a)
#pragma unroll
        for (int b = 0; b < Q; ++b) { acc[a][b] = 0; ah_[a][b] = 0.f; al_[a][b] = 0.f; }

    int kt_count = 0;
    for (int kt = kbeg; kt < kend; kt += GBK) {
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            int e = tid + 256 * u;
            int il, pl;
            if (g.ta == 0) { il = e >> 4; pl = e & 15; } else { pl = e / GBM; il = e % GBM; }
            int i = i0 + il, p = kt + pl;
            bool ok = (i < g.m) && (p < kend);
            if (g.triA == TRI_LOWER) ok = ok && (p <= i);
            if (g.triA == TRI_UPPER) ok = ok && (p >= i);
            if (MODE == GM_DF) {
                float hi = 0.f, lo = 0.f;
                if (ok) {
                    hi = load_op(Ah, g.lda, g.ta, i, p); lo = load_op(Al, g.lda, g.ta, i, p);
                    if (ks) { float f = (float)ks[p]; hi *= f; lo *= f; }
                }
                As[pl][il] = hi;
                Asl[pl][il] = lo;
            } else {
                T v = 0;
                if (ok) {
                    v = load_op(A, g.lda, g.ta, i, p);
                    if (ks) v *= ks[p];
                }
                As[pl][il] = (S)v;
            }
        }
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            int e = tid + 256 * u;
            int jl, pl;
            if (g.tb == 0) { pl = e / GBN; jl = e % GBN; } else { jl = e >> 4; pl = e & 15; }
            int j = j0 + jl, p = kt + pl;
            bool ok = (j < g.n) && (p < kend);
            if (g.triB == TRI_LOWER) ok = ok && (p >= j);
            if (g.triB == TRI_UPPER) ok = ok && (p <= j);
            if (MODE == GM_DF) {
                float hi = 0.f, lo = 0.f;
                if (ok) { hi = load_op(Bh, g.ldb, g.tb, p, j); lo = load_op(Bl, g.ldb, g.tb, p, j); }
                Bs[pl][jl] = hi;
                Bsl[pl][jl] = lo;
            } else {
                T v = 0;
                if (ok) v = load_op(B, g.ldb, g.tb, p, j);
                Bs[pl][jl] = (S)v;
            }
        }
        __syncthreads();
        if (MODE != GM_DF) {
#pragma unroll
            for (int p = 0; p < GBK; ++p) {
                S a[Q], b[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) { a[q] = As[p][ty + 16 * q]; b[q] = Bs[p][tx + 16 * q]; }
#pragma unroll
                for (int qa = 0; qa < Q; ++qa)
#pragma unroll
                    for (int qb = 0; qb < Q; ++qb) acc[qa][qb] = fma((T)a[qa], (T)b[qb], acc[qa][qb]);
            }
        } else {
#pragma unroll 4
            for (int p = 0; p < GBK; ++p) {
                float ahv[Q], alv[Q], bhv[Q], blv[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    ahv[q] = As[p][ty + 16 * q]; alv[q] = Asl[p][ty + 16 * q];
                    bhv[q] = Bs[p][tx + 16 * q]; blv[q] = Bsl[p][tx + 16 * q];
                }
#pragma unroll
                for (int qa = 0; qa < Q; ++qa)
#pragma unroll
                    for (int qb = 0; qb < Q; ++qb) {
                        // rounded intrinsics: never contracted, so the transformations stay error-free
                        float ph = __fmul_rn(ahv[qa], bhv[qb]);
                        float pe = __fmaf_rn(ahv[qa], bhv[qb], -ph);                 // hi*hi = ph + pe exactly
                        float cr = __fmaf_rn(ahv[qa], blv[qb], __fmul_rn(alv[qa], bhv[qb]));
                        float x = ah_[qa][qb];
                        float s = __fadd_rn(x, ph);                                  // TwoSum(x, ph)
                        float bp = __fsub_rn(s, x);
                        float er = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bp)), __fsub_rn(ph, bp));
                        ah_[qa][qb] = s;
                        al_[qa][qb] = __fadd_rn(al_[qa][qb], __fadd_rn(er, __fadd_rn(pe, cr)));
                    }
            }
            if (((++kt_count) & 7) == 0) {   // flush the float pairs into FP64 every 128 k
#pragma unroll
                for (int qa = 0; qa < Q; ++qa)
#pragma unroll
                    for (int qb = 0; qb < Q; ++qb) {
                        acc[qa][qb] += (double)ah_[qa][qb] + (double)al_[qa][qb];
                        ah_[qa][qb] = 0.f; al_[qa][qb] = 0.f;
                    }
            }
        }
        __syncthreads();
    }
    if (MODE == GM_DF) {
#pragma unroll
        for (int qa = 0; qa < Q; ++qa)
#pragma unroll
            for (int qb = 0; qb < Q; ++qb) acc[qa][qb] += (double)ah_[qa][qb] + (double)al_[qa][qb];
    }

    T *C = (T *)g.C + (long long)z * g.sC;
    const T *Cin = g.Cin ? (const T *)g.Cin + (long long)z * g.sCin : nullptr;
    const T alpha = (T)g.alpha, beta = (T)g.beta;
#pragma unroll
    for (int qa = 0; qa < Q; ++qa) {
        int i = i0 + ty + 16 * qa;
        if (i >= g.m) continue;
#pragma unroll
        for (int qb = 0; qb < Q; ++qb) {
            int j = j0 + tx + 16 * qb;
            if (j >= g.n) continue;
            if (g.lowerC && j > i) continue;
            T v = alpha * acc[qa][qb];
            if (g.beta != 0.0) v += beta * Cin[(long long)i * g.ldcin + j];
            C[(long long)i * g.ldc + j] = v;
        }
    }
}

// --------------------------------------------------------------------------
// FP64 GEMM on the DFMA pipe.  The pipe retires 2 DFMA per clock and SM -- a
// warp's DFMA occupies its sub-partition for 64 clocks -- so a tile needs only
// enough warps (8) and no register blocking to keep it busy: shared-memory and
// L2 traffic stay below a tenth of their rates even with 16 x 16 tiles.  What
// bounds a product is then how evenly its multiply-adds spread over the 152
// pipes, so the tile is chosen per launch (dgemm_tile) among
//   32 x 32 (2 x 2 outputs per thread), 16 x 16 (one output per thread) and
//   8 x 8 (four threads per output, each every fourth k; sums added in order).
// Each k block is prefetched into registers while the previous one is used.
// Measured (one launch, GB300): 128^3 113 us with 64 x 64 tiles on four SMs -> 9 us;
// 2048^3 14.4 ms, 1.19 TFLOP/s of the pipe's 1.26.
// --------------------------------------------------------------------------
template <int TS> struct DgemmTile;
template <> struct DgemmTile<32> { static constexpr int R = 2, KS = 1, BK = 16; };
template <> struct DgemmTile<16> { static constexpr int R = 1, KS = 1, BK = 32; };
template <> struct DgemmTile<8> { static constexpr int R = 1, KS = 4, BK = 64; };

// tile t of a row-by-row count of the tiles (bi, bj) with bj <= bi and bj < nt
__device__ __forceinline__ void dgemm_lower_tile(int t, int nt, int &bi, int &bj)
{
    const int tri = nt * (nt + 1) / 2;
    if (t >= tri) {
        bi = nt + (t - tri) / nt;
        bj = (t - tri) % nt;
        return;
    }
    bi = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (bi * (bi + 1) / 2 > t) --bi;
    while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
    bj = t - bi * (bi + 1) / 2;
}

template <int TS>
__global__ void __launch_bounds__(256) dgemm_kernel(GemmArgs g)
{
    constexpr int R = DgemmTile<TS>::R, KS = DgemmTile<TS>::KS, BK = DgemmTile<TS>::BK, TD = TS / R;
    static_assert(TD * TD * KS == 256 && TS * BK == 512, "256 threads, two elements per thread and operand");
    // tile of this CTA; long k ranges first: with op(A) lower or op(B) upper triangular they
    // are at the far end.  lowerC: the grid counts the tiles on and below the diagonal alone
    // (CTAs that leave at once would take their turn in the round-robin over the SMs).
    int bi, bj;
    const int z = blockIdx.z;
    if (g.lowerC) {
        const int t = g.triA == TRI_LOWER ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
        dgemm_lower_tile(t, (g.n + TS - 1) / TS, bi, bj);
    } else {
        bi = g.triA == TRI_LOWER ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
        bj = g.triB == TRI_UPPER ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    }
    const int i0 = bi * TS, j0 = bj * TS;
    const double *A = (const double *)g.A + (long long)z * g.sA;
    const double *B = (const double *)g.B + (long long)z * g.sB;
    const double *ks = (const double *)g.kscale;
    int kbeg = 0, kend = g.k;
    if (g.triA == TRI_LOWER) kend = min(kend, i0 + TS);
    if (g.triA == TRI_UPPER) kbeg = max(kbeg, i0);
    if (g.triB == TRI_LOWER) kbeg = max(kbeg, j0);
    if (g.triB == TRI_UPPER) kend = min(kend, j0 + TS);

    __shared__ double As[2][BK][TS + 1], Bs[2][BK][TS + 1];
    __shared__ double red[KS > 1 ? KS - 1 : 1][KS > 1 ? TD * TD : 1];
    const int tid = threadIdx.x, kg = tid / (TD * TD), tx = tid % TD, ty = (tid / TD) % TD;
    double acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] = 0.0;

    double ra[2], rb[2];
    auto fetch = [&](int kt) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = tid + 256 * u;
            {   // consecutive threads along the operand's memory rows
                const int il = g.ta ? e % TS : e / BK, pl = g.ta ? e / TS : e % BK, i = i0 + il, p = kt + pl;
                bool ok = i < g.m && p < kend;
                if (g.triA == TRI_LOWER) ok = ok && p <= i;
                if (g.triA == TRI_UPPER) ok = ok && p >= i;
                double v = 0.0;
                if (ok) {
                    v = load_op(A, g.lda, g.ta, i, p);
                    if (ks) v *= ks[p];
                }
                ra[u] = v;
            }
            {
                const int jl = g.tb ? e / BK : e % TS, pl = g.tb ? e % BK : e / TS, j = j0 + jl, p = kt + pl;
                bool ok = j < g.n && p < kend;
                if (g.triB == TRI_LOWER) ok = ok && p >= j;
                if (g.triB == TRI_UPPER) ok = ok && p <= j;
                rb[u] = ok ? load_op(B, g.ldb, g.tb, p, j) : 0.0;
            }
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = tid + 256 * u;
            As[s][g.ta ? e / TS : e % BK][g.ta ? e % TS : e / BK] = ra[u];
            Bs[s][g.tb ? e % BK : e / TS][g.tb ? e / BK : e % TS] = rb[u];
        }
    };
    if (kbeg < kend) {
        fetch(kbeg);
        store(0);
        __syncthreads();
        for (int kt = kbeg, s = 0; kt < kend; kt += BK, s ^= 1) {
            const bool more = kt + BK < kend;
            if (more) fetch(kt + BK);
#pragma unroll 8
            for (int p = kg; p < BK; p += KS) {
                double a[R], b[R];
#pragma unroll
                for (int q = 0; q < R; ++q) { a[q] = As[s][p][ty + TD * q]; b[q] = Bs[s][p][tx + TD * q]; }
#pragma unroll
                for (int qa = 0; qa < R; ++qa)
#pragma unroll
                    for (int qb = 0; qb < R; ++qb) acc[qa][qb] = fma(a[qa], b[qb], acc[qa][qb]);
            }
            if (more) store(s ^ 1);
            __syncthreads();
        }
    }
    if (KS > 1) {
        if (kg > 0) red[kg - 1][tid % (TD * TD)] = acc[0][0];
        __syncthreads();
        if (kg > 0) return;
#pragma unroll
        for (int q = 0; q < KS - 1; ++q) acc[0][0] += red[q][tid];
    }
    double *C = (double *)g.C + (long long)z * g.sC;
    const double *Cin = g.Cin ? (const double *)g.Cin + (long long)z * g.sCin : nullptr;
#pragma unroll
    for (int qa = 0; qa < R; ++qa) {
        const int i = i0 + ty + TD * qa;
        if (i >= g.m) continue;
#pragma unroll
        for (int qb = 0; qb < R; ++qb) {
            const int j = j0 + tx + TD * qb;
            if (j >= g.n || (g.lowerC && j > i)) continue;
            double v = g.alpha * acc[qa][qb];
            if (g.beta != 0.0) v += g.beta * Cin[(long long)i * g.ldcin + j];
            C[(long long)i * g.ldc + j] = v;
        }
    }
}

// tiles of order ts that are worked on, per batch matrix
static long long dgemm_tiles(const GemmArgs &g, int ts)
{
    const long long mt = (g.m + ts - 1) / ts, nt = (g.n + ts - 1) / ts;
    if (!g.lowerC) return mt * nt;
    const long long d = std::min(mt, nt);
    return d * (d + 1) / 2 + (mt > nt ? (mt - nt) * nt : 0);
}

// time of the busiest pipe in units of outputs x k, the tiles dealt out over 152 SMs
static double dgemm_cost(const GemmArgs &g, int ts)
{
    return std::ceil((double)dgemm_tiles(g, ts) * g.batch / 152.0) * ts * ts;
}

// The largest tile whose busiest SM has no more work than the smaller tiles' allow for: a
// smaller tile costs a few percent more instructions per DFMA, hence its handicap.
static int dgemm_tile(const GemmArgs &g)
{
    const double c32 = dgemm_cost(g, 32), c16 = 1.04 * dgemm_cost(g, 16), c8 = 1.15 * dgemm_cost(g, 8);
    if (c32 <= c16 && c32 <= c8) return 32;
    return c16 <= c8 ? 16 : 8;
}

// estimate of the DFMA engine's time in microseconds: the busiest SM's multiply-adds at
// 2 per clock and 2 GHz, and the launch
double dgemm_time_us(const GemmArgs &g)
{
    return dgemm_cost(g, dgemm_tile(g)) * g.k / 4000.0 + 4.0;
}

static void dgemm_launch(const GemmArgs &g, cudaStream_t s)
{
    const int ts = dgemm_tile(g);
    const dim3 grid = g.lowerC ? dim3((unsigned)dgemm_tiles(g, ts), 1, g.batch)
                               : dim3((g.n + ts - 1) / ts, (g.m + ts - 1) / ts, g.batch);
    if (ts == 32) dgemm_kernel<32><<<grid, 256, 0, s>>>(g);
    else if (ts == 16) dgemm_kernel<16><<<grid, 256, 0, s>>>(g);
    else dgemm_kernel<8><<<grid, 256, 0, s>>>(g);
    count_launch();
}

void gemm_launch(const GemmArgs &g, cudaStream_t s)
{
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return;
    const auto grid = [&](int tile) { return dim3((g.n + tile - 1) / tile, (g.m + tile - 1) / tile, g.batch); };
    const dim3 g64 = grid(64);
    switch (g.mode) {
    case GM_F32: gemm_kernel<GM_F32, 4><<<g64, 256, 0, s>>>(g); count_launch(); break;
    case GM_DF:
        // A float-pair multiply-add is 13 instructions, so a small product takes as long as a thread's
        // share of it: tiles of 16 while they fit on the chip (32 x 64 x 64: 22 us, 2 us with them).
        // Up to k = 128, where no flush lies inside the product, a tile's k range does not show in the
        // result's bits.
        if (g.k <= 128 && 16ll * g64.x * g64.y * g64.z <= 4 * 152)
            gemm_kernel<GM_DF, 1><<<grid(16), 256, 0, s>>>(g);
        else
            gemm_kernel<GM_DF, 4><<<g64, 256, 0, s>>>(g);
        count_launch();
        break;
    default: dgemm_launch(g, s); break;
    }
}

// --------------------------------------------------------------------------
// Cholesky of one diagonal block (<= 128 in FP32, <= 64 in FP64) and its
// triangular inverse, blocked by 32 columns, one CTA per batch matrix
// --------------------------------------------------------------------------
struct LeafPivot {
    static __device__ __forceinline__ void get(float d, float &piv, float &r) { piv = sqrtf(d); r = 1.0f / piv; }
    // 1/sqrt(d) for a positive finite d.  The FP64 pipe is narrow: a float reciprocal square
    // root refined by two Newton steps y <- y (3 - d y^2) / 2 (each doubles the number of
    // correct bits) replaces the square root and the division; outside the float range the
    // library functions are used.  Comparisons, conversions (to float: to nearest even) and the
    // halving work on the bit patterns, since the FP64 pipe would take 64 clocks for each.
    static __device__ __forceinline__ bool in_range(double d)   // 1e-30 < d < 1e30
    {
        const long long u = __double_as_longlong(d);
        return u > __double_as_longlong(1e-30) && u < __double_as_longlong(1e30);
    }
    static __device__ __forceinline__ bool positive_finite(double d)
    {
        const long long u = __double_as_longlong(d);
        return u > 0 && u < 0x7FF0000000000000LL;
    }
    static __device__ __forceinline__ double rsqrt_start(double d)     // of float accuracy, for d in range
    {
        const unsigned long long u = (unsigned long long)__double_as_longlong(d);
        const unsigned int f = (unsigned int)((u + 0x0FFFFFFFull + ((u >> 29) & 1ull)) >> 29) - (896u << 23);
        float g;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(__uint_as_float(f)));
        return __longlong_as_double((long long)(((unsigned long long)__float_as_uint(g) << 29) + (896ull << 52)));
    }
    static __device__ __forceinline__ double rsqrt_newton(double d, double y)
    {
        const double h = __longlong_as_double(__double_as_longlong(d) - (1ll << 52));   // d / 2
        return y * fma(-(h * y), y, 1.5);
    }
};

// ---- FP64: blocks of at most 64, two block columns of 32 ----
//
// What bounds it: a warp's FP64 instruction occupies its sub-partition for 64 clocks and its
// result is there after 66, so a sub-partition is a queue of one instruction at a time and
// latency cannot be hidden, only shared out over the four of them.  The chain is the 64
// columns one after another: update, reciprocal square root (six dependent FP64
// instructions), scale, about 800 clocks each.  So one warp does nothing but that chain on a
// sub-partition of its own; a column is published through an mbarrier as soon as it is
// final; the three warps that bring the later columns up to date begin with the one the chain
// takes next, and the inverse follows row by row in three other warps.  The products around
// the two diagonal blocks are laid out so that every lane has an entry inside the triangles.
// Measured (64 x 64, one CTA): 52 us; 105 us with all warps meeting at two barriers per
// column and half of the lanes idle.

constexpr int LEAF64_WARPS = 12, LEAF64_THREADS = 32 * LEAF64_WARPS;
constexpr unsigned int LEAF_WAIT_LIMIT = 1u << 20;    // polls of one wait

// The waits of one warp of a leaf (every barrier is used for one phase), at most LIMIT polls each.
// One that runs out is reported at the leaf's end (leaf_lost); the warp goes on, what it forms
// being thrown away with the call.  The bound is known at compile time and the outcome one
// integer: 59.4 us an FP64 leaf as against 59.2 without a report, 61 with a bound in a register.
template <unsigned int LIMIT> struct LeafWaits {
    uint32_t ok = 1;
    __device__ __forceinline__ void wait(uint32_t bar) { ok &= mbar_wait_first<LIMIT>(bar); }
    __device__ __forceinline__ void report(int *lost) const { if (!ok) *lost = 1; }
};

// one thread, after every warp: a wait ran out, so the block is not factorised
__device__ __forceinline__ void leaf_lost(int lost, int *err, int *info, int z, int off)
{
    if (!lost) return;
    if (err) atomicExch(err, 5);
    if (info[z] == 0) info[z] = off + 1;
}

// Warp 0: the chain of a w x w (w <= 32) diagonal block at Lb (row stride ls, zeros above the
// diagonal), D = L_D L_D^T.  Lane i has row i.  Column c, brought up to date with the columns
// before c - 1 and signalled in ready[c] (c >= 2), takes its last update, is scaled, goes back
// to Lb with rv[c] = 1/L_cc, and is signalled in done[c].  A pivot that is not positive and
// finite is recorded in info[z] (global index gpiv + c + 1, first one only) and taken as 1.
//
// Every lane forms the pivot itself, from L_c,c-1 and the diagonal entry, so that it does not
// wait for lane c's; the next column is loaded while the square root is under way.
template <class W>
__device__ __forceinline__ void leaf64_chain(double *Lb, int ls, int w, double *rv, uint32_t done, uint32_t ready,
                                             int lane, int *info, int z, int gpiv, int *bad, W &waits)
{
    double *row = Lb + min(lane, w - 1) * ls;         // (lanes beyond the last row repeat it)
    double v = 0.0, vc = 0.0, d = row[0], dc = Lb[0];
    for (int c = 0; c < w; ++c) {
        double pv = fma(-vc, vc, dc);
        const int cn = min(c + 1, w - 1);
        const double y = LeafPivot::rsqrt_start(pv);  // (any bits, if pv is out of range)
        d = fma(-v, vc, d);
        const double y1 = LeafPivot::rsqrt_newton(pv, y);
        if (cn >= 2 && cn > c) waits.wait(ready + 8 * cn);
        const double dn = row[cn];
        dc = Lb[cn * ls + cn];
        double r = LeafPivot::rsqrt_newton(pv, y1);   // 1/L_cc; lane c: L_cc = pv r
        v = (lane == c ? pv : d) * r;
        if (!LeafPivot::in_range(pv)) {
            if (!LeafPivot::positive_finite(pv)) {
                if (lane == 0 && !*bad) { *bad = 1; if (info[z] == 0) info[z] = gpiv + c + 1; }
                pv = 1.0;
            }
            const double piv = sqrt(pv);
            r = 1.0 / piv;
            v = lane == c ? piv : d * r;
        }
        vc = __shfl_sync(0xffffffffu, v, cn);
        if (lane >= c && lane < w) row[c] = v;
        if (lane == 0) rv[c] = r;
        __syncwarp();
        mbar_arrive_if(done + 8 * c, lane == 0);
        d = dn;
    }
}

// Three warps (u = 0 .. 2): columns u, u + 3, ... of the same block, lane i row i, take the
// columns before their last but one in turn and are signalled in ready.
template <class W>
__device__ __forceinline__ void leaf64_update(double *Lb, int ls, int w, uint32_t done, uint32_t ready, int u, int lane,
                                              W &waits)
{
    double d[11];
#pragma unroll
    for (int p = 0; p < 11; ++p) {
        const int c = 3 * p + u;
        d[p] = (lane < w && c <= lane) ? Lb[lane * ls + c] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < 30; ++j) {
        if (j + 2 < w) {
            waits.wait(done + 8 * j);
            const double li = lane < w ? Lb[lane * ls + j] : 0.0;
#pragma unroll
            for (int p = 0; p < 11; ++p) {
                if (3 * p + 2 < j + 2) continue;
                const int c = 3 * p + u;
                if (c >= j + 2 && c < w) {
                    d[p] = fma(-li, Lb[c * ls + j], d[p]);
                    if (c == j + 2) {
                        if (lane >= c && lane < w) Lb[lane * ls + c] = d[p];
                        __syncwarp();
                        if (lane == 0) mbar_arrive(ready + 8 * c);
                    }
                }
            }
        }
    }
}

// Three warps (iw = 0 .. 2): X_D = L_D^{-1} into Xb, zeros above the diagonal, behind the
// factorisation: lane c holds column c, warp iw the rows iw, iw + 3, ...
//   x_cc = 1/L_cc,  x_kc = -(sum_{m=c}^{k-1} L_km x_mc) / L_kk,
// the sum in four parts, m - c = 0 .. 3 (mod 4), added as (0 + 1) + (2 + 3).  Part p of column
// c is slot (c + p) mod 4 = m mod 4, so that a slot is the same register in every lane.  Row j
// is signalled in row[j]; the warp of row j + 1 finishes that one before its other rows.
template <class W>
__device__ __forceinline__ void leaf64_invert(const double *Lb, double *Xb, int ls, int w, const double *rv,
                                              uint32_t done, uint32_t row, int iw, int lane, W &waits)
{
    double a[11][4];
#pragma unroll
    for (int p = 0; p < 11; ++p)
#pragma unroll
        for (int t = 0; t < 4; ++t) a[p][t] = 0.0;
    const bool even = !(lane & 1);
    auto finish = [&](int j, const double *s) {
        waits.wait(done + 8 * j);
        const double r = rv[j];
        const double sum = ((even ? s[0] : s[2]) + s[1]) + ((even ? s[2] : s[0]) + s[3]);
        if (lane < w) Xb[j * ls + lane] = lane < j ? -sum * r : (lane == j ? r : 0.0);
        __syncwarp();
        if (lane == 0) mbar_arrive(row + 8 * j);
    };
    if (iw == 0) finish(0, a[0]);
#pragma unroll
    for (int j = 0; j < 31; ++j) {
        if (j + 1 < w) {
            waits.wait(row + 8 * j);      // (row j was finished after column j)
            const double x = lane <= j ? Xb[j * ls + lane] : 0.0;
#pragma unroll
            for (int p = 0; p < 11; ++p) {
                if (3 * p + 2 < j + 1) continue;
                const int k = 3 * p + iw;
                if (k >= j + 1 && k < w) {
                    a[p][j & 3] = fma(Lb[k * ls + j], x, a[p][j & 3]);
                    if (k == j + 1) finish(j + 1, a[p]);
                }
            }
        }
    }
}

// The s x s (s <= 64) diagonal block at (off, off) of batch matrix blockIdx.x:
//   1. L_11 (warps 0-3) and X_11 = L_11^{-1} (warps 5-7);
//   2. L_21 = A_21 X_11^T: lane i has row i, warp v the columns v, 15 - v, 16 + v, 31 - v
//      (66 multiply-adds each), in short loops -- code that runs once is bound by its fetch;
//   3. A_22 -= L_21 L_21^T, lower part: columns j and 32 - j share a warp's lanes;
//   4. L_22 and X_22, while warps 9-11 form W = L_21 X_11;
//   5. X_21 = -X_22 W.
// Every sum runs over its index in ascending order.  Warps 0, 4 and 8 share a sub-partition,
// which 2 and 3 apart is left to the chain.
template <unsigned int LIMIT>
__global__ void __launch_bounds__(LEAF64_THREADS)
chol_leaf64_kernel(double *A, long long lda, long long sA, double *Rinv, long long ldr, long long sR, int off, int s,
                   int *info, int *err)
{
    extern __shared__ unsigned char leaf_smem[];
    const int ls = s | 1;                            // odd: a column is free of bank conflicts
    double *L = (double *)leaf_smem, *X = L + (size_t)s * ls, *W = X + (size_t)s * ls;   // W: 32 x 33
    double *rv = W + 32 * 33;
    __shared__ int bad, lost;
    __shared__ unsigned long long bars[192];         // columns of L done, ready for the chain, rows of X
    const int z = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t done = smem_u32(bars), ready = smem_u32(bars + 64), row = smem_u32(bars + 128);
    A += (long long)z * sA + (long long)off * lda + off;
    Rinv += (long long)z * sR + (long long)off * ldr + off;
    if (tid == 0) { bad = 0; lost = 0; }
    LeafWaits<LIMIT> waits;
    if (tid < 192) mbar_init(done + 8 * tid, 1);
    {   // all loads of a thread in flight at once
        constexpr int NL = (64 * 64 + LEAF64_THREADS - 1) / LEAF64_THREADS;
        double v[NL];
#pragma unroll
        for (int t = 0; t < NL; ++t) {
            const int e = tid + t * LEAF64_THREADS, r = e >> 6, c = e & 63;
            v[t] = (r < s && c <= r) ? A[(long long)r * lda + c] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < NL; ++t) {
            const int e = tid + t * LEAF64_THREADS, r = e >> 6, c = e & 63;
            if (r < s && c < s) { L[r * ls + c] = v[t]; X[r * ls + c] = 0.0; }
        }
    }
    __syncthreads();
    const int w1 = min(32, s), w2 = s - w1;
    if (warp == 0) leaf64_chain(L, ls, w1, rv, done, ready, lane, info, z, off, &bad, waits);
    else if (warp < 4) leaf64_update(L, ls, w1, done, ready, warp - 1, lane, waits);
    else if (warp > 4 && warp < 8) leaf64_invert(L, X, ls, w1, rv, done, row, warp - 5, lane, waits);
    waits.report(&lost);
    __syncthreads();
    if (w2 > 0) {
        double *L21 = L + 32 * ls;
        if (warp < 8) {
            const double *a = L21 + min(lane, w2 - 1) * ls;      // (rows beyond the last repeat it, unused)
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
                const int c = 8 * t + ((t & 1) ? 7 - warp : warp);
                const double *x = X + c * ls;
                double acc = 0.0;
#pragma unroll 4
                for (int m = 0; m <= c; ++m) acc = fma(a[m], x[m], acc);
                W[lane * 33 + c] = acc;
            }
        }
        __syncthreads();
        for (int e = tid; e < w2 * 32; e += LEAF64_THREADS) L21[(e >> 5) * ls + (e & 31)] = W[(e >> 5) * 33 + (e & 31)];
        for (int t = warp; t < 17; t += LEAF64_WARPS) {
            const bool hi = lane >= t;
            const int i = hi ? lane : 32 - t + lane, j = hi ? t : 32 - t;
            double acc = 0.0;
#pragma unroll 8
            for (int c = 0; c < 32; ++c) acc = fma(W[i * 33 + c], W[j * 33 + c], acc);
            if (i < w2 && (t < 16 || hi)) L[(32 + i) * ls + 32 + j] -= acc;
        }
        __syncthreads();
        double *L22 = L + 32 * ls + 32;
        if (warp == 0) {
            leaf64_chain(L22, ls, w2, rv + 32, done + 256, ready + 256, lane, info, z, off + 32, &bad,
                         waits);
        } else if (warp < 4) {
            leaf64_update(L22, ls, w2, done + 256, ready + 256, warp - 1, lane, waits);
        } else if (warp > 4 && warp < 8) {
            leaf64_invert(L22, X + 32 * ls + 32, ls, w2, rv + 32, done + 256, row + 256, warp - 5, lane,
                          waits);
        } else if (warp > 8) {
            const double *l = L21 + min(lane, w2 - 1) * ls;
            for (int c = warp - 9; c < 32; c += 3) {
                double acc = 0.0;
#pragma unroll 4
                for (int q = c; q < 32; ++q) acc = fma(l[q], X[q * ls + c], acc);
                W[lane * 33 + c] = acc;
            }
        }
        waits.report(&lost);
        __syncthreads();
        if (warp < 8) {
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
                const int r = 8 * t + ((t & 1) ? 7 - warp : warp);
                if (r >= w2) break;                  // (r ascends)
                double *x = X + (32 + r) * ls;
                double acc = 0.0;
#pragma unroll 4
                for (int q = 0; q <= r; ++q) acc = fma(x[32 + q], W[q * 33 + lane], acc);
                x[lane] = -acc;
            }
        }
        __syncthreads();
    }
    if (tid == 0) leaf_lost(lost, err, info, z, off);
    for (int r = warp; r < s; r += LEAF64_WARPS)
        for (int c = lane; c < s; c += 32) {
            A[(long long)r * lda + c] = (c <= r) ? L[r * ls + c] : 0.0;
            Rinv[(long long)r * ldr + c] = (c <= r) ? X[r * ls + c] : 0.0;
        }
}

// ---- FP32: blocks of at most 128, four block columns of 32 ----
//
// The same division of work as in FP64: a chain warp that publishes column after column, three
// warps that bring the later columns up to date in shared memory, three that follow with the
// inverse.  What bounds it here is latency -- a column's square root, reciprocal and hand-over,
// about 200 clocks -- and, for code that runs a few times per launch, its fetch: with a block
// unrolled in the registers of one warp a leaf took 100 us.  Measured (128 x 128): 62 us.

template <class W>
__device__ __forceinline__ void leaf32_chain(float *Lb, int ls, int w, float *rv, uint32_t done, uint32_t ready,
                                             int lane, int *info, int z, int gpiv, int *bad, W &waits)
{
    float *row = Lb + min(lane, w - 1) * ls;          // (lanes beyond the last row repeat it)
    float v = 0.f, vc = 0.f, d = row[0], dc = Lb[0];
    for (int c = 0; c < w; ++c) {
        float pv = fmaf(-vc, vc, dc);
        d = fmaf(-v, vc, d);
        if (!(pv > 0.f) || !isfinite(pv)) {
            if (lane == 0 && !*bad) { *bad = 1; if (info[z] == 0) info[z] = gpiv + c + 1; }
            pv = 1.f;
        }
        const int cn = min(c + 1, w - 1);
        float piv, r;
        LeafPivot::get(pv, piv, r);
        v = lane == c ? piv : d * r;
        vc = __shfl_sync(0xffffffffu, v, cn);
        if (lane >= c && lane < w) row[c] = v;
        if (lane == 0) rv[c] = r;
        __syncwarp();
        mbar_arrive_if(done + 8 * c, lane == 0);
        if (cn >= 2 && cn > c) waits.wait(ready + 8 * cn);
        d = row[cn];
        dc = Lb[cn * ls + cn];
    }
}

// columns u, u + 3, ...: the columns before their last but one, in turn
template <class W>
__device__ __forceinline__ void leaf32_update(float *Lb, int ls, int w, uint32_t done, uint32_t ready, int u, int lane,
                                              W &waits)
{
    float *row = Lb + min(lane, w - 1) * ls;
    for (int j = 0; j + 2 < w; ++j) {
        waits.wait(done + 8 * j);
        const float li = row[j];
        for (int c0 = j + 2 + (u + 6 - (j + 2) % 3) % 3; c0 < w; c0 += 12) {
            float v[4];                               // four columns' loads, then their stores
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int c = min(c0 + 3 * t, w - 1);
                v[t] = fmaf(-li, Lb[c * ls + j], row[c]);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (c0 + 3 * t < w && lane >= c0 + 3 * t && lane < w) row[c0 + 3 * t] = v[t];
            if (c0 == j + 2) {
                __syncwarp();
                mbar_arrive_if(ready + 8 * c0, lane == 0);
            }
        }
    }
}

// rows iw, iw + 3, ... of X_D = L_D^{-1}: x_kc = -(sum_m L_km x_mc) / L_kk, m ascending, the
// sums growing in Xb (zero at first)
template <class W>
__device__ __forceinline__ void leaf32_invert(const float *Lb, float *Xb, int ls, int w, const float *rv, uint32_t done,
                                              uint32_t row, int iw, int lane, W &waits)
{
    const int col = min(lane, w - 1);
    auto finish = [&](int j) {
        waits.wait(done + 8 * j);
        const float r = rv[j], acc = Xb[j * ls + col];
        if (lane < w) Xb[j * ls + lane] = lane < j ? -acc * r : (lane == j ? r : 0.f);
        __syncwarp();
        mbar_arrive_if(row + 8 * j, lane == 0);
    };
    if (iw == 0) finish(0);
    for (int j = 0; j + 1 < w; ++j) {
        waits.wait(row + 8 * j);
        const float x = Xb[j * ls + col];
        for (int k0 = j + 1 + (iw + 6 - (j + 1) % 3) % 3; k0 < w; k0 += 12) {
            float v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int k = min(k0 + 3 * t, w - 1);
                v[t] = fmaf(Lb[k * ls + j], x, Xb[k * ls + col]);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (k0 + 3 * t < w && lane < w) Xb[(k0 + 3 * t) * ls + lane] = v[t];
            if (k0 == j + 1) { __syncwarp(); finish(k0); }
        }
    }
}

// The s x s (s <= 128) diagonal block at (off, off) of batch matrix blockIdx.x, right-looking by
// blocks of 32 columns with 8 warps:
//   1. the diagonal block and its inverse X_D (warp 0, warps 1-3, warps 5-7);
//   2. panel L_21 = A_21 X_D^T: a warp per row of A_21, lane c holding row c of X_D in
//      registers, the row of A_21 read as shared-memory broadcasts;
//   3. trailing update A_22 -= L_21 L_21^T: lane j holding rows j, j + 32, j + 64 of L_21 in
//      registers, a warp per row i, the lower triangle stored.
// Then the off-diagonal blocks of X = L^{-1}, block row i after block row i - 1:
// X_ik = -X_ii (sum_{m=k}^{i-1} L_im X_mk), all k < i at once, four rows per warp.
template <unsigned int LIMIT>
__global__ void __launch_bounds__(256) chol_leaf128_kernel(float *A, long long lda, long long sA, float *Rinv,
                                                           long long ldr, long long sR, int off, int s, int *info,
                                                           int *err)
{
    constexpr int NQ = 3;                     // 32-row groups of a panel
    extern __shared__ unsigned char leaf_smem[];
    const int ls = s | 1;
    float *L = (float *)leaf_smem;            // the block, then L
    float *X = L + (size_t)s * ls;            // L^{-1}
    float *W = X + (size_t)s * ls;            // s x 33: the panel, then block products of the inverse
    float *rv = W + (size_t)s * 33;           // 1 / L_jj
    __shared__ int bad, lost;
    __shared__ unsigned long long bars[4 * 96];   // per block column: done, ready, rows of X
    const int z = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    A += (long long)z * sA + (long long)off * lda + off;
    Rinv += (long long)z * sR + (long long)off * ldr + off;
    if (tid == 0) { bad = 0; lost = 0; }
    LeafWaits<LIMIT> waits;
    for (int e = tid; e < 4 * 96; e += 256) mbar_init(smem_u32(bars + e), 1);
    for (int e0 = tid; e0 < 128 * 128; e0 += 256 * 16) {   // 16 loads of a thread in flight at once
        float v[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const int e = e0 + 256 * t, r = e >> 7, c = e & 127;
            v[t] = (r < s && c <= r) ? A[(long long)r * lda + c] : 0.f;
        }
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const int e = e0 + 256 * t, r = e >> 7, c = e & 127;
            if (r < s && c < s) { L[r * ls + c] = v[t]; X[r * ls + c] = 0.f; }
        }
    }
    __syncthreads();
    const int nb = (s + 31) >> 5;
    for (int kb = 0; kb < nb; ++kb) {
        const int o = kb * 32, w = min(32, s - o), o2 = o + w, rows = s - o2;
        {
            float *Ld = L + o * ls + o;
            const uint32_t done = smem_u32(bars + 96 * kb), ready = done + 256, row = done + 512;
            if (warp == 0) leaf32_chain(Ld, ls, w, rv + o, done, ready, lane, info, z, off + o, &bad, waits);
            else if (warp < 4) leaf32_update(Ld, ls, w, done, ready, warp - 1, lane, waits);
            else if (warp > 4) leaf32_invert(Ld, X + o * ls + o, ls, w, rv + o, done, row, warp - 5, lane, waits);
            waits.report(&lost);
        }
        __syncthreads();
        if (rows > 0) {                       // (w = 32)
            {   // W[i][c] = sum_{m <= c} A[o2 + i][o + m] X_D[c][m]
                float xd[32];
#pragma unroll
                for (int m = 0; m < 32; ++m) xd[m] = X[(o + lane) * ls + o + m];
                for (int i = warp; i < rows; i += 8) {
                    const float *a = L + (o2 + i) * ls + o;
                    float acc = 0.f;
#pragma unroll
                    for (int m = 0; m < 32; ++m) acc += a[m] * xd[m];
                    W[i * 33 + lane] = acc;
                }
            }
            __syncthreads();
            {
                float wr[NQ][32];
#pragma unroll
                for (int q = 0; q < NQ; ++q)
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        const int j = lane + 32 * q;
                        wr[q][c] = j < rows ? W[j * 33 + c] : 0.f;
                    }
                for (int i = warp; i < rows; i += 8) {
                    const float *wi = W + i * 33;
                    float acc[NQ];
#pragma unroll
                    for (int q = 0; q < NQ; ++q) acc[q] = 0.f;
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        const float v = wi[c];
#pragma unroll
                        for (int q = 0; q < NQ; ++q) acc[q] += v * wr[q][c];
                    }
                    float *lrow = L + (o2 + i) * ls;
                    lrow[o + lane] = wi[lane];
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int j = lane + 32 * q;
                        if (j <= i) lrow[o2 + j] -= acc[q];
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int ib = 1; ib < nb; ++ib) {
        const int o = ib * 32, w = min(32, s - o), hw = (w + 3) >> 2;
        for (int idx = warp; idx < ib * hw; idx += 8) {    // W[32 k + r][c] = sum_{q in [32 k, o)} L[o + r][q] X[q][32 k + c]
            const int k = idx / hw, r0 = 4 * (idx - k * hw);
            const float *l[4];
            float a[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) { l[t] = L + (o + min(r0 + t, w - 1)) * ls; a[t] = 0.f; }
#pragma unroll 8
            for (int q = k * 32; q < o; ++q) {
                const float xv = X[q * ls + k * 32 + lane];
#pragma unroll
                for (int t = 0; t < 4; ++t) a[t] += l[t][q] * xv;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (r0 + t < w) W[(k * 32 + r0 + t) * 33 + lane] = a[t];
        }
        __syncthreads();
        for (int idx = warp; idx < ib * hw; idx += 8) {    // X[o + r][32 k + c] = -sum_{q <= r} X_ii[r][q] W[32 k + q][c]
            const int k = idx / hw, r0 = 4 * (idx - k * hw);
            const float *d[4];
            float a[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) { d[t] = X + (o + min(r0 + t, w - 1)) * ls + o; a[t] = 0.f; }
            const int qn = min(r0 + 4, w);                 // (X_ii is zero above its diagonal)
#pragma unroll 4
            for (int q = 0; q < qn; ++q) {
                const float wv = W[(k * 32 + q) * 33 + lane];
#pragma unroll
                for (int t = 0; t < 4; ++t) a[t] += d[t][q] * wv;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (r0 + t < w) X[(o + r0 + t) * ls + k * 32 + lane] = -a[t];
        }
        __syncthreads();
    }
    if (tid == 0) leaf_lost(lost, err, info, z, off);
    for (int r = warp; r < s; r += 8)
        for (int c = lane; c < s; c += 32) {
            A[(long long)r * lda + c] = (c <= r) ? L[r * ls + c] : 0.f;
            Rinv[(long long)r * ldr + c] = (c <= r) ? X[r * ls + c] : 0.f;
        }
}

// dynamic shared memory: the block, its inverse, a panel, the reciprocals of the diagonal
static size_t chol_leaf_smem(int s, bool fp64)
{
    return fp64 ? (2 * (size_t)s * (s | 1) + 32 * 33 + 64) * sizeof(double)
                : (2 * (size_t)s * (s | 1) + 34 * (size_t)s) * sizeof(float);
}

template <class T>
int chol_leaf(T *A, long long lda, long long sA, T *Rinv, long long ldr, long long sR, int off, int s, int batch,
              int *info, int *err, bool one_poll, cudaStream_t st)
{
    constexpr bool fp64 = sizeof(T) == 8;
    if (s <= 0 || s > CholLeaf<T>::max_s) return -2;
    const auto launch = [&](auto kernel) {
        if (!ensure_dynamic_smem((const void *)kernel, (int)chol_leaf_smem(CholLeaf<T>::max_s, fp64))) return false;
        kernel<<<batch, fp64 ? LEAF64_THREADS : 256, chol_leaf_smem(s, fp64), st>>>(A, lda, sA, Rinv, ldr, sR, off, s, info,
                                                                                    err);
        return true;
    };
    bool ok;
    if constexpr (fp64) ok = one_poll ? launch(chol_leaf64_kernel<1>) : launch(chol_leaf64_kernel<LEAF_WAIT_LIMIT>);
    else ok = one_poll ? launch(chol_leaf128_kernel<1>) : launch(chol_leaf128_kernel<LEAF_WAIT_LIMIT>);
    if (!ok) return -1;
    count_launch();
    return 0;
}

template int chol_leaf<double>(double *, long long, long long, double *, long long, long long, int, int, int, int *,
                               int *, bool, cudaStream_t);
template int chol_leaf<float>(float *, long long, long long, float *, long long, long long, int, int, int, int *, int *,
                              bool, cudaStream_t);

// --------------------------------------------------------------------------
// HBM passes with 32x32 shared-memory tiles
// --------------------------------------------------------------------------
constexpr int TT = 32;

// M = (Sig H + (Sig H)^T)/2 and the squared defect ||Sig H - (Sig H)^T||_F^2 and
// ||Sig H||_F^2, block partials, over tile pairs (bi >= bj).
__global__ void __launch_bounds__(256) sym_prepare_kernel(const double *H, long long ldh, const double *sig,
                                                          int n, double *M, long long ldm, double *partials)
{
    const int bi = blockIdx.y, bj = blockIdx.x;
    const int blin = blockIdx.y * gridDim.x + blockIdx.x;
    __shared__ double P[TT][TT + 1], Q[TT][TT + 1];
    __shared__ double red[2][256];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
    double dsum = 0.0, nsum = 0.0;
    if (bi >= bj) {
        for (int yy = ty; yy < TT; yy += 8) {
            int i = bi * TT + yy, j = bj * TT + tx;
            P[yy][tx] = (i < n && j < n) ? sig[i] * H[(long long)i * ldh + j] : 0.0;
            int i2 = bj * TT + yy, j2 = bi * TT + tx;
            Q[yy][tx] = (i2 < n && j2 < n) ? sig[i2] * H[(long long)i2 * ldh + j2] : 0.0;
        }
        __syncthreads();
        for (int yy = ty; yy < TT; yy += 8) {
            int i = bi * TT + yy, j = bj * TT + tx;
            double a = P[yy][tx], b = Q[tx][yy];     // (Sig H)[i][j] and (Sig H)[j][i]
            if (i < n && j < n) {
                double m = 0.5 * (a + b);
                M[(long long)i * ldm + j] = m;
                double d = a - b;
                double w = (bi == bj) ? 1.0 : 2.0;     // off-diagonal tile pairs count twice
                if (bi == bj) { dsum += d * d; nsum += a * a; }
                else { dsum += w * d * d; nsum += a * a + b * b; }
            }
            int i2 = bj * TT + yy, j2 = bi * TT + tx;
            if (bi != bj && i2 < n && j2 < n) M[(long long)i2 * ldm + j2] = 0.5 * (Q[yy][tx] + P[tx][yy]);
        }
    }
    red[0][threadIdx.x] = dsum; red[1][threadIdx.x] = nsum;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            red[0][threadIdx.x] += red[0][threadIdx.x + st];
            red[1][threadIdx.x] += red[1][threadIdx.x + st];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { partials[2 * blin] = red[0][0]; partials[2 * blin + 1] = red[1][0]; }
}

int sym_prepare_blocks(int n) { int t = (n + TT - 1) / TT; return t * t; }

void sym_prepare(const double *H, long long ldh, const double *sig, int n, double *M, long long ldm,
                 double *partials, cudaStream_t s)
{
    int t = (n + TT - 1) / TT;
    sym_prepare_kernel<<<dim3(t, t), 256, 0, s>>>(H, ldh, sig, n, M, ldm, partials); count_launch();
}

// Casida blocks (Eq. Casida): P = sym(A + B), R = sym(A - B) over 32x32 tile pairs;
// partials[2 b] = squared symmetry defects ||A - A^T||^2 + ||B - B^T||^2 of the tile pair,
// partials[2 b + 1] = its share of ||H||_F^2 = 2 (||A||_F^2 + ||B||_F^2).
__global__ void __launch_bounds__(256) casida_prepare_kernel(const double *A, long long lda, const double *B,
                                                             long long ldb, int k, double *P, double *R,
                                                             long long ldp, double *partials)
{
    const int bi = blockIdx.y, bj = blockIdx.x;
    const int blin = blockIdx.y * gridDim.x + blockIdx.x;
    __shared__ double Ta[TT][TT + 1], Tb[TT][TT + 1], Ua[TT][TT + 1], Ub[TT][TT + 1];
    __shared__ double red[2][256];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    double dsum = 0.0, nsum = 0.0;
    if (bi >= bj) {
        for (int yy = ty; yy < TT; yy += 8) {
            int i = bi * TT + yy, j = bj * TT + tx;
            bool in = i < k && j < k;
            Ta[yy][tx] = in ? A[(long long)i * lda + j] : 0.0;
            Tb[yy][tx] = in ? B[(long long)i * ldb + j] : 0.0;
            int i2 = bj * TT + yy, j2 = bi * TT + tx;
            bool in2 = i2 < k && j2 < k;
            Ua[yy][tx] = in2 ? A[(long long)i2 * lda + j2] : 0.0;
            Ub[yy][tx] = in2 ? B[(long long)i2 * ldb + j2] : 0.0;
        }
        __syncthreads();
        for (int yy = ty; yy < TT; yy += 8) {
            int i = bi * TT + yy, j = bj * TT + tx;
            double a = Ta[yy][tx], at = Ua[tx][yy], b = Tb[yy][tx], bt = Ub[tx][yy];   // (i,j) and (j,i)
            if (i < k && j < k) {
                double sa = 0.5 * (a + at), sb = 0.5 * (b + bt);
                P[(long long)i * ldp + j] = sa + sb;
                R[(long long)i * ldp + j] = sa - sb;
                double da = a - at, db = b - bt;
                if (bi == bj) { dsum += da * da + db * db; nsum += 2.0 * (a * a + b * b); }
                else { dsum += 2.0 * (da * da + db * db); nsum += 2.0 * (a * a + at * at + b * b + bt * bt); }
            }
            int i2 = bj * TT + yy, j2 = bi * TT + tx;
            if (bi != bj && i2 < k && j2 < k) {
                double sa = 0.5 * (Ua[yy][tx] + Ta[tx][yy]), sb = 0.5 * (Ub[yy][tx] + Tb[tx][yy]);
                P[(long long)i2 * ldp + j2] = sa + sb;
                R[(long long)i2 * ldp + j2] = sa - sb;
            }
        }
    }
    red[0][threadIdx.x] = dsum; red[1][threadIdx.x] = nsum;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            red[0][threadIdx.x] += red[0][threadIdx.x + st];
            red[1][threadIdx.x] += red[1][threadIdx.x + st];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { partials[2 * blin] = red[0][0]; partials[2 * blin + 1] = red[1][0]; }
}

void casida_prepare(const double *A, long long lda, const double *B, long long ldb, int k, double *P, double *R,
                    long long ldp, double *partials, cudaStream_t s)
{
    int t = (k + TT - 1) / TT;
    casida_prepare_kernel<<<dim3(t, t), 256, 0, s>>>(A, lda, B, ldb, k, P, R, ldp, partials); count_launch();
}

// The orthogonal change of basis T = [[I, I], [I, -I]] / sqrt 2 applied to a pair of k x m
// blocks: top = c (sx X + sy Y), bottom = c (sx X - sy Y), written to rows 0..k-1 and
// k..2k-1 of `out` (ld ldo).  Two doubles per thread, coalesced along rows.
__global__ void casida_combine_kernel(const double *X, long long ldx, const double *Y, long long ldy, int k, int m,
                                      double sx, double sy, double c, double *out, long long ldo)
{
    const long long total = (long long)k * m;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / m), j = (int)(e % m);
        const double x = sx * X[(long long)i * ldx + j], y = sy * Y[(long long)i * ldy + j];
        out[(long long)i * ldo + j] = c * (x + y);
        out[(long long)(i + k) * ldo + j] = c * (x - y);
    }
}

void casida_combine(const double *X, long long ldx, const double *Y, long long ldy, int k, int m, double sx,
                    double sy, double c, double *out, long long ldo, cudaStream_t s)
{
    const long long total = (long long)k * m;
    int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 16);
    if (blocks < 1) blocks = 1;
    casida_combine_kernel<<<blocks, 256, 0, s>>>(X, ldx, Y, ldy, k, m, sx, sy, c, out, ldo); count_launch();
}

// H = [[A, B], [-B, -A]] (Eq. Casida) assembled from its blocks
__global__ void casida_build_kernel(const double *A, long long lda, const double *B, long long ldb, int k, double *H,
                                    long long ldh)
{
    const long long total = (long long)k * k;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / k), j = (int)(e % k);
        const double a = A[(long long)i * lda + j], b = B[(long long)i * ldb + j];
        H[(long long)i * ldh + j] = a;
        H[(long long)i * ldh + j + k] = b;
        H[(long long)(i + k) * ldh + j] = -b;
        H[(long long)(i + k) * ldh + j + k] = -a;
    }
}

void casida_build(const double *A, long long lda, const double *B, long long ldb, int k, double *H, long long ldh,
                  cudaStream_t s)
{
    const long long total = (long long)k * k;
    int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 16);
    if (blocks < 1) blocks = 1;
    casida_build_kernel<<<blocks, 256, 0, s>>>(A, lda, B, ldb, k, H, ldh); count_launch();
}

// S <- (S + S^T) / 2 in place, over 32x32 tile pairs: the symmetric part of a product of
// two commuting symmetric matrices, whose computed value carries a first-order commutator
// error that averaging cancels (taking one triangle would keep it)
template <class T>
__global__ void __launch_bounds__(256) sym_average_kernel(T *S, long long lds, int n)
{
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bi < bj) return;
    __shared__ T P[TT][TT + 1], Q[TT][TT + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bi * TT + yy, j = bj * TT + tx;
        P[yy][tx] = (i < n && j < n) ? S[(long long)i * lds + j] : (T)0;
        int i2 = bj * TT + yy, j2 = bi * TT + tx;
        Q[yy][tx] = (i2 < n && j2 < n) ? S[(long long)i2 * lds + j2] : (T)0;
    }
    __syncthreads();
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bi * TT + yy, j = bj * TT + tx;
        if (i < n && j < n) S[(long long)i * lds + j] = (T)0.5 * (P[yy][tx] + Q[tx][yy]);
        int i2 = bj * TT + yy, j2 = bi * TT + tx;
        if (bi != bj && i2 < n && j2 < n) S[(long long)i2 * lds + j2] = (T)0.5 * (Q[yy][tx] + P[tx][yy]);
    }
}

template <class T>
void sym_average(T *S, long long lds, int n, cudaStream_t s)
{
    int t = (n + TT - 1) / TT;
    sym_average_kernel<T><<<dim3(t, t), 256, 0, s>>>(S, lds, n); count_launch();
}
template void sym_average<double>(double *, long long, int, cudaStream_t);
template void sym_average<float>(float *, long long, int, cudaStream_t);

// S <- (S + Sigma S^T Sigma) / 2: the nearest Sigma-symmetric matrix (Sigma S symmetric), in
// place, over 32x32 tile pairs
__global__ void __launch_bounds__(256) j_resym_kernel(double *S, long long lds, const double *sig, int n)
{
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bi < bj) return;
    __shared__ double P[TT][TT + 1], Q[TT][TT + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bi * TT + yy, j = bj * TT + tx;
        P[yy][tx] = (i < n && j < n) ? S[(long long)i * lds + j] : 0.0;
        int i2 = bj * TT + yy, j2 = bi * TT + tx;
        Q[yy][tx] = (i2 < n && j2 < n) ? S[(long long)i2 * lds + j2] : 0.0;
    }
    __syncthreads();
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bi * TT + yy, j = bj * TT + tx;
        if (i < n && j < n) S[(long long)i * lds + j] = 0.5 * (P[yy][tx] + sig[i] * sig[j] * Q[tx][yy]);
        int i2 = bj * TT + yy, j2 = bi * TT + tx;
        if (bi != bj && i2 < n && j2 < n)
            S[(long long)i2 * lds + j2] = 0.5 * (Q[yy][tx] + sig[i2] * sig[j2] * P[tx][yy]);
    }
}

void j_resym(double *S, long long lds, const double *sig, int n, cudaStream_t s)
{
    int t = (n + TT - 1) / TT;
    j_resym_kernel<<<dim3(t, t), 256, 0, s>>>(S, lds, sig, n); count_launch();
}

// Daleckii-Krein weights of the sign function:
//   X[i][j] = W[i][j] (s_i - s_j) / (lam_i - lam_j) + [i == j] lambar_i,  s = sign(lam)
// (divided differences of sign(x); zero between eigenvalues of the same sign)
__global__ void dk_combine_kernel(const double *W, long long ldw, const double *lam, const double *lambar, int n,
                                  double *X, long long ldx)
{
    const int i = blockIdx.y;
    const double li = lam[i];
    const double si = li > 0.0 ? 1.0 : -1.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double lj = lam[j];
        const double sj = lj > 0.0 ? 1.0 : -1.0;
        double v = (si != sj) ? W[(long long)i * ldw + j] * (si - sj) / (li - lj) : 0.0;
        if (i == j && lambar) v += lambar[i];
        X[(long long)i * ldx + j] = v;
    }
}

void dk_combine(const double *W, long long ldw, const double *lam, const double *lambar, int n, double *X,
                long long ldx, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    dk_combine_kernel<<<dim3(gx, n), 256, 0, s>>>(W, ldw, lam, lambar, n, X, ldx); count_launch();
}

// Correction of one refinement step of an approximate symmetric eigendecomposition
// A ~ Z diag(lam) Z^T (Ogita and Aishima's iteration): with S = Z^T A Z and
// Gm = Z^T Z - I (both full, symmetric), R = -Gm and
//   F_ii = R_ii / 2,
//   F_ij = (S_ij + lam_j R_ij) / (lam_j - lam_i)   if |lam_j - lam_i| > omega,
//   F_ij = R_ij / 2                                  otherwise (a cluster: keep orthogonality only).
__global__ void eig_refine_correction_kernel(const double *S, long long lds, const double *Gm, long long ldg,
                                             const double *lam, int n, double omega, double *F, long long ldf)
{
    const int i = blockIdx.y;
    const double li = lam[i];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double r = -Gm[(long long)i * ldg + j];
        const double d = lam[j] - li;
        double v = 0.5 * r;
        if (i != j && fabs(d) > omega) v = (S[(long long)i * lds + j] + lam[j] * r) / d;
        F[(long long)i * ldf + j] = v;
    }
}

void eig_refine_correction(const double *S, long long lds, const double *Gm, long long ldg, const double *lam, int n,
                           double omega, double *F, long long ldf, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    eig_refine_correction_kernel<<<dim3(gx, n), 256, 0, s>>>(S, lds, Gm, ldg, lam, n, omega, F, ldf);
    count_launch();
}

// Phi(X): the lower triangle with its diagonal halved, the strict upper triangle zeroed
// (the operator of the Cholesky factorisation's adjoint)
__global__ void tril_half_diag_kernel(double *X, long long ldx, int n)
{
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        double *x = X + (long long)i * ldx + j;
        if (j > i) *x = 0.0;
        else if (j == i) *x *= 0.5;
    }
}

void tril_half_diag(double *X, long long ldx, int n, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    tril_half_diag_kernel<<<dim3(gx, n), 256, 0, s>>>(X, ldx, n); count_launch();
}

// Real embedding of a complex n x n matrix Z (interleaved re/im doubles, row-major, ld in
// complex elements): R = [[Re Z, -Im Z], [Im Z, Re Z]] (2n x 2n, ld ldr).  Z -> R is an
// injective real algebra homomorphism with R(Z^H) = R(Z)^T.
__global__ void complex_embed_kernel(const double *Z, long long ldz, int n, double *R, long long ldr)
{
    const int i = blockIdx.y;
    const double2 *z = reinterpret_cast<const double2 *>(Z) + (long long)i * ldz;
    double *r0 = R + (long long)i * ldr, *r1 = R + (long long)(i + n) * ldr;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double2 v = z[j];
        r0[j] = v.x; r0[j + n] = -v.y;
        r1[j] = v.y; r1[j + n] = v.x;
    }
}

void complex_embed(const double *Z, long long ldz, int n, double *R, long long ldr, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    complex_embed_kernel<<<dim3(gx, n), 256, 0, s>>>(Z, ldz, n, R, ldr); count_launch();
}

// The inverse on the first block column: Z[i][j] = R[i][j] + i R[i + n][j] for j < m
// (columns j of R taken in the order perm[0..m) when perm is given)
__global__ void complex_extract_kernel(const double *R, long long ldr, int n, int m, const int *perm, double *Z,
                                       long long ldz)
{
    const int i = blockIdx.y;
    double2 *z = reinterpret_cast<double2 *>(Z) + (long long)i * ldz;
    const double *r0 = R + (long long)i * ldr, *r1 = R + (long long)(i + n) * ldr;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
        const int c = perm ? perm[j] : j;
        z[j] = make_double2(r0[c], r1[c]);
    }
}

void complex_extract(const double *R, long long ldr, int n, int m, const int *perm, double *Z, long long ldz,
                     cudaStream_t s)
{
    int gx = (m + 255) / 256; if (gx > 16) gx = 16;
    complex_extract_kernel<<<dim3(gx, n), 256, 0, s>>>(R, ldr, n, m, perm, Z, ldz); count_launch();
}

// Column phase convention for complex eigenvectors: each column of Z (m x n, interleaved)
// is multiplied by conj(z_max)/|z_max|, z_max its entry of largest modulus (first one on
// ties), so that entry becomes real and positive.  One block per column.
__global__ void complex_phase_fix_kernel(double *Z, long long ldz, int m, int n)
{
    __shared__ double bm[256];
    __shared__ int bi[256];
    const int c = blockIdx.x, t = threadIdx.x;
    double2 *z = reinterpret_cast<double2 *>(Z);
    double best = -1.0; int bidx = 0;
    for (int i = t; i < m; i += blockDim.x) {
        const double2 v = z[(long long)i * ldz + c];
        const double a = v.x * v.x + v.y * v.y;
        if (a > best) { best = a; bidx = i; }
    }
    bm[t] = best; bi[t] = bidx;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (t < o && (bm[t + o] > bm[t] || (bm[t + o] == bm[t] && bi[t + o] < bi[t]))) {
            bm[t] = bm[t + o]; bi[t] = bi[t + o];
        }
        __syncthreads();
    }
    const double2 p = z[(long long)bi[0] * ldz + c];
    const double a = sqrt(p.x * p.x + p.y * p.y);
    if (!(a > 0.0)) return;
    const double cr = p.x / a, ci = -p.y / a;     // conj(p) / |p|
    for (int i = t; i < m; i += blockDim.x) {
        double2 &v = z[(long long)i * ldz + c];
        const double x = v.x * cr - v.y * ci, y = v.x * ci + v.y * cr;
        v = make_double2(x, y);
    }
}

void complex_phase_fix(double *Z, long long ldz, int m, int n, cudaStream_t s)
{
    complex_phase_fix_kernel<<<n, 256, 0, s>>>(Z, ldz, m, n); count_launch();
}

// X[i][j] *= r[i] (row scaling)
__global__ void scale_rows_kernel(double *X, long long ldx, int m, int n, const double *r)
{
    const int i = blockIdx.y;
    const double f = r[i];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        X[(long long)i * ldx + j] *= f;
}

void scale_rows(double *X, long long ldx, int m, int n, const double *r, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    scale_rows_kernel<<<dim3(gx, m), 256, 0, s>>>(X, ldx, m, n, r); count_launch();
}

// (hi, lo) = (fl32(x), fl32(x - hi)) for a batch of rows x cols blocks (source
// leading dimension ld, batch stride sb), written compactly (ld = cols)
__global__ void split_pairs_kernel(const double *x, long long ld, long long sb, int rows, int cols, float *hi,
                                   float *lo)
{
    const int z = blockIdx.z, i = blockIdx.y;
    const double *xr = x + (long long)z * sb + (long long)i * ld;
    const long long o = ((long long)z * rows + i) * cols;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < cols; j += gridDim.x * blockDim.x) {
        double v = xr[j];
        float h = __double2float_rn(v);
        hi[o + j] = h;
        lo[o + j] = __double2float_rn(v - (double)h);
    }
}

void split_pairs(const double *x, long long ld, long long sb, int rows, int cols, int batch, float *hi, float *lo,
                 cudaStream_t s)
{
    int gx = (cols + 255) / 256; if (gx > 16) gx = 16;
    split_pairs_kernel<<<dim3(gx, rows, batch), 256, 0, s>>>(x, ld, sb, rows, cols, hi, lo); count_launch();
}

// fixed-order single-block sum (deterministic)
__global__ void reduce_sum_kernel(const double *x, int count, int stride, double *out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (int i = threadIdx.x; i < count; i += 1024) s += x[(long long)i * stride];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

void reduce_sum(const double *x, int count, double *out, cudaStream_t s)
{
    reduce_sum_kernel<<<1, 1024, 0, s>>>(x, count, 1, out); count_launch();
}

// copy the strictly lower triangle onto the upper one
template <class T>
__global__ void __launch_bounds__(256) mirror_lower_kernel(T *A, long long lda, long long sA, int n)
{
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bi < bj) return;
    A += (long long)blockIdx.z * sA;
    __shared__ T P[TT][TT + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bi * TT + yy, j = bj * TT + tx;
        P[yy][tx] = (i < n && j < n) ? A[(long long)i * lda + j] : (T)0;
    }
    __syncthreads();
    for (int yy = ty; yy < TT; yy += 8) {
        int i = bj * TT + yy, j = bi * TT + tx;   // target (i, j) in the upper tile
        if (i < n && j < n && j > i) A[(long long)i * lda + j] = P[tx][yy];
    }
}

template <class T>
void mirror_lower(T *A, long long lda, long long sA, int n, int batch, cudaStream_t s)
{
    int t = (n + TT - 1) / TT;
    mirror_lower_kernel<T><<<dim3(t, t, batch), 256, 0, s>>>(A, lda, sA, n); count_launch();
}
template void mirror_lower<double>(double *, long long, long long, int, int, cudaStream_t);
template void mirror_lower<float>(float *, long long, long long, int, int, cudaStream_t);

template <class T>
__global__ void shift_copy_lower_kernel(const T *G, long long ldg, T *Z, long long ldz, long long sZ, int n,
                                        const double *shifts)
{
    const int z = blockIdx.z;
    const int i = blockIdx.y;
    const T c = (T)shifts[z];
    T *Zr = Z + (long long)z * sZ + (long long)i * ldz;
    const T *Gr = G + (long long)i * ldg;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= i && j < n; j += gridDim.x * blockDim.x)
        Zr[j] = Gr[j] + (i == j ? c : (T)0);
}

template <class T>
void shift_copy_lower(const T *G, long long ldg, T *Z, long long ldz, long long sZ, int n, const double *shifts,
                      int batch, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 8) gx = 8;
    shift_copy_lower_kernel<T><<<dim3(gx, n, batch), 256, 0, s>>>(G, ldg, Z, ldz, sZ, n, shifts); count_launch();
}
template void shift_copy_lower<double>(const double *, long long, double *, long long, long long, int,
                                       const double *, int, cudaStream_t);
template void shift_copy_lower<float>(const float *, long long, float *, long long, long long, int,
                                      const double *, int, cudaStream_t);

template <class T>
__global__ void combine_lower_kernel(const T *Zinv, long long ldz, long long sZ, const double *a, int r, int n,
                                     T *Tm, long long ldt)
{
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= i && j < n; j += gridDim.x * blockDim.x) {
        T v = 0;
        for (int q = 0; q < r; ++q) v = fma((T)a[q], Zinv[(long long)q * sZ + (long long)i * ldz + j], v);
        Tm[(long long)i * ldt + j] = v;
    }
}

template <class T>
void combine_lower(const T *Zinv, long long ldz, long long sZ, const double *a, int r, int n, T *Tm, long long ldt,
                   cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 8) gx = 8;
    combine_lower_kernel<T><<<dim3(gx, n), 256, 0, s>>>(Zinv, ldz, sZ, a, r, n, Tm, ldt); count_launch();
}
template void combine_lower<double>(const double *, long long, long long, const double *, int, int, double *,
                                    long long, cudaStream_t);
template void combine_lower<float>(const float *, long long, long long, const double *, int, int, float *,
                                   long long, cudaStream_t);

template <class TI, class TO>
__global__ void scale_copy_kernel(const TI *X, long long ldx, TO *Y, long long ldy, int m, int n, double alpha)
{
    const int i = blockIdx.y;
    if (i >= m) return;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        Y[(long long)i * ldy + j] = (TO)(alpha * (double)X[(long long)i * ldx + j]);
}

template <class TI, class TO>
void scale_copy(const TI *X, long long ldx, TO *Y, long long ldy, int m, int n, double alpha, cudaStream_t s)
{
    if (m <= 0 || n <= 0) return;
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    scale_copy_kernel<TI, TO><<<dim3(gx, m), 256, 0, s>>>(X, ldx, Y, ldy, m, n, alpha); count_launch();
}
template void scale_copy<double, double>(const double *, long long, double *, long long, int, int, double, cudaStream_t);
template void scale_copy<double, float>(const double *, long long, float *, long long, int, int, double, cudaStream_t);
template void scale_copy<float, double>(const float *, long long, double *, long long, int, int, double, cudaStream_t);
template void scale_copy<float, float>(const float *, long long, float *, long long, int, int, double, cudaStream_t);

void copy_matrix(const double *X, long long ldx, double *Y, long long ldy, int m, int n, cudaStream_t s)
{
    scale_copy<double, double>(X, ldx, Y, ldy, m, n, 1.0, s);
}

// Y[z] = X[z] for z < batch (m x n blocks, strides sX, sY): one launch for the batch
template <class T>
__global__ void copy_batched_kernel(const T *X, long long ldx, long long sX, T *Y, long long ldy, long long sY, int m,
                                    int n)
{
    const int i = blockIdx.y;
    const T *x = X + (long long)blockIdx.z * sX + (long long)i * ldx;
    T *y = Y + (long long)blockIdx.z * sY + (long long)i * ldy;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) y[j] = x[j];
}

template <class T>
void copy_batched(const T *X, long long ldx, long long sX, T *Y, long long ldy, long long sY, int m, int n, int batch,
                  cudaStream_t s)
{
    if (m <= 0 || n <= 0 || batch <= 0) return;
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    copy_batched_kernel<T><<<dim3(gx, m, batch), 256, 0, s>>>(X, ldx, sX, Y, ldy, sY, m, n); count_launch();
}
template void copy_batched<double>(const double *, long long, long long, double *, long long, long long, int, int, int,
                                   cudaStream_t);
template void copy_batched<float>(const float *, long long, long long, float *, long long, long long, int, int, int,
                                  cudaStream_t);

// Z[i][j] <- (B[i][j] + Z[i][j]) / 2 for j < p, (B[i][j] - Z[i][j]) / 2 for j >= p (m x n):
// with Z = Y B on entry, the columns (I + Y)/2 B_+ and (I - Y)/2 B_- of the two projectors
__global__ void half_sum_diff_kernel(const double *B, long long ldb, double *Z, long long ldz, int m, int n, int p)
{
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double b = B[(long long)i * ldb + j], z = Z[(long long)i * ldz + j];
        Z[(long long)i * ldz + j] = 0.5 * (j < p ? b + z : b - z);
    }
}

void half_sum_diff(const double *B, long long ldb, double *Z, long long ldz, int m, int n, int p, cudaStream_t s)
{
    if (m <= 0 || n <= 0) return;
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    half_sum_diff_kernel<<<dim3(gx, m), 256, 0, s>>>(B, ldb, Z, ldz, m, n, p); count_launch();
}

// Y = a diag(sig)^rx X + b diag(sig) T diag(sig) (n x n; T may be null): the signature
// scalings of the general sign iteration, one pass (Y may alias X or T: entry by entry)
__global__ void sig_affine_kernel(const double *X, long long ldx, int rx, const double *T, long long ldt,
                                  const double *sig, int n, double a, double b, double *Y, long long ldy)
{
    const int i = blockIdx.y;
    const double si = sig[i], ai = rx ? a * si : a;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        double v = ai * X[(long long)i * ldx + j];
        if (T) v += b * si * sig[j] * T[(long long)i * ldt + j];
        Y[(long long)i * ldy + j] = v;
    }
}

void sig_affine(const double *X, long long ldx, int rx, const double *T, long long ldt, const double *sig, int n,
                double a, double b, double *Y, long long ldy, cudaStream_t s)
{
    if (n <= 0) return;
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    sig_affine_kernel<<<dim3(gx, n), 256, 0, s>>>(X, ldx, rx, T, ldt, sig, n, a, b, Y, ldy); count_launch();
}

template <class T>
__global__ void add_diag_kernel(T *X, long long ldx, int n, double v)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        X[(long long)i * ldx + i] += (T)v;
}

template <class T>
void add_diag(T *X, long long ldx, int n, double v, cudaStream_t s)
{
    add_diag_kernel<T><<<(n + 255) / 256, 256, 0, s>>>(X, ldx, n, v); count_launch();
}
template void add_diag<double>(double *, long long, int, double, cudaStream_t);
template void add_diag<float>(float *, long long, int, double, cudaStream_t);

// per-block partials of ||X - Y||_F^2 and ||Y||_F^2 (grid-stride over rows)
constexpr int FROB_BLOCKS = 608;  // 4 x 152 SMs

template <class T>
__global__ void __launch_bounds__(256) frob_diff_kernel(const T *X, long long ldx, const T *Y, long long ldy, int m,
                                                        int n, double *partials)
{
    __shared__ double red[2][256];
    double d2 = 0.0, y2 = 0.0;
    for (int i = blockIdx.x; i < m; i += gridDim.x) {
        for (int j = threadIdx.x; j < n; j += 256) {
            double y = (double)Y[(long long)i * ldy + j];
            double d = (X ? (double)X[(long long)i * ldx + j] : 0.0) - y;
            d2 += d * d; y2 += y * y;
        }
    }
    red[0][threadIdx.x] = d2; red[1][threadIdx.x] = y2;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            red[0][threadIdx.x] += red[0][threadIdx.x + st];
            red[1][threadIdx.x] += red[1][threadIdx.x + st];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { partials[2 * blockIdx.x] = red[0][0]; partials[2 * blockIdx.x + 1] = red[1][0]; }
}

int frob_blocks(int m, int n) { (void)n; return m < FROB_BLOCKS ? (m > 0 ? m : 1) : FROB_BLOCKS; }

template <class T>
void frob_diff(const T *X, long long ldx, const T *Y, long long ldy, int m, int n, double *partials, cudaStream_t s)
{
    frob_diff_kernel<T><<<frob_blocks(m, n), 256, 0, s>>>(X, ldx, Y, ldy, m, n, partials); count_launch();
}
template void frob_diff<double>(const double *, long long, const double *, long long, int, int, double *, cudaStream_t);
template void frob_diff<float>(const float *, long long, const float *, long long, int, int, double *, cudaStream_t);

// counter-based normal variates: splitmix64 hash of (seed, index) -> two
// uniforms -> Box-Muller
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// entry `idx` of the seeded Gaussian stream (Box-Muller on two splitmix64 draws)
__device__ __forceinline__ double gauss_at(uint64_t seed, uint64_t idx)
{
    uint64_t h1 = splitmix64(seed ^ (idx * 2 + 1)), h2 = splitmix64(seed + idx * 2 + 0x1234567ull);
    double u1 = ((h1 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);
    return sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
}

__global__ void fill_gaussian_kernel(double *X, long long ldx, int m, int n, uint64_t seed)
{
    for (int i = blockIdx.y; i < m; i += gridDim.y)
        for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
            X[(long long)i * ldx + j] = gauss_at(seed, (uint64_t)i * (uint64_t)n + (uint64_t)j);
}

void fill_gaussian(double *X, long long ldx, int m, int n, uint64_t seed, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    const int gy = m < 65535 ? m : 65535;
    if (gy <= 0) return;
    fill_gaussian_kernel<<<dim3(gx, gy), 256, 0, s>>>(X, ldx, m, n, seed); count_launch();
}

__global__ void trace_kernel(const double *X, long long ldx, int n, double *out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) s += X[(long long)i * ldx + i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

void trace_partial(const double *X, long long ldx, int n, double *out, cudaStream_t s)
{
    trace_kernel<<<1, 1024, 0, s>>>(X, ldx, n, out); count_launch();
}

__global__ void get_diag_kernel(const double *X, long long ldx, int n, double *d)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        d[i] = X[(long long)i * ldx + i];
}

void get_diag(const double *X, long long ldx, int n, double *d, cudaStream_t s)
{
    get_diag_kernel<<<(n + 255) / 256, 256, 0, s>>>(X, ldx, n, d); count_launch();
}

// max over rows of sum_j |X[i][j]| (the infinity norm, an upper bound on
// ||X||_2 for symmetric X): one warp per row, then a fixed-order max.
__global__ void row_abs_sums_kernel(const double *X, long long ldx, int n, double *sums)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= n) return;
    double s = 0.0;
    for (int j = lane; j < n; j += 32) s += fabs(X[(long long)warp * ldx + j]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) sums[warp] = s;
}

__global__ void reduce_max_kernel(const double *x, int n, double *out)
{
    __shared__ double red[1024];
    double b = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) b = fmax(b, x[i]);
    red[threadIdx.x] = b;
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + st]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

void row_abs_sum_max(const double *X, long long ldx, int n, double *tmp, double *out, cudaStream_t s)
{
    row_abs_sums_kernel<<<(n * 32 + 255) / 256, 256, 0, s>>>(X, ldx, n, tmp); count_launch();
    reduce_max_kernel<<<1, 1024, 0, s>>>(tmp, n, out); count_launch();
}

// y = op(A) x for square n, op(A) optionally triangular (masked)
__global__ void gemv_n_kernel(const double *A, long long lda, int tri, int n, const double *x, double *y)
{
    // one warp per row
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= n) return;
    const int i = warp;
    int jb = 0, je = n;
    if (tri == TRI_LOWER) je = i + 1;
    if (tri == TRI_UPPER) jb = i;
    double s = 0.0;
    for (int j = jb + lane; j < je; j += 32) s = fma(A[(long long)i * lda + j], x[j], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) y[i] = s;
}

// y[i] = sum_p A[p][i] x[p] (op(A) = A^T, `tri` describes op(A)); rows are
// split into GEMV_CHUNKS slices whose partial sums are added in a fixed order.
constexpr int GEMV_CHUNKS = 32;

__global__ void gemv_t_partial_kernel(const double *A, long long lda, int tri, int n, const double *x,
                                      double *part)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int ch = blockIdx.y;
    if (i >= n) return;
    const int len = (n + GEMV_CHUNKS - 1) / GEMV_CHUNKS;
    int pb = ch * len, pe = min(n, pb + len);
    if (tri == TRI_LOWER) pe = min(pe, i + 1);   // op(A)[i][p] = A[p][i] nonzero for p <= i
    if (tri == TRI_UPPER) pb = max(pb, i);
    double s = 0.0;
    for (int p = pb; p < pe; ++p) s = fma(A[(long long)p * lda + i], x[p], s);
    part[(long long)ch * n + i] = s;
}

__global__ void gemv_t_reduce_kernel(const double *part, int n, double *y)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int c = 0; c < GEMV_CHUNKS; ++c) s += part[(long long)c * n + i];
    y[i] = s;
}

void gemv(const double *A, long long lda, int ta, int tri, int n, const double *x, double *y, double *tmp,
          cudaStream_t s)
{
    if (ta == 0) {
        gemv_n_kernel<<<(n * 32 + 255) / 256, 256, 0, s>>>(A, lda, tri, n, x, y); count_launch();
    } else {
        gemv_t_partial_kernel<<<dim3((n + 127) / 128, GEMV_CHUNKS), 128, 0, s>>>(A, lda, tri, n, x, tmp); count_launch();
        gemv_t_reduce_kernel<<<(n + 255) / 256, 256, 0, s>>>(tmp, n, y); count_launch();
    }
}

__global__ void normalize_kernel(double *y, double *x, int n, double *norm_out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) s += y[i] * y[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    double nrm = sqrt(red[0]);
    double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) x[i] = y[i] * inv;
    if (threadIdx.x == 0 && norm_out) norm_out[0] = nrm;
}

void normalize_vec(double *y, double *x, int n, double *norm_out, cudaStream_t s)
{
    normalize_kernel<<<1, 1024, 0, s>>>(y, x, n, norm_out); count_launch();
}

// Lanczos three-term update w <- w - alpha v - beta vprev with alpha, beta read
// from device memory (beta may be null): no host round trip per step
__global__ void lanczos_update_kernel(double *w, const double *v, const double *vprev, const double *alpha,
                                      const double *beta, int n)
{
    const double a = alpha[0], b = beta ? beta[0] : 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        w[i] = w[i] - a * v[i] - (vprev ? b * vprev[i] : 0.0);
}

void lanczos_update(double *w, const double *v, const double *vprev, const double *alpha, const double *beta, int n,
                    cudaStream_t s)
{
    int blocks = (n + 255) / 256; if (blocks > 64) blocks = 64;
    lanczos_update_kernel<<<blocks, 256, 0, s>>>(w, v, vprev, alpha, beta, n); count_launch();
}

__global__ void dot_kernel(const double *x, const double *y, int n, double *out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) s += x[i] * y[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 512; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

void dot_vec(const double *x, const double *y, int n, double *out, cudaStream_t s)
{
    dot_kernel<<<1, 1024, 0, s>>>(x, y, n, out); count_launch();
}

// ---------------------------------------------------------------------------
// Krylov loops in one launch.  Step by step, a Lanczos step takes four launches
// (product, alpha, three-term update, beta with the new vector) and a power
// step three or four; the recursion's nodes, the bounds of small inputs and
// the shift screening run such loops hundreds of times on operators of order
// at most KRY_MAX_M.  What bounds a loop is the FP64 pipe (m^2 multiply-adds a
// step, 2 per clock and SM) and then the exchanges, so the rows are spread over
// m / 8 CTAs of 8 warps, one row (and, for L^T, one column) to a warp, held in
// its registers for the whole loop.  A product's entries go through global
// memory to every CTA (two buffers in turn) behind one grid barrier; the dot
// products, the three-term update and the normalisation are then done by every
// CTA for itself, in the same order, so all hold the same bits.  The launch is
// cooperative -- all CTAs are resident before any waits.  A CTA whose wait runs
// out of polls leaves without another arrival, so that nobody passes a later
// barrier: CTA 0, which writes the results, either passed every barrier or gives up
// as well, writes NaN and sets the error flag.
// Sums: 32 consecutive entries by a shuffle tree, the trees' results in order,
// over KRY_SEGMENTS equal segments of the vector first, then those in order.
// Measured, 24 Lanczos steps: m = 128 190 us, m = 1000 400 us; on one cluster of 8
// CTAs, which these loops ran on before, 440 and 1940 us.
// ---------------------------------------------------------------------------
constexpr int KRY_ROWS = 8, KRY_THREADS = 32 * KRY_ROWS, KRY_SEGMENTS = 8;
constexpr int KRY_T = KRY_MAX_M / 32;                  // entries of a row per lane
constexpr int KRY_GROUPS = KRY_SEGMENTS * (KRY_MAX_M / KRY_SEGMENTS / 32);   // sums of 32 entries, at most
constexpr unsigned int KRY_WAIT_LIMIT = 1u << 22;      // default bound of a wait, in polls

// every CTA of the grid has arrived (count: 0 at launch; target: arrivals so far times CTAs)
__device__ __forceinline__ bool kry_grid_sync(unsigned int *count, unsigned int target, unsigned int limit, int *sm_ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int v;
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        int ok = 0;
        for (unsigned int it = 0; it < limit; ++it) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            if (v >= target) { ok = 1; break; }
        }
        *sm_ok = ok;
    }
    __syncthreads();
    return *sm_ok != 0;
}

// sum of f(i), i < m, returned to every thread: groups of 32 from the start of each segment of
// `seg` entries, the groups of a segment in order, the segments in order.  root: the square root
// of the sum instead, and its reciprocal (0 for 0) in bc[1], by one warp (each takes some ten
// dependent FP64 instructions, which eight warps would issue one after the other)
template <class F>
__device__ __forceinline__ double kry_sum(int m, int seg, F f, double *red, double *bc, bool root = false)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = (seg + 31) / 32, ns = (m + seg - 1) / seg;
    for (int g = warp; g < ns * per; g += KRY_ROWS) {
        const int s0 = (g / per) * seg, i = s0 + (g % per) * 32 + lane;
        double x = (i < m && i < s0 + seg) ? f(i) : 0.0;
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[g] = x;
    }
    __syncthreads();
    if (warp == 0) {
        double p = 0.0;                                // lane c: segment c
        if (lane < ns)
            for (int j = 0; j < per; ++j) p += red[lane * per + j];
        double s = 0.0;
        for (int c = 0; c < ns; ++c) s += __shfl_sync(0xffffffffu, p, c);
        if (root) {
            s = sqrt(s);
            const double inv = s > 0.0 ? 1.0 / s : 0.0;
            if (lane == 0) bc[1] = inv;
        }
        if (lane == 0) bc[0] = s;
    }
    __syncthreads();
    return bc[0];
}

// row . x for a row of `len` entries held by a warp (lane l: entries l, l + 32, ...; zero
// beyond): eight running sums over blocks of 256, a block of 128 into four of them where one is
// left, the rest into the first, added pairwise and over the lanes by a shuffle tree
__device__ __forceinline__ double kry_row_dot(const double *row, int len, const double *x, int lane)
{
    double a[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int nb = max(0, (len - 224 - lane + 255) / 256);         // whole blocks of this lane (len - 224 - lane > 256 b)
    const bool four = lane + 256 * nb + 96 < len;
    const int nb_all = max(0, (len - 224 - 31 + 255) / 256);       // of every lane
#pragma unroll
    for (int t = 0; t < KRY_T; ++t) {
        if (32 * t >= len) break;
        const int b = t >> 3, q = t & 7, i = lane + 32 * t;
        const double v = row[t];
        if (b < nb_all || q == 0) {
            if (i < len) a[q] = fma(v, x[i], a[q]);
        } else {
            const bool own = b < nb || (b == nb && four && q < 4);
            if (i < len) {
                if (own) a[q] = fma(v, x[i], a[q]);
                else a[0] = fma(v, x[i], a[0]);
            }
        }
    }
    double s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

template <int OP>
__global__ void __launch_bounds__(KRY_THREADS, 1)
krylov_grid_kernel(const double *__restrict__ A, long long lda, int m, int steps, int power, uint64_t seed, double *out,
                   double *ex, unsigned int *count, int *err, unsigned int limit)
{
    __shared__ double cur[KRY_MAX_M], prv[KRY_MAX_M], w[KRY_MAX_M];
    __shared__ double red[KRY_GROUPS + 8], bc[2];
    __shared__ int sm_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r = blockIdx.x * KRY_ROWS + warp;
    const int seg = (m + KRY_SEGMENTS - 1) / KRY_SEGMENTS;
    unsigned int arrived = 0;
    int turn = 0;
    // entry r of a vector (lane 0's v) -> dst, whole in every CTA; false if a wait ran out
    auto exchange = [&](double v, double *dst) -> bool {
        double *buf = ex + turn * m;
        turn ^= 1;
        if (r < m && lane == 0) __stcg(buf + r, v);
        arrived += gridDim.x;
        if (!kry_grid_sync(count, arrived, limit, &sm_ok)) return false;
        for (int i = tid; i < m; i += KRY_THREADS) dst[i] = __ldcg(buf + i);
        __syncthreads();
        return true;
    };
    auto give_up = [&]() {
        if (blockIdx.x != 0 || tid != 0) return;
        for (int j = 0; j < (power > 0 ? 1 : steps); ++j) {
            out[j] = NAN;
            if (power == 0) out[steps + 1 + j] = NAN;
        }
        if (err) atomicExch(err, 6);
    };
    // this warp's row of A (of L), and column of L
    const int rlen = r < m ? (OP == KRY_SYM ? m : r + 1) : 0;
    double row[KRY_T], col[OP == KRY_TRI_PAIR ? KRY_T : 1];
#pragma unroll
    for (int t = 0; t < KRY_T; ++t) {
        const int i = lane + 32 * t;
        row[t] = i < rlen ? __ldg(A + (long long)r * lda + i) : 0.0;
        if (OP == KRY_TRI_PAIR) col[t] = (r < m && i >= r && i < m) ? __ldg(A + (long long)i * lda + r) : 0.0;
    }
    if (!exchange(r < m && lane == 0 ? gauss_at(seed, (uint64_t)r) : 0.0, cur)) return give_up();
    kry_sum(m, KRY_MAX_M, [&](int i) { return cur[i] * cur[i]; }, red, bc, true);
    const double inv0 = bc[1];
    for (int i = tid; i < m; i += KRY_THREADS) { cur[i] *= inv0; prv[i] = 0.0; }
    __syncthreads();
    auto apply = [&]() -> bool {                       // op(A) cur -> w
        if (!exchange(kry_row_dot(row, rlen, cur, lane), w)) return false;
        // w = u = L x: L^T u (zeros above the diagonal)
        return OP == KRY_SYM || exchange(kry_row_dot(col, r < m ? m : 0, w, lane), w);
    };
    if (power == 0) {
        double beta_prev = 0.0;
        for (int j = 0; j < steps; ++j) {
            if (!apply()) return give_up();
            const double alpha = kry_sum(m, seg, [&](int i) { return cur[i] * w[i]; }, red, bc);
            for (int i = tid; i < m; i += KRY_THREADS) w[i] = w[i] - alpha * cur[i] - beta_prev * prv[i];
            __syncthreads();
            const double beta = kry_sum(m, seg, [&](int i) { return w[i] * w[i]; }, red, bc, true);
            if (blockIdx.x == 0 && tid == 0) { out[j] = alpha; out[steps + 1 + j] = beta; }
            const double scale = bc[1];
            for (int i = tid; i < m; i += KRY_THREADS) { prv[i] = cur[i]; cur[i] = w[i] * scale; }
            __syncthreads();
            beta_prev = beta;
        }
    } else {
        for (int it = 0; it < power; ++it) {
            if (!apply()) return give_up();
            kry_sum(m, seg, [&](int i) { return w[i] * w[i]; }, red, bc, true);
            const double scale = bc[1];
            for (int i = tid; i < m; i += KRY_THREADS) cur[i] = w[i] * scale;
            __syncthreads();
        }
        if (!apply()) return give_up();
        const double rq = kry_sum(m, seg, [&](int i) { return cur[i] * w[i]; }, red, bc);
        if (blockIdx.x == 0 && tid == 0) out[0] = rq;
    }
}

size_t krylov_scratch_doubles(int m) { return 2 * (size_t)m + 8; }

bool krylov_fused(const double *A, long long lda, int op, int m, int steps, int power, uint64_t seed, double *out,
                  double *scratch, int *err, unsigned int wait_limit, cudaStream_t s)
{
    if (m < 1 || m > KRY_MAX_M || steps < 0 || power < 0) return false;
    unsigned int *count = (unsigned int *)(scratch + 2 * (size_t)m);
    if (cudaMemsetAsync(count, 0, sizeof(unsigned int), s) != cudaSuccess) return false;
    unsigned int limit = wait_limit ? wait_limit : KRY_WAIT_LIMIT;
    void *args[] = {&A, &lda, &m, &steps, &power, &seed, &out, &scratch, &count, &err, &limit};
    const void *kernel = op == KRY_SYM ? (const void *)krylov_grid_kernel<KRY_SYM>
                                       : (const void *)krylov_grid_kernel<KRY_TRI_PAIR>;
    if (cudaLaunchCooperativeKernel(kernel, dim3((m + KRY_ROWS - 1) / KRY_ROWS), dim3(KRY_THREADS), args, 0, s) !=
        cudaSuccess)
        return false;
    count_launch();
    return true;
}

__global__ void scale_columns_kernel(double *X, long long ldx, int m, int n, const double *d, int use_sqrt_abs)
{
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        double f = use_sqrt_abs ? sqrt(fabs(d[j])) : d[j];
        X[(long long)i * ldx + j] *= f;
    }
}

void scale_columns(double *X, long long ldx, int m, int n, const double *d, int use_sqrt_abs, cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    scale_columns_kernel<<<dim3(gx, m), 256, 0, s>>>(X, ldx, m, n, d, use_sqrt_abs); count_launch();
}

// make the largest-magnitude entry of each column positive (ties: lowest row)
__global__ void sign_fix_columns_kernel(double *X, long long ldx, int m, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double best = -1.0, val = 0.0;
    for (int i = 0; i < m; ++i) {
        double v = X[(long long)i * ldx + j];
        if (fabs(v) > best) { best = fabs(v); val = v; }
    }
    if (val < 0.0)
        for (int i = 0; i < m; ++i) X[(long long)i * ldx + j] = -X[(long long)i * ldx + j];
}

void sign_fix_columns(double *X, long long ldx, int m, int n, cudaStream_t s)
{
    sign_fix_columns_kernel<<<(n + 127) / 128, 128, 0, s>>>(X, ldx, m, n); count_launch();
}

__global__ void gather_columns_kernel(const double *X, long long ldx, double *Y, long long ldy, int m, int n,
                                      const int *perm)
{
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        Y[(long long)i * ldy + j] = X[(long long)i * ldx + perm[j]];
}

void gather_columns(const double *X, long long ldx, double *Y, long long ldy, int m, int n, const int *perm,
                    cudaStream_t s)
{
    int gx = (n + 255) / 256; if (gx > 16) gx = 16;
    gather_columns_kernel<<<dim3(gx, m), 256, 0, s>>>(X, ldx, Y, ldy, m, n, perm); count_launch();
}

// --------------------------------------------------------------------------
// Jacobi eigensolver for one symmetric matrix of order m <= 64 (one CTA).
// Parallel cyclic order: in each of the m'-1 rounds (m' = m rounded up to even)
// the pairs of a round-robin tournament are disjoint, so all their rotations
// are applied together.
//
// What bounds it: a round's rotations of A and V are about 33 000 FP64
// operations, 8000 clocks of one SM's FP64 pipe, and eight or nine sweeps of 63
// rounds would be needed.  So the sweeps are made in FP32 (64 times the rate)
// until they end at rounding, A ~ V32 diag V32^T; V32 is made orthogonal to FP64
// accuracy -- with E = I - V32^T V32 (~1e-6), V = V32 (I + E/2 + 3 E^2/8 +
// 5 E^3/16) leaves O(E^4) -- and A <- V^T A V, formed in FP64, is so nearly diagonal that two FP64
// sweeps finish it (more where eigenvalues coincide).  Fewer FP64 rotations are also fewer roundings:
// orthogonality and residual are 3 to 8 times smaller than after FP64 sweeps alone.  A rotation need not annihilate exactly, only be orthogonal:
// its tangent is taken in FP32, its cosine from that in FP64.  A keeps both
// triangles; a round updates the 2 x 2 blocks of pairs k >= l and mirrors them.
// Measured (m = 64): 0.9 ms, 1.6 ms with every eigenvalue double; 2.2 and 3.1 ms with every sweep in FP64.
// --------------------------------------------------------------------------
constexpr int JAC_LD = 65, JAC_THREADS = 256, JAC_WARPS = JAC_THREADS / 32;
constexpr int JAC_SMEM = 5 * 64 * JAC_LD * (int)sizeof(double);

__device__ __forceinline__ void jac_rotation(float app, float aqq, float apq, float &c, float &s)
{
    const float tau = (aqq - app) / (2.0f * apq);
    const float t = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
    c = 1.0f / sqrtf(1.0f + t * t);
    s = t * c;
}

__device__ __forceinline__ void jac_rotation(double app, double aqq, double apq, double &c, double &s)
{
    const float tau = (float)(aqq - app) / (2.0f * (float)apq);
    const double t = (double)(copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau)));
    const double x = fma(t, t, 1.0);              // 1 .. 2
    double y = (double)rsqrtf((float)x);
    y = y * (1.5 - 0.5 * x * y * y);
    y = y * (1.5 - 0.5 * x * y * y);
    c = y;
    s = t * y;
}

// squared norms of the off-diagonal part and of the diagonal of A, to every thread
template <class T>
__device__ __forceinline__ void jac_norms(const T *A, int m, double *red, double &off, double &dia)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    T o = 0, d = 0;
    for (int e = tid; e < m * m; e += JAC_THREADS) {
        const int i = e / m, j = e - i * m;
        const T v = A[i * JAC_LD + j];
        if (i == j) d += v * v;
        else o += v * v;
    }
    for (int q = 16; q > 0; q >>= 1) {
        o += __shfl_xor_sync(0xffffffffu, o, q);
        d += __shfl_xor_sync(0xffffffffu, d, q);
    }
    if (lane == 0) { red[warp] = (double)o; red[JAC_WARPS + warp] = (double)d; }
    __syncthreads();
    off = dia = 0.0;
    for (int w = 0; w < JAC_WARPS; ++w) { off += red[w]; dia += red[JAC_WARPS + w]; }
    __syncthreads();
}

// sweeps until off^2 <= tol dia^2, at most `most`; returns the number made
template <class T>
__device__ int jac_sweeps(T *A, T *V, int m, double tol, int most, T *cs, T *sn, int *pp, int *qq, double *red)
{
    const int tid = threadIdx.x, me = (m + 1) & ~1, np = me / 2, nb = np * (np + 1) / 2;
    int sweep = 0;
    for (; sweep < most; ++sweep) {
        double off, dia;
        jac_norms<T>(A, m, red, off, dia);
        if (!(off > tol * dia)) break;
        for (int round = 0; round < me - 1; ++round) {
            if (tid < np) {     // round-robin: me - 1 stays, the others turn (me > m: a zero row and column)
                int p = tid == 0 ? round : round + tid, q = tid == 0 ? me - 1 : round - tid;
                if (p >= me - 1) p -= me - 1;
                if (q < 0) q += me - 1;
                if (p > q) { const int t = p; p = q; q = t; }
                pp[tid] = p;
                qq[tid] = q;
                const T apq = A[p * JAC_LD + q];
                T c = 1, s = 0;
                if (apq != (T)0) jac_rotation(A[p * JAC_LD + p], A[q * JAC_LD + q], apq, c, s);
                if (!(c <= (T)1.0001)) { c = 1; s = 0; }            // (not finite)
                cs[tid] = c;
                sn[tid] = s;
            }
            __syncthreads();
            for (int e = tid; e < nb; e += JAC_THREADS) {   // A <- J^T A J, block of pairs k >= l
                int k = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                while (k * (k + 1) / 2 > e) --k;
                while ((k + 1) * (k + 2) / 2 <= e) ++k;
                const int l = e - k * (k + 1) / 2;
                const int p = pp[k], q = qq[k], u = pp[l], v = qq[l];
                const T ck = cs[k], sk = sn[k], cl = cs[l], sl = sn[l];
                const T apu = A[p * JAC_LD + u], apv = A[p * JAC_LD + v], aqu = A[q * JAC_LD + u], aqv = A[q * JAC_LD + v];
                const T bpu = ck * apu - sk * aqu, bqu = sk * apu + ck * aqu;
                const T bpv = ck * apv - sk * aqv, bqv = sk * apv + ck * aqv;
                const T npu = cl * bpu - sl * bpv, npv = sl * bpu + cl * bpv;
                const T nqu = cl * bqu - sl * bqv, nqv = sl * bqu + cl * bqv;
                if (k == l) {
                    A[p * JAC_LD + p] = npu;
                    A[q * JAC_LD + q] = nqv;
                    A[p * JAC_LD + q] = A[q * JAC_LD + p] = nqu;
                } else {
                    A[p * JAC_LD + u] = A[u * JAC_LD + p] = npu;
                    A[p * JAC_LD + v] = A[v * JAC_LD + p] = npv;
                    A[q * JAC_LD + u] = A[u * JAC_LD + q] = nqu;
                    A[q * JAC_LD + v] = A[v * JAC_LD + q] = nqv;
                }
            }
            for (int e = tid; e < np * 64; e += JAC_THREADS) {   // V <- V J
                const int k = e >> 6, row = e & 63;
                if (row >= m) continue;
                const int p = pp[k], q = qq[k];
                const T c = cs[k], s = sn[k];
                const T vp = V[row * JAC_LD + p], vq = V[row * JAC_LD + q];
                V[row * JAC_LD + p] = c * vp - s * vq;
                V[row * JAC_LD + q] = s * vp + c * vq;
            }
            __syncthreads();
        }
    }
    return sweep;
}

// C = op(X) Y for m x m blocks in shared memory (row stride JAC_LD), op = transpose if tx; sym:
// the result is symmetric, its lower part is formed and mirrored; then C <- a I + b C + c D
// entry by entry (D may be C's own input).  C differs from X and Y.
__device__ void jac_product(const double *X, int tx, const double *Y, double *C, int m, bool sym, double a, double b,
                            double c, const double *D)
{
    const int jx = threadIdx.x & 15, iy = threadIdx.x >> 4;
    double acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0;
    for (int p = 0; p < m; ++p) {
        double x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = iy + 16 * u;
            x[u] = tx ? X[p * JAC_LD + i] : X[i * JAC_LD + p];
            y[u] = Y[p * JAC_LD + jx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v)
                if (!sym || v <= u) acc[u][v] = fma(x[u], y[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int i = iy + 16 * u, j = jx + 16 * v;
            if (i >= m || j >= m || (sym && j > i)) continue;
            double r = b * acc[u][v] + (i == j ? a : 0.0);
            if (c != 0.0) r += c * D[i * JAC_LD + j];
            C[i * JAC_LD + j] = r;
            if (sym) C[j * JAC_LD + i] = r;
        }
    __syncthreads();
}

__global__ void __launch_bounds__(JAC_THREADS) jacobi_leaf_kernel(const double *Ag, long long lda, int m, double *W,
                                                                  long long ldw, double *w, int *sweeps_out)
{
    extern __shared__ __align__(16) unsigned char jac_smem[];
    double *A = (double *)jac_smem, *V = A + 64 * JAC_LD, *T1 = V + 64 * JAC_LD, *T2 = T1 + 64 * JAC_LD;
    double *T3 = T2 + 64 * JAC_LD;
    __shared__ double cs[32], sn[32], red[2 * JAC_WARPS];
    __shared__ int pp[32], qq[32];
    const int tid = threadIdx.x;
    // A and the FP32 matrices, scaled by a power of two to entries below 1
    double amax = 0.0;
    for (int e = tid; e < 64 * 64; e += JAC_THREADS) {
        const int i = e >> 6, j = e & 63;
        const double v = (i < m && j < m) ? 0.5 * (Ag[(long long)i * lda + j] + Ag[(long long)j * lda + i]) : 0.0;
        A[i * JAC_LD + j] = v;
        amax = fmax(amax, fabs(v));
    }
    for (int q = 16; q > 0; q >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, q));
    if ((tid & 31) == 0) red[tid >> 5] = amax;
    __syncthreads();
    for (int q = 0; q < JAC_WARPS; ++q) amax = fmax(amax, red[q]);
    __syncthreads();
    int ex = 0;
    if (amax > 0.0 && isfinite(amax)) frexp(amax, &ex);
    const double up = ldexp(1.0, max(-1000, min(1000, ex))), down = ldexp(1.0, -max(-1000, min(1000, ex)));
    float *A32 = (float *)T1, *V32 = (float *)T2;
    for (int e = tid; e < 64 * 64; e += JAC_THREADS) {
        const int i = e >> 6, j = e & 63;
        A[i * JAC_LD + j] *= down;
        A32[i * JAC_LD + j] = (float)A[i * JAC_LD + j];
        V32[i * JAC_LD + j] = i == j ? 1.0f : 0.0f;
    }
    __syncthreads();
    int sweeps = jac_sweeps<float>(A32, V32, m, 3e-12, 12, (float *)cs, (float *)sn, pp, qq, red);
    for (int e = tid; e < 64 * 64; e += JAC_THREADS) {
        const int i = e >> 6, j = e & 63;
        V[i * JAC_LD + j] = (double)V32[i * JAC_LD + j];
    }
    __syncthreads();
    jac_product(V, 1, V, T1, m, true, 1.0, -1.0, 0.0, nullptr);       // E = I - V^T V
    jac_product(T1, 0, T1, T2, m, true, 0.5, 0.3125, 0.375, T1);      // I/2 + 3 E/8 + 5 E^2/16
    jac_product(T1, 0, T2, T3, m, true, 1.0, 1.0, 0.0, nullptr);      // I + E times that
    jac_product(V, 0, T3, T1, m, false, 0.0, 1.0, 0.0, nullptr);      // V, orthogonal
    double *Vo = T1;
    jac_product(A, 0, Vo, T2, m, false, 0.0, 1.0, 0.0, nullptr);      // A V
    jac_product(Vo, 1, T2, A, m, true, 0.0, 1.0, 0.0, nullptr);       // V^T A V
    if (tid < 64 && (m & 1)) {                                        // the zero row and column of an odd order
        A[m * JAC_LD + tid] = A[tid * JAC_LD + m] = 0.0;
        Vo[tid * JAC_LD + m] = 0.0;
    }
    __syncthreads();
    sweeps += jac_sweeps<double>(A, Vo, m, 1e-30, 40, cs, sn, pp, qq, red);
    for (int e = tid; e < m * m; e += JAC_THREADS) {
        const int i = e / m, j = e % m;
        W[(long long)i * ldw + j] = Vo[i * JAC_LD + j];
    }
    if (tid < m) w[tid] = A[tid * JAC_LD + tid] * up;
    if (tid == 0 && sweeps_out) sweeps_out[0] = sweeps;
}

int jacobi_leaf(const double *A, long long lda, int m, double *W, long long ldw, double *w, int *sweeps_out,
                cudaStream_t s)
{
    if (!ensure_dynamic_smem((const void *)jacobi_leaf_kernel, JAC_SMEM)) return -1;
    jacobi_leaf_kernel<<<1, JAC_THREADS, JAC_SMEM, s>>>(A, lda, m, W, ldw, w, sweeps_out); count_launch();
    return 0;
}

}  // namespace pssd
