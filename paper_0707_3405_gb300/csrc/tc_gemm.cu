// Complex64 GEMMs on the 5th-generation tensor cores (tcgen05, accumulators in
// TMEM) with split TF32 operands: the projector, Gram, constraint and update
// contractions of Algorithm 1 (Sec. 3.2 and 4.1, zgemm in the paper) on the
// mixed-precision path.
//
// Precision ("3xTF32"): every FP32 operand x is split as x = hi + lo with hi
// and lo rounded to TF32 (10-bit mantissa); a product is hi*hi + hi*lo + lo*hi
// (the lo*lo term is below FP32 resolution), accumulated in FP32 by the tensor
// core.  The relative error per product is about 2^-21, i.e. FP32 class.
//
// Complex arithmetic as one real GEMM per tile, re / im interleaved along K.  The left factor's
// vectors (columns of A, or rows of A) are the 128 MMA rows [re, im, re, im, ...]; each of the NT
// columns of the right factor is two MMA columns, j (the real part) and NT + j (the imaginary one):
//   C = A^H B:  [re, im, ...] and [im, -re, ...] of B's column;
//   D = A B:    [re, -im, ...] and [im, re, ...] of B's column.
//
// One persistent CTA per SM takes every gridDim-th item (an output tile, and for A^H B a part of
// the reduction, which is split over the GPU).  Sixteen warps in four groups, one per ring slot, load FP32
// from HBM ahead into registers, split it and store hi / lo into 64-byte-swizzled K-major shared tiles of a
// 4-stage ring (8 complex K a stage); one warp issues a stage's six MMAs of M = 128, N = 2 NT and
// commits them to the stage's mbarrier; four warps read the accumulator of the finished item from
// TMEM, which holds two, and write it out while the next item runs.  FP32 partial tiles of a split
// reduction are summed afterwards in a fixed order (reproducible).
//
// What bounds it (NT = 128): a stage's MMAs take 768 cycles of the tensor pipe and, with the left
// rows kept in the collector, 64 KB of shared-memory reads beside the loaders' 48 KB of stores, 896
// cycles of shared-memory bandwidth.  Measured on a GB300 (tensor rate: 3 x 8 m n K flops), before
// (256 threads loading, splitting and storing in lockstep, one of them issuing) and after:
//   A B    113081 x 128 x 256    330 -> 134 us  (269 -> 664 TFLOP/s of about 960 for TF32)
//          113081 x 128 x 1024  1070 -> 420 us;  57925 x 64 x 128  50 -> 33 us
//   A^H B  432 x 128 x 113081    333 -> 289 us;  384 x 256 x 113081  468 -> 403 us
//          64 x 64 x 57925        65 -> 40 us
// All loaders filling one stage together (8 or 16 warps, 2 to 4 stages ahead in registers) took 179 to
// 197 us for the first: each stage then costs one group's whole chain of wait, stores, fence and
// signal, which the slot groups overlap.
//
// Every mbarrier wait is bounded.  A loader's first wait for its slot, whose limit tests lower, raises a device flag
// (read by tc_check_error) and is repeated with the full limit.  When that or another wait runs out, the flag is
// raised, the other waits end at their next poll, and every warp goes on without what it waited for, so that the
// CTA ends with its copies and MMAs done and its TMEM freed.
#include "common.cuh"
#include "df64.cuh"
#include "tc.cuh"

#include <algorithm>
#include <cfloat>

namespace lg {

namespace {

using namespace tc;

constexpr int kLoaders = 16, kReaders = 4;                   // warps
constexpr int kThreads = 32 * (kLoaders + 1 + kReaders);     // + the MMA warp
constexpr int KST = 8;       // complex K per stage: 16 floats = one 64-byte shared row
constexpr int ROWB = 64;     // bytes per shared row
constexpr int kRing = 4;
constexpr int kRows = 128;   // vectors of the left factor per tile (MMA M)

__device__ int g_tc_err = 0;
// Poll limit of the loaders' first wait for a stage (lowered only by tests of the timeout path).
__device__ long long g_tc_spin = kSpinLimit;

__device__ __forceinline__ unsigned char *align1k(unsigned char *p) {
    return reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

constexpr int stage_bytes(int NT) { return 2 * kRows * ROWB + 2 * 2 * NT * ROWB; }
constexpr size_t smem_bytes(int NT) { return (size_t)kRing * stage_bytes(NT) + 1024 + 256; }

// Byte offset of complex element k (0 .. 7) of row r in a 64-byte-swizzled tile.
__device__ __forceinline__ uint32_t elem_at(int r, int k) {
    return (uint32_t)r * (uint32_t)ROWB + ((uint32_t)((k >> 1) ^ ((r >> 1) & 3)) << 4) + (uint32_t)((k & 1) << 3);
}

// hi and lo parts of a complex number to the same place of a hi and a lo tile.
__device__ __forceinline__ void put2(unsigned char *hi, unsigned char *lo, uint32_t off, float x, float y) {
    const float2 h = make_float2(to_tf32(x), to_tf32(y));
    *reinterpret_cast<float2 *>(hi + off) = h;
    *reinterpret_cast<float2 *>(lo + off) = make_float2(to_tf32(x - h.x), to_tf32(y - h.y));
}

// hi and lo parts of four floats to the same place of a hi and a lo tile.
__device__ __forceinline__ void put4(unsigned char *hi, unsigned char *lo, uint32_t off, float4 v) {
    const float4 h = make_float4(to_tf32(v.x), to_tf32(v.y), to_tf32(v.z), to_tf32(v.w));
    *reinterpret_cast<float4 *>(hi + off) = h;
    *reinterpret_cast<float4 *>(lo + off) =
        make_float4(to_tf32(v.x - h.x), to_tf32(v.y - h.y), to_tf32(v.z - h.z), to_tf32(v.w - h.w));
}

struct TcArgs {
    int m, n, K;                 // left vectors, right columns, reduction
    const c32 *A, *B;
    int lda, ldb;
    int tm, tn, nsplit, kchunk;  // tiles, splits of the reduction and their length (a multiple of KST)
    float alpha, beta;           // A B
    const c32 *C;
    c32 *D;
    int ldc, ldd;
    c32 *part;                   // A^H B: FP32 partial tiles [split][j][i]
};

struct TcItem {
    int i0, j0, z, kbeg, kend, nst;   // first left vector and right column, split, reduction range, stages
};
template <int NT>
__device__ __forceinline__ TcItem tc_item(const TcArgs &a, int it) {
    TcItem w;
    const int tiles = a.tm * a.tn;
    w.z = it / tiles;
    const int t = it - w.z * tiles, ti = t / a.tn;
    w.i0 = ti * kRows;
    w.j0 = (t - ti * a.tn) * NT;
    w.kbeg = w.z * a.kchunk;
    w.kend = min(a.K, w.kbeg + a.kchunk);
    w.nst = (w.kend - w.kbeg + KST - 1) / KST;
    return w;
}

// CN: C = A^H B (partial tiles), else D = alpha A B + beta C.
template <bool CN, int NT>
__device__ __forceinline__ void tc_body(const TcArgs &a) {
    constexpr int A_BYTES = kRows * ROWB, B_BYTES = 2 * NT * ROWB, STAGE = stage_bytes(NT);
    constexpr int ACC = 2 * NT, TCOLS = 2 * ACC;           // TMEM columns of an accumulator, of both
    extern __shared__ unsigned char smraw[];
    unsigned char *base = align1k(smraw);
    uint64_t *full = reinterpret_cast<uint64_t *>(base + kRing * STAGE);
    uint64_t *empty = full + kRing, *accf = empty + kRing, *acce = accf + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + 2);
    volatile int *quit = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
    if (warp == kLoaders) tmem_alloc(tslot, TCOLS);
    if (tid == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(&full[s], kLoaders / kRing);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], kReaders);
        }
        *quit = 0;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = uniform(*tslot);
    const int nit = a.tm * a.tn * a.nsplit, it0 = blockIdx.x, step = gridDim.x;
    if (warp < kLoaders) {
        // ---- loaders: group w / 4 fills ring slot w / 4, that is every kRing-th stage, so that one
        // group's wait, stores and proxy fence overlap the others'.  Operands that are contiguous along
        // K: eight threads take a vector's eight numbers (64 bytes), or, for the right factor of A B,
        // which is small and stays in L2, four threads take two numbers each (fewer, 16-byte stores).
        // The left factor of A B is contiguous along its vectors: a warp takes 256 bytes of two columns,
        // a thread one vector's two consecutive K.
        constexpr int TH = 32 * kLoaders / kRing, EA = kRows * KST / TH, EB = NT * KST / TH;
        static_assert(EA * TH == kRows * KST && EB * TH == NT * KST, "whole elements per thread");
        const int t = tid % TH, s = warp / (kLoaders / kRing), tk = t & 7, tv = t >> 3;
        constexpr int VS = TH / KST;                       // vectors between a thread's elements
        float2 ra[EA], rb[EB];
        int li = it0, lk = s;                              // load cursor: item, stage
        TcItem lw{};
        auto settle = [&]() {                              // carry the cursor into the next items
            while (li < nit) {
                lw = tc_item<NT>(a, li);
                if (lk < lw.nst) return true;
                lk -= lw.nst;
                li += step;
            }
            return false;
        };
        bool more = settle();
        const float2 zero = make_float2(0.f, 0.f);
        auto load = [&]() {
            const int k0 = lw.kbeg + lk * KST;
#pragma unroll
            for (int q = 0; q < EA; ++q) {
                const int i = lw.i0 + (CN ? tv + VS * q : t % kRows);
                const int k = k0 + (CN ? tk : 2 * (t / kRows + TH / kRows * (q >> 1)) + (q & 1));
                const c32 *src = CN ? a.A + (size_t)i * a.lda + k : a.A + (size_t)k * a.lda + i;
                ra[q] = (i < a.m && k < lw.kend) ? __ldg(reinterpret_cast<const float2 *>(src)) : zero;
            }
#pragma unroll
            for (int q = 0; q < EB; ++q) {
                const int j = lw.j0 + (CN ? tv + VS * q : (t >> 2) + 2 * VS * (q >> 1));
                const int k = k0 + (CN ? tk : 2 * (t & 3) + (q & 1));
                rb[q] = (j < a.n && k < lw.kend) ? __ldg(reinterpret_cast<const float2 *>(a.B + (size_t)j * a.ldb + k)) : zero;
            }
        };
        // the first polls (a millisecond) do not look at *quit, which would cost a shared-memory read a stage (2 %)
        const long long spin = g_tc_spin, first = min(spin, 256LL);
        unsigned char *sAh = base + s * STAGE, *sAl = sAh + A_BYTES, *sBh = sAl + A_BYTES, *sBl = sBh + B_BYTES;
        if (more) load();
        for (uint32_t n = 0; more; ++n) {                  // n-th filling of the slot
            if (n > 0 && !mbar_wait(&empty[s], (n - 1) & 1u, first)) {
                bool ok = false;
                for (long long p = first; p < spin && !ok && !*quit; ++p) ok = mbar_wait(&empty[s], (n - 1) & 1u, 1);
                if (!ok) {
                    atomicExch(&g_tc_err, 1);
                    mbar_wait_quit(&empty[s], (n - 1) & 1u, quit);
                }
            }
            if (CN) {
#pragma unroll
                for (int q = 0; q < EA; ++q) put2(sAh, sAl, elem_at(tv + VS * q, tk), ra[q].x, ra[q].y);
            } else {
#pragma unroll
                for (int q = 0; q < EA; q += 2)
                    put4(sAh, sAl, elem_at(t % kRows, 2 * (t / kRows + TH / kRows * (q >> 1))),
                         make_float4(ra[q].x, ra[q].y, ra[q + 1].x, ra[q + 1].y));
            }
            if (CN) {
#pragma unroll
                for (int q = 0; q < EB; ++q) {
                    const float x = rb[q].x, y = rb[q].y;
                    put2(sBh, sBl, elem_at(tv + VS * q, tk), x, y);
                    put2(sBh, sBl, elem_at(NT + tv + VS * q, tk), y, -x);
                }
            } else {
#pragma unroll
                for (int q = 0; q < EB; q += 2) {
                    const int j = (t >> 2) + 2 * VS * (q >> 1), k = 2 * (t & 3);
                    const float2 x = rb[q], y = rb[q + 1];
                    put4(sBh, sBl, elem_at(j, k), make_float4(x.x, -x.y, y.x, -y.y));
                    put4(sBh, sBl, elem_at(NT + j, k), make_float4(x.y, x.x, y.y, y.x));
                }
            }
            lk += kRing;
            more = settle();
            if (more) load();                              // in flight during the fence and the next wait
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s]);
        }
    } else if (warp == kLoaders) {
        // ---- MMA issuer: the whole warp, one elected lane issuing; nothing in the loop depends on how a
        // wait ended (see tc.cuh)
        const uint32_t el = elect_one();
        constexpr uint32_t HI = (uint32_t)(make_desc_sw64(0) >> 32), IDESC = make_idesc_tf32(kRows, ACC);
        const uint32_t d0 = (uint32_t)make_desc_sw64(uniform(smem_u32(base)));
        int s = 0, g = 0;
        uint32_t ph = 0;
        int q = 0;                                         // items so far
        for (int it = it0; it < nit; it += step, ++q) {
            const int z = it / (a.tm * a.tn), kbeg = z * a.kchunk;
            const int nst = (min(a.K, kbeg + a.kchunk) - kbeg + KST - 1) / KST;
            const int b = q & 1;
            const uint32_t dt = tmem + (uint32_t)(b * ACC);
            if (q >= 2) mbar_wait_quit(&acce[b], (uint32_t)((q / 2 - 1) & 1), quit);
            for (int t = 0; t < nst; ++t, ++g) {
                mbar_wait_quit(&full[s], ph, quit);
                __syncwarp();
                fence_after_sync();
                const uint32_t ah = d0 + ((uint32_t)(s * STAGE) >> 4), bh = ah + ((2 * A_BYTES) >> 4);
                const uint32_t first = t == 0 ? 0u : 1u;
                mma_tf32_warp<kFill, HI, 0, 0>(el, dt, ah, bh, IDESC, first);
                mma_tf32_warp<kLastUse, HI, 0, B_BYTES>(el, dt, ah, bh, IDESC, 1u);
                mma_tf32_warp<kDiscard, HI, A_BYTES, 0>(el, dt, ah, bh, IDESC, 1u);
                mma_tf32_warp<kFill, HI, 32, 32>(el, dt, ah, bh, IDESC, 1u);
                mma_tf32_warp<kLastUse, HI, 32, B_BYTES + 32>(el, dt, ah, bh, IDESC, 1u);
                mma_tf32_warp<kDiscard, HI, A_BYTES + 32, 32>(el, dt, ah, bh, IDESC, 1u);
                mma_commit_warp(el, &empty[s]);
                if (++s == kRing) { s = 0; ph ^= 1; }
            }
            mma_commit_warp(el, &accf[b]);
        }
        if (*quit && el) atomicExch(&g_tc_err, 1);
        // every MMA is done before the CTA frees its TMEM
        if (g > 0) mbar_wait(&empty[(g - 1) % kRing], (uint32_t)(((g - 1) / kRing) & 1));
    } else {
        // ---- readers: warp w reads TMEM lanes 32 (w % 4) .. (the left vectors), 16 columns at a time
        const int quarter = warp & 3, r = quarter * 32 + lane;
        int q = 0;
        bool late = false;
        for (int it = it0; it < nit; it += step, ++q) {
            const TcItem w = tc_item<NT>(a, it);
            const int b = q & 1, i = w.i0 + r, nj = min(NT, a.n - w.j0);
            const bool row_ok = i < a.m;
            late |= !mbar_wait(&accf[b], (uint32_t)((q / 2) & 1));
            __syncwarp();
            fence_after_sync();
            const uint32_t t0 = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * ACC);
#pragma unroll 1
            for (int c0 = 0; c0 < nj; c0 += 16) {
                float re[16], im[16];
                tmem_ld16_nowait(t0 + (uint32_t)c0, re);
                tmem_ld16_nowait(t0 + (uint32_t)(NT + c0), im);
                if (CN) {
                    tmem_wait_ld(re, im);
                    c32 *P = a.part + ((size_t)w.z * a.n + w.j0 + c0) * a.m + i;
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj)
                        if (row_ok && c0 + jj < nj) P[(size_t)jj * a.m] = mkc(re[jj], im[jj]);
                } else {
                    // C may be D (in-place accumulate): the 16 loads of the step come before its stores
                    float2 cv[16];
                    const c32 *Cp = a.C + (size_t)(w.j0 + c0) * a.ldc + i;
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj)
                        cv[jj] = (row_ok && c0 + jj < nj && a.beta != 0.f)
                                     ? *reinterpret_cast<const float2 *>(Cp + (size_t)jj * a.ldc)
                                     : make_float2(0.f, 0.f);
                    tmem_wait_ld(re, im);
                    c32 *Dp = a.D + (size_t)(w.j0 + c0) * a.ldd + i;
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj)
                        if (row_ok && c0 + jj < nj)
                            Dp[(size_t)jj * a.ldd] =
                                mkc(fmaf(a.beta, cv[jj].x, a.alpha * re[jj]), fmaf(a.beta, cv[jj].y, a.alpha * im[jj]));
                }
            }
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[b]);
        }
        if (late && lane == 0) atomicExch(&g_tc_err, 1);
    }
    fence_before_sync();
    __syncthreads();
    if (warp == kLoaders) tmem_dealloc(tmem, TCOLS);
}

template <int NT>
__global__ void __launch_bounds__(kThreads, 1) k_tc_cn(TcArgs a) { tc_body<true, NT>(a); }
template <int NT>
__global__ void __launch_bounds__(kThreads, 1) k_tc_nn(TcArgs a) { tc_body<false, NT>(a); }

// One entry of k_tc_reduce in FP64, for sums that leave the FP32 range on the way.
__device__ __noinline__ c32 tc_reduce_fp64(const c32 *part, size_t tot, int nsplit, float alpha, float beta, c32 c) {
    double re = 0.0, im = 0.0;
    for (int z = 0; z < nsplit; ++z) {
        re += part[(size_t)z * tot].x;
        im += part[(size_t)z * tot].y;
    }
    re *= alpha;
    im *= alpha;
    if (beta != 0.f) {
        re += (double)beta * c.x;
        im += (double)beta * c.y;
    }
    return mkc((float)re, (float)im);
}

// C = alpha (sum of the partial tiles, in split order) + beta C.  The sum is a double-FP32 pair (TwoSum), its
// products with alpha and beta are exact, and the result is rounded once: FP64 arithmetic would cost 64
// cycles a warp and instruction.
__global__ void k_tc_reduce(int m, int n, int nsplit, float alpha, const c32 *__restrict__ part, float beta,
                            c32 *C, int ldc) {
    const size_t tot = (size_t)m * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = (int)(e / m);
        float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
        auto add = [](float &h, float &l, float x) {
            float err;
            df64::two_sum(h, x, h, err);
            l = __fadd_rn(l, err);
        };
#pragma unroll 8
        for (int z = 0; z < nsplit; ++z) {
            const c32 v = part[(size_t)z * tot + e];
            add(rh, rl, v.x);
            add(ih, il, v.y);
        }
        const c32 c = beta != 0.f ? C[(size_t)j * ldc + i] : mkc(0.f, 0.f);
        auto out = [alpha, beta](float h, float l, float x) {
            const float p = __fmul_rn(alpha, h), q = __fmul_rn(beta, x);
            float s, t;
            df64::two_sum(p, q, s, t);
            t = __fadd_rn(t, __fadd_rn(__fmaf_rn(alpha, h, -p), __fmaf_rn(beta, x, -q)));
            return __fadd_rn(s, __fmaf_rn(alpha, l, t));
        };
        c32 v = mkc(out(rh, rl, c.x), out(ih, il, c.y));
        if (!(fabsf(v.x) <= FLT_MAX && fabsf(v.y) <= FLT_MAX)) v = tc_reduce_fp64(part + e, tot, nsplit, alpha, beta, c);
        C[(size_t)j * ldc + i] = v;
    }
}

template <typename Kern>
int ensure_smem(Kern kern, size_t bytes, DeviceOnce &once) {
    const int dev = current_device();
    if (!once.done(dev)) {
        LG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
        once.mark(dev);
    }
    return LOBPCG_OK;
}

int num_sms_tc() {
    static std::atomic<int> cached{0};
    int v = cached.load();
    if (!v) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
        cached.store(v);
    }
    return v;
}

// Cycles of a stage (MMAs and shared-memory traffic) by NT.
constexpr int stage_cycles(int NT) { return NT == 128 ? 900 : NT == 64 ? 600 : 450; }

// NT of the cheapest tiling of n columns.
int pick_nt(int n) {
    int best = 128;
    for (int nt : {64, 32})
        if ((long long)((n + nt - 1) / nt) * stage_cycles(nt) < (long long)((n + best - 1) / best) * stage_cycles(best))
            best = nt;
    return best;
}

// Terms of one FP32 accumulation of A^H B, from K alone.  The tensor core truncates as it accumulates, so a
// sum loses about half a unit in the last place per MMA: entries of a Gram with chunks of c terms come out
// about 0.3 c 2^-24 too small.  A Rayleigh-Ritz step on nearly dependent directions divides by the small
// eigenvalues of S: where A's blocks lose more than S's, spurious low Ritz values appear.  (With the chunks
// chosen by the time of each shape, 2264 terms for the S and 2976 for the A of a 128-band block of the 120^3
// cell, its last block left orthonormality by 0.1 to 1e5 and one solve in seven broke down; with 744 for
// both, by 1e-6.)  So all products of one K have the same chunks, of at most 1024 terms, their number a
// multiple of the SMs, so that any number of tiles keeps them all busy to the end.  More partial tiles cost,
// GB300, K = 113081: 384 x 256 374 -> 403 us, 432 x 128 259 -> 289, 1152 x 1152 4.61 -> 5.53 ms; 128 x 128 92 as
// before.  At least 128 terms, where K is short: a tile's 128 KB of partial sums are then written in about the
// time of its stages (512 x 512 x 5000 56 -> 79 us, 16 x 16 x 3000 16.5 -> 15.1).
constexpr int kMinChunk = 128, kMaxChunk = 1024;
int cn_chunk(int K) {
    const long long sms = num_sms_tc(), rounds = (K + sms * kMaxChunk - 1) / (sms * kMaxChunk);
    const long long kc = (K + sms * rounds - 1) / (sms * rounds);
    return std::max(kMinChunk, (int)((kc + KST - 1) / KST * KST));
}
// Partial tiles at a time: larger products run in panels of rows and columns.
constexpr size_t kPartBytes = (size_t)256 << 20;

template <int NT>
int launch_cn(GemmWork &w, const TcArgs &all, float beta, c32 *C, int ldc, cudaStream_t s) {
    static DeviceOnce attr;
    LG_TRY(ensure_smem(k_tc_cn<NT>, smem_bytes(NT), attr));
    const int sms = num_sms_tc(), kchunk = cn_chunk(all.K), nsplit = (all.K + kchunk - 1) / kchunk;
    const long long units = std::max<long long>(1, (long long)(kPartBytes / (sizeof(c32) * nsplit)) / (kRows * NT));
    const int tm_all = (all.m + kRows - 1) / kRows, tn_all = (all.n + NT - 1) / NT;   // tiles of a panel: tmp x tnp <= units
    const int tmp = (int)std::min<long long>(tm_all, units), tnp = (int)std::min<long long>(tn_all, units / tmp);
    const int pm = std::min(all.m, tmp * kRows), pn = std::min(all.n, tnp * NT);
    LG_TRY(w.alloc->ensure(w.part, sizeof(c32) * (size_t)nsplit * pm * pn));
    for (int j0 = 0; j0 < all.n; j0 += tnp * NT)
        for (int i0 = 0; i0 < all.m; i0 += tmp * kRows) {
            TcArgs a = all;
            a.m = std::min(pm, all.m - i0);
            a.n = std::min(pn, all.n - j0);
            a.A = all.A + (size_t)i0 * all.lda;
            a.B = all.B + (size_t)j0 * all.ldb;
            a.tm = (a.m + kRows - 1) / kRows;
            a.tn = (a.n + NT - 1) / NT;
            a.kchunk = kchunk;
            a.nsplit = nsplit;
            a.part = reinterpret_cast<c32 *>(w.part.p);
            const int grid = (int)std::min<long long>(sms, (long long)a.tm * a.tn * nsplit);
            k_tc_cn<NT><<<grid, kThreads, smem_bytes(NT), s>>>(a);
            LG_TRY(check_launch("tensor-core gemm A^H B"));
            const size_t tot = (size_t)a.m * a.n;
            const int blocks = (int)std::min<size_t>((tot + 127) / 128, 4096);
            k_tc_reduce<<<blocks, 128, 0, s>>>(a.m, a.n, nsplit, a.alpha, a.part, beta, C + (size_t)j0 * ldc + i0, ldc);
            LG_TRY(check_launch("tensor-core gemm reduce"));
        }
    return LOBPCG_OK;
}

template <int NT>
int launch_nn(TcArgs &a, cudaStream_t s) {
    static DeviceOnce attr;
    LG_TRY(ensure_smem(k_tc_nn<NT>, smem_bytes(NT), attr));
    a.tm = (a.m + kRows - 1) / kRows;
    a.tn = (a.n + NT - 1) / NT;
    a.nsplit = 1;
    a.kchunk = (a.K + KST - 1) / KST * KST;
    k_tc_nn<NT><<<(int)std::min<long long>(num_sms_tc(), (long long)a.tm * a.tn), kThreads, smem_bytes(NT), s>>>(a);
    return check_launch("tensor-core gemm A B");
}

}  // namespace

int tc_gemm_cn(GemmWork &w, int m, int n, int K, float alpha, const c32 *A, int lda, const c32 *B, int ldb,
               float beta, c32 *C, int ldc, cudaStream_t s) {
    if (m <= 0 || n <= 0) return LOBPCG_OK;
    TcArgs a{};
    a.m = m;
    a.n = n;
    a.K = K;
    a.A = A;
    a.B = B;
    a.lda = lda;
    a.ldb = ldb;
    a.alpha = alpha;
    const int nt = pick_nt(n);
    if (nt == 128) return launch_cn<128>(w, a, beta, C, ldc, s);
    if (nt == 64) return launch_cn<64>(w, a, beta, C, ldc, s);
    return launch_cn<32>(w, a, beta, C, ldc, s);
}

int tc_gemm_nn(int M, int n, int k, float alpha, const c32 *A, int lda, const c32 *B, int ldb, float beta,
               const c32 *C, int ldc, c32 *D, int ldd, cudaStream_t s) {
    if (M <= 0 || n <= 0) return LOBPCG_OK;
    TcArgs a{};
    a.m = M;
    a.n = n;
    a.K = k;
    a.A = A;
    a.B = B;
    a.lda = lda;
    a.ldb = ldb;
    a.alpha = alpha;
    a.beta = beta;
    a.C = beta != 0.f ? C : D;
    a.ldc = beta != 0.f ? ldc : ldd;
    a.D = D;
    a.ldd = ldd;
    const int nt = pick_nt(n);
    if (nt == 128) return launch_nn<128>(a, s);
    if (nt == 64) return launch_nn<64>(a, s);
    return launch_nn<32>(a, s);
}

int *device_wait_flag() {
    static std::atomic<int *> cached{nullptr};
    int *p = cached.load();
    if (!p) {
        void *q = nullptr;
        if (cudaGetSymbolAddress(&q, g_tc_err) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        p = static_cast<int *>(q);
        cached.store(p);
    }
    return p;
}

int tc_set_spin_limit(long long polls) {
    const long long v = polls < 0 ? kSpinLimit : polls;
    LG_CUDA_TRY(cudaMemcpyToSymbol(g_tc_spin, &v, sizeof(v)));
    return oz_set_spin_limit(polls);
}

int tc_check_error() {
    const int oz = oz_check_error();   // (both flags are read and cleared)
    int h = 0;
    LG_CUDA_TRY(cudaMemcpyFromSymbol(&h, g_tc_err, sizeof(int)));
    if (h) {
        const int z = 0;
        LG_CUDA_TRY(cudaMemcpyToSymbol(g_tc_err, &z, sizeof(int)));
        return fail(LOBPCG_ERR_TIMEOUT,
                    "a bounded device wait ran out (tensor-core GEMM mbarrier or tridiagonalisation grid barrier)");
    }
    return oz;
}

}  // namespace lg
