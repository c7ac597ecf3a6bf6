// FP64-class complex128 GEMMs on the 5th-generation tensor cores (tcgen05, BF16
// operands, FP32 accumulators in TMEM): the tall contractions of the FP64-class
// work of the mixed schedule (all-band Grams, constraint projections and
// updates, block and sweep-end Ritz rotations, the KB projections of the FP64
// H X refresh) -- zgemm in the paper (Sec. 4.1), where it dominates.
//
// Arithmetic (error-free slicing after Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 2012; integer slices with exact
// fixed-point accumulation as in Ootomo, Ozaki and Yokota 2024):
//   * The reduction dimension is cut into chunks of 64 complex terms.  Within a
//     chunk every operand vector (a row of the product's left or right factor)
//     gets one power-of-two scale 2^e with max |x| < 2^e, and each real part is
//     written as x = 2^e sum_{p=1..6} d_p 2^{-8p} + (rest at most 2^{e-49}),
//     with integer digits |d_1| <= 256, |d_p| <= 128: x 2^{48-e} is rounded to
//     an integer from its FP64 bit pattern and peeled into signed base-256
//     digits with integer operations.  Integers of that size are exact BF16
//     numbers.
//   * x y = 2^{e_x + e_y} sum_{p,q} d_p d'_q 2^{-8(p+q)}: the digit products of
//     one "level" l = p + q (l = 2..7; products with p + q > 7 are below 2^-48
//     relative and dropped) are summed by the tensor core into one FP32
//     accumulator.  Each product is at most 2^16 and a level holds at most
//     2^17 per real term, so over the 128 real terms of a chunk every partial
//     sum is an integer below 2^24: FP32 accumulation is exact.
//   * After each chunk the six level accumulators are read from TMEM, scaled by
//     2^{e_x + e_y - 8 l} (exact) and added into a double-FP32 accumulator per
//     output (pairs of FP32 numbers, TwoSum; about 2^-48 relative), which is
//     written out as FP64.
//   Result: error about 2^-44 of sum |x||y| at worst (chunk scales are shared by
//   64 consecutive plane waves), FP64 class, at BF16 tensor throughput / 21.
//
// Complex arithmetic as one real product (re / im interleaved along K):
//   C = A^H B:  rows of the left factor: columns of A as (re, im) pairs; right
//               factor: two rows per column of B, (re, im) and (im, -re);
//               C_ij = P[2j][i] + i P[2j+1][i].
//   D = A B:    left factor: two rows per row of A, (re, -im) and (im, re);
//               right factor: columns of B as (re, im); D_ij = P[j][2i] + i P[j][2i+1].
//
// Data path: a split kernel writes each operand's digits once, as 64-byte-swizzled
// K-major BF16 tiles in the exact order one pipeline stage needs them (six slices
// of a 128- or 64-row tile x 32 K values, contiguous), plus the chunk scales.
// The product kernel (k_oz_mma: persistent, one CTA of 18 warps per SM, each taking every
// gridDim-th item, an output tile and a part of its reduction) streams the stages with one bulk
// copy per operand (cp.async.bulk into a 3-stage ring, mbarrier transaction counts), one warp
// issues the 42 MMAs of a stage (21 slice pairs x 2 K-steps of 16, M = 128, N = 64), and sixteen
// warps read the six levels of every chunk (tcgen05.ld) and fold them into the double-FP32 sums.
// The level accumulators rotate through eight slots of TMEM, so a chunk starts while the last
// levels of the one before it, and an item while the output of the one before it, are still read.
// Long reductions (A^H B) are split over the GPU and cut into K slabs that bound the digit
// scratch; FP64 partial tiles are summed in a fixed order (reproducible).  Every mbarrier wait is
// bounded; one that runs out sets a device flag (read by oz_check_error), the CTA's warps leave their
// loops, and it waits (bounded) for its copies and MMAs in flight, frees its TMEM and returns.  (The
// producer's first wait for a stage, whose limit tests lower, is repeated with the full limit.)
//
// What bounds it: the tensor cores would take 36 cycles an MMA (the left slice held in the
// collector, the right one read at 128 bytes a cycle), 6000 a chunk; issue, the waits for the
// stages and the slots and the folding leave about 9300.  Measured on a GB300 (SM clock
// 1.93 GHz), before and after the issue by a whole warp, the rotating slots, the folding without
// FP64 instructions and the persistent schedule:
//   A B    57925 x 320 x 320     1.97 -> 0.99 ms   (24 -> 48 TFLOP/s complex128)
//   A^H B  512 x 128 x 113081    2.66 -> 1.64 ms   (0.66 ms of it the split into digits)
//   Gram   1152, K = 113081      25.8 -> 12.0 ms   (2.7 ms of it the split)
#include "common.cuh"
#include "df64.cuh"
#include "tc.cuh"

#include <algorithm>
#include <cmath>
#include <utility>

namespace lg {

namespace {

using namespace tc;

constexpr int kSlices = 6;                   // 8-bit digits per real value
constexpr int kLevels = kSlices;             // p + q = 2 .. 7
constexpr int kStageK = 32;                  // real K (BF16) per stage: 64-byte tile rows
constexpr int kChunkStages = 4;              // 128 real K = 64 complex terms per exact chunk
constexpr int kChunkC = kStageK * kChunkStages / 2;
constexpr int TM = 128;                      // left-factor tile rows (MMA M)
constexpr int TQ = 64;                       // right-factor tile rows (MMA N)
constexpr int kTileA = TM * 64;              // bytes of one slice of a left tile stage
constexpr int kTileB = TQ * 64;
constexpr int kStageA = kSlices * kTileA;    // 48 KB
constexpr int kStageB = kSlices * kTileB;    // 24 KB
constexpr int kStageBytes = kStageA + kStageB;
constexpr int kRing = 3;
constexpr int kEpiWarps = 16;
constexpr int kCols = TQ / (kEpiWarps / 4);  // columns of a tile row that one epilogue warp folds
constexpr int kThreads = 32 * (kEpiWarps + 2);   // + producer warp + MMA warp
constexpr int kSlots = 8;                    // level accumulators of 64 columns in TMEM
constexpr int kTmemCols = kSlots * TQ;       // all 512
constexpr size_t kSmem = (size_t)kRing * kStageBytes + 1024 + 256;   // ring + alignment + barriers

// split modes: how a complex vector becomes real rows of a factor
constexpr int kRowsPlain = 0;   // one row (re, im)                     left of A^H B, right of A B
constexpr int kRowsCnB = 1;     // two rows (re, im), (im, -re)         right of A^H B
constexpr int kRowsNnA = 2;     // two rows (re, -im), (im, re)         left of A B

constexpr long long kMmaSpin = 1 << 15;      // polls of one wait of the MMA warp (an eighth of a second)

__device__ int g_oz_err = 0;
// Poll limit of the producer's first wait for a stage (lowered only by tests of the timeout path).
__device__ long long g_oz_spin = kSpinLimit;

// Byte offset of BF16 element (r, c) (c < 32) in a 64-byte-swizzled K-major tile:
// the 16-byte chunk c / 8 of row r sits at chunk position (c / 8) ^ ((r / 2) % 4).
__device__ __forceinline__ uint32_t swz64(int r, int c) {
    return (uint32_t)r * 64u + ((((uint32_t)c >> 3) ^ (((uint32_t)r >> 1) & 3u)) << 4) + (((uint32_t)c & 7u) << 1);
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Knuth TwoSum: s + err = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &err) {
    s = a + b;
    const float bb = s - a;
    err = (a - (s - bb)) + (b - bb);
}

// (hi, lo) += (x, y) in double-FP32 arithmetic, renormalised.
__device__ __forceinline__ void df_add(float &hi, float &lo, float x, float y) {
    float s, e;
    two_sum(hi, x, s, e);
    e += lo + y;
    hi = s + e;
    lo = e - (hi - s);
}

// The six base-256 digits of x relative to the chunk scale 2^e (|x| < 2^e), most significant
// first: F = round(x 2^(48 - e)) is formed exactly from the mantissa with a rounding shift, then
// peeled into signed digits d_6 .. d_2 in [-128, 127] from the low end; the rest, |d_1| <= 256,
// is the top digit.  x = 2^e sum_p d_p 2^(-8p) up to 2^(e-49).  Integer operations only.
__device__ __forceinline__ void digits(double x, int e, float (&d)[kSlices]) {
    const long long bits = __double_as_longlong(x);
    const int b = (int)((bits >> 52) & 0x7FF);
    long long F = 0;
    if (b > 0) {
        const unsigned long long m = (unsigned long long)(bits & 0xFFFFFFFFFFFFFLL) | (1ULL << 52);
        const int sh = 1027 + e - b;                       // >= 5 because |x| < 2^e
        if (sh < 60) F = (long long)((m + (1ULL << (sh - 1))) >> sh);
        if (bits < 0) F = -F;
    }
#pragma unroll
    for (int p = kSlices - 1; p >= 1; --p) {
        const long long dp = ((F + 128) & 0xFF) - 128;
        d[p] = (float)dp;
        F = (F - dp) >> 8;
    }
    d[0] = (float)F;
}

// ------------------------------------------------------------------ split
// One CTA: 32 complex vectors x one chunk (64 complex terms) of the K range
// [k0, k0 + nchunks * 64) of the operand X (element (v, k) at X[v * rs + k * ks]).
// Writes the chunk's digit tiles and the vectors' chunk exponents.
template <int TR, int MODE>
__global__ void __launch_bounds__(256)
k_oz_split(const z64 *__restrict__ X, long long rs, long long ks, int nvec, int K, int k0, int KS,
           unsigned char *__restrict__ T, int *__restrict__ E, int nvec_pad) {
    constexpr int RPC = MODE == kRowsPlain ? 1 : 2;
    __shared__ double2 tile[32][kChunkC + 1];
    __shared__ int ex[32];
    const int v0 = blockIdx.x * 32, chunk = blockIdx.y;
    const int kb = k0 + chunk * kChunkC;
    const int tid = threadIdx.x;
    if (ks == 1) {   // K contiguous: threads along K
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int v = tid / 64 + 4 * i, k = tid % 64;
            const int gv = v0 + v, gk = kb + k;
            double2 a = make_double2(0.0, 0.0);
            if (gv < nvec && gk < K) {
                const z64 z = X[(size_t)gv * rs + (size_t)gk];
                a = make_double2(z.x, z.y);
            }
            tile[v][k] = a;
        }
    } else {         // vectors contiguous: threads along the vectors
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int v = tid % 32, k = tid / 32 + 8 * i;
            const int gv = v0 + v, gk = kb + k;
            double2 a = make_double2(0.0, 0.0);
            if (gv < nvec && gk < K) {
                const z64 z = X[(size_t)gv * rs + (size_t)gk * ks];
                a = make_double2(z.x, z.y);
            }
            tile[v][k] = a;
        }
    }
    __syncthreads();
    // chunk exponent of each vector: 2^e > max |re|, |im| (e = 0 for an all-zero chunk).  Taken from
    // the FP64 exponent fields with integer operations (this GPU's FP64 units are slow): a normal
    // x with biased exponent b has |x| < 2^(b - 1022); subnormals count as zero.
    const int warp = tid >> 5, lane = tid & 31;
    for (int v = warp; v < 32; v += 8) {
        int bmax = 0;
        for (int k = lane; k < kChunkC; k += 32) {
            const int br = (int)((__double_as_longlong(tile[v][k].x) >> 52) & 0x7FF);
            const int bi = (int)((__double_as_longlong(tile[v][k].y) >> 52) & 0x7FF);
            bmax = max(bmax, max(br, bi));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bmax = max(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
        if (lane == 0) {
            const int e = bmax > 0 ? bmax - 1022 : 0;
            ex[v] = e;
            if (v0 + v < nvec_pad) E[(size_t)chunk * nvec_pad + v0 + v] = e;
        }
    }
    __syncthreads();
    // digits: 8 elements per thread, integer arithmetic on the FP64 bit patterns
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        const int idx = tid + 256 * i;
        const int v = idx / kChunkC, k = idx % kChunkC;
        if (v0 + v >= nvec_pad) continue;
        const double2 a = tile[v][k];
        const int e = ex[v];
        float dr[kSlices], di[kSlices];
        digits(a.x, e, dr);
        digits(a.y, e, di);
        const int kk = 2 * k;                       // real K of the re part within the chunk
        const int stage = chunk * kChunkStages + kk / kStageK, col = kk % kStageK;
#pragma unroll
        for (int sub = 0; sub < RPC; ++sub) {
            const int rr = RPC * (v0 + v) + sub;    // real row
            unsigned char *base = T + ((size_t)(rr / TR) * KS + stage) * (size_t)(kSlices * TR * 64) +
                                  swz64(rr % TR, col);
#pragma unroll
            for (int p = 0; p < kSlices; ++p) {
                float u0 = dr[p], u1 = di[p];
                if (MODE == kRowsCnB && sub == 1) { u0 = di[p]; u1 = -dr[p]; }
                if (MODE == kRowsNnA) {
                    if (sub == 0) { u0 = dr[p]; u1 = -di[p]; }
                    else { u0 = di[p]; u1 = dr[p]; }
                }
                __nv_bfloat162 pr = __floats2bfloat162_rn(u0, u1);   // integers <= 256: exact
                *reinterpret_cast<__nv_bfloat162 *>(base + (size_t)p * TR * 64) = pr;
            }
        }
    }
}

// ------------------------------------------------------------------ product
// Order of a stage's 42 MMAs (21 slice pairs x 2 K-steps): the MMAs of one left slice and K-step
// together, so that the slice is read from shared memory once (collector), slice 1 first, so that
// the levels are complete in the order 0 .. 5.
constexpr int kMmas = kSlices * (kSlices + 1);
struct MmaOrder {
    int L[kMmas], p[kMmas], kk[kMmas], col[kMmas];
    bool first[kMmas], last[kMmas];          // first / last MMA of its level in the stage
};
constexpr MmaOrder make_order() {
    MmaOrder o{};
    int i = 0;
    for (int p = 0; p < kSlices; ++p)
        for (int kk = 0; kk < 2; ++kk)
            for (int L = p; L < kLevels; ++L, ++i) {
                o.L[i] = L;
                o.p[i] = p;
                o.kk[i] = kk;
                o.col[i] = p + 1 == kLevels ? kDiscard : L == p ? kFill : L + 1 == kLevels ? kLastUse : kUse;
                o.first[i] = p == 0 && kk == 0;
                o.last[i] = p == L && kk == 1;
            }
    return o;
}

struct OzArgs {
    const unsigned char *At, *Bt;   // digit tiles of the left / right factor
    const int *EA, *EB;             // chunk exponents [chunk][vector]
    int KS;                         // stages per tile row (4 x chunks of the slab)
    int nvA_pad, nvB_pad;           // padded vector counts of the exponent tables
    int nchunks, cps;               // chunks of the slab, chunks per K split
    int lower;                      // skip tiles with every output column j above every row i
    int tq, tiles, nsplit;          // right tiles; output tiles that are computed; K splits
    // mode 0: FP64 partial tiles P[split][q][r] (written, or added to when accumulate)
    double *P;
    int ldp;
    size_t pstride;
    int accumulate;
    // mode 1: D = alpha (product) + beta C for complex rows row0 .. of A B
    int M, n, row0;
    double alpha, beta;
    int scaled;                     // alpha != 1 or beta != 0
    const z64 *C;
    int ldc;
    z64 *D;
    int ldd;
};

// One unit of work: output tile (rt, qt) and chunks [c0, c0 + nch) of its reduction.
struct OzItem {
    int rt, qt, z, c0, nch;
};
__device__ __forceinline__ OzItem oz_item(const OzArgs &a, int it) {
    OzItem w;
    w.z = it / a.tiles;
    int t = it - w.z * a.tiles;
    if (a.lower) {   // row tile rt has right tiles 0 .. 4 rt + 3 (right rows 64 qt .. are columns j >= 32 qt)
        w.rt = 0;
        for (int n = min(a.tq, 4); t >= n; n = min(a.tq, 4 * w.rt + 4)) {
            t -= n;
            ++w.rt;
        }
        w.qt = t;
    } else {
        w.rt = t / a.tq;
        w.qt = t - w.rt * a.tq;
    }
    w.c0 = w.z * a.cps;
    w.nch = max(0, min(a.nchunks - w.c0, a.cps));
    return w;
}

// MMA I of a stage (stage st of the chunk whose levels are u0 ..), with the waits and signals of its level.
template <int I>
__device__ __forceinline__ void issue_one(uint32_t el, uint32_t tmem, int u0, int st, uint32_t alo, uint32_t blo,
                                          uint64_t *accf, uint64_t *acce, bool &late) {
    constexpr MmaOrder O = make_order();
    constexpr int L = O.L[I], p = O.p[I], kk = O.kk[I];
    constexpr uint32_t HI = (uint32_t)(make_desc_sw64(0) >> 32);
    const int u = u0 + L, slot = u & (kSlots - 1);
    if (O.first[I] && st == 0 && u >= kSlots) {
        late |= !mbar_wait(&acce[slot], (uint32_t)((u / kSlots - 1) & 1), kMmaSpin);
        __syncwarp();
        fence_after_sync();
    }
    mma_bf16_warp<O.col[I], HI, p * kTileA + kk * 32, (L - p) * kTileB + kk * 32>(
        el, tmem + (uint32_t)(slot * TQ), alo, blo, make_idesc_bf16(TM, TQ), (O.first[I] && st == 0) ? 0u : 1u);
    if (O.last[I] && st == kChunkStages - 1) mma_commit_warp(el, &accf[slot]);
}
template <int... I>
__device__ __forceinline__ void issue_stage(std::integer_sequence<int, I...>, uint32_t el, uint32_t tmem, int u0, int st,
                                            uint32_t alo, uint32_t blo, uint64_t *accf, uint64_t *acce,
                                            bool &late) {
    (issue_one<I>(el, tmem, u0, st, alo, blo, accf, acce, late), ...);
}

template <int OUT>
__global__ void __launch_bounds__(kThreads, 1) k_oz_mma(OzArgs a) {
    extern __shared__ unsigned char smraw[];
    unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) &
                                                            ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(base + kRing * kStageBytes);
    uint64_t *empty = full + kRing;
    uint64_t *accf = empty + kRing;         // one per slot: its level's sums of the chunk are complete
    uint64_t *acce = accf + kSlots;         // one per slot: its level has been read
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + kSlots);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
    if (warp == kEpiWarps + 1) tmem_alloc(tslot, kTmemCols);
    if (tid == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int k = 0; k < kSlots; ++k) {
            mbar_init(&accf[k], 1);
            mbar_init(&acce[k], kEpiWarps);
        }
        *abort_flag = 0;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = uniform(*tslot);
    const int it0 = blockIdx.x, nit = a.tiles * a.nsplit, step = gridDim.x;
    if (warp == kEpiWarps) {
        // ---- producer: one bulk copy per factor per stage
        if (lane == 0) {
            const long long spin = g_oz_spin;
            int g = 0;
            for (int it = it0; it < nit && !*abort_flag; it += step) {
                const OzItem w = oz_item(a, it);
                const unsigned char *gA = a.At + ((size_t)w.rt * a.KS + (size_t)w.c0 * kChunkStages) * kStageA;
                const unsigned char *gB = a.Bt + ((size_t)w.qt * a.KS + (size_t)w.c0 * kChunkStages) * kStageB;
                for (int t = 0; t < w.nch * kChunkStages && !*abort_flag; ++t, ++g) {
                    const int s = g % kRing;
                    const uint32_t par = (uint32_t)((g / kRing - 1) & 1);
                    if (g >= kRing && !mbar_wait(&empty[s], par, spin)) {
                        atomicExch(&g_oz_err, 1);
                        if (!mbar_wait(&empty[s], par)) {
                            *abort_flag = 1;
                            break;
                        }
                    }
                    unsigned char *sA = base + s * kStageBytes, *sB = sA + kStageA;
                    mbar_expect_tx(&full[s], kStageBytes);
                    bulk_g2s(sA, gA + (size_t)t * kStageA, kStageA, &full[s]);
                    bulk_g2s(sB, gB + (size_t)t * kStageB, kStageB, &full[s]);
                }
            }
            // drain: the copies of the last (up to kRing) issued stages must land before exit
            for (int h = max(0, g - kRing); h < g; ++h) mbar_wait(&full[h % kRing], (uint32_t)((h / kRing) & 1));
        }
    } else if (warp == kEpiWarps + 1) {
        // ---- MMA issuer: the whole warp, one elected lane issuing.  Nothing in a chunk depends on how
        // a wait ended: a branch or a predicate that does, or a look at the abort flag between the polls of a
        // wait, makes the compiler give up uniform registers (80 cycles an MMA instead of 45, the whole kernel
        // 20 % slower).  A wait that runs out is recorded, the rest of the chunk is issued on whatever the
        // ring holds, and the error flag discards the result; the abort flag, which the other warps raise when
        // theirs run out, is looked at before every chunk.
        const uint32_t el = elect_one();
        const uint32_t d0 = (uint32_t)make_desc_sw64(uniform(smem_u32(base)));
        bool late = false;
        int s = 0;                           // ring position
        uint32_t ph = 0;                     // and its phase
        int nc = 0;                          // chunks of all this CTA's items
        for (int it = it0; it < nit; it += step) nc += max(0, min(a.nchunks - it / a.tiles * a.cps, a.cps));
        int ci = 0;
        for (; ci < nc; ++ci) {
            if (uniform((uint32_t)*abort_flag)) break;
            const int u0 = kLevels * ci;     // level L of chunk ci is the (u0 + L)-th level of the CTA
            for (int st = 0; st < kChunkStages; ++st) {
                late |= !mbar_wait(&full[s], ph, kMmaSpin);
                __syncwarp();
                fence_after_sync();
                const uint32_t alo = d0 + ((uint32_t)(s * kStageBytes) >> 4), blo = alo + (kStageA >> 4);
                issue_stage(std::make_integer_sequence<int, kMmas>{}, el, tmem, u0, st, alo, blo, accf, acce, late);
                mma_commit_warp(el, &empty[s]);
                if (++s == kRing) { s = 0; ph ^= 1; }
            }
        }
        if (late && el) {
            *abort_flag = 1;
            atomicExch(&g_oz_err, 1);
        }
        // wait (bounded) for the last stage's MMAs: its arrival follows that of the last level, which is all the
        // epilogue waits for, and neither it nor an MMA may outlive the CTA's shared memory and TMEM
        const int nst = ci * kChunkStages;
        if (nst > 0) mbar_wait(&empty[(nst - 1) % kRing], (uint32_t)(((nst - 1) / kRing) & 1));
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .., columns kCols (w / 4) ..
        const int wq = warp & 3, h = warp >> 2;
        const int row = wq * 32 + lane;
        const uint32_t taddr = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)(h * kCols);
        constexpr int rpcA = OUT == 0 ? 1 : 2, rpcB = OUT == 0 ? 2 : 1;
        bool ok = true;
        int u0 = 0;                                        // levels read so far
        for (int it = it0; it < nit; it += step) {
            const OzItem w = oz_item(a, it);
            const int rr = w.rt * TM + row;                // real left row
            const int *EA = a.EA + (size_t)w.c0 * a.nvA_pad + rr / rpcA;
            const int4 *EB =
                reinterpret_cast<const int4 *>(a.EB + (size_t)w.c0 * a.nvB_pad + (w.qt * TQ + h * kCols) / rpcB);
            float ah[kCols], al[kCols];
#pragma unroll
            for (int j = 0; j < kCols; ++j) ah[j] = al[j] = 0.f;
            for (int ci = 0; ci < w.nch; ++ci, u0 += kLevels) {
                // Chunk sum per column as a double-FP32 pair (ch, cl) in units of level 2.  The levels are
                // integers below 2^24, each worth 256 of the next: t = 256 hi + v and its rounding error
                // v - (t - 256 hi) are exact (a fast TwoSum: either |256 hi| >= |v|, or every term is an
                // integer below 2^25).  Levels 3-5 (at most 2^-16 of the chunk's scale) go into the low
                // part, whose FP32 rounding then stays below 2^-40 of that scale.
                // Levels 0-3 are read together as soon as the last of them is complete: the next chunk's
                // levels 2-5 wait for their slots.
                float ch[kCols], cl[kCols];
                {
                    const int k = (u0 + 3) & (kSlots - 1);
                    ok = __all_sync(0xffffffffu,
                                    !*abort_flag && mbar_wait(&accf[k], (uint32_t)(((u0 + 3) / kSlots) & 1)));
                    if (!ok) break;
                    fence_after_sync();
                    float v1[kCols], v2[kCols], v3[kCols];
                    tmem_ld16_nowait(taddr + (uint32_t)(((u0 + 0) & (kSlots - 1)) * TQ), ch);
                    tmem_ld16_nowait(taddr + (uint32_t)(((u0 + 1) & (kSlots - 1)) * TQ), v1);
                    tmem_ld16_nowait(taddr + (uint32_t)(((u0 + 2) & (kSlots - 1)) * TQ), v2);
                    tmem_ld16_nowait(taddr + (uint32_t)(k * TQ), v3);
                    tmem_wait_ld(ch, v1, v2, v3);
                    fence_before_sync();
                    __syncwarp();
                    if (lane < 4) mbar_arrive(&acce[(u0 + lane) & (kSlots - 1)]);
#pragma unroll
                    for (int j = 0; j < kCols; ++j) {
                        const float t1 = fmaf(ch[j], 256.f, v1[j]), e1 = v1[j] - fmaf(ch[j], -256.f, t1);
                        const float t2 = fmaf(t1, 256.f, v2[j]), e2 = v2[j] - fmaf(t1, -256.f, t2);
                        ch[j] = t2;
                        cl[j] = fmaf(v3[j], 0x1p-8f, fmaf(e1, 256.f, e2));
                    }
                }
                {
                    const int k = (u0 + 5) & (kSlots - 1);
                    ok = __all_sync(0xffffffffu,
                                    !*abort_flag && mbar_wait(&accf[k], (uint32_t)(((u0 + 5) / kSlots) & 1)));
                    if (!ok) break;
                    fence_after_sync();
                    float v4[kCols], v5[kCols];
                    tmem_ld16_nowait(taddr + (uint32_t)(((u0 + 4) & (kSlots - 1)) * TQ), v4);
                    tmem_ld16_nowait(taddr + (uint32_t)(k * TQ), v5);
                    tmem_wait_ld(v4, v5);
                    fence_before_sync();
                    __syncwarp();
                    if (lane < 2) mbar_arrive(&acce[(u0 + 4 + lane) & (kSlots - 1)]);
#pragma unroll
                    for (int j = 0; j < kCols; ++j) cl[j] = fmaf(v5[j], 0x1p-24f, fmaf(v4[j], 0x1p-16f, cl[j]));
                }
                // one unit of level 2 is 2^(er + eb - 32): the exponent field alone where the scales of four
                // neighbouring vectors are normal numbers
                const int er = EA[(size_t)ci * a.nvA_pad];
#pragma unroll
                for (int j0 = 0; j0 < kCols; j0 += 4 * rpcB) {
                    const int4 t = EB[(size_t)ci * (a.nvB_pad / 4) + j0 / (4 * rpcB)];
                    const int e[4] = {er + t.x, er + t.y, er + t.z, er + t.w};
                    const int lo4 = min(min(e[0], e[1]), min(e[2], e[3]));
                    const int hi4 = max(max(e[0], e[1]), max(e[2], e[3]));
                    if (lo4 > 32 - 127 && hi4 < 32 + 128) {
#pragma unroll
                        for (int k = 0; k < 4 * rpcB; ++k) {
                            const float S = __int_as_float((e[k / rpcB] + (127 - 32)) << 23);
                            df_add(ah[j0 + k], al[j0 + k], ch[j0 + k] * S, cl[j0 + k] * S);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 4 * rpcB; ++k) {   // 2^e as a product of two normal numbers
                            const int ek = min(max(e[k / rpcB] - 32, -252), 254), e1 = ek >> 1;
                            const float S1 = __int_as_float((e1 + 127) << 23), S2 = __int_as_float((ek - e1 + 127) << 23);
                            df_add(ah[j0 + k], al[j0 + k], ch[j0 + k] * S1 * S2, cl[j0 + k] * S1 * S2);
                        }
                    }
                }
            }
            if (!ok) break;
            // The two forms of the output are separate loops: an FP64 instruction that is predicated off
            // costs its 64 cycles all the same.
            if (OUT == 0) {
                double *P = a.P + (size_t)w.z * a.pstride + (size_t)(w.qt * TQ + h * kCols) * a.ldp + rr;
                if (a.accumulate) {
#pragma unroll
                    for (int j = 0; j < kCols; ++j) P[(size_t)j * a.ldp] += pair_to_double(ah[j], al[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < kCols; ++j) P[(size_t)j * a.ldp] = pair_to_double(ah[j], al[j]);
                }
            } else if ((rr >> 1) < a.M) {
                const size_t at = 2 * (size_t)(a.row0 + (rr >> 1)) + (rr & 1);   // of the column, in reals
                const int jc = w.qt * TQ + h * kCols;
                double *Dd = reinterpret_cast<double *>(a.D) + at;
                if (a.scaled) {
                    const double *Cd = reinterpret_cast<const double *>(a.C) + at;
#pragma unroll
                    for (int j = 0; j < kCols; ++j) {
                        if (jc + j >= a.n) break;
                        double val = a.alpha * pair_to_double(ah[j], al[j]);
                        if (a.beta != 0.0) val += a.beta * Cd[2 * (size_t)(jc + j) * a.ldc];
                        Dd[2 * (size_t)(jc + j) * a.ldd] = val;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < kCols; ++j) {
                        if (jc + j >= a.n) break;
                        Dd[2 * (size_t)(jc + j) * a.ldd] = pair_to_double(ah[j], al[j]);
                    }
                }
            }
        }
        if (!ok) {
            *abort_flag = 1;
            atomicExch(&g_oz_err, 1);
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == kEpiWarps + 1) tmem_dealloc(tmem, kTmemCols);
}

// C = alpha (P-assembled A^H B) + beta C, P[split][q][r] with q = 2 j + (0: re, 1: im).
__global__ void k_oz_finish_cn(int m, int n, int nsplit, const double *__restrict__ P, int ldp, size_t pstride,
                               double alpha, double beta, z64 *C, int ldc, int lower) {
    const size_t tot = (size_t)m * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = (int)(e / m);
        if (lower && i < j) continue;
        double re = 0.0, im = 0.0;
        for (int zz = 0; zz < nsplit; ++zz) {
            re += P[zz * pstride + (size_t)(2 * j) * ldp + i];
            im += P[zz * pstride + (size_t)(2 * j + 1) * ldp + i];
        }
        z64 v = mkc(alpha * re, alpha * im);
        if (beta != 0.0) v = v + beta * C[(size_t)j * ldc + i];
        C[(size_t)j * ldc + i] = v;
    }
}

int ensure_attr() {
    static DeviceOnce once;
    const int dev = current_device();
    if (!once.done(dev)) {
        LG_CUDA_TRY(cudaFuncSetAttribute(k_oz_mma<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
        LG_CUDA_TRY(cudaFuncSetAttribute(k_oz_mma<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
        once.mark(dev);
    }
    return LOBPCG_OK;
}

int num_sms() {
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

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Digits of nvec vectors over K range [k0, k0 + nchunks * 64) into tiles of TR real rows.
template <int TR, int MODE>
int split(const z64 *X, long long rs, long long ks, int nvec, int K, int k0, int nchunks, unsigned char *T, int *E,
          int nvec_pad, cudaStream_t s) {
    const int KS = nchunks * kChunkStages;
    k_oz_split<TR, MODE><<<dim3((nvec_pad + 31) / 32, nchunks), 256, 0, s>>>(X, rs, ks, nvec, K, k0, KS, T, E,
                                                                             nvec_pad);
    return check_launch("FP64-class tensor-core GEMM: operand digits");
}

// Chunks per K split of `tiles` output tiles over `chunks` chunks: every SM takes whole items (a tile
// and a split), so the makespan is the items of the busiest SM times a split's chunks plus about one
// chunk's time for an item's output; the shortest wins, of two alike the fewer splits.  At least two
// items per SM: a split's chunks are summed in double-FP32, whose rounding grows with their number (A^H B
// 300 x 300 x 20000, error against 64 bits: one sum of 63 chunks 4.5e-15, of 29 3.8e-15), the splits in FP64.
int pick_cps(long long tiles, int chunks) {
    const int least = (int)std::min<long long>(chunks, (2LL * num_sms() + tiles - 1) / tiles);
    int best_cps = chunks;
    double best = 1e300;
    for (int ns = least; ns <= std::max(128, 2 * least) && ns <= chunks; ++ns) {
        const int cps = (chunks + ns - 1) / ns;
        const long long items = tiles * ((chunks + cps - 1) / cps);
        const double t = (double)((items + num_sms() - 1) / num_sms()) * (cps + 1.0) + 0.05 * ns;
        if (t < best) {
            best = t;
            best_cps = cps;
        }
    }
    return std::max(1, best_cps);
}

// Scratch budget of the digit tiles of one slab (bytes).
constexpr size_t kSlabBytes = (size_t)768 << 20;

}  // namespace

// C = alpha A^H B + beta C, complex128, A: K x m (lda), B: K x n (ldb), C: m x n (ldc).
// lower: only entries i >= j are written (and tiles wholly above the diagonal skipped).
int oz_gemm_cn(GemmWork &w, int m, int n, int K, double alpha, const z64 *A, int lda, const z64 *B, int ldb,
               double beta, z64 *C, int ldc, cudaStream_t s, bool lower) {
    if (m <= 0 || n <= 0) return LOBPCG_OK;
    LG_TRY(ensure_attr());
    const int mA = round_up(m, TM);            // left real rows (one per column of A)
    const int qB = round_up(2 * n, TQ);        // right real rows (two per column of B)
    const int nvA = mA, nvB = qB / 2;          // padded vector counts
    const int Kc = std::max(1, (K + kChunkC - 1) / kChunkC);   // chunks of the whole reduction
    // slab: chunks whose digits fit the scratch budget
    const size_t per_chunk = (size_t)kChunkStages * ((size_t)(mA / TM) * kStageA + (size_t)(qB / TQ) * kStageB);
    const int slab = std::max(1, std::min(Kc, (int)(kSlabBytes / per_chunk)));
    const int tm = mA / TM, tq = qB / TQ;
    long long tiles = 0;
    for (int rt = 0; rt < tm; ++rt)
        for (int qt = 0; qt < tq; ++qt)
            if (!lower || 32 * qt <= TM * rt + TM - 1) ++tiles;
    const int cps = pick_cps(tiles, slab);
    const int nsplit = (slab + cps - 1) / cps;
    LG_TRY(w.alloc->ensure(w.oz_a, per_chunk * slab));
    LG_TRY(w.alloc->ensure(w.oz_e, sizeof(int) * (size_t)slab * (nvA + nvB)));
    LG_TRY(w.alloc->ensure(w.oz_p, sizeof(double) * (size_t)nsplit * qB * mA));
    unsigned char *At = static_cast<unsigned char *>(w.oz_a.p);
    unsigned char *Bt = At + (size_t)slab * kChunkStages * tm * kStageA;
    int *EA = static_cast<int *>(w.oz_e.p), *EB = EA + (size_t)slab * nvA;
    double *P = static_cast<double *>(w.oz_p.p);
    for (int cb = 0, first = 1; cb < Kc; cb += slab, first = 0) {
        const int nc = std::min(slab, Kc - cb);
        const int k0 = cb * kChunkC;
        LG_TRY((split<TM, kRowsPlain>(A, lda, 1, m, K, k0, nc, At, EA, nvA, s)));
        LG_TRY((split<TQ, kRowsCnB>(B, ldb, 1, n, K, k0, nc, Bt, EB, nvB, s)));
        OzArgs a{};
        a.At = At;
        a.Bt = Bt;
        a.EA = EA;
        a.EB = EB;
        a.KS = nc * kChunkStages;
        a.nvA_pad = nvA;
        a.nvB_pad = nvB;
        a.nchunks = nc;
        a.cps = cps;
        a.lower = lower ? 1 : 0;
        a.P = P;
        a.ldp = mA;
        a.pstride = (size_t)qB * mA;
        a.accumulate = first ? 0 : 1;
        a.tq = tq;
        a.tiles = (int)tiles;
        a.nsplit = nsplit;
        k_oz_mma<0><<<(int)std::min<long long>(num_sms(), tiles * nsplit), kThreads, kSmem, s>>>(a);
        LG_TRY(check_launch("FP64-class tensor-core GEMM A^H B"));
    }
    const size_t tot = (size_t)m * n;
    const int blocks = (int)std::min<size_t>((tot + 255) / 256, 4096);
    k_oz_finish_cn<<<blocks, 256, 0, s>>>(m, n, nsplit, P, mA, (size_t)qB * mA, alpha, beta, C, ldc,
                                          lower ? 1 : 0);
    return check_launch("FP64-class tensor-core GEMM: partial sums");
}

// D = alpha A B + beta C, complex128, A: M x k (lda), B: k x n (ldb), C, D: M x n.
int oz_gemm_nn(GemmWork &w, int M, int n, int k, double alpha, const z64 *A, int lda, const z64 *B, int ldb,
               double beta, const z64 *C, int ldc, z64 *D, int ldd, cudaStream_t s) {
    if (M <= 0 || n <= 0) return LOBPCG_OK;
    LG_TRY(ensure_attr());
    const int Kc = std::max(1, (k + kChunkC - 1) / kChunkC);
    const int qB = round_up(n, TQ);
    const int nvB = qB;
    // slab of complex rows of A (two real rows each): a multiple of 64 rows (one left tile)
    const size_t per_row = (size_t)2 * Kc * kChunkStages * kSlices * 64;   // bytes of digits per complex row
    int rows = (int)std::min<size_t>((size_t)round_up(M, TM / 2), std::max<size_t>(TM / 2, kSlabBytes / per_row));
    rows = std::max(TM / 2, rows / (TM / 2) * (TM / 2));
    const int nvA = rows;
    const size_t bytesA = (size_t)(2 * rows / TM) * Kc * kChunkStages * kStageA;
    const size_t bytesB = (size_t)(qB / TQ) * Kc * kChunkStages * kStageB;
    LG_TRY(w.alloc->ensure(w.oz_a, bytesA + bytesB));
    LG_TRY(w.alloc->ensure(w.oz_e, sizeof(int) * (size_t)Kc * (nvA + nvB)));
    unsigned char *At = static_cast<unsigned char *>(w.oz_a.p), *Bt = At + bytesA;
    int *EA = static_cast<int *>(w.oz_e.p), *EB = EA + (size_t)Kc * nvA;
    LG_TRY((split<TQ, kRowsPlain>(B, ldb, 1, n, k, 0, Kc, Bt, EB, nvB, s)));
    for (int r0 = 0; r0 < M; r0 += rows) {
        const int mr = std::min(rows, M - r0);
        LG_TRY((split<TM, kRowsNnA>(A + r0, 1, lda, mr, k, 0, Kc, At, EA, nvA, s)));
        OzArgs a{};
        a.At = At;
        a.Bt = Bt;
        a.EA = EA;
        a.EB = EB;
        a.KS = Kc * kChunkStages;
        a.nvA_pad = nvA;
        a.nvB_pad = nvB;
        a.nchunks = Kc;
        a.cps = Kc;
        a.M = mr;
        a.n = n;
        a.row0 = r0;
        a.alpha = alpha;
        a.beta = beta;
        a.scaled = alpha != 1.0 || beta != 0.0;
        a.C = beta != 0.0 ? C : D;
        a.ldc = beta != 0.0 ? ldc : ldd;
        a.D = D;
        a.ldd = ldd;
        const int tm = (2 * mr + TM - 1) / TM;
        a.tq = qB / TQ;
        a.tiles = a.tq * tm;
        a.nsplit = 1;
        k_oz_mma<1><<<std::min(num_sms(), a.tiles), kThreads, kSmem, s>>>(a);
        LG_TRY(check_launch("FP64-class tensor-core GEMM A B"));
    }
    return LOBPCG_OK;
}

int oz_set_spin_limit(long long polls) {
    const long long v = polls < 0 ? kSpinLimit : polls;
    LG_CUDA_TRY(cudaMemcpyToSymbol(g_oz_spin, &v, sizeof(v)));
    return LOBPCG_OK;
}

int oz_check_error() {
    int h = 0;
    LG_CUDA_TRY(cudaMemcpyFromSymbol(&h, g_oz_err, sizeof(int)));
    if (h) {
        const int zero = 0;
        LG_CUDA_TRY(cudaMemcpyToSymbol(g_oz_err, &zero, sizeof(int)));
        return fail(LOBPCG_ERR_TIMEOUT, "a bounded device wait ran out (FP64-class tensor-core GEMM)");
    }
    return LOBPCG_OK;
}

}  // namespace lg
