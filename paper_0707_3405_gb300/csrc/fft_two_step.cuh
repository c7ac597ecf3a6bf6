// Double-FP32, FP64 and FP32 passes of the local potential (Sec. 4.1: Goedecker's zero-padded FFT) for grid edges
// N = R1 R2 with both factors small enough for a thread's registers.
//
// Same three passes as fft.cu (A: sphere -> z-FFT -> y-FFT, B: x-FFT, V, x-FFT, C: y-FFT -> z-FFT ->
// sphere), with these differences:
//   * A line is transformed in two steps.  Inverse, n = a + R2 b, k = k1 + R1 k2: a thread takes the R1
//     values of one a, transforms over b, multiplies by W_N^{a k1} and puts them back where they
//     were; after one barrier a thread takes the R2 values of one k1 and transforms over a.  The forward
//     transform runs the same two steps backwards (over k2 first).  Every thread writes only where
//     it has read, so a step needs no barrier inside, and a line has one exchange through shared
//     memory instead of one per radix.
//   * Pass B keeps the second inverse step, the product with V and the first forward step in registers: one
//     round trip through shared memory per line and direction, three barriers a block.
//   * Factors that split into coprime ones (6, 10, 12, 15) are transformed without inner twiddles (Good
//     1958; Thomas 1963).
//   * x and y are indexed from the first occupied plane and row: that multiplies the real-space values by
//     a phase exp(-2 pi i (x nx0 + y ny0) / N), which V commutes with and the way back undoes.  With at
//     most N / 2 + 1 occupied planes and rows (the half box of Sec. 5.1) the zero inputs and unneeded outputs
//     of the 8-point steps are then known at compile time and left out.
//   * The twiddle products and the 3- and 5-point constants' sums add their exact FP32 products before they
//     are renormalised (19 instead of 25 operations per two-term sum).
// What bounds it: FP32 issue.  Measured on a GB300, 9 bands of the 120^3 cell a launch, us, against the
// shared-memory passes with one exchange and two barriers per radix (4, 2, 5, 3): pass A 227 -> 122,
// B 675 -> 295, C 288 -> 155; H on 128 bands with 432 projectors 20.7 -> 12.1 ms.  FP64 is bound by its
// units: 64 bands of the 72^3 cell, pass A 540 -> 390, B 1620 -> 1000, C 614 -> 405.  FP32, 19 bands of the
// 120^3 cell against the register passes (fft_reg.cu): A 67 -> 53, B 119 -> 92 (issuing 41 % of the cycles, the
// shared-memory pipe 68 % busy, 200 MB of DRAM), C 71 -> 61; both twiddle products of pass B in its second step
// (one read instead of two), five or seven blocks an SM, 16 lines a block, 256 threads or 16-line chunks in the
// plane passes: 2 to 5 % slower.
#pragma once

#include "common.cuh"
#include "df64.cuh"

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace lg {

// One application of the passes: S the type of the transforms and of the half box T2, R that of the bands.
template <typename S, typename R>
struct Fft2Args {
    const FFTGeom *g;
    const cx<R> *X;
    int ldx;
    cx<R> *Y;
    int ldy, nb;
    const R *kin;
    const S *vt;        // V / N^3 as [z][x][y]
    const cx<R> *tw;
    cx<S> *T2;
    int nbatch, smem_max;
    cudaStream_t s;
};

// The passes for the grid edges of one source file each; 1 where they do not apply.
#define LG_FFT2(n)                                   \
    int fft2_df_##n(const Fft2Args<df64f, double> &); \
    int fft2_f64_##n(const Fft2Args<double, double> &); \
    int fft2_f32_##n(const Fft2Args<float, float> &);
LG_FFT2(1) LG_FFT2(2) LG_FFT2(3) LG_FFT2(4)
#undef LG_FFT2

namespace f2s {

using D = df64f;

// exact product pieces of two pairs: p + e = a b up to 2^-48 |a b|
__device__ __forceinline__ void prod(D a, D b, float &p, float &e) {
    p = __fmul_rn(a.hi, b.hi);
    e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
}
// a x + b y
__device__ __forceinline__ D dot2(D a, D x, D b, D y) {
    float p, e, q, f, s, t;
    prod(a, x, p, e);
    prod(b, y, q, f);
    df64::two_sum(p, q, s, t);
    D r;
    df64::fast_two_sum(s, __fadd_rn(t, __fadd_rn(e, f)), r.hi, r.lo);
    return r;
}
// c + a x + b y
__device__ __forceinline__ D dot2_add(D c, D a, D x, D b, D y) {
    float p, e, q, f, s, t, s2, t2;
    prod(a, x, p, e);
    prod(b, y, q, f);
    df64::two_sum(c.hi, p, s, t);
    df64::two_sum(s, q, s2, t2);
    D r;
    df64::fast_two_sum(s2, __fadd_rn(__fadd_rn(t, t2), __fadd_rn(c.lo, __fadd_rn(e, f))), r.hi, r.lo);
    return r;
}
// The same sums in plain arithmetic.
template <typename R>
__device__ __forceinline__ R dot2(R a, R x, R b, R y) { return fma(a, x, b * y); }
template <typename R>
__device__ __forceinline__ R dot2_add(R c, R a, R x, R b, R y) { return fma(a, x, fma(b, y, c)); }
__device__ __forceinline__ D half(D a) { return D(0.5f * a.hi, 0.5f * a.lo); }
template <typename R>
__device__ __forceinline__ R half(R a) { return R(0.5) * a; }

template <typename S>
__device__ __forceinline__ cx<S> cmul(cx<S> a, cx<S> w) {
    return mkc<S>(dot2(a.x, w.x, -a.y, w.y), dot2(a.x, w.y, a.y, w.x));
}
// a conj(w)
template <typename S>
__device__ __forceinline__ cx<S> cmulc(cx<S> a, cx<S> w) {
    return mkc<S>(dot2(a.x, w.x, a.y, w.y), dot2(a.y, w.x, -a.x, w.y));
}
template <bool INV, typename S>
__device__ __forceinline__ cx<S> mul_i(cx<S> a) { return INV ? mkc<S>(-a.y, a.x) : mkc<S>(a.y, -a.x); }
template <bool INV, typename S>
__device__ __forceinline__ cx<S> twid(cx<S> a, cx<S> w) { return INV ? cmulc(a, w) : cmul(a, w); }   // w = W_N^j (forward)

// ------------------------------------------------------------- small transforms in registers
// P<R, INV>::run(v, tw): v <- DFT_R v; tw: the N-entry table, TS = N / R its stride for W_R.
template <typename S, int R, bool INV, int N>
struct P;
template <typename S, bool INV, int N>
struct P<S, 1, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&)[1], const C *) {}
};
template <typename S, bool INV, int N>
struct P<S, 2, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&v)[2], const C *) {
        const C a = v[0], b = v[1];
        v[0] = a + b;
        v[1] = a - b;
    }
};
template <typename S, bool INV, int N>
struct P<S, 3, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&v)[3], const C *) {
        const S s3 = (S)0.86602540378443864676;   // sin(2 pi / 3)
        const C a = v[0], t1 = v[1] + v[2], t2 = mkc<S>(a.x - half(t1.x), a.y - half(t1.y));
        const C t3 = s3 * mul_i<INV>(v[1] - v[2]);
        v[0] = a + t1;
        v[1] = t2 + t3;
        v[2] = t2 - t3;
    }
};
template <typename S, bool INV, int N>
struct P<S, 4, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&v)[4], const C *) {
        const C t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], t3 = mul_i<INV>(v[1] - v[3]);
        v[0] = t0 + t2;
        v[2] = t0 - t2;
        v[1] = t1 + t3;
        v[3] = t1 - t3;
    }
};
template <typename S, bool INV, int N>
struct P<S, 5, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&v)[5], const C *) {
        const S c1 = (S)0.30901699437494742410, c2 = (S)-0.80901699437494742410;   // cos(2 pi / 5), cos(4 pi / 5)
        const S s1 = (S)0.95105651629515357212, s2 = (S)0.58778525229247312917;    // sin(2 pi / 5), sin(4 pi / 5)
        const C a = v[0], p = v[1] + v[4], q = v[2] + v[3];
        const C m = mul_i<INV>(v[1] - v[4]), k = mul_i<INV>(v[2] - v[3]);
        const C r1 = mkc<S>(dot2_add(a.x, c1, p.x, c2, q.x), dot2_add(a.y, c1, p.y, c2, q.y));
        const C r2 = mkc<S>(dot2_add(a.x, c2, p.x, c1, q.x), dot2_add(a.y, c2, p.y, c1, q.y));
        const C i1 = mkc<S>(dot2(s1, m.x, s2, k.x), dot2(s1, m.y, s2, k.y));
        const C i2 = mkc<S>(dot2(s2, m.x, -s1, k.x), dot2(s2, m.y, -s1, k.y));
        v[0] = a + p + q;
        v[1] = r1 + i1;
        v[4] = r1 - i1;
        v[2] = r2 + i2;
        v[3] = r2 - i2;
    }
};
// 8 points; ZIN: v[5..7] are zero; NOUT: outputs 5..7 are not needed.
template <typename S, bool INV, bool ZIN, bool NOUT>
__device__ __forceinline__ void dft8(cx<S> (&v)[8]) {
    using C = cx<S>;
    const S h = (S)0.70710678118654752440;   // 1 / sqrt(2)
    // even half: 0 2 4 6, odd half: 1 3 5 7
    const C e0 = v[0] + v[4], e1 = v[0] - v[4];
    const C e2 = ZIN ? v[2] : v[2] + v[6], e3 = mul_i<INV>(ZIN ? v[2] : v[2] - v[6]);
    const C o0 = ZIN ? v[1] : v[1] + v[5], o1 = ZIN ? v[1] : v[1] - v[5];
    const C o2 = ZIN ? v[3] : v[3] + v[7], o3 = mul_i<INV>(ZIN ? v[3] : v[3] - v[7]);
    const C E0 = e0 + e2, E2 = e0 - e2, E1 = e1 + e3, E3 = e1 - e3;
    C O0 = o0 + o2, O2 = mul_i<INV>(o0 - o2), O1 = o1 + o3, O3 = o1 - o3;
    O1 = h * (O1 + mul_i<INV>(O1));
    O3 = h * (mul_i<INV>(O3) - O3);
    v[0] = E0 + O0;
    v[1] = E1 + O1;
    v[2] = E2 + O2;
    v[3] = E3 + O3;
    v[4] = E0 - O0;
    if (!NOUT) {
        v[5] = E1 - O1;
        v[6] = E2 - O2;
        v[7] = E3 - O3;
    }
}
template <typename S, bool INV, int N>
struct P<S, 8, INV, N> {
    using C = cx<S>;
    static __device__ __forceinline__ void run(C (&v)[8], const C *) { dft8<S, INV, false, false>(v); }
};
// R = A B, coprime: n = (B n1 + A n2) mod R, k = (B (1/B mod A) k1 + A (1/A mod B) k2) mod R.
constexpr int inv_mod(int x, int m) {
    for (int i = 1; i < m; ++i)
        if ((x % m) * i % m == 1) return i;
    return 1;
}
template <typename S, int A, int B, bool INV, int N>
__device__ __forceinline__ void pfa(cx<S> (&v)[A * B], const cx<S> *tw) {
    using C = cx<S>;
    constexpr int R = A * B, qa = B * inv_mod(B, A), qb = A * inv_mod(A, B);
    C t[R];   // [n1][k2]
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
        C u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = v[(B * n1 + A * n2) % R];
        P<S, B, INV, N>::run(u, tw);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) t[n1 * B + k2] = u[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        C u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1 * B + k2];
        P<S, A, INV, N>::run(u, tw);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[(qa * k1 + qb * k2) % R] = u[k1];
    }
}
// R = A B by Cooley and Tukey, inner twiddles W_R^{n1 k2} from the table.
template <typename S, int A, int B, bool INV, int N>
__device__ __forceinline__ void ct(cx<S> (&v)[A * B], const cx<S> *tw) {
    using C = cx<S>;
    constexpr int R = A * B;
    C t[R];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
        C u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = v[n1 + A * n2];
        P<S, B, INV, N>::run(u, tw);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) t[n1 * B + k2] = n1 * k2 ? twid<INV>(u[k2], tw[n1 * k2 * (N / R)]) : u[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        C u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1 * B + k2];
        P<S, A, INV, N>::run(u, tw);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[k2 + B * k1] = u[k1];
    }
}
#define LG_FFT2_P(R, expr)                                                                         \
    template <typename S, bool INV, int N>                                                         \
    struct P<S, R, INV, N> {                                                                       \
        static __device__ __forceinline__ void run(cx<S> (&v)[R], const cx<S> *tw) { expr; }       \
    };
LG_FFT2_P(6, (pfa<S, 2, 3, INV, N>(v, tw)))
LG_FFT2_P(9, (ct<S, 3, 3, INV, N>(v, tw)))
LG_FFT2_P(10, (pfa<S, 2, 5, INV, N>(v, tw)))
LG_FFT2_P(12, (pfa<S, 3, 4, INV, N>(v, tw)))
LG_FFT2_P(15, (pfa<S, 3, 5, INV, N>(v, tw)))
LG_FFT2_P(16, (ct<S, 4, 4, INV, N>(v, tw)))
#undef LG_FFT2_P

// The R1-point step: HALF: inputs (inverse) beyond R1 / 2 are zero, outputs (forward) beyond it unneeded.
template <typename S, int R1, bool INV, int N, bool HALF>
__device__ __forceinline__ void step1(cx<S> (&v)[R1], const cx<S> *tw) {
    if constexpr (R1 == 8 && HALF) dft8<S, INV, INV, !INV>(v);
    else P<S, R1, INV, N>::run(v, tw);
}

// Blocks: FP32 lines are half as long in bytes and registers, so pass B takes a warp's width of lines (twiddle
// reads are then broadcasts) and the plane passes share an SM in pairs.
template <typename S>
struct Shape {
    static constexpr bool F32 = std::is_same<S, float>::value;
    static constexpr int LB = F32 ? 32 : 16;   // lines per block of pass B
    static constexpr int LP = LB + 1;          // entries between positions of the line buffer (bank spread)
    static constexpr int NB = F32 ? 6 : 4;     // blocks of pass B an SM: one's barriers overlap the others' work
    static constexpr int NP = F32 ? 2 : 1;     // blocks of the plane passes, as many as their tile leaves room for
};
constexpr int TH = 128;   // threads of pass B
constexpr int TP = 512;   // threads of the plane passes

template <int N, typename S, typename R>
__device__ __forceinline__ void load_tw(cx<S> *tw, const cx<R> *__restrict__ twg) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = mkc<S>((S)twg[i].x, (S)twg[i].y);
}

// ------------------------------------------------------------- pass B
template <typename S, typename R, int N, int R1, bool HALF>
__global__ void __launch_bounds__(TH, Shape<S>::NB)
k_2b(cx<S> *__restrict__ T2, int Px, const S *__restrict__ vt, const cx<R> *__restrict__ twg) {
    using C = cx<S>;
    constexpr int R2 = N / R1;
    constexpr int LB = Shape<S>::LB, LP = Shape<S>::LP;
    __shared__ C tw[N];
    __shared__ C L[N * LP];
    const int y0 = blockIdx.x * LB, z = blockIdx.y;
    const size_t NN = (size_t)N * N;
    C *base = T2 + (size_t)blockIdx.z * Px * NN + (size_t)z * N + y0;
    const C zero = mkc<S>(S(0), S(0));
    const int ny = min(LB, N - y0);
    load_tw<N>(tw, twg);
    __syncthreads();
    for (int it = threadIdx.x; it < R2 * LB; it += TH) {
        const int l = it % LB, a = it / LB;
        if (l >= ny) continue;
        C v[R1];
#pragma unroll
        for (int b = 0; b < R1; ++b) {
            const int px = a + R2 * b;
            v[b] = (HALF && b > R1 / 2) ? zero : px < Px ? base[(size_t)px * NN + l] : zero;
        }
        step1<S, R1, true, N, HALF>(v, tw);
#pragma unroll
        for (int k = 0; k < R1; ++k) L[(a + R2 * k) * LP + l] = k ? cmulc(v[k], tw[a * k]) : v[k];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R1 * LB; it += TH) {
        const int l = it % LB, k1 = it / LB;
        if (l >= ny) continue;
        const S *vx = vt + (size_t)z * NN + y0 + l;   // [z][x][y]
        C v[R2];
#pragma unroll
        for (int a = 0; a < R2; ++a) v[a] = L[(a + R2 * k1) * LP + l];
        P<S, R2, true, N>::run(v, tw);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[k2] = vx[(size_t)(k1 + R1 * k2) * N] * v[k2];
        P<S, R2, false, N>::run(v, tw);
#pragma unroll
        for (int a = 0; a < R2; ++a) L[(a + R2 * k1) * LP + l] = a ? cmul(v[a], tw[a * k1]) : v[a];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R2 * LB; it += TH) {
        const int l = it % LB, a = it / LB;
        if (l >= ny) continue;
        C v[R1];
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = L[(a + R2 * k) * LP + l];
        step1<S, R1, false, N, HALF>(v, tw);
#pragma unroll
        for (int b = 0; b < R1; ++b) {
            const int px = a + R2 * b;
            if (!(HALF && b > R1 / 2) && px < Px) base[(size_t)px * NN + l] = v[b];
        }
    }
}

// ------------------------------------------------------------- pass A
// One block per (band, x-plane).  Tile A[z][py] (pitch P1, odd).  After the z-FFT, slot k2 + R2 k1 of a row
// holds z = k1 + R1 k2.  Dynamic shared memory: tw, tile, line buffer.
template <typename S, typename R, int N, int R1, bool HALF>
__global__ void __launch_bounds__(TP, Shape<S>::NP)
k_2a(const cx<R> *__restrict__ X, int ldx, cx<S> *__restrict__ T2, int Px, int Py, const int *__restrict__ plane_begin,
     const int2 *__restrict__ yrange, const int *__restrict__ gmap, const cx<R> *__restrict__ twg, int lbs) {
    using C = cx<S>;
    constexpr int R2 = N / R1;
    const int LB = 1 << lbs, LP = LB | 1;   // lines of a chunk
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = Py | 1;
    C *tw = reinterpret_cast<C *>(smem_raw), *A = tw + N, *L = A + (size_t)N * P1;
    const int px = blockIdx.x, bd = blockIdx.y;
    const cx<R> *Xb = X + (size_t)bd * ldx;
    const C zero = mkc<S>(S(0), S(0));
    load_tw<N>(tw, twg);
    for (int i = threadIdx.x; i < N * P1; i += TP) A[i] = zero;
    __syncthreads();
    const int g1 = plane_begin[px + 1];
    for (int g = plane_begin[px] + threadIdx.x; g < g1; g += TP) {
        const int m = gmap[g], py = m / N, iz = m - py * N;
        const cx<R> x = Xb[g];
        A[iz * P1 + py] = mkc<S>((S)x.x, (S)x.y);
    }
    __syncthreads();
    const int2 yr = yrange[px];
    const int rows = yr.y - yr.x + 1;
    for (int it = threadIdx.x; it < R2 * rows; it += TP) {
        const int py = yr.x + it % rows, a = it / rows;
        C v[R1];
#pragma unroll
        for (int b = 0; b < R1; ++b) v[b] = A[(a + R2 * b) * P1 + py];
        P<S, R1, true, N>::run(v, tw);
#pragma unroll
        for (int k = 0; k < R1; ++k) A[(a + R2 * k) * P1 + py] = k ? cmulc(v[k], tw[a * k]) : v[k];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R1 * rows; it += TP) {
        const int py = yr.x + it % rows, k1 = it / rows;
        C v[R2];
#pragma unroll
        for (int a = 0; a < R2; ++a) v[a] = A[(a + R2 * k1) * P1 + py];
        P<S, R2, true, N>::run(v, tw);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) A[(k2 + R2 * k1) * P1 + py] = v[k2];
    }
    __syncthreads();
    C *out = T2 + ((size_t)bd * Px + px) * (size_t)N * N;   // [z][y]
    for (int s0 = 0; s0 < N; s0 += LB) {                     // LB slots of the tile at a time
        const int nl = min(LB, N - s0);
        for (int it = threadIdx.x; it < R2 * LB; it += TP) {
            const int l = it & (LB - 1), a = it >> lbs;
            if (l >= nl) continue;
            C v[R1];
#pragma unroll
            for (int b = 0; b < R1; ++b) {
                const int py = a + R2 * b;
                v[b] = (HALF && b > R1 / 2) ? zero : py < Py ? A[(s0 + l) * P1 + py] : zero;
            }
            step1<S, R1, true, N, HALF>(v, tw);
#pragma unroll
            for (int k = 0; k < R1; ++k) L[(a + R2 * k) * LP + l] = k ? cmulc(v[k], tw[a * k]) : v[k];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < R1 * LB; it += TP) {   // neighbouring threads on neighbouring y
            const int k1 = it % R1, l = it / R1;
            if (l >= nl) continue;
            const int sl = s0 + l, z = sl / R2 + R1 * (sl % R2);
            C v[R2];
#pragma unroll
            for (int a = 0; a < R2; ++a) v[a] = L[(a + R2 * k1) * LP + l];
            P<S, R2, true, N>::run(v, tw);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) out[(size_t)z * N + k1 + R1 * k2] = v[k2];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------- pass C
// One block per (band, x-plane), pass A backwards: slot b + R1 a of a row holds the z coefficient a + R2 b.
template <typename S, typename R, int N, int R1, bool HALF>
__global__ void __launch_bounds__(TP, Shape<S>::NP)
k_2c(const cx<S> *__restrict__ T2, cx<R> *__restrict__ Y, int ldy, const cx<R> *__restrict__ X, int ldx,
     const R *__restrict__ kin, int Px, int Py, const int *__restrict__ plane_begin,
     const int2 *__restrict__ yrange, const int *__restrict__ gmap, const cx<R> *__restrict__ twg, int lbs) {
    using C = cx<S>;
    constexpr int R2 = N / R1;
    const int LB = 1 << lbs, LP = LB | 1;   // lines of a chunk
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = Py | 1;
    C *tw = reinterpret_cast<C *>(smem_raw), *A = tw + N, *L = A + (size_t)N * P1;
    const int px = blockIdx.x, bd = blockIdx.y;
    load_tw<N>(tw, twg);
    __syncthreads();
    const C *in = T2 + ((size_t)bd * Px + px) * (size_t)N * N;   // [z][y]
    for (int z0 = 0; z0 < N; z0 += LB) {
        const int nl = min(LB, N - z0);
        for (int it = threadIdx.x; it < R1 * LB; it += TP) {
            const int k1 = it % R1, l = it / R1;
            if (l >= nl) continue;
            C v[R2];
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) v[k2] = in[(size_t)(z0 + l) * N + k1 + R1 * k2];
            P<S, R2, false, N>::run(v, tw);
#pragma unroll
            for (int a = 0; a < R2; ++a) L[(a + R2 * k1) * LP + l] = a ? cmul(v[a], tw[a * k1]) : v[a];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < R2 * LB; it += TP) {
            const int l = it & (LB - 1), a = it >> lbs;
            if (l >= nl) continue;
            C v[R1];
#pragma unroll
            for (int k = 0; k < R1; ++k) v[k] = L[(a + R2 * k) * LP + l];
            step1<S, R1, false, N, HALF>(v, tw);
#pragma unroll
            for (int b = 0; b < R1; ++b) {
                const int py = a + R2 * b;
                if (!(HALF && b > R1 / 2) && py < Py) A[(z0 + l) * P1 + py] = v[b];
            }
        }
        __syncthreads();
    }
    const int2 yr = yrange[px];
    const int rows = yr.y - yr.x + 1;
    for (int it = threadIdx.x; it < R1 * rows; it += TP) {
        const int py = yr.x + it % rows, k1 = it / rows;
        C v[R2];
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[k2] = A[(k1 + R1 * k2) * P1 + py];
        P<S, R2, false, N>::run(v, tw);
#pragma unroll
        for (int a = 0; a < R2; ++a) A[(k1 + R1 * a) * P1 + py] = a ? cmul(v[a], tw[a * k1]) : v[a];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R2 * rows; it += TP) {
        const int py = yr.x + it % rows, a = it / rows;
        C v[R1];
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = A[(k + R1 * a) * P1 + py];
        P<S, R1, false, N>::run(v, tw);
#pragma unroll
        for (int b = 0; b < R1; ++b) A[(b + R1 * a) * P1 + py] = v[b];
    }
    __syncthreads();
    cx<R> *Yb = Y + (size_t)bd * ldy;
    const cx<R> *Xb = X + (size_t)bd * ldx;
    const int g1 = plane_begin[px + 1];
    for (int g = plane_begin[px] + threadIdx.x; g < g1; g += TP) {
        const int m = gmap[g], py = m / N, iz = m - py * N;
        C v = A[(iz / R2 + R1 * (iz % R2)) * P1 + py];
        if (kin) {
            const S t = (S)kin[g];
            const cx<R> x = Xb[g];
            v = v + t * mkc<S>((S)x.x, (S)x.y);
        }
        Yb[g] = mkc<R>((R)v.x, (R)v.y);
    }
}

// Lines of a chunk of the plane passes (a power of two, its logarithm) for the shared memory at hand; -1: the
// plane tile does not fit.
template <typename S>
int chunk_log2(const FFTGeom &g, int smem_max) {
    for (int l = 5; l >= 1; --l)
        if (sizeof(cx<S>) * (size_t)g.N * (1 + (g.Py | 1) + ((1 << l) | 1)) <= (size_t)smem_max) return l;
    return -1;
}

// 1: the geometry does not fit (the caller's general passes take it).
template <typename S, typename R, int N, int R1>
int run(const Fft2Args<S, R> &a) {
    const FFTGeom &g = *a.g;
    const int lbs = chunk_log2<S>(g, a.smem_max);
    if (lbs < 0) return 1;
    const size_t sm = sizeof(cx<S>) * (size_t)N * (1 + (g.Py | 1) + ((1 << lbs) | 1));
    const bool half = g.Px <= N / 2 + 1 && g.Py <= N / 2 + 1;
    static DeviceOnce attr;
    const int dev = current_device();
    if (!attr.done(dev)) {
        const void *fns[] = {(const void *)k_2a<S, R, N, R1, true>, (const void *)k_2c<S, R, N, R1, true>,
                             (const void *)k_2a<S, R, N, R1, false>, (const void *)k_2c<S, R, N, R1, false>};
        for (const void *f : fns)
            LG_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, a.smem_max));
        attr.mark(dev);
    }
    auto passes = [&](auto ka, auto kb, auto kc) -> int {
        for (int b0 = 0; b0 < a.nb; b0 += a.nbatch) {
            const int nbb = std::min(a.nbatch, a.nb - b0);
            const cx<R> *Xb = a.X + (size_t)b0 * a.ldx;
            cx<R> *Yb = a.Y + (size_t)b0 * a.ldy;
            ka<<<dim3(g.Px, nbb), TP, sm, a.s>>>(Xb, a.ldx, a.T2, g.Px, g.Py, g.plane_begin, g.plane_yrange, g.gmap, a.tw, lbs);
            LG_TRY(check_launch("fft pass A (two-step)"));
            kb<<<dim3((N + Shape<S>::LB - 1) / Shape<S>::LB, N, nbb), TH, 0, a.s>>>(a.T2, g.Px, a.vt, a.tw);
            LG_TRY(check_launch("fft pass B (two-step)"));
            kc<<<dim3(g.Px, nbb), TP, sm, a.s>>>(a.T2, Yb, a.ldy, Xb, a.ldx, a.kin, g.Px, g.Py, g.plane_begin,
                                                g.plane_yrange, g.gmap, a.tw, lbs);
            LG_TRY(check_launch("fft pass C (two-step)"));
        }
        return LOBPCG_OK;
    };
    if (half) return passes(k_2a<S, R, N, R1, true>, k_2b<S, R, N, R1, true>, k_2c<S, R, N, R1, true>);
    return passes(k_2a<S, R, N, R1, false>, k_2b<S, R, N, R1, false>, k_2c<S, R, N, R1, false>);
}

}  // namespace f2s
}  // namespace lg
