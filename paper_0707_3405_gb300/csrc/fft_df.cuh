// Double-FP32 passes of the local potential (Sec. 4.1: Goedecker's zero-padded FFT) for grid edges
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
// B 675 -> 295, C 288 -> 155; H on 128 bands with 432 projectors 20.7 -> 12.1 ms.
#pragma once

#include "common.cuh"
#include "df64.cuh"

#include <algorithm>
#include <atomic>

namespace lg {
namespace fdf {

using D = df64f;
using C = cx<df64f>;

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
__device__ __forceinline__ C cmul(C a, C w) { return mkc<D>(dot2(a.x, w.x, -a.y, w.y), dot2(a.x, w.y, a.y, w.x)); }
// a conj(w)
__device__ __forceinline__ C cmulc(C a, C w) { return mkc<D>(dot2(a.x, w.x, a.y, w.y), dot2(a.y, w.x, -a.x, w.y)); }
__device__ __forceinline__ D half(D a) { return D(0.5f * a.hi, 0.5f * a.lo); }
template <bool INV>
__device__ __forceinline__ C mul_i(C a) { return INV ? mkc<D>(-a.y, a.x) : mkc<D>(a.y, -a.x); }
template <bool INV>
__device__ __forceinline__ C twid(C a, C w) { return INV ? cmulc(a, w) : cmul(a, w); }   // w = W_N^j (forward)

// ------------------------------------------------------------- small transforms in registers
// P<R, INV>::run(v, tw): v <- DFT_R v; tw: the N-entry table, TS = N / R its stride for W_R.
template <int R, bool INV, int N>
struct P;
template <bool INV, int N>
struct P<1, INV, N> {
    static __device__ __forceinline__ void run(C (&)[1], const C *) {}
};
template <bool INV, int N>
struct P<2, INV, N> {
    static __device__ __forceinline__ void run(C (&v)[2], const C *) {
        const C a = v[0], b = v[1];
        v[0] = a + b;
        v[1] = a - b;
    }
};
template <bool INV, int N>
struct P<3, INV, N> {
    static __device__ __forceinline__ void run(C (&v)[3], const C *) {
        const D s3 = (D)0.86602540378443864676;   // sin(2 pi / 3)
        const C a = v[0], t1 = v[1] + v[2], t2 = mkc<D>(a.x - half(t1.x), a.y - half(t1.y));
        const C t3 = s3 * mul_i<INV>(v[1] - v[2]);
        v[0] = a + t1;
        v[1] = t2 + t3;
        v[2] = t2 - t3;
    }
};
template <bool INV, int N>
struct P<4, INV, N> {
    static __device__ __forceinline__ void run(C (&v)[4], const C *) {
        const C t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], t3 = mul_i<INV>(v[1] - v[3]);
        v[0] = t0 + t2;
        v[2] = t0 - t2;
        v[1] = t1 + t3;
        v[3] = t1 - t3;
    }
};
template <bool INV, int N>
struct P<5, INV, N> {
    static __device__ __forceinline__ void run(C (&v)[5], const C *) {
        const D c1 = (D)0.30901699437494742410, c2 = (D)-0.80901699437494742410;   // cos(2 pi / 5), cos(4 pi / 5)
        const D s1 = (D)0.95105651629515357212, s2 = (D)0.58778525229247312917;    // sin(2 pi / 5), sin(4 pi / 5)
        const C a = v[0], p = v[1] + v[4], q = v[2] + v[3];
        const C m = mul_i<INV>(v[1] - v[4]), k = mul_i<INV>(v[2] - v[3]);
        const C r1 = mkc<D>(dot2_add(a.x, c1, p.x, c2, q.x), dot2_add(a.y, c1, p.y, c2, q.y));
        const C r2 = mkc<D>(dot2_add(a.x, c2, p.x, c1, q.x), dot2_add(a.y, c2, p.y, c1, q.y));
        const C i1 = mkc<D>(dot2(s1, m.x, s2, k.x), dot2(s1, m.y, s2, k.y));
        const C i2 = mkc<D>(dot2(s2, m.x, -s1, k.x), dot2(s2, m.y, -s1, k.y));
        v[0] = a + p + q;
        v[1] = r1 + i1;
        v[4] = r1 - i1;
        v[2] = r2 + i2;
        v[3] = r2 - i2;
    }
};
// 8 points; ZIN: v[5..7] are zero; NOUT: outputs 5..7 are not needed.
template <bool INV, bool ZIN, bool NOUT>
__device__ __forceinline__ void dft8(C (&v)[8]) {
    const D h = (D)0.70710678118654752440;   // 1 / sqrt(2)
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
template <bool INV, int N>
struct P<8, INV, N> {
    static __device__ __forceinline__ void run(C (&v)[8], const C *) { dft8<INV, false, false>(v); }
};
// R = A B, coprime: n = (B n1 + A n2) mod R, k = (B (1/B mod A) k1 + A (1/A mod B) k2) mod R.
constexpr int inv_mod(int x, int m) {
    for (int i = 1; i < m; ++i)
        if ((x % m) * i % m == 1) return i;
    return 1;
}
template <int A, int B, bool INV, int N>
__device__ __forceinline__ void pfa(C (&v)[A * B], const C *tw) {
    constexpr int R = A * B, qa = B * inv_mod(B, A), qb = A * inv_mod(A, B);
    C t[R];   // [n1][k2]
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
        C u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = v[(B * n1 + A * n2) % R];
        P<B, INV, N>::run(u, tw);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) t[n1 * B + k2] = u[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        C u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1 * B + k2];
        P<A, INV, N>::run(u, tw);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[(qa * k1 + qb * k2) % R] = u[k1];
    }
}
// R = A B by Cooley and Tukey, inner twiddles W_R^{n1 k2} from the table.
template <int A, int B, bool INV, int N>
__device__ __forceinline__ void ct(C (&v)[A * B], const C *tw) {
    constexpr int R = A * B;
    C t[R];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
        C u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = v[n1 + A * n2];
        P<B, INV, N>::run(u, tw);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) t[n1 * B + k2] = n1 * k2 ? twid<INV>(u[k2], tw[n1 * k2 * (N / R)]) : u[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        C u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1 * B + k2];
        P<A, INV, N>::run(u, tw);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[k2 + B * k1] = u[k1];
    }
}
#define LG_FDF_P(R, expr)                                                                             \
    template <bool INV, int N>                                                                        \
    struct P<R, INV, N> {                                                                             \
        static __device__ __forceinline__ void run(C (&v)[R], const C *tw) { expr; }                 \
    };
LG_FDF_P(6, (pfa<2, 3, INV, N>(v, tw)))
LG_FDF_P(9, (ct<3, 3, INV, N>(v, tw)))
LG_FDF_P(10, (pfa<2, 5, INV, N>(v, tw)))
LG_FDF_P(12, (pfa<3, 4, INV, N>(v, tw)))
LG_FDF_P(15, (pfa<3, 5, INV, N>(v, tw)))
LG_FDF_P(16, (ct<4, 4, INV, N>(v, tw)))
#undef LG_FDF_P

// The R1-point step: HALF: inputs (inverse) beyond R1 / 2 are zero, outputs (forward) beyond it unneeded.
template <int R1, bool INV, int N, bool HALF>
__device__ __forceinline__ void step1(C (&v)[R1], const C *tw) {
    if constexpr (R1 == 8 && HALF) dft8<INV, INV, !INV>(v);
    else P<R1, INV, N>::run(v, tw);
}

constexpr int LB = 16;    // lines per block of pass B
constexpr int LP = 17;    // entries between positions of the line buffer (bank spread)
constexpr int TH = 128;   // threads of pass B: four blocks an SM, so that one's barriers overlap the others' work
constexpr int TP = 512;   // threads of the plane passes, whose tile leaves room for one block

template <int N>
__device__ __forceinline__ void load_tw(C *tw, const z64 *__restrict__ twg) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = mkc<D>((D)twg[i].x, (D)twg[i].y);
}

// ------------------------------------------------------------- pass B
template <int N, int R1, bool HALF>
__global__ void __launch_bounds__(TH, 4)
k_db(C *__restrict__ T2, int Px, const D *__restrict__ vt, const z64 *__restrict__ twg) {
    constexpr int R2 = N / R1;
    __shared__ C tw[N];
    __shared__ C S[N * LP];
    const int y0 = blockIdx.x * LB, z = blockIdx.y;
    const size_t NN = (size_t)N * N;
    C *base = T2 + (size_t)blockIdx.z * Px * NN + (size_t)z * N + y0;
    const C zero = mkc<D>(D(0), D(0));
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
        step1<R1, true, N, HALF>(v, tw);
#pragma unroll
        for (int k = 0; k < R1; ++k) S[(a + R2 * k) * LP + l] = k ? cmulc(v[k], tw[a * k]) : v[k];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R1 * LB; it += TH) {
        const int l = it % LB, k1 = it / LB;
        if (l >= ny) continue;
        const D *vx = vt + (size_t)z * NN + y0 + l;   // [z][x][y]
        C v[R2];
#pragma unroll
        for (int a = 0; a < R2; ++a) v[a] = S[(a + R2 * k1) * LP + l];
        P<R2, true, N>::run(v, tw);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[k2] = vx[(size_t)(k1 + R1 * k2) * N] * v[k2];
        P<R2, false, N>::run(v, tw);
#pragma unroll
        for (int a = 0; a < R2; ++a) S[(a + R2 * k1) * LP + l] = a ? cmul(v[a], tw[a * k1]) : v[a];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R2 * LB; it += TH) {
        const int l = it % LB, a = it / LB;
        if (l >= ny) continue;
        C v[R1];
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = S[(a + R2 * k) * LP + l];
        step1<R1, false, N, HALF>(v, tw);
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
template <int N, int R1, bool HALF>
__global__ void __launch_bounds__(TP, 1)
k_da(const z64 *__restrict__ X, int ldx, C *__restrict__ T2, int Px, int Py, const int *__restrict__ plane_begin,
     const int2 *__restrict__ yrange, const int *__restrict__ gmap, const z64 *__restrict__ twg, int lbs) {
    constexpr int R2 = N / R1;
    const int LB = 1 << lbs, LP = LB | 1;   // lines of a chunk
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = Py | 1;
    C *tw = reinterpret_cast<C *>(smem_raw), *A = tw + N, *S = A + (size_t)N * P1;
    const int px = blockIdx.x, bd = blockIdx.y;
    const z64 *Xb = X + (size_t)bd * ldx;
    const C zero = mkc<D>(D(0), D(0));
    load_tw<N>(tw, twg);
    for (int i = threadIdx.x; i < N * P1; i += TP) A[i] = zero;
    __syncthreads();
    const int g1 = plane_begin[px + 1];
    for (int g = plane_begin[px] + threadIdx.x; g < g1; g += TP) {
        const int m = gmap[g], py = m / N, iz = m - py * N;
        const z64 x = Xb[g];
        A[iz * P1 + py] = mkc<D>((D)x.x, (D)x.y);
    }
    __syncthreads();
    const int2 yr = yrange[px];
    const int rows = yr.y - yr.x + 1;
    for (int it = threadIdx.x; it < R2 * rows; it += TP) {
        const int py = yr.x + it % rows, a = it / rows;
        C v[R1];
#pragma unroll
        for (int b = 0; b < R1; ++b) v[b] = A[(a + R2 * b) * P1 + py];
        P<R1, true, N>::run(v, tw);
#pragma unroll
        for (int k = 0; k < R1; ++k) A[(a + R2 * k) * P1 + py] = k ? cmulc(v[k], tw[a * k]) : v[k];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R1 * rows; it += TP) {
        const int py = yr.x + it % rows, k1 = it / rows;
        C v[R2];
#pragma unroll
        for (int a = 0; a < R2; ++a) v[a] = A[(a + R2 * k1) * P1 + py];
        P<R2, true, N>::run(v, tw);
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
            step1<R1, true, N, HALF>(v, tw);
#pragma unroll
            for (int k = 0; k < R1; ++k) S[(a + R2 * k) * LP + l] = k ? cmulc(v[k], tw[a * k]) : v[k];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < R1 * LB; it += TP) {   // neighbouring threads on neighbouring y
            const int k1 = it % R1, l = it / R1;
            if (l >= nl) continue;
            const int sl = s0 + l, z = sl / R2 + R1 * (sl % R2);
            C v[R2];
#pragma unroll
            for (int a = 0; a < R2; ++a) v[a] = S[(a + R2 * k1) * LP + l];
            P<R2, true, N>::run(v, tw);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) out[(size_t)z * N + k1 + R1 * k2] = v[k2];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------- pass C
// One block per (band, x-plane), pass A backwards: slot b + R1 a of a row holds the z coefficient a + R2 b.
template <int N, int R1, bool HALF>
__global__ void __launch_bounds__(TP, 1)
k_dc(const C *__restrict__ T2, z64 *__restrict__ Y, int ldy, const z64 *__restrict__ X, int ldx,
     const double *__restrict__ kin, int Px, int Py, const int *__restrict__ plane_begin,
     const int2 *__restrict__ yrange, const int *__restrict__ gmap, const z64 *__restrict__ twg, int lbs) {
    constexpr int R2 = N / R1;
    const int LB = 1 << lbs, LP = LB | 1;   // lines of a chunk
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = Py | 1;
    C *tw = reinterpret_cast<C *>(smem_raw), *A = tw + N, *S = A + (size_t)N * P1;
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
            P<R2, false, N>::run(v, tw);
#pragma unroll
            for (int a = 0; a < R2; ++a) S[(a + R2 * k1) * LP + l] = a ? cmul(v[a], tw[a * k1]) : v[a];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < R2 * LB; it += TP) {
            const int l = it & (LB - 1), a = it >> lbs;
            if (l >= nl) continue;
            C v[R1];
#pragma unroll
            for (int k = 0; k < R1; ++k) v[k] = S[(a + R2 * k) * LP + l];
            step1<R1, false, N, HALF>(v, tw);
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
        P<R2, false, N>::run(v, tw);
#pragma unroll
        for (int a = 0; a < R2; ++a) A[(k1 + R1 * a) * P1 + py] = a ? cmul(v[a], tw[a * k1]) : v[a];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < R2 * rows; it += TP) {
        const int py = yr.x + it % rows, a = it / rows;
        C v[R1];
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = A[(k + R1 * a) * P1 + py];
        P<R1, false, N>::run(v, tw);
#pragma unroll
        for (int b = 0; b < R1; ++b) A[(b + R1 * a) * P1 + py] = v[b];
    }
    __syncthreads();
    z64 *Yb = Y + (size_t)bd * ldy;
    const z64 *Xb = X + (size_t)bd * ldx;
    const int g1 = plane_begin[px + 1];
    for (int g = plane_begin[px] + threadIdx.x; g < g1; g += TP) {
        const int m = gmap[g], py = m / N, iz = m - py * N;
        C v = A[(iz / R2 + R1 * (iz % R2)) * P1 + py];
        if (kin) {
            const D t = (D)kin[g];
            const z64 x = Xb[g];
            v = v + t * mkc<D>((D)x.x, (D)x.y);
        }
        Yb[g] = mkc((double)v.x, (double)v.y);
    }
}

// Lines of a chunk of the plane passes (a power of two, its logarithm) for the shared memory at hand; -1: the
// plane tile does not fit.
inline int chunk_log2(const FFTGeom &g, int smem_max) {
    for (int l = 5; l >= 1; --l)
        if (sizeof(C) * (size_t)g.N * (1 + (g.Py | 1) + ((1 << l) | 1)) <= (size_t)smem_max) return l;
    return -1;
}

// 1: the geometry does not fit (the caller's general passes take it).
template <int N, int R1>
int run(const FFTGeom &g, const z64 *X, int ldx, z64 *Y, int ldy, int nb, const double *kin, const D *vt, const z64 *tw,
        C *T2, int nbatch, int smem_max, cudaStream_t s) {
    const int lbs = chunk_log2(g, smem_max);
    if (lbs < 0) return 1;
    const size_t sm = sizeof(C) * (size_t)N * (1 + (g.Py | 1) + ((1 << lbs) | 1));
    const bool half = g.Px <= N / 2 + 1 && g.Py <= N / 2 + 1;
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        LG_CUDA_TRY(cudaFuncSetAttribute(k_da<N, R1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
        LG_CUDA_TRY(cudaFuncSetAttribute(k_dc<N, R1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
        LG_CUDA_TRY(cudaFuncSetAttribute(k_da<N, R1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
        LG_CUDA_TRY(cudaFuncSetAttribute(k_dc<N, R1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
        attr.store(true);
    }
    auto passes = [&](auto ka, auto kb, auto kc) -> int {
        for (int b0 = 0; b0 < nb; b0 += nbatch) {
            const int nbb = std::min(nbatch, nb - b0);
            const z64 *Xb = X + (size_t)b0 * ldx;
            z64 *Yb = Y + (size_t)b0 * ldy;
            ka<<<dim3(g.Px, nbb), TP, sm, s>>>(Xb, ldx, T2, g.Px, g.Py, g.plane_begin, g.plane_yrange, g.gmap, tw, lbs);
            LG_TRY(check_launch("fft pass A (double-FP32)"));
            kb<<<dim3((N + LB - 1) / LB, N, nbb), TH, 0, s>>>(T2, g.Px, vt, tw);
            LG_TRY(check_launch("fft pass B (double-FP32)"));
            kc<<<dim3(g.Px, nbb), TP, sm, s>>>(T2, Yb, ldy, Xb, ldx, kin, g.Px, g.Py, g.plane_begin, g.plane_yrange,
                                              g.gmap, tw, lbs);
            LG_TRY(check_launch("fft pass C (double-FP32)"));
        }
        return LOBPCG_OK;
    };
    if (half) return passes(k_da<N, R1, true>, k_db<N, R1, true>, k_dc<N, R1, true>);
    return passes(k_da<N, R1, false>, k_db<N, R1, false>, k_dc<N, R1, false>);
}

}  // namespace fdf
}  // namespace lg
