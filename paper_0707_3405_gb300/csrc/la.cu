// FP64 Rayleigh-Ritz for block LOBPCG (Algorithm 1, step 4 of Bottin et al.
// 2007: "apply the Rayleigh-Ritz method within the subspace spanned by the
// columns of Psi, W and P"; the paper calls LAPACK for it, Sec. 4.2) and the
// all-band subspace diagonalisation that closes each sweep (Sec. 3.2).
//
// Given the Gram matrix S = Z^H Z and A = Z^H H Z of a basis Z (n x n):
//   1. scale to unit diagonal, S' = D S D, A' = D A D, D = diag(S)^-1/2;
//   2. blocked Cholesky S' = L L^H; a column whose pivot^2 is below drop_tol
//      is dependent on the earlier ones and is removed (its L column becomes
//      e_j, its L row is cleared), which turns the problem into plain RR on
//      the remaining columns;
//   3. Ahat = L^-1 A' L^-H (explicit blocked triangular inverse);
//   4. lowest m eigenpairs of Ahat: complex Householder tridiagonalisation
//      (reflectors in the LAPACK larfg convention, real sub-diagonal),
//      eigenvalues by multisection on Sturm counts (a warp per eigenvalue),
//      eigenvectors by inverse iteration with partial-pivoting tridiagonal
//      LU and modified Gram-Schmidt inside clusters of close eigenvalues,
//      back-transformation by the reflectors in blocks of 32 (compact WY form);
//   5. C = D L^-H Q.
// Every step runs on the GPU in FP64; no host synchronisation.
#include "common.cuh"
#include "df64.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

namespace lg {

namespace {

constexpr int NBK = 32;  // Cholesky / inverse block size

template <typename RT> struct Lim;
template <> struct Lim<double> {
    static __device__ __forceinline__ double eps() { return DBL_EPSILON; }
    static __device__ __forceinline__ double tiny() { return DBL_MIN; }
    static __device__ __forceinline__ double big() { return DBL_MAX; }
};
template <> struct Lim<float> {
    static __device__ __forceinline__ float eps() { return FLT_EPSILON; }
    static __device__ __forceinline__ float tiny() { return FLT_MIN; }
    static __device__ __forceinline__ float big() { return FLT_MAX; }
};
__device__ __forceinline__ z64 ldcg_cx(const z64 *p) {
    const double2 t = __ldcg(reinterpret_cast<const double2 *>(p));
    return mkc(t.x, t.y);
}
__device__ __forceinline__ c32 ldcg_cx(const c32 *p) {
    const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
    return mkc(t.x, t.y);
}
__device__ __forceinline__ cx<df64> ldcg_cx(const cx<df64> *p) {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
    return mkc(df64(t.x, t.y), df64(t.z, t.w));
}
// Load a complex stored as cx<PT> into the compute type CT.
template <typename CT, typename PT>
__device__ __forceinline__ cx<CT> ld_as(const cx<PT> *p) {
    if constexpr (std::is_same<CT, PT>::value) return *p;
    else return mkc<CT>((CT)p->x, (CT)p->y);
}
template <typename CT, typename PT>
__device__ __forceinline__ cx<CT> ldcg_as(const cx<PT> *p) {
    const cx<PT> v = ldcg_cx(p);
    if constexpr (std::is_same<CT, PT>::value) return v;
    else return mkc<CT>((CT)v.x, (CT)v.y);
}
template <typename PT, typename CT>
__device__ __forceinline__ cx<PT> as_store(cx<CT> v) {
    if constexpr (std::is_same<CT, PT>::value) return v;
    else return mkc<PT>((PT)v.x, (PT)v.y);
}


template <typename RT>
__device__ __forceinline__ RT warp_sum(RT v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic block sum (blockDim.x multiple of 32, <= 1024). Result on all threads.
template <typename RT>
__device__ RT block_sum(RT v, RT *sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    RT t = 0.0;
    for (int i = 0; i < nw; ++i) t += sh[i];
    return t;
}

// acc + a b
template <typename CT>
__device__ __forceinline__ cx<CT> cmac(cx<CT> acc, cx<CT> a, cx<CT> b) {
    CT re = fma(a.x, b.x, acc.x);
    re = fma(-a.y, b.y, re);
    CT im = fma(a.x, b.y, acc.y);
    im = fma(a.y, b.x, im);
    return mkc<CT>(re, im);
}

// ------------------------------------------------------------------ scaling
template <typename RT>
__global__ void k_scale_gram(int n, const cx<RT> *__restrict__ S, int lds, const cx<RT> *__restrict__ A, int lda,
                             cx<RT> *__restrict__ Ss, cx<RT> *__restrict__ As, RT *__restrict__ d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n) return;
    const RT si = S[(size_t)i * lds + i].x, sj = S[(size_t)j * lds + j].x;
    const RT di = si > 0.0 ? 1.0 / sqrt(si) : 0.0;
    const RT dj = sj > 0.0 ? 1.0 / sqrt(sj) : 0.0;
    if (j == 0) d[i] = di;
    cx<RT> s, a;
    if (i >= j) {
        s = S[(size_t)j * lds + i];
        a = A[(size_t)j * lda + i];
    } else {
        s = conjc(S[(size_t)i * lds + j]);
        a = conjc(A[(size_t)i * lda + j]);
    }
    if (i == j) { s.y = 0.0; a.y = 0.0; }
    Ss[(size_t)j * n + i] = (di * dj) * s;
    As[(size_t)j * n + i] = (di * dj) * a;
}

// ------------------------------------------------------------------ Cholesky with dropping
// Factor the kb x kb diagonal block at k0 (already updated by earlier panels),
// write L_kk over it and its inverse into Linv.
// (FP64 and FP32 arithmetic.  The FP64 schedule's steps on nearly dependent bases follow the exact
// roundings of this form; the elimination form below gained nothing there, the FP64 units bounding both.)
template <typename RT>
__global__ void __launch_bounds__(256)
k_chol_diag(int n, int k0, int kb, cx<RT> *__restrict__ L, cx<RT> *__restrict__ Linv, RT drop_tol,
            int *__restrict__ dropped, int *__restrict__ ndrop) {
    __shared__ cx<RT> T[NBK][NBK + 1];
    __shared__ cx<RT> I[NBK][NBK + 1];
    __shared__ int dflag[NBK];
    const int tid = threadIdx.x;
    for (int e = tid; e < NBK * NBK; e += blockDim.x) {
        const int r = e % NBK, c = e / NBK;
        cx<RT> v = mkc<RT>(0.0, 0.0);
        if (r < kb && c < kb && r >= c) v = L[(size_t)(k0 + c) * n + k0 + r];
        T[r][c] = v;
        I[r][c] = mkc<RT>(0.0, 0.0);
    }
    __syncthreads();
    for (int j = 0; j < kb; ++j) {
        const RT p = T[j][j].x;
        const bool drop = !(p > drop_tol);
        __syncthreads();
        if (drop) {
            for (int r = j + 1 + tid; r < kb; r += blockDim.x) T[r][j] = mkc<RT>(0.0, 0.0);
            if (tid == 0) { T[j][j] = mkc<RT>(1.0, 0.0); dflag[j] = 1; }
        } else {
            const RT rt = sqrt(p), inv = (RT)1.0 / rt;
            for (int r = j + 1 + tid; r < kb; r += blockDim.x) T[r][j] = inv * T[r][j];
            if (tid == 0) { T[j][j] = mkc<RT>(rt, 0.0); dflag[j] = 0; }
        }
        __syncthreads();
        if (!drop) {
            const int rem = kb - j - 1;
            for (int e = tid; e < rem * rem; e += blockDim.x) {
                const int r = j + 1 + e % rem, c = j + 1 + e / rem;
                if (r >= c) T[r][c] = T[r][c] - mul_conj(T[r][j], T[c][j]);
            }
        }
        __syncthreads();
    }
    // clear the rows of dropped columns inside the block
    for (int e = tid; e < kb * kb; e += blockDim.x) {
        const int r = e % kb, c = e / kb;
        if (c < r && dflag[r]) T[r][c] = mkc<RT>(0.0, 0.0);
    }
    __syncthreads();
    // inverse of the lower-triangular block (real positive diagonal) by forward substitution,
    // column c on the 8 lanes of one warp segment: I[r][c] = -(1 / T[r][r]) sum_{l=c}^{r-1} T[r][l] I[l][c],
    // each lane taking every 8th l, the segment adding its partial sums by shuffles (fixed order)
    __shared__ RT rdiag[NBK];
    if (tid < kb) rdiag[tid] = (RT)1.0 / T[tid][tid].x;
    __syncthreads();
    {
        const int c = tid >> 3, sub = tid & 7;
        const bool on = c < kb;
        for (int r = 0; r < kb; ++r) {
            cx<RT> sacc = mkc<RT>(0.0, 0.0);
            if (on && c < r)
                for (int l = c + sub; l < r; l += 8) sacc = sacc + T[r][l] * I[l][c];
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                sacc.x += __shfl_xor_sync(0xffffffffu, sacc.x, o);
                sacc.y += __shfl_xor_sync(0xffffffffu, sacc.y, o);
            }
            if (on && sub == 0) {
                if (c < r) I[r][c] = (-rdiag[r]) * sacc;
                else if (c == r) I[r][r] = mkc<RT>(rdiag[r], 0.0);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int e = tid; e < kb * kb; e += blockDim.x) {
        const int r = e % kb, c = e / kb;
        L[(size_t)(k0 + c) * n + k0 + r] = (r >= c) ? T[r][c] : mkc<RT>(0.0, 0.0);
        Linv[(size_t)(k0 + c) * n + k0 + r] = (r >= c) ? I[r][c] : mkc<RT>(0.0, 0.0);
    }
    if (tid < kb) {
        dropped[k0 + tid] = dflag[tid];
        if (dflag[tid]) atomicAdd(ndrop, 1);
    }
}

// The same in double-FP32 (one SM's FP64 units would be the limit).  Elimination in the form Lu D Lu^H with the identity beside it: column j's pivot p, m_r = T[r][j] / p, then
// T[r][c] -= m_r conj(T[c][j]) for j < c <= r and I[r][c] -= m_r I[j][c] for c <= j, so that the
// inverse of Lu grows in the same step.  A step is one division, one multiply-add and one block
// barrier; the square roots come once at the end, for all columns together (L = Lu D^1/2).  A chain
// of 32 steps is what bounds it: double-FP32 52 -> 31 us per block, against
// square root, column scaling, update and a separate forward substitution.
__global__ void __launch_bounds__(256)
k_chol_diag_df(int n, int k0, int kb, z64 *__restrict__ L, z64 *__restrict__ Linv, double drop_tol_in,
               int *__restrict__ dropped, int *__restrict__ ndrop) {
    using CT = df64;
    __shared__ cx<CT> T[NBK][NBK + 1];
    __shared__ cx<CT> I[NBK][NBK + 1];
    __shared__ CT rs[NBK];     // 1 / sqrt(pivot)
    __shared__ int dflag[NBK];
    const CT drop_tol = (CT)drop_tol_in;
    const int tid = threadIdx.x, r = tid & (NBK - 1), w = tid / NBK;   // a thread has row r, columns w, w + 8, ...
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < NBK / 8; ++k) {
        const int c = w + 8 * k;
        T[r][c] = (r < kb && r >= c) ? ld_as<CT>(L + (size_t)(k0 + c) * n + k0 + r) : zero;
        I[r][c] = mkc<CT>(r == c ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    for (int j = 0; j < kb; ++j) {
        const CT p = T[j][j].x;
        const bool drop = !(p > drop_tol);
        if (tid == 0) dflag[j] = drop;
        if (drop) {            // row and column j become those of the identity
            if (r == j)
                for (int c = w; c < j; c += 8) I[j][c] = zero;
        } else if (r > j && r < kb) {
            const cx<CT> mm = ((CT)-1.0 / p) * T[r][j];
#pragma unroll
            for (int k = 0; k < NBK / 8; ++k) {
                const int c = w + 8 * k;
                if (c > r) continue;
                cx<CT> *e = c > j ? &T[r][c] : &I[r][c];
                *e = cmac(*e, mm, c > j ? conjc(T[c][j]) : I[j][c]);
            }
        }
        __syncthreads();
    }
    if (tid < kb) {
        const CT p = T[tid][tid].x;
        rs[tid] = dflag[tid] ? CT(1.0) : (CT)1.0 / sqrt(p);
        dropped[k0 + tid] = dflag[tid];
        if (dflag[tid]) atomicAdd(ndrop, 1);
    }
    __syncthreads();
    if (r < kb)
#pragma unroll
        for (int k = 0; k < NBK / 8; ++k) {
            const int c = w + 8 * k;
            if (c >= kb) continue;
            cx<CT> l = zero, li = zero;
            if (r == c) {
                l = mkc<CT>(dflag[c] ? CT(1.0) : rs[c] * T[c][c].x, 0.0);
                li = mkc<CT>(rs[c], 0.0);
            } else if (r > c) {
                if (!dflag[r] && !dflag[c]) l = rs[c] * T[r][c];
                li = rs[r] * I[r][c];
            }
            L[(size_t)(k0 + c) * n + k0 + r] = as_store<double>(l);
            Linv[(size_t)(k0 + c) * n + k0 + r] = as_store<double>(li);
        }
}

// Panel: L21 = S21 Linv_kk^H for rows k0+kb..n-1 (kPanelRows rows per block, 32 columns).  FP64 throughput
// bounds it: four rows rather than eight per block spread it over twice the SMs (n = 384: 21 -> 13 us).
constexpr int kPanelRows = 4;
template <typename RT>
__global__ void __launch_bounds__(32 * kPanelRows)
k_chol_panel(int n, int k0, int kb, cx<RT> *__restrict__ L, const cx<RT> *__restrict__ Linv,
             const int *__restrict__ dropped) {
    __shared__ cx<RT> Di[NBK][NBK + 1];
    __shared__ cx<RT> Srow[kPanelRows][NBK + 1];
    const int tid = threadIdx.x;
    for (int e = tid; e < NBK * NBK; e += blockDim.x) {
        const int r = e % NBK, c = e / NBK;
        Di[r][c] = (r < kb && c < kb) ? Linv[(size_t)(k0 + c) * n + k0 + r] : mkc<RT>(0.0, 0.0);
    }
    const int rl = tid / NBK, c = tid % NBK;
    const int row = k0 + kb + blockIdx.x * kPanelRows + rl;
    if (row < n && c < kb) Srow[rl][c] = L[(size_t)(k0 + c) * n + row];
    __syncthreads();
    if (row < n && c < kb) {
        cx<RT> s = mkc<RT>(0.0, 0.0);
        for (int l = 0; l <= c; ++l) s = s + mul_conj(Srow[rl][l], Di[c][l]);
        if (dropped[k0 + c]) s = mkc<RT>(0.0, 0.0);
        L[(size_t)(k0 + c) * n + row] = s;
    }
}

// Leading identity block (a basis whose first `lead` vectors are orthonormal and orthogonal to the
// rest, as [X W P] of a mixed block iteration): its Cholesky factor and inverse are the identity.
template <typename RT>
__global__ void k_lead_identity(int n, int lead, cx<RT> *__restrict__ L, cx<RT> *__restrict__ Linv,
                                int *__restrict__ dropped) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= n) return;
    const cx<RT> v = mkc<RT>(i == j ? 1.0 : 0.0, 0.0);
    L[(size_t)j * n + i] = v;
    if (i < lead) Linv[(size_t)j * n + i] = v;
    if (i == 0) dropped[j] = 0;
}

template <typename RT>
__global__ void k_zero_dropped_rows(int n, cx<RT> *__restrict__ L, const int *__restrict__ dropped) {
    const int j = blockIdx.x;
    if (!dropped[j]) return;
    for (int c = threadIdx.x; c < j; c += blockDim.x) L[(size_t)c * n + j] = mkc<RT>(0.0, 0.0);
}

// ------------------------------------------------------------------ hermitize / dropped rows
template <typename RT>
__global__ void k_hermitize_rowsum(int n, cx<RT> *__restrict__ A, const int *__restrict__ dropped,
                                   RT *__restrict__ rowsum) {
    const int i = blockIdx.x;
    __shared__ RT sh[32];
    RT s = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        cx<RT> v = (i >= j) ? A[(size_t)j * n + i] : conjc(A[(size_t)i * n + j]);
        if (i == j) v.y = 0.0;
        if (dropped && (dropped[i] || dropped[j])) v = mkc<RT>(0.0, 0.0);
        s += sqrt(abs2(v));
        if (i >= j) {
            A[(size_t)j * n + i] = v;
            A[(size_t)i * n + j] = conjc(v);
        }
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) rowsum[i] = s;
}

template <typename RT>
__global__ void k_set_dropped_diag(int n, cx<RT> *__restrict__ A, const int *__restrict__ dropped,
                                   const int *__restrict__ ndrop, const RT *__restrict__ rowsum) {
    if (*ndrop == 0) return;
    __shared__ RT sh[32];
    RT mx = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) mx = fmax(mx, rowsum[i]);
    // deterministic max via shuffles
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
    __syncthreads();
    RT m2 = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m2 = fmax(m2, sh[w]);
    const RT sigma = 2.0 * m2 + 1.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (dropped[i]) A[(size_t)i * n + i] = mkc<RT>(sigma, 0.0);
}

// ------------------------------------------------------------------ tridiagonalisation
// Range of a column: the sums of squares below keep their type's precision for |x|^2 in [lo, hi]
// (double-FP32: the low part of a square is 2^-48 of it, and FP32 ends at 2^-149); a column outside is
// brought to about one by a power of two f, whose inverse is a normal number.
template <typename RT> struct ColRange {
    using F = RT;
    static __device__ __forceinline__ bool ok(RT t) {
        return sizeof(RT) == 8 ? t >= (RT)0x1p-900 && t <= (RT)0x1p900 : t >= (RT)0x1p-96 && t <= (RT)0x1p96;
    }
};
template <> struct ColRange<df64> {
    using F = float;
    static __device__ __forceinline__ bool ok(df64 t) { return t.hi >= 0x1p-96f && t.hi <= 0x1p96f; }
};
__device__ __forceinline__ float col_factor(float m) { return scalbnf(1.f, min(126, max(-100, -ilogbf(m)))); }
__device__ __forceinline__ double col_factor(double m) { return scalbn(1.0, min(1000, max(-900, -ilogb(m)))); }
__device__ __forceinline__ float scaled(float a, float f) { return a * f; }
__device__ __forceinline__ double scaled(double a, double f) { return a * f; }
__device__ __forceinline__ df64 scaled(df64 a, float f) { return df64(a.hi * f, a.lo * f); }
template <typename RT>
__device__ __forceinline__ cx<RT> scaled(cx<RT> a, typename ColRange<RT>::F f) {
    return mkc<RT>(scaled(a.x, f), scaled(a.y, f));
}
__device__ __forceinline__ float high(float a) { return a; }
__device__ __forceinline__ double high(double a) { return a; }
__device__ __forceinline__ float high(df64 a) { return a.hi; }

// Reflector of x = A[i+1:n, i] in the LAPACK larfg convention:
//   H = I - tau v v^H, v[0] = 1, H^H x = beta e_1 with beta real.
template <typename RT>
struct Refl {
    cx<RT> tau;
    RT beta;
    cx<RT> scal;                         // v[r] = (x[r] pre) scal for r >= 1
    typename ColRange<RT>::F pre;        // a power of two; 0: x is out of range (reflector_rescaled)
    __device__ __forceinline__ cx<RT> of(cx<RT> x) const { return (pre != 1 ? scaled<RT>(x, pre) : x) * scal; }
};

// Reflector from alpha = x[0] and s = sum_{r>=1} |x[r]|^2 (LAPACK larfg convention).
template <typename RT>
__device__ __forceinline__ Refl<RT> reflector_from(cx<RT> alpha, RT s) {
    Refl<RT> R;
    const RT t = abs2(alpha) + s;
    R.pre = ColRange<RT>::ok(t) ? 1 : 0;
    if (R.pre == 0 || (s == 0.0 && alpha.y == 0.0)) {
        R.tau = mkc<RT>(0.0, 0.0);
        R.beta = alpha.x;
        R.scal = mkc<RT>(0.0, 0.0);
        return R;
    }
    const RT beta = -copysign(sqrt(t), alpha.x);
    R.beta = beta;
    R.tau = mkc<RT>((beta - alpha.x) / beta, -alpha.y / beta);
    const cx<RT> den = mkc<RT>(alpha.x - beta, alpha.y);
    const RT dd = abs2(den);
    R.scal = mkc<RT>(den.x / dd, -den.y / dd);
    return R;
}

// The reflector of a column of L entries whose |x|^2 is out of range (zero, nearly decoupled or huge columns): as
// above on x times a power of two.  Every thread of the block calls it, and gets the result; sh holds 32
// entries.  (Without it a double-FP32 column of norm 5e-20 or less, whose |den|^2 has no FP32
// reciprocal, made the whole eigen-decomposition not a number, and columns below 1e-15 lost digits.)
template <typename RT, bool CG, typename PT>
__device__ __noinline__ Refl<RT> reflector_rescaled(const cx<PT> *col, int L, RT *sh) {
    using F = typename ColRange<RT>::F;
    F m = 0;                             // largest part, or not a number where one is
    auto larger = [&m](F a) { m = a > m || a != a ? a : m; };
    for (int r = threadIdx.x; r < L; r += blockDim.x) {
        const cx<RT> x = CG ? ldcg_as<RT>(col + r) : ld_as<RT>(col + r);
        larger(fabs(high(x.x)));
        larger(fabs(high(x.y)));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) larger(__shfl_xor_sync(0xffffffffu, m, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = RT(m);
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) larger(high(sh[w]));
    const cx<RT> alpha = CG ? ldcg_as<RT>(col) : ld_as<RT>(col);
    if (m == 0) {
        Refl<RT> R = reflector_from<RT>(mkc<RT>(0.0, 0.0), RT(0.0));
        R.pre = 1;
        return R;
    }
    const F f = col_factor(m);
    RT s = 0.0;
    for (int r = 1 + threadIdx.x; r < L; r += blockDim.x)
        s += abs2(scaled<RT>(CG ? ldcg_as<RT>(col + r) : ld_as<RT>(col + r), f));
    s = block_sum(s, sh);
    Refl<RT> R = reflector_from<RT>(scaled<RT>(alpha, f), s);
    if (R.pre == 0) {                    // infinite or not a number: so is the result
        const RT t = abs2(scaled<RT>(alpha, f)) + s, nan = t - t;
        R.beta = nan;
        R.tau = R.scal = mkc<RT>(nan, nan);
    }
    R.beta = scaled(R.beta, 1 / f);
    R.pre = f;
    return R;
}

template <typename RT, bool CG = false, typename PT = RT>
__device__ Refl<RT> make_reflector(const cx<PT> *__restrict__ col, int L, RT *sh) {
    RT s = 0.0;
    for (int r = 1 + threadIdx.x; r < L; r += blockDim.x) s += abs2(CG ? ldcg_as<RT>(col + r) : ld_as<RT>(col + r));
    s = block_sum(s, sh);
    const Refl<RT> R = reflector_from<RT>(CG ? ldcg_as<RT>(col) : ld_as<RT>(col), s);
    return R.pre != 0 ? R : reflector_rescaled<RT, CG, PT>(col, L, sh);
}

// Block sum whose cross-warp step is one warp's shuffle tree (a fixed order): for large
// blocks, where every thread summing all warp partials would cost more issue slots than
// the rest of the step.  sh holds 33 entries; every thread gets the result.
template <typename RT>
__device__ RT block_sum_tree(RT v, RT *sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        RT t = lane < nw ? sh[lane] : RT(0.0);
        t = warp_sum(t);
        if (lane == 0) sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

// make_reflector with the tree sum and the scalar arithmetic in one thread, broadcast
// through shared memory (*rb).
template <typename RT, typename PT = RT>
__device__ Refl<RT> make_reflector_bc(const cx<PT> *__restrict__ col, int L, RT *sh, Refl<RT> *rb) {
    RT s = 0.0;
    for (int r = 1 + threadIdx.x; r < L; r += blockDim.x) s += abs2(ld_as<RT>(col + r));
    s = block_sum_tree(s, sh);
    if (threadIdx.x == 0) *rb = reflector_from<RT>(ld_as<RT>(col), s);
    __syncthreads();
    const Refl<RT> R = *rb;
    return R.pre != 0 ? R : reflector_rescaled<RT, false, PT>(col, L, sh);
}

// Step i, part 1: reflector (every block, redundantly) and y = A22 v by 32x32 tiles;
// the last block to finish forms w = tau y - |tau|^2/2 (v^H y) v.
template <typename RT>
__global__ void __launch_bounds__(256)
k_tri_step1(int n, int i, cx<RT> *__restrict__ A, int lda, cx<RT> *__restrict__ Hv, cx<RT> *__restrict__ taus,
            RT *__restrict__ dg, RT *__restrict__ eg, cx<RT> *__restrict__ ypart, cx<RT> *__restrict__ wv,
            unsigned int *__restrict__ counter) {
    __shared__ RT sh[32];
    __shared__ cx<RT> vs[32];
    __shared__ cx<RT> acc[8][33];
    __shared__ bool last;
    const int L = n - i - 1;
    const cx<RT> *col = A + (size_t)i * lda + i + 1;
    const Refl<RT> R = make_reflector<RT>(col, L, sh);
    const int tr = blockIdx.x, tc = blockIdx.y;
    const int tid = threadIdx.x;
    if (tr == 0 && tc == 0) {
        for (int r = tid; r < L; r += blockDim.x) Hv[(size_t)i * n + i + 1 + r] = (r == 0) ? mkc<RT>(1.0, 0.0) : R.of(col[r]);
        if (tid == 0) {
            taus[i] = R.tau;
            dg[i] = A[(size_t)i * lda + i].x;
            eg[i] = R.beta;
        }
    }
    // v entries of this column tile
    if (tid < 32) {
        const int c = tc * 32 + tid;
        vs[tid] = (c < L) ? ((c == 0) ? mkc<RT>(1.0, 0.0) : R.of(col[c])) : mkc<RT>(0.0, 0.0);
    }
    __syncthreads();
    const int rl = tid & 31, cg = tid >> 5;  // 32 rows x 8 column groups of 4
    const int r = tr * 32 + rl;
    cx<RT> s = mkc<RT>(0.0, 0.0);
    if (r < L) {
        const cx<RT> *A22 = A + (size_t)(i + 1) * lda + i + 1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int cl = cg * 4 + q, c = tc * 32 + cl;
            if (c < L) s = s + A22[(size_t)c * lda + r] * vs[cl];
        }
    }
    acc[cg][rl] = s;
    __syncthreads();
    if (tid < 32) {
        cx<RT> t = acc[0][tid];
        for (int g = 1; g < 8; ++g) t = t + acc[g][tid];
        const int rr = tr * 32 + tid;
        if (rr < L) ypart[(size_t)tc * n + rr] = t;
    }
    // last-block reduction (no waiting: only the block that arrives last continues)
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const unsigned int total = gridDim.x * gridDim.y;
        const unsigned int prev = atomicAdd(counter + i, 1u);
        last = (prev == total - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int ncb = gridDim.y;
    // y = sum of partials (fixed order), dot = v^H y
    RT dre = 0.0, dim = 0.0;
    for (int rr = tid; rr < L; rr += blockDim.x) {
        cx<RT> y = mkc<RT>(0.0, 0.0);
        for (int c = 0; c < ncb; ++c) {
            y = y + ldcg_cx(ypart + (size_t)c * n + rr);
        }
        const cx<RT> v = (rr == 0) ? mkc<RT>(1.0, 0.0) : R.of(col[rr]);
        // conj(v) * y
        dre += v.x * y.x + v.y * y.y;
        dim += v.x * y.y - v.y * y.x;
        wv[rr] = y;  // stash y, scaled below
    }
    dre = block_sum(dre, sh);
    (void)dim;  // v^H A v is real for Hermitian A
    const RT t2 = 0.5 * abs2(R.tau) * dre;
    __syncthreads();
    for (int rr = tid; rr < L; rr += blockDim.x) {
        const cx<RT> v = (rr == 0) ? mkc<RT>(1.0, 0.0) : R.of(col[rr]);
        const cx<RT> y = wv[rr];
        wv[rr] = R.tau * y - t2 * v;
    }
}

// Step i, part 2: A22 -= w v^H + v w^H on 32x32 tiles.
template <typename RT>
__global__ void __launch_bounds__(256)
k_tri_step2(int n, int i, cx<RT> *__restrict__ A, int lda, const cx<RT> *__restrict__ Hv, const cx<RT> *__restrict__ wv) {
    __shared__ cx<RT> vr[32], wr[32], vc[32], wc[32];
    const int L = n - i - 1;
    const int tr = blockIdx.x, tc = blockIdx.y, tid = threadIdx.x;
    const cx<RT> *v = Hv + (size_t)i * n + i + 1;
    if (tid < 32) {
        const int r = tr * 32 + tid, c = tc * 32 + tid;
        vr[tid] = r < L ? v[r] : mkc<RT>(0.0, 0.0);
        wr[tid] = r < L ? wv[r] : mkc<RT>(0.0, 0.0);
        vc[tid] = c < L ? v[c] : mkc<RT>(0.0, 0.0);
        wc[tid] = c < L ? wv[c] : mkc<RT>(0.0, 0.0);
    }
    __syncthreads();
    cx<RT> *A22 = A + (size_t)(i + 1) * lda + i + 1;
    for (int e = tid; e < 32 * 32; e += blockDim.x) {
        const int rl = e & 31, cl = e >> 5;
        const int r = tr * 32 + rl, c = tc * 32 + cl;
        if (r < L && c < L) {
            cx<RT> a = A22[(size_t)c * lda + r];
            a = a - mul_conj(wr[rl], vc[cl]) - mul_conj(vr[rl], wc[cl]);
            A22[(size_t)c * lda + r] = a;
        }
    }
}

// Grid-wide barrier for co-resident blocks (cooperative launch): a monotone arrival
// counter; block 0 thread 0 of every block waits for `target` arrivals.  Bounded: a
// wait that runs out (or sees another block's failure) sets *err and the blocks leave.
__device__ __forceinline__ bool grid_barrier(unsigned int *count, unsigned int target, int *err) {
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        int ok = 0;
        for (long long it = 0; it < (1LL << 22); ++it) {
            if (*reinterpret_cast<volatile unsigned int *>(count) >= target) { ok = 1; break; }
            if (*reinterpret_cast<volatile int *>(err)) break;
        }
        if (!ok) atomicExch(err, 1);
        __threadfence();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// Whole Householder tridiagonalisation in one cooperative launch (same arithmetic as
// k_tri_step1 / k_tri_step2, same fixed summation order): per column, every block
// forms the reflector, multiplies its 32 x 32 tiles of A22 by v, [barrier], sums the
// partial products for all rows and forms w, updates its tiles, [barrier].  Data
// written by other blocks is read through L2 (__ldcg).  Dynamic shared memory: v and w
// (2 n complex).
template <typename RT>
__global__ void __launch_bounds__(256)
k_tri_coop(int n, cx<RT> *__restrict__ A, int lda, cx<RT> *__restrict__ Hv, cx<RT> *__restrict__ taus,
           RT *__restrict__ dg, RT *__restrict__ eg, cx<RT> *__restrict__ ypart, unsigned int *bar, int *err) {
    extern __shared__ __align__(16) unsigned char dsm[];
    cx<RT> *vsh = reinterpret_cast<cx<RT> *>(dsm);
    cx<RT> *wsh = vsh + n;
    __shared__ RT sh[32];
    __shared__ cx<RT> acc[8][33];
    const int tid = threadIdx.x, G = gridDim.x;
    unsigned int arrivals = 0;
    for (int i = 0; i + 1 < n; ++i) {
        const int L = n - i - 1;
        const int tl = (L + 31) / 32, ntiles = tl * tl;
        const cx<RT> *col = A + (size_t)i * lda + i + 1;
        const Refl<RT> R = make_reflector<RT, true>(col, L, sh);
        for (int r = tid; r < L; r += blockDim.x) vsh[r] = (r == 0) ? mkc<RT>(1.0, 0.0) : R.of(ldcg_cx(col + r));
        if (blockIdx.x == 0) {
            for (int r = tid; r < L; r += blockDim.x) Hv[(size_t)i * n + i + 1 + r] = vsh[r];
            if (tid == 0) {
                taus[i] = R.tau;
                dg[i] = ldcg_cx(A + (size_t)i * lda + i).x;
                eg[i] = R.beta;
            }
        }
        __syncthreads();
        const cx<RT> *A22 = A + (size_t)(i + 1) * lda + i + 1;
        const int rl = tid & 31, cg = tid >> 5;
        for (int t = blockIdx.x; t < ntiles; t += G) {
            const int tr = t % tl, tc = t / tl;
            const int r = tr * 32 + rl;
            cx<RT> sacc = mkc<RT>(0.0, 0.0);
            if (r < L) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = tc * 32 + cg * 4 + q;
                    if (c < L) sacc = sacc + ldcg_cx(A22 + (size_t)c * lda + r) * vsh[c];
                }
            }
            acc[cg][rl] = sacc;
            __syncthreads();
            if (tid < 32) {
                cx<RT> u = acc[0][tid];
                for (int g = 1; g < 8; ++g) u = u + acc[g][tid];
                const int rr = tr * 32 + tid;
                if (rr < L) ypart[(size_t)tc * n + rr] = u;
            }
            __syncthreads();
        }
        arrivals += G;
        if (!grid_barrier(bar, arrivals, err)) return;
        // y = sum of the tile-column partials (fixed order), dot = v^H y, w = tau y - |tau|^2/2 (v^H y) v
        RT dre = 0.0;
        for (int rr = tid; rr < L; rr += blockDim.x) {
            cx<RT> y = mkc<RT>(0.0, 0.0);
            for (int c = 0; c < tl; ++c) y = y + ldcg_cx(ypart + (size_t)c * n + rr);
            const cx<RT> v = vsh[rr];
            dre += v.x * y.x + v.y * y.y;
            wsh[rr] = y;
        }
        dre = block_sum(dre, sh);
        const RT t2 = 0.5 * abs2(R.tau) * dre;
        for (int rr = tid; rr < L; rr += blockDim.x) wsh[rr] = R.tau * wsh[rr] - t2 * vsh[rr];
        __syncthreads();
        // A22 -= w v^H + v w^H on this block's tiles
        cx<RT> *A22w = A + (size_t)(i + 1) * lda + i + 1;
        for (int t = blockIdx.x; t < ntiles; t += G) {
            const int tr = t % tl, tc = t / tl;
            for (int e = tid; e < 32 * 32; e += blockDim.x) {
                const int r = tr * 32 + (e & 31), c = tc * 32 + (e >> 5);
                if (r < L && c < L) {
                    cx<RT> a = ldcg_cx(A22w + (size_t)c * lda + r);
                    a = a - mul_conj(wsh[r], vsh[c]) - mul_conj(vsh[r], wsh[c]);
                    A22w[(size_t)c * lda + r] = a;
                }
            }
        }
        arrivals += G;
        if (!grid_barrier(bar, arrivals, err)) return;
    }
    if (blockIdx.x == 0 && tid == 0) dg[n - 1] = ldcg_cx(A + (size_t)(n - 1) * lda + n - 1).x;
}

// a - w_r conj(v_c) - v_r conj(w_c), each real part through fused multiply-adds
template <typename CT>
__device__ __forceinline__ cx<CT> rank2_entry(cx<CT> a, cx<CT> wr, cx<CT> vr, cx<CT> vc, cx<CT> wc) {
    CT re = fma(-wr.x, vc.x, a.x);
    re = fma(-wr.y, vc.y, re);
    re = fma(-vr.x, wc.x, re);
    re = fma(-vr.y, wc.y, re);
    CT im = fma(-wr.y, vc.x, a.y);
    im = fma(wr.x, vc.y, im);
    im = fma(-vr.y, wc.x, im);
    im = fma(vr.x, wc.y, im);
    return mkc<CT>(re, im);
}
// The reduction held in the shared memory of one thread-block cluster of CS CTAs, for small
// matrices (see kTriClusterMaxN).  CTA q keeps the rows
// r = q + CS j of the full Hermitian matrix, row-major, so that y = A v needs no reduction
// across CTAs.  Per column i, after one cluster barrier every CTA holds y_i = A^(i) v_i and
// column i+1 of A^(i), both gathered through distributed shared memory, and forms w_i, the
// next column, d, e and reflector i+1 on its own: the same operations on the same values in
// the same order, so the same bits in every CTA.  Then each CTA applies the rank-2 update to
// its rows of the trailing block and, in the same pass, multiplies them by v_{i+1} (one warp
// per row), and sends its entries of y_{i+1} and of column i+2 to every CTA.  The gathered
// vectors alternate between two buffers, so that one barrier per column orders every write
// after the reads of the buffer it overwrites.  Outputs: Hv, taus in the
// compute type; d, e.  Dynamic shared memory: nr x n matrix entries (nr = ceil(n / CS)) and
// 7 n vector entries.
template <typename RT, typename CT>
__global__ void __launch_bounds__(1024, 1)
k_tri_cluster(int n, const cx<RT> *__restrict__ A, int lda, cx<RT> *__restrict__ Hv, cx<RT> *__restrict__ taus,
              RT *__restrict__ dg, RT *__restrict__ eg) {
    static_assert(sizeof(cx<CT>) == sizeof(cx<RT>), "the compute type keeps the storage size");
    namespace cgn = cooperative_groups;
    cgn::cluster_group cl = cgn::this_cluster();
    const int CS = (int)cl.num_blocks(), q = (int)cl.block_rank();
    const int nr = (n + CS - 1) / CS;
    extern __shared__ __align__(16) unsigned char dsm[];
    cx<CT> *M = reinterpret_cast<cx<CT> *>(dsm);       // local row j = global row q + CS j
    cx<CT> *vb = M + (size_t)nr * n;                    // v_i and v_{i+1}, by parity of i
    cx<CT> *w = vb + 2 * n;                             // w_i
    cx<CT> *yg = w + n;                                 // gathered y, two parities
    cx<CT> *cg = yg + 2 * n;                            // gathered next column, two parities
    __shared__ CT sh[33];
    __shared__ Refl<CT> rb;
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, nw = blockDim.x >> 5;
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
    // every CTA of the cluster running before any of them writes another's shared memory
    cl.sync();
    for (size_t e = tid; e < (size_t)nr * n; e += blockDim.x) {
        const int j = (int)(e / n), c = (int)(e % n), r = q + CS * j;
        M[e] = r < n ? ld_as<CT>(A + (size_t)c * lda + r) : zero;
    }
    // reflector 0 from column 0 of A, d[0]
    Refl<CT> R = make_reflector_bc<CT, RT>(A + 1, n - 1, sh, &rb);
    for (int r = tid; r < n; r += blockDim.x)
        vb[r] = (r < 1) ? zero : (r == 1 ? mkc<CT>(1.0, 0.0) : R.of(ld_as<CT>(A + r)));
    if (q == 0 && tid == 0) dg[0] = A[0].x;
    __syncthreads();
    // y_0 = A[J,J] v_0 and column 1 on the owned rows of J = [1, n), sent to every CTA
    for (int j = wp; j < nr; j += nw) {
        const int r = q + CS * j;
        if (r < 1 || r >= n) continue;
        const cx<CT> *Mr = M + (size_t)j * n;
        cx<CT> acc = zero;
        for (int c = 1 + lane; c < n; c += 32) acc = cmac(acc, Mr[c], vb[c]);
        acc.x = warp_sum(acc.x);
        acc.y = warp_sum(acc.y);
        if (lane < CS) {
            cl.map_shared_rank(yg, lane)[r] = acc;
            cl.map_shared_rank(cg, lane)[r] = Mr[1];
        }
    }
    cl.sync();
    for (int i = 0; i + 1 < n; ++i) {
        const int par = i & 1;
        cx<CT> *v = vb + (size_t)par * n, *vn = vb + (size_t)(1 - par) * n;
        const cx<CT> *yv = yg + (size_t)par * n;
        cx<CT> *x = cg + (size_t)par * n;
        // w_i = tau y - |tau|^2 / 2 (v^H y) v on J = [i+1, n)
        CT dre = 0.0;
        for (int r = i + 1 + tid; r < n; r += blockDim.x) dre += v[r].x * yv[r].x + v[r].y * yv[r].y;
        dre = block_sum_tree(dre, sh);
        const CT t2 = (CT)0.5 * abs2(R.tau) * dre;
        for (int r = i + 1 + tid; r < n; r += blockDim.x) w[r] = R.tau * yv[r] - t2 * v[r];
        __syncthreads();
        // column i+1 of A^(i+1) (in place of the gathered column of A^(i)), d[i+1]
        const cx<CT> vi1 = v[i + 1], wi1 = w[i + 1];
        for (int r = i + 1 + tid; r < n; r += blockDim.x) x[r] = x[r] - mul_conj(w[r], vi1) - mul_conj(v[r], wi1);
        __syncthreads();
        if (q == 0) {
            cx<CT> *HvC = reinterpret_cast<cx<CT> *>(Hv);
            for (int r = i + 1 + tid; r < n; r += blockDim.x) HvC[(size_t)i * n + r] = v[r];
            if (tid == 0) {
                reinterpret_cast<cx<CT> *>(taus)[i] = R.tau;
                eg[i] = (RT)R.beta;
                dg[i + 1] = (RT)x[i + 1].x;
            }
        }
        if (i + 2 >= n) break;  // last column: nothing left to transform
        const Refl<CT> Rn = make_reflector_bc<CT>(x + i + 2, n - i - 2, sh, &rb);
        for (int r = tid; r < n; r += blockDim.x)
            vn[r] = (r < i + 2) ? zero : (r == i + 2 ? mkc<CT>(1.0, 0.0) : Rn.of(x[r]));
        __syncthreads();
        // rank-2 update of the owned rows of the trailing block [i+2, n)^2, times v_{i+1}
        const int c2 = i + 2, nxt = 1 - par;
        for (int j = wp; j < nr; j += nw) {
            const int r = q + CS * j;
            if (r < c2 || r >= n) continue;
            cx<CT> *Mr = M + (size_t)j * n;
            const cx<CT> wr = w[r], vr = v[r];
            cx<CT> acc = zero;
            for (int c = c2 + lane; c < n; c += 32) {
                const cx<CT> a = rank2_entry(Mr[c], wr, vr, v[c], w[c]);
                Mr[c] = a;
                acc = cmac(acc, a, vn[c]);
            }
            acc.x = warp_sum(acc.x);
            acc.y = warp_sum(acc.y);
            __syncwarp();
            if (lane < CS) {
                cl.map_shared_rank(yg, lane)[(size_t)nxt * n + r] = acc;
                cl.map_shared_rank(cg, lane)[(size_t)nxt * n + r] = Mr[c2];
            }
        }
        R = Rn;
        cl.sync();
    }
}

// ---- light sums, for the few steps of a shuffle tree: double-FP32 pairs whose low part is renormalised
// only at the end.  Each step keeps the exact error of the high parts' sum; the low part, a few units
// of 2^-24 of the high one, rounds at 2^-48 of it.  Plain arithmetic for other types.
template <typename CT>
__device__ __forceinline__ CT light_add(CT a, CT b) { return a + b; }
template <>
__device__ __forceinline__ df64 light_add<df64>(df64 a, df64 b) {
    df64 r;
    df64::two_sum(a.hi, b.hi, r.hi, r.lo);
    r.lo = __fadd_rn(r.lo, __fadd_rn(a.lo, b.lo));
    return r;
}
template <typename CT>
__device__ __forceinline__ CT light_norm(CT a) { return a; }
template <>
__device__ __forceinline__ df64 light_norm<df64>(df64 a) { return df64::norm(a.hi, a.lo); }

template <typename CT>
__device__ __forceinline__ CT light_warp_sum(CT v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = light_add<CT>(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The warps' partial sums into sh (one entry per warp, not reused before another barrier), and, in one
// warp after the barrier, their sum.
template <typename CT>
__device__ __forceinline__ void light_partial(CT v, CT *sh) {
    v = light_warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
}
template <typename CT>
__device__ __forceinline__ CT light_total(const CT *sh) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    return light_norm(light_warp_sum(lane < nw ? sh[lane] : CT(0.0)));
}

// Reflector from alpha = x[0] and s = sum_{r>=1} |x[r]|^2 (as reflector_from), by a whole warp: lanes 0-3
// each take one of the four divisions.
template <typename CT>
__device__ __forceinline__ Refl<CT> reflector_warp(cx<CT> alpha, CT s) {
    Refl<CT> R;
    const CT t = abs2(alpha) + s;
    R.pre = ColRange<CT>::ok(t) ? 1 : 0;
    if (R.pre == 0 || (s == CT(0.0) && alpha.y == CT(0.0))) {
        R.tau = mkc<CT>(0.0, 0.0);
        R.beta = alpha.x;
        R.scal = mkc<CT>(0.0, 0.0);
        return R;
    }
    const int lane = threadIdx.x & 31;
    const CT beta = -copysign(sqrt(t), alpha.x);
    const cx<CT> den = mkc<CT>(alpha.x - beta, alpha.y);
    const CT num = (lane & 3) == 0 ? beta - alpha.x : (lane & 3) == 2 ? den.x : (lane & 3) == 1 ? -alpha.y : -den.y;
    const CT quo = num / ((lane & 2) ? abs2(den) : beta);
    R.beta = beta;
    R.tau = mkc<CT>(__shfl_sync(0xffffffffu, quo, 0), __shfl_sync(0xffffffffu, quo, 1));
    R.scal = mkc<CT>(__shfl_sync(0xffffffffu, quo, 2), __shfl_sync(0xffffffffu, quo, 3));
    return R;
}

// Grid barrier of co-resident blocks: one counter, arrival by a releasing reduction, one polling thread
// per block with acquiring loads.  2250 cycles on 152 blocks (fences around a plain atomic: 2850;
// a flag per block, polled by a warp or by every thread: 7000 to 9000, the polls delay the stores).
// Bounded like grid_barrier.
__device__ __forceinline__ bool release_barrier(unsigned int *count, unsigned int target, int *err) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        ok = false;
        for (long long it = 0; it < (1LL << 22); ++it) {
            unsigned int c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
            if (c >= target) { ok = true; break; }
            if ((it & 255) == 255 && *reinterpret_cast<volatile int *>(err)) break;
        }
        if (!ok) atomicExch(err, 1);
    }
    return __syncthreads_and(ok) != 0;
}

// Householder tridiagonalisation with the rows of the full Hermitian matrix dealt cyclically to the
// blocks of one cooperative grid (row r to block r mod G), in shared memory, so that y = A v needs
// no reduction across blocks.  Per column i, after one grid barrier every block reads y_i = A^(i) v_i and
// column i+1 of A^(i) (2 n entries through L2) and forms w_i, the next column, d, e and reflector i+1
// itself: the same operations on the same values in the same order, so the same bits in every
// block.  Then each block updates its rows of the trailing block and in the same pass multiplies
// them by v_{i+1} (WPR warps per row), and publishes its entries of y_{i+1} and of column i+2 in the other of
// two buffers.  v_i[i+1] = 1, so column i+1 needs only each thread's own w and the scalar w[i+1].
// What bounds it: the chain of a column (grid barrier, the L2 reads, two block sums, square root and
// divisions), about 4 us, and above n = 800 the double-FP32 updates of the rows.  Cycles of a column at
// n = 384 / 1152: grid barrier 2250, L2 reads 900 / 1500, sums and scalars 2500, vectors 1500 / 3000, rows
// 1500 / 7000.  Measured (Rayleigh-Ritz step, m = n / 3, double-FP32 / FP64, ms), the cluster kernel
// (n = 384) or the tile kernel (n = 1152), whose blocks each summed 36 partial products per row, before:
//   n = 192  2.50 -> 2.26 / 5.45 -> 4.51;  384  5.96 -> 5.05 / 13.8 -> 10.1;  1152  62 -> 34 / 140 -> 84
// Dynamic shared memory: nr x n matrix entries (nr = ceil(n / G)), 3 n vector entries.
template <typename RT, typename CT>
__global__ void __launch_bounds__(512)
k_tri_rows(int n, const cx<RT> *__restrict__ A, int lda, cx<RT> *__restrict__ Hv, cx<RT> *__restrict__ taus,
           RT *__restrict__ dg, RT *__restrict__ eg, cx<RT> *__restrict__ xch_st, unsigned int *count, int *err) {
    static_assert(sizeof(cx<CT>) == sizeof(cx<RT>), "the compute type keeps the storage size");
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ CT sh[2][16], dots;   // (reflector_rescaled takes sh as 32 entries)
    __shared__ cx<CT> part[512 / 32], al;
    __shared__ Refl<CT> rs;
    const int G = gridDim.x, q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, nw = blockDim.x >> 5;
    const int nr = (n + G - 1) / G;
    const int WPR = max(1, nw / nr), rstep = nw / WPR;   // warps per row, rows at a time
    cx<CT> *M = reinterpret_cast<cx<CT> *>(dsm);          // local row j = global row q + G j
    cx<CT> *v = M + (size_t)nr * n, *w = v + n, *x = w + n;
    cx<CT> *xch = reinterpret_cast<cx<CT> *>(xch_st);     // [parity][y, column][n]
    cx<CT> *HvC = reinterpret_cast<cx<CT> *>(Hv);
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
    for (size_t e = tid; e < (size_t)nr * n; e += blockDim.x) {
        const int r = q + G * (int)(e % nr), c = (int)(e / nr);   // neighbouring threads on neighbouring owned rows
        M[(size_t)(e % nr) * n + c] = r < n ? ld_as<CT>(A + (size_t)c * lda + r) : zero;
    }
    // reflector 0 from column 0 of A, d[0]
    CT sq = 0.0;
    for (int r = 2 + tid; r < n; r += blockDim.x) sq = light_add<CT>(sq, abs2(ld_as<CT>(A + r)));
    light_partial(sq, sh[0]);
    Refl<CT> R = reflector_warp<CT>(ld_as<CT>(A + 1), light_total(sh[0]));
    if (R.pre == 0) R = reflector_rescaled<CT, false, RT>(A + 1, n - 1, sh[0]);
    for (int r = tid; r < n; r += blockDim.x) v[r] = (r < 1) ? zero : (r == 1 ? mkc<CT>(1.0, 0.0) : R.of(ld_as<CT>(A + r)));
    if (q == 0 && tid == 0) dg[0] = A[0].x;
    __syncthreads();
    for (int i = -1; i + 1 < n; ++i) {
        // i = -1: only the products A^(0) v_0 and column 1 of A^(0)
        const int c2 = i + 2;
        cx<CT> *vn = v;
        if (i >= 0) {
            const cx<CT> *yv = xch + (size_t)(i & 1) * 2 * n, *cv = yv + n;
            const cx<CT> y1 = ldcg_cx(yv + i + 1);
            CT dre = 0.0;
            for (int r = i + 1 + tid; r < n; r += blockDim.x) {
                const cx<CT> y = ldcg_cx(yv + r), vr = v[r];
                x[r] = ldcg_cx(cv + r);
                w[r] = y;
                dre = fma(vr.x, y.x, fma(vr.y, y.y, dre));
            }
            light_partial(dre, sh[1]);
            if (wp == 0) {
                const CT t = light_total(sh[1]);
                if (lane == 0) dots = (CT)0.5 * abs2(R.tau) * t;
            }
            __syncthreads();
            // w = tau y - |tau|^2 / 2 (v^H y) v, column i+1 of A^(i+1) = c - w - conj(w[i+1]) v on J = [i+1, n)
            const CT t2 = dots;
            cx<CT> w1 = R.tau * y1;
            w1.x = w1.x - t2;
            CT s = 0.0;
            for (int r = i + 1 + tid; r < n; r += blockDim.x) {
                const cx<CT> vr = v[r], y = w[r], c = x[r];
                cx<CT> wr, xr;
                wr.x = fma(R.tau.x, y.x, fma(-R.tau.y, y.y, -(t2 * vr.x)));
                wr.y = fma(R.tau.x, y.y, fma(R.tau.y, y.x, -(t2 * vr.y)));
                xr.x = fma(-vr.x, w1.x, fma(-vr.y, w1.y, c.x - wr.x));
                xr.y = fma(-vr.y, w1.x, fma(vr.x, w1.y, c.y - wr.y));
                w[r] = wr;
                x[r] = xr;
                if (r == c2) al = xr;
                if (r > c2) s = fma(xr.x, xr.x, fma(xr.y, xr.y, s));
                if (q == i % G) HvC[(size_t)i * n + r] = vr;
                if (r == i + 1 && q == 0) {
                    reinterpret_cast<cx<CT> *>(taus)[i] = R.tau;
                    eg[i] = (RT)R.beta;
                    dg[i + 1] = (RT)xr.x;
                }
            }
            if (c2 >= n) break;   // last column: nothing left to transform
            light_partial(s, sh[0]);
            if (wp == 0) {        // one warp: every warp at once would share the FP64 units' and divisions' time
                const Refl<CT> t = reflector_warp<CT>(al, light_total(sh[0]));
                if (lane == 0) rs = t;
            }
            __syncthreads();
            R = rs;
            if (R.pre == 0) R = reflector_rescaled<CT, false, CT>(x + c2, n - c2, sh[0]);
            for (int r = c2 + tid; r < n; r += blockDim.x) x[r] = r == c2 ? mkc<CT>(1.0, 0.0) : R.of(x[r]);
            vn = x;
            __syncthreads();
        }
        // rank-2 update of the owned rows of [c2, n)^2 (columns and rows from 1 on at i = -1), times vn
        cx<CT> *yo = xch + (size_t)((i + 1) & 1) * 2 * n, *co = yo + n;
        for (int j0 = 0; j0 < nr; j0 += rstep) {
            const int j = j0 + wp / WPR, sub = wp % WPR, r = q + G * j;
            const bool on = wp < rstep * WPR && j < nr && r >= c2 && r < n;
            if (on) {
                cx<CT> *Mr = M + (size_t)j * n;
                cx<CT> acc = zero;
                const cx<CT> wr = i >= 0 ? w[r] : zero, vr = i >= 0 ? v[r] : zero;
                for (int c = c2 + lane + 32 * sub; c < n; c += 32 * WPR) {
                    cx<CT> a = Mr[c];
                    if (i >= 0) {
                        const cx<CT> vc = v[c], wc = w[c];
                        // pairs: accurate sums here (a third more instructions of this line); the chain of
                        // multiply-adds leaves a tenth to a quarter more error in the eigenvectors at n = 640
                        if constexpr (std::is_same<CT, df64>::value) a = a - mul_conj(wr, vc) - mul_conj(vr, wc);
                        else a = rank2_entry(a, wr, vr, vc, wc);
                        Mr[c] = a;
                    }
                    acc = cmac(acc, a, vn[c]);
                }
                // both parts in one tree: after the first step the lower half warp has re, the upper im
                const bool up = lane >= 16;
                const CT mine = up ? acc.y : acc.x, other = __shfl_xor_sync(0xffffffffu, up ? acc.x : acc.y, 16);
                CT t = light_add<CT>(mine, other);
#pragma unroll
                for (int o = 8; o; o >>= 1) t = light_add<CT>(t, __shfl_xor_sync(0xffffffffu, t, o));
                const CT im = __shfl_sync(0xffffffffu, t, 16);
                if (lane == 0) part[wp] = mkc<CT>(t, im);
            }
            __syncthreads();
            if (on && sub == 0 && lane == 0) {
                cx<CT> t = part[wp];
                for (int k = 1; k < WPR; ++k) t = mkc<CT>(light_add<CT>(t.x, part[wp + k].x), light_add<CT>(t.y, part[wp + k].y));
                yo[r] = mkc<CT>(light_norm(t.x), light_norm(t.y));
                co[r] = M[(size_t)j * n + c2];
            }
            if (j0 + rstep < nr) __syncthreads();
        }
        if (i >= 0) {
            cx<CT> *t = v;
            v = x;
            x = t;
        }
        if (!release_barrier(count, (unsigned int)(i + 2) * (unsigned int)G, err)) return;
    }
}

template <typename RT>
__global__ void k_tri_last(int n, const cx<RT> *__restrict__ A, int lda, RT *__restrict__ dg) {
    if (threadIdx.x == 0) dg[n - 1] = A[(size_t)(n - 1) * lda + n - 1].x;
}

// ------------------------------------------------------------------ eigenvalues (multisection)
template <typename RT>
__device__ __forceinline__ int sturm_count(const RT *__restrict__ d, const RT *__restrict__ e, int n,
                                           RT x, RT pivmin) {
    int c = 0;
    RT q = d[0] - x;
    if (fabs(q) < pivmin) q = -pivmin;
    c += (q < 0.0);
    for (int i = 1; i < n; ++i) {
        const RT ei = e[i - 1];
        q = d[i] - x - (ei * ei) / q;
        if (fabs(q) < pivmin) q = -pivmin;
        c += (q < 0.0);
    }
    return c;
}

template <typename RT>
__device__ void tri_bounds(const RT *__restrict__ d, const RT *__restrict__ e, int n, RT &lo,
                           RT &hi, RT &tnorm, RT &pivmin) {
    lo = Lim<RT>::big();
    hi = -Lim<RT>::big();
    RT emax2 = 0.0;
    for (int i = 0; i < n; ++i) {
        RT r = 0.0;
        if (i > 0) r += fabs(e[i - 1]);
        if (i < n - 1) { r += fabs(e[i]); emax2 = fmax(emax2, e[i] * e[i]); }
        lo = fmin(lo, d[i] - r);
        hi = fmax(hi, d[i] + r);
    }
    tnorm = fmax(fabs(lo), fabs(hi));
    pivmin = Lim<RT>::tiny() * fmax((RT)1.0, emax2);
    const RT pad = 2.0 * Lim<RT>::eps() * tnorm * n + 2.0 * pivmin;
    lo -= pad;
    hi += pad;
}

// Multisection: each round the 32 lanes of a warp evaluate Sturm counts at 32
// points inside the bracket and keep the 1/33 of it that holds eigenvalue k
// (about 5 bits per round).  The FP64 divisions of the Sturm counts are the cost
// (this GPU has few FP64 units per SM).
constexpr int kMsLanes = 32;
// FP32 Sturm count on FP32 copies of d and e^2 (shared memory).
__device__ __forceinline__ int sturm_count32(const float *__restrict__ d, const float *__restrict__ e2, int n, float x,
                                             float pivmin) {
    int c = 0;
    float q = d[0] - x;
    if (fabsf(q) < pivmin) q = -pivmin;
    c += (q < 0.f);
    for (int i = 1; i < n; ++i) {
        q = d[i] - x - e2[i - 1] / q;
        if (fabsf(q) < pivmin) q = -pivmin;
        c += (q < 0.f);
    }
    return c;
}

// FP64 rounds of one eigenvalue index k by a warp, from the bracket [lo, hi] (have: it may be trusted, but
// is checked by the first round, whose end lanes evaluate its ends) or from [lo_g, hi_g].
__device__ void multisect_fp64(int n, int k, const double *__restrict__ d, const double *__restrict__ e, bool have,
                               double lo, double hi, double lo_g, double hi_g, double pivmin,
                               double *__restrict__ theta) {
    const int sub = threadIdx.x;
    if (!have) {
        double tnorm;
        tri_bounds(d, e, n, lo_g, hi_g, tnorm, pivmin);
        lo = lo_g;
        hi = hi_g;
    }
    bool check = have;
    for (int it = 0; it < 32; ++it) {
        const double w = hi - lo;
        if (w <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 4.0 * pivmin) break;  // warp-uniform
        double x;
        if (check)  // bracket ends on the end lanes, 30 points between
            x = (sub == 0) ? lo : (sub == kMsLanes - 1) ? hi : lo + w * (double)sub / (double)(kMsLanes - 1);
        else
            x = lo + w * (double)(sub + 1) / (double)(kMsLanes + 1);
        const int c = sturm_count(d, e, n, x, pivmin);
        if (check) {
            check = false;
            const bool ok = __shfl_sync(0xffffffffu, c, 0) <= k && __shfl_sync(0xffffffffu, c, kMsLanes - 1) > k;
            if (!ok) {  // the bracket missed (not expected): restart from Gershgorin
                lo = lo_g;
                hi = hi_g;
                continue;
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, c <= k);
        const int T = __popc(mask) - 1;  // counts are monotone in sub: lanes 0..T have c <= k
        const double xlo = __shfl_sync(0xffffffffu, x, T < 0 ? 0 : T);
        const double xhi = __shfl_sync(0xffffffffu, x, T < kMsLanes - 1 ? T + 1 : kMsLanes - 1);
        if (T >= 0) lo = xlo;
        if (T < kMsLanes - 1) hi = xhi;
    }
    if (sub == 0) theta[k] = 0.5 * (lo + hi);
}

// FP32 (the complex64 step): one warp per eigenvalue index, one warp per block so that the m warps
// spread over the SMs.  FP32 Sturm counts are exact for a matrix whose entries are within a few
// FP32 roundings of T (Kahan; Demmel, Dhillon and Ren 1995); the same holds in each arithmetic
// below, so a bracket widened by a margin well above that perturbation still holds the
// eigenvalue in a finer one.
__global__ void __launch_bounds__(32)
k_multisect32(int n, int m, const float *__restrict__ d, const float *__restrict__ e, float *__restrict__ theta) {
    const int k = blockIdx.x, sub = threadIdx.x;
    if (k >= m) return;
    float lo, hi, tnorm, pivmin;
    tri_bounds(d, e, n, lo, hi, tnorm, pivmin);
    for (int it = 0; it < 32; ++it) {
        const float w = hi - lo;
        if (w <= 2.f * FLT_EPSILON * fmaxf(fabsf(lo), fabsf(hi)) + 4.f * pivmin) break;  // warp-uniform
        const float x = lo + w * (float)(sub + 1) / (float)(kMsLanes + 1);
        const int c = sturm_count(d, e, n, x, pivmin);
        const unsigned mask = __ballot_sync(0xffffffffu, c <= k);
        const int T = __popc(mask) - 1;
        const float xlo = __shfl_sync(0xffffffffu, x, T < 0 ? 0 : T);
        const float xhi = __shfl_sync(0xffffffffu, x, T < kMsLanes - 1 ? T + 1 : kMsLanes - 1);
        if (T >= 0) lo = xlo;
        if (T < kMsLanes - 1) hi = xhi;
    }
    if (sub == 0) theta[k] = 0.5f * (lo + hi);
}

// Double-FP32 Sturm count on pair copies of d and e^2 (shared memory): the same recurrence,
// its divisions on the FP32 units (one SM sub-partition issues an FP64 instruction for a whole
// warp in 64 cycles on this GPU, an FP32 one in 1).  About 2^-47 relative per operation: the
// count is exact for a matrix within a few such roundings of T.
__device__ __forceinline__ int sturm_count_df(const df64 *__restrict__ d, const df64 *__restrict__ e2, int n, df64 x,
                                              float pivmin) {
    int c = 0;
    df64 q = d[0] - x;
    if (fabsf(q.hi) < pivmin) q = df64(-pivmin);
    c += (q.hi < 0.f);
    for (int i = 1; i < n; ++i) {
        q = (d[i] - x) - e2[i - 1] / q;
        if (fabsf(q.hi) < pivmin) q = df64(-pivmin);
        c += (q.hi < 0.f);
    }
    return c;
}

// Multisection with FP32 rounds, then double-FP32 rounds; the bracket bounds come from FP32 copies of
// T with a generous pad.  The FP64-class Rayleigh-Ritz step ends there.  FINE64 (FP64 steps): the
// double-FP32 rounds stop at the perturbation their counts are exact for, the bracket is widened by
// it, and FP64 rounds, of which the first checks the bracket, finish: three of them instead of eight
// (an FP64 round is the dear one: n divisions of ten instructions at 64 cycles a warp).  A matrix
// outside the FP32 range takes FP64 rounds only.  FP64 Rayleigh-Ritz step, m = n / 3:
//   n = 48 1.08 -> 0.97 ms, 96 2.18 -> 1.99, 200 4.80 -> 4.36.
// Dynamic shared memory: d, e^2 as pairs, then as floats (24 n bytes).
template <bool FINE64>
__global__ void __launch_bounds__(32)
k_multisect_df(int n, int m, const double *__restrict__ d, const double *__restrict__ e, double *__restrict__ theta) {
    extern __shared__ __align__(16) unsigned char smraw[];
    df64 *dd = reinterpret_cast<df64 *>(smraw);
    df64 *de2 = dd + n;
    float *ds = reinterpret_cast<float *>(de2 + n);
    float *e2s = ds + n;
    const int k = blockIdx.x, sub = threadIdx.x;
    if (k >= m) return;
    for (int i = sub; i < n; i += kMsLanes) {
        dd[i] = df64(d[i]);
        const df64 ei = (i + 1 < n) ? df64(e[i]) : df64(0.f);
        de2[i] = ei * ei;
        ds[i] = dd[i].hi;
        e2s[i] = de2[i].hi;
    }
    __syncwarp();
    // Gershgorin bracket in FP32, padded well above its rounding
    float lo_f = FLT_MAX, hi_f = -FLT_MAX, emax2 = 0.f;
    bool finite = true;
    for (int i = 0; i < n; ++i) {
        float r = 0.f;
        if (i > 0) r += sqrtf(e2s[i - 1]);
        if (i < n - 1) { r += sqrtf(e2s[i]); emax2 = fmaxf(emax2, e2s[i]); }
        lo_f = fminf(lo_f, ds[i] - r);
        hi_f = fmaxf(hi_f, ds[i] + r);
        finite = finite && fabsf(ds[i]) + r <= FLT_MAX;
    }
    if (!FINE64 && !finite) {   // the minima, maxima and counts would pass over what is not a number
        if (sub == 0) theta[k] = nan("");
        return;
    }
    const float tn = fmaxf(fabsf(lo_f), fabsf(hi_f));
    const float piv = FLT_MIN * fmaxf(1.f, fmaxf(emax2, tn * tn));
    const float gpad = 64.f * FLT_EPSILON * tn * (float)n + 4.f * piv;
    lo_f -= gpad;
    hi_f += gpad;
    const float margin = 32.f * FLT_EPSILON * tn + 4.f * piv;
    float l32 = lo_f, h32 = hi_f;
    for (int it = 0; it < 8 && h32 - l32 > 4.f * margin; ++it) {  // warp-uniform
        const float w = h32 - l32;
        const float x = l32 + w * (float)(sub + 1) / (float)(kMsLanes + 1);
        const int c = sturm_count32(ds, e2s, n, x, piv);
        const unsigned mask = __ballot_sync(0xffffffffu, c <= k);
        const int T = __popc(mask) - 1;
        const float xlo = __shfl_sync(0xffffffffu, x, T < 0 ? 0 : T);
        const float xhi = __shfl_sync(0xffffffffu, x, T < kMsLanes - 1 ? T + 1 : kMsLanes - 1);
        if (T >= 0) l32 = xlo;
        if (T < kMsLanes - 1) h32 = xhi;
    }
    const df64 lo_g(lo_f), hi_g(hi_f);
    df64 lo = fmax(lo_g, df64(l32) - df64(margin)), hi = fmin(hi_g, df64(h32) + df64(margin));
    bool check = true;
    const float eps_df = 0x1p-45f, margin_df = 0x1p-42f * tn + 4.f * piv;
    const bool in_range = tn < 1e15f && tn > 1e-15f;
    for (int it = 0; it < 40; ++it) {
        const df64 w = hi - lo;
        if (FINE64 && (!in_range || w.hi <= 4.f * margin_df)) break;
        if (w.hi <= 2.f * eps_df * fmaxf(fabsf(lo.hi), fabsf(hi.hi)) + 4.f * piv) break;  // warp-uniform
        df64 x;
        if (check)  // bracket ends on the end lanes, 30 points between
            x = (sub == 0) ? lo : (sub == kMsLanes - 1) ? hi : lo + w * df64((float)sub / (float)(kMsLanes - 1));
        else
            x = lo + w * df64((float)(sub + 1) / (float)(kMsLanes + 1));
        const int c = sturm_count_df(dd, de2, n, x, piv);
        if (check) {
            check = false;
            const bool ok = __shfl_sync(0xffffffffu, c, 0) <= k && __shfl_sync(0xffffffffu, c, kMsLanes - 1) > k;
            if (!ok) {  // the FP32 bracket missed (not expected): restart from Gershgorin
                lo = lo_g;
                hi = hi_g;
                continue;
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, c <= k);
        const int T = __popc(mask) - 1;
        const df64 xlo = __shfl_sync(0xffffffffu, x, T < 0 ? 0 : T);
        const df64 xhi = __shfl_sync(0xffffffffu, x, T < kMsLanes - 1 ? T + 1 : kMsLanes - 1);
        if (T >= 0) lo = xlo;
        if (T < kMsLanes - 1) hi = xhi;
    }
    if (!FINE64) {
        if (sub == 0) theta[k] = (double)((lo + hi) * df64(0.5f));
        return;
    }
    multisect_fp64(n, k, d, e, in_range, (double)lo - (double)margin_df, (double)hi + (double)margin_df, (double)lo_f,
                   (double)hi_f, DBL_MIN * fmax(1.0, (double)emax2), theta);
}

// ------------------------------------------------------------------ eigenvectors (inverse iteration)
template <typename RT>
__device__ __forceinline__ RT hash_uniform(unsigned int a, unsigned int b) {
    unsigned int h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 16; h *= 0x7FEB352Du; h ^= h >> 15; h *= 0x846CA68Bu; h ^= h >> 16;
    return (RT)h * (2.0 / 4294967296.0) - 1.0;
}

// |a| < |b| and a == 0; for FP64 on the bits, without an FP64 instruction
__device__ __forceinline__ bool mag_less(float a, float b) { return fabsf(a) < fabsf(b); }
__device__ __forceinline__ bool is_zero(float a) { return a == 0.f; }
__device__ __forceinline__ bool mag_less(double a, double b) {
    constexpr unsigned long long M = 0x7FFFFFFFFFFFFFFFULL;
    return ((unsigned long long)__double_as_longlong(a) & M) < ((unsigned long long)__double_as_longlong(b) & M);
}
__device__ __forceinline__ bool is_zero(double a) { return (__double_as_longlong(a) << 1) == 0; }

// One warp per eigenvalue index; the warp whose eigenvalue starts a cluster of
// close eigenvalues computes all vectors of that cluster, in order: lane 0 runs the
// LU of T - lambda I with partial pivoting and the solves (sequential recurrences,
// kept in shared memory), from a pseudo-random start; after each solve the warp
// orthogonalises against the cluster's earlier vectors (modified Gram-Schmidt) and
// normalises.  Dynamic shared memory: 6 n reals + n pivots.
// What bounds it: lane 0's chain of dependent FP64 instructions, 64 cycles or more each (with few clusters, of
// the longest one).  So comparisons run on the bits, rows are swapped by selects (a predicated-off
// instruction costs the same), each pivot is inverted once (the multiplier is its product with the
// reciprocal, corrected by its remainder; the rows of U are divided by their pivots by all lanes).  Three
// solves for every vector: two for eigenvalues far from all others take 1 % off the step at n = 1152 and
// nothing below.  GB300, the step with 128 vectors of n = 384 in double-FP32 4.57 -> 4.45 ms, all of n = 1152
// 33.0 -> 32.2.
template <typename RT>
__global__ void __launch_bounds__(32)
k_inviter(int n, int m, const RT *__restrict__ d, const RT *__restrict__ e, const RT *__restrict__ theta,
          RT *Z) {
    extern __shared__ __align__(16) unsigned char smraw[];
    RT *dd = reinterpret_cast<RT *>(smraw);
    RT *du = dd + n, *du2 = du + n, *dl = du2 + n, *z = dl + n, *rdd = z + n;
    signed char *pv = reinterpret_cast<signed char *>(rdd + n);
    const int k = blockIdx.x, lane = threadIdx.x;
    if (k >= m) return;
    RT lo, hi, tnorm, pivmin;
    tri_bounds(d, e, n, lo, hi, tnorm, pivmin);
    // vectors of eigenvalues closer than gaptol are orthogonalised against each other;
    // elsewhere orthogonality is ~ eps |T| / gap (LAPACK uses 1e-3 |T| for single precision)
    const RT gaptol = (sizeof(RT) == 4 ? (RT)1e-3 : (RT)1e-5) * fmax(tnorm, Lim<RT>::tiny());
    const RT pert = 10.0 * Lim<RT>::eps() * fmax(tnorm, Lim<RT>::tiny());
    // pivots below a hundredth of a rounding of |T| are raised to it: where lam is a decoupled diagonal entry
    // to the last bit, the pivot is the coupling itself, and the solution its inverse squared, which overflowed
    // (a zero vector)
    const RT low = pert * (RT)1e-3;
    if (k > 0 && theta[k] - theta[k - 1] <= gaptol) return;  // not a cluster start
    RT lam_prev = -Lim<RT>::big();
    for (int j = k; j < m; ++j) {
        if (j > k && theta[j] - theta[j - 1] > gaptol) break;
        RT lam = theta[j];
        if (j > k && lam < lam_prev + pert) lam = lam_prev + pert;
        lam_prev = lam;
        RT *zj = Z + (size_t)j * n;
        for (int i = lane; i < n; i += 32) {
            dd[i] = d[i] - lam;
            dl[i] = i + 1 < n ? e[i] : (RT)0.0;
            z[i] = hash_uniform<RT>((unsigned)j, (unsigned)i);
        }
        __syncwarp();
        if (lane == 0) {
            RT p = dd[0], u = dl[0];            // the row being eliminated: pivot candidate and its right neighbour
            for (int i = 0; i + 1 < n; ++i) {
                const RT l = dl[i], dn = dd[i + 1], un = dl[i + 1];
                const bool sw = mag_less(p, l);
                RT piv = sw ? l : p;
                const RT o = sw ? p : l, u0 = sw ? dn : u, u1 = sw ? u : dn;
                piv = is_zero(piv) ? pert : mag_less(piv, low) ? copysign(low, piv) : piv;
                const RT r = (RT)1.0 / piv, f0 = o * r;
                const RT f = fma(fma(-f0, piv, o), r, f0);   // o / piv
                rdd[i] = r;
                dl[i] = f;
                du[i] = u0;
                du2[i] = sw ? un : (RT)0.0;
                pv[i] = sw;
                p = fma(-f, u0, u1);
                const RT t = -f * un;
                u = sw ? t : un;
            }
            p = is_zero(p) ? pert : mag_less(p, low) ? copysign(low, p) : p;
            rdd[n - 1] = (RT)1.0 / p;
        }
        __syncwarp();
        for (int i = lane; i + 1 < n; i += 32) {   // rows of U over their pivots
            du[i] *= rdd[i];
            du2[i] *= rdd[i];
        }
        __syncwarp();
        for (int it = 0; it < 3; ++it) {
            if (lane == 0) {
                RT zi = z[0];
                for (int i = 0; i + 1 < n; ++i) {
                    const RT zn = z[i + 1], f = dl[i];
                    const bool sw = pv[i];
                    const RT x = sw ? zn : zi, y = sw ? zi : zn;
                    z[i] = x;
                    zi = fma(-f, x, y);
                }
                z[n - 1] = zi;
            }
            __syncwarp();
            for (int i = lane; i < n; i += 32) z[i] *= rdd[i];
            __syncwarp();
            if (lane == 0) {
                RT z1 = z[n - 1], z2 = 0.0;
                for (int i = n - 2; i >= 0; --i) {
                    const RT x = fma(-du[i], z1, fma(-du2[i], z2, z[i]));
                    z[i] = x;
                    z2 = z1;
                    z1 = x;
                }
            }
            __syncwarp();
            for (int p = k; p < j; ++p) {
                const RT *zp = Z + (size_t)p * n;
                RT sp = 0.0;
                for (int i = lane; i < n; i += 32) sp += z[i] * zp[i];
                sp = warp_sum(sp);
                for (int i = lane; i < n; i += 32) z[i] -= sp * zp[i];
                __syncwarp();
            }
            RT nr = 0.0;
            for (int i = lane; i < n; i += 32) nr += z[i] * z[i];
            nr = warp_sum(nr);
            const RT inv = nr > 0.0 ? 1.0 / sqrt(nr) : 0.0;
            for (int i = lane; i < n; i += 32) z[i] *= inv;
            __syncwarp();
        }
        for (int i = lane; i < n; i += 32) zj[i] = z[i];
        __syncwarp();
    }
}

// ------------------------------------------------------------------ back-transformation
// V = H_0 H_1 ... H_{n-2} Z with H_i = I - tau_i v_i v_i^H, applied kWy reflectors at a time in
// the compact WY form (Schreiber and Van Loan, 1989): H_{i0} ... H_{i0+k-1} = I - Y T Y^H with
// Y = [v_{i0} ... v_{i0+k-1}] and T upper triangular, T_jj = tau_j and
// T[0:j, j] = -tau_j T[0:j, 0:j] (Y[:, 0:j]^H v_j).  Each block then costs one reduction
// (t = Y^H z) instead of one per reflector.  v_i is read only on its support r >= i + 1.
constexpr int kWy = 32;

// Partial Gram matrices G = Y^H Y of each block of kWy reflectors (block b: reflectors
// 32 b ...), over row chunk ch of the block's rows [32 b + 1, n): grid (blocks, chunks).  The
// chunk of Y is staged in shared memory (zero where v_k has no support, r <= 32 b + k); thread
// (k, g) accumulates G[k][g + 8 u], u = 0..3.  Gp[b][ch] is a full kWy x kWy row-major matrix.
constexpr int kWyRows = 64;   // rows of a chunk
template <typename CT>
__global__ void __launch_bounds__(256)
k_wy_gram(int n, int nch, const cx<CT> *__restrict__ Hv, cx<CT> *__restrict__ Gp) {
    __shared__ cx<CT> Ys[kWyRows][kWy + 1];
    const int b = blockIdx.x, ch = blockIdx.y, i0 = b * kWy, kb = min(kWy, n - 1 - i0);
    const int rows = n - (i0 + 1), per = (rows + nch - 1) / nch;
    const int r0 = i0 + 1 + ch * per, r1 = min(n, r0 + per);
    const int tid = threadIdx.x, k = tid >> 3, g = tid & 7;
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
    cx<CT> acc[4] = {zero, zero, zero, zero};
    for (int c0 = r0; c0 < r1; c0 += kWyRows) {
        __syncthreads();
        for (int e = tid; e < kWyRows * kWy; e += blockDim.x) {
            const int kk = e / kWyRows, rr = e % kWyRows, r = c0 + rr;
            Ys[rr][kk] = (kk < kb && r < r1 && r > i0 + kk) ? Hv[(size_t)(i0 + kk) * n + r] : zero;
        }
        __syncthreads();
        const int nr = min(kWyRows, r1 - c0);
        for (int rr = 0; rr < nr; ++rr) {
            const cx<CT> a = conjc(Ys[rr][k]);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = cmac(acc[u], a, Ys[rr][g + 8 * u]);
        }
    }
    cx<CT> *out = Gp + ((size_t)b * nch + ch) * kWy * kWy;
#pragma unroll
    for (int u = 0; u < 4; ++u) out[k * kWy + g + 8 * u] = acc[u];
}

// T of each block from its Gram (chunk partials summed in chunk order): T_jj = tau_j, then
// pairs of adjacent diagonal blocks of width h = 1, 2, 4, 8, 16 merged by
// T12 = -T11 G12 T22 (the product of the two blocks' WY forms), each merge level in two
// parallel matrix products.  kWy x kWy row-major into Tf[b], zero outside the reflectors.
template <typename CT>
__global__ void __launch_bounds__(256)
k_wy_t(int n, int nch, const cx<CT> *__restrict__ Gp, const cx<CT> *__restrict__ taus, cx<CT> *__restrict__ Tf) {
    __shared__ cx<CT> G[kWy][kWy + 1];
    __shared__ cx<CT> T[kWy][kWy + 1];
    __shared__ cx<CT> X[kWy][kWy + 1];
    const int b = blockIdx.x, i0 = b * kWy, kb = min(kWy, n - 1 - i0), tid = threadIdx.x;
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
    for (int e = tid; e < kWy * kWy; e += blockDim.x) {
        const int k = e / kWy, j = e % kWy;
        cx<CT> sum = zero;
        for (int ch = 0; ch < nch; ++ch) sum = sum + Gp[((size_t)b * nch + ch) * kWy * kWy + e];
        G[k][j] = sum;
        T[k][j] = (k == j && k < kb) ? taus[i0 + k] : zero;
    }
    __syncthreads();
    for (int h = 1; h < kWy; h *= 2) {
        // entries of the merges at this level: (kWy / 2h) merges x h x h
        const int nent = (kWy / (2 * h)) * h * h;
        // X = T11 G12
        for (int e = tid; e < nent; e += blockDim.x) {
            const int mg = e / (h * h), k = (e % (h * h)) / h, l = e % h;
            const int a = mg * 2 * h;
            cx<CT> u = zero;
            for (int p = k; p < h; ++p) u = cmac(u, T[a + k][a + p], G[a + p][a + h + l]);
            X[a + k][a + h + l] = u;
        }
        __syncthreads();
        // T12 = -X T22
        for (int e = tid; e < nent; e += blockDim.x) {
            const int mg = e / (h * h), k = (e % (h * h)) / h, l = e % h;
            const int a = mg * 2 * h;
            cx<CT> u = zero;
            for (int p = 0; p <= l; ++p) u = cmac(u, X[a + k][a + h + p], T[a + h + p][a + h + l]);
            T[a + k][a + h + l] = zero - u;
        }
        __syncthreads();
    }
    for (int e = tid; e < kWy * kWy; e += blockDim.x) Tf[(size_t)b * kWy * kWy + e] = T[e / kWy][e % kWy];
}

// NV eigenvectors per CTA (z in shared memory in the compute type CT), blocks from the last
// to the first: t = Y^H z (a warp per reflector, KU reflectors at once for independent
// accumulation chains, fixed-order warp sums), s = T t (eight lanes per entry, combined by a
// shuffle tree), z -= Y s (a thread per row, KU partial sums).  Dynamic shared memory:
// NV n entries.
template <typename RT, typename CT, int NV>
__global__ void __launch_bounds__(256)
k_backtransform_wy(int n, int m, const cx<CT> *__restrict__ Hv, const cx<CT> *__restrict__ Tf,
                   const RT *__restrict__ Z, cx<RT> *__restrict__ V, int ldv) {
    constexpr int KU = NV >= 4 ? 1 : 4;
    extern __shared__ __align__(16) unsigned char smraw[];
    cx<CT> *z = reinterpret_cast<cx<CT> *>(smraw);   // [NV][n]
    __shared__ cx<CT> t[NV][kWy], sv[NV][kWy];
    const int j0 = blockIdx.x * NV, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, nw = blockDim.x >> 5;
    const cx<CT> zero = mkc<CT>(0.0, 0.0);
    for (int e = tid; e < NV * n; e += blockDim.x) {
        const int vv = e / n, r = e % n;
        z[e] = (j0 + vv < m) ? mkc<CT>((CT)Z[(size_t)(j0 + vv) * n + r], CT(0.0)) : zero;
    }
    __syncthreads();
    const int nblk = (n - 1 + kWy - 1) / kWy;
    for (int b = nblk - 1; b >= 0; --b) {
        const int i0 = b * kWy, kb = min(kWy, n - 1 - i0);
        // t_k = v_{i0+k}^H z, reflectors k = k0 + nw u (u < KU) together
        for (int k0 = wp; k0 < kWy; k0 += nw * KU) {
            cx<CT> acc[KU][NV];
#pragma unroll
            for (int u = 0; u < KU; ++u)
#pragma unroll
                for (int vv = 0; vv < NV; ++vv) acc[u][vv] = zero;
            for (int r = i0 + 1 + lane; r < n; r += 32) {
                cx<CT> zr[NV];
#pragma unroll
                for (int vv = 0; vv < NV; ++vv) zr[vv] = z[vv * n + r];
#pragma unroll
                for (int u = 0; u < KU; ++u) {
                    const int k = k0 + nw * u;
                    if (k < kb && r > i0 + k) {   // v_{i0+k} lives on r >= i0 + k + 1
                        const cx<CT> a = conjc(Hv[(size_t)(i0 + k) * n + r]);
#pragma unroll
                        for (int vv = 0; vv < NV; ++vv) acc[u][vv] = cmac(acc[u][vv], a, zr[vv]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < KU; ++u) {
                const int k = k0 + nw * u;
#pragma unroll
                for (int vv = 0; vv < NV; ++vv) {
                    const CT re = warp_sum(acc[u][vv].x), im = warp_sum(acc[u][vv].y);
                    if (lane == 0 && k < kWy) t[vv][k] = mkc<CT>(re, im);
                }
            }
        }
        __syncthreads();
        // s = T t: entry (vv, k) from eight lanes, lane part p taking l = k + p, k + p + 8, ...
        const cx<CT> *Tb = Tf + (size_t)b * kWy * kWy;
        for (int e = tid; e < NV * kWy * 8; e += blockDim.x) {
            const int p = e & 7, k = (e >> 3) % kWy, vv = (e >> 3) / kWy;
            cx<CT> u = zero;
            for (int l = k + p; l < kb; l += 8) u = cmac(u, Tb[k * kWy + l], t[vv][l]);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
                u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
            }
            if (p == 0) sv[vv][k] = u;
        }
        __syncthreads();
        // z -= Y s on the rows the block touches
        for (int r = i0 + 1 + tid; r < n; r += blockDim.x) {
            const int kmax = min(kb, r - i0);   // v_{i0+k}[r] is zero for r <= i0 + k
            cx<CT> d[NV][KU];                   // KU partial sums per vector
#pragma unroll
            for (int vv = 0; vv < NV; ++vv)
#pragma unroll
                for (int q = 0; q < KU; ++q) d[vv][q] = zero;
            for (int k = 0; k < kmax; k += KU) {
#pragma unroll
                for (int q = 0; q < KU; ++q) {
                    if (k + q < kmax) {
                        const cx<CT> a = Hv[(size_t)(i0 + k + q) * n + r];
#pragma unroll
                        for (int vv = 0; vv < NV; ++vv) d[vv][q] = cmac(d[vv][q], a, sv[vv][k + q]);
                    }
                }
            }
#pragma unroll
            for (int vv = 0; vv < NV; ++vv) {
                cx<CT> tot = d[vv][0];
#pragma unroll
                for (int q = 1; q < KU; ++q) tot = tot + d[vv][q];
                z[vv * n + r] = z[vv * n + r] - tot;
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < NV * n; e += blockDim.x) {
        const int vv = e / n, r = e % n;
        if (j0 + vv < m) V[(size_t)(j0 + vv) * ldv + r] = mkc<RT>((RT)z[e].x, (RT)z[e].y);
    }
}

template <typename RT>
__global__ void k_scale_rows_copy(int n, int m, const RT *__restrict__ d, const cx<RT> *__restrict__ T, int ldt,
                                  cx<RT> *__restrict__ C, int ldc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i < n) C[(size_t)j * ldc + i] = d[i] * T[(size_t)j * ldt + i];
}

__global__ void k_copy_int(const int *__restrict__ a, int *__restrict__ b) { *b = *a; }

size_t align_up(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// Raise a kernel's dynamic shared-memory ceiling to the device maximum.  The attribute is
// process-wide, so it is never lowered: launches of different sizes on concurrent streams
// then never see a ceiling below their own request.
int allow_max_dyn_smem(const void *fn) {
    int dev = 0, smem_max = 0;
    LG_CUDA_TRY(cudaGetDevice(&dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa;
    LG_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
    LG_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     smem_max - (int)fa.sharedSizeBytes));
    return LOBPCG_OK;
}

// The cluster-resident tridiagonalisation (8 CTAs) when the device can place such a cluster;
// done = false leaves the reduction to the grid-wide kernels.
template <typename RT, typename CT>
int launch_tri_cluster(int n, const cx<RT> *A, int lda, cx<RT> *Hv, cx<RT> *taus, RT *dg, RT *eg, cudaStream_t s,
                       bool &done) {
    done = false;
    const int CS = 8;
    const int nr = (n + CS - 1) / CS;
    const size_t dsm = sizeof(cx<CT>) * ((size_t)nr * n + 7 * (size_t)n);
    int dev = 0, smem_max = 0, cl_ok = 0;
    LG_CUDA_TRY(cudaGetDevice(&dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&cl_ok, cudaDevAttrClusterLaunch, dev));
    const void *fn = (const void *)k_tri_cluster<RT, CT>;
    cudaFuncAttributes fa;
    LG_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
    if (!cl_ok || dsm + fa.sharedSizeBytes > (size_t)smem_max) return LOBPCG_OK;
    // the same (largest) limit from every caller: concurrent lanes launch this kernel with
    // different sizes, and a per-call limit set by one would invalidate another's launch
    LG_TRY(allow_max_dyn_smem(fn));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS);
    cfg.blockDim = dim3(std::min(1024, 32 * nr));  // one warp per owned row
    cfg.dynamicSmemBytes = dsm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) != cudaSuccess || ncl < 1) {
        (void)cudaGetLastError();  // this cluster shape cannot be placed: not an error
        return LOBPCG_OK;
    }
    LG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_tri_cluster<RT, CT>, n, A, lda, Hv, taus, dg, eg));
    LG_TRY(check_launch("tridiagonalisation (cluster)"));
    done = true;
    return LOBPCG_OK;
}
// The row-cyclic cooperative tridiagonalisation, when the rows of a block and three vectors fit its
// shared memory; done = false leaves the reduction to the other kernels.  With concurrent streams
// each grid takes its share of the SMs (so that all of them are resident together).
template <typename RT, typename CT>
int launch_tri_rows(EigWork &w, int n, const cx<RT> *A, int lda, cx<RT> *Hv, cx<RT> *taus, RT *dg, RT *eg, cx<RT> *xch,
                    unsigned int *count, cudaStream_t s, bool &done) {
    done = false;
    int dev = 0, sms = 0, coop = 0, smem_max = 0;
    LG_CUDA_TRY(cudaGetDevice(&dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    LG_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    int *err = device_wait_flag();
    const int share = std::max(1, w.coop_share);
    int G = std::max(1, std::min(n, sms / share));
    const int nr = (n + G - 1) / G;
    G = (n + nr - 1) / nr;   // as few blocks as give the same rows per block
    const size_t dsm = sizeof(cx<CT>) * ((size_t)nr * n + 3 * (size_t)n);
    const void *fn = (const void *)k_tri_rows<RT, CT>;
    cudaFuncAttributes fa;
    LG_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
    if (!coop || !err || dsm + fa.sharedSizeBytes > (size_t)smem_max) return LOBPCG_OK;
    LG_TRY(allow_max_dyn_smem(fn));
    int per_sm = 0;
    LG_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 512, dsm));
    if (per_sm < 1 || (size_t)G * share > (size_t)sms * per_sm) return LOBPCG_OK;
    void *args[] = {(void *)&n, (void *)&A, (void *)&lda, (void *)&Hv, (void *)&taus, (void *)&dg,
                    (void *)&eg, (void *)&xch, (void *)&count, (void *)&err};
    if (w.gate && share == 1) {
        // one cooperative grid at a time across concurrent streams
        std::lock_guard<std::mutex> lk(w.gate->mu);
        if (w.gate->used) LG_CUDA_TRY(cudaStreamWaitEvent(s, w.gate->ev, 0));
        LG_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(512), args, dsm, s));
        LG_CUDA_TRY(cudaEventRecord(w.gate->ev, s));
        w.gate->used = true;
    } else {
        LG_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(512), args, dsm, s));
    }
    LG_TRY(check_launch("tridiagonalisation (rows)"));
    done = true;
    return LOBPCG_OK;
}
// One cluster's barrier is cheaper than the grid's, its eight SMs' arithmetic dearer: 1.48 against
// 1.52 ms at n = 128 (double-FP32 step, m = n / 3), 2.50 against 2.26 at n = 192; FP64 3.10 / 3.03, 5.45 / 4.51.
constexpr int kTriClusterMaxN = 128;
constexpr int kWyChunks = 8;   // row chunks of the back-transformation's Gram partials

// T factors, then the blocked application; NV eigenvectors per CTA, as many as keep about
// 128 CTAs or more (each CTA reads every reflector once) and fit its shared memory (8 up to n = 1752,
// 4 up to 3568).
template <typename RT, typename CT>
int backtransform_wy(int n, int m, const cx<CT> *Hv, const cx<CT> *taus, cx<CT> *Tf, cx<CT> *Gp, const RT *Z,
                     cx<RT> *V, int ldv, cudaStream_t s) {
    const int nblk = (n - 1 + kWy - 1) / kWy;
    const int nch = kWyChunks;
    k_wy_gram<CT><<<dim3(nblk, nch), 256, 0, s>>>(n, nch, Hv, Gp);
    LG_TRY(check_launch("back-transform Gram partials"));
    k_wy_t<CT><<<nblk, 256, 0, s>>>(n, nch, Gp, taus, Tf);
    LG_TRY(check_launch("back-transform T factors"));
    int NV = m >= 8 * 128 ? 8 : m >= 4 * 128 ? 4 : m >= 2 * 128 ? 2 : 1;
    int smem_max = 0;
    LG_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, current_device()));
    while (NV > 1 && sizeof(cx<CT>) * (size_t)NV * (n + 2 * kWy) > (size_t)smem_max) NV /= 2;
    const size_t smem = sizeof(cx<CT>) * (size_t)NV * n;
    const int grid = (m + NV - 1) / NV;
    auto run = [&](auto kern) -> int {
        if (smem > 48 * 1024) LG_TRY(allow_max_dyn_smem((const void *)kern));
        kern<<<grid, 256, smem, s>>>(n, m, Hv, Tf, Z, V, ldv);
        return check_launch("back-transform (compact WY)");
    };
    if (NV == 8) return run(k_backtransform_wy<RT, CT, 8>);
    if (NV == 4) return run(k_backtransform_wy<RT, CT, 4>);
    if (NV == 2) return run(k_backtransform_wy<RT, CT, 2>);
    return run(k_backtransform_wy<RT, CT, 1>);
}

template <typename RT>
int heev_lowest_t(EigWork &w, int n, int m, cx<RT> *A, int lda, RT *theta, cx<RT> *V, int ldv, cudaStream_t s) {
    if (n <= 0 || m <= 0) return LOBPCG_OK;
    if (m > n) return fail(LOBPCG_ERR_ARG, "heev: m > n");
    // workspace carve-up
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    const size_t o_hv = take(sizeof(cx<RT>) * (size_t)n * n);
    const size_t o_tau = take(sizeof(cx<RT>) * n);
    const size_t o_d = take(sizeof(RT) * n);
    const size_t o_e = take(sizeof(RT) * n);
    const size_t o_yp = take(sizeof(cx<RT>) * (size_t)((n + 31) / 32) * n);
    const size_t o_wv = take(sizeof(cx<RT>) * 4 * (size_t)n);
    const size_t o_z = take(sizeof(RT) * (size_t)n * m);
    const size_t o_cnt = take(sizeof(unsigned int) * n);
    const size_t o_tf = take(sizeof(cx<RT>) * (size_t)kWy * kWy * ((n + kWy - 1) / kWy));
    const size_t o_gp = take(sizeof(cx<RT>) * (size_t)kWy * kWy * kWyChunks * ((n + kWy - 1) / kWy));
    LG_TRY(w.alloc->ensure(w.buf, off));
    char *base = reinterpret_cast<char *>(w.buf.p);
    cx<RT> *Hv = reinterpret_cast<cx<RT> *>(base + o_hv);
    cx<RT> *taus = reinterpret_cast<cx<RT> *>(base + o_tau);
    RT *dg = reinterpret_cast<RT *>(base + o_d);
    RT *eg = reinterpret_cast<RT *>(base + o_e);
    cx<RT> *yp = reinterpret_cast<cx<RT> *>(base + o_yp);
    cx<RT> *wv = reinterpret_cast<cx<RT> *>(base + o_wv);
    RT *Z = reinterpret_cast<RT *>(base + o_z);
    unsigned int *cnt = reinterpret_cast<unsigned int *>(base + o_cnt);
    cx<RT> *Tf = reinterpret_cast<cx<RT> *>(base + o_tf);
    cx<RT> *Gp = reinterpret_cast<cx<RT> *>(base + o_gp);
    LG_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned int) * n, s));
    LG_CUDA_TRY(cudaMemsetAsync(taus, 0, sizeof(cx<RT>) * n, s));
    bool coop_done = false, hv_df = false;
    if (n >= 2 && n <= kTriClusterMaxN) {
        bool done = false, df = false;
        if constexpr (std::is_same<RT, double>::value) {
            df = w.df;  // the double-FP32 compute type, as in the grid-wide kernel below
            if (df) LG_TRY((launch_tri_cluster<RT, df64>(n, A, lda, Hv, taus, dg, eg, s, done)));
        }
        if (!df) LG_TRY((launch_tri_cluster<RT, RT>(n, A, lda, Hv, taus, dg, eg, s, done)));
        coop_done = done;
        hv_df = done && df;
    }
    if (!coop_done && n >= 2) {
        bool done = false, df = false;
        if constexpr (std::is_same<RT, double>::value) {
            df = w.df;
            if (df) LG_TRY((launch_tri_rows<RT, df64>(w, n, A, lda, Hv, taus, dg, eg, wv, cnt, s, done)));
        }
        if (!df) LG_TRY((launch_tri_rows<RT, RT>(w, n, A, lda, Hv, taus, dg, eg, wv, cnt, s, done)));
        coop_done = done;
        hv_df = done && df;
    }
    if (!coop_done && n >= 2 && n <= 1024) {
        // one cooperative launch; falls back to two launches per column if it cannot run
        const int tl0 = (n - 1 + 31) / 32;
        const size_t dsm = 2 * sizeof(cx<RT>) * (size_t)n;
        int per_sm = 0, dev = 0, sms = 0, coop = 0;
        LG_CUDA_TRY(cudaGetDevice(&dev));
        LG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        LG_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        if (dsm > 48 * 1024)
            LG_TRY(allow_max_dyn_smem((const void *)k_tri_coop<RT>));
        LG_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tri_coop<RT>, 256, dsm));
        const int G = std::min(tl0 * tl0, sms * std::max(per_sm, 0));
        int *err = device_wait_flag();
        if (coop && G >= 1 && err) {
            unsigned int *bar = cnt;            // arrival counter (zeroed above)
            void *args[] = {(void *)&n, (void *)&A, (void *)&lda, (void *)&Hv, (void *)&taus, (void *)&dg, (void *)&eg,
                            (void *)&yp, (void *)&bar, (void *)&err};
            if (w.gate) {
                std::lock_guard<std::mutex> lk(w.gate->mu);
                if (w.gate->used) LG_CUDA_TRY(cudaStreamWaitEvent(s, w.gate->ev, 0));
                LG_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_tri_coop<RT>, dim3(G), dim3(256), args, dsm, s));
                LG_CUDA_TRY(cudaEventRecord(w.gate->ev, s));
                w.gate->used = true;
            } else {
                LG_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_tri_coop<RT>, dim3(G), dim3(256), args, dsm, s));
            }
            LG_TRY(check_launch("tridiagonalisation (cooperative)"));
            coop_done = true;
        }
    }
    if (!coop_done) {
        for (int i = 0; i + 1 < n; ++i) {
            const int L = n - i - 1;
            const int tl = (L + 31) / 32;
            k_tri_step1<RT><<<dim3(tl, tl), 256, 0, s>>>(n, i, A, lda, Hv, taus, dg, eg, yp, wv, cnt);
            LG_TRY(check_launch("tridiag step 1"));
            k_tri_step2<RT><<<dim3(tl, tl), 256, 0, s>>>(n, i, A, lda, Hv, wv);
            LG_TRY(check_launch("tridiag step 2"));
        }
        k_tri_last<RT><<<1, 32, 0, s>>>(n, A, lda, dg);
        LG_TRY(check_launch("tridiag last"));
    }
    if constexpr (std::is_same<RT, double>::value) {
        const size_t smem_ms = 24 * (size_t)n;
        auto ms = w.df ? k_multisect_df<false> : k_multisect_df<true>;
        if (smem_ms > 48 * 1024) LG_TRY(allow_max_dyn_smem((const void *)ms));
        ms<<<m, kMsLanes, smem_ms, s>>>(n, m, dg, eg, theta);
    } else {
        k_multisect32<<<m, kMsLanes, 0, s>>>(n, m, dg, eg, theta);
    }
    LG_TRY(check_launch("multisection"));
    const size_t smem_ii = 6 * sizeof(RT) * (size_t)n + (size_t)n;
    if (smem_ii > 48 * 1024)
        LG_TRY(allow_max_dyn_smem((const void *)k_inviter<RT>));
    k_inviter<RT><<<m, 32, smem_ii, s>>>(n, m, dg, eg, theta, Z);
    LG_TRY(check_launch("inverse iteration"));
    if (n == 1) {
        LG_CUDA_TRY(cudaMemcpy2DAsync(V, sizeof(cx<RT>) * ldv, Z, sizeof(RT), sizeof(RT), m, cudaMemcpyDeviceToDevice, s));
        LG_CUDA_TRY(cudaMemset2DAsync(reinterpret_cast<char *>(V) + sizeof(RT), sizeof(cx<RT>) * ldv, 0, sizeof(RT), m, s));
        return check_launch("back-transform (n = 1)");
    }
    if constexpr (sizeof(cx<RT>) == sizeof(cx<df64>)) {
        if (hv_df)
            return backtransform_wy<RT, df64>(n, m, reinterpret_cast<const cx<df64> *>(Hv),
                                              reinterpret_cast<const cx<df64> *>(taus),
                                              reinterpret_cast<cx<df64> *>(Tf), reinterpret_cast<cx<df64> *>(Gp), Z,
                                              V, ldv, s);
    }
    return backtransform_wy<RT, RT>(n, m, Hv, taus, Tf, Gp, Z, V, ldv, s);
}

template <typename RT>
int hermitize_lower_t(EigWork &w, int n, cx<RT> *A, cudaStream_t s) {
    LG_TRY(w.alloc->ensure(w.ibuf, sizeof(RT) * (size_t)n + 256));
    k_hermitize_rowsum<RT><<<n, 128, 0, s>>>(n, A, nullptr, reinterpret_cast<RT *>(w.ibuf.p));
    return check_launch("hermitize");
}

template <typename RT>
int rayleigh_ritz_t(EigWork &w, int n, int m, const cx<RT> *S, int lds, const cx<RT> *A, int lda, double drop_tol,
                    RT *theta, cx<RT> *C, int ldc, int *ndropped, cudaStream_t s, int lead = 0) {
    if (n <= 0 || m <= 0) return LOBPCG_OK;
    if (m > n) return fail(LOBPCG_ERR_ARG, "rayleigh_ritz: m > n");
    if (n > 4096) return fail(LOBPCG_ERR_ARG, "rayleigh_ritz: n > 4096");
    // own workspace (separate from heev's)
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    const size_t o_ss = take(sizeof(cx<RT>) * (size_t)n * n);
    const size_t o_as = take(sizeof(cx<RT>) * (size_t)n * n);
    const size_t o_li = take(sizeof(cx<RT>) * (size_t)n * n);
    const size_t o_tm = take(sizeof(cx<RT>) * (size_t)n * n);
    const size_t o_q = take(sizeof(cx<RT>) * (size_t)n * m);
    const size_t o_d = take(sizeof(RT) * n);
    const size_t o_rs = take(sizeof(RT) * n);
    const size_t o_dr = take(sizeof(int) * n);
    const size_t o_nd = take(sizeof(int));
    LG_TRY(w.alloc->ensure(w.ibuf, off));
    char *base = reinterpret_cast<char *>(w.ibuf.p);
    cx<RT> *Ss = reinterpret_cast<cx<RT> *>(base + o_ss);
    cx<RT> *As = reinterpret_cast<cx<RT> *>(base + o_as);
    cx<RT> *Li = reinterpret_cast<cx<RT> *>(base + o_li);
    cx<RT> *Tm = reinterpret_cast<cx<RT> *>(base + o_tm);
    cx<RT> *Q = reinterpret_cast<cx<RT> *>(base + o_q);
    RT *d = reinterpret_cast<RT *>(base + o_d);
    RT *rs = reinterpret_cast<RT *>(base + o_rs);
    int *dr = reinterpret_cast<int *>(base + o_dr);
    int *nd = reinterpret_cast<int *>(base + o_nd);

    w.gw.df = std::is_same<RT, double>::value && w.df;  // the small products below
    LG_CUDA_TRY(cudaMemsetAsync(nd, 0, sizeof(int), s));
    LG_CUDA_TRY(cudaMemsetAsync(Li, 0, sizeof(cx<RT>) * (size_t)n * n, s));
    k_scale_gram<RT><<<dim3((n + 127) / 128, n), 128, 0, s>>>(n, S, lds, A, lda, Ss, As, d);
    LG_TRY(check_launch("scale gram"));
    if (lead % NBK != 0 || lead > n || lead < 0) lead = 0;
    if (lead > 0) {
        k_lead_identity<RT><<<dim3((n + 127) / 128, lead), 128, 0, s>>>(n, lead, Ss, Li, dr);
        LG_TRY(check_launch("leading identity"));
    }
    // blocked Cholesky with dropping (L overwrites Ss), after the leading identity columns
    for (int k0 = lead; k0 < n; k0 += NBK) {
        const int kb = std::min(NBK, n - k0);
        bool chol_done = false;
        if constexpr (std::is_same<RT, double>::value) {
            if (w.df) {  // one block: double-FP32 instead of that SM's FP64 units
                k_chol_diag_df<<<1, 256, 0, s>>>(n, k0, kb, Ss, Li, drop_tol, dr, nd);
                chol_done = true;
            }
        }
        if (!chol_done) k_chol_diag<RT><<<1, 256, 0, s>>>(n, k0, kb, Ss, Li, (RT)drop_tol, dr, nd);
        LG_TRY(check_launch("cholesky diag"));
        const int rem = n - k0 - kb;
        if (rem > 0) {
            k_chol_panel<RT><<<(rem + kPanelRows - 1) / kPanelRows, 32 * kPanelRows, 0, s>>>(n, k0, kb, Ss, Li, dr);
            LG_TRY(check_launch("cholesky panel"));
            const cx<RT> *L21 = Ss + (size_t)k0 * n + k0 + kb;
            cx<RT> *S22 = Ss + (size_t)(k0 + kb) * n + k0 + kb;
            LG_TRY(gemm_small<RT>(&w.gw, 'N', 'C', rem, rem, kb, -1.0, L21, n, L21, n, 1.0, S22, n, s, kLowerOut));
        }
    }
    k_zero_dropped_rows<RT><<<n, 128, 0, s>>>(n, Ss, dr);
    LG_TRY(check_launch("zero dropped rows"));
    // off-diagonal blocks of L^-1 by doubling: with the inverses of two adjacent diagonal blocks of
    // width h known, the block below the first is -L22^-1 (L21 L11^-1); all pairs of a width in one launch
    // per product (log2(n / 32) levels instead of n / 32 block rows)
    for (int h = NBK; h < n; h *= 2) {
        const int pairs = (n + h - 1) / (2 * h);                       // pairs with a second block
        const int last = std::min(h, n - (2 * (pairs - 1) + 1) * h);   // its width in the last pair
        const long long st = 2LL * h * (n + 1);
        GemmBatch b1{st, st, st, pairs, last, h};
        LG_TRY(gemm_batch<RT>(w.gw, h, h, h, 1.0, Ss + h, n, Li, n, Tm + h, n, b1, s));
        GemmBatch b2{st, st, st, pairs, last, last};
        LG_TRY(gemm_batch<RT>(w.gw, h, h, h, -1.0, Li + (size_t)h * (n + 1), n, Tm + h, n, Li + h, n, b2, s));
    }
    // Ahat = Li As Li^H (its lower triangle).  Li is lower triangular: the products skip its zeros, and
    // are a half, a sixth and (below) a half of full ones
    LG_TRY(gemm_small<RT>(&w.gw, 'N', 'N', n, n, n, 1.0, Li, n, As, n, 0.0, Tm, n, s, kTriA));
    LG_TRY(gemm_small<RT>(&w.gw, 'N', 'C', n, n, n, 1.0, Tm, n, Li, n, 0.0, As, n, s, kTriB | kLowerOut));
    k_hermitize_rowsum<RT><<<n, 128, 0, s>>>(n, As, dr, rs);
    LG_TRY(check_launch("hermitize"));
    k_set_dropped_diag<RT><<<1, 1024, 0, s>>>(n, As, dr, nd, rs);
    LG_TRY(check_launch("dropped diag"));
    LG_TRY(heev_lowest_t<RT>(w, n, m, As, n, theta, Q, n, s));
    // C = D Li^H Q
    LG_TRY(gemm_small<RT>(&w.gw, 'C', 'N', n, m, n, 1.0, Li, n, Q, n, 0.0, Tm, n, s, kTriA));
    k_scale_rows_copy<RT><<<dim3((n + 127) / 128, m), 128, 0, s>>>(n, m, d, Tm, n, C, ldc);
    LG_TRY(check_launch("scale C"));
    if (ndropped) {
        k_copy_int<<<1, 1, 0, s>>>(nd, ndropped);
        LG_TRY(check_launch("copy ndropped"));
    }
    return LOBPCG_OK;
}

int heev_lowest(EigWork &w, int n, int m, z64 *A, int lda, double *theta, z64 *V, int ldv, cudaStream_t s) {
    return heev_lowest_t<double>(w, n, m, A, lda, theta, V, ldv, s);
}
int hermitize_lower(EigWork &w, int n, z64 *A, cudaStream_t s) { return hermitize_lower_t<double>(w, n, A, s); }
int rayleigh_ritz(EigWork &w, int n, int m, const z64 *S, int lds, const z64 *A, int lda, double drop_tol,
                  double *theta, z64 *C, int ldc, int *ndropped, cudaStream_t s, int lead) {
    return rayleigh_ritz_t<double>(w, n, m, S, lds, A, lda, drop_tol, theta, C, ldc, ndropped, s, lead);
}
int rayleigh_ritz32(EigWork &w, int n, int m, const c32 *S, int lds, const c32 *A, int lda, double drop_tol,
                    float *theta, c32 *C, int ldc, int *ndropped, cudaStream_t s) {
    return rayleigh_ritz_t<float>(w, n, m, S, lds, A, lda, drop_tol, theta, C, ldc, ndropped, s);
}

}  // namespace lg
