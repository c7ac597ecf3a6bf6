// Double-FP32 ("double-word") real scalar for the FP64-class dense algebra of
// the Rayleigh-Ritz step on a GPU whose FP64 units are few: a value is an
// unevaluated pair hi + lo of FP32 numbers with |lo| <= ulp(hi) / 2, which
// carries about 48 significant bits in the FP32 exponent range.
//
// Building blocks (the error-free transformations of floating-point
// arithmetic):
//   TwoSum (Knuth, TAOCP vol. 2, 4.2.2): s + e = a + b exactly, s = fl(a + b);
//   FastTwoSum (Dekker 1971): the same when |a| >= |b|, in three operations;
//   TwoProd through one FMA: p + e = a b exactly, p = fl(a b).
// Addition is the accurate double-word sum (both parts through TwoSum, two
// renormalisations), multiplication TwoProd plus the two cross terms,
// division three quotient digits from one FP32 reciprocal with double-word
// remainders, square root one Newton correction of the FP32 root.  Relative
// error of each operation: a few units of 2^-48.  Every step uses the _rn
// intrinsics so that the compiler cannot contract or reorder it.
//
// The operators and math functions are hidden friends: they are found only
// for df64 arguments, so they never capture calls on double or float.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace lg {

// hi + lo as an FP64 number, rounded to nearest, in integer arithmetic: a warp-wide FP64 instruction
// occupies its sub-partition for 64 cycles on this GPU.  (hi, lo) is normalised (|lo| at most half a
// unit in the last place of hi).  With e the exponent of hi, hi = mh 2^(e - 23) and lo, in units of
// 2^(e - 52), is an integer of at most 2^28 once rounded; their sum is the mantissa up to one
// renormalisation (a power of two less something).
__device__ __forceinline__ double pair_to_double(float hi, float lo) {
    // tiny and huge numbers by 2^64 or 2^-64, exactly, into the middle of the exponent range
    const uint32_t b0 = (__float_as_uint(hi) >> 23) & 255u;
    const float fac = b0 < 64u ? 0x1p64f : b0 > 190u ? 0x1p-64f : 1.f;
    const int adj = b0 < 64u ? -64 : b0 > 190u ? 64 : 0;
    const uint32_t u = __float_as_uint(hi * fac), be = (u >> 23) & 255u;
    // lo 2^(52 - e) as two exact factors, e = be - 127
    const float f = (u >> 31 ? -lo : lo) * fac * __uint_as_float((254u - be) << 23) * 0x1p52f;
    unsigned long long m = ((unsigned long long)((u & 0x7FFFFFu) | 0x800000u) << 29) + (long long)__float2int_rn(f);
    const uint32_t under = (m >> 52) == 0 ? 1u : 0u;            // hi a power of two and lo against it
    m <<= under;
    uint32_t top = (be - under + (uint32_t)(adj + 1023 - 127 - 1)) << 20;   // the leading one adds the exponent
    if (be == 0) { m = 0; top = 0; }                             // zero
    if (be == 255) { m = (unsigned long long)(u & 0x7FFFFFu) << 29; top = 0x7FF00000u; }   // infinite, not a number
    return __hiloint2double((int)((top + (uint32_t)(m >> 32)) | (u & 0x80000000u)), (int)(uint32_t)m);
}

// The pair of an FP64 number, hi = x rounded to nearest and lo = x - hi likewise, in integer arithmetic
// for the same reason (and with no FP64 instruction in a rare branch: predicated off it costs the
// same): the 53-bit mantissa is cut into 24 bits, rounded, and the signed rest.  Numbers whose low
// part would leave the FP32 range are brought into it by 2^64 or 2^-64; below 2^-138, where hi is subnormal, lo
// is zero.
__device__ __forceinline__ void double_to_pair(double x, float &hi, float &lo) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);   // (folds for constants)
    const uint32_t top = (uint32_t)(b >> 32), sign = top & 0x80000000u;
    const int e0 = (int)((top >> 20) & 0x7FFu) - 1023;
    const int e = e0 < -74 ? e0 + 64 : e0 > 126 ? e0 - 64 : e0;
    const float fac = e0 < -74 ? 0x1p-64f : e0 > 126 ? 0x1p64f : 1.f;
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
    const uint32_t mh = (uint32_t)((m + (1ULL << 28)) >> 29);                       // in [2^23, 2^24]
    const int ml = (int)(uint32_t)((uint32_t)m - (mh << 29));                       // in [-2^28, 2^28], mod 2^32
    hi = __uint_as_float((((uint32_t)(e + 126) << 23) + mh) | sign) * fac;           // the leading one adds the exponent
    lo = (float)ml * __uint_as_float(((uint32_t)(e - 52 + 127) << 23) | sign) * fac;
    if (e < -74) lo = 0.f;
    if (e < -86) hi = 0.f;   // below half of FP32's smallest number
    if (e > 126) {   // beyond FP32's range, infinite or not a number
        const bool nan = e0 == 1024 && (b & 0xFFFFFFFFFFFFFULL) != 0;
        hi = __uint_as_float((nan ? 0x7FC00000u : 0x7F800000u) | sign);
        lo = 0.f;
    }
}

struct alignas(8) df64 {
    float hi, lo;

    df64() = default;
    __host__ __device__ __forceinline__ df64(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ __forceinline__ df64(float f) : hi(f), lo(0.f) {}
    __host__ __device__ __forceinline__ df64(int i) : df64((double)i) {}
    __host__ __device__ __forceinline__ df64(unsigned int i) : df64((double)i) {}
    __host__ __device__ __forceinline__ df64(double d) {
#ifdef __CUDA_ARCH__
        double_to_pair(d, hi, lo);
#else
        hi = (float)d;
        lo = (float)(d - (double)hi);
#endif
    }
    __host__ __device__ __forceinline__ explicit operator double() const {
#ifdef __CUDA_ARCH__
        return pair_to_double(hi, lo);
#else
        return (double)hi + (double)lo;
#endif
    }

    // ---- error-free transformations
    static __device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
        s = __fadd_rn(a, b);
        const float bb = __fsub_rn(s, a);
        e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    }
    static __device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e) {
        s = __fadd_rn(a, b);
        e = __fsub_rn(b, __fsub_rn(s, a));
    }
    static __device__ __forceinline__ void fast_two_sum_any(float &h, float &l) {   // in place, any order of size
        float s, e;
        two_sum(h, l, s, e);
        h = s;
        l = e;
    }
    static __device__ __forceinline__ df64 norm(float a, float b) {
        df64 r;
        fast_two_sum(a, b, r.hi, r.lo);
        return r;
    }

    // ---- arithmetic
    friend __device__ __forceinline__ df64 operator-(df64 a) { return df64(-a.hi, -a.lo); }
    friend __device__ __forceinline__ df64 operator+(df64 a, df64 b) {
        float s, e, t, f;
        two_sum(a.hi, b.hi, s, e);
        two_sum(a.lo, b.lo, t, f);
        e = __fadd_rn(e, t);
        fast_two_sum(s, e, s, e);
        e = __fadd_rn(e, f);
        return norm(s, e);
    }
    friend __device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }
    friend __device__ __forceinline__ df64 operator*(df64 a, df64 b) {
        const float p = __fmul_rn(a.hi, b.hi);
        float e = __fmaf_rn(a.hi, b.hi, -p);
        e = __fmaf_rn(a.hi, b.lo, e);
        e = __fmaf_rn(a.lo, b.hi, e);
        return norm(p, e);
    }
    // Three quotient digits from one reciprocal r of b.hi: each digit is the remainder's high part times
    // r, and the remainder a - q b stays a pair (the high parts' difference is exact: q b.hi is within
    // a few units in the last place of what it is subtracted from).  A third of the instructions of
    // three FP32 divisions with double-word remainders, to the same few units of 2^-48, for |b| in
    // [2^-126, 2^126] and a remainder that FP32 holds (|a| >= 2^-100).  Smaller |b|: the reciprocal is infinite and
    // the quotient not a number, which callers keep away from (reflectors scale their column, Sturm
    // counts replace small pivots).
    friend __device__ __forceinline__ df64 operator/(df64 a, df64 b) {
        const float r = __frcp_rn(b.hi);
        const float q1 = __fmul_rn(a.hi, r);
        // remainder a - q1 b = h + l
        float h = __fmaf_rn(-q1, b.hi, a.hi), l = __fmaf_rn(-q1, b.lo, a.lo);
        fast_two_sum_any(h, l);
        const float q2 = __fmul_rn(h, r);
        const float q3 = __fmul_rn(__fadd_rn(__fmaf_rn(-q2, b.hi, h), __fmaf_rn(-q2, b.lo, l)), r);
        float s, e;
        fast_two_sum(q1, q2, s, e);
        return norm(s, __fadd_rn(e, q3));
    }
    // a b + c with a single renormalisation (the accumulation form of the GEMM kernels)
    friend __device__ __forceinline__ df64 fma(df64 a, df64 b, df64 c) {
        const float p = __fmul_rn(a.hi, b.hi);
        float e = __fmaf_rn(a.hi, b.hi, -p);
        e = __fmaf_rn(a.hi, b.lo, e);
        e = __fmaf_rn(a.lo, b.hi, e);
        float s, t;
        two_sum(c.hi, p, s, t);
        t = __fadd_rn(t, __fadd_rn(c.lo, e));
        return norm(s, t);
    }
    friend __device__ __forceinline__ df64 sqrt(df64 a) {
        if (!(a.hi > 0.f)) return df64(__fsqrt_rn(a.hi), 0.f);  // 0 -> 0, negative -> NaN
        const float s = __fsqrt_rn(a.hi);
        const float p = __fmul_rn(s, s);
        const float e = __fmaf_rn(s, s, -p);
        const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), e), a.lo);
        return norm(s, __fdiv_rn(r, __fmul_rn(2.f, s)));
    }
    friend __device__ __forceinline__ df64 fabs(df64 a) { return a.hi < 0.f ? -a : a; }
    friend __device__ __forceinline__ df64 copysign(df64 a, df64 b) {
        return (signbit(a.hi) != signbit(b.hi)) ? -a : a;
    }

    // ---- comparisons (normalised pairs compare lexicographically)
    friend __device__ __forceinline__ bool operator<(df64 a, df64 b) {
        return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
    }
    friend __device__ __forceinline__ bool operator>(df64 a, df64 b) { return b < a; }
    friend __device__ __forceinline__ bool operator<=(df64 a, df64 b) { return !(b < a) && a.hi == a.hi && b.hi == b.hi; }
    friend __device__ __forceinline__ bool operator>=(df64 a, df64 b) { return b <= a; }
    friend __device__ __forceinline__ bool operator==(df64 a, df64 b) { return a.hi == b.hi && a.lo == b.lo; }
    friend __device__ __forceinline__ bool operator!=(df64 a, df64 b) { return !(a == b); }
    friend __device__ __forceinline__ df64 fmax(df64 a, df64 b) { return (a < b) ? b : a; }
    friend __device__ __forceinline__ df64 fmin(df64 a, df64 b) { return (b < a) ? b : a; }

    friend __device__ __forceinline__ df64 &operator+=(df64 &a, df64 b) { return a = a + b; }
    friend __device__ __forceinline__ df64 &operator-=(df64 &a, df64 b) { return a = a - b; }
    friend __device__ __forceinline__ df64 &operator*=(df64 &a, df64 b) { return a = a * b; }
    friend __device__ __forceinline__ df64 &operator/=(df64 &a, df64 b) { return a = a / b; }

    // ---- warp exchange
    friend __device__ __forceinline__ df64 __shfl_xor_sync(unsigned mask, df64 v, int m) {
        return df64(__shfl_xor_sync(mask, v.hi, m), __shfl_xor_sync(mask, v.lo, m));
    }
    friend __device__ __forceinline__ df64 __shfl_sync(unsigned mask, df64 v, int src) {
        return df64(__shfl_sync(mask, v.hi, src), __shfl_sync(mask, v.lo, src));
    }
};

static_assert(sizeof(df64) == 8, "df64 is two floats");

// The same pair with the "sloppy" double-word sum (one TwoSum on the high parts, the low parts
// added, one renormalisation: 11 instead of 20 FP32 operations).  Its error is bounded by a few
// units of 2^-48 of |a| + |b| rather than of |a + b|: enough wherever the error analysis is
// norm-wise, as in the butterflies of an FFT, whose outputs carry errors relative to the
// transform's norm anyway.  Multiplication and the conversions are df64's.
struct alignas(8) df64f {
    float hi, lo;

    df64f() = default;
    __host__ __device__ __forceinline__ df64f(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ __forceinline__ df64f(float f) : hi(f), lo(0.f) {}
    __host__ __device__ __forceinline__ df64f(int i) : df64f((double)i) {}
    __host__ __device__ __forceinline__ df64f(double d) {
#ifdef __CUDA_ARCH__
        double_to_pair(d, hi, lo);
#else
        hi = (float)d;
        lo = (float)(d - (double)hi);
#endif
    }
    __host__ __device__ __forceinline__ explicit operator double() const {
#ifdef __CUDA_ARCH__
        return pair_to_double(hi, lo);
#else
        return (double)hi + (double)lo;
#endif
    }

    friend __device__ __forceinline__ df64f operator-(df64f a) { return df64f(-a.hi, -a.lo); }
    friend __device__ __forceinline__ df64f operator+(df64f a, df64f b) {
        float s, e;
        df64::two_sum(a.hi, b.hi, s, e);
        e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
        df64f r;
        df64::fast_two_sum(s, e, r.hi, r.lo);
        return r;
    }
    friend __device__ __forceinline__ df64f operator-(df64f a, df64f b) { return a + (-b); }
    friend __device__ __forceinline__ df64f operator*(df64f a, df64f b) {
        const float p = __fmul_rn(a.hi, b.hi);
        float e = __fmaf_rn(a.hi, b.hi, -p);
        e = __fmaf_rn(a.hi, b.lo, e);
        e = __fmaf_rn(a.lo, b.hi, e);
        df64f r;
        df64::fast_two_sum(p, e, r.hi, r.lo);
        return r;
    }
    friend __device__ __forceinline__ df64f &operator+=(df64f &a, df64f b) { return a = a + b; }
    friend __device__ __forceinline__ df64f &operator-=(df64f &a, df64f b) { return a = a - b; }
    friend __device__ __forceinline__ df64f &operator*=(df64f &a, df64f b) { return a = a * b; }
};

static_assert(sizeof(df64f) == 8, "df64f is two floats");

}  // namespace lg
