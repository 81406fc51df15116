// Fixed-point factor entries of the double-precision selections (select_fx.cu, select_single.cu; the format and why it
// holds what FP64 holds: select_fx.cu).
#pragma once

#include "sic_internal.cuh"

constexpr int FXS = 58;  // fixed point: 2^FXS stands for 2^e (factor entries) or 2^(2e) (products)

// the format's exponent: 1.9 2^(2e) >= variance + nugget
static inline int fx_exponent(const sic_kernel* kp) {
    int e2 = 0;
    frexp((kp->variance + kp->nugget) / 1.9, &e2);  // (variance + nugget) / 1.9 < 2^e2
    return e2 >= 0 ? (e2 + 1) / 2 : -((-e2) / 2);
}

__device__ __forceinline__ int2 fx_split(long long x) {
    const int h = (int)((x + (1LL << 28)) >> 29);
    return make_int2(h, (int)(x - ((long long)h << 29)));
}

// round(x 2^sh), x >= 0 finite (0 below the resolution); integer operations only
__device__ __forceinline__ long long fx_of_positive(double x, int sh) {
    const long long u = __double_as_longlong(x);
    const int s = (int)(u >> 52) - 1075 + sh;  // x = mant 2^(E - 1075)
    const long long mant = (u & 0xfffffffffffffLL) | 0x10000000000000LL;
    if (s >= 0) return mant << s;
    return s > -55 ? ((mant >> (-s - 1)) + 1) >> 1 : 0LL;
}

// x 2^e2 in FP64 (significand rounded to nearest, ties away), integer operations only
__device__ __forceinline__ double fx_to_double(long long x, int e2) {
    if (x == 0) return 0.0;
    const unsigned long long sg = (unsigned long long)x & (1ULL << 63);
    const unsigned long long mag = x < 0 ? 0ULL - (unsigned long long)x : (unsigned long long)x;
    const int z = __clzll((long long)mag);
    const unsigned long long m = (((mag << z) >> 10) + 1ULL) >> 1;  // 53 bits, or 2^53 after rounding
    // the significand's leading bit (or the carry to 2^53) adds to the exponent field
    return __longlong_as_double((long long)(sg | ((((unsigned long long)(e2 + 63 - z + 1022)) << 52) + m)));
}

// multiplier and shift of a positive FP64 factor r: fx_mul(n, M) 2^s = n r 2^e, for |n| <= 2^59
__device__ __forceinline__ void fx_factor(double r, int e, long long& M, int& s) {
    const long long u = __double_as_longlong(r);
    M = (((u & 0xfffffffffffffLL) | 0x10000000000000LL)) << 9;
    s = (int)((u >> 52) & 0x7ff) - 1023 + e - 1;
}
__device__ __forceinline__ long long fx_mul(long long n, long long M, int s) {
    const long long p = __mul64hi(n << 4, M);
    return s >= 0 ? p << s : (p + (1LL << (-s - 1))) >> -s;  // s >= -2: r^2 >= 2^(-2e) / 1.9
}

// binary exponent of x (-1023 for zero); integer operations only
__device__ __forceinline__ int exponent_of(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

// covariances with the target below 2^(2e - FX_COV_BITS) are selected with FP64 rows (select_fx.cu)
constexpr int FX_COV_BITS = 30;

__device__ __forceinline__ bool not_finite(double x) {
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}

struct FxSum {
    long long hh, cr;
    __device__ __forceinline__ void add(int2 a, int2 b) {
        hh += (long long)a.x * b.x;
        cr += (long long)a.x * b.y + (long long)a.y * b.x;
    }
    __device__ __forceinline__ void add2(int4 a, int4 b) {
        add(make_int2(a.x, a.y), make_int2(b.x, b.y));
        add(make_int2(a.z, a.w), make_int2(b.z, b.w));
    }
    __device__ __forceinline__ long long value() const { return hh + (cr >> 29); }
};

// ---- 60 bits: factors that are themselves the result (fill_columns.cu) ----

constexpr int FCS = 60;  // 2^FCS stands for 2^e (factor entries) or 2^(2e) (products)

__device__ __forceinline__ int2 fc_split(long long x) {
    const int h = (int)((x + (1LL << 29)) >> 30);  // |h| < 2^30.5, |l| <= 2^29
    return make_int2(h, (int)(x - ((long long)h << 30)));
}
// sum of products: up to 48 terms of a row keep every word below 2^63 (the entries' squares sum to at most
// 1.9 2^(2 FCS))
struct FcSum {
    long long hh, c1, c2;
    __device__ __forceinline__ void add(int2 a, int2 b) {
        hh += (long long)a.x * b.x;
        c1 += (long long)a.x * b.y;
        c2 += (long long)a.y * b.x;
    }
    __device__ __forceinline__ void add2(int4 a, int4 b) {
        add(make_int2(a.x, a.y), make_int2(b.x, b.y));
        add(make_int2(a.z, a.w), make_int2(b.z, b.w));
    }
    __device__ __forceinline__ long long value() const { return hh + (((c1 >> 2) + (c2 >> 2)) >> 28); }
};
// round(n r 2^e) for r by fc_pivot, |n| < 2^61: the top of the 128-bit product
__device__ __forceinline__ long long fc_mul(long long n, long long M, int h) {
    const long long a = n << 1, hi = __mul64hi(a, M);  // hi 2^64 + lo = n M 2
    const unsigned long long lo = (unsigned long long)a * (unsigned long long)M;
    const int s = h + 3;  // n M 2^-63 2^s, s >= 1
    return (hi << s) | (long long)(lo >> (64 - s));
}

// Multiplier M (60 bits) and shift h of r = d^(-1/2), fc_mul's, for the pivot d = dj 2^(2e - FCS), dj > 0: an FP32
// reciprocal square root of the normalised pivot, one Newton step in double-float (2^-42), one on the residual
// 1 - d r^2 formed in integers (2^-61).  No FP64 operation (a chain of them takes 64 cycles each).  A factor rounded to
// FP64 would put an update F_i F_l off by 2^-52 of itself, 2e-16 of the variance in the first columns, whatever the
// products' exactness.
__device__ __forceinline__ void fc_pivot(long long dj, long long& M, int& h) {
    const int z = __clzll(dj) - 1;
    const unsigned long long D = (unsigned long long)dj << z;  // [2^62, 2^63)
    const int odd = z & 1;
    h = ((z + 1) >> 1) - 3;
    // X = D 2^-62 (z even) or twice that: [1, 4), in two floats
    const float xh = (float)(int)(D >> 39) * __uint_as_float((unsigned)(127 - 23 + odd) << 23);
    const float xl = (float)(int)((D >> 15) & 0xffffffULL) * __uint_as_float((unsigned)(127 - 47 + odd) << 23);
    const float y = rsqrtf(xh);  // (0.5, 1]
    const float y2 = __fmul_rn(y, y);
    const float y2e = __fmaf_rn(y, y, -y2);
    const float p = __fmul_rn(xh, y2);
    const float pe = __fmaf_rn(xh, y2, -p);
    const float e0 = __fmaf_rn(-xl, y2, __fmaf_rn(-xh, y2e, __fsub_rn(__fsub_rn(1.f, p), pe)));
    const float c = __fmul_rn(0.5f * y, e0);
    const unsigned yb = __float_as_uint(y);
    const long long TOP = (1LL << 62) - 1;
    long long m = ((long long)((yb & 0x7fffffu) | 0x800000u) << (38 + (int)(yb >> 23) - 126)) +
                  ((long long)__float2int_rn(c * 0x1p50f) << 12);  // r 2^62, off by 2^-42
    m = m < TOP ? m : TOP;
    const unsigned long long t = __umul64hi(D << 1, (unsigned long long)m << 2);  // D m 2^-61
    const unsigned long long hi = __umul64hi(t, (unsigned long long)m), lo = t * (unsigned long long)m;
    // 2^K (1 - E): K = 125 - odd; R = E 2^71, below 2^31 in magnitude
    const unsigned long long rl = 0ULL - lo, rh = (1ULL << (61 - odd)) - hi - (lo ? 1ULL : 0ULL);
    const int R = odd ? (int)((rh << 11) | (rl >> 53)) : (int)((rh << 10) | (rl >> 54));
    m += __float2int_rn((float)R * y * 0x1p-10f);  // m E / 2
    M = m < TOP ? m : TOP;
}

// FP32 value (truncated) of a double scaled by 2^-off, by its bits; 0 below FP32's range and for
// negative values
__device__ __forceinline__ float fx_f32(double x, int off) {
    const unsigned H = (unsigned)__double2hiint(x), L = (unsigned)__double2loint(x);
    const int e = (int)((H >> 20) & 0x7ffu) - 896 - off;
    if (e <= 0 || (int)H < 0) return 0.f;
    return e >= 255 ? INFINITY : __uint_as_float(((unsigned)e << 23) | ((H & 0xfffffu) << 3) | (L >> 29));
}
