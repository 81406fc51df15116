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

// FP32 value (truncated) of a double scaled by 2^-off, by its bits; 0 below FP32's range and for
// negative values
__device__ __forceinline__ float fx_f32(double x, int off) {
    const unsigned H = (unsigned)__double2hiint(x), L = (unsigned)__double2loint(x);
    const int e = (int)((H >> 20) & 0x7ffu) - 896 - off;
    if (e <= 0 || (int)H < 0) return 0.f;
    return e >= 255 ? INFINITY : __uint_as_float(((unsigned)e << 23) | ((H & 0xfffffu) << 3) | (L >> 29));
}
