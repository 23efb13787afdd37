// 64-bit fixed-point arithmetic shared by the GKB products (fx.cu) and the
// reconstruction (evaluate.cu): rounding of FP64 values at a common scale, balanced
// 21-bit limbs and exact limb products.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

constexpr int FX_NONFINITE = 2047;  // exponent field of Inf and NaN

__device__ __forceinline__ int fx_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7FF8000000000000LL); }

// round(x 2^s) for |x| 2^s < 2^62 (s = 1084 - E with E at least the exponent
// field of x and at least 1); 0 for a non-finite x (flagged by E = 2047).
// Normal x: integer operations on the significand (the FP64 pipe is not used).
__device__ __forceinline__ long long fx_round(double x, int s) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    if (e == 0x7FF) return 0;
    long long q;
    if (e == 0) {
        if ((b << 1) == 0) return 0;                // +-0
        q = __double2ll_rn(ldexp(fabs(x), s));      // subnormal: exact scaling, one rounding
    } else {
        const long long m = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;  // 53-bit significand
        const int d = 1075 - e - s;                 // |x| 2^s = m 2^-d with d >= -9
        if (d <= 0) q = m << (-d);
        else if (d > 54) q = 0;
        else q = (m + (1LL << (d - 1))) >> d;       // round half up
    }
    return b < 0 ? -q : q;
}

// Balanced 21-bit limbs of a vector value: q = z2 2^42 + z1 2^21 + z0 with
// z0, z1 in [-2^20, 2^20) and |z2| <= 2^20 + 1 (|q| < 2^62).
__device__ __forceinline__ int4 fx_limbs_bal(long long q) {
    const int z0 = (int)((q << 43) >> 43);
    q = (q - z0) >> 21;
    const int z1 = (int)((q << 43) >> 43);
    q = (q - z1) >> 21;
    return make_int4(z0, z1, (int)q, 0);
}

__device__ __forceinline__ long long imad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// acc += N * Z over the limb products of weight >= 2^42: N's limbs are its
// bit fields (a0, a1 in [0, 2^21), a2 = N >> 42 signed), Z's the balanced ones.
struct FxAcc {
    long long c2 = 0, c1 = 0, c0 = 0;  // weights 2^84, 2^63, 2^42
    __device__ __forceinline__ void add(long long N, int z0, int z1, int z2) {
        const unsigned lo = (unsigned)N, hi = (unsigned)(N >> 32);
        const int a0 = (int)(lo & 0x1FFFFFu);
        const int a1 = (int)(__funnelshift_r(lo, hi, 21) & 0x1FFFFFu);
        const int a2 = (int)hi >> 10;
        c2 = imad_wide(a2, z2, c2);
        c1 = imad_wide(a2, z1, c1);
        c1 = imad_wide(a1, z2, c1);
        c0 = imad_wide(a2, z0, c0);
        c0 = imad_wide(a1, z1, c0);
        c0 = imad_wide(a0, z2, c0);
    }
    // the accumulated value in units of 2^42, rounded to FP64
    __device__ __forceinline__ double value() const {
        return fma((double)c2, 0x1p42, fma((double)c1, 0x1p21, (double)c0));
    }
};
