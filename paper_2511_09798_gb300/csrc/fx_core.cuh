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

// Sum of products N Z, both split into a high and a signed 32-bit low part, |N| <
// 2^61 and |Z| < 2^62 (so |n1| <= 2^29 and |z1| <= 2^30).  n1 z1 goes to c (units of
// 2^64), which holds FX_FOLD terms of at most 2^59 + 2^32 before it is folded; the
// cross products, below 2^62 together and made positive by FX_BIAS, add their
// upper word to c and carry their lower word into the next term and, after the
// last, into the result.  n0 z0 is left out: an error of at most a quarter of a
// unit of 2^64 per term, of either sign (a twelfth in the root mean square).  What
// that is relative to a term depends on how large N and Z are: 2^-61 for N = 2^61
// and Z = 2^62, 2^-52 for N = 2^53 and Z = 2^61.  Three wide
// products per term where 21-bit limbs that accumulate without folds take six:
// those bound the reconstruction of 8 vectors (the pipe of the wide products 63 %
// busy): 816 -> 608 us for 150 vectors, 8000 nodes and 500 points, 1.70 -> 1.59 ms
// for one vector and 20 000 nodes and points (a fourth for the upper half of n0 z0
// 1.68 ms, and a solve with 2161 rows and 140 steps 8.94 -> 9.28 ms).  (16 vectors
// per CTA: no gain, 12 warps per SM.)
constexpr int FX_FOLD = 8;
constexpr unsigned FX_BIAS = 1u << 30;  // in the upper word
constexpr int FX_UNIT = 44;             // the result's low part is in units of 2^FX_UNIT

struct FxAcc32 {
    long long c = 0, hi = 0, lo = 0;  // value c + hi 2^32 + lo
    unsigned rem = 0;
    __device__ __forceinline__ void add(int n1, int n0, int z1, int z0) {
        const long long x =
            imad_wide(n0, z1, imad_wide(n1, z0, (long long)(((unsigned long long)FX_BIAS << 32) | rem)));
        rem = (unsigned)x;
        c = imad_wide(n1, z1, c) + (long long)((unsigned long long)x >> 32);
    }
    __device__ __forceinline__ void fold() {
        hi += c >> 32;
        lo += (long long)((unsigned long long)c & 0xffffffffu);
        c = 0;
    }
    // (folded) the sum of up to 2^12 terms as h 2^96 + l 2^FX_UNIT; such pairs add
    __device__ __forceinline__ longlong2 pair(int64_t terms) const {
        return make_longlong2(hi, ((lo - terms * (long long)FX_BIAS) << (64 - FX_UNIT)) | (rem >> (FX_UNIT - 32)));
    }
    // a pair in units of 2^FX_UNIT
    static __device__ __forceinline__ double value(longlong2 p) {
        return fma((double)p.x, 0x1p52, (double)p.y);
    }
};

__device__ __forceinline__ int2 fx_split(long long v) {  // (low, high) with a signed low part
    const int l = (int)v;
    return make_int2(l, (int)(v >> 32) - (l >> 31));
}
