// Projected SVD of the lower-bidiagonal C_l ((l+1) x l) of Algorithms 2 and 4:
// C_l = U~ S~ V~^T, f~ = U~^T (beta_1 e_1).
//
// On GB300 a dependent FP64 operation costs ~64 cycles (FP64 division ~640), so
// a sequential bidiagonal QR sweep would take tens of milliseconds.  This
// implementation instead works on the Golub-Kahan tridiagonal T (order 2l+1,
// zero diagonal, off-diagonal alpha_1, beta_2, alpha_2, ..., alpha_l, beta_{l+1},
// eigenvalues +-s~_i and 0, eigenvectors (u~_i, v~_i interleaved)/sqrt(2)),
// which exposes parallelism over the singular values:
//
//  1. k_tgk_bisect  32 or 8 lanes per singular value: brackets in the IEEE bit
//     pattern of the shift (nearly geometric for positive doubles), Sturm counts
//     from the division-free three-term recurrence of the leading principal
//     minors with power-of-two rescaling; an FP32 guess and secant steps on the
//     determinant place the sample points.  Ends at adjacent doubles.
//  2. k_tgk_vectors one warp per singular value: twisted factorization
//     (top-down and bottom-up LDL^T of T - s I, twist where |gamma| is
//     smallest) gives the eigenvector without iteration; the pivots are ratios
//     of the minors.
//  3. k_tgk_clusters one warp per cluster of close singular values (relative
//     gap < cluster_tol; as many CTAs as needed for one cluster per warp):
//     three steps of inverse iteration with the stored
//     factorizations, all members in parallel lanes, Gram-Schmidt in order
//     (the scheme of LAPACK's dstein), so the cluster basis is orthonormal.
//  4. k_tgk_finalize split into u~ and v~, normalise, f~_i = beta_1 u~_i[0];
//     f~_{l+1} = beta_1 / |u| with u the null vector of C^T (u_1 = 1,
//     u_{j+1} = -alpha_j u_j / beta_{j+1}), accumulated in log space.
// Every result is FP64; the FP32 counts, secant roots and square roots only place the
// points at which the FP64 counts are taken.
#include <cfloat>

#include "common.cuh"
#include "internal.h"

namespace {

constexpr int BS_WARPS = 4;
constexpr int SVD_MAX_L = 8192;  // bidiagonal dimension (shared memory: 2 L doubles and 2 L floats)

__device__ __forceinline__ int proj_l(const ProjDims& d, int b) { return d.l_arr ? d.l_arr[b] : d.l; }

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double bitsd(long long b) { return __longlong_as_double(b); }

// Normalised off-diagonal of T: e_{2m} = alpha_{m+1}, e_{2m+1} = beta_{m+2}; / bound.
__device__ void load_e(const double* __restrict__ alpha, const double* __restrict__ beta, int l,
                       double* e, double* bound_out) {
    __shared__ double red[32];
    const int ne = 2 * l;
    for (int k = threadIdx.x; k < ne; k += blockDim.x) e[k] = (k & 1) ? beta[(k >> 1) + 1] : alpha[k >> 1];
    __syncthreads();
    double b = 0.0;
    for (int k = threadIdx.x; k < ne; k += blockDim.x) {
        double g = fabs(e[k]) + (k + 1 < ne ? fabs(e[k + 1]) : 0.0);
        b = fmax(b, g);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b = fmax(b, __shfl_xor_sync(RBF_FULL_MASK, b, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = b;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, red[w]);
        red[0] = t > 0.0 ? t : 1.0;
    }
    __syncthreads();
    const double bound = red[0];
    const double inv = 1.0 / bound;
    for (int k = threadIdx.x; k < ne; k += blockDim.x) e[k] *= inv;
    __syncthreads();
    *bound_out = bound;
}

// power of two that brings max(|a|, |b|) near 1 (integer ops on the exponents)
__device__ __forceinline__ double rescale_factor(double a, double b) {
    int ea = (__double2hiint(a) >> 20) & 0x7ff;
    int eb = (__double2hiint(b) >> 20) & 0x7ff;
    int e = max(ea, eb);                 // biased exponent of the larger
    int t = 2046 - e;                    // biased exponent of 2^-(e - 1023)
    t = max(1, min(2046, t));
    return __hiloint2double(t << 20, 0);
}

__device__ __forceinline__ bool is_zero(double p) {  // integer test: DSETP would take an FP64 slot
    return (((unsigned)__double2hiint(p) << 1) | (unsigned)__double2loint(p)) == 0;
}

// -2^-996 v with its exponent field kept at 24 or above: stands in for a zero
// minor that follows v (counts as a negative pivot).
__device__ __forceinline__ double tiny_after(double v) {
    const unsigned h = (unsigned)__double2hiint(v);
    const int e = max((int)((h >> 20) & 0x7ffu) - 996, 24);
    return __hiloint2double((int)(((h ^ 0x80000000u) & 0x800fffffu) | ((unsigned)e << 20)), 0);
}

// One step of the leading principal minors of T - x I: p_{k+1} = -x p_k -
// e_{k-1}^2 p_{k-1}.  Two FP64 instructions, one of them on the chain.
__device__ __forceinline__ double minor_raw(double x, double pm1, double pm2, double e2) {
    return fma(-x, pm1, -(e2 * pm2));
}
__device__ __forceinline__ double minor_step(double x, double pm1, double pm2, double e2) {
    const double p = minor_raw(x, pm1, pm2, e2);
    return is_zero(p) ? tiny_after(pm1) : p;
}

// Eight steps from (pm2, pm1) with e2[dir u], u = 0..7, each minor passed to
// put(u, p); returns the sign changes.  A zero minor inside the group needs no
// care as long as the next coupling is not zero: the minors around it differ in
// sign, so either sign of the zero gives the one change that a tiny negative
// pivot gives.  Otherwise all later ones are zero, which the last one shows, and
// the group is taken again with tiny_after in the zeros' places: no test on the
// chain of the usual case.
template <typename Put>
__device__ __forceinline__ int minor_group(const double* __restrict__ e2, int dir, double x, double& pm2, double& pm1,
                                           Put put) {
    double a = pm2, c = pm1;
    int neg = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const double p = minor_raw(x, c, a, e2[dir * u]);
        neg += (int)(sign_bit(p) ^ sign_bit(c));
        put(u, p);
        a = c;
        c = p;
    }
    if (is_zero(c)) {
        a = pm2;
        c = pm1;
        neg = 0;
#pragma unroll 1
        for (int u = 0; u < 8; ++u) {
            const double p = minor_step(x, c, a, e2[dir * u]);
            neg += (int)(sign_bit(p) ^ sign_bit(c));
            put(u, p);
            a = c;
            c = p;
        }
    }
    pm2 = a;
    pm1 = c;
    return neg;
}

// number of eigenvalues of the normalised T below x > 0; *det, *dexp: det(T -
// x I) = det 2^dexp
__device__ __forceinline__ int sturm_count(const double* __restrict__ e2, int nt, double x, double* det,
                                           int* dexp) {
    double pm2 = 1.0, pm1 = -x;
    int neg = 1;  // d_0 = -x < 0
    int ex = 0;
    int k = 1;
    for (; k + 7 < nt; k += 8) {
        neg += minor_group(e2 + (k - 1), 1, x, pm2, pm1, [](int, double) {});
        const double f = rescale_factor(pm1, pm2);
        ex += 1023 - (__double2hiint(f) >> 20);
        pm1 *= f;
        pm2 *= f;
    }
    for (; k < nt; ++k) {
        const double p = minor_step(x, pm1, pm2, e2[k - 1]);
        neg += (int)(sign_bit(p) ^ sign_bit(pm1));
        pm2 = pm1;
        pm1 = p;
    }
    *det = pm1;
    *dexp = ex;
    return neg;
}

// The same count in FP32, rescaled every second step (every fourth underflows
// on graded bidiagonals: l = 1000 1.42 -> 2.62 ms): exact for a matrix whose
// entries differ from T's by a few FP32 roundings, unless a minor underflows.
// Used for a first guess only.
__device__ __forceinline__ int sturm_count_f32(const float* __restrict__ e2, int nt, float x) {
    float pm2 = 1.f, pm1 = -x;
    int neg = 1;
    auto step = [&](float e) {
        const float p = fmaf(-x, pm1, -(e * pm2));
        neg += (int)((__float_as_uint(p) ^ __float_as_uint(pm1)) >> 31);
        pm2 = pm1;
        pm1 = p;
    };
    int k = 1;
#pragma unroll 2
    for (; k + 1 < nt; k += 2) {
        step(e2[k - 1]);
        step(e2[k]);
        const int e = __float_as_int(fmaxf(fabsf(pm1), fabsf(pm2))) & 0x7f800000;
        const float f = __int_as_float(min(0x7f000000 - e, 0x7e800000));  // 2^-(exponent), at most 2^126
        pm1 *= f;
        pm2 *= f;
    }
    if (k < nt) step(e2[k - 1]);
    return neg;
}

// Singular value i (descending) as the m-th positive eigenvalue of T, m = l -
// 1 - i from below, LPV lanes per value.  The bracket [lo, hi) holds count(lo)
// <= m < count(hi) throughout, in the order of the doubles' bit patterns, and
// ends at adjacent doubles; only the choice of the sample points varies:
//   - a multisection with FP32 counts from [2^-90, 1] to a few FP32 ulps;
//   - one FP64 round with points at geometric distances 2^-22 .. 2^-7
//     (relative) on both sides of that guess, which brackets the value to about
//     2^-20 when the guess is good and leaves a valid, wider bracket otherwise;
//   - then, while the bracket holds one eigenvalue, points at geometric
//     distances from the secant root of det(T - x I) (its error is quadratic in
//     the bracket's width), otherwise, and after a secant round that gained
//     little, an even multisection.
// The FP64 counts bound the kernel: 2 n_t FP64 instructions of 64 cycles per
// round and warp.  About 4 FP64 rounds with 32 lanes (6 with 8) replace the 12
// to 14 of an even multisection of the whole range (kernel times): l = 150 668 -> 147
// us, l = 3001 84.5 -> 5.7 ms.  LPV = 32 takes the fewest rounds, 8 the fewest counts (the
// launcher chooses by the number of values).
constexpr int BI_ROUNDS = 64;

template <int LPV>
__global__ void k_tgk_bisect(ProjDims d, const double* __restrict__ alpha_all,
                             const double* __restrict__ beta_all, double* __restrict__ sigma_all,
                             double* __restrict__ bound_all) {
    extern __shared__ double sh[];
    constexpr int VPW = 32 / LPV, H = LPV / 2;  // values per warp, points per side
    const int b = blockIdx.y;
    const int l = proj_l(d, b);
    if (l < 1) return;
    const double* alpha = alpha_all + (size_t)b * d.L;
    const double* beta = beta_all + (size_t)b * (d.L + 1);
    double* sigma = sigma_all + (size_t)b * d.L;
    double* e2 = sh;                      // [2l] the normalised off-diagonal, squared in place
    float* e2f = (float*)(sh + 2 * l);    // [2l] its FP32 copy
    const int nwarp = blockDim.x >> 5;
    if (blockIdx.x * nwarp * VPW >= l) return;
    double bound;
    load_e(alpha, beta, l, e2, &bound);
    for (int k = threadIdx.x; k < 2 * l; k += blockDim.x) {
        const double t = e2[k] * e2[k];
        e2[k] = t;
        e2f[k] = (float)t;
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) bound_all[b] = bound;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane / LPV, g = lane % LPV;  // value of the warp, point of the value
    const int i0 = (blockIdx.x * nwarp + warp) * VPW;
    if (i0 >= l) return;
    const int i = i0 + grp;                      // descending index
    const bool live = i < l;
    const int m = live ? l - 1 - i : 0;          // ascending rank
    const int nt = 2 * l + 1;
    const unsigned gmask = LPV == 32 ? 0xffffffffu : ((1u << LPV) - 1u) << (grp * LPV);
    const int first = grp * LPV;                 // the group's first lane
    // ---- FP32 guess
    int flo = __float_as_int(0x1p-90f), fhi = __float_as_int(1.001f);
    while (__any_sync(RBF_FULL_MASK, fhi - flo > 4)) {
        const int dd = fhi - flo;
        const int xb = dd >= LPV + 1 ? flo + (int)(((long long)dd * (g + 1)) / (LPV + 1)) : flo + min(g + 1, dd - 1);
        const int cnt = sturm_count_f32(e2f, nt, __int_as_float(xb)) - (l + 1);
        const unsigned above = __ballot_sync(RBF_FULL_MASK, cnt > m) & gmask;
        const int f = above ? __ffs(above) - 1 : first + LPV - 1;
        const int xf = __shfl_sync(RBF_FULL_MASK, xb, f);
        const int xp = __shfl_sync(RBF_FULL_MASK, xb, max(f - 1, first));
        if (dd > 4) {
            if (above == 0) {
                flo = xf;
            } else {
                if (f > first) flo = xp;
                fhi = xf;
            }
        }
    }
    // ---- FP64 bracket
    long long lo = 0, hi = dbits(1.0 + 1.0 / 1024.0);
    int clo = -1, chi = -1;          // counts at lo, hi (valid with their dets), -1: not sampled
    double dlo = 0.0, dhi = 0.0;     // det mantissas and exponents there
    int xlo = 0, xhi = 0;
    bool secant = false;
    const double guess = (double)__int_as_float(flo + (fhi - flo) / 2);
    for (int round = 0; round < BI_ROUNDS; ++round) {
        const long long dd = hi - lo;
        const bool open = live && dd > 1;
        if (!__any_sync(RBF_FULL_MASK, open)) break;
        long long xb;
        secant = round > 0 && !secant && dd > LPV && clo >= 0 && chi == clo + 1;
        if (round == 0) {
            const int q = g < H ? H - 1 - g : g - H;  // 0 .. H-1 outwards
            const double rel = (double)exp2f(-22.f + 15.f * (float)q / (float)(H - 1));
            xb = dbits(g < H ? guess - guess * rel : guess + guess * rel);
        } else if (secant) {
            // root of the secant through (lo, det) and (hi, det), in FP32
            // relative to the bracket; points at distances of 2^-step, 2^-2 step, ... of each side
            const float r = (float)(fabs(dhi) / fabs(dlo)) * exp2f((float)max(-120, min(120, xhi - xlo)));
            const float t = 1.f / (1.f + r);
            long long sb = lo + (long long)((double)t * (double)dd);
            sb = max(lo + 1, min(hi - 1, sb));
            const float A = (float)(sb - lo), C = (float)(hi - sb);
            constexpr float STEP = LPV == 32 ? 2.f : 4.f;
            if (g < H) xb = sb - (long long)(A * exp2f(-STEP * (float)(g + 1) + STEP * 0.75f));
            else xb = sb + 1 + (long long)(C * exp2f(-STEP * (float)(LPV - g) + STEP * 0.75f));
        } else if (dd >= LPV + 1) {
            xb = lo + (dd / (LPV + 1)) * (g + 1);
        } else {
            xb = lo + min((long long)(g + 1), dd - 1);
        }
        xb = max(lo + 1, min(hi - 1, xb));
        double det;
        int ex;
        const int cnt = sturm_count(e2, nt, bitsd(max(xb, 1LL)), &det, &ex) - (l + 1);
        const unsigned above = __ballot_sync(RBF_FULL_MASK, cnt > m) & gmask;
        const int f = above ? __ffs(above) - 1 : first + LPV;  // first lane above, or past the group
        const int up = min(f, first + LPV - 1), dn = max(f - 1, first);
        const long long xu = __shfl_sync(RBF_FULL_MASK, xb, up), xd = __shfl_sync(RBF_FULL_MASK, xb, dn);
        const double du = __shfl_sync(RBF_FULL_MASK, det, up), de = __shfl_sync(RBF_FULL_MASK, det, dn);
        const int eu = __shfl_sync(RBF_FULL_MASK, ex, up), ee = __shfl_sync(RBF_FULL_MASK, ex, dn);
        const int cu = __shfl_sync(RBF_FULL_MASK, cnt, up), cd = __shfl_sync(RBF_FULL_MASK, cnt, dn);
        if (open) {
            if (above && f < first + LPV) {
                hi = xu;
                dhi = du;
                xhi = eu;
                chi = cu;
            }
            if (f > first) {
                lo = xd;
                dlo = de;
                xlo = ee;
                clo = cd;
            }
            // a secant round is followed by another one only after a gain of at least 2^8
            if (secant && (hi - lo) < (dd >> 8)) secant = false;
        }
    }
    if (live && g == 0) sigma[i] = 0.5 * (bitsd(lo) + bitsd(hi)) * bound;
}

// Eigenvector of the normalised T for s = sigma_i / bound by the twisted
// factorization, one warp per value.  The pivots are ratios of minors, d+_k =
// p_{k+1} / p_k from the top and d-_k = q_k+1 / q_k from the bottom: two lanes
// run the two division-free recurrences (the only serial chains, one FP64
// instruction per step on each), then all lanes take the pivots, gamma_k =
// d+_k + d-_k + s, and the twist r where |gamma| is smallest (largest index on
// ties), and the vector is a running product of -e_k / d+_k upwards and -e_{k-1}
// / d-_k downwards from x_r = 1 (warp scans).  Against one thread per value
// with two IEEE divisions per step on its chain: l = 150 490 -> 61 us, l = 3001
// 13.8 -> 6.5 ms.
// Scratch rows (stride NT) per value: invdp = 1 / d+_k, rp = e_k / d+_k (the
// cluster step's factors), rm; X: the result.
constexpr int VEC_WARPS = 4;

__device__ __forceinline__ double off_diag(const double* __restrict__ alpha, const double* __restrict__ beta, int k,
                                           double inv) {
    return ((k & 1) ? beta[(k >> 1) + 1] : alpha[k >> 1]) * inv;
}

// The minor before index k as step k's recurrence used it: stored minors p
// (running in direction dir, `steps` steps before k), rescaled when that step
// closed a group of 8; 1 before the first.
__device__ __forceinline__ double minor_before(const double* p, int dir, int k, int steps) {
    if (steps < 1) return 1.0;
    const double v = p[k - dir];
    return steps > 1 && ((steps - 1) & 7) == 0 ? v * rescale_factor(v, p[k - 2 * dir]) : v;
}

// One warp: the `cnt` entries x[k], k = r + dir, r + 2 dir, ..., as running
// products of -fac[k] from x_r = 1; their squares are added to *nrm2.
__device__ __forceinline__ void product_scan(const double* fac, double* x, int r, int dir, int cnt, int lane,
                                             double* nrm2) {
    double carry = 1.0;
    for (int t0 = 0; t0 < cnt; t0 += 32) {
        const int t = t0 + lane;
        const int k = r + dir * (t + 1);
        const double f = t < cnt ? -fac[k] : 1.0;
        double v = f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double w = __shfl_up_sync(RBF_FULL_MASK, v, o);
            if (lane >= o) v *= w;
        }
        const bool bad = !isfinite(v);
        if (__any_sync(RBF_FULL_MASK, bad)) {
            // a partial product over the chunk left the range of doubles: in order from the carry
            double c = carry, mine = 0.0;
            for (int q = 0; q < 32; ++q) {
                c *= __shfl_sync(RBF_FULL_MASK, f, q);
                if (q == lane) mine = c;
            }
            v = mine;
            carry = c;
        } else {
            v *= carry;
            carry = __shfl_sync(RBF_FULL_MASK, v, 31);
        }
        if (t < cnt) {
            x[k] = v;
            *nrm2 = fma(v, v, *nrm2);
        }
    }
}

__global__ void __launch_bounds__(VEC_WARPS * 32)
    k_tgk_vectors(ProjDims d, const double* __restrict__ alpha_all, const double* __restrict__ beta_all,
                  const double* __restrict__ sigma_all, const double* __restrict__ bound_all,
                  double* __restrict__ invdp_all, double* __restrict__ rp_all, double* __restrict__ rm_all,
                  double* __restrict__ X_all) {
    extern __shared__ double e2[];  // [2l]
    const int b = blockIdx.y;
    const int l = proj_l(d, b);
    if (l < 1 || blockIdx.x * VEC_WARPS >= l) return;
    const int L = d.L, NT = 2 * d.L + 1;
    const double* alpha = alpha_all + (size_t)b * L;
    const double* beta = beta_all + (size_t)b * (L + 1);
    double bound;
    load_e(alpha, beta, l, e2, &bound);
    for (int k = threadIdx.x; k < 2 * l; k += blockDim.x) e2[k] = e2[k] * e2[k];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * VEC_WARPS + (threadIdx.x >> 5);
    if (i >= l) return;
    const size_t row = ((size_t)b * L + i) * NT;
    double* invdp = invdp_all + row;
    double* rp = rp_all + row;
    double* rm = rm_all + row;  // the bottom-up minors, then e_{k-1} / d-_k
    double* x = X_all + row;    // the top-down minors, then the vector
    const int nt = 2 * l + 1;
    const double s = sigma_all[(size_t)b * L + i] / bound;
    const double inv_bound = 1.0 / bound;
    // ---- minors: step k (pivot k from the lane's end) stored at its pivot's index
    {
        const bool dn = lane & 1;
        double* out = dn ? rm : x;
        const double* ee = dn ? e2 + (nt - 2) : e2;  // e2 entry of step k: ee[+-(k - 1)]
        const int dir = dn ? -1 : 1, at = dn ? nt - 1 : 0;
        double pm2 = 1.0, pm1 = s == 0.0 ? -1e-300 : -s;
        if (lane < 2) out[at] = pm1;
        int k = 1;
        for (; k + 7 < nt; k += 8) {
            double* o = out + at + dir * k;
            minor_group(ee + dir * (k - 1), dir, s, pm2, pm1, [&](int u, double p) {
                if (lane < 2) o[dir * u] = p;
            });
            const double f = rescale_factor(pm1, pm2);
            pm1 *= f;
            pm2 *= f;
        }
        for (; k < nt; ++k) {
            const double p = minor_step(s, pm1, pm2, ee[dir * (k - 1)]);
            if (lane < 2) out[at + dir * k] = p;
            pm2 = pm1;
            pm1 = p;
        }
    }
    __syncwarp();
    // ---- pivots, gamma and the twist.  Step k's minor was formed from the one
    // before it rescaled when k - 1 closed a group of 8 (k - 1 = 8, 16, ...;
    // the last group of fewer than 8 steps is not rescaled).
    double best = INFINITY;
    int r = 0;
    for (int k0 = 0; k0 < nt; k0 += 32) {
        const int k = k0 + lane;
        double iv = 0.0, rpk = 0.0, rmk = 0.0;
        if (k < nt) {
            double den = minor_before(x, 1, k, k), pk = x[k];
            if (is_zero(den)) den = tiny_after(minor_before(x, 1, k - 1, k - 1));  // (two zeros never follow one another)
            if (is_zero(pk)) pk = tiny_after(den);
            iv = den / pk;  // 1 / d+_k
            const double dp = pk / den;
            if (k < nt - 1) rpk = off_diag(alpha, beta, k, inv_bound) * iv;
            const int kb = nt - 1 - k;  // steps from the bottom
            double denb = minor_before(rm, -1, k, kb), qk = rm[k];
            if (is_zero(denb)) denb = tiny_after(minor_before(rm, -1, k + 1, kb - 1));
            if (is_zero(qk)) qk = tiny_after(denb);
            const double dm = qk / denb;
            if (k > 0) rmk = off_diag(alpha, beta, k - 1, inv_bound) / dm;
            const double gm = fabs(dp + dm + s);
            if (gm <= best) {
                best = gm;
                r = k;
            }
        }
        __syncwarp();
        if (k < nt) {
            invdp[k] = iv;
            rp[k] = rpk;
            rm[k] = rmk;
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(RBF_FULL_MASK, best, o);
        const int orr = __shfl_xor_sync(RBF_FULL_MASK, r, o);
        if (ob < best || (ob == best && orr > r)) {
            best = ob;
            r = orr;
        }
    }
    __syncwarp();
    // ---- x_r = 1; upward x_k = -rp_k x_{k+1}; downward x_k = -rm_k x_{k-1}
    double nrm2 = 0.0;
    if (lane == 0) {
        x[r] = 1.0;
        nrm2 = 1.0;
    }
    product_scan(rp, x, r, -1, r, lane, &nrm2);
    product_scan(rm, x, r, 1, nt - 1 - r, lane, &nrm2);
    const double inv = rsqrt(warp_sum(nrm2));
    __syncwarp();
    for (int k = lane; k < nt; k += 32) x[k] *= inv;
}

// Clusters of close singular values: inverse iteration (3 steps) with the
// stored LDL^T factors of T - s_a I, all members in parallel lanes, then
// modified Gram-Schmidt in order.  One warp per cluster.  Bound by the dependent FP64
// operations of the solves (~64 cycles each, 600 per step): 15 values of l up to
// 150 with 8 warps per CTA, the loads in front of each block of the chain and the
// scaling inside it 240 us, now 194.
constexpr int CL_WARPS = 4;  // one per FP64 unit of an SM
constexpr int CL_MAX = 32;
constexpr int CL_BLK = 8;  // steps of a triangular solve whose operands are loaded together

// One lane: v[k] += -f[k - 1] v[k - 1] for k = 1 .. nt - 1 (forward), or
// v[k] += -f[k] v[k + 1] for k = nt - 2 .. 0 (backward).  The operands of a block
// are loaded while the block before it is in its chain.
template <int DIR>
__device__ __forceinline__ void solve_chain(double* v, const double* f, int nt) {
    double* x = DIR > 0 ? v : v + nt - 1;
    const double* g = DIR > 0 ? f : f + nt - 2;
    double c = x[0];
    double a[2][CL_BLK], y[2][CL_BLK];
    auto load = [&](int k, double* a, double* y) {
#pragma unroll
        for (int u = 0; u < CL_BLK; ++u) {
            const bool in = k + u < nt;
            a[u] = in ? g[DIR * (k + u - 1)] : 0.0;
            y[u] = in ? x[DIR * (k + u)] : 0.0;
        }
    };
    auto chain = [&](int k, const double* a, const double* y) {
#pragma unroll
        for (int u = 0; u < CL_BLK; ++u)
            if (k + u < nt) x[DIR * (k + u)] = c = fma(-a[u], c, y[u]);
    };
    load(1, a[0], y[0]);
    for (int k = 1; k < nt; k += 2 * CL_BLK) {
        load(k + CL_BLK, a[1], y[1]);
        chain(k, a[0], y[0]);
        load(k + 2 * CL_BLK, a[0], y[0]);
        chain(k + CL_BLK, a[1], y[1]);
    }
}

// Grid (B, gy): CTA y takes the clusters of index y CL_WARPS .. y CL_WARPS +
// CL_WARPS - 1 (in the order of the descending singular values), one per warp;
// every CTA finds them with the same scan over one bit per value ("close to
// the next one").  A cluster's member vectors are iterated in place in X.
__global__ void k_tgk_clusters(ProjDims d, const double* __restrict__ sigma_all, double tol,
                               const double* __restrict__ invdp_all, const double* __restrict__ rp_all,
                               double* __restrict__ X_all) {
    __shared__ int own_start[CL_WARPS], own_end[CL_WARPS];
    __shared__ unsigned near_bits[SVD_MAX_L / 32];
    const int b = blockIdx.x;
    const int l = proj_l(d, b);
    if (l < 1) return;
    const int L = d.L, NT = 2 * d.L + 1;
    const double* sigma = sigma_all + (size_t)b * L;
    if (threadIdx.x < CL_WARPS) own_start[threadIdx.x] = -1;
    for (int j = threadIdx.x; j < (l + 31) / 32 * 32; j += blockDim.x) {
        const bool near = j + 1 < l && fabs(sigma[j] - sigma[j + 1]) < tol * sigma[j];
        const unsigned w = __ballot_sync(RBF_FULL_MASK, near);
        if ((j & 31) == 0) near_bits[j >> 5] = w;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int c0 = blockIdx.y * CL_WARPS;
        int c = 0;
        int i = 0;
        while (i < l && c < c0 + CL_WARPS) {
            int j = i;
            while (j + 1 < l && j - i + 1 < CL_MAX && ((near_bits[j >> 5] >> (j & 31)) & 1u)) ++j;
            if (j > i) {
                if (c >= c0) {
                    own_start[c - c0] = i;
                    own_end[c - c0] = j;
                }
                ++c;
            }
            i = j + 1;
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nt = 2 * l + 1;
    const int a0 = own_start[warp];
    if (a0 < 0) return;
    const int a1 = own_end[warp];
    const int mcnt = a1 - a0 + 1;
    const size_t row0 = ((size_t)b * L + a0) * NT;
    double* y = X_all + row0;  // member vectors of this warp's cluster, in place
    // deterministic start vectors
    for (int a = 0; a < mcnt; ++a)
        for (int k = lane; k < nt; k += 32) y[(size_t)a * NT + k] = sin(0.7 * (double)(k + 1) * (a + 1) + 0.3);
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
        // lane a solves (T - s_a I) x = y_a:  L D L^T with L_{k+1,k} = rp_k
        // (a lane's warp instruction takes the FP64 unit as long as a full warp's: the
        // scaling by the inverse pivots runs over the lanes, not in the chain)
        if (lane < mcnt) solve_chain<1>(y + (size_t)lane * NT, rp_all + row0 + (size_t)lane * NT, nt);
        __syncwarp();
        for (int a = 0; a < mcnt; ++a)
            for (int k = lane; k < nt; k += 32) y[(size_t)a * NT + k] *= invdp_all[row0 + (size_t)a * NT + k];
        __syncwarp();
        if (lane < mcnt) solve_chain<-1>(y + (size_t)lane * NT, rp_all + row0 + (size_t)lane * NT, nt);
        __syncwarp();
        // modified Gram-Schmidt in member order
        for (int a = 0; a < mcnt; ++a) {
            double* va = y + (size_t)a * NT;
            for (int bb = 0; bb < a; ++bb) {
                const double* vb = y + (size_t)bb * NT;
                double dot = 0.0;
                for (int k = lane; k < nt; k += 32) dot = fma(vb[k], va[k], dot);
                dot = warp_sum(dot);
                for (int k = lane; k < nt; k += 32) va[k] = fma(-dot, vb[k], va[k]);
                __syncwarp();
            }
            double n2 = 0.0;
            for (int k = lane; k < nt; k += 32) n2 = fma(va[k], va[k], n2);
            n2 = warp_sum(n2);
            const double inv = rsqrt(n2);
            for (int k = lane; k < nt; k += 32) va[k] *= inv;
            __syncwarp();
        }
    }
}

// Split the eigenvectors into u~, v~ (normalised), write V~ (and U~ when
// asked: column i = u~_i, l+1 entries, ld ldu) and f~: one warp per vector over
// the CTAs 0 .. gridDim.x - 2 of an instance; the last CTA takes f~_{l+1} (one
// CTA per instance for everything took 23 ms of an l = 3001 SVD).
constexpr int FIN_WARPS = 8;

__global__ void __launch_bounds__(FIN_WARPS * 32)
    k_tgk_finalize(ProjDims d, const double* __restrict__ alpha_all, const double* __restrict__ beta_all,
                   const double* __restrict__ X_all, double* __restrict__ ftil_all, double* __restrict__ V_all,
                   int64_t ldv, rbf_dev_state* __restrict__ stt, const double* __restrict__ sigma_all,
                   double* __restrict__ sigma1_out, double* __restrict__ ftil_last_out, double* __restrict__ U_all,
                   int64_t ldu) {
    extern __shared__ double Ls[];  // l + 1 (last CTA)
    __shared__ double red[FIN_WARPS], red2[FIN_WARPS];
    const int b = blockIdx.y;
    const int l = proj_l(d, b);
    if (l < 1) return;
    const int L = d.L, NT = 2 * d.L + 1;
    const double* alpha = alpha_all + (size_t)b * L;
    const double* beta = beta_all + (size_t)b * (L + 1);
    double* ftil = ftil_all + (size_t)b * (L + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nt = 2 * l + 1;
    const double beta1 = beta[0];
    if (blockIdx.x + 1 < gridDim.x) {
        const int i = blockIdx.x * FIN_WARPS + warp;
        if (i >= l) return;
        const double* x = X_all + ((size_t)b * L + i) * NT;
        double* V = V_all + (size_t)b * L * ldv;
        double nu = 0.0, nv = 0.0;
        for (int k = lane; k < nt; k += 32) {
            double t = x[k] * x[k];
            if (k & 1) nv += t; else nu += t;
        }
        nu = warp_sum(nu);
        nv = warp_sum(nv);
        const double iv = rsqrt(nv);
        for (int k = 2 * lane + 1; k < nt; k += 64) V[(int64_t)i * ldv + (k >> 1)] = x[k] * iv;
        if (U_all) {
            const double iu = rsqrt(nu);
            double* U = U_all + (size_t)b * L * ldu;
            for (int k = 2 * lane; k < nt; k += 64) U[(int64_t)i * ldu + (k >> 1)] = x[k] * iu;
        }
        if (lane == 0) ftil[i] = beta1 * x[0] * rsqrt(nu);
        return;
    }
    // f~_{l+1} = beta_1 / |u|, u_1 = 1, log|u_{j+1}| = log|u_j| + log(alpha_j / beta_{j+1})
    // Ls[j] = log|u_{j+1}| for j = 0..l (inclusive prefix sums, each thread a
    // contiguous run of them after the sum of the runs before it)
    const bool zero_tail = beta[l] == 0.0;
    for (int j = threadIdx.x; j <= l; j += blockDim.x)
        Ls[j] = (j == 0 || zero_tail) ? 0.0 : log(alpha[j - 1]) - log(beta[j]);
    __syncthreads();
    const int per = (l + FIN_WARPS * 32) / (FIN_WARPS * 32);  // ceil((l + 1) / threads)
    const int j0 = min(l + 1, (int)threadIdx.x * per), j1 = min(l + 1, j0 + per);
    double run = 0.0;
    for (int j = j0; j < j1; ++j) run += Ls[j];
    double pre = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(RBF_FULL_MASK, pre, o);
        if (lane >= o) pre += t;
    }
    if (lane == 31) red[warp] = pre;
    __syncthreads();
    double acc = pre - run;
    for (int w = 0; w < warp; ++w) acc += red[w];
    double mx = 0.0;
    for (int j = j0; j < j1; ++j) {
        acc += Ls[j];
        Ls[j] = acc;
        mx = fmax(mx, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(RBF_FULL_MASK, mx, o));
    if (lane == 0) red2[warp] = mx;
    __syncthreads();
    for (int w = 0; w < FIN_WARPS; ++w) mx = fmax(mx, red2[w]);
    double part = 0.0;
    for (int j = threadIdx.x; j <= l; j += blockDim.x) part += exp(2.0 * (Ls[j] - mx));
    part = warp_sum(part);
    if (lane == 0) red[warp] = part;  // (read for the last time before the barrier above)
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < FIN_WARPS; ++w) s += red[w];
        // a zero coupling inside the run makes |u| infinite
        double ft = zero_tail || mx == INFINITY ? 0.0 : beta1 * exp(-mx) / sqrt(s);
        ftil[l] = ft;
        if (sigma1_out) sigma1_out[b] = sigma_all[(size_t)b * L];
        if (ftil_last_out) ftil_last_out[b] = ft;
        if (stt && b == 0) {
            stt->scal[SC_FTIL_LAST] = ft;
            stt->scal[SC_SIGMA1] = sigma_all[0];
        }
    }
}

}  // namespace

size_t svd_ws_bytes(int l) { return svd_ws_bytes_batch(l, 1); }

size_t svd_ws_bytes_batch(int L, int B) {
    const size_t NT = 2 * (size_t)L + 1;
    size_t b = 0;
    b += 4 * ws_align(NT * L * 8 * B);            // X, invdp, rp, rm
    b += ws_align((size_t)8 * B);
    return b + 4096;
}

rbf_status launch_projected_svd_batch(rbf_ctx* ctx, ProjDims d, const double* alpha, const double* beta,
                                      double* sigma, double* ftil, double* V, int64_t ldv, void* ws,
                                      double* sigma1_out, double* ftil_last_out, double* U, int64_t ldu) {
    const int L = d.L, B = d.B;
    if (L < 1 || L > SVD_MAX_L)
        return rbf_fail(ctx, RBF_ERR_INVALID, "bidiagonal dimension %d outside [1, %d]", L, SVD_MAX_L);
    const size_t NT = 2 * (size_t)L + 1;
    WsCarve wc(ws);
    double* X = wc.take<double>(NT * L * B);
    double* invdp = wc.take<double>(NT * L * B);
    double* rp = wc.take<double>(NT * L * B);
    double* rm = wc.take<double>(NT * L * B);
    double* bound = wc.take<double>((size_t)B);
    cudaStream_t s = ctx->stream;
    const size_t sh_b = 2 * (size_t)L * (sizeof(double) + sizeof(float));
    const size_t sh_v = 2 * (size_t)L * sizeof(double);
    const size_t sh_f = ((size_t)L + 1) * sizeof(double);
    // 32 lanes per value up to three warps per SM scheduler, 8 lanes beyond, where
    // the number of counts bounds it (kernel times with 32 and 8 lanes: l = 150 0.147 and
    // 0.219 ms, l = 1000 1.32 and 1.40, 15 runs of up to l = 150 0.240 and 0.218, l = 3001 10.6 and 5.7)
    const bool wide = (int64_t)L * B <= (int64_t)ctx->sm_count * 12;
    const int warps = L > 4096 ? 2 * BS_WARPS : BS_WARPS;  // one CTA per SM holds the tables above 4096
    const int per_cta = warps * (wide ? 1 : 4);
    if (wide) RBF_CUDA(ctx, smem_limit<k_tgk_bisect<32>>(ctx, sh_b));
    else RBF_CUDA(ctx, smem_limit<k_tgk_bisect<8>>(ctx, sh_b));
    RBF_CUDA(ctx, smem_limit<k_tgk_vectors>(ctx, sh_v));
    RBF_CUDA(ctx, smem_limit<k_tgk_finalize>(ctx, sh_f));
    const dim3 gb((L + per_cta - 1) / per_cta, B);
    if (wide) k_tgk_bisect<32><<<gb, warps * 32, sh_b, s>>>(d, alpha, beta, sigma, bound);
    else k_tgk_bisect<8><<<gb, warps * 32, sh_b, s>>>(d, alpha, beta, sigma, bound);
    RBF_LAUNCHED(ctx, "k_tgk_bisect");
    k_tgk_vectors<<<dim3((L + VEC_WARPS - 1) / VEC_WARPS, B), VEC_WARPS * 32, sh_v, s>>>(d, alpha, beta, sigma, bound,
                                                                                     invdp, rp, rm, X);
    RBF_LAUNCHED(ctx, "k_tgk_vectors");
    // at most l / 2 clusters of two or more: one warp each
    const int gy = ((L + 1) / 2 + CL_WARPS - 1) / CL_WARPS;
    if (gy > 65535) return rbf_fail(ctx, RBF_ERR_UNSUPPORTED, "too many clusters for the grid");
    k_tgk_clusters<<<dim3(B, gy), CL_WARPS * 32, 0, s>>>(d, sigma, ctx->opt.cluster_tol, invdp, rp, X);
    RBF_LAUNCHED(ctx, "k_tgk_clusters");
    k_tgk_finalize<<<dim3((L + FIN_WARPS - 1) / FIN_WARPS + 1, B), FIN_WARPS * 32, sh_f, s>>>(
        d, alpha, beta, X, ftil, V, ldv, B == 1 ? ctx->d_state : nullptr, sigma, sigma1_out, ftil_last_out, U, ldu);
    RBF_LAUNCHED(ctx, "k_tgk_finalize");
    return RBF_OK;
}

rbf_status launch_projected_svd(rbf_ctx* ctx, const double* alpha, const double* beta, int l,
                                double* sigma, double* ftil, double* V, int64_t ldv, void* ws) {
    if (l < 1 || l > 1023) return rbf_fail(ctx, RBF_ERR_INVALID, "projected dimension %d outside [1, 1023]", l);
    ProjDims d{1, l, l, nullptr};
    return launch_projected_svd_batch(ctx, d, alpha, beta, sigma, ftil, V, ldv, ws, nullptr, nullptr);
}

extern "C" rbf_status rbf_projected_svd(rbf_ctx* ctx, const rbf_gkb_state* st, double* d_sigma,
                                        double* d_ftil, double* d_V, int64_t ldv) {
    RbfRange range_("rbf_projected_svd");
    if (!ctx) return RBF_ERR_INVALID;
    if (!st || !d_sigma || !d_ftil || !d_V) return rbf_fail(ctx, RBF_ERR_INVALID, "NULL argument");
    const int l = st->steps_done;
    if (l < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "state has no completed step");
    if (ldv < l) return rbf_fail(ctx, RBF_ERR_INVALID, "ldv < l");
    RBF_TRY(rbf_ws_reserve(ctx, svd_ws_bytes(l)));
    rbf_timer_start(ctx);
    RBF_TRY(launch_projected_svd(ctx, st->d_alpha, st->d_beta, l, d_sigma, d_ftil, d_V, ldv, ctx->ws));
    ctx->tim.svd_ms = rbf_timer_stop(ctx);
    return RBF_OK;
}
