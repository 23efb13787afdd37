// Reconstruction u(P_t) = sum_j coef_j Phi(|P_t - X_j|), Phi(r) = sqrt(r^2 + c^2)
// (eq. u_reconstruction), for one or several coefficient vectors that share Phi.
//
// In FP64 a pair costs 12 FP64-pipe operations for Phi and an FMA per vector, at
// 2 operations per clock per SM: 10.3 ms for 20 000 points and nodes (0.80 of the
// pipe).  The pairs are therefore evaluated in 64-bit fixed point on the integer
// and FP32 pipes, at 32 to 64 times the FP64 rate: 10.3 -> 1.59 ms.
//
//   - the coordinates and c are rounded at 2^-k, k such that the largest of them
//     stays below 2^60: q = round(x 2^k) (exact for values within 2^7 of the
//     largest, |error| <= 2^-61 of it otherwise);
//   - with d = q_P - q_X = h 2^32 + l (l signed 32 bits), s = |P - X|^2 + c^2 in
//     units of 2^(64-2k) is sum h^2 + (2 sum h l + (sum l^2 >> 32)) / 2^32, kept as 64
//     integer and 32 fraction bits;
//   - sqrt(s): FP32 estimate R0 = s rsqrt(s); with the exact residual e0 = s - R0^2,
//     R1 = 2^12 R0 + round(2^12 e0 rsqrt(s) / 2); with the residual e1 = 2^24 s -
//     R1^2, small enough to be taken modulo 2^64, N = 2^19 R1 + round(2^19 e1 rsqrt(s) /
//     2^13): |N - 2^31 sqrt(s)| is at most 1 unit (0.8 from N = 2^54 on, 0.3 in the root
//     mean square) wherever the rule below admits;
//   - the coefficients are rounded at 2^-62 of the largest of a stage of 128 nodes
//     and the products N coef are added in 64-bit integers (FxAcc32), then
//     rounded to FP64 once per stage (one scale for all the nodes of a CTA loses more
//     of the small coefficients, and its sums live through the whole kernel: 1.59 ms at
//     20 000 points and nodes instead of 1.53).
// What that is relative to Phi depends on the smallest N, 2^53 where c is smallest
// beside the coordinates: Phi is good to 2^-53 there, to 2^-61 where it is as large
// as they are; a stage's sum to FxAcc32's error.  c may be smaller than the
// largest coordinate by an exponent of at most 5 (at 6 Phi would be good to 2^-51.4).
// Below that, and with any Inf or NaN, a CTA takes the FP64 form (a first launch
// finds the coordinates' largest exponent, the CTA whether its coefficients are
// finite).
// Errors against extended precision, root mean square over 128 points and 4000 random
// nodes in units of 2^-53 of the sum of magnitudes, with an FP64 kernel and with this:
// unit cube and c = 0.2 0.080 and 0.039, c = 0.04 0.073 and 0.046, coefficients over 8
// decades 0.255 and 0.078, of alternating sign 0.529 and 0.011; [10, 10.5]^3 and c = 0.5
// 0.083 and 0.032; a cluster of size 0.01 at 1 and c = 1/32 0.068 and 0.035; one large
// coefficient before 20 000 of 1e-12 7.9 and 3.6, after them 1.4 and 1.3.
#include "common.cuh"
#include "fx_core.cuh"
#include "internal.h"

namespace {

constexpr int EV_T = 128;           // points per CTA, one per thread; nodes per stage
constexpr int EV_MIN_CHUNK = 64;     // nodes per CTA
constexpr int EX_CTAS = 64;         // partial maxima of the exponent scan

// Largest exponent field of the nodes' and points' coordinates, one partial per CTA.
__global__ void __launch_bounds__(256) k_eval_exps(const double* __restrict__ X, int64_t n3,
                                                   const double* __restrict__ P, int64_t m3, int* __restrict__ out) {
    __shared__ int red[8];
    const int64_t t0 = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
    int ex = 0;
    for (int64_t i = t0; i < n3; i += step) ex = max(ex, fx_exp(X[i]));
    for (int64_t i = t0; i < m3; i += step) ex = max(ex, fx_exp(P[i]));
    ex = __reduce_max_sync(RBF_FULL_MASK, ex);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ex;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < 8; ++w) ex = max(ex, red[w]);
        out[blockIdx.x] = ex;
    }
}

// 2^31 sqrt(s) for s = |d|^2 + c^2 from the fixed-point differences d = (hx, lx),
// ..., and c's parts: hh0 = h_c^2, hl0 = h_c l_c + (l_c^2 >> 33).
__device__ __forceinline__ long long eval_phi(long long dx, long long dy, long long dz, long long hh0, long long hl0) {
    const int lx = (int)dx, ly = (int)dy, lz = (int)dz;
    const int hx = (int)(dx >> 32) - (lx >> 31), hy = (int)(dy >> 32) - (ly >> 31), hz = (int)(dz >> 32) - (lz >> 31);
    const long long hh = imad_wide(hx, hx, imad_wide(hy, hy, imad_wide(hz, hz, hh0)));
    const long long hl = imad_wide(hx, lx, imad_wide(hy, ly, imad_wide(hz, lz, hl0)));
    const unsigned long long ll = (unsigned long long)imad_wide(lx, lx, imad_wide(ly, ly, imad_wide(lz, lz, 0)));
    const long long T = 2 * hl + (long long)(ll >> 32);
    const long long s = hh + (T >> 32);  // >= 2^36
    const unsigned frac = (unsigned)T, s0 = (unsigned)s, s1 = (unsigned)((unsigned long long)s >> 32);
    const float sf = fmaf((float)s1, 4294967296.f, (float)s0);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(sf));
    const int R0 = (int)(sf * y);                           // < 2^30, within 2^8 of sqrt(s)
    const long long e0 = imad_wide(-R0, R0, s);             // |e0| < 2^39
    // d1 = 2^12 e0 y / 2, rounded to an integer by the addition of 1.5 2^23
    const int b1 = __float_as_int(fmaf((float)(int)(e0 >> 9), y * 1048576.f, 12582912.f));
    const long long R1 = (long long)R0 * 4096 + (b1 - 0x4B400000);
    // e1 = 2^24 s - R1^2 modulo 2^64 (|e1| < 2^46)
    const unsigned w0 = __funnelshift_l(frac, s0, 24), w1 = __funnelshift_l(s0, s1, 24);
    const unsigned r0 = (unsigned)R1, r1 = (unsigned)((unsigned long long)R1 >> 32);
    const unsigned long long sq = (unsigned long long)r0 * r0 + ((unsigned long long)(2u * r1 * r0) << 32);
    const long long e1 = (long long)((((unsigned long long)w1 << 32) | w0) - sq);
    const int b2 = __float_as_int(fmaf((float)(int)(e1 >> 15), y * 2097152.f, 12582912.f));  // 2^19 e1 y / 2^13
    return (R1 << 19) + (b2 - 0x4B400000);
}

// u = sum of the chunks' partials: eight chains over the chunks, one per warp of a
// CTA of 32 outputs (a serial sum rounds once per chunk at the size of a large early
// partial, and its loads wait for one another: 20 000 nodes and 100 points, 304 chunks, 54
// -> 31 us in all).
__global__ void __launch_bounds__(256) k_eval_reduce(int64_t total, int chunks, const double* __restrict__ part,
                                                     double* __restrict__ u) {
    __shared__ double t[8][32];
    const int lane = threadIdx.x & 31, e = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    double s = 0.0;
    if (i < total)
#pragma unroll 8
        for (int q = e; q < chunks; q += 8) s += part[(int64_t)q * total + i];
    t[e][lane] = s;
    __syncthreads();
    if (e == 0 && i < total)
        u[i] = ((t[0][lane] + t[1][lane]) + (t[2][lane] + t[3][lane])) +
               ((t[4][lane] + t[5][lane]) + (t[6][lane] + t[7][lane]));
}

// Partials over the centre chunk blockIdx.y for the NC vectors blockIdx.z NC ..:
// part[chunk][vector][t].
template <int NC>
__global__ void __launch_bounds__(EV_T) k_evaluate(const double* __restrict__ X, int64_t n,
                                                   const double* __restrict__ coefs, int64_t ldc, int ncoef,
                                                   const double* __restrict__ Pts, int64_t m, double c, double scale,
                                                   int64_t chunk, const int* __restrict__ exps,
                                                   double* __restrict__ part) {
    __shared__ long long qx[EV_T], qy[EV_T], qz[EV_T];  // staged nodes (FP64 form: their bits)
    __shared__ int2 qa[NC][EV_T];                       // staged coefficients, split (FP64 form: values)
    __shared__ int red[EV_T / 32][NC + 1];
    const int64_t t = (int64_t)blockIdx.x * EV_T + threadIdx.x;
    const bool active = t < m;
    const int c0 = blockIdx.z * NC;
    const int nc = min(NC, ncoef - c0);
    const int64_t j0 = (int64_t)blockIdx.y * chunk;
    const int64_t j1 = min(n, j0 + chunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double px = active ? Pts[t] : 0.0, py = active ? Pts[m + t] : 0.0, pz = active ? Pts[2 * m + t] : 0.0;
    // largest exponents: of all coordinates (ev[NC]), of the chunk's coefficients
    int ev[NC + 1], ea = 0;
    ev[NC] = threadIdx.x < EX_CTAS ? exps[threadIdx.x] : 0;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        ev[q] = 0;
        if (q < nc)
            for (int64_t j = j0 + threadIdx.x; j < j1; j += EV_T)
                ev[q] = max(ev[q], fx_exp(coefs[(int64_t)(c0 + q) * ldc + j]));
    }
#pragma unroll
    for (int q = 0; q < NC + 1; ++q) {
        ev[q] = __reduce_max_sync(RBF_FULL_MASK, ev[q]);
        if (lane == 0) red[warp][q] = ev[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NC + 1; ++q) {
        for (int w = 0; w < EV_T / 32; ++w) ev[q] = max(ev[q], red[w][q]);
        if (q < NC) ea = max(ea, ev[q]);
    }
    const int ec = fx_exp(c), es = max(max(ev[NC], ec), 1);
    double res[NC];
    if (es < FX_NONFINITE && ea < FX_NONFINITE && ec >= es - 5) {
        const int k = 1082 - es;
        const long long ux = fx_round(px, k), uy = fx_round(py, k), uz = fx_round(pz, k), qc = fx_round(c, k);
        const int lc = (int)qc, hc = (int)(qc >> 32) - (lc >> 31);
        auto stage_exp = [&](int q) {
            int e = 1;
#pragma unroll
            for (int w = 0; w < EV_T / 32; ++w) e = max(e, red[w][q]);
            return e;
        };
        const long long hh0 = imad_wide(hc, hc, 0), hl0 = imad_wide(hc, lc, imad_wide(lc, lc, 0) >> 33);
#pragma unroll
        for (int q = 0; q < NC; ++q) res[q] = 0.0;
        for (int64_t jb = j0; jb < j1; jb += EV_T) {
            FxAcc32 acc[NC];
            __syncthreads();
            const int64_t j = jb + threadIdx.x;
            const bool ok = j < j1;
            qx[threadIdx.x] = ok ? fx_round(X[j], k) : 0;
            qy[threadIdx.x] = ok ? fx_round(X[n + j], k) : 0;
            qz[threadIdx.x] = ok ? fx_round(X[2 * n + j], k) : 0;
            double cf[NC];
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                cf[q] = ok && q < nc ? coefs[(int64_t)(c0 + q) * ldc + j] : 0.0;
                const int e = __reduce_max_sync(RBF_FULL_MASK, fx_exp(cf[q]));
                if (lane == 0) red[warp][q] = e;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < NC; ++q) qa[q][threadIdx.x] = fx_split(fx_round(cf[q], 1084 - stage_exp(q)));
            __syncthreads();
            const int cnt = (int)min((int64_t)EV_T, j1 - jb);
            for (int rb = 0; rb < cnt; rb += FX_FOLD) {
                const int re = min(rb + FX_FOLD, cnt);
#pragma unroll 2
                for (int r = rb; r < re; ++r) {
                    const int2 N = fx_split(eval_phi(ux - qx[r], uy - qy[r], uz - qz[r], hh0, hl0));
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        const int2 a = qa[q][r];
                        acc[q].add(N.y, N.x, a.y, a.x);
                    }
                }
#pragma unroll
                for (int q = 0; q < NC; ++q) acc[q].fold();
            }
#pragma unroll
            for (int q = 0; q < NC; ++q)
                res[q] += ldexp(FxAcc32::value(acc[q].pair(cnt)), FX_UNIT + 1 - k - (1084 - stage_exp(q)));
        }
    } else {
        const double c2 = c * c;
        const bool far = ec < 1023 - 490 || es > 1023 + 490;  // s may leave the normal numbers
        double* sx = (double*)qx;
        double* sy = (double*)qy;
        double* sz = (double*)qz;
#pragma unroll
        for (int q = 0; q < NC; ++q) res[q] = 0.0;
        for (int64_t jb = j0; jb < j1; jb += EV_T) {
            __syncthreads();
            const int64_t j = jb + threadIdx.x;
            const bool ok = j < j1;
            sx[threadIdx.x] = ok ? X[j] : 0.0;
            sy[threadIdx.x] = ok ? X[n + j] : 0.0;
            sz[threadIdx.x] = ok ? X[2 * n + j] : 0.0;
#pragma unroll
            for (int q = 0; q < NC; ++q)
                *(double*)&qa[q][threadIdx.x] = ok && q < nc ? coefs[(int64_t)(c0 + q) * ldc + j] : 0.0;
            __syncthreads();
            const int cnt = (int)min((int64_t)EV_T, j1 - jb);
            for (int r = 0; r < cnt; ++r) {
                const double dx = px - sx[r], dy = py - sy[r], dz = pz - sz[r];
                const double s = fma(dx, dx, fma(dy, dy, fma(dz, dz, c2)));
                const double ph = far ? sqrt(s) : s * rsqrt_f64(s);
#pragma unroll
                for (int q = 0; q < NC; ++q) res[q] = fma(*(const double*)&qa[q][r], ph, res[q]);
            }
        }
    }
    if (active)
#pragma unroll
        for (int q = 0; q < NC; ++q)
            if (q < nc) part[((int64_t)blockIdx.y * ncoef + c0 + q) * m + t] = res[q] * scale;
}

// Centre chunks for `ctas` CTAs per chunk.  At most one wave of resident CTAs (the
// chains of a pair need all the warps that fit: 8 CTAs per SM took 5 % longer than a
// full wave at 20 000 points and nodes) and at least 64 nodes each; among these down to
// 3/4 as many (up to eight per point tile where one wave holds a single one), the number that fills
// the SMs most evenly: ceil(CTAs per SM) times a CTA's nodes and its fixed part,
// about 24 nodes.  One full wave against this, 8000 nodes: 500 points and 150 vectors 612
// and 549 us, 8 vectors 69 and 49 (in FP64 198 and 160), 20 000 points and 17 vectors 4.69 and
// 3.13 ms (21.4 and 17.3).
int64_t eval_chunks(int64_t n, int64_t ctas, int64_t sms, int64_t per_sm) {
    int64_t top = sms * per_sm / ctas;
    if (top < 2) top = 8;
    const int64_t most = (n + EV_MIN_CHUNK - 1) / EV_MIN_CHUNK;
    if (top > most) top = most;
    int64_t low = sms * per_sm / ctas < 2 ? 1 : (3 * top + 3) / 4;
    int64_t best = top, least = INT64_MAX;
    for (int64_t c = top; c >= low; --c) {
        const int64_t cost = (ctas * c + sms - 1) / sms * ((n + c - 1) / c + 24);
        if (cost < least) {
            least = cost;
            best = c;
        }
    }
    return best;
}

rbf_status evaluate_vectors(rbf_ctx* ctx, const rbf_operator* op, const double* coefs, int64_t ldc, int ncoef,
                            const double* pts, int64_t m, double* u) {
    const int64_t n = op->n;
    const int64_t tiles = (m + EV_T - 1) / EV_T;
    // vectors per CTA: the smallest of 1, 2, 4, 8 that holds them all (8 beyond)
    const int nc = ncoef <= 1 ? 1 : ncoef <= 2 ? 2 : ncoef <= 4 ? 4 : 8;
    const int zs = (ncoef + nc - 1) / nc;
    const void* kern = nc == 1 ? (const void*)k_evaluate<1> : nc == 2 ? (const void*)k_evaluate<2>
                       : nc == 4 ? (const void*)k_evaluate<4> : (const void*)k_evaluate<8>;
    int per_sm = 0;
    RBF_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, EV_T, 0));
    int64_t chunks = eval_chunks(n, tiles * zs, ctx->sm_count, per_sm);
    if (chunks > 65535) chunks = 65535;
    const int64_t total = m * ncoef;
    int64_t chunk;
    for (;;) {  // fewer chunks where the partials of so many do not fit the workspace cap
        chunk = (n + chunks - 1) / chunks;
        chunks = (n + chunk - 1) / chunk;
        const rbf_status st = rbf_ws_reserve(ctx, ws_align((size_t)chunks * total * sizeof(double)) +
                                                      ws_align(EX_CTAS * sizeof(int)));
        if (st == RBF_OK) break;
        if (chunks == 1) return st;
        chunks = (chunks + 1) / 2;
    }
    WsCarve wc(ctx->ws);
    double* part = wc.take<double>((size_t)chunks * total);
    int* exps = wc.take<int>(EX_CTAS);
    k_eval_exps<<<EX_CTAS, 256, 0, ctx->stream>>>(op->d_nodes, 3 * n, pts, 3 * m, exps);
    RBF_LAUNCHED(ctx, "k_eval_exps");
    const double scale = op->form == RBF_FORM_EPS ? 1.0 / op->c : 1.0;
    const dim3 grid((unsigned)tiles, (unsigned)chunks, (unsigned)zs);
#define EV_LAUNCH(NC_)                                                                                            \
    k_evaluate<NC_><<<grid, EV_T, 0, ctx->stream>>>(op->d_nodes, n, coefs, ldc, ncoef, pts, m, op->c, scale, chunk, \
                                                    exps, part)
    if (nc == 1) EV_LAUNCH(1);
    else if (nc == 2) EV_LAUNCH(2);
    else if (nc == 4) EV_LAUNCH(4);
    else EV_LAUNCH(8);
#undef EV_LAUNCH
    RBF_LAUNCHED(ctx, "k_evaluate");
    if (chunks < 16) return launch_reduce_partials(ctx, total, (int)chunks, part, u);
    k_eval_reduce<<<(unsigned)((total + 31) / 32), 256, 0, ctx->stream>>>(total, (int)chunks, part, u);
    RBF_LAUNCHED(ctx, "k_eval_reduce");
    return RBF_OK;
}

}  // namespace

rbf_status launch_evaluate(rbf_ctx* ctx, const rbf_operator* op, const double* coef, const double* pts, int64_t m,
                           double* u) {
    return evaluate_vectors(ctx, op, coef, op->n, 1, pts, m, u);
}

extern "C" rbf_status rbf_evaluate_many(rbf_ctx* ctx, const rbf_operator* op, const double* d_coefs, int64_t ldc,
                                        int ncoef, const double* d_points, int64_t m, double* d_u) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!op || !d_coefs || !d_points || !d_u || m < 1 || ncoef < 1 || ldc < op->n)
        return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_evaluate_many: bad argument");
    return evaluate_vectors(ctx, op, d_coefs, ldc, ncoef, d_points, m, d_u);
}
