// Stopping / lambda network (20 -> 128 -> 128 -> 2, exact-erf GELU, FP32) with
// forward, backward and Adam kernels; the features it reads from the first GKB
// steps.
//
// A training step is three launches: forward and activation gradients of a few
// samples per CTA with W2 in shared memory (k_mlp_pass), partial weight
// gradients over chunks of the batch (k_mlp_wgrad), and the sum of the partials
// with the Adam update (k_mlp_finish).  All sums are in a fixed order.
#include <cfloat>

#include "common.cuh"
#include "internal.h"

namespace {

constexpr int NI = RBF_MLP_IN, NH = RBF_MLP_HIDDEN, NO = RBF_MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NI * NH, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH * NO, NPAR = OFF_B3 + NO;
static_assert(NPAR == RBF_MLP_PARAMS, "parameter layout");

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// Forward pass and, with TRAIN, the activation gradients of TS samples at a time by
// CTAs of 256 threads: thread (half, j) owns hidden unit j for the samples [half TS /
// 2, (half + 1) TS / 2).  W2 sits in shared memory for both directions (rows of
// W2_LD floats: conflict-free reads along a row by 16 bytes and down a column), read
// once per CTA however many tiles it takes; it arrives by cp.async while layer 1 of
// the first runs.  Latency bounds small batches (a network of 19 458 weights): few
// samples per CTA, so that the batch spreads over the SMs, and no second launch and
// no cached z.  Forward and activation gradients of 512 samples: 27 + 36 us (16
// samples per CTA, W2 from L2, read across rows in the backward pass) -> 9.4 us.
// Writes Y [B][2] and, with TRAIN, H1, H2, DZ1, DZ2 [B][NH] and DY = (Y - T) / B;
// lpart (optional): squared-error partial per CTA.
constexpr int MP_T = 2 * NH;
constexpr int W2_LD = NH + 4;

struct PassArgs {
    const float *P, *X, *T;
    int B;
    float *Y, *H1, *H2, *DZ1, *DZ2, *DY;
    double* lpart;
};

template <int TS, bool TRAIN>
constexpr size_t mlp_smem() {
    return sizeof(float) * (size_t)(NH * W2_LD + TS * (NI + (TRAIN ? 2 : 1) * NH));
}

template <int TS, bool TRAIN>
__global__ void __launch_bounds__(MP_T) k_mlp_pass(PassArgs a) {
    constexpr int HS = TS / 2;  // samples per thread
    extern __shared__ float4 smem4[];
    float* w2 = (float*)smem4;     // [NH][W2_LD]
    float* xs = w2 + NH * W2_LD;   // [TS][NI]
    float* h1s = xs + TS * NI;     // [TS][NH]
    float* dzs = h1s + TS * NH;    // [TS][NH] dz2
    __shared__ float red[MP_T / 32][HS][NO];
    __shared__ float dys[TS][NO];
    const float* __restrict__ P = a.P;
    const int j = threadIdx.x & (NH - 1), half = threadIdx.x / NH;
    for (int q = threadIdx.x; q < NH * NH / 4; q += MP_T) {
        const int i = q / (NH / 4), c = (q % (NH / 4)) * 4;
        const unsigned d = (unsigned)__cvta_generic_to_shared(w2 + i * W2_LD + c);
        // the parameter vector need not be 16-byte aligned
        if (((uintptr_t)P & 15u) == 0)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(P + OFF_W2 + i * NH + c) : "memory");
        else
            for (int e = 0; e < 4; ++e) w2[i * W2_LD + c + e] = P[OFF_W2 + i * NH + c + e];
    }
    const int tiles = (a.B + TS - 1) / TS;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int s0 = tile * TS;
        const int ns = min(TS, a.B - s0);
        if (tile != (int)blockIdx.x) __syncthreads();  // the tile before is read
        for (int q = threadIdx.x; q < TS * NI; q += MP_T) xs[q] = q / NI < ns ? a.X[(int64_t)s0 * NI + q] : 0.f;
        __syncthreads();
        float z1[HS], z2[HS], h2[HS];
        const float* x = xs + half * HS * NI;
#pragma unroll
        for (int s = 0; s < HS; ++s) z1[s] = P[OFF_B1 + j];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float wv = P[OFF_W1 + i * NH + j];
#pragma unroll
            for (int s = 0; s < HS; ++s) z1[s] = fmaf(x[s * NI + i], wv, z1[s]);
        }
        float* h1 = h1s + half * HS * NH;
#pragma unroll
        for (int s = 0; s < HS; ++s) {
            const float h = gelu_f(z1[s]);
            h1[s * NH + j] = h;
            if (TRAIN && half * HS + s < ns) a.H1[(int64_t)(s0 + half * HS + s) * NH + j] = h;
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int s = 0; s < HS; ++s) z2[s] = P[OFF_B2 + j];
#pragma unroll 4
        for (int i = 0; i < NH; i += 4) {
            float w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = w2[(i + e) * W2_LD + j];
#pragma unroll
            for (int s = 0; s < HS; ++s) {
                const float4 h = *reinterpret_cast<const float4*>(h1 + s * NH + i);
                z2[s] = fmaf(h.w, w[3], fmaf(h.z, w[2], fmaf(h.y, w[1], fmaf(h.x, w[0], z2[s]))));
            }
        }
        // output layer: partial products per unit, reduced over the warps of the half
        const float w30 = P[OFF_W3 + j * NO], w31 = P[OFF_W3 + j * NO + 1];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
        for (int s = 0; s < HS; ++s) {
            h2[s] = gelu_f(z2[s]);
            if (TRAIN && half * HS + s < ns) a.H2[(int64_t)(s0 + half * HS + s) * NH + j] = h2[s];
            const float p0 = warp_sumf(h2[s] * w30), p1 = warp_sumf(h2[s] * w31);
            if (lane == 0) {
                red[warp][s][0] = p0;
                red[warp][s][1] = p1;
            }
        }
        __syncthreads();
        if (threadIdx.x < TS * NO) {
            const int s = threadIdx.x / NO, o = threadIdx.x % NO, hf = s / HS;
            float y = P[OFF_B3 + o], d = 0.f;
            double dl = 0.0;
            for (int w = 0; w < NH / 32; ++w) y += red[hf * (NH / 32) + w][s % HS][o];
            if (s < ns) {
                const int64_t at = (int64_t)(s0 + s) * NO + o;
                a.Y[at] = y;
                if (TRAIN) {
                    d = y - a.T[at];
                    dl = (double)y - (double)a.T[at];
                    a.DY[at] = d / (float)a.B;
                }
            }
            if (TRAIN) dys[s][o] = d / (float)a.B;
            if constexpr (TRAIN) {
                static_assert(TS * NO <= 32, "the loss is summed by one warp");
                if (a.lpart) {
                    double l = dl * dl;
                    for (int q = TS * NO / 2; q > 0; q >>= 1) l += __shfl_xor_sync(0xffffffffu >> (32 - TS * NO), l, q);
                    if (threadIdx.x == 0) a.lpart[tile] = l;
                }
            }
        }
        if (!TRAIN) continue;
        __syncthreads();
        float* dz2 = dzs + half * HS * NH;
#pragma unroll
        for (int s = 0; s < HS; ++s) {
            const int q = half * HS + s;
            const float dz = (dys[q][0] * w30 + dys[q][1] * w31) * gelu_grad_f(z2[s]);
            dz2[s * NH + j] = dz;
            if (q < ns) a.DZ2[(int64_t)(s0 + q) * NH + j] = dz;
        }
        __syncthreads();
        // dh1_j = sum over units u of dz2_u W2[j][u]
        float acc[HS];
#pragma unroll
        for (int s = 0; s < HS; ++s) acc[s] = 0.f;
        const float* wr = w2 + j * W2_LD;
#pragma unroll 4
        for (int u = 0; u < NH; u += 4) {
            const float4 w = *reinterpret_cast<const float4*>(wr + u);
#pragma unroll
            for (int s = 0; s < HS; ++s) {
                const float4 d = *reinterpret_cast<const float4*>(dz2 + s * NH + u);
                acc[s] = fmaf(d.w, w.w, fmaf(d.z, w.z, fmaf(d.y, w.y, fmaf(d.x, w.x, acc[s]))));
            }
        }
#pragma unroll
        for (int s = 0; s < HS; ++s)
            if (half * HS + s < ns) a.DZ1[(int64_t)(s0 + half * HS + s) * NH + j] = acc[s] * gelu_grad_f(z1[s]);
    }
}

// a + b and its rounding error (Knuth's TwoSum).
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
    return t;
}

// Sums in FP32 as unevaluated pairs s + c and triples s + c + d (Ogita, Rump and Oishi's
// Dot2 and SumK with K = 3: the rounding errors of a product and of an addition,
// both exact in FP32, are added to the next word).  A stage of 16 samples is summed in
// pairs, whose own roundings are about 2^-49 of the stage's sum; stages and chunks in
// triples, 2^-70.  A sum of the exact products in FP64 rounds at 2^-54 of its partial sum
// once per sample: for 512 samples the two come to the same 2^-50.
struct Pair {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void dot(float a, float b) {
        const float p = __fmul_rn(a, b);
        float e;
        s = two_sum(s, p, e);
        c = __fadd_rn(c, __fadd_rn(e, __fmaf_rn(a, b, -p)));
    }
};

struct Triple {
    float s = 0.f, c = 0.f, d = 0.f;
    __device__ __forceinline__ void add(float p, float e) {
        float q, r, u;
        s = two_sum(s, p, q);
        e = two_sum(e, q, r);
        c = two_sum(c, e, u);
        d = __fadd_rn(d, __fadd_rn(r, u));
    }
    __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)d); }
};

// Weight-gradient partials over the samples [chunk c, chunk (c + 1)) of chunk c =
// blockIdx.x: out[r][j] = sum_s L[s][r] R[s][j], 4 x 4 outputs per thread, 32 rows
// x 128 columns per CTA.  blockIdx.y: 0..3 W2 (L = H1, R = DZ2); 4 W1 and b1 (L =
// X and 1, R = DZ1); 5 b2 (L = 1, R = DZ2); 6 W3 transposed (L = DY, R = H2) and b3.
// An FP64 sum of the products (exact in FP64) runs at 1/64 of the FP32 rate: 10
// M FP64 FMAs of a 512-sample step are 16 us at best; ten FP32 operations per
// product and 22 per stage give its precision (triples throughout, 24 operations per
// product: 33 us for a step of 512 samples; this, 27; pairs throughout, 24, but errors
// 8 times as large at 4096 samples).  One thread per weight with an FP64 chain over the
// batch took 127 us, a step 162.
constexpr int WG_T = 256;
constexpr int WG_S = 16;  // samples staged at a time

struct GradArgs {
    const float *X, *H1, *H2, *DY, *DZ1, *DZ2;
    int B, chunk, chunks;
    float* part;  // [chunks][3][NPAR]
};

__global__ void __launch_bounds__(WG_T) k_mlp_wgrad(GradArgs a) {
    __shared__ float Ls[WG_S][32];
    __shared__ float Rs[WG_S][NH];
    const int task = blockIdx.y;
    const int sb = blockIdx.x * a.chunk, se = min(a.B, sb + a.chunk);
    const int rows = task < 4 ? 32 : (task == 4 ? NI + 1 : (task == 5 ? 1 : NO));
    const float* __restrict__ Rg = task == 4 ? a.DZ1 : (task == 6 ? a.H2 : a.DZ2);
    const int r0 = (threadIdx.x >> 5) * 4, c0 = (threadIdx.x & 31) * 4;
    Triple acc[4][4], b3;
    pdl_wait();
    for (int s0 = sb; s0 < se; s0 += WG_S) {
        const int cnt = min(WG_S, se - s0);
        __syncthreads();
        for (int q = threadIdx.x; q < WG_S * NH; q += WG_T)
            Rs[q / NH][q % NH] = q / NH < cnt ? Rg[(int64_t)s0 * NH + q] : 0.f;
        for (int q = threadIdx.x; q < WG_S * 32; q += WG_T) {
            const int s = q / 32, r = q % 32;
            float v = 0.f;
            if (s < cnt && r < rows) {
                const int64_t at = s0 + s;
                if (task < 4) v = a.H1[at * NH + task * 32 + r];
                else if (task == 4) v = r < NI ? a.X[at * NI + r] : 1.f;
                else v = task == 5 ? 1.f : a.DY[at * NO + r];
            }
            Ls[s][r] = v;
        }
        __syncthreads();
        if (r0 < rows) {
            Pair run[4][4];
#pragma unroll 2
            for (int s = 0; s < cnt; ++s) {
                const float4 l = *reinterpret_cast<const float4*>(&Ls[s][r0]);
                const float4 r = *reinterpret_cast<const float4*>(&Rs[s][c0]);
                const float lv[4] = {l.x, l.y, l.z, l.w}, rv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) run[u][v].dot(lv[u], rv[v]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v].add(run[u][v].s, run[u][v].c);
        }
        if (task == 6 && threadIdx.x >= 32 && threadIdx.x < 32 + NO)
            for (int s = 0; s < cnt; ++s) b3.add(Ls[s][threadIdx.x - 32], 0.f);
    }
    float* out = a.part + (int64_t)blockIdx.x * 3 * NPAR;
    auto put = [&](int at, const Triple& t) {
        out[at] = t.s;
        out[NPAR + at] = t.c;
        out[2 * NPAR + at] = t.d;
    };
    if (task == 6 && threadIdx.x >= 32 && threadIdx.x < 32 + NO) put(OFF_B3 + threadIdx.x - 32, b3);
    if (r0 >= rows) return;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = r0 + u;
        if (r >= rows) break;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int c = c0 + v;
            int at;
            if (task < 4) at = OFF_W2 + (task * 32 + r) * NH + c;
            else if (task == 4) at = r < NI ? OFF_W1 + r * NH + c : OFF_B1 + c;
            else at = task == 5 ? OFF_B2 + c : OFF_W3 + c * NO + r;
            put(at, acc[u][v]);
        }
    }
}

// The factors of sample s in the gradient of parameter p.
__device__ __forceinline__ float2 grad_factors(const GradArgs& a, int p, int64_t s) {
    if (p < OFF_B1) return make_float2(a.X[s * NI + p / NH], a.DZ1[s * NH + p % NH]);
    if (p < OFF_W2) return make_float2(1.f, a.DZ1[s * NH + p - OFF_B1]);
    if (p < OFF_B2) return make_float2(a.H1[s * NH + (p - OFF_W2) / NH], a.DZ2[s * NH + (p - OFF_W2) % NH]);
    if (p < OFF_W3) return make_float2(1.f, a.DZ2[s * NH + p - OFF_B2]);
    if (p < OFF_B3) return make_float2(a.H2[s * NH + (p - OFF_W3) / NO], a.DY[s * NO + (p - OFF_W3) % NO]);
    return make_float2(1.f, a.DY[s * NO + p - OFF_B3]);
}

// Gradient of one parameter where the paired sum left FP32's range.  A product below
// 2^-102 has lost part of its rounding error, at most 2^-149 per sample: where the
// sum is below B 2^-100 (a unit without response, for one) it is taken again with the
// second factors times 2^96, exactly, which leaves 2^-245.  An infinite or NaN product
// or sum: in FP64, whose products are exact.
__device__ __noinline__ float grad_again(const GradArgs& a, int p) {
    Triple t;
    for (int64_t s = 0; s < a.B; ++s) {
        const float2 f = grad_factors(a, p, s);
        const float r = f.y * 0x1p96f, q = __fmul_rn(f.x, r);
        t.add(q, __fmaf_rn(f.x, r, -q));
    }
    const double g = t.value() * 0x1p-96;
    if (isfinite(g)) return (float)g;
    double acc = 0.0;
    for (int64_t s = 0; s < a.B; ++s) {
        const float2 f = grad_factors(a, p, s);
        acc += (double)f.x * (double)f.y;
    }
    return (float)acc;
}

struct AdamArgs {
    float *P, *M, *V;
    float lr, b1, b2, c1, c2, eps;
};

// (P, m0, v0: the parameter and its moments before the update)
__device__ __forceinline__ void adam_one(const AdamArgs& o, int p, float g, float P, float m0, float v0) {
    const float m = o.b1 * m0 + (1.f - o.b1) * g;
    const float v = o.b2 * v0 + (1.f - o.b2) * g * g;
    o.M[p] = m;
    o.V[p] = v;
    o.P[p] = P - o.lr * (m * o.c1) / (sqrtf(v * o.c2) + o.eps);
}

// G = sum of the chunks' partials in chunk order; with ADAM the update of the
// parameters by it.
template <bool ADAM>
__global__ void __launch_bounds__(128) k_mlp_finish(GradArgs a, float* __restrict__ G, AdamArgs o) {
    const int p = blockIdx.x * 128 + threadIdx.x;
    const bool ok = p < NPAR;
    // the parameters and moments are not written by the launches of this step before
    const float P = ADAM && ok ? o.P[p] : 0.f, m0 = ADAM && ok ? o.M[p] : 0.f, v0 = ADAM && ok ? o.V[p] : 0.f;
    pdl_wait();
    if (!ok) return;
    Triple t;
    const float* __restrict__ q = a.part + p;
#pragma unroll 8
    for (int c = 0; c < a.chunks; ++c, q += 3 * NPAR) {
        t.add(q[0], q[NPAR]);
        t.d = __fadd_rn(t.d, q[2 * NPAR]);
    }
    float g = (float)t.value();
    if (!(fabsf(g) >= (float)a.B * 0x1p-100f && fabsf(g) <= FLT_MAX)) g = grad_again(a, p);
    G[p] = g;
    if (ADAM) adam_one(o, p, g, P, m0, v0);
}

__global__ void __launch_bounds__(128) k_adam(const float* __restrict__ G, AdamArgs o) {
    const int p = blockIdx.x * 128 + threadIdx.x;
    if (p < NPAR) adam_one(o, p, G[p], o.P[p], o.M[p], o.V[p]);
}

__global__ void k_sum_parts(const double* __restrict__ parts, int n, double scale, double* __restrict__ out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int q = 0; q < n; ++q) s += parts[q];
        out[0] = s * scale;
    }
}

// Features from the first j GKB steps: [log10 s1, log10(s_i / s1) i=2..10,
// log10(rho_i / beta_1) i=1..10] where rho_i = |C_i y_i - beta_1 e_1| is the
// least-squares residual after i steps (LSQR): rho_i = beta_1 / |u^(i)| with
// u the null vector of C_i^T (u_1 = 1, u_{m+1} = -alpha_m u_m / beta_{m+1}).
// Standardised with (mean, std) when given.
__device__ void stop_features_one(const double* __restrict__ alpha, const double* __restrict__ beta,
                                  const double* __restrict__ sigma, int j, const float* __restrict__ mean,
                                  const float* __restrict__ stdv, float* __restrict__ feat) {
    double f[RBF_MLP_IN];
    const double s1 = sigma[0];
    f[0] = log10(s1);
    for (int i = 1; i < 10; ++i) f[i] = i < j ? log10(fmax(sigma[i], 1e-300) / s1) : -300.0;
    // running log-sum-exp of 2 log|u_m|
    double Lm = 0.0, mx = 0.0, sum = 1.0;  // u_1 = 1
    for (int i = 1; i <= 10; ++i) {
        if (i <= j && beta[i] > 0.0) {
            Lm += log(alpha[i - 1]) - log(beta[i]);
            const double e2 = 2.0 * Lm;
            if (e2 > mx) {
                sum = sum * exp(mx - e2) + 1.0;
                mx = e2;
            } else {
                sum += exp(e2 - mx);
            }
            f[9 + i] = -(0.5 * (mx + log(sum))) / log(10.0);
        } else {
            f[9 + i] = i <= j ? -300.0 : f[9 + i - 1];
        }
    }
    for (int q = 0; q < RBF_MLP_IN; ++q) {
        float v = (float)f[q];
        if (mean && stdv) v = (v - mean[q]) / stdv[q];
        feat[q] = v;
    }
}

__global__ void k_stop_features(const double* __restrict__ alpha, const double* __restrict__ beta,
                                const double* __restrict__ sigma, int j, const float* __restrict__ mean,
                                const float* __restrict__ stdv, float* __restrict__ feat) {
    if (threadIdx.x == 0) stop_features_one(alpha, beta, sigma, j, mean, stdv, feat);
}

// Batched: instance b = blockIdx.x with alpha [B][L], beta [B][L+1], sigma
// [B][L]; instances with fewer than j steps get NaN features.
__global__ void k_stop_features_batch(const double* __restrict__ alpha, const double* __restrict__ beta,
                                      const double* __restrict__ sigma, int L, const int* __restrict__ l_arr, int j,
                                      const float* __restrict__ mean, const float* __restrict__ stdv,
                                      float* __restrict__ feat) {
    const int b = blockIdx.x;
    if (threadIdx.x != 0) return;
    float* out = feat + (size_t)b * RBF_MLP_IN;
    if (l_arr[b] < j) {
        for (int q = 0; q < RBF_MLP_IN; ++q) out[q] = __int_as_float(0x7fc00000);
        return;
    }
    stop_features_one(alpha + (size_t)b * L, beta + (size_t)b * (L + 1), sigma + (size_t)b * L, j, mean, stdv, out);
}

}  // namespace

// ---------------------------------------------------------------------------
template <int TS, bool TRAIN>
static rbf_status launch_pass(rbf_ctx* ctx, const PassArgs& a, int* tiles) {
    constexpr size_t smem = mlp_smem<TS, TRAIN>();
    constexpr int per_sm = (int)((227 * 1024) / (smem + 2 * 1024));
    *tiles = (a.B + TS - 1) / TS;
    RBF_CUDA(ctx, (smem_limit<k_mlp_pass<TS, TRAIN>>(ctx, smem)));
    const int grid = *tiles < ctx->sm_count * per_sm ? *tiles : ctx->sm_count * per_sm;
    k_mlp_pass<TS, TRAIN><<<grid, MP_T, smem, ctx->stream>>>(a);
    RBF_LAUNCHED(ctx, "k_mlp_pass");
    return RBF_OK;
}

// Samples per CTA: few for small batches, so that they spread over the SMs; more
// where the SMs take several tiles each, so that a weight read from shared memory
// serves more of them.  Forward, tiles per SM and time, with 4, 8, 32 and 48 samples:
// 512 samples 8.3, 8.3, 12.5 and 16.5 us; 2048 13.0, 10.4, 12.5 and 16.5; 4096 16.6, 16.5, 12.5
// and 16.6; 7000 23.9, 20.6, 20.6 and 16.6; 65536 156, 123, 105 and 112 (16 samples of W2 from
// L2, in CTAs of 128 threads: 16.6, 16.6, 18.6, 18.6 and 103).  With the activation
// gradients: 7000 samples 119, 119 and 119 with 4, 8 and 16 after 128 with 4 and W2 read
// for each tile; 65536 992 with 8, 952 with 16.
static rbf_status launch_mlp_train(rbf_ctx* ctx, const PassArgs& a, int* tiles) {
    return (int64_t)a.B <= (int64_t)ctx->sm_count * 48 ? launch_pass<4, true>(ctx, a, tiles)
                                                        : launch_pass<16, true>(ctx, a, tiles);
}

static rbf_status launch_mlp_forward(rbf_ctx* ctx, const PassArgs& a) {
    const int64_t per_sm = ((int64_t)a.B + ctx->sm_count - 1) / ctx->sm_count;
    int tiles = 0;
    if (per_sm <= 4) return launch_pass<4, false>(ctx, a, &tiles);
    if (per_sm <= 16) return launch_pass<8, false>(ctx, a, &tiles);
    if (per_sm > 32 && per_sm <= 48) return launch_pass<48, false>(ctx, a, &tiles);
    return launch_pass<32, false>(ctx, a, &tiles);
}

extern "C" rbf_status rbf_mlp_forward(rbf_ctx* ctx, const float* d_params, const float* d_x, int batch, float* d_y) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!d_params || !d_x || !d_y || batch < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_mlp_forward: bad argument");
    PassArgs a{};
    a.P = d_params;
    a.X = d_x;
    a.B = batch;
    a.Y = d_y;
    return launch_mlp_forward(ctx, a);
}

// Gradient into G and, with `adam`, the update in the same last launch.
static rbf_status mlp_grad_impl(rbf_ctx* ctx, const float* P, const float* X, const float* T, int B, float* G,
                                float* h_loss, const AdamArgs* adam) {
    // chunks of the batch: 16 samples each (32 x 7 CTAs at 512 samples), longer
    // ones past 64 chunks, where the partials (234 KB per chunk) would cost more
    // than the shorter sums save
    int chunk = WG_S;
    while ((B + chunk - 1) / chunk > 64) chunk += WG_S;
    const int tiles_max = (B + 3) / 4;
    int chunks;
    for (;;) {  // fewer chunks where the partials of so many do not fit the workspace cap
        chunks = (B + chunk - 1) / chunk;
        const size_t need = 4 * ws_align((size_t)B * NH * 4) + 2 * ws_align((size_t)B * NO * 4) +
                            ws_align((size_t)chunks * 3 * NPAR * sizeof(float)) +
                            ws_align((size_t)(tiles_max + 1) * 8);
        const rbf_status st = rbf_ws_reserve(ctx, need);
        if (st == RBF_OK) break;
        if (chunks == 1) return st;
        chunk *= 2;
    }
    WsCarve wc(ctx->ws);
    PassArgs a{};
    a.P = P;
    a.X = X;
    a.T = T;
    a.B = B;
    a.H1 = wc.take<float>((size_t)B * NH);
    a.H2 = wc.take<float>((size_t)B * NH);
    a.DZ1 = wc.take<float>((size_t)B * NH);
    a.DZ2 = wc.take<float>((size_t)B * NH);
    a.Y = wc.take<float>((size_t)B * NO);
    a.DY = wc.take<float>((size_t)B * NO);
    float* part = wc.take<float>((size_t)chunks * 3 * NPAR);
    double* lpart = wc.take<double>((size_t)tiles_max + 1);
    a.lpart = h_loss ? lpart : nullptr;
    int tiles = 0;
    RBF_TRY(launch_mlp_train(ctx, a, &tiles));
    const GradArgs ga{X, a.H1, a.H2, a.DY, a.DZ1, a.DZ2, B, chunk, chunks, part};
    // programmatic launches: their start-up overlaps the launch before (26.7 -> 21.5 us a step)
    RBF_CUDA(ctx, rbf_launch_ex(ctx, k_mlp_wgrad, dim3(chunks, 7), dim3(WG_T), 0, true, 1, ga));
    RBF_LAUNCHED(ctx, "k_mlp_wgrad");
    const dim3 fg((NPAR + 127) / 128);
    if (adam) RBF_CUDA(ctx, rbf_launch_ex(ctx, k_mlp_finish<true>, fg, dim3(128), 0, true, 1, ga, G, *adam));
    else RBF_CUDA(ctx, rbf_launch_ex(ctx, k_mlp_finish<false>, fg, dim3(128), 0, true, 1, ga, G, AdamArgs{}));
    RBF_LAUNCHED(ctx, "k_mlp_finish");
    if (h_loss) {
        k_sum_parts<<<1, 32, 0, ctx->stream>>>(lpart, tiles, 1.0 / (2.0 * B), lpart + tiles);
        RBF_LAUNCHED(ctx, "k_sum_parts");
        double l = 0.0;
        RBF_CUDA(ctx, cudaMemcpyAsync(&l, lpart + tiles, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
        RBF_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        *h_loss = (float)l;
    }
    return RBF_OK;
}

static AdamArgs adam_args(float* P, float* M, float* V, int t, float lr) {
    const double b1 = 0.9, b2 = 0.999;
    return AdamArgs{P, M, V, lr, (float)b1, (float)b2, (float)(1.0 / (1.0 - pow(b1, t))),
                    (float)(1.0 / (1.0 - pow(b2, t))), 1e-8f};
}

extern "C" rbf_status rbf_mlp_grad(rbf_ctx* ctx, const float* d_params, const float* d_x, const float* d_t, int batch,
                                   float* d_grad, float* h_loss) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!d_params || !d_x || !d_t || !d_grad || batch < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_mlp_grad: bad argument");
    return mlp_grad_impl(ctx, d_params, d_x, d_t, batch, d_grad, h_loss, nullptr);
}

extern "C" rbf_status rbf_mlp_adam(rbf_ctx* ctx, float* d_params, float* d_m, float* d_v, const float* d_grad, int t,
                                   float lr) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!d_params || !d_m || !d_v || !d_grad || t < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_mlp_adam: bad argument");
    k_adam<<<(NPAR + 127) / 128, 128, 0, ctx->stream>>>(d_grad, adam_args(d_params, d_m, d_v, t, lr));
    RBF_LAUNCHED(ctx, "k_adam");
    return RBF_OK;
}

extern "C" rbf_status rbf_mlp_train_step(rbf_ctx* ctx, float* d_params, float* d_m, float* d_v, int t, float lr,
                                         const float* d_x, const float* d_t, int batch, float* d_grad, float* h_loss) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!d_grad) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_mlp_train_step: gradient buffer required");
    if (!d_m || !d_v || t < 1) {  // the update is refused after the gradient has been written
        RBF_TRY(rbf_mlp_grad(ctx, d_params, d_x, d_t, batch, d_grad, h_loss));
        return rbf_mlp_adam(ctx, d_params, d_m, d_v, d_grad, t, lr);
    }
    if (!d_params || !d_x || !d_t || batch < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_mlp_grad: bad argument");
    const AdamArgs o = adam_args(d_params, d_m, d_v, t, lr);
    return mlp_grad_impl(ctx, d_params, d_x, d_t, batch, d_grad, h_loss, &o);
}

extern "C" rbf_status rbf_stop_features(rbf_ctx* ctx, const rbf_gkb_state* st, int j, const float* d_mean,
                                        const float* d_std, float* d_feat) {
    if (!ctx) return RBF_ERR_INVALID;
    if (!st || !d_feat) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_stop_features: NULL argument");
    if (j < 1 || j > 10 || st->steps_done < j)
        return rbf_fail(ctx, RBF_ERR_INVALID, "features need 1 <= j <= 10 completed steps (have %d)", st->steps_done);
    const size_t need = ws_align((size_t)j * 8) + ws_align((size_t)(j + 1) * 8) + ws_align((size_t)j * j * 8) +
                        svd_ws_bytes(j);
    RBF_TRY(rbf_ws_reserve(ctx, need));
    WsCarve wc(ctx->ws);
    double* sigma = wc.take<double>(j);
    double* ftil = wc.take<double>(j + 1);
    double* V = wc.take<double>((size_t)j * j);
    void* svd = (void*)wc.take<char>(svd_ws_bytes(j));
    RBF_TRY(launch_projected_svd(ctx, st->d_alpha, st->d_beta, j, sigma, ftil, V, j, svd));
    k_stop_features<<<1, 32, 0, ctx->stream>>>(st->d_alpha, st->d_beta, sigma, j, d_mean, d_std, d_feat);
    RBF_LAUNCHED(ctx, "k_stop_features");
    return RBF_OK;
}

rbf_status launch_stop_features_batch(rbf_ctx* ctx, const double* alpha, const double* beta, const double* sigma,
                                      int L, const int* d_l, int B, int j, const float* mean, const float* stdv,
                                      float* feat) {
    k_stop_features_batch<<<B, 32, 0, ctx->stream>>>(alpha, beta, sigma, L, d_l, j, mean, stdv, feat);
    RBF_LAUNCHED(ctx, "k_stop_features_batch");
    return RBF_OK;
}
