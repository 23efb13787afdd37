// Full SVD of the assembled FP64 collocation matrix (Algorithm 3 step 1) and
// the full-SVD methods on top of it: Tikhonov with GCV (Algorithm 3, eqs.
// gcv_svd and tikh_svd_solution) and TSVD (eq. tsvd_solution).
//
// Default: Householder bidiagonalization A = Q_L B Q_R^T in one cooperative
// kernel (f rides along as an extra column, so that g = Q_L^T f comes out of
// the same passes; two bounded grid barriers per step), then the SVD of
// the bidiagonal through the Golub-Kahan tridiagonal (the projected-SVD
// kernels with C = [B^T; 0]: sigma, V~ = U_B and U~ = V_B), f^ = V~^T g and
// alpha = Q_R (U~ d).
//
// Option svd_method = 1: one-sided (Hestenes) Jacobi (high relative accuracy
// for small singular values, far more work): the columns of W = A are rotated in
// pairs until they are mutually orthogonal (W = U Sigma, V = product of the
// rotations).  One cooperative kernel per sweep: each round pairs the columns
// by the circle method (n/2 disjoint pairs), one CTA per pair: the three dot
// products |w_i|^2, |w_j|^2, w_i.w_j in one pass, the rotation that zeroes
// w_i.w_j applied to w_i, w_j and v_i, v_j; a bounded grid barrier separates
// the rounds.  Sweeps repeat until no pair needed a rotation (|w_i.w_j| <=
// sqrt(n) eps |w_i| |w_j|).  Then sigma_j = |w_j| sorted descending and
// f^ = W^T f / sigma.
//
// Both: numerical rank r = #{sigma_i > N eps sigma_1}, s_perp = sum_{i>r}
// f^_i^2, the GCV grid (Tikhonov) or rank curve (TSVD), the solution alpha.
#include <algorithm>
#include <cfloat>
#include <vector>

#include "common.cuh"
#include "grid_sync.cuh"
#include "internal.h"

namespace {

constexpr int JT = 256;
constexpr int JW = JT / 32;
constexpr int MAX_SWEEPS = 40;

// W[j ldw + i] = A[i lda + j] (column j of A contiguous), V = I when given.
__global__ void k_fsvd_init(const double* __restrict__ A, int64_t lda, int64_t n, double* __restrict__ W, int64_t ldw,
                            double* __restrict__ V) {
    __shared__ double t[32][33];
    const int64_t i0 = (int64_t)blockIdx.y * 32, j0 = (int64_t)blockIdx.x * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int64_t i = i0 + r, j = j0 + threadIdx.x;
        t[r][threadIdx.x] = (i < n && j < n) ? A[i * lda + j] : 0.0;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int64_t j = j0 + r, i = i0 + threadIdx.x;
        if (i < n && j < n) {
            W[j * ldw + i] = t[threadIdx.x][r];
            if (V) V[j * n + i] = i == j ? 1.0 : 0.0;
        }
    }
}

__device__ __forceinline__ int circle_pos(int k, int r, int np) { return k == 0 ? 0 : 1 + (k - 1 + r) % (np - 1); }

// Block-wide sums of three values, result in every thread.
__device__ __forceinline__ void block_sum3(double& a, double& b, double& c, double (*red)[JW]) {
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) {
        red[0][warp] = a;
        red[1][warp] = b;
        red[2][warp] = c;
    }
    __syncthreads();
    a = b = c = 0.0;
#pragma unroll
    for (int w = 0; w < JW; ++w) {
        a += red[0][w];
        b += red[1][w];
        c += red[2][w];
    }
}

__global__ void __launch_bounds__(JT) k_jacobi_sweep(double* __restrict__ W, double* __restrict__ V, int64_t n,
                                                     int np, double tol, rbf_dev_state* __restrict__ stt,
                                                     unsigned* __restrict__ bar, int group, long long budget,
                                                     int* __restrict__ rot_out) {
    __shared__ double red[3][JW];
    int nrot = 0;
    for (int r = 0; r < np - 1; ++r) {
        for (int p = blockIdx.x; p < np / 2; p += gridDim.x) {
            int i = circle_pos(p, r, np), j = circle_pos(np - 1 - p, r, np);
            if (i >= n || j >= n) continue;  // the dummy column of an odd n
            if (i > j) {
                const int t = i;
                i = j;
                j = t;
            }
            double* wi = W + (int64_t)i * n;
            double* wj = W + (int64_t)j * n;
            double a = 0.0, b = 0.0, g = 0.0;
            for (int64_t k = threadIdx.x; k < n; k += JT) {
                const double x = wi[k], y = wj[k];
                a = fma(x, x, a);
                b = fma(y, y, b);
                g = fma(x, y, g);
            }
            block_sum3(a, b, g, red);
            if (g == 0.0 || !(fabs(g) > tol * sqrt(a) * sqrt(b))) continue;
            const double zeta = (b - a) / (2.0 * g);
            const double t = fabs(zeta) > 1e150 ? 0.5 / zeta
                                                 : copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
            const double c = 1.0 / sqrt(fma(t, t, 1.0));
            const double s = c * t;
            for (int64_t k = threadIdx.x; k < n; k += JT) {
                const double x = wi[k], y = wj[k];
                wi[k] = c * x - s * y;
                wj[k] = fma(s, x, c * y);
            }
            double* vi = V + (int64_t)i * n;
            double* vj = V + (int64_t)j * n;
            for (int64_t k = threadIdx.x; k < n; k += JT) {
                const double x = vi[k], y = vj[k];
                vi[k] = c * x - s * y;
                vj[k] = fma(s, x, c * y);
            }
            ++nrot;
        }
        if (!grid_sync(stt, bar, group, budget)) return;
    }
    if (threadIdx.x == 0) rot_out[blockIdx.x] = nrot;
}

// sigma_j = |w_j| (one CTA per column)
__global__ void __launch_bounds__(JT) k_colnorm(const double* __restrict__ W, int64_t n, double* __restrict__ sig) {
    __shared__ double red[3][JW];
    const double* w = W + (int64_t)blockIdx.x * n;
    double a = 0.0, b = 0.0, c = 0.0;
    for (int64_t k = threadIdx.x; k < n; k += JT) a = fma(w[k], w[k], a);
    block_sum3(a, b, c, red);
    if (threadIdx.x == 0) sig[blockIdx.x] = sqrt(a);
}

// perm[rank] = j, descending sigma, ties by index
__global__ void k_sort_rank(const double* __restrict__ sig, int64_t n, int* __restrict__ perm,
                            double* __restrict__ sig_sorted) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double s = sig[j];
    int64_t rank = 0;
    for (int64_t i = 0; i < n; ++i) {
        const double t = sig[i];
        rank += (t > s || (t == s && i < j)) ? 1 : 0;
    }
    perm[rank] = (int)j;
    sig_sorted[rank] = s;
}

// fhat[k] = w_{perm k} . f / sigma_k (0 for a zero column)
__global__ void __launch_bounds__(JT) k_fhat(const double* __restrict__ W, int64_t n, const int* __restrict__ perm,
                                             const double* __restrict__ sig_sorted, const double* __restrict__ f,
                                             double* __restrict__ fhat) {
    __shared__ double red[3][JW];
    const int kk = blockIdx.x;
    const double* w = W + (int64_t)perm[kk] * n;
    double a = 0.0, b = 0.0, c = 0.0;
    for (int64_t k = threadIdx.x; k < n; k += JT) a = fma(w[k], f[k], a);
    block_sum3(a, b, c, red);
    if (threadIdx.x == 0) fhat[kk] = sig_sorted[kk] > 0.0 ? a / sig_sorted[kk] : 0.0;
}

constexpr int FT = 1024;  // threads of the one-block kernels over n

// Block sum of one value over FT threads, in every thread.
__device__ __forceinline__ double ft_sum(double v, double* red) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_sum(red[threadIdx.x & 31]);
}

// rank r = #{sigma_i > n eps sigma_1} (sigma descending) and s_perp = sum_{i >=
// r} fhat_i^2, one block (one thread took 344 us at n = 3001)
__global__ void __launch_bounds__(FT) k_fsvd_rank(const double* __restrict__ sig, const double* __restrict__ fhat,
                                                  int64_t n, int* __restrict__ r_out, double* __restrict__ sperp_out) {
    __shared__ double red[FT / 32];
    const double thr = (double)n * DBL_EPSILON * sig[0];
    const bool some = sig[0] > 0.0;
    double cnt = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += FT) cnt += some && sig[i] > thr ? 1.0 : 0.0;
    const int64_t r = (int64_t)ft_sum(cnt, red);
    double sp = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += FT)
        if (i >= r) sp = fma(fhat[i], fhat[i], sp);
    sp = ft_sum(sp, red);
    if (threadIdx.x == 0) {
        *r_out = (int)r;
        *sperp_out = sp;
    }
}

// Tikhonov GCV on the grid: (sum_{i<r} (1-phi_i)^2 fhat_i^2 + s_perp) / ((n - r) + sum_{i<r} (1-phi_i))^2,
// one CTA per grid point (one thread per point: 1.54 ms at n = 3001)
constexpr int GCV_T = 128;
__global__ void __launch_bounds__(GCV_T)
    k_fsvd_gcv(const double* __restrict__ sig, const double* __restrict__ fhat, int64_t n,
               const int* __restrict__ r_in, const double* __restrict__ sperp, int J, double t_lo, double t_hi,
               double* __restrict__ gcv) {
    __shared__ double red[2][GCV_T / 32];
    const int t = blockIdx.x;
    const int r = *r_in;
    const double lam = sig[0] * exp10(grid_t(t, J, t_lo, t_hi));
    const double l2 = lam * lam;
    double num = 0.0, den = 0.0;
    for (int i = threadIdx.x; i < r; i += GCV_T) {
        const double s = sig[i];
        const double q = l2 / fma(s, s, l2);
        num = fma(q * q, fhat[i] * fhat[i], num);
        den += q;
    }
    num = warp_sum(num);
    den = warp_sum(den);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = num;
        red[1][threadIdx.x >> 5] = den;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    num = 0.0;
    den = (double)(n - r);
    for (int w = 0; w < GCV_T / 32; ++w) {
        num += red[0][w];
        den += red[1][w];
    }
    gcv[t] = (num + *sperp) / (den * den);
}

// TSVD GCV over k = 1..min(r, n-1): (sum_{k<=i<r} fhat_i^2 + s_perp) / (n -
// k)^2, one block: suffix sums by a scan from the end (a thread per k summing
// its own tail did O(n^2) dependent additions)
__global__ void __launch_bounds__(FT)
    k_fsvd_gcv_rank(const double* __restrict__ fhat, int64_t n, const int* __restrict__ r_in,
                    const double* __restrict__ sperp, double* __restrict__ curve) {
    __shared__ double wsum[FT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = *r_in;
    const int64_t kmax = r < n - 1 ? r : n - 1;
    // thread t: terms r - (t + 1) per .. r - t per - 1, added downwards
    const int64_t per = (r + FT - 1) / FT;
    const int64_t i1 = r - (int64_t)threadIdx.x * per > 0 ? r - (int64_t)threadIdx.x * per : 0;
    const int64_t i0 = i1 - per > 0 ? i1 - per : 0;
    double run = 0.0;
    for (int64_t i = i1 - 1; i >= i0; --i) run = fma(fhat[i], fhat[i], run);
    double pre = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(RBF_FULL_MASK, pre, o);
        if (lane >= o) pre += t;
    }
    if (lane == 31) wsum[warp] = pre;
    __syncthreads();
    double acc = *sperp;
    for (int w = 0; w < warp; ++w) acc += wsum[w];
    acc += pre - run;
    for (int64_t i = i1 - 1; i >= i0; --i) {  // acc = sum over the terms past i: k = i + 1
        if (i + 1 <= kmax) {
            const double d = (double)(n - (i + 1));
            curve[i] = acc / (d * d);
        }
        acc = fma(fhat[i], fhat[i], acc);
    }
}

// argmin with lowest index on ties (one block); method 0: Tikhonov (index into
// the grid), 1: TSVD (k = index + 1).  Writes d_i and the choice.
__global__ void k_fsvd_choose(const double* __restrict__ curve, int count, int method, int fixed_mode,
                              double lambda_in, int rank_in, const double* __restrict__ sig,
                              const double* __restrict__ fhat, const int* __restrict__ r_in, int J, double t_lo,
                              double t_hi, double* __restrict__ d, int64_t n, rbf_dev_state* __restrict__ stt) {
    __shared__ double bv[1024];
    __shared__ int bi[1024];
    __shared__ double lam_s;
    __shared__ int k_s;
    double best = INFINITY;
    int besti = 0x7fffffff;
    if (!fixed_mode)
        for (int t = threadIdx.x; t < count; t += blockDim.x) {
            double v = curve[t];
            if (isnan(v)) v = INFINITY;
            if (v < best || (v == best && t < besti)) { best = v; besti = t; }
        }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = besti;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) {
            const double ov = bv[threadIdx.x + off], mv = bv[threadIdx.x];
            const int oi = bi[threadIdx.x + off], mi = bi[threadIdx.x];
            if (ov < mv || (ov == mv && oi < mi)) {
                bv[threadIdx.x] = ov;
                bi[threadIdx.x] = oi;
            }
        }
        __syncthreads();
    }
    const int r = *r_in;
    if (threadIdx.x == 0) {
        int idx = bi[0];
        if (idx < 0 || idx >= count) idx = 0;
        if (method == 0) {
            lam_s = fixed_mode ? lambda_in : sig[0] * exp10(grid_t(idx, J, t_lo, t_hi));
            k_s = r;
            stt->info[IN_INDEX] = fixed_mode ? -1 : idx;
            stt->scal[SC_LAMBDA] = lam_s;
        } else {
            k_s = fixed_mode ? rank_in : idx + 1;
            lam_s = 0.0;
            stt->info[IN_RANK] = k_s;
            stt->scal[SC_LAMBDA] = 0.0;
        }
        stt->scal[SC_SIGMA1] = sig[0];
    }
    __syncthreads();
    const double l2 = lam_s * lam_s;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        double v = 0.0;
        if (method == 0) {
            if (i < r) v = sig[i] * fhat[i] / fma(sig[i], sig[i], l2);
        } else if (i < k_s && sig[i] > 0.0) {
            v = fhat[i] / sig[i];
        }
        d[i] = v;
    }
}

// coef[row] = sum_k V[perm k][row] d_k (V column-major; one thread per row)
__global__ void k_fsvd_lift(const double* __restrict__ V, int64_t n, const int* __restrict__ perm,
                            const double* __restrict__ d, double* __restrict__ coef) {
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= n) return;
    double acc = 0.0;
    for (int64_t k = 0; k < n; ++k) {
        const double dk = d[k];
        if (dk != 0.0) acc = fma(V[(int64_t)perm[k] * n + row], dk, acc);
    }
    coef[row] = acc;
}

// ---------------------------------------------------------------------------
// Householder bidiagonalization path
// ---------------------------------------------------------------------------
constexpr int BT = 256;
constexpr int BW = BT / 32;
template <int NW>
__device__ __forceinline__ double block_sum1(double v, double* red) {
    v = warp_sum(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += red[w];
    return t;
}

// Householder reflector of x = [x0; rest], ss = |rest|^2, in the unnormalised
// form H = I - t w w^T, w = [x0 - beta; rest], H x = beta e_1: t = 1 / (nrm (nrm
// + |x0|)) with nrm = |x| and beta = -sign(x0) nrm; t = 0 (w_0 = 0, beta = x0)
// when the rest is zero or |x|^2 no normal number (|x| < 2^-511, what a matrix of
// low rank leaves after several steps: t would overflow).  The library's square
// root and division: refined estimates in their place shortened the chain by 1 % of
// a solve at n = 1000 (21.3 and 21.1 ms), at an ulp more in t and beta.
struct Refl {
    double t, w0, beta;
};

__device__ __forceinline__ Refl reflector(double x0, double ss) {
    const double q = fma(x0, x0, ss), ax = fabs(x0);
    const unsigned qh = __double2hiint(q);  // (integer tests: a comparison would take its turn in the FP64 chain)
    if (qh < 0x00100000u || (__double2hiint(ss) | __double2loint(ss)) == 0) return Refl{0.0, 0.0, x0};
    const double nrm = sqrt(q), t = qh < 0x7e700000u ? 1.0 / (nrm * (nrm + ax)) : 1.0 / nrm / (nrm + ax);
    const double beta = x0 >= 0.0 ? -nrm : nrm;
    return Refl{t, x0 - beta, beta};
}

// Householder bidiagonalization, one cooperative kernel of one CTA per SM.
// W column-major n x (n+1), the last column f.  On return: dg = diag of
// B, eg = superdiagonal, column n = Q_L^T f, the right reflectors in rows k
// (entries k+2..n-1, unscaled) with taur / scaler.
//
// The stored matrix S lags the reduced one by the rank-2 update of the step
// before: A = S - u y^T - x v^T.  Step k, with two grid barriers:
//   A  (whole columns, column j on CTA j mod G, pieces of 256 rows per warp):
//      apply that update, write S, and take u'^T s_j with the new left reflector
//      u' in the same pass: y'_j = t u'^T s_j, row k: r_j = s_kj - u'_k y'_j
//   -- barrier --  right reflector v' from r
//   B  (blocks of 4 rows over all columns): x'_i = t' sum_j (S_ij - u'_i y'_j)
//      v'_j, and column k + 1 of A with its norm: the next left reflector
//   -- barrier --
// so S is read twice and written once per step (a pass for the products and one
// for the update of each reflector read it four times and wrote it twice), the
// vectors u, x and v sit in shared memory, and the norms come from one partial
// per CTA instead of a pass over the vector in every CTA.  Pass B applies u' to
// the entries first: sum_j S_ij v'_j - u'_i y'^T v' saves an FMA per entry, but
// its difference cancels, and Tikhonov solutions of collocation matrices (singular
// values that fall off fast) come out 2.4 times as far off (n = 1000; n = 500
// 1.6 times).  The FP64 pipe bounds it (5 n^3 / 3 FMAs: 71 ms at n = 3001, 2.7 ms
// at 1000) together with the two barriers and reflector chains per step.  Whole GCV
// Tikhonov solves 46.5 -> 21.1 ms at n = 1000, 386 -> 161 ms at 3001 (21.2 and
// 148 with the cancelling difference).
constexpr int BD_T = 512;
constexpr int BD_W = BD_T / 32;
constexpr int BD_ROWS = 256;  // rows of a column piece (8 per lane)
constexpr int BD_RB = 4;      // rows of a block of pass B: one 32-byte sector per column

struct BidiagArgs {
    double* W;  // ld a multiple of 4
    int64_t n, ld;
    double *dg, *eg, *taur, *scaler;
    double *y, *r, *x, *a;  // [n+1] y' and r by column, x' and column k + 1 of A by row
    ulonglong2* slot;       // [2][G to][G from] |r|^2 (columns past k + 1), |a|^2 (rows past k + 1), with epochs
    rbf_dev_state* stt;
    long long budget;
};

// doubles of dynamic shared memory: u, x (or v) and the new u; partial dots;
// row-k entries; row-block partials
__host__ __device__ inline int64_t bd_cols(int64_t n, int G) { return (n + G) / G + 1; }
__host__ __device__ inline int64_t bd_pieces(int64_t n) { return n / BD_ROWS + 2; }
__host__ __device__ inline int64_t bd_blocks(int64_t n, int G) { return (n / BD_RB + G + 1) / G + 1; }
inline size_t bd_smem(int64_t n, int G) {
    return sizeof(double) * (size_t)(3 * n + bd_cols(n, G) * (bd_pieces(n) + 1) + bd_blocks(n, G) * BD_W * BD_RB);
}

// Grid barrier that carries its own reduction: a CTA sends its partial sum and
// the barrier's number as one 128-bit word to a slot of its own in every CTA's
// row of slots, and one warp of each CTA polls that CTA's row and adds the values
// (in a fixed order).  One store and one load across the L2, where arriving at a
// counter, polling it and then loading the partials takes three trips: the whole
// solve 24.2 -> 21.5 ms at n = 1000 and 157 -> 150 ms at 3001 (with the loads
// ahead of the barriers below and one FMA less per entry in pass B).  All CTAs
// polling one shared row of slots: 22.9 and 154.5 ms, its lines are too hot; one
// load after the other: 27.4 and 166.
__device__ __forceinline__ void bd_fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void bd_publish(ulonglong2* slot, double v, unsigned long long epoch) {
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(slot),
                 "l"(__double_as_longlong(v)), "l"(epoch)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 bd_peek(const ulonglong2* slot) {
    ulonglong2 r;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
                 : "=l"(r.x), "=l"(r.y)
                 : "l"(slot)
                 : "memory");
    return r;
}

// The calling warp waits until all G slots carry `epoch` and adds their values;
// all loads of a lane are in flight together.  Bounded: false after `budget` polls
// (the run is then stopped).
constexpr int BD_SLOTS = 5;  // slots per lane in flight: 160 CTAs in one go
__device__ __forceinline__ bool bd_collect(const ulonglong2* slot, int G, unsigned long long epoch, long long budget,
                                           int lane, double* sum) {
    bool ok = true;
    double t = 0.0;
    for (int b0 = lane; b0 < G; b0 += 32 * BD_SLOTS) {
        ulonglong2 v[BD_SLOTS];
        for (long long it = 0;; ++it) {
            bool all = true;
#pragma unroll
            for (int q = 0; q < BD_SLOTS; ++q)
                v[q] = b0 + 32 * q < G ? bd_peek(slot + b0 + 32 * q) : make_ulonglong2(0, epoch);
#pragma unroll
            for (int q = 0; q < BD_SLOTS; ++q) all = all && v[q].y == epoch;
            if (all) break;
            if (it > budget) {
                ok = false;
                break;
            }
        }
        double d[BD_SLOTS];
#pragma unroll
        for (int q = 0; q < BD_SLOTS; ++q) d[q] = __longlong_as_double((long long)v[q].x);
        t += ((d[0] + d[1]) + (d[2] + d[3])) + d[4];
    }
    *sum = warp_sum(t);
    return __all_sync(RBF_FULL_MASK, ok);
}

__global__ void __launch_bounds__(BD_T) k_bidiag(BidiagArgs g) {
    extern __shared__ double sm[];
    __shared__ double sc[4];
    const int64_t n = g.n, ld = g.ld;
    const int G = gridDim.x, cta = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* W = g.W;
    double* uo = sm;          // left reflector of the step before, then y' of this step
    double* un = sm + n;      // left reflector of this step
    double* xs = sm + 2 * n;  // x of the step before, then v' of this step
    const int pmax = (int)bd_pieces(n);
    double* pd = sm + 3 * n;                 // [columns][pieces] partial dots
    double* sk = pd + bd_cols(n, G) * pmax;  // [columns] row k of the updated columns
    double* rp = sk + bd_cols(n, G);         // [row blocks][warps][rows]
    __shared__ int go;
    unsigned long long epoch = 1;
    const ulonglong2* mine = g.slot + (int64_t)cta * G;
    // warp 0 sends v (the same in every lane) to all CTAs
    auto publish = [&](int e, double v) {
        for (int b = lane; b < G; b += 32) bd_publish(g.slot + ((int64_t)e * G + b) * G + cta, v, epoch);
    };
    // a collected barrier: warp 0 waits; false stops the CTA
    double sum = 0.0;  // (warp 0)
    auto collect = [&](int e) -> bool {
        if (warp == 0) {
            const bool ok = bd_collect(mine + (int64_t)e * G * G, G, epoch, g.budget, lane, &sum);
            bd_fence();  // the others' stores, made before they published, are visible from here on
            if (lane == 0) {
                go = ok;
                if (!ok) {
                    atomicExch(&g.stt->info[IN_ERR], (int)RBF_ERR_TIMEOUT);
                    atomicExch(&g.stt->info[IN_DONE], 1);
                }
            }
        }
        ++epoch;
        __syncthreads();
        return go != 0;
    };
    // column 0 and its norm
    {
        double ss = 0.0;
        for (int64_t i = cta * (int64_t)BD_T + threadIdx.x; i < n; i += (int64_t)G * BD_T) {
            const double v = W[i];
            g.a[i] = v;
            g.x[i] = 0.0;
            if (i > 0) ss = fma(v, v, ss);
        }
        ss = block_sum1<BD_W>(ss, pd);
        for (int64_t i = threadIdx.x; i < n; i += BD_T) uo[i] = 0.0;
        __syncthreads();
        if (warp == 0) {
            bd_fence();
            publish(1, ss);
        }
    }
    double vscale = 0.0;  // 1 once a right reflector is pending
    for (int64_t k = 0; k < n; ++k) {
        // the columns of pass A and the values they need were written by this CTA:
        // the first piece is loaded ahead of the barrier
        const int64_t j0 = k + 1 + (((int64_t)cta - (k + 1)) % G + G) % G;  // first own column past k
        const int nc = j0 <= n ? (int)((n - j0) / G) + 1 : 0;
        const int64_t base = k & ~(int64_t)31;
        const int np = (int)((n - base + BD_ROWS - 1) / BD_ROWS);
        double v[8], yj = 0.0, vj = 0.0;
        auto load = [&](int u, double* v, double* yj, double* vj) {
            const int c = u / np, piece = u - c * np;
            const int64_t j = j0 + (int64_t)c * G;
            const double* col = W + j * ld;
            const int64_t i0 = base + (int64_t)piece * BD_ROWS + lane;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int64_t i = i0 + 32 * q;
                v[q] = i >= k && i < n ? __ldcg(col + i) : 0.0;
            }
            *yj = k > 0 ? __ldcg(g.y + j) : 0.0;
            *vj = j < n && vscale != 0.0 ? __ldcg(g.r + j) : 0.0;
        };
        if (warp < nc * np) load(warp, v, &yj, &vj);
        if (!collect(1)) return;
        // ---- left reflector of column k
        if (warp == 0) {
            const Refl h = reflector(__ldcg(g.a + k), sum);
            if (lane == 0) {
                sc[0] = h.t;
                sc[1] = h.w0;
                un[k] = h.w0;
                xs[k] = 0.0;
                if (cta == 0) g.dg[k] = h.beta;
            }
        }
        for (int64_t i = k + 1 + threadIdx.x; i < n; i += BD_T) {
            un[i] = __ldcg(g.a + i);
            xs[i] = __ldcg(g.x + i);
        }
        // x at row k: its own value, needed by row k of the update
        if (threadIdx.x == BD_T - 1) sc[2] = __ldcg(g.x + k);
        __syncthreads();
        const double t1 = sc[0], uk = sc[1], xk = sc[2];
        // ---- pass A
        for (int u = warp; u < nc * np; u += BD_W) {
            const int c = u / np, piece = u - c * np;
            const int64_t j = j0 + (int64_t)c * G;
            double* col = W + j * ld;
            const int64_t i0 = base + (int64_t)piece * BD_ROWS + lane;
            double vn[8], yn = 0.0, rn = 0.0, dot = 0.0, dot1 = 0.0;
            if (u + BD_W < nc * np) load(u + BD_W, vn, &yn, &rn);  // the next piece while this one is updated
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int64_t i = i0 + 32 * q;
                if (i > k && i < n) {
                    v[q] = fma(-xs[i], vj, fma(-uo[i], yj, v[q]));
                    col[i] = v[q];
                    if (q & 1) dot1 = fma(un[i], v[q], dot1);
                    else dot = fma(un[i], v[q], dot);
                } else if (i == k) {
                    const double s = fma(-xk, vj, fma(-uo[i], yj, v[q]));
                    sk[c] = s;
                    dot = fma(uk, s, dot);
                }
            }
            dot = warp_sum(dot + dot1);
            if (lane == 0) pd[(int64_t)c * pmax + piece] = dot;
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = vn[q];
            yj = yn;
            vj = rn;
        }
        __syncthreads();
        if (warp == 0) {
            double rr = 0.0;
            for (int c = lane; c < nc; c += 32) {
                const int64_t j = j0 + (int64_t)c * G;
                double d = 0.0;
                for (int q = 0; q < np; ++q) d += pd[(int64_t)c * pmax + q];
                const double yj = t1 * d;
                const double r = fma(-uk, yj, sk[c]);
                g.y[j] = yj;
                g.r[j] = r;
                W[j * ld + k] = r;
                if (j > k + 1 && j < n) rr = fma(r, r, rr);
            }
            rr = warp_sum(rr);
            __syncwarp();
            if (k < n - 1) {  // (the other warps' stores came before the barrier above)
                bd_fence();
                publish(0, rr);
            }
        }
        if (k == n - 1) break;
        if (!collect(0)) return;
        // the first entries of pass B, ahead of the reflector
        const int64_t rbase = (k + 1) & ~(int64_t)(BD_RB - 1);
        const int64_t nblk = (n - rbase + BD_RB - 1) / BD_RB;
        const int rl = lane & (BD_RB - 1), cl = lane / BD_RB;
        constexpr int CPW = 32 / BD_RB, CW = BD_W * CPW;  // columns of a warp step, of a CTA step
        const int64_t jb = k + 1 + warp * CPW + cl;
        double first[4];
        {
            const int64_t i = rbase + (int64_t)cta * BD_RB + rl;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                first[q] = cta < nblk && i > k && i < n && jb + q * CW < n ? __ldcg(W + i + (jb + q * CW) * ld) : 0.0;
        }
        // ---- right reflector of row k
        if (warp == 0) {
            const double x0 = __ldcg(g.r + k + 1);
            const Refl h = reflector(x0, sum);
            if (lane == 0) {
                sc[0] = h.t;
                xs[k + 1] = h.w0;
                if (cta == 0) {
                    g.eg[k] = h.beta;
                    g.taur[k] = h.t;  // (k_bidiag_ab turns the two into tau and 1 / w_0)
                    g.scaler[k] = h.w0;
                }
            }
        }
        for (int64_t j = k + 1 + threadIdx.x; j < n; j += BD_T) {
            if (j > k + 1) xs[j] = __ldcg(g.r + j);
            uo[j] = __ldcg(g.y + j);
        }
        __syncthreads();
        const double t2 = sc[0], y1 = uo[k + 1], v1 = xs[k + 1];
        // ---- pass B
        int nb = 0;
        for (int64_t rb = cta; rb < nblk; rb += G, ++nb) {
            const int64_t i = rbase + rb * BD_RB + rl;
            const bool ok = i > k && i < n;
            double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
            if (ok) {
                const double* p = W + i;
                const double ui = un[i];
                auto add = [&](double s, int64_t j, double& acc) { acc = fma(fma(-ui, uo[j], s), xs[j], acc); };
                int64_t j = jb;
                if (nb == 0) {
                    if (j < n) add(first[0], j, a0);
                    if (j + CW < n) add(first[1], j + CW, a1);
                    if (j + 2 * CW < n) add(first[2], j + 2 * CW, a2);
                    if (j + 3 * CW < n) add(first[3], j + 3 * CW, a3);
                    j += 4 * CW;
                }
                for (; j + 3 * CW < n; j += 4 * CW) {
                    const double s0 = __ldcg(p + j * ld), s1 = __ldcg(p + (j + CW) * ld);
                    const double s2 = __ldcg(p + (j + 2 * CW) * ld), s3 = __ldcg(p + (j + 3 * CW) * ld);
                    add(s0, j, a0);
                    add(s1, j + CW, a1);
                    add(s2, j + 2 * CW, a2);
                    add(s3, j + 3 * CW, a3);
                }
                for (; j < n; j += CW) add(__ldcg(p + j * ld), j, a0);
            }
            a0 = (a0 + a1) + (a2 + a3);
#pragma unroll
            for (int o = BD_RB; o < 32; o <<= 1) a0 += __shfl_xor_sync(RBF_FULL_MASK, a0, o);
            if (lane < BD_RB) rp[((int64_t)nb * BD_W + warp) * BD_RB + lane] = a0;
        }
        __syncthreads();
        double ss = 0.0;
        for (int e = threadIdx.x; warp == 0 && e < nb * BD_RB; e += 32) {
            const int q = e / BD_RB, rr = e - q * BD_RB;
            const int64_t i = rbase + ((int64_t)cta + (int64_t)q * G) * BD_RB + rr;
            if (i <= k || i >= n) continue;
            double z0 = 0.0, z1 = 0.0;
#pragma unroll
            for (int w = 0; w < BD_W; w += 2) {
                z0 += rp[((int64_t)q * BD_W + w) * BD_RB + rr];
                z1 += rp[((int64_t)q * BD_W + w + 1) * BD_RB + rr];
            }
            const double xi = t2 * (z0 + z1);
            const double ai = fma(-xi, v1, fma(-un[i], y1, __ldcg(W + (k + 1) * ld + i)));
            g.x[i] = xi;
            g.a[i] = ai;
            if (i > k + 1) ss = fma(ai, ai, ss);
        }
        if (warp == 0) {
            ss = warp_sum(ss);
            __syncwarp();
            bd_fence();
            publish(1, ss);
        }
        double* t = uo;
        uo = un;
        un = t;
        vscale = 1.0;
    }
}

// alpha / beta of C = [B^T; 0] for the tridiagonal SVD: alpha = dg, beta =
// (1, eg, 0); beta_1 only scales f~, which is not used here.  The right
// reflectors (t, w_0) become (t w_0^2, 1 / w_0): I - tau w' w'^T with w'_0 = 1.
__global__ void k_bidiag_ab(const double* __restrict__ dg, const double* __restrict__ eg, int64_t n,
                            double* __restrict__ alpha, double* __restrict__ beta, double* __restrict__ taur,
                            double* __restrict__ scaler) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n - 1) {
        const double t = taur[i], w0 = scaler[i];
        taur[i] = t * w0 * w0;
        scaler[i] = t != 0.0 ? 1.0 / w0 : 0.0;
    }
    if (i < n) alpha[i] = dg[i];
    if (i <= n) beta[i] = i == 0 ? 1.0 : (i < n ? eg[i - 1] : 0.0);
}

// fhat[i] = V~_i . g  (V~ column-major, ld n; one CTA per i)
__global__ void __launch_bounds__(BT) k_vt_g(const double* __restrict__ Vt, int64_t n, const double* __restrict__ g,
                                             double* __restrict__ fhat) {
    __shared__ double red[BW];
    const double* v = Vt + (int64_t)blockIdx.x * n;
    double a = 0.0;
    for (int64_t k = threadIdx.x; k < n; k += BT) a = fma(v[k], g[k], a);
    a = block_sum1<BW>(a, red);
    if (threadIdx.x == 0) fhat[blockIdx.x] = a;
}

// x[row] = sum_i U~[row][i] d_i over the first n rows of U~ (ld n+1): 32 rows x
// 32 column groups per CTA, four chains each (one thread per row: 1.45 ms at n =
// 3001, latency of n dependent FMAs).  Columns with d_i = 0 (beyond the rank) are
// left out: the vector of a zero singular value may have no u part to normalise.
__global__ void __launch_bounds__(1024) k_u_d(const double* __restrict__ Ut, int64_t n, const double* __restrict__ d,
                                              double* __restrict__ x) {
    __shared__ double red[32][33];
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * 32 + lane, ldu = n + 1;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    if (row < n) {
        const double* p = Ut + row;
        int64_t i = grp;
        auto add = [&](int64_t c, double& acc) {
            const double dc = d[c], t = fma(p[c * ldu], dc, acc);
            acc = dc != 0.0 ? t : acc;
        };
        for (; i + 96 < n; i += 128)
#pragma unroll
            for (int u = 0; u < 4; ++u) add(i + 32 * u, a[u]);
        for (; i < n; i += 32) add(i, a[0]);
    }
    red[grp][lane] = (a[0] + a[1]) + (a[2] + a[3]);
    __syncthreads();
    const double t = warp_sum(red[lane][grp]);  // warp grp: row grp of the CTA
    const int64_t out = (int64_t)blockIdx.x * 32 + grp;
    if (lane == 0 && out < n) x[out] = t;
}

// alpha = Q_R z for one vector, by blocks of QB reflectors H_k = I - tau_k v_k
// v_k^T (v_k: 1 at k+1, W's row k times scaler_k beyond): all QB dots of a
// block at once, z' = z - V a with a from the dots and the Gram matrix of the
// block's reflectors (a_q = tau_q (w_q - sum_{p > q} G_qp a_p)).  The Gram
// matrices of all blocks come first (k_qr_gram, one launch).  One grid barrier
// per block; a reflector at a time on one CTA took 17.8 ms at n = 3001 and 2.8
// at 1000 (1.6 and 0.55 ms now, Gram matrices included).
constexpr int QB = 32;
constexpr int QG_ROWS = 512;  // entries of the reflectors per Gram partial
constexpr int QA_T = 256;

__device__ __forceinline__ double refl_entry(const double* __restrict__ W, int64_t ld, const double* scaler,
                                             int64_t k, int64_t j, int64_t last) {
    if (k >= last || j <= k) return 0.0;
    return j == k + 1 ? 1.0 : W[j * ld + k] * scaler[k];
}

// part[chunk][block][p][q] = sum over QG_ROWS entries of v_p v_q, p < q (others 0)
__global__ void __launch_bounds__(QA_T) k_qr_gram(const double* __restrict__ W, int64_t n, int64_t ld,
                                                  const double* __restrict__ scaler, double* __restrict__ part) {
    __shared__ double t[64][QB + 1];
    const int64_t k0 = (int64_t)blockIdx.x * QB;
    const int64_t j0 = (int64_t)blockIdx.y * QG_ROWS, j1 = j0 + QG_ROWS < n ? j0 + QG_ROWS : n;
    const int q = threadIdx.x & (QB - 1), p0 = threadIdx.x / QB;  // pairs (p0 + 8 r, q), r < 4
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t jb = j0; jb < j1; jb += 64) {
        if (jb + 64 > k0 + 1)
            for (int r = p0; r < 64; r += QA_T / QB)
                t[r][q] = jb + r < j1 ? refl_entry(W, ld, scaler, k0 + q, jb + r, n - 1) : 0.0;
        __syncthreads();
        if (jb + 64 > k0 + 1)
            for (int r = 0; r < 64; ++r) {
                const double vq = t[r][q];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (p0 + 8 * u < q) acc[u] = fma(t[r][p0 + 8 * u], vq, acc[u]);
            }
        __syncthreads();
    }
    double* out = part + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * QB * QB;
#pragma unroll
    for (int u = 0; u < 4; ++u) out[(p0 + 8 * u) * QB + q] = acc[u];
}

struct QrArgs {
    const double* W;
    int64_t n, ld;
    const double *taur, *scaler, *gram;
    double* z;
    double *hpart, *gpart;  // [QB][G] and 2 x [QB][groups]
    rbf_dev_state* stt;
    unsigned* bar;
    int group;
    long long budget;
};

// CTA b owns the entries [n b / G, n (b+1) / G) of z, in shared memory with the
// current block's reflectors at them.
__global__ void __launch_bounds__(QA_T) k_qr_apply(QrArgs a) {
    extern __shared__ double qs[];
    __shared__ double dots[QA_T / 32][QB], hs[QB], al[QB], Gs[QB][QB + 1], tau[QB];
    const int64_t n = a.n;
    const int G = gridDim.x;
    const int64_t r0 = n * blockIdx.x / G;
    const int R = (int)(n * (blockIdx.x + 1) / G - r0);
    double* z = qs;            // [R]
    double* vt = qs + R;       // [R][QB + 1]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = threadIdx.x; r < R; r += QA_T) z[r] = a.z[r0 + r];
    unsigned epoch = 0;
    const int64_t nblk = (n - 1 + QB - 1) / QB;
    for (int64_t blk = nblk - 1; blk >= 0; --blk) {
        const int64_t k0 = blk * QB;
        __syncthreads();
        for (int r = warp; r < R; r += QA_T / 32)
            vt[r * (QB + 1) + lane] = refl_entry(a.W, a.ld, a.scaler, k0 + lane, r0 + r, n - 1);
        if (warp == 0) tau[lane] = k0 + lane < n - 1 ? a.taur[k0 + lane] : 0.0;
        for (int e = threadIdx.x; e < QB * QB; e += QA_T) Gs[e / QB][e % QB] = a.gram[blk * QB * QB + e];
        __syncthreads();
        double d = 0.0;
        for (int r = warp; r < R; r += QA_T / 32) d = fma(vt[r * (QB + 1) + lane], z[r], d);
        dots[warp][lane] = d;
        __syncthreads();
        if (warp == 0) {
            d = 0.0;
            for (int w = 0; w < QA_T / 32; ++w) d += dots[w][lane];
            a.hpart[(int64_t)lane * G + blockIdx.x] = d;
        }
        if (!grid_reduce_sync(a.stt, a.bar, a.group, a.budget, ++epoch, a.hpart, a.gpart, hs, QB, (int64_t)2 * QB * G))
            return;
        if (warp == 0) {  // lane p: w_p, the later reflectors' parts removed in order
            double w = hs[lane];
            for (int q = QB - 1; q > 0; --q) {
                const double aq = tau[q] * __shfl_sync(RBF_FULL_MASK, w, q);
                if (lane < q) w = fma(-Gs[lane][q], aq, w);
            }
            al[lane] = tau[lane] * w;
        }
        __syncthreads();
        for (int rr = 0; rr < R; rr += QA_T / 8) {  // 8 lanes per entry
            const int r = rr + threadIdx.x / 8, g8 = threadIdx.x & 7;
            double t = 0.0;
            if (r < R)
#pragma unroll
                for (int u = 0; u < QB / 8; ++u) t = fma(vt[r * (QB + 1) + g8 + 8 * u], al[g8 + 8 * u], t);
            t += __shfl_xor_sync(RBF_FULL_MASK, t, 1);
            t += __shfl_xor_sync(RBF_FULL_MASK, t, 2);
            t += __shfl_xor_sync(RBF_FULL_MASK, t, 4);
            if (g8 == 0 && r < R) z[r] -= t;
        }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < R; r += QA_T) a.z[r0 + r] = z[r];
}

// Z <- Q_R Z, one CTA per column (ld ldz): the right reflectors in reverse order.
__global__ void __launch_bounds__(BT) k_apply_qr(const double* __restrict__ W, int64_t n, int64_t ld,
                                                 const double* __restrict__ taur, const double* __restrict__ scaler,
                                                 double* __restrict__ Z, int64_t ldz) {
    __shared__ double red[BW];
    double* z = Z + (int64_t)blockIdx.x * ldz;
    for (int64_t k = n - 2; k >= 0; --k) {
        const double tau = taur[k];
        if (tau == 0.0) continue;
        const double scale = scaler[k];
        const int64_t m2 = n - k - 1;
        const double z0 = z[k + 1];
        double sd = 0.0;
        for (int64_t c = 1 + threadIdx.x; c < m2; c += BT) sd = fma(W[(k + 1 + c) * ld + k], z[k + 1 + c], sd);
        sd = block_sum1<BW>(sd, red);
        const double t = tau * fma(scale, sd, z0);
        const double ts = t * scale;
        for (int64_t c = 1 + threadIdx.x; c < m2; c += BT) z[k + 1 + c] = fma(-ts, W[(k + 1 + c) * ld + k], z[k + 1 + c]);
        if (threadIdx.x == 0) z[k + 1] = z0 - t;
        __syncthreads();
    }
}

// out[:, k] = V[:, perm k] (column-major)
__global__ void k_gather_cols(const double* __restrict__ V, int64_t n, const int* __restrict__ perm,
                              double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t k = blockIdx.y;
    if (i < n) out[k * n + i] = V[(int64_t)perm[k] * n + i];
}

// out[:, k] = U~[0..n-1, k] (drop the last row of U~, ld n+1 -> n)
__global__ void k_copy_ut(const double* __restrict__ Ut, int64_t n, double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t k = blockIdx.y;
    if (i < n) out[k * n + i] = Ut[k * (n + 1) + i];
}

constexpr int64_t TGK_MAX_N = 8192;

// Result of either path.
struct Fsvd {
    bool tgk;
    int64_t n;
    double *sig, *fhat, *d, *curve, *sperp;
    int* r;
    // Jacobi
    double *W, *V;
    int* perm;
    // bidiagonalization
    double *Wb, *taur, *scaler, *Vt, *Ut;
    int64_t ldw;
    double *gram, *gram_part, *hpart, *gpart;  // blocked application of Q_R
    unsigned* bar;
    int G, group, bar_k;
    int sweeps;
};

int coop_grid(rbf_ctx* ctx, const void* kernel, int threads, int cap, int* group, int* bar_k, size_t smem = 0) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        occ = 1;
    }
    int G = ctx->sm_count * (occ < 1 ? 1 : occ);
    if (G > cap) G = cap;
    if (G < 1) G = 1;
    int gr = 1;
    while (gr * gr < G) ++gr;
    *group = gr;
    *bar_k = (G + gr - 1) / gr;
    return G;
}

rbf_status fsvd_common_tail(rbf_ctx* ctx, Fsvd* F, const double* f) {
    cudaStream_t s = ctx->stream;
    if (f) {
        k_fsvd_rank<<<1, FT, 0, s>>>(F->sig, F->fhat, F->n, F->r, F->sperp);
        RBF_LAUNCHED(ctx, "k_fsvd_rank");
    }
    return RBF_OK;
}

// Jacobi path
rbf_status fsvd_jacobi(rbf_ctx* ctx, const rbf_operator* op, const double* f, Fsvd* F) {
    const int64_t n = op->n;
    const int np = (int)(n + (n & 1));
    int group, bar_k;
    const int G = coop_grid(ctx, (const void*)k_jacobi_sweep, JT, np / 2, &group, &bar_k);
    const int J = ctx->opt.grid_j;
    const size_t need = 2 * ws_align((size_t)n * n * 8) + 5 * ws_align((size_t)n * 8) +
                        ws_align((size_t)(J > n ? J : n) * 8) + ws_align(8) + ws_align((size_t)n * 4) + ws_align(4) +
                        ws_align((size_t)G * 4) + ws_align((size_t)(bar_k + 2) * BAR_STRIDE * 4) + 4096;
    RBF_TRY(rbf_ws_reserve(ctx, need));
    WsCarve wc(ctx->ws);
    F->tgk = false;
    F->n = n;
    F->W = wc.take<double>((size_t)n * n);
    F->V = wc.take<double>((size_t)n * n);
    double* sig_raw = wc.take<double>((size_t)n);
    F->sig = wc.take<double>((size_t)n);
    F->fhat = wc.take<double>((size_t)n);
    F->d = wc.take<double>((size_t)n);
    F->curve = wc.take<double>((size_t)(J > n ? J : n));
    F->sperp = wc.take<double>(1);
    F->perm = wc.take<int>((size_t)n);
    F->r = wc.take<int>(1);
    int* rotc = wc.take<int>((size_t)G);
    unsigned* bar = wc.take<unsigned>((size_t)(bar_k + 2) * BAR_STRIDE);
    cudaStream_t s = ctx->stream;
    RBF_CUDA(ctx, cudaMemsetAsync(bar, 0, (size_t)(bar_k + 2) * BAR_STRIDE * sizeof(unsigned), s));
    RBF_CUDA(ctx, cudaMemsetAsync(&ctx->d_state->info[IN_ERR], 0, 2 * sizeof(int), s));  // IN_DONE, IN_ERR
    dim3 tb(32, 8), tg((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32));
    k_fsvd_init<<<tg, tb, 0, s>>>((const double*)op->d_A, op->lda, n, F->W, n, F->V);
    RBF_LAUNCHED(ctx, "k_fsvd_init");
    double tol = sqrt((double)n) * DBL_EPSILON;
    long long budget = ctx->opt.wait_budget;
    std::vector<int> rot((size_t)G);
    int sweeps = 0;
    for (; sweeps < MAX_SWEEPS; ++sweeps) {
        double* Wp = F->W;
        double* Vp = F->V;
        int64_t nn = n;
        int npp = np;
        rbf_dev_state* stt = ctx->d_state;
        int grp = group;
        int* rp = rotc;
        unsigned* bp = bar;
        void* args[] = {&Wp, &Vp, &nn, &npp, &tol, &stt, &bp, &grp, &budget, &rp};
        RBF_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)k_jacobi_sweep, dim3(G), dim3(JT), args, 0, s));
        ctx->launches++;
        int err = 0;
        RBF_CUDA(ctx, cudaMemcpyAsync(rot.data(), rotc, sizeof(int) * G, cudaMemcpyDeviceToHost, s));
        RBF_CUDA(ctx, cudaMemcpyAsync(&err, &ctx->d_state->info[IN_ERR], sizeof(int), cudaMemcpyDeviceToHost, s));
        RBF_CUDA(ctx, cudaStreamSynchronize(s));
        if (err) return rbf_fail(ctx, (rbf_status)err, "a bounded grid barrier of the Jacobi sweep gave up");
        long long total = 0;
        for (int q = 0; q < G; ++q) total += rot[q];
        if (total == 0) {
            ++sweeps;
            break;
        }
    }
    F->sweeps = sweeps;
    k_colnorm<<<(unsigned)n, JT, 0, s>>>(F->W, n, sig_raw);
    RBF_LAUNCHED(ctx, "k_colnorm");
    k_sort_rank<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(sig_raw, n, F->perm, F->sig);
    RBF_LAUNCHED(ctx, "k_sort_rank");
    if (f) {
        k_fhat<<<(unsigned)n, JT, 0, s>>>(F->W, n, F->perm, F->sig, f, F->fhat);
        RBF_LAUNCHED(ctx, "k_fhat");
    }
    return fsvd_common_tail(ctx, F, f);
}

// Bidiagonalization path
rbf_status fsvd_bidiag(rbf_ctx* ctx, const rbf_operator* op, const double* f, Fsvd* F) {
    const int64_t n = op->n;
    const int J = ctx->opt.grid_j;
    const int L = (int)n;
    const size_t smem = bd_smem(n, ctx->sm_count);
    RBF_CUDA(ctx, smem_limit<k_bidiag>(ctx, smem));
    F->G = coop_grid(ctx, (const void*)k_bidiag, BD_T, ctx->sm_count, &F->group, &F->bar_k, smem);
    const int G = F->G;
    if (G != ctx->sm_count) return rbf_fail(ctx, RBF_ERR_INTERNAL, "bidiagonalization grid of %d CTAs", G);
    const int64_t qblk = (n - 1 + QB - 1) / QB, qchunk = (n + QG_ROWS - 1) / QG_ROWS;
    F->ldw = (n + 3) & ~(int64_t)3;
    // the bidiagonalization's vectors and slots are needed before the tridiagonal SVD's
    // scratch is, the dot products and Gram matrices of Q_R after it: one place for all
    const size_t early = 4 * ws_align((size_t)(n + 2) * 8) + ws_align((size_t)2 * G * G * sizeof(ulonglong2));
    const size_t late = 2 * ws_align((size_t)2 * QB * G * 8) + ws_align((size_t)qchunk * qblk * QB * QB * 8) +
                        ws_align((size_t)qblk * QB * QB * 8);
    const size_t scratch = std::max(svd_ws_bytes(L), std::max(early, late));
    const size_t need = ws_align((size_t)F->ldw * (n + 1) * 8) + ws_align((size_t)n * n * 8) +
                        ws_align((size_t)(n + 1) * n * 8) + 10 * ws_align((size_t)(n + 2) * 8) +
                        ws_align((size_t)(J > n ? J : n) * 8) + ws_align(8) + ws_align(4) +
                        ws_align((size_t)(F->bar_k + 2) * BAR_STRIDE * 4) + ws_align(scratch);
    RBF_TRY(rbf_ws_reserve(ctx, need));
    WsCarve wc(ctx->ws);
    F->tgk = true;
    F->n = n;
    F->sweeps = 0;
    F->Wb = wc.take<double>((size_t)F->ldw * (n + 1));
    F->Vt = wc.take<double>((size_t)n * n);
    F->Ut = wc.take<double>((size_t)(n + 1) * n);
    double* dg = wc.take<double>((size_t)n + 2);
    double* eg = wc.take<double>((size_t)n + 2);
    F->taur = wc.take<double>((size_t)n + 2);
    F->scaler = wc.take<double>((size_t)n + 2);
    double* alpha = wc.take<double>((size_t)n + 2);
    double* beta = wc.take<double>((size_t)n + 2);
    double* ftil = wc.take<double>((size_t)n + 2);
    F->sig = wc.take<double>((size_t)n + 2);
    F->fhat = wc.take<double>((size_t)n + 2);
    F->d = wc.take<double>((size_t)n + 2);
    F->curve = wc.take<double>((size_t)(J > n ? J : n));
    F->sperp = wc.take<double>(1);
    F->r = wc.take<int>(1);
    F->bar = wc.take<unsigned>((size_t)(F->bar_k + 2) * BAR_STRIDE);
    void* svd = (void*)wc.take<char>(scratch);
    WsCarve before(svd), after(svd);
    double* vec[4];
    for (double*& v : vec) v = before.take<double>((size_t)n + 2);
    ulonglong2* slot = before.take<ulonglong2>((size_t)2 * G * G);
    F->hpart = after.take<double>((size_t)QB * G);
    F->gpart = after.take<double>((size_t)2 * QB * G);
    F->gram_part = after.take<double>((size_t)qchunk * qblk * QB * QB);
    F->gram = after.take<double>((size_t)qblk * QB * QB);
    cudaStream_t s = ctx->stream;
    const size_t bar_bytes = (size_t)(F->bar_k + 2) * BAR_STRIDE * sizeof(unsigned);
    RBF_CUDA(ctx, cudaMemsetAsync(slot, 0, (size_t)2 * G * G * sizeof(ulonglong2), s));
    RBF_CUDA(ctx, cudaMemsetAsync(F->bar, 0, bar_bytes, s));
    RBF_CUDA(ctx, cudaMemsetAsync(&ctx->d_state->info[IN_ERR], 0, 2 * sizeof(int), s));
    RBF_CUDA(ctx, cudaMemsetAsync(F->taur, 0, sizeof(double) * (n + 2), s));
    // W = [A f] column-major
    dim3 tb(32, 8), tg((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32));
    k_fsvd_init<<<tg, tb, 0, s>>>((const double*)op->d_A, op->lda, n, F->Wb, F->ldw, nullptr);
    RBF_LAUNCHED(ctx, "k_fsvd_init");
    double* g = F->Wb + n * F->ldw;  // f, then Q_L^T f
    if (f) RBF_CUDA(ctx, cudaMemcpyAsync(g, f, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    else RBF_CUDA(ctx, cudaMemsetAsync(g, 0, sizeof(double) * n, s));
    {
        BidiagArgs a{F->Wb, n,      F->ldw, dg,     eg,   F->taur,      F->scaler, vec[0], vec[1],
                     vec[2], vec[3], slot,   ctx->d_state, ctx->opt.wait_budget};
        void* args[] = {&a};
        RBF_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)k_bidiag, dim3(G), dim3(BD_T), args, smem, s));
        ctx->launches++;
    }
    int err = 0;
    RBF_CUDA(ctx, cudaMemcpyAsync(&err, &ctx->d_state->info[IN_ERR], sizeof(int), cudaMemcpyDeviceToHost, s));
    RBF_CUDA(ctx, cudaStreamSynchronize(s));
    if (err) return rbf_fail(ctx, (rbf_status)err, "a bounded grid barrier of the bidiagonalization gave up");
    k_bidiag_ab<<<(unsigned)((n + 256) / 256), 256, 0, s>>>(dg, eg, n, alpha, beta, F->taur, F->scaler);
    RBF_LAUNCHED(ctx, "k_bidiag_ab");
    ProjDims dd{1, L, L, nullptr};
    RBF_TRY(launch_projected_svd_batch(ctx, dd, alpha, beta, F->sig, ftil, F->Vt, n, svd, nullptr, nullptr, F->Ut,
                                       n + 1));
    if (f) {
        k_vt_g<<<(unsigned)n, BT, 0, s>>>(F->Vt, n, g, F->fhat);
        RBF_LAUNCHED(ctx, "k_vt_g");
    }
    return fsvd_common_tail(ctx, F, f);
}

// z <- Q_R z for one vector
rbf_status fsvd_apply_qr(rbf_ctx* ctx, const Fsvd* F, double* z) {
    const int64_t n = F->n;
    cudaStream_t s = ctx->stream;
    const int64_t qblk = (n - 1 + QB - 1) / QB, qchunk = (n + QG_ROWS - 1) / QG_ROWS;
    k_qr_gram<<<dim3((unsigned)qblk, (unsigned)qchunk), QA_T, 0, s>>>(F->Wb, n, F->ldw, F->scaler, F->gram_part);
    RBF_LAUNCHED(ctx, "k_qr_gram");
    RBF_TRY(launch_reduce_partials(ctx, qblk * QB * QB, (int)qchunk, F->gram_part, F->gram));
    const size_t smem = sizeof(double) * (size_t)((n + F->G - 1) / F->G + 1) * (QB + 2);
    QrArgs a{F->Wb, n, F->ldw, F->taur, F->scaler, F->gram, z, F->hpart, F->gpart, ctx->d_state, F->bar, F->group,
             ctx->opt.wait_budget};
    void* args[] = {&a};
    RBF_CUDA(ctx, smem_limit<k_qr_apply>(ctx, smem));
    RBF_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)k_qr_apply, dim3(F->G), dim3(QA_T), args, smem, s));
    ctx->launches++;
    return RBF_OK;
}

rbf_status fsvd_run(rbf_ctx* ctx, const rbf_operator* op, const double* f, Fsvd* F) {
    const int64_t n = op->n;
    if (op->storage != RBF_ASSEMBLED || op->precision != RBF_FP64 || !op->d_A)
        return rbf_fail(ctx, RBF_ERR_UNSUPPORTED, "the full SVD needs an assembled FP64 operator");
    if (n < 2 || n > 8192)
        return rbf_fail(ctx, RBF_ERR_UNSUPPORTED, "full SVD for 2 <= n <= 8192 (n = %lld)", (long long)n);
    return (n <= TGK_MAX_N && ctx->opt.svd_method == 0) ? fsvd_bidiag(ctx, op, f, F) : fsvd_jacobi(ctx, op, f, F);
}

// coef = V d
rbf_status fsvd_lift(rbf_ctx* ctx, const Fsvd* F, double* coef) {
    const int64_t n = F->n;
    cudaStream_t s = ctx->stream;
    if (!F->tgk) {
        k_fsvd_lift<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(F->V, n, F->perm, F->d, coef);
        RBF_LAUNCHED(ctx, "k_fsvd_lift");
        return RBF_OK;
    }
    k_u_d<<<(unsigned)((n + 31) / 32), 1024, 0, s>>>(F->Ut, n, F->d, coef);
    RBF_LAUNCHED(ctx, "k_u_d");
    return fsvd_apply_qr(ctx, F, coef);
}

rbf_status read_state(rbf_ctx* ctx) {
    RBF_CUDA(ctx, cudaMemcpyAsync(ctx->h_state, ctx->d_state, sizeof(rbf_dev_state), cudaMemcpyDeviceToHost,
                                  ctx->stream));
    RBF_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    RBF_CUDA(ctx, cudaGetLastError());
    if (ctx->h_state->info[IN_ERR] != 0)
        return rbf_fail(ctx, (rbf_status)ctx->h_state->info[IN_ERR], "a bounded grid barrier of the full SVD gave up");
    return RBF_OK;
}

}  // namespace

extern "C" rbf_status rbf_svd_full(rbf_ctx* ctx, const rbf_operator* op, const double* d_f, double* d_sigma,
                                   double* d_fhat, double* d_V, int* sweeps) {
    RbfRange range_("rbf_svd_full");
    if (!ctx) return RBF_ERR_INVALID;
    if (!op || !d_sigma || (d_fhat && !d_f)) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_svd_full: bad argument");
    Fsvd F;
    RBF_TRY(fsvd_run(ctx, op, d_fhat ? d_f : nullptr, &F));
    const int64_t n = op->n;
    cudaStream_t s = ctx->stream;
    RBF_CUDA(ctx, cudaMemcpyAsync(d_sigma, F.sig, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    if (d_fhat) RBF_CUDA(ctx, cudaMemcpyAsync(d_fhat, F.fhat, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    if (d_V) {
        if (F.tgk) {
            k_copy_ut<<<dim3((unsigned)((n + 255) / 256), (unsigned)n), 256, 0, s>>>(F.Ut, n, d_V);
            RBF_LAUNCHED(ctx, "k_copy_ut");
            k_apply_qr<<<(unsigned)n, BT, 0, s>>>(F.Wb, n, F.ldw, F.taur, F.scaler, d_V, n);
            RBF_LAUNCHED(ctx, "k_apply_qr");
        } else {
            k_gather_cols<<<dim3((unsigned)((n + 255) / 256), (unsigned)n), 256, 0, s>>>(F.V, n, F.perm, d_V);
            RBF_LAUNCHED(ctx, "k_gather_cols");
        }
    }
    if (sweeps) *sweeps = F.sweeps;
    RBF_CUDA(ctx, cudaStreamSynchronize(s));
    RBF_CUDA(ctx, cudaGetLastError());
    return RBF_OK;
}

extern "C" rbf_status rbf_tikhonov(rbf_ctx* ctx, const rbf_operator* op, const double* d_f, int rule,
                                   double lambda_in, double* d_coef, rbf_solve_info* info) {
    RbfRange range_("rbf_tikhonov");
    if (!ctx) return RBF_ERR_INVALID;
    if (!op || !d_f || !d_coef) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_tikhonov: NULL argument");
    if (rule != RBF_GCV && rule != RBF_FIXED) return rbf_fail(ctx, RBF_ERR_INVALID, "rule must be RBF_GCV or RBF_FIXED");
    if (rule == RBF_FIXED && !(lambda_in >= 0.0)) return rbf_fail(ctx, RBF_ERR_INVALID, "fixed lambda must be >= 0");
    Fsvd F;
    RBF_TRY(fsvd_run(ctx, op, d_f, &F));
    const int64_t n = op->n;
    const int J = ctx->opt.grid_j;
    cudaStream_t s = ctx->stream;
    const double tlo = ctx->opt.grid_t_lo, thi = ctx->opt.grid_t_hi;
    if (rule == RBF_GCV) {
        k_fsvd_gcv<<<J, GCV_T, 0, s>>>(F.sig, F.fhat, n, F.r, F.sperp, J, tlo, thi, F.curve);
        RBF_LAUNCHED(ctx, "k_fsvd_gcv");
    }
    k_fsvd_choose<<<1, 1024, 0, s>>>(F.curve, J, 0, rule == RBF_FIXED, lambda_in, 0, F.sig, F.fhat, F.r, J, tlo, thi,
                                      F.d, n, ctx->d_state);
    RBF_LAUNCHED(ctx, "k_fsvd_choose");
    RBF_TRY(fsvd_lift(ctx, &F, d_coef));
    int r = 0;
    RBF_CUDA(ctx, cudaMemcpyAsync(&r, F.r, sizeof(int), cudaMemcpyDeviceToHost, s));
    RBF_TRY(read_state(ctx));
    if (info) {
        info->lambda = ctx->h_state->scal[SC_LAMBDA];
        info->index = ctx->h_state->info[IN_INDEX];
        info->rank = r;
        info->steps = F.sweeps;
        info->sigma1 = ctx->h_state->scal[SC_SIGMA1];
        info->eta = 0.0;
        info->rho = 0.0;
    }
    return RBF_OK;
}

extern "C" rbf_status rbf_tsvd(rbf_ctx* ctx, const rbf_operator* op, const double* d_f, int rank, double* d_coef,
                               rbf_solve_info* info) {
    RbfRange range_("rbf_tsvd");
    if (!ctx) return RBF_ERR_INVALID;
    if (!op || !d_f || !d_coef) return rbf_fail(ctx, RBF_ERR_INVALID, "rbf_tsvd: NULL argument");
    if (rank < 0 || rank > op->n) return rbf_fail(ctx, RBF_ERR_INVALID, "rank %d outside [0, n]", rank);
    Fsvd F;
    RBF_TRY(fsvd_run(ctx, op, d_f, &F));
    const int64_t n = op->n;
    cudaStream_t s = ctx->stream;
    if (rank == 0) {
        k_fsvd_gcv_rank<<<1, FT, 0, s>>>(F.fhat, n, F.r, F.sperp, F.curve);
        RBF_LAUNCHED(ctx, "k_fsvd_gcv_rank");
    }
    int r = 0;
    RBF_CUDA(ctx, cudaMemcpyAsync(&r, F.r, sizeof(int), cudaMemcpyDeviceToHost, s));
    RBF_CUDA(ctx, cudaStreamSynchronize(s));
    const int kmax = (int)(r < n - 1 ? r : n - 1);
    if (rank == 0 && kmax < 1) return rbf_fail(ctx, RBF_ERR_INVALID, "numerical rank 0: no TSVD solution");
    k_fsvd_choose<<<1, 1024, 0, s>>>(F.curve, kmax, 1, rank != 0, 0.0, rank, F.sig, F.fhat, F.r, ctx->opt.grid_j,
                                      ctx->opt.grid_t_lo, ctx->opt.grid_t_hi, F.d, n, ctx->d_state);
    RBF_LAUNCHED(ctx, "k_fsvd_choose");
    RBF_TRY(fsvd_lift(ctx, &F, d_coef));
    RBF_TRY(read_state(ctx));
    if (info) {
        info->lambda = 0.0;
        info->index = -1;
        info->rank = ctx->h_state->info[IN_RANK];
        info->steps = F.sweeps;
        info->sigma1 = ctx->h_state->scal[SC_SIGMA1];
        info->eta = 0.0;
        info->rho = 0.0;
    }
    return RBF_OK;
}
