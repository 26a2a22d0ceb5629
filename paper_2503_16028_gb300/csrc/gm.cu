// Gaussian-mixture estimation of Alg. 3 / Sec. 2.4 ("estimate a Gaussian
// mixture by samples"; the paper delegates the estimator to Feng2018): EM for
// K diagonal Gaussians on the r leading KL coordinates S of the equally
// weighted particles, prior on every other coordinate.
//   E-step: log p_nj = log w_j + sum_s [-1/2 log(2 pi lambda_js) - (x_ns - m_js)^2 / (2 lambda_js)],
//           g_nj = exp(log p_nj - LSE_j), loglik = sum_n LSE_j.
//   M-step: N_j = sum_n g_nj, w_j = N_j / N, m_j = sum_n g_nj x_n / N_j,
//           lambda_js = max(sum_n g_nj (x_ns - m_js)^2 / N_j, floor * lambda_s).
//   A component with N_j < 2 is re-seeded at the particle with the lowest
//   max_j g_nj (pooled variances, w_j = 1/N); weights are renormalised.
// Initial means: K distinct particles from Philox (purpose EMINIT), variances
// the pooled population variance, w_j = 1/K.  A fixed number of iterations.
#include <algorithm>
#include <cmath>
#include "smcgm_internal.cuh"
#include "common.cuh"

namespace smcgm {

// xsT[s][n] = X[n][S[s]]
__global__ void k_gather_modes(int N, int d, int r, const double* __restrict__ X, const int* __restrict__ S, double* __restrict__ xsT) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)N * r) return;
    const int s = (int)(t / N), n = (int)(t % N);
    xsT[t] = X[(size_t)n * d + S[s]];
}

// pooled population variance per mode (block per s), floored.
__global__ void k_pooled(int N, int r, const double* __restrict__ xsT, const double* __restrict__ lamS, double floor_frac,
                         double* __restrict__ pooled) {
    __shared__ double red[32];
    __shared__ double s_m;
    const int s = blockIdx.x;
    const double* x = xsT + (size_t)s * N;
    double a = 0.0;
    for (int n = threadIdx.x; n < N; n += blockDim.x) a += x[n];
    a = block_sum(a, red);
    if (threadIdx.x == 0) s_m = a / N;
    __syncthreads();
    double v = 0.0;
    for (int n = threadIdx.x; n < N; n += blockDim.x) { const double e = x[n] - s_m; v += e * e; }
    v = block_sum(v, red);
    if (threadIdx.x == 0) pooled[s] = fmax(v / N, floor_frac * lamS[s]);
}

// Initial particles of the components (the Philox picks), passed by value.
struct EmPicks { int idx[MAXK]; };

__global__ void k_em_init(int N, int K, int r, EmPicks init, const double* __restrict__ xsT,
                          const double* __restrict__ pooled, double* __restrict__ w, double* __restrict__ m, double* __restrict__ lam) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < K * r) {
        const int j = t / r, s = t % r;
        m[t] = xsT[(size_t)s * N + init.idx[j]];
        lam[t] = pooled[s];
    }
    if (t < K) w[t] = 1.0 / K;
}

// ------------------------------------------------------------------------
// The whole diagonal EM fit in one cooperative launch.  The work of an iteration is
// small (3 N K r FP64 operations for the E-step, 4 N K r for the M-step: 23 us at N = 4096,
// K = 8, r = 64 on the FP64 pipes of 152 SMs) against the launches and the serial parts of
// separate kernels, so each block keeps its N / gridDim particles in shared memory for all
// iterations and an iteration has two grid barriers:
//   1. E-step and the block's sums of g, g (x - c) and g (x - c)^2 about the pivot c = the
//      component's current mean, to `part` (one row of 2 K r + K values per block);
//   2. each block adds the rows for its slice of the (j, s) pairs, in a fixed order, and
//      writes m = c + S1 / N_j and lambda = max(S2 / N_j - (S1 / N_j)^2, floor lambda_s).
// The pivot moves with the fit, so the subtraction loses nothing once the means settle.  Where a mean moved by more
// than half a standard deviation it could cancel digits (all but 1 / N of S2 at worst), so in such an iteration,
// mostly the first few, all blocks form the sums about the new means again, with two barriers more.
// A collapsed component (N_j < 2) is found by every block alike (same sums, same order).
// Measured (r = 64, 50 iterations, the whole fit): N = 1024, K = 4 9.0 -> 0.97 ms, N = 256, K = 2 7.2 -> 0.84 ms
// (what is left is the chain of FP64 latencies through an iteration, 16 us: an exponential takes 1250
// cycles, a logarithm 2200, a division 500; the FP64 pipe is 6 % busy).
// ------------------------------------------------------------------------
constexpr int EM_THREADS = 256;
constexpr int EM_BLOCKS = 152;      // most blocks of the launch (rows of `part`)
constexpr int EM_MINP = 8;          // least particles per block: fewer blocks make cheaper barriers
constexpr int EM_ETHREADS = EM_THREADS - 32;   // threads of the E-step's densities; the last warp forms the constants meanwhile
constexpr int EM_SPLIT = 4;         // most groups of threads sharing the M-step sums' particles

__host__ __device__ inline int em_pad(int r) { return ((r + 11) / 16) * 16 + 4; }   // >= r, 4 mod 16: rows of 4 s fall on other banks
static size_t em_smem(int K, int r, int per, bool xs_in_smem) {
    return sizeof(double) * ((size_t)2 * K * em_pad(r) + 2 * (size_t)K * per + 3 * (size_t)K + 40 + 2 * EM_THREADS +
                             (xs_in_smem ? (size_t)per * em_pad(r) : 0));
}
size_t em_partial_doubles(int K, int r) { return 2 * (size_t)EM_BLOCKS * (2 * (size_t)K * r + K + 2) + (size_t)K * r; }

struct EmArgs {
    int N, K, r, iters, lg_lanes;   // lanes per (particle, component) in the E-step: 2^lg_lanes
    double floor_frac;
    const double *xsT, *pooled, *lamS;
    double *w, *m, *lam;          // in: the initial mixture; out: the fitted one
    double *part;                 // two buffers of gridDim rows (S1, S2: K r; N_j: K; min of gmax, its particle), then 1 / (2 lambda): K r
    double *loglik;
    unsigned *bar, *again;        // the barrier's counter; the last iteration whose variances need the sums about the new means, plus one
    int* err;
};
constexpr double EM_AGAIN = 0.25;   // |m - c|^2 / lambda above which they do: below it the subtraction costs at most a third of a bit

// Division of a small index (< 2^16) by a divisor known per launch: the high word of a product.
struct EmDiv {
    int d;
    unsigned m;
    __device__ explicit EmDiv(int dd) : d(dd), m(dd > 1 ? 0xffffffffu / (unsigned)dd + 1u : 0u) {}
    __device__ __forceinline__ int quot(int x) const { return d > 1 ? (int)__umulhi((unsigned)x, m) : x; }
};

template <bool XS>
__global__ void __launch_bounds__(EM_THREADS) k_em(EmArgs A) {
    extern __shared__ __align__(16) double sh[];
    const int N = A.N, K = A.K, r = A.r, Kr = K * r, rp = em_pad(r), G = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
    const int per = (N + G - 1) / G, n0 = min(N, b * per), np = min(N, n0 + per) - n0;
    const int row = 2 * Kr + K + 2;
    double* sm = sh;                       // means [K][rp]
    double* si = sm + (size_t)K * rp;      // 1 / (2 lambda) [K][rp]
    double* lp = si + (size_t)K * rp;      // log densities, then responsibilities [K][per]
    double* ex = lp + (size_t)K * per;     // exp(lp - max) [K][per]
    double* cst = ex + (size_t)K * per;    // constants of the log densities
    double* nj = cst + K;
    double* sw = nj + K;                   // weights
    double* red = sw + K;                  // 40
    double* spl = red + 40;                // 2 EM_THREADS: the M-step sums of the second and later thread groups
    double* xs = spl + 2 * EM_THREADS;     // [per][rp]
    double* g_si = A.part + 2 * (size_t)G * row;
    const EmDiv by_np(max(1, np)), by_K(K), by_r(r);
    const int lanes = 1 << A.lg_lanes, split = max(1, min(EM_SPLIT, EM_THREADS / Kr));
    auto X = [&](int p, int s) -> double { return XS ? xs[(size_t)p * rp + s] : A.xsT[(size_t)s * N + n0 + p]; };
    if (XS)
        for (int t = tid; t < np * r; t += EM_THREADS) {
            const int s = t / np, p = t % np;
            xs[(size_t)p * rp + s] = A.xsT[(size_t)s * N + n0 + p];
        }
    for (int t = tid; t < Kr; t += EM_THREADS) {
        const int j = by_r.quot(t), s = t - j * r;
        const double l = A.lam[t];
        sm[(size_t)j * rp + s] = A.m[t];
        si[(size_t)j * rp + s] = 1.0 / (2.0 * l);
    }
    for (int j = tid; j < K; j += EM_THREADS) sw[j] = A.w[j];
    // constants of the initial mixture: lambda = pooled for every component
    {
        double c = 0.0;
        for (int s = tid; s < r; s += EM_THREADS) c += -0.5 * log(2.0 * M_PI * A.lam[s]);
        c = block_sum(c, red);
        if (tid == 0) red[32] = c;
        __syncthreads();
        for (int j = tid; j < K; j += EM_THREADS) cst[j] = log(sw[j]) + red[32];
        __syncthreads();
    }
    const double log_2pi = log(2.0 * M_PI);
    unsigned arrivals = 0;
    for (int it = 0;; ++it) {
        // log densities: 2^lg_lanes lanes per (particle, component)
        const int items = np * K;
        if (tid >= EM_ETHREADS && tid - EM_ETHREADS < K && it > 0) {   // the last warp: the constants, one logarithm each
            const int j = tid - EM_ETHREADS;
            cst[j] = 0.5 * (log(sw[j] * sw[j] / spl[j]) - M_LN2 * spl[MAXK + j]) - 0.5 * r * log_2pi;
        }
        for (int base = 0; tid < EM_ETHREADS && base < items << A.lg_lanes; base += EM_ETHREADS) {
            const int item = (base + tid) >> A.lg_lanes, ln = tid & (lanes - 1);
            const bool on = item < items;
            const int p = on ? by_K.quot(item) : 0, j = on ? item - p * K : 0;
            double acc = 0.0;
            if (on) {
                const double *mj = sm + (size_t)j * rp, *ij = si + (size_t)j * rp;
#pragma unroll 4
                for (int s = ln; s < r; s += lanes) {
                    const double e = X(p, s) - mj[s];
                    acc -= e * e * ij[s];
                }
            }
            for (int o = lanes >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (on && ln == 0) lp[(size_t)j * per + p] = acc;
        }
        __syncthreads();
        for (int t = tid; t < items; t += EM_THREADS) {
            const int j = by_np.quot(t), p = t - j * np;
            double mx = -1.0 / 0.0;
            for (int q = 0; q < K; ++q) mx = fmax(mx, lp[(size_t)q * per + p] + cst[q]);
            ex[(size_t)j * per + p] = exp(lp[(size_t)j * per + p] + cst[j] - mx);
        }
        __syncthreads();
        if (it == A.iters) {               // the final log-likelihood: sum over the particles of LSE_j
            double a = 0.0;
            for (int p = tid; p < np; p += EM_THREADS) {
                double mx = -1.0 / 0.0, sum = 0.0;
                for (int q = 0; q < K; ++q) mx = fmax(mx, lp[(size_t)q * per + p] + cst[q]);
                for (int q = 0; q < K; ++q) sum += ex[(size_t)q * per + p];
                a += mx + log(sum);
            }
            a = block_sum(a, red);
            double* fin = A.part + (size_t)(it & 1) * G * row;
            if (tid == 0) fin[(size_t)b * row] = a;
            if (!grid_barrier(A.bar, arrivals += G, A.err)) return;
            if (b == 0) {
                a = 0.0;
                for (int k = tid; k < G; k += EM_THREADS) a += __ldcg(&fin[(size_t)k * row]);
                a = block_sum(a, red);
                if (tid == 0) *A.loglik = a;
                for (int j = tid; j < K; j += EM_THREADS) A.w[j] = sw[j];
            }
            return;
        }
        double gmin = 1.0 / 0.0;           // least max_j g of the block's particles, lowest index on ties
        int imin = N;
        for (int t = tid; t < items; t += EM_THREADS) {   // responsibilities
            const int j = by_np.quot(t), p = t - j * np;
            double sum = 0.0;
            for (int q = 0; q < K; ++q) sum += ex[(size_t)q * per + p];
            lp[(size_t)j * per + p] = ex[(size_t)j * per + p] / sum;
        }
        __syncthreads();
        double* part = A.part + (size_t)(it & 1) * G * row;   // the other buffer may still be read
        double* out = part + (size_t)b * row;
        auto sums = [&] {                  // of g (x - c) and g (x - c)^2 about the means c in shared memory
            if (split > 1) {                   // few pairs: groups of Kr threads share the particles
                const int h = tid / Kr, q = tid - h * Kr, j = by_r.quot(q), s = q - j * r;
                double s1 = 0.0, s2 = 0.0;
                if (h < split) {
                    const double c = sm[(size_t)j * rp + s];
                    const double* g = lp + (size_t)j * per;
                    for (int p = h; p < np; p += split) {
                        const double e = X(p, s) - c, ge = g[p] * e;
                        s1 += ge;
                        s2 = fma(ge, e, s2);
                    }
                    spl[tid] = s1;
                    spl[EM_THREADS + tid] = s2;
                }
                __syncthreads();
                if (h == 0) {
                    for (int k = 1; k < split; ++k) { s1 += spl[k * Kr + q]; s2 += spl[EM_THREADS + k * Kr + q]; }
                    out[q] = s1;
                    out[Kr + q] = s2;
                }
            } else {
                for (int t = tid; t < Kr; t += EM_THREADS) {
                    const int j = by_r.quot(t), s = t - j * r;
                    const double c = sm[(size_t)j * rp + s];
                    const double* g = lp + (size_t)j * per;
                    double s1 = 0.0, s2 = 0.0;
                    for (int p = 0; p < np; ++p) {
                        const double e = X(p, s) - c, ge = g[p] * e;
                        s1 += ge;
                        s2 = fma(ge, e, s2);
                    }
                    out[t] = s1;
                    out[Kr + t] = s2;
                }
            }
        };
        sums();
        for (int j = tid >> 5; j < K; j += EM_THREADS / 32) {
            double a = 0.0;
            for (int p = tid & 31; p < np; p += 32) a += lp[(size_t)j * per + p];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if ((tid & 31) == 0) out[2 * Kr + j] = a;
        }
        if (tid < 32) {
            for (int p = tid; p < np; p += 32) {
                double gm = 0.0;
                for (int j = 0; j < K; ++j) gm = fmax(gm, lp[(size_t)j * per + p]);
                if (gm < gmin) { gmin = gm; imin = n0 + p; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double og = __shfl_xor_sync(0xffffffffu, gmin, o);
                const int oi = __shfl_xor_sync(0xffffffffu, imin, o);
                if (og < gmin || (og == gmin && oi < imin)) { gmin = og; imin = oi; }
            }
            if (tid == 0) { out[2 * Kr + K] = gmin; out[2 * Kr + K + 1] = (double)imin; }
        }
        if (!grid_barrier(A.bar, arrivals += G, A.err)) return;
        // this block's slice of the pairs, a warp per pair (and N_j alike in every warp that needs it)
        const int lo = (int)((size_t)Kr * b / G), hi = (int)((size_t)Kr * (b + 1) / G), lane = tid & 31, wid = tid >> 5;
        auto nj_of = [&](int j) {
            double a = 0.0;
            for (int k = lane; k < G; k += 32) a += __ldcg(&part[(size_t)k * row + 2 * Kr + j]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            return a;
        };
        for (int q = lo + wid; q < hi; q += EM_THREADS / 32) {
            const int j = by_r.quot(q), s = q - j * r;
            double s1 = 0.0, s2 = 0.0, n = 0.0;
            for (int k = lane; k < G; k += 32) {
                const double* pr = part + (size_t)k * row;
                s1 += __ldcg(&pr[q]);
                s2 += __ldcg(&pr[Kr + q]);
                n += __ldcg(&pr[2 * Kr + j]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
                n += __shfl_xor_sync(0xffffffffu, n, o);
            }
            double mv, lv;
            bool jump = false;
            if (n < 2.0) {                  // rare: re-seeded at the particle with the lowest max_j g
                double bg = 1.0 / 0.0, bi = (double)N;
                for (int k = 0; k < G; ++k) {
                    const double vg = __ldcg(&part[(size_t)k * row + 2 * Kr + K]), vi = __ldcg(&part[(size_t)k * row + 2 * Kr + K + 1]);
                    if (vg < bg || (vg == bg && vi < bi)) { bg = vg; bi = vi; }
                }
                mv = A.xsT[(size_t)s * N + (int)bi];
                lv = A.pooled[s];
            } else {
                const double dm = s1 / n;
                mv = sm[(size_t)j * rp + s] + dm;
                lv = fmax(s2 / n - dm * dm, A.floor_frac * A.lamS[s]);
                jump = dm * dm > EM_AGAIN * lv;
            }
            if (lane == 0) {
                A.m[q] = mv;
                if (jump) atomicExch(A.again, (unsigned)it + 1u);
                A.lam[q] = lv;
                g_si[q] = 1.0 / (2.0 * lv);
            }
        }
        // while the other blocks arrive: N_j, the weights and their logarithms (every block alike)
        grid_arrive(A.bar);
        for (int j = wid; j < K; j += EM_THREADS / 32) {
            const double a = nj_of(j);
            if (lane == 0) nj[j] = a;
        }
        __syncthreads();
        if (tid < K) {                       // w_j = N_j / N (1 / N for a re-seeded one), normalised: N cancels
            double tot = 0.0;
            for (int j = 0; j < K; ++j) tot += nj[j] < 2.0 ? 1.0 : nj[j];
            sw[tid] = (nj[tid] < 2.0 ? 1.0 : nj[tid]) / tot;
        }
        if (!grid_wait(A.bar, arrivals += G, A.err)) return;
        const bool again = __ldcg(A.again) == (unsigned)it + 1u;   // the same in every block: written before the barrier
        for (int t = tid; t < Kr; t += EM_THREADS) {
            const int j = by_r.quot(t), s = t - j * r;
            sm[(size_t)j * rp + s] = __ldcg(&A.m[t]);
            si[(size_t)j * rp + s] = __ldcg(&g_si[t]);
        }
        if (again) {
            // means and variances once more, about the new means: the sums' part of the rows is free (N_j, beside it, may still be read)
            __syncthreads();
            sums();
            if (!grid_barrier(A.bar, arrivals += G, A.err)) return;
            for (int q = lo + wid; q < hi; q += EM_THREADS / 32) {
                const int j = by_r.quot(q), s = q - j * r;
                double s1 = 0.0, s2 = 0.0;
                for (int k = lane; k < G; k += 32) {
                    const double* pr = part + (size_t)k * row;
                    s1 += __ldcg(&pr[q]);
                    s2 += __ldcg(&pr[Kr + q]);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
                }
                if (lane == 0 && !(nj[j] < 2.0)) {
                    const double n = nj[j], dm = s1 / n, lv = fmax(s2 / n - dm * dm, A.floor_frac * A.lamS[s]);
                    A.m[q] = sm[(size_t)j * rp + s] + dm;
                    A.lam[q] = lv;
                    g_si[q] = 1.0 / (2.0 * lv);
                }
            }
            if (!grid_barrier(A.bar, arrivals += G, A.err)) return;
            for (int t = tid; t < Kr; t += EM_THREADS) {
                const int j = by_r.quot(t), s = t - j * r;
                sm[(size_t)j * rp + s] = __ldcg(&A.m[t]);
                si[(size_t)j * rp + s] = __ldcg(&g_si[t]);
            }
        }
        // sum_s log lambda_js as one logarithm per component: the product of the mantissas (in [1, 2), at most 256 of
        // them: no overflow) and the sum of the exponents
        for (int j = wid; j < K; j += EM_THREADS / 32) {
            double prod = 1.0;
            int ex2 = 0;
            for (int s = lane; s < r; s += 32) {
                const double v = __ldcg(&A.lam[(size_t)j * r + s]);
                const int hi2 = __double2hiint(v), e = (hi2 >> 20) & 0x7ff;
                if (e > 0 && e < 0x7ff) {
                    prod *= __hiloint2double((hi2 & 0x800fffff) | 0x3ff00000, __double2loint(v));
                    ex2 += e - 1023;
                } else {
                    prod *= v;               // zero, denormal, infinity, NaN
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                prod *= __shfl_xor_sync(0xffffffffu, prod, o);
                ex2 += __shfl_xor_sync(0xffffffffu, ex2, o);
            }
            if (lane == 0) { spl[j] = prod; spl[MAXK + j] = (double)ex2; }
        }
        __syncthreads();
    }
}

__global__ void k_lamS(int r, const double* __restrict__ lam, const int* __restrict__ S, double* __restrict__ out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < r) out[s] = lam[S[s]];
}

__global__ void k_sum(int N, const double* __restrict__ a, double* __restrict__ out) {
    __shared__ double red[32];
    double s = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) s += a[i];
    s = block_sum(s, red);
    if (threadIdx.x == 0) *out = s;
}

// ------------------------------------------------------------------------
// Full covariances on the mixture modes (cfg.full_cov; a reading beyond the
// paper, whose C_j are diagonal in the KL basis):
//   E-step: log p_nj = log w_j - r/2 log(2 pi) - log det L_j - |L_j^{-1}(x_n - m_j)|^2 / 2,
//   M-step: C_j = sum_n g_nj (x_n - m_j)(x_n - m_j)^T / N_j + floor diag(lambda_S),
//   initial and re-seeded covariances diag(pooled variances).
// An iteration is k_chol, k_estep_full, k_resp, k_cov_mean, k_cov_acc, k_cov_finish.  The E-step and the
// contraction are N K r^2 / 2 FP64 multiply-adds each (108 us at N = 4096, K = 8, r = 64 on the
// FP64 pipes), everything else should stay small beside them.  Measured per 50-iteration fit
// there: 70.2 -> 20.7 ms (one block per particle reading rows of L^-1 uncoalesced 631 -> 150 us, FP64
// pipe 81 % busy: 1.7 warps per scheduler, so some have two; the factor with its column sums in global memory
// 416 -> 69 us; the contraction on 32 x 32 tiles 292 -> 152 us, the pipe all but full).
// ------------------------------------------------------------------------

// Rows in blocks of four: block I holds L[4I + q][k] at 8 I (I + 1) + 4 k + q, k < 4 I + 4, with
// 1 / L_kk on the diagonal (rows beyond r: zero, diagonal 1), so that a substitution step reads the
// four rows' entries of one column as two 16-byte words.
__host__ __device__ inline int row_blocks(int r) { return (r + 3) / 4; }
__host__ __device__ inline int lb_size(int r) { const int R = row_blocks(r); return 8 * R * (R + 1); }
size_t cov_lb_doubles(int K, int r) { return (size_t)K * lb_size(r) + K; }

// Cholesky factor L_j (lower), log det L_j and the blocked rows above of every C_j, one block per
// component, FP64: right-looking in panels of four columns, W_ic -= sum W_ik W_ck / W_kk on the trailing triangle (all
// threads), L_ik = W_ik / sqrt(W_kk) at the end; in shared memory while it fits (r <= CHOL_SMEM_R), else in
// L_j's own storage.  A pivot that is not positive (C_j not positive definite) sets *bad and counts
// as 1 so the rest stays finite.  cst_j = log w_j - r/2 log(2 pi) - log det L_j when w is given.
// Bound by the FP64 pipe of one SM and the pivots' chain: about 48 operations of 64 cycles per panel and
// scheduler, then the update (r^3 / 6 multiply-adds, 11 us at r = 64).  With a column per step, two barriers
// and a pivot chain each: 79 us at r = 64, K = 8; in panels 69.
constexpr int CHOL_SMEM_R = 160;

// 1 / d to an ulp for d in [2^-1000, 2^1000]: the Newton-Raphson iteration y <- y + y (1 - d y) from the hardware's approximate
// reciprocal (some 20 bits), which squares the relative error at each of its two steps; half the latency of a rounded
// division.
__device__ __forceinline__ double rcp_newton(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    y = fma(y, fma(-d, y, 1.0), y);
    return fma(y, fma(-d, y, 1.0), y);
}
// Pivots at the ends of the range, subnormal ones included: a call, so that the common path has no instruction of it.
__device__ __noinline__ double divide(double a, double b) { return a / b; }
template <bool SMEM>
__global__ void __launch_bounds__(256) k_chol(int r, const double* __restrict__ cov, const double* __restrict__ w, double* __restrict__ L,
                                              double* __restrict__ Lb, double* __restrict__ logdet, double* __restrict__ cst,
                                              int* __restrict__ bad) {
    extern __shared__ __align__(16) double chsm[];
    __shared__ double T[4][MAXR], rs[MAXR], red[32];
    const int j = blockIdx.x, tid = threadIdx.x;
    const size_t rr = (size_t)r * r;
    const double* A = cov + j * rr;
    double* Lj = L + j * rr;
    double* Wk = SMEM ? chsm : Lj;
    const int ws = SMEM ? r + 1 : r;
    for (int i = tid >> 5; i < r; i += 8)
        for (int c = tid & 31; c <= i; c += 32) Wk[i * ws + c] = A[i * r + c];
    __syncthreads();
    const int tx = tid & 15, ty = tid >> 4;
    for (int k = 0; k < r; k += 4) {
        // columns k .. k + 3 (beyond r: those of the identity): a thread per row eliminates the 4 x 4 diagonal block, then its row
        const int ri = k + tid;                               // r <= 256 = the threads
        double w[4];
        if (ri < r) {
            double d[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
#pragma unroll
                for (int b = 0; b <= a; ++b) d[a][b] = k + a < r ? Wk[(k + a) * ws + k + b] : a == b ? 1.0 : 0.0;
                w[a] = a <= tid ? Wk[ri * ws + k + a] : 0.0;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const bool pos = d[c][c] > 0.0;
                const double dc = pos ? d[c][c] : 1.0;
                const bool far = (unsigned)((__double2hiint(dc) >> 20) - 23) >= 2000u;    // not in [2^-1000, 2^1000); no FP64 operation
                const double rinv = rcp_newton(dc);
                auto over = [&](double x) { return far ? divide(x, dc) : x * rinv; };
                if (tid == 0 && k + c < r) {
                    rs[k + c] = dc;
                    if (!pos) atomicExch(bad, 1);
                }
#pragma unroll
                for (int b = c + 1; b < 4; ++b) {
                    const double tb = over(d[b][c]);
#pragma unroll
                    for (int a = b; a < 4; ++a) d[a][b] = fma(-d[a][c], tb, d[a][b]);
                    w[b] = fma(-w[c], tb, w[b]);
                }
                T[c][ri] = over(w[c]);
            }
            if (tid >= 4)
#pragma unroll
                for (int a = 0; a < 4; ++a) Wk[ri * ws + k + a] = w[a];
        }
        __syncthreads();
        if (tid < 4 && ri < r)                                // the diagonal block's rows, which every row's thread has read
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (a <= tid) Wk[ri * ws + k + a] = w[a];
        // the trailing triangle, two of a thread's elements at a time
        for (int c0 = k + 4 + tx; c0 < r; c0 += 16) {
            const double t0 = T[0][c0], t1 = T[1][c0], t2 = T[2][c0], t3 = T[3][c0];
            auto upd = [&](int i) {
                const double* q = Wk + i * ws + k;
                return fma(-q[0], t0, fma(-q[1], t1, fma(-q[2], t2, fma(-q[3], t3, Wk[i * ws + c0]))));
            };
            int i = c0 + ((ty - c0) & 15);                    // the first row >= c0 of this thread's rows (ty mod 16)
            for (; i + 16 < r; i += 32) {
                const double u = upd(i), v = upd(i + 16);
                Wk[i * ws + c0] = u;
                Wk[(i + 16) * ws + c0] = v;
            }
            if (i < r) Wk[i * ws + c0] = upd(i);
        }
        __syncthreads();
    }
    double ld = 0.0;
    for (int k = tid; k < r; k += 256) {
        const double sq = sqrt(rs[k]);
        rs[k] = 1.0 / sq;
        T[0][k] = sq;
        ld += log(sq);
    }
    ld = block_sum(ld, red);                 // its barriers also publish rs and T
    if (tid == 0) {
        logdet[j] = ld;
        if (cst) cst[j] = log(w[j]) - 0.5 * r * log(2.0 * M_PI) - ld;
    }
    __syncthreads();
    double* Lbj = Lb + (size_t)j * lb_size(r);
    const int R = row_blocks(r);
    for (int i = tid >> 5; i < 4 * R; i += 8)
        for (int c = tid & 31; c <= (i | 3); c += 32) {
            double v = 0.0;
            if (c == i) v = i < r ? rs[i] : 1.0;
            else if (c < i && i < r) v = Wk[i * ws + c] * rs[c];
            Lbj[8 * (i >> 2) * ((i >> 2) + 1) + 4 * c + (i & 3)] = v;
        }
    __syncthreads();
    for (int i = tid >> 5; i < r; i += 8)
        for (int c = tid & 31; c < r; c += 32) {
            double v = 0.0;
            if (c == i) v = T[0][i];
            else if (c < i) v = Wk[i * ws + c] * rs[c];
            Lj[i * r + c] = v;                // in place when the work array is L_j itself
        }
}

// Forward substitution L y = rhs for 32 right-hand sides, one per lane; ys[i][lane] in shared memory,
// four rows at a time: a step loads one y and two uniform 16-byte words of L for four multiply-adds.
template <class Rhs, class Out>
__device__ __forceinline__ void tri_subst(int r, const double* __restrict__ Lb, double* ys, int lane, Rhs rhs, Out out) {
    const int R = row_blocks(r);
    for (int I = 0; I < R; ++I) {
        const double2* Lp = reinterpret_cast<const double2*>(Lb + 8 * I * (I + 1));
        double a0 = rhs(4 * I), a1 = rhs(4 * I + 1), a2 = rhs(4 * I + 2), a3 = rhs(4 * I + 3);
#pragma unroll 4
        for (int k = 0; k < 4 * I; ++k) {
            const double y = ys[k * 32 + lane];
            const double2 l01 = __ldg(Lp + 2 * k), l23 = __ldg(Lp + 2 * k + 1);
            a0 = fma(-l01.x, y, a0);
            a1 = fma(-l01.y, y, a1);
            a2 = fma(-l23.x, y, a2);
            a3 = fma(-l23.y, y, a3);
        }
        const double2* D = Lp + 8 * I;
        const double2 c0a = __ldg(D), c0b = __ldg(D + 1), c1a = __ldg(D + 2), c1b = __ldg(D + 3), c2b = __ldg(D + 5), c3b = __ldg(D + 7);
        a0 *= c0a.x;
        a1 = fma(-c0a.y, a0, a1) * c1a.y;
        a2 = fma(-c1b.x, a1, fma(-c0b.x, a0, a2)) * c2b.x;
        a3 = fma(-c2b.y, a2, fma(-c1b.y, a1, fma(-c0b.y, a0, a3))) * c3b.y;
        ys[(4 * I) * 32 + lane] = a0;
        ys[(4 * I + 1) * 32 + lane] = a1;
        ys[(4 * I + 2) * 32 + lane] = a2;
        ys[(4 * I + 3) * 32 + lane] = a3;
        out(4 * I, a0, a1, a2, a3);
    }
}

// L_j^{-1} (the proposal's terms use it): its columns are the substitutions of the unit vectors, a
// warp per 32 columns.
__global__ void __launch_bounds__(32) k_tri_inverse(int r, const double* __restrict__ Lb, double* __restrict__ Li) {
    extern __shared__ __align__(16) double ysm[];
    const int j = blockIdx.y, lane = threadIdx.x, col = blockIdx.x * 32 + lane;
    double* out = Li + (size_t)j * r * r;
    tri_subst(r, Lb + (size_t)j * lb_size(r), ysm, lane, [&](int i) { return i == col ? 1.0 : 0.0; },
              [&](int i, double a, double b, double c, double d) {
                  const double v[4] = {a, b, c, d};
#pragma unroll
                  for (int q = 0; q < 4; ++q)
                      if (col < r && i + q < r) out[(size_t)(i + q) * r + col] = v[q];
              });
}

// E-step: log p_nj, a warp per 32 particles of one component (grid y), a particle per lane.
constexpr int ESF_WARPS = 2;
__global__ void __launch_bounds__(32 * ESF_WARPS) k_estep_full(int N, int r, const double* __restrict__ xsT, const double* __restrict__ m,
                                                               const double* __restrict__ Lb, const double* __restrict__ cst,
                                                               double* __restrict__ lp) {
    extern __shared__ __align__(16) double ysm[];
    const int j = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = (blockIdx.x * ESF_WARPS + wid) * 32 + lane, nc = min(n, N - 1);
    const double* mj = m + (size_t)j * r;
    double q = 0.0;
    tri_subst(r, Lb + (size_t)j * lb_size(r), ysm + (size_t)wid * 32 * 4 * row_blocks(r), lane,
              [&](int i) { return i < r ? xsT[(size_t)i * N + nc] - mj[i] : 0.0; },
              [&](int, double a, double b, double c, double d) { q = fma(d, d, fma(c, c, fma(b, b, fma(a, a, q)))); });
    if (n < N) lp[(size_t)j * N + n] = cst[j] - 0.5 * q;
}

// Responsibilities from the log densities (in place), log-sum-exp and largest responsibility of every
// particle: a thread per (component, particle).
__global__ void __launch_bounds__(256) k_resp(int N, int K, double* __restrict__ lp, double* __restrict__ lse, double* __restrict__ gmax) {
    __shared__ double l[256], e[256];
    const int P = 256 / K, p = threadIdx.x % P, j = threadIdx.x / P;
    const int n = blockIdx.x * P + p;
    const bool on = j < K && n < N;
    double v = 0.0, mx = -1.0 / 0.0;
    if (on) v = lp[(size_t)j * N + n];
    l[threadIdx.x] = v;
    __syncthreads();
    if (on) {
        for (int q = 0; q < K; ++q) mx = fmax(mx, l[q * P + p]);
        e[threadIdx.x] = exp(v - mx);
    }
    __syncthreads();
    double g = 0.0, ls = 0.0;
    if (on) {
        double sum = 0.0;
        for (int q = 0; q < K; ++q) sum += e[q * P + p];
        ls = mx + log(sum);
        g = exp(v - ls);
        lp[(size_t)j * N + n] = g;
    }
    __syncthreads();
    l[threadIdx.x] = g;
    __syncthreads();
    if (on && j == 0) {
        double gm = 0.0;
        for (int q = 0; q < K; ++q) gm = fmax(gm, l[q * P + p]);
        lse[n] = ls;
        gmax[n] = gm;
    }
}

// The pivots of the contraction: sums_j[s] = sum_n g_nj x_ns, sums_j[r] = N_j, a block each.  Their quotient is the new mean to
// rounding (about the old one the subtraction of (m - c)(m - c)^T cancels digits where a mean jumps, all but
// 1 / N at worst); k_cov_finish corrects it by the sums about itself.  One FP64 operation per element, 4 us at
// N = 4096, K = 8, r = 64 on the pipe; 8 us per iteration in the fit.
__global__ void __launch_bounds__(256) k_cov_mean(int N, int r, const double* __restrict__ xsT, const double* __restrict__ resp,
                                                  double* __restrict__ sums) {
    __shared__ double red[32];
    const int s = blockIdx.x, j = blockIdx.y;
    const double *x = xsT + (size_t)s * N, *g = resp + (size_t)j * N;
    double b = 0.0;
    if (s < r) {
#pragma unroll 8
        for (int n = threadIdx.x; n < N; n += 256) b = fma(g[n], x[n], b);
    } else {
#pragma unroll 8
        for (int n = threadIdx.x; n < N; n += 256) b += g[n];
    }
    b = block_sum(b, red);
    if (threadIdx.x == 0) sums[(size_t)j * (r + 1) + s] = b;
}

// The contraction sum_n g_nj (x_n - c_j)(x_n - c_j)^T about the pivot c_j of k_cov_mean,
// with sum_n g_nj (x_n - c_j) and N_j, over one chunk of the particles (grid z): each thread
// holds one 4 x 4 tile of the lower triangle (136 tiles at r = 64: 5 % more products than the triangle
// itself; 32 x 32 tiles took 48 % more), 16 particles' deviations staged in shared memory per step.
// 136 tiles are four warps and a quarter: the lanes of the partial warp divide each step's particles among
// them, so that it costs the FP64 pipe a quarter of a warp (173 -> 152 us at N = 4096, K = 8, r = 64).
// k_cov_finish adds the chunks in a fixed order.
constexpr int COV_PN = 16;
__host__ __device__ inline int cov_tiles(int r) { const int R = row_blocks(r); return R * (R + 1) / 2; }
__host__ __device__ inline size_t cov_row(int r) { return (size_t)cov_tiles(r) * 16 + r + 1; }   // values per (component, chunk)
// chunks: about two blocks of 256 threads per SM in all
__host__ __device__ inline int cov_chunks(int K, int r) {
    const int c = 304 / (K * ((cov_tiles(r) + 255) / 256));
    return c < 1 ? 1 : c > 64 ? 64 : c;
}
static size_t cov_sums_at(int K, int r) { return (size_t)K * cov_chunks(K, r) * cov_row(r); }   // k_cov_mean's sums, after the chunks
size_t cov_partial_doubles(int K, int r) { return cov_sums_at(K, r) + (size_t)K * (r + 1); }
static size_t cov_smem(int r) { return sizeof(double) * ((2 * (size_t)COV_PN + 1) * 4 * row_blocks(r) + COV_PN); }

__global__ void __launch_bounds__(256) k_cov_acc(int N, int r, const double* __restrict__ xsT, const double* __restrict__ resp,
                                                 const double* __restrict__ sums, double* __restrict__ part) {
    extern __shared__ __align__(16) double csm[];
    const int j = blockIdx.y, chunk = blockIdx.z, nch = gridDim.z, tid = threadIdx.x, rp = 4 * row_blocks(r);
    double* D = csm;                      // [COV_PN][rp] deviations
    double* Wd = D + COV_PN * rp;         // [COV_PN][rp] weighted deviations
    double* pv = Wd + COV_PN * rp;        // [rp] pivots
    double* gs = pv + rp;
    if (tid < r) pv[tid] = sums[(size_t)j * (r + 1) + tid] / sums[(size_t)j * (r + 1) + r];
    const int T = cov_tiles(r), base = T & ~31, left = T - base;
    // a tile per thread; the last, partial warp's `left` tiles with S lanes each, which share a step's particles
    int t = blockIdx.x * 256 + tid, S = 1, slice = 0;
    if (left && (t & ~31) == base) {
        while (2 * S * left <= 32 && 2 * S <= COV_PN) S *= 2;
        slice = (tid & 31) / left;
        t = slice < S ? base + (tid & 31) % left : T;
    }
    int ta = 0, tb = 0;
    if (t < T) {
        ta = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
        while (ta * (ta + 1) / 2 > t) --ta;
        while ((ta + 1) * (ta + 2) / 2 <= t) ++ta;
        tb = t - ta * (ta + 1) / 2;
    }
    const int per = (N + nch - 1) / nch, n_lo = min(N, chunk * per), n_hi = min(N, n_lo + per);
    const double* g = resp + (size_t)j * N;
    double acc[4][4] = {}, s1 = 0.0, sn = 0.0;
    for (int n0 = n_lo; n0 < n_hi; n0 += COV_PN) {
        if (tid < COV_PN) gs[tid] = n0 + tid < n_hi ? g[n0 + tid] : 0.0;
        __syncthreads();
        for (int e = tid; e < COV_PN * rp; e += 256) {
            const int s = e / COV_PN, p = e % COV_PN;
            const double dv = (s < r && n0 + p < n_hi) ? xsT[(size_t)s * N + n0 + p] - pv[s] : 0.0;
            D[p * rp + s] = dv;
            Wd[p * rp + s] = gs[p] * dv;
        }
        __syncthreads();
        if (t < T) {
            const double *wa = Wd + slice * rp + 4 * ta, *db = D + slice * rp + 4 * tb;
#pragma unroll 4
            for (int p = slice; p < COV_PN; p += S, wa += S * rp, db += S * rp) {
                const double2 a01 = *reinterpret_cast<const double2*>(wa), a23 = *reinterpret_cast<const double2*>(wa + 2);
                const double2 b01 = *reinterpret_cast<const double2*>(db), b23 = *reinterpret_cast<const double2*>(db + 2);
                const double a[4] = {a01.x, a01.y, a23.x, a23.y}, b[4] = {b01.x, b01.y, b23.x, b23.y};
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
            }
        }
        if (blockIdx.x == 0) {
            if (tid < r)
                for (int p = 0; p < COV_PN; ++p) s1 += Wd[p * rp + tid];
            if (tid == 0)
                for (int p = 0; p < COV_PN; ++p) sn += gs[p];
        }
        __syncthreads();
    }
    double* out = part + ((size_t)j * nch + chunk) * cov_row(r);
    for (int h = S / 2; h > 0; h >>= 1)       // the slices of a tile (S differs from 1 in whole warps)
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) acc[x][y] += __shfl_down_sync(0xffffffffu, acc[x][y], h * left);
    if (t < T && slice == 0)
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) out[(size_t)t * 16 + 4 * x + y] = acc[x][y];
    if (blockIdx.x == 0) {
        if (tid < r) out[(size_t)T * 16 + tid] = s1;
        if (tid == 0) out[(size_t)T * 16 + r] = sn;
    }
}

// Adds the chunks and writes C_j (both triangles), its diagonal, m_j and the weights; a component with
// N_j < 2 is re-seeded at the particle with the lowest largest responsibility.  Latency: every chunk is requested
// before the first barrier (one sum after the other 35 us, so 19, caches cold).
__global__ void __launch_bounds__(256) k_cov_finish(int N, int K, int r, int nch, const double* __restrict__ part, const double* __restrict__ sums,
                                                    const double* __restrict__ gmax, const double* __restrict__ xsT, const double* __restrict__ pooled,
                                                    const double* __restrict__ lamS, double floor_frac, double* __restrict__ w,
                                                    double* __restrict__ m, double* __restrict__ lam, double* __restrict__ cov) {
    // four threads per element (and per mode, component) share the chunks
    __shared__ double dm[MAXR], s_nj[MAXK], s_v[2 + MAXR / 64][256];
    __shared__ int s_i[256];
    const int j = blockIdx.y, tid = threadIdx.x, T = cov_tiles(r), cg = tid >> 6, el = tid & 63;
    const size_t row = cov_row(r);
    const double* pj = part + (size_t)j * nch * row;
    auto partial = [&](const double* p0, bool on) {         // a quarter of the sum over the chunks of p0[c * row]
        double a = 0.0;
        if (on)
#pragma unroll 5
            for (int c = cg; c < nch; c += 4) a += p0[c * row];
        return a;
    };
    auto whole = [&](int k) { return (s_v[k][el] + s_v[k][64 + el]) + (s_v[k][128 + el] + s_v[k][192 + el]); };
    const size_t e = (size_t)blockIdx.x * 64 + el;
    // every load before the first barrier: the kernel is their latency
    s_v[0][tid] = partial(part + (size_t)min(el, K - 1) * nch * row + (size_t)T * 16 + r, el < K);
    s_v[1][tid] = partial(pj + e, e < (size_t)T * 16);
    for (int k = 0; 64 * k < r; ++k) s_v[2 + k][tid] = partial(pj + (size_t)T * 16 + 64 * k + el, 64 * k + el < r);
    __syncthreads();
    if (tid < K) s_nj[tid] = whole(0);
    __syncthreads();
    const double nj = s_nj[j];
    const bool low = nj < 2.0;
    if (tid < 64)
        for (int k = 0; 64 * k + tid < r; ++k) dm[64 * k + tid] = whole(2 + k) / nj;
    const double s = whole(1);
    __syncthreads();
    if (tid < 64 && e < (size_t)T * 16) {
        const int t = (int)(e >> 4), q = (int)(e & 15);
        int ta = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
        while (ta * (ta + 1) / 2 > t) --ta;
        while ((ta + 1) * (ta + 2) / 2 <= t) ++ta;
        const int a = 4 * ta + (q >> 2), b = 4 * (t - ta * (ta + 1) / 2) + (q & 3);
        if (a < r && b <= a) {
            double v = s / nj - dm[a] * dm[b] + (a == b ? floor_frac * lamS[a] : 0.0);
            if (low) v = a == b ? pooled[a] : 0.0;
            cov[((size_t)j * r + a) * r + b] = v;
            cov[((size_t)j * r + b) * r + a] = v;
            if (a == b) lam[(size_t)j * r + a] = v;
        }
    }
    if (blockIdx.x != 0) return;
    __syncthreads();
    if (low) {
        double best = 1.0 / 0.0;
        int bi = N;
        for (int n = tid; n < N; n += 256)
            if (gmax[n] < best) { best = gmax[n]; bi = n; }
        s_v[0][tid] = best;
        s_i[tid] = bi;
        __syncthreads();
        if (tid == 0)
            for (int k = 1; k < 256; ++k)
                if (s_v[0][k] < s_v[0][0] || (s_v[0][k] == s_v[0][0] && s_i[k] < s_i[0])) { s_v[0][0] = s_v[0][k]; s_i[0] = s_i[k]; }
        __syncthreads();
        if (tid < r) m[(size_t)j * r + tid] = xsT[(size_t)tid * N + s_i[0]];
    } else if (tid < r) {
        m[(size_t)j * r + tid] = sums[(size_t)j * (r + 1) + tid] / sums[(size_t)j * (r + 1) + r] + dm[tid];
    }
    if (j == 0 && tid == 0) {
        double tot = 0.0;
        for (int k = 0; k < K; ++k) { w[k] = s_nj[k] < 2.0 ? 1.0 / N : s_nj[k] / N; tot += w[k]; }
        for (int k = 0; k < K; ++k) w[k] = w[k] / tot;
    }
}

// cov_j = diag(lam_j) for every component (the initial covariances).
__global__ void k_cov_diag(int K, int r, const double* __restrict__ lam, double* __restrict__ cov) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= K * r * r) return;
    const int j = t / (r * r), a = (t / r) % r, b = t % r;
    cov[t] = a == b ? lam[(size_t)j * r + a] : 0.0;
}

static int* factor_flag(Ctx& c) { return c.icount + 40; }

// L_j, log det L_j and the blocked rows of every C_j; with w also the E-step's constants.
static void launch_chol(Ctx& c, bool estep_constants) {
    double* cst = estep_constants ? c.gLb + (size_t)c.K * lb_size(c.r) : nullptr;
    if (c.r <= CHOL_SMEM_R) {
        check(cudaFuncSetAttribute(k_chol<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * CHOL_SMEM_R * (CHOL_SMEM_R + 1))), "attr");
        k_chol<true><<<c.K, 256, sizeof(double) * (size_t)c.r * (c.r + 1), c.stream>>>(c.r, c.gcov, c.gw, c.gL, c.gLb, c.glogdet, cst, factor_flag(c));
    } else {
        k_chol<false><<<c.K, 256, 0, c.stream>>>(c.r, c.gcov, c.gw, c.gL, c.gLb, c.glogdet, cst, factor_flag(c));
    }
    ++c.pc.launches;
    check(cudaGetLastError(), "factor launch");
}

// L_j, L_j^{-1} and log det L_j of every C_j.
static void launch_factor(Ctx& c) {
    launch_chol(c, false);
    const size_t sm = sizeof(double) * 32 * 4 * row_blocks(c.r);
    check(cudaFuncSetAttribute(k_tri_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * 32 * MAXR)), "attr");
    k_tri_inverse<<<dim3((c.r + 31) / 32, c.K), 32, sm, c.stream>>>(c.r, c.gLb, c.gLi); ++c.pc.launches;
    check(cudaGetLastError(), "inverse launch");
}

static void check_factor_flag(Ctx& c) {
    int bad = 0;
    check(cudaMemcpyAsync(&bad, factor_flag(c), sizeof(int), cudaMemcpyDeviceToHost, c.stream), "factor flag");
    sync_stream(c);
    if (bad) {
        c.fitted = false;   // the stored mixture is no longer usable
        throw InputError{"a mixture covariance is not positive definite"};
    }
}

// Factors every C_j on the device; with cov_host the covariances are uploaded first.  Waits, and
// fails (InputError) if a C_j is not positive definite.
void factor_mixture(Ctx& c, const double* cov_host) {
    const size_t n = (size_t)c.K * c.r * c.r;
    check(cudaMemsetAsync(factor_flag(c), 0, sizeof(int), c.stream), "memset");
    if (cov_host) check(cudaMemcpyAsync(c.gcov, cov_host, n * sizeof(double), cudaMemcpyHostToDevice, c.stream), "cov");
    launch_factor(c);
    check_factor_flag(c);
}

// EM with full covariances; the log-likelihood goes to ll (device).
static void em_full(Ctx& c, const double* lamS, double* ll) {
    const int N = c.N, K = c.K, r = c.r, kr2 = K * r * r;
    const int nch = cov_chunks(K, r), tg = (cov_tiles(r) + 255) / 256, P = 256 / K;
    const size_t esm = sizeof(double) * ESF_WARPS * 32 * 4 * row_blocks(r), csm = cov_smem(r);
    check(cudaFuncSetAttribute(k_estep_full, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * ESF_WARPS * 32 * MAXR)), "attr");
    check(cudaFuncSetAttribute(k_cov_acc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cov_smem(MAXR)), "attr");
    const double* cst = c.gLb + (size_t)K * lb_size(r);
    double* sums = c.covpart + cov_sums_at(K, r);
    auto estep = [&] {
        k_estep_full<<<dim3((N + 32 * ESF_WARPS - 1) / (32 * ESF_WARPS), K), 32 * ESF_WARPS, esm, c.stream>>>(N, r, c.xsT, c.gmu, c.gLb, cst, c.resp);
        k_resp<<<(N + P - 1) / P, 256, 0, c.stream>>>(N, K, c.resp, c.lse, c.gmax);
        c.pc.launches += 2;
    };
    check(cudaMemsetAsync(factor_flag(c), 0, sizeof(int), c.stream), "memset");
    k_cov_diag<<<(kr2 + 255) / 256, 256, 0, c.stream>>>(K, r, c.glam, c.gcov); ++c.pc.launches;
    for (int it = 0; it < c.cfg.em_iters; ++it) {
        launch_chol(c, true);
        estep();
        k_cov_mean<<<dim3(r + 1, K), 256, 0, c.stream>>>(N, r, c.xsT, c.resp, sums);
        k_cov_acc<<<dim3(tg, K, nch), 256, csm, c.stream>>>(N, r, c.xsT, c.resp, sums, c.covpart);
        k_cov_finish<<<dim3((cov_tiles(r) * 16 + 63) / 64, K), 256, 0, c.stream>>>(N, K, r, nch, c.covpart, sums, c.gmax, c.xsT, c.pooled, lamS,
                                                                                   c.cfg.var_floor, c.gw, c.gmu, c.glam, c.gcov);
        c.pc.launches += 3;
    }
    launch_chol(c, true);
    estep();
    launch_factor(c);                                    // the proposal's L_j^{-1}
    k_sum<<<1, 1024, 0, c.stream>>>(N, c.lse, ll); ++c.pc.launches;
    check(cudaGetLastError(), "full-covariance fit");
}

// EM with diagonal covariances; the log-likelihood goes to ll (device).
static void em_diag(Ctx& c, const double* lamS, double* ll) {
    const int N = c.N, K = c.K, r = c.r;
    EmArgs A{};
    A.N = N; A.K = K; A.r = r; A.iters = c.cfg.em_iters; A.lg_lanes = 2; A.floor_frac = c.cfg.var_floor;
    A.xsT = c.xsT; A.pooled = c.pooled; A.lamS = lamS; A.w = c.gw; A.m = c.gmu; A.lam = c.glam;
    A.part = c.empart; A.loglik = ll; A.bar = reinterpret_cast<unsigned*>(c.icount + 44); A.again = A.bar + 1; A.err = c.dev_err;
    const int G = std::max(1, std::min({EM_BLOCKS, c.sm_count, (N + EM_MINP - 1) / EM_MINP}));
    const int per = (N + G - 1) / G;
    while (A.lg_lanes < 5 && (per * K << (A.lg_lanes + 1)) <= EM_ETHREADS) ++A.lg_lanes;   // the chain of FP64 latencies is what bounds small fits
    constexpr size_t LIMIT = 200 * 1024;
    const bool xs = em_smem(K, r, per, true) <= LIMIT;
    const size_t sm = em_smem(K, r, per, xs);
    const void* fn = xs ? reinterpret_cast<const void*>(&k_em<true>) : reinterpret_cast<const void*>(&k_em<false>);
    check(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LIMIT), "attr");
    check(cudaMemsetAsync(A.bar, 0, 2 * sizeof(unsigned), c.stream), "memset");
    void* args[] = {&A};
    check(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(EM_THREADS), args, sm, c.stream), "EM launch"); ++c.pc.launches;
}

double gm_fit_device(Ctx& c) {
    const int N = c.N, K = c.K, r = c.r;
    double* lamS = c.pooled + r;          // second half of the pooled scratch
    k_gather_modes<<<(unsigned)(((size_t)N * r + 255) / 256), 256, 0, c.stream>>>(N, c.d, r, c.X, c.S, c.xsT); ++c.pc.launches;
    k_lamS<<<(r + 127) / 128, 128, 0, c.stream>>>(r, c.lam, c.S, lamS); ++c.pc.launches;
    k_pooled<<<r, 256, 0, c.stream>>>(N, r, c.xsT, lamS, c.cfg.var_floor, c.pooled); ++c.pc.launches;
    // initial picks (host Philox, the same definition as on the device)
    EmPicks picks{};
    for (int k = 0; k < K; ++k) {
        const U4 w = philox((uint32_t)k, 0u, (uint32_t)c.layer, P_EMINIT, c.key.k0, c.key.k1);
        int cidx = (int)(((unsigned long long)w.x * (unsigned long long)N) >> 32);
        bool clash = true;
        while (clash) {
            clash = false;
            for (int q = 0; q < k; ++q) if (picks.idx[q] == cidx) { clash = true; break; }
            if (clash) cidx = (cidx + 1) % N;
        }
        picks.idx[k] = cidx;
    }
    k_em_init<<<(K * r + 127) / 128, 128, 0, c.stream>>>(N, K, r, picks, c.xsT, c.pooled, c.gw, c.gmu, c.glam); ++c.pc.launches;
    double* ll_dev = c.dscal + 8;
    if (c.cfg.full_cov) em_full(c, lamS, ll_dev);
    else em_diag(c, lamS, ll_dev);
    double ll = 0.0;
    check(cudaMemcpyAsync(&ll, ll_dev, sizeof(double), cudaMemcpyDeviceToHost, c.stream), "ll");
    if (c.cfg.full_cov) check_factor_flag(c);            // one wait for the whole fit
    else sync_and_check_barrier(c);
    return ll;
}

}  // namespace smcgm
