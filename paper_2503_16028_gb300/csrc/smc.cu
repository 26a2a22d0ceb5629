// Reweighting, tempering, resampling and moments of Alg. 1 (Sec. 2.1) with
// the temperature rule of App. C.
//
// Tempering: with uniform weights before reweighting, the weights of step h
// are exp(-h Phi_n) and ESS(h) = (sum e^{-h Phi})^2 / sum e^{-2 h Phi} (the
// paper's (sum w^2)^-1 for normalised w).  h = 1 - t when ESS(1 - t) meets
// the target, else 64 bisection steps on [0, 1 - t] keeping the lower bracket.
//
// Resampling: systematic, on an integer CDF: normalised weights scaled by
// T = 2^48 and floored, the remainder added to the largest weight, inclusive
// prefix sums CDF_i; particle k takes min{i : N CDF_i > k T + u48} with u48 one
// Philox draw.  Integer arithmetic makes the indices independent of summation
// order.
#include <algorithm>
#include <type_traits>
#include "smcgm_internal.cuh"
#include "common.cuh"

namespace smcgm {

// Both kernels are cooperative launches over up to SMC_BLOCKS blocks with grid barriers: their
// cost is FP64 exponentials (some 30 FP64 operations each, and one SM's FP64 pipe does two lanes a
// cycle), so one block took 2.0 ms for the 66 x 4096 exponentials of a tempering step and 3.5 ms
// for 8192 particles, however fast its reductions, and resampling 8192 another 206 us.  Reweighting
// and resampling 8192 particles of 1024 modes, as called: 3.85 -> 0.41 ms.
constexpr int SMC_BLOCKS = 152;
constexpr int SMC_THREADS = 256;
constexpr int TEMPER_LEVELS = 4, TEMPER_C = 1 << TEMPER_LEVELS;   // decisions per round; candidates: one less, and 1 - t
constexpr int TEMPER_MINP = SMC_THREADS / TEMPER_C;   // least particles per block: one exponential per thread and round

static int smc_grid(int N, int per_block, int sms) {
    return std::max(1, std::min({SMC_BLOCKS, sms, (N + per_block - 1) / per_block}));
}
size_t smc_partial_doubles() { return 2 * SMC_BLOCKS * 2 * TEMPER_C + 2 * SMC_BLOCKS; }

// Value v (of 2 TEMPER_C) of all blocks' partials, added in a fixed order; every thread of every block
// gets the same sums in `tot`.
__device__ inline void sum_partials(const double* part, int G, double* scr, double* tot) {
    constexpr int V = 2 * TEMPER_C, CH = SMC_THREADS / V;
    const int v = threadIdx.x % V, ch = threadIdx.x / V;
    double a = 0.0;
#pragma unroll 4
    for (int g = ch; g < G; g += CH) a += __ldcg(&part[(size_t)g * V + v]);
    __syncthreads();
    scr[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x < V) {
        a = 0.0;
        for (int k = 0; k < CH; ++k) a += scr[k * V + threadIdx.x];
        tot[threadIdx.x] = a;
    }
    __syncthreads();
}

// Tempering.  The 64 bisection decisions are taken four at a time: a round evaluates the ESS at
// the fifteen points that the next four halvings can visit (the same midpoints, formed the same
// way) and then walks down, so 16 rounds of one barrier replace 64; the sixteenth lane of the first
// round evaluates h = 1 - t.
// out: [0] h, [1] ESS(h), [2] log Z increment, [3] new t
__global__ void __launch_bounds__(SMC_THREADS) k_temper(int N, const double* __restrict__ phi, double t, double target,
                                                        double* __restrict__ logw, double* __restrict__ out, double* part, unsigned* bar,
                                                        int* err) {
    __shared__ double red[32], scr[SMC_THREADS], tot[2 * TEMPER_C], cand[TEMPER_C + 1], ess[TEMPER_C];
    const int G = gridDim.x, tid = threadIdx.x;
    const int per = (N + G - 1) / G, n0 = min(N, (int)blockIdx.x * per), n1 = min(N, n0 + per);
    double* pmin = part + 2 * SMC_BLOCKS * 2 * TEMPER_C;
    unsigned arrivals = 0;
    double mn = 1.0 / 0.0;
    for (int i = n0 + tid; i < n1; i += SMC_THREADS) mn = fmin(mn, phi[i]);
    mn = -block_max(-mn, red);
    if (tid == 0) pmin[blockIdx.x] = mn;
    if (!grid_barrier(bar, arrivals += G, err)) return;
    mn = 1.0 / 0.0;
    for (int g = tid; g < G; g += SMC_THREADS) mn = fmin(mn, __ldcg(&pmin[g]));
    mn = -block_max(-mn, red);
    if (tid == 0) tot[0] = mn;
    __syncthreads();
    const double phimin = tot[0];
    const double rest = 1.0 - t;
    double lo = 0.0, hi = rest, ess_lo = 0.0, h;
    for (int round = 0;; ++round) {
        // cand[m], m = 1 .. 15: the midpoint of cand[m - s] and cand[m + s], s the lowest set bit of m (cand[0] = lo,
        // cand[16] = hi), level by level as the halvings would form them; slot 0 then holds 1 - t
        __syncthreads();
        if (tid == 0) {
            cand[0] = lo;
            cand[TEMPER_C] = hi;
            for (int st = TEMPER_C / 2; st >= 1; st >>= 1)
                for (int m = st; m < TEMPER_C; m += 2 * st) cand[m] = 0.5 * (cand[m - st] + cand[m + st]);
            cand[0] = rest;
        }
        __syncthreads();
        const int k = tid % TEMPER_C;
        const double hk = cand[k];
        double s1 = 0.0, s2 = 0.0;
        if (round == 0 || k > 0)
            for (int i = n0 + tid / TEMPER_C; i < n1; i += SMC_THREADS / TEMPER_C) {
                const double e = exp(-hk * (phi[i] - phimin));
                s1 += e;
                s2 += e * e;
            }
        s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
        s2 += __shfl_xor_sync(0xffffffffu, s2, 16);
        if ((tid & 31) < TEMPER_C) { scr[(tid >> 5) * 2 * TEMPER_C + k] = s1; scr[(tid >> 5) * 2 * TEMPER_C + TEMPER_C + k] = s2; }
        __syncthreads();
        double* pr = part + (size_t)(round & 1) * SMC_BLOCKS * 2 * TEMPER_C;   // the other half is still being read
        if (tid < 2 * TEMPER_C) {
            double a = 0.0;
            for (int w = 0; w < SMC_THREADS / 32; ++w) a += scr[w * 2 * TEMPER_C + tid];
            pr[(size_t)blockIdx.x * 2 * TEMPER_C + tid] = a;
        }
        if (!grid_barrier(bar, arrivals += G, err)) return;
        sum_partials(pr, G, scr, tot);
        if (tid < TEMPER_C) ess[tid] = tot[tid] * tot[tid] / tot[TEMPER_C + tid];
        __syncthreads();
        if (round == 0 && ess[0] >= target) { h = rest; ess_lo = ess[0]; break; }
        int at = TEMPER_C / 2;                   // walk down: the middle, a quarter point, ...
        for (int st = TEMPER_C / 4, l = 0; l < TEMPER_LEVELS; ++l, st >>= 1) {
            if (ess[at] >= target) { lo = cand[at]; ess_lo = ess[at]; at += st; }
            else { hi = cand[at]; at -= st; }
        }
        if (round == 64 / TEMPER_LEVELS - 1) { h = lo; break; }
    }
    // log weights -h Phi, their LSE (the largest is -h min Phi), normalised weights; log Z increment = LSE - log N
    const double mx = -h * phimin;
    double s = 0.0;
    for (int i = n0 + tid; i < n1; i += SMC_THREADS) s += exp(-h * phi[i] - mx);
    s = block_sum(s, red);
    if (tid == 0) pmin[SMC_BLOCKS + blockIdx.x] = s;
    if (!grid_barrier(bar, arrivals += G, err)) return;
    s = 0.0;
    for (int g = tid; g < G; g += SMC_THREADS) s += __ldcg(&pmin[SMC_BLOCKS + g]);
    s = block_sum(s, red);
    if (tid == 0) tot[0] = mx + log(s);
    __syncthreads();
    const double lse = tot[0];
    for (int i = n0 + tid; i < n1; i += SMC_THREADS) logw[i] = -h * phi[i] - lse;
    if (blockIdx.x == 0 && tid == 0) {
        out[0] = h;
        out[1] = h > 0.0 ? ess_lo : s;   // at h = 0 the sum of N ones, or NaN with a potential that is not finite
        out[2] = lse - log((double)N);
        out[3] = (h == rest) ? 1.0 : t + h;
    }
}

void launch_temper(Ctx& c, double* out) {
    unsigned* bar = reinterpret_cast<unsigned*>(c.icount + 44);
    int N = c.N;
    const double* phi = c.Phi;
    double t = c.t, target = c.cfg.ess_frac * c.N;
    void* args[] = {&N, &phi, &t, &target, &c.logw, &out, &c.smcpart, &bar, &c.dev_err};
    check(cudaMemsetAsync(bar, 0, sizeof(unsigned), c.stream), "memset");
    check(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_temper), dim3(smc_grid(N, TEMPER_MINP, c.sm_count)), dim3(SMC_THREADS),
                                      args, 0, c.stream), "temper"); ++c.pc.launches;
}

// Systematic resampling on the 2^48 fixed-point CDF; writes idx[N].  A particle per thread: q_i =
// floor(w_i T), the remainder to the largest weight (lowest index on ties), inclusive prefix sums
// (integers: any order), then a binary search per output.
__global__ void __launch_bounds__(SMC_THREADS) k_resample(int N, const double* __restrict__ logw, unsigned long long u48,
                                                          unsigned long long* cdf, int* __restrict__ idx, double* part, unsigned* bar,
                                                          int* err) {
    __shared__ double red[32], s_w[SMC_THREADS / 32], s_b;
    __shared__ unsigned long long s_q[SMC_THREADS / 32], s_off, s_tot;
    __shared__ int s_i[SMC_THREADS / 32], s_ib;
    const unsigned long long T = 1ull << 48;
    const int G = gridDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int i = blockIdx.x * SMC_THREADS + tid;
    const bool on = i < N;
    unsigned arrivals = 0;
    auto meet = [&] {                                        // a wait that ran out leaves the error flag and -1, never an old index
        const bool ok = grid_barrier(bar, arrivals += G, err);
        if (!ok && on) idx[i] = -1;
        return ok;
    };
    const double lw = on ? logw[i] : -1.0 / 0.0;
    auto gather = [&](const double* p, bool maximum) {      // the blocks' values p[g], combined alike in every block
        double a = maximum ? -1.0 / 0.0 : 0.0;
        for (int g = tid; g < G; g += SMC_THREADS) { const double v = __ldcg(&p[g]); a = maximum ? fmax(a, v) : a + v; }
        a = maximum ? block_max(a, red) : block_sum(a, red);
        if (tid == 0) s_b = a;
        __syncthreads();
        const double r = s_b;
        __syncthreads();
        return r;
    };
    double v = block_max(lw, red);
    if (tid == 0) part[blockIdx.x] = v;
    if (!meet()) return;
    const double mx = gather(part, true);
    v = block_sum(on ? exp(lw - mx) : 0.0, red);
    if (tid == 0) part[SMC_BLOCKS + blockIdx.x] = v;
    if (!meet()) return;
    const double lse = mx + log(gather(part + SMC_BLOCKS, false));
    const double w = on ? exp(lw - lse) : -1.0;
    unsigned long long q = on ? (unsigned long long)floor(w * (double)T) : 0;
    {
        unsigned long long qs = q;
        double wb = w;
        int ib = on ? i : N;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            qs += __shfl_xor_sync(0xffffffffu, qs, o);
            const double ow = __shfl_xor_sync(0xffffffffu, wb, o);
            const int oi = __shfl_xor_sync(0xffffffffu, ib, o);
            if (ow > wb || (ow == wb && oi < ib)) { wb = ow; ib = oi; }
        }
        if (lane == 0) { s_q[wid] = qs; s_w[wid] = wb; s_i[wid] = ib; }
        __syncthreads();
        if (tid == 0) {
            for (int k = 1; k < SMC_THREADS / 32; ++k) {
                qs += s_q[k];
                if (s_w[k] > wb || (s_w[k] == wb && s_i[k] < ib)) { wb = s_w[k]; ib = s_i[k]; }
            }
            double* pb = part + 2 * SMC_BLOCKS + 4 * blockIdx.x;
            pb[0] = __longlong_as_double((long long)qs);
            pb[1] = wb;
            pb[2] = (double)ib;
        }
    }
    if (!meet()) return;
    if (wid == 0) {                              // total, prefix of the earlier blocks, and the largest weight
        unsigned long long tot = 0, off = 0;
        double wb = -2.0;
        int ib = N;
        for (int g = lane; g < G; g += 32) {
            const double* pb = part + 2 * SMC_BLOCKS + 4 * g;
            const unsigned long long qg = (unsigned long long)__double_as_longlong(__ldcg(&pb[0]));
            const double ow = __ldcg(&pb[1]);
            const int oi = (int)__ldcg(&pb[2]);
            tot += qg;
            if (g < (int)blockIdx.x) off += qg;
            if (ow > wb || (ow == wb && oi < ib)) { wb = ow; ib = oi; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
            off += __shfl_xor_sync(0xffffffffu, off, o);
            const double ow = __shfl_xor_sync(0xffffffffu, wb, o);
            const int oi = __shfl_xor_sync(0xffffffffu, ib, o);
            if (ow > wb || (ow == wb && oi < ib)) { wb = ow; ib = oi; }
        }
        if (lane == 0) {
            s_tot = tot;
            s_ib = ib;
            s_off = off + (ib < (int)blockIdx.x * SMC_THREADS ? T - tot : 0);   // the remainder, modulo 2^64
        }
    }
    __syncthreads();
    if (i == s_ib) q += T - s_tot;
    unsigned long long run = q;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += u;
    }
    if (lane == 31) s_q[wid] = run;
    __syncthreads();
    run += s_off;
    for (int k = 0; k < wid; ++k) run += s_q[k];
    if (on) cdf[i] = run;
    if (!meet()) return;
    // particle k: smallest i with N * CDF_i > k T + u48
    if (on) {
        const unsigned long long target = (unsigned long long)i * T + u48;
        int lo = 0, hi = N - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((unsigned long long)N * __ldcg(&cdf[mid]) > target) hi = mid;
            else lo = mid + 1;
        }
        idx[i] = lo;
    }
}

// Issues k_resample; a block per 256 particles (N <= 32768: 128 blocks, all resident).
static void launch_resample_indices(int N, const double* logw, unsigned long long u48, unsigned long long* cdf, int* idx, double* part,
                                    unsigned* bar, int* err, cudaStream_t stream) {
    void* args[] = {&N, &logw, &u48, &cdf, &idx, &part, &bar, &err};
    check(cudaMemsetAsync(bar, 0, sizeof(unsigned), stream), "memset");
    check(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_resample), dim3((N + SMC_THREADS - 1) / SMC_THREADS), dim3(SMC_THREADS),
                                      args, 0, stream), "k_resample launch");
}

__global__ void k_gather(int d, const int* __restrict__ idx, const double* __restrict__ X, double* __restrict__ X2,
                         const double* __restrict__ Phi, double* __restrict__ Phi2) {
    const int k = blockIdx.x;
    const int src = idx[k];
    const double2* a = reinterpret_cast<const double2*>(X + (size_t)src * d);
    double2* b = reinterpret_cast<double2*>(X2 + (size_t)k * d);
    for (int i = threadIdx.x; i < d / 2; i += blockDim.x) b[i] = a[i];
    if (threadIdx.x == 0) Phi2[k] = Phi[src];
}

void launch_resample(Ctx& c) {
    const U4 w = philox(0u, 0u, (uint32_t)c.layer, P_RESAMPLE, c.key.k0, c.key.k1);
    const unsigned long long u48 = ((unsigned long long)w.x << 16) | (unsigned long long)(w.y >> 16);
    launch_resample_indices(c.N, c.logw, u48, reinterpret_cast<unsigned long long*>(c.gridtmp), c.idx, c.smcpart,
                            reinterpret_cast<unsigned*>(c.icount + 44), c.dev_err, c.stream); ++c.pc.launches;
    k_gather<<<c.N, 256, 0, c.stream>>>(c.d, c.idx, c.X, c.X2, c.Phi, c.Phi2); ++c.pc.launches;
    check(cudaGetLastError(), "resample");
    std::swap(c.X, c.X2);
    std::swap(c.Phi, c.Phi2);
}

// Posterior moments over the particles: mean and population variance per coordinate, two passes
// over X, each bound by HBM.  A block sums one chunk of the particles for 64 columns (32 lanes of
// 16 bytes, 8 rows at a time); k_col_finish adds the chunks in a fixed order.  One thread per
// column summing all particles took 1664 us at N = 4096, d = 16384 (now 290 us: 537 MB read twice at
// 3.7 TB/s); the grid's variance over 4096 fields of 256^2 1791 -> 1115 us, where two FP64
// operations per value (850 us on the FP64 pipes) bound it.
constexpr int MOM_ROWS = 8;

// Sums over a chunk of rows of (x - mean)^2 (SQ) or x, per column, to part[chunk][cols].  A: rows x cols;
// VEC columns per lane (2 when cols is even: every row and chunk starts on 16 bytes).
template <bool SQ, int VEC>
__global__ void __launch_bounds__(32 * MOM_ROWS) k_col_sums(int rows, size_t cols, const double* __restrict__ A, const double* __restrict__ mean,
                                                            double* __restrict__ part) {
    using V = typename std::conditional<VEC == 2, double2, double>::type;
    __shared__ double sh[MOM_ROWS][VEC][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t c = ((size_t)blockIdx.x * 32 + lane) * VEC;
    const int per = (rows + gridDim.y - 1) / gridDim.y, r0 = min(rows, (int)blockIdx.y * per), r1 = min(rows, r0 + per);
    double s[VEC] = {}, m[VEC] = {};
    if (c < cols) {
        if (SQ) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) m[q] = mean[c + q];
        }
#pragma unroll 4
        for (int r = r0 + wid; r < r1; r += MOM_ROWS) {
            const V v = *reinterpret_cast<const V*>(A + (size_t)r * cols + c);
            const double* x = reinterpret_cast<const double*>(&v);
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                const double e = x[q] - m[q];
                s[q] = SQ ? fma(e, e, s[q]) : s[q] + e;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < VEC; ++q) sh[wid][q][lane] = s[q];
    __syncthreads();
    if (wid == 0 && c < cols) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            double t = s[q];
            for (int k = 1; k < MOM_ROWS; ++k) t += sh[k][q][lane];
            part[(size_t)blockIdx.y * cols + c + q] = t;
        }
    }
}

// out = (add ? out : 0) + the sum over the chunks / n.
__global__ void k_col_finish(int chunks, size_t cols, const double* __restrict__ part, double n, int add, double* __restrict__ out) {
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols) return;
    double s = 0.0;
    for (int k = 0; k < chunks; ++k) s += part[(size_t)k * cols + c];
    out[c] = (add ? out[c] : 0.0) + s / n;
}

// Chunks of the rows: about eight blocks per SM in all, at least 32 rows each, and no more than `most`.
static int col_chunks(const Ctx& c, int rows, size_t cols, int most) {
    const size_t bx = (cols + 63) / 64, want = std::max<size_t>(1, 8 * (size_t)c.sm_count / bx);
    return (int)std::max<size_t>(1, std::min({want, (size_t)(rows + 31) / 32, (size_t)most, (size_t)65535}));
}

// part: scratch of chunks x cols doubles (most = the chunks it holds)
template <bool SQ>
static void col_reduce(Ctx& c, int rows, size_t cols, const double* A, const double* mean, double* part, int most, bool add, double* out) {
    const int ch = col_chunks(c, rows, cols, most);
    if (cols % 2 == 0)
        k_col_sums<SQ, 2><<<dim3((unsigned)((cols + 63) / 64), ch), 32 * MOM_ROWS, 0, c.stream>>>(rows, cols, A, mean, part);
    else
        k_col_sums<SQ, 1><<<dim3((unsigned)((cols + 31) / 32), ch), 32 * MOM_ROWS, 0, c.stream>>>(rows, cols, A, mean, part);
    k_col_finish<<<(unsigned)((cols + 255) / 256), 256, 0, c.stream>>>(ch, cols, part, (double)c.N, add ? 1 : 0, out);
    c.pc.launches += 2;
}

void launch_moments(Ctx& c, double* mean, double* var) {
    // the partials go to X2 (the gather's target, N x d, free here)
    col_reduce<false>(c, c.N, c.d, c.X, nullptr, c.X2, c.N, false, mean);
    col_reduce<true>(c, c.N, c.d, c.X, mean, c.X2, c.N, false, var);
    check(cudaGetLastError(), "moments");
}

// 1D field at the midpoints for `count` particles.
__global__ void k_synth1d(int n, int Km, int count, const double* __restrict__ X, const double* __restrict__ S, double* __restrict__ U) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)count * n) return;
    const int p = (int)(t / n), i = (int)(t % n);
    double u = 0.0;
    for (int k = 0; k < Km; ++k) u = fma(X[(size_t)p * Km + k], S[(size_t)i * Km + k], u);
    U[t] = u;
}

void launch_grid_moments(Ctx& c, const double* mean_kl, double* mean_grid, double* var_grid) {
    const size_t cells = c.dim == 2 ? (size_t)c.n * c.n : (size_t)c.n;
    auto synth = [&](const double* X, int count, double* U) {
        if (c.dim == 2) launch_synth2d(c, X, count, U);
        else { k_synth1d<<<(unsigned)(((size_t)count * c.n + 255) / 256), 256, 0, c.stream>>>(c.n, c.Km, count, X, c.basis, U); ++c.pc.launches; }
    };
    synth(mean_kl, 1, mean_grid);
    check(cudaMemsetAsync(var_grid, 0, cells * sizeof(double), c.stream), "memset");
    // partials: the solutions' batch array in 2D; in 1D what the fields leave of the batch scratch
    double* part = c.dim == 2 ? c.w64 : c.u64 + (size_t)c.B * c.n;
    for (int off = 0; off < c.N; off += c.B) {
        const int cnt = std::min(c.B, c.N - off);
        synth(c.X + (size_t)off * c.d, cnt, c.u64);
        col_reduce<true>(c, cnt, cells, c.u64, mean_grid, part, c.B, true, var_grid);
    }
    check(cudaGetLastError(), "grid moments");
}

// ---------------------------------------------------------------------------
// Resampling without any allocation.
//
// Some callers cannot hand the library a device buffer at all: a host
// application that owns every byte of device memory through its own pool and
// forbids other allocations, or a loop where a cudaMalloc (which may
// synchronise the device) is not acceptable.  For them the systematic-
// resampling indices can be computed with scratch that lives in this file: a
// fixed array of device memory that every GPU loading the library keeps until
// the process exits.  The caller passes the log weights and the output array;
// the library allocates nothing.
// ---------------------------------------------------------------------------
constexpr int STATIC_PART = 6 * SMC_BLOCKS;   // the blocks' partials
// the CDF, the partials, then the grid barrier's counter and its error flag (which nobody reads: the indices of -1 say it)
static __device__ __align__(256) unsigned long long g_static_scratch[SMC_STATIC_RESAMPLE_MAX + STATIC_PART + 1];

// Device address of g_static_scratch on the current device.  It is looked up on every
// call (the lookup allocates nothing): a cached address would go stale if the
// process reset the device, which unloads the library's module there.  The first
// lookup on a device also loads the module's copy of the array onto it.
static unsigned long long* static_scratch_ptr() {
    void* p = nullptr;
    check(cudaGetSymbolAddress(&p, g_static_scratch), "cudaGetSymbolAddress(g_static_scratch)");
    return reinterpret_cast<unsigned long long*>(p);
}

}  // namespace smcgm

extern "C" smc_status smc_resample_indices_static(const double* d_logw, int n_particles, unsigned long long seed, int layer,
                                                  int* d_indices, void* stream) {
    using namespace smcgm;
    if (!d_logw || !d_indices || layer < 0) {
        set_global_error("smc_resample_indices_static: null pointer or negative layer");
        return SMC_EINVAL;
    }
    if (n_particles < 1 || n_particles > SMC_STATIC_RESAMPLE_MAX) {
        set_global_error("smc_resample_indices_static: n_particles must be in [1, SMC_STATIC_RESAMPLE_MAX] (32768)");
        return SMC_EINVAL;
    }
    if (!device_visible(d_logw) || !device_visible(d_indices)) {
        set_global_error("smc_resample_indices_static: d_logw and d_indices must be device memory");
        return SMC_EINVAL;
    }
    try {
        unsigned long long* scratch = static_scratch_ptr();
        unsigned long long* cdf = scratch;
        unsigned* counters = reinterpret_cast<unsigned*>(scratch + SMC_STATIC_RESAMPLE_MAX + STATIC_PART);
        const Key key = key_of(seed);
        const U4 w = philox(0u, 0u, (uint32_t)layer, P_RESAMPLE, key.k0, key.k1);
        const unsigned long long u48 = ((unsigned long long)w.x << 16) | (unsigned long long)(w.y >> 16);
        // every entry of the CDF scratch below n_particles is written before it is read; only the barrier's counter is cleared
        launch_resample_indices(n_particles, d_logw, u48, cdf, d_indices, reinterpret_cast<double*>(scratch + SMC_STATIC_RESAMPLE_MAX),
                                counters, reinterpret_cast<int*>(counters + 1),
                                reinterpret_cast<cudaStream_t>(stream));
    } catch (const CudaError& ce) {
        set_global_error((std::string(ce.what) + ": " + cudaGetErrorString(ce.e)).c_str());
        return SMC_ECUDA;
    }
    return SMC_OK;
}
