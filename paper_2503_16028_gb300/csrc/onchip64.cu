// The FP64 solve of a batch of particles on chip: as onchip.cu (one launch, a block of 64^2 or a
// cluster of 4 blocks of 128^2 per particle), in FP64 throughout.
//
// What bounds it: the FP64 pipe, two lanes per SM and cycle (a warp's instruction takes its scheduler's share 64
// cycles).  So the layout spends registers, instructions and shared memory freely and FP64 operations
// sparingly, about 22 per cell and CG iteration on the finest level and 7.5 below it (the multi-pass
// solver: 29 and, with both colours of a checkerboard in each warp, 19, times 1.56 for the halo cells that
// its tiles smooth again):
//  - neighbour sums are one chain of multiply-adds; latency hides behind the pipe's other warps;
//  - 1/D comes from the set-up's arrays, restriction takes the red residuals alone (the black ones vanish);
//  - on levels with a cell per thread a warp holds one colour, so a half sweep issues on half the warps;
//  - A z is r on the cells smoothed last and is formed on the others only; A p follows by recurrence and
//    p.Ap from z.Az, which also makes one exchange of two sums out of two exchanges;
//  - sums over the block are trees over few warps, scalars are formed by one thread.
// Measured, forward maps with FP64 solves: 2048 of 64^2 14.5 ms in passes, 9.4 on chip (14.4 before the last
// three of the above); 1024 of 128^2 29.2 and 22.5; 2 of 64^2 1.8 and 0.74, 2 of 128^2 2.1 and 0.89.
// A strip of 256^2 would need 16 blocks and 4 cells a thread at one block per SM: 7 such clusters leave 40 SMs idle.
//
// Layout: 1024 threads per block, a 2 x 2 patch of the finest level each (faces, residual and
// correction in registers, 64 a thread; 1/D and the next level's faces in shared memory), one cell of
// the next level; CG's p, q and x go through L2.  Below that a block of 64^2 has the 16^2 level on its
// first 256 threads; a cluster gathers the 32^2 level in every block (one cell per thread) and goes
// on as one block does.  8^2 is smoothed by 64 threads and 4^2 solved with its dense inverse.
#include "smcgm_internal.cuh"
#include "common.cuh"
#include "onchip.cuh"

namespace smcgm {

constexpr int O6_T = 1024;

struct O6Level { const double *Kw, *Ks, *E, *Nn, *inv; };
struct O6Args {
    int n, max_outer, maxit, nu_f, nu_c;
    double cc, tol2, floor2, tolout2, b2const;
    const double* b2pp;
    O6Level lv[6];               // levels n, n/2, .. 4 (as many as there are)
    const double* b;
    size_t bstride;
    double2 *x, *p, *q;          // per particle n^2 doubles, [block][patch row][thread]
    double* W;
    GraphCounters* cnt;
    int* err;
    const double* inv4;          // per particle: the dense inverse of the 4^2 level, 16 x 16
    // the V-cycle alone: right-hand sides, corrections, the active particles
    const double* vr;
    double* ve;
    const int *list, *nact;
};

// Shared memory, in doubles.
template <int C_>
struct O6Mem {
    static constexpr int C = C_, CC = C * C, W = 32 * C, H = 32 / C, PT = W + 2, PL = (H + 2) * PT;
    static constexpr int FP = 0;                        // finest level: 4 planes, cell (i, j) of each patch
    static constexpr int HPL = FP + 4 * PL;             // the next level's plane
    static constexpr int P32 = HPL + PL;                // C = 2: the gathered 32^2 level's plane (34 x 34)
    static constexpr int P16 = P32 + (C > 1 ? 1156 : 0);   // 18 x 18
    static constexpr int P8 = P16 + 324;                // 10 x 10
    static constexpr int ZEROED = P8 + 100;             // all planes: guards stay zero at the walls
    static constexpr int INVF = ZEROED;                 // 1/D: [cell][thread]
    static constexpr int HF = INVF + 4 * O6_T;          // the next level's faces w, e, s, n and 1/D: [5][thread]
    static constexpr int F32 = HF + 5 * O6_T;           // C = 2: as HF for the 32^2 level
    static constexpr int F16 = F32 + (C > 1 ? 5 * O6_T : 0);   // [5][256]
    static constexpr int F8 = F16 + 5 * 256;            // [5][64]
    static constexpr int INV4 = F8 + 5 * 64;            // dense inverse of the 4^2 level, 16 x 16
    static constexpr int RES = INV4 + 256;              // residuals to restrict, one per thread
    static constexpr int RB = RES + O6_T;               // C = 2: the gathered right-hand side
    static constexpr int R4 = RB + (C > 1 ? O6_T : 0);
    static constexpr int E4 = R4 + 16;
    static constexpr int BUF = E4 + 16;                 // block sums of two values: 2 x 1024, then 2 x 4
    static constexpr int RED = BUF + 2 * O6_T + 8;      // the cluster's: slots of 2 x CC
    static constexpr int SC = RED + 4 * CC;             // scalars for all threads
    static constexpr int ENDD = SC + 4;
    static constexpr int BARS = 8 * ENDD;               // bytes
    static constexpr size_t BYTES = BARS + 64;
    static_assert(BYTES <= 227 * 1024, "one block per SM");
};

// ---- finest level: cells 0 (0,0), 1 (1,0), 2 (0,1), 3 (1,1); red: 0 and 3 ----
template <class M>
__device__ __forceinline__ void pub_f6(double* sm, const OcPos<M>& t, int col, const double (&e)[4]) {
    if (M::C > 1 && t.nbase) {
        const int plane = t.lower ? (col ? 1 : 0) : (col ? 2 : 3);
        oc_store(t.nbase + 8 * (M::FP + plane * M::PL + (t.lower ? (M::H + 1) * M::PT : 0) + t.tx + 1),
                 t.lower ? (col ? e[1] : e[0]) : (col ? e[2] : e[3]), t.nbase + nb_bar(t, !t.lower));
    }
    const int at = (t.ty + 1) * M::PT + t.tx + 1;
    sm[M::FP + (col ? 1 : 0) * M::PL + at] = e[col ? 1 : 0];
    sm[M::FP + (col ? 2 : 3) * M::PL + at] = e[col ? 2 : 3];
}
// The outer neighbours of the two cells of a colour: a cell's horizontal and vertical one (the other two are its patch's).
template <class M>
__device__ __forceinline__ void out_f6(const double* sm, const OcPos<M>& t, int col, double& ah, double& av, double& bh, double& bv) {
    const double *p0 = sm + M::FP + (t.ty + 1) * M::PT + t.tx + 1, *p1 = p0 + M::PL, *p2 = p1 + M::PL, *p3 = p2 + M::PL;
    if (col == 0) { ah = p1[-1]; av = p2[-M::PT]; bh = p2[1]; bv = p1[M::PT]; }     // cell 0: west, south; cell 3: east, north
    else { ah = p0[1]; av = p3[-M::PT]; bh = p3[-1]; bv = p0[M::PT]; }              // cell 1: east, south; cell 2: west, north
}
// Adds the sum of k e over the neighbours of the two cells of a colour; w: west faces [j][0..2], s: south faces [0..2][i].
// One chain of multiply-adds: the pipe takes 64 cycles per instruction of a scheduler, more than its latency.
template <class M>
__device__ __forceinline__ void nb_f6(const double* sm, const OcPos<M>& t, int col, const double (&w)[6], const double (&s)[6], const double (&e)[4],
                                      double& a, double& b) {
    double ah, av, bh, bv;
    out_f6(sm, t, col, ah, av, bh, bv);
    if (col == 0) {
        a = fma(w[0], ah, fma(w[1], e[1], fma(s[0], av, fma(s[2], e[2], a))));
        b = fma(w[5], bh, fma(w[4], e[2], fma(s[5], bv, fma(s[3], e[1], b))));
    } else {
        a = fma(w[2], ah, fma(w[1], e[0], fma(s[1], av, fma(s[3], e[3], a))));
        b = fma(w[3], bh, fma(w[4], e[3], fma(s[4], bv, fma(s[2], e[0], b))));
    }
}
template <class M>
__device__ __forceinline__ void sweep_f6(const double* sm, const OcPos<M>& t, int col, const double (&w)[6], const double (&s)[6],
                                         const double (&r)[4], double (&e)[4]) {
    const int i = col ? 1 : 0, j = col ? 2 : 3;
    double a = r[i], b = r[j];
    nb_f6(sm, t, col, w, s, e, a, b);
    e[i] = a * sm[M::INVF + i * O6_T + t.tid];
    e[j] = b * sm[M::INVF + j * O6_T + t.tid];
}

// ---- levels with one cell per thread: SIDE > 0: a local SIDE^2 level on its first SIDE^2 threads; 0: the block's ----
// Even warps hold the red cells, odd warps the black ones, so a half sweep issues on half the warps (with both
// colours in a warp it costs the pipe all of them).
template <class M, int SIDE>
struct Lev6 {
    static constexpr int WID = SIDE ? SIDE : M::W;
    static constexpr int PT = WID + 2;
    static constexpr int NT = SIDE ? SIDE * SIDE : O6_T;
    static __device__ __forceinline__ int idx(int tid) { return (tid >> 6) * 32 + (tid & 31); }
    static __device__ __forceinline__ int y(int tid) { return idx(tid) / (WID / 2); }
    static __device__ __forceinline__ int x(int tid) { return 2 * (idx(tid) % (WID / 2)) + ((y(tid) + (tid >> 5)) & 1); }
    static __device__ __forceinline__ int at(int tid) { return (y(tid) + 1) * PT + x(tid) + 1; }
    static __device__ __forceinline__ bool red(int tid) { return ((tid >> 5) & 1) == 0; }
};
// Barrier of a level: the exchange with the neighbouring blocks, the block, or the first 256 threads (16^2 and below).
template <class M, int SIDE>
__device__ __forceinline__ void sync6(double* sm, OcPos<M>& t) {
    if (SIDE == 0) nb_sync(sm, t, 4 * M::W);
    else if (SIDE == 32) __syncthreads();
    else asm volatile("bar.sync 1, 256;" ::: "memory");
}
template <class M, int SIDE>
__device__ __forceinline__ void pub6(double* sm, double* pl, const OcPos<M>& t, double e) {
    if (SIDE == 0 && M::C > 1 && t.nbase)
        oc_store(t.nbase + 8 * (M::HPL + (t.lower ? (M::H + 1) * M::PT : 0) + t.tx + 1), e, t.nbase + nb_bar(t, !t.lower));
    pl[Lev6<M, SIDE>::at(t.tid)] = e;
}
// c plus the sum of k e over the neighbours; f: faces w, e, s, n at stride NT.
template <class M, int SIDE>
__device__ __forceinline__ double nb6(const double* pl, const OcPos<M>& t, const double* f, double c) {
    using L = Lev6<M, SIDE>;
    const double* p = pl + L::at(t.tid);
    return fma(f[0], p[-1], fma(f[L::NT], p[1], fma(f[2 * L::NT], p[-L::PT], fma(f[3 * L::NT], p[L::PT], c))));
}
// Pre-smoothing from e = 0; writes the residual of red cells to RES[cell] (the black ones' vanish).
template <class M, int SIDE>
__device__ __forceinline__ void pre6(double* sm, double* pl, const double* f, OcPos<M>& t, int nu, double r, double& e) {
    using L = Lev6<M, SIDE>;
    const bool on = t.tid < L::NT, red = L::red(t.tid);
    double nb = 0.0;                                     // red cells: D e = r + nb
    e = 0.0;
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        if (on && red) {
            if (sw > 0) nb = nb6<M, SIDE>(pl, t, f, 0.0);
            e = (r + nb) * f[4 * L::NT];
            pub6<M, SIDE>(sm, pl, t, e);
        }
        sync6<M, SIDE>(sm, t);
        if (on && !red) {
            e = nb6<M, SIDE>(pl, t, f, r) * f[4 * L::NT];
            pub6<M, SIDE>(sm, pl, t, e);
        }
        sync6<M, SIDE>(sm, t);
    }
    if (on && red) sm[M::RES + L::y(t.tid) * L::WID + L::x(t.tid)] = nb6<M, SIDE>(pl, t, f, -nb);
}
// Post-smoothing; e already holds the corrected value.  The last red values are not published.
template <class M, int SIDE>
__device__ __forceinline__ void post6(double* sm, double* pl, const double* f, OcPos<M>& t, int nu, double r, double& e) {
    using L = Lev6<M, SIDE>;
    const bool on = t.tid < L::NT, red = L::red(t.tid);
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        if (on && red) pub6<M, SIDE>(sm, pl, t, e);
        sync6<M, SIDE>(sm, t);
        if (on && !red) {
            e = nb6<M, SIDE>(pl, t, f, r) * f[4 * L::NT];
            pub6<M, SIDE>(sm, pl, t, e);
        }
        sync6<M, SIDE>(sm, t);
        if (on && red) e = nb6<M, SIDE>(pl, t, f, r) * f[4 * L::NT];
    }
}

// Sums of NV values over the particle's cells, then fin(sums) by thread 0 of every block (the same bits everywhere),
// whose scalars in SC all threads may read afterwards.  `edges`: bytes of an edge exchange that goes with it, or 0.
// True if a wait ran out in any thread of the block.
template <int NV, class M, class Fin>
__device__ __forceinline__ bool sum6(double* sm, OcPos<M>& t, int slot, const double (&v)[NV], int edges, Fin fin) {
    double* buf = sm + M::BUF;
#pragma unroll
    for (int k = 0; k < NV; ++k) buf[k * O6_T + t.tid] = v[k];
    if (M::C > 1 && t.tid == 0) oc_expect(t, all_bar<M>(sm, slot), 8 * NV * M::CC);
    __syncthreads();
    if (t.tid < 128 * NV) {                    // per value one warp per scheduler: 8 values each, then the warp
        const double* q = buf + (t.tid >> 7) * O6_T + (t.tid & 127);
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int k = 0; k < 8; k += 2) { a += q[128 * k]; b += q[128 * (k + 1)]; }
        a += b;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((t.tid & 31) == 0) buf[2 * O6_T + (t.tid >> 5)] = a;
        asm volatile("bar.sync 2, %0;" ::"n"(128 * NV) : "memory");
        if (t.tid < M::CC) {
            double s[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double* w = buf + 2 * O6_T + 4 * k;
                s[k] = (w[0] + w[1]) + (w[2] + w[3]);
            }
            if (M::C == 1) {
                fin(s);
            } else {
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    oc_store(oc_map(sm + M::RED + (2 * slot + k) * M::CC + t.rank, t.tid), s[k], oc_map(all_bar<M>(sm, slot), t.tid));
            }
        }
    }
    if (M::C > 1) {
        if (edges) nb_wait(sm, t, edges);
        if (t.tid < 32) {
            oc_wait(t, all_bar<M>(sm, slot), (t.par >> slot) & 1);
            if (t.tid == 0) {
                double s[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const double* q = sm + M::RED + (2 * slot + k) * M::CC;
                    s[k] = q[0];
                    for (int d = 1; d < M::CC; ++d) s[k] += q[d];
                }
                fin(s);
            }
        }
        t.par ^= 1u << slot;
        return __syncthreads_or(t.dead);
    }
    __syncthreads();
    return false;
}

// V: one V-cycle only, for the levels from 128^2 down of a larger grid's multi-pass solver.
template <int C, bool V>
__global__ void __launch_bounds__(O6_T, 1) k_onchip64(const O6Args A) {
    using M = O6Mem<C>;
    extern __shared__ __align__(16) double sm6[];
    double* sm = sm6;
    constexpr int n = 64 * C;
    if (V && A.nact && (int)(blockIdx.x / M::CC) >= *A.nact) return;
    const int p = V ? A.list[blockIdx.x / M::CC] : (int)(blockIdx.x / M::CC);
    OcPos<M> t;
    oc_place(t, sm, Lev6<M, 0>::x(threadIdx.x), Lev6<M, 0>::y(threadIdx.x));
    const int gx = 2 * t.tx, gy = 2 * ((int)t.rank * M::H + t.ty);
    const size_t base = (size_t)p * n * n;
    const double b2 = V ? 1.0 : A.b2pp ? A.b2pp[p] : A.b2const;
    double* W = (V ? A.ve : A.W) + base + (size_t)gy * n + gx;
    if (!(b2 > 0.0)) {                                      // not solved: w = 0 (the whole cluster alike)
        *reinterpret_cast<double2*>(W) = *reinterpret_cast<double2*>(W + n) = make_double2(0.0, 0.0);
        return;
    }
    for (int i = t.tid; i < M::ZEROED; i += O6_T) sm[i] = 0.0;
    if (C > 1 && t.tid == 0) oc_init_bars<M>(sm);
    double kw[6], ks[6], r[4], e[4];
    {
        const O6Level& L = A.lv[0];
        const double *Kw = L.Kw + base, *Ks = L.Ks + base, *inv = L.inv + base;
        const size_t c = (size_t)gy * n + gx;
        auto two = [](const double* q) { return *reinterpret_cast<const double2*>(q); };
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const double2 k = two(Kw + c + j * n), v = two(inv + c + j * n);
            kw[3 * j] = k.x;
            kw[3 * j + 1] = k.y;
            kw[3 * j + 2] = gx + 2 < n ? Kw[c + j * n + 2] : L.E[(size_t)p * n + gy + j];
            sm[M::INVF + 2 * j * O6_T + t.tid] = v.x;
            sm[M::INVF + (2 * j + 1) * O6_T + t.tid] = v.y;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double2 k = two(gy + j < n ? Ks + c + (size_t)j * n : L.Nn + (size_t)p * n + gx);
            ks[2 * j] = k.x;
            ks[2 * j + 1] = k.y;
        }
        const double* B = V ? A.vr + base + c : A.b + (size_t)p * A.bstride + c;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const double2 v = two(B + j * n);
            r[2 * j] = v.x;
            r[2 * j + 1] = v.y;
        }
    }
    // the coarser levels' faces: cell (x, y) of a level of side m
    auto load_level = [&](const O6Level& L, int m, int x, int y, double* f, int nt) {
        const size_t c = (size_t)p * m * m + (size_t)y * m + x;
        f[0] = L.Kw[c];
        f[nt] = x + 1 < m ? L.Kw[c + 1] : L.E[(size_t)p * m + y];
        f[2 * nt] = L.Ks[c];
        f[3 * nt] = y + 1 < m ? L.Ks[c + m] : L.Nn[(size_t)p * m + x];
        f[4 * nt] = L.inv[c];
    };
    load_level(A.lv[1], n / 2, t.tx, (int)t.rank * M::H + t.ty, sm + M::HF + t.tid, O6_T);
    if (C == 2) load_level(A.lv[2], 32, Lev6<M, 32>::x(t.tid), Lev6<M, 32>::y(t.tid), sm + M::F32 + t.tid, O6_T);
    constexpr int l16 = C == 1 ? 2 : 3;
    if (t.tid < 256) load_level(A.lv[l16], 16, Lev6<M, 16>::x(t.tid), Lev6<M, 16>::y(t.tid), sm + M::F16 + t.tid, 256);
    if (t.tid < 64) load_level(A.lv[l16 + 1], 8, Lev6<M, 8>::x(t.tid), Lev6<M, 8>::y(t.tid), sm + M::F8 + t.tid, 64);
    if (t.tid < 256) sm[M::INV4 + t.tid] = A.inv4[(size_t)p * 256 + t.tid];
    oc_sync<C>();                                            // every block of the cluster runs, its mbarriers are ready
    const size_t pb = (size_t)blockIdx.x * 2 * O6_T + t.tid;   // this thread's patch rows in x, p and q
    double *HPL = sm + M::HPL, *P32 = sm + M::P32, *P16 = sm + M::P16, *P8 = sm + M::P8;
    const double *HF = sm + M::HF + t.tid, *F32 = sm + M::F32 + t.tid, *F16 = sm + M::F16 + (t.tid & 255), *F8 = sm + M::F8 + (t.tid & 63);
    double* SC = sm + M::SC;
    int iters = 0, phases = 0, inner = 0;
    bool converged = false;
#pragma unroll 1
    for (int o = 0; o < A.max_outer; ++o) {
        // ---- CG on A x = r from x = 0, with A p by recurrence from A z (which is r on the cells smoothed last, so half of it
        // costs nothing) and p.Ap from z.Az, so that one exchange serves both sums of an iteration.
        // SC[0]: whether to go on; SC[1], SC[2]: beta, alpha; thread 0 keeps the threshold, r.z and alpha ----
        double thr = 0.0, rz = 0.0, al = 0.0;
        bool first = true, dead = false;
        for (;;) {
            e[0] = r[0] * sm[M::INVF + t.tid];
            e[3] = r[3] * sm[M::INVF + 3 * O6_T + t.tid];
            pub_f6(sm, t, 0, e);
            if (V) {
                nb_sync(sm, t, 8 * M::W);
            } else {
                const double s[1] = {fma(r[0], r[0], r[1] * r[1]) + fma(r[2], r[2], r[3] * r[3])};
                if (!first) ++iters;
                dead = sum6(sm, t, OC_RR, s, 8 * M::W, [&](const double (&v)[1]) {
                    const double rr = v[0];
                    if (first) thr = fmax(A.tol2 * rr, A.floor2 * b2);
                    SC[0] = first ? (rr > 0.0 ? 1.0 : 0.0) : (rr <= thr || iters >= A.maxit || !(rr == rr)) ? 0.0 : 1.0;
                });
                if (dead || SC[0] == 0.0) break;
                if (first) ++inner;
            }
            // V-cycle: z = M r in e
            double nb0 = 0.0, nb3 = 0.0;                      // red cells: D e = r + nb
#pragma unroll 1
            for (int sw = 0; sw < A.nu_f; ++sw) {
                if (sw > 0) {
                    nb0 = nb3 = 0.0;
                    nb_f6(sm, t, 0, kw, ks, e, nb0, nb3);
                    e[0] = (r[0] + nb0) * sm[M::INVF + t.tid];
                    e[3] = (r[3] + nb3) * sm[M::INVF + 3 * O6_T + t.tid];
                    pub_f6(sm, t, 0, e);
                    nb_sync(sm, t, 8 * M::W);
                }
                sweep_f6(sm, t, 1, kw, ks, r, e);
                pub_f6(sm, t, 1, e);
                nb_sync(sm, t, 8 * M::W);
            }
            nb0 = -nb0;
            nb3 = -nb3;
            nb_f6(sm, t, 0, kw, ks, e, nb0, nb3);
            double rh = nb0 + nb3, eh;
            pre6<M, 0>(sm, HPL, HF, t, A.nu_c, rh, eh);
            __syncthreads();
            double e32 = 0.0, r32 = 0.0;
            // the red residuals of a coarse cell's four children lie at (2x, 2y) and (2x + 1, 2y + 1)
            if (C == 2) {
                if (t.tid < 256) {
                    const int x = t.tid & 31, y = t.tid >> 5;   // this block's 8 rows of the 32^2 level
                    const double* q = sm + M::RES + (2 * y) * M::W + 2 * x;
                    const double v = q[0] + q[M::W + 1];
                    for (int d = 0; d < M::CC; ++d) {
                        double* dst = sm + M::RB + (int)t.rank * 256 + t.tid;
                        oc_store(oc_map(dst, d), v, oc_map(all_bar<M>(sm, OC_GATHER), d));
                    }
                }
                all_sync(sm, t, OC_GATHER, 8 * 1024);
                r32 = sm[M::RB + Lev6<M, 32>::y(t.tid) * 32 + Lev6<M, 32>::x(t.tid)];
                pre6<M, 32>(sm, P32, F32, t, A.nu_c, r32, e32);
                __syncthreads();
            }
            if (t.tid < 256) {
                constexpr int CW = C == 1 ? M::W : 32;        // width of the level above in RES
                double e16, e8 = 0.0, r8 = 0.0;
                const int x = Lev6<M, 16>::x(t.tid), y = Lev6<M, 16>::y(t.tid), x8 = Lev6<M, 8>::x(t.tid & 63), y8 = Lev6<M, 8>::y(t.tid & 63);
                const double* q = sm + M::RES + (2 * y) * CW + 2 * x;
                const double r16 = q[0] + q[CW + 1];
                asm volatile("bar.sync 1, 256;" ::: "memory");
                pre6<M, 16>(sm, P16, F16, t, A.nu_c, r16, e16);
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (t.tid < 64) {
                    const double* q8 = sm + M::RES + 2 * y8 * 16 + 2 * x8;
                    r8 = q8[0] + q8[17];
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                pre6<M, 8>(sm, P8, F8, t, A.nu_c, r8, e8);
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (t.tid < 16) {
                    const double* q4 = sm + M::RES + 2 * (t.tid >> 2) * 8 + 2 * (t.tid & 3);
                    sm[M::R4 + t.tid] = q4[0] + q4[9];
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                double v = sm[M::INV4 + t.tid] * sm[M::R4 + (t.tid & 15)];
#pragma unroll
                for (int k = 8; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
                if ((t.tid & 15) == 0) sm[M::E4 + (t.tid >> 4)] = v;
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (t.tid < 64) e8 = fma(A.cc, sm[M::E4 + (y8 >> 1) * 4 + (x8 >> 1)], e8);
                post6<M, 8>(sm, P8, F8, t, A.nu_c, r8, e8);
                if (t.tid < 64 && Lev6<M, 8>::red(t.tid)) P8[Lev6<M, 8>::at(t.tid)] = e8;
                asm volatile("bar.sync 1, 256;" ::: "memory");
                e16 = fma(A.cc, P8[((y >> 1) + 1) * 10 + (x >> 1) + 1], e16);
                post6<M, 16>(sm, P16, F16, t, A.nu_c, r16, e16);
                if (Lev6<M, 16>::red(t.tid)) P16[Lev6<M, 16>::at(t.tid)] = e16;
            }
            __syncthreads();
            if (C == 2) {
                e32 = fma(A.cc, P16[((Lev6<M, 32>::y(t.tid) >> 1) + 1) * 18 + (Lev6<M, 32>::x(t.tid) >> 1) + 1], e32);
                post6<M, 32>(sm, P32, F32, t, A.nu_c, r32, e32);
                if (Lev6<M, 32>::red(t.tid)) P32[Lev6<M, 32>::at(t.tid)] = e32;
                __syncthreads();
                const int py = ((int)t.rank * M::H + t.ty) >> 1;
                eh = fma(A.cc, P32[(py + 1) * 34 + (t.tx >> 1) + 1], eh);
            } else {
                eh = fma(A.cc, P16[((t.ty >> 1) + 1) * 18 + (t.tx >> 1) + 1], eh);
            }
            post6<M, 0>(sm, HPL, HF, t, A.nu_c, rh, eh);
#pragma unroll
            for (int k = 0; k < 4; ++k) e[k] = fma(A.cc, eh, e[k]);
#pragma unroll 1
            for (int sw = 0; sw < A.nu_f; ++sw) {
                pub_f6(sm, t, 0, e);
                nb_sync(sm, t, 8 * M::W);
                sweep_f6(sm, t, 1, kw, ks, r, e);
                pub_f6(sm, t, 1, e);
                nb_sync(sm, t, 8 * M::W);
                sweep_f6(sm, t, 0, kw, ks, r, e);
            }
            if (V) break;
            // A z: r on the red cells, in flux form on the black ones
            pub_f6(sm, t, 0, e);
            nb_sync(sm, t, 8 * M::W);
            double z1, z2;
            {
                double ah, av, bh, bv;
                out_f6(sm, t, 1, ah, av, bh, bv);
                z1 = fma(kw[2], e[1] - ah, fma(kw[1], e[1] - e[0], fma(ks[1], e[1] - av, ks[3] * (e[1] - e[3]))));
                z2 = fma(kw[3], e[2] - bh, fma(kw[4], e[2] - e[3], fma(ks[4], e[2] - bv, ks[2] * (e[2] - e[0]))));
            }
            const double red = fma(r[0], e[0], r[3] * e[3]);
            const double zz[2] = {fma(r[1], e[1], fma(r[2], e[2], red)), fma(z1, e[1], fma(z2, e[2], red))};
            dead = sum6(sm, t, OC_RZ, zz, 0, [&](const double (&v)[2]) {
                const double beta = first ? 0.0 : v[0] / rz, pq = first ? v[1] : v[1] - beta * (v[0] / al);
                rz = v[0];
                al = pq > 0.0 ? rz / pq : 0.0;
                SC[1] = beta;
                SC[2] = al;
            });
            if (dead) break;
            const double alpha = SC[2];
            double2 a = make_double2(e[0], e[1]), b = make_double2(e[2], e[3]);
            double2 x0 = make_double2(0.0, 0.0), x1 = x0, q0 = make_double2(r[0], z1), q1 = make_double2(z2, r[3]);
            if (!first) {
                const double beta = SC[1];
                const double2 p0 = A.p[pb], p1 = A.p[pb + O6_T], o0 = A.q[pb], o1 = A.q[pb + O6_T];
                x0 = A.x[pb];
                x1 = A.x[pb + O6_T];
                a.x = fma(beta, p0.x, a.x); a.y = fma(beta, p0.y, a.y);
                b.x = fma(beta, p1.x, b.x); b.y = fma(beta, p1.y, b.y);
                q0.x = fma(beta, o0.x, q0.x); q0.y = fma(beta, o0.y, q0.y);
                q1.x = fma(beta, o1.x, q1.x); q1.y = fma(beta, o1.y, q1.y);
            }
            A.p[pb] = a;
            A.p[pb + O6_T] = b;
            A.q[pb] = q0;
            A.q[pb + O6_T] = q1;
            x0.x = fma(alpha, a.x, x0.x); x0.y = fma(alpha, a.y, x0.y);
            x1.x = fma(alpha, b.x, x1.x); x1.y = fma(alpha, b.y, x1.y);
            A.x[pb] = x0;
            A.x[pb + O6_T] = x1;
            r[0] = fma(-alpha, q0.x, r[0]); r[1] = fma(-alpha, q0.y, r[1]);
            r[2] = fma(-alpha, q1.x, r[2]); r[3] = fma(-alpha, q1.y, r[3]);
            first = false;
        }
        if (V) {
            *reinterpret_cast<double2*>(W) = make_double2(e[0], e[1]);
            *reinterpret_cast<double2*>(W + n) = make_double2(e[2], e[3]);
            break;
        }
        // ---- w += x; residual b - A w in flux form, the neighbours' w through the finest planes ----
        ++phases;
        {
            double2 w0 = make_double2(0.0, 0.0), w1 = w0;
            if (o > 0) { w0 = *reinterpret_cast<double2*>(W); w1 = *reinterpret_cast<double2*>(W + n); }
            if (!first) {
                const double2 x0 = A.x[pb], x1 = A.x[pb + O6_T];
                w0.x += x0.x; w0.y += x0.y; w1.x += x1.x; w1.y += x1.y;
            }
            *reinterpret_cast<double2*>(W) = w0;
            *reinterpret_cast<double2*>(W + n) = w1;
            e[0] = w0.x; e[1] = w0.y; e[2] = w1.x; e[3] = w1.y;
        }
        if (dead) break;
        __syncthreads();
        pub_f6(sm, t, 0, e);
        pub_f6(sm, t, 1, e);
        nb_sync(sm, t, 16 * M::W);
        double s[1];
        {
            const double* B = A.b + (size_t)p * A.bstride + (size_t)gy * n + gx;
            double ah, av, bh, bv;
            out_f6(sm, t, 0, ah, av, bh, bv);
            r[0] = B[0] - (fma(kw[0], e[0] - ah, kw[1] * (e[0] - e[1])) + fma(ks[0], e[0] - av, ks[2] * (e[0] - e[2])));
            r[3] = B[n + 1] - (fma(kw[5], e[3] - bh, kw[4] * (e[3] - e[2])) + fma(ks[5], e[3] - bv, ks[3] * (e[3] - e[1])));
            out_f6(sm, t, 1, ah, av, bh, bv);
            r[1] = B[1] - (fma(kw[2], e[1] - ah, kw[1] * (e[1] - e[0])) + fma(ks[1], e[1] - av, ks[3] * (e[1] - e[3])));
            r[2] = B[n] - (fma(kw[3], e[2] - bh, kw[4] * (e[2] - e[3])) + fma(ks[4], e[2] - bv, ks[2] * (e[2] - e[0])));
            s[0] = (r[0] * r[0] + r[1] * r[1]) + (r[2] * r[2] + r[3] * r[3]);
        }
        if (sum6(sm, t, OC_RZ, s, 0, [&](const double (&v)[1]) { SC[0] = v[0] <= A.tolout2 * b2 ? 1.0 : 0.0; })) break;
        if (SC[0] == 1.0) { converged = true; break; }
        __syncthreads();                                     // SC[0] is read before the next phase writes it
    }
    if (!V && t.rank == 0 && t.tid == 0) {
        GraphCounters* g = A.cnt;
        atomicAdd(&g->cg_iterations, (unsigned long long)iters);
        atomicAdd(&g->inner_solves, (unsigned long long)inner);
        atomicAdd(&g->residuals, (unsigned long long)phases);
        if (!converged) atomicAdd(&g->nonconv, 1ull);
        atomicMax(&g->itmax, iters);
    }
    oc_leave(t, A.err);
}

// Dense inverses of the 4^2 level's operators, a warp per particle: lane l holds half a row, Gauss-Jordan
// elimination (symmetric positive definite: no pivoting) by shuffles.  A block of the solver's 1024 threads took 15 us for
// it, on one entry a thread; 14 operations a step of one warp cost the FP64 pipe an eighth of that.
__global__ void __launch_bounds__(128) k_inv4(int count, const double* __restrict__ Kw, const double* __restrict__ Ks, const double* __restrict__ E,
                                              const double* __restrict__ Nn, double* __restrict__ out) {
    __shared__ double T[4][16][17];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, p = blockIdx.x * 4 + wp;
    if (p >= count) return;
    const int i = lane >> 1, h = lane & 1, x = i & 3, y = i >> 2, c = p * 16 + i;
    const double kW = Kw[c], kS = Ks[c], kE = x < 3 ? Kw[c + 1] : E[p * 4 + y], kN = y < 3 ? Ks[c + 4] : Nn[p * 4 + x];
    double a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int j = 8 * h + q;
        a[q] = j == i ? (kW + kE) + (kS + kN) : j == i - 1 && x > 0 ? -kW : j == i + 1 && x < 3 ? -kE : j == i - 4 ? -kS : j == i + 4 ? -kN : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const double rp = 1.0 / __shfl_sync(0xffffffffu, a[k & 7], 2 * k + (k >> 3)), f = __shfl_sync(0xffffffffu, a[k & 7], 2 * i + (k >> 3));
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const double rk = __shfl_sync(0xffffffffu, a[q], 2 * k + h) * rp;
            const bool col = 8 * h + q == k;
            a[q] = i == k ? (col ? rp : rk) : col ? -f * rp : fma(-f, rk, a[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) T[wp][i][8 * h + q] = a[q];
    __syncwarp();
    for (int k = lane; k < 256; k += 32) out[(size_t)p * 256 + k] = 0.5 * (T[wp][k >> 4][k & 15] + T[wp][k & 15][k >> 4]);
}

void launch_inv4(Ctx& c, int count) {
    const LevelArrays<double>& L = c.s64.lv[c.s64.nlev - 3];
    k_inv4<<<(count + 3) / 4, 128, 0, c.stream>>>(count, L.Kw, L.Ks, L.E, L.Nn, c.s64.binv); ++c.pc.launches;
}

template <int C, bool V>
static void o6_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int count, cudaStream_t st) {
    check(cudaFuncSetAttribute(k_onchip64<C, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)O6Mem<C>::BYTES), "attr");
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(count * C * C));
    cfg.blockDim = dim3(O6_T);
    cfg.dynamicSmemBytes = O6Mem<C>::BYTES;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C * C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
}

template <int C, bool V>
static bool o6_fits() {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int nc = 0;
    o6_config<C, V>(cfg, attr, 1, nullptr);
    if (C == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nc, k_onchip64<C, V>, O6_T, O6Mem<C>::BYTES) != cudaSuccess) nc = 0;
    } else if (cudaOccupancyMaxActiveClusters(&nc, k_onchip64<C, V>, &cfg) != cudaSuccess) {
        nc = 0;
    }
    (void)cudaGetLastError();
    return nc > 0;
}

// Whether the FP64 solves run on chip: 64^2 or 128^2, the sizes whose faces fit the registers of one block or of a
// cluster of 4 with one block per SM (both measured faster than the passes from 2 particles to thousands, above).
bool onchip64_supported(const Ctx& c) {
    if (c.dim != 2 || mixed_precision(c.cfg) || c.cfg.tile_kernel != 0) return false;
    return c.n == 64 ? o6_fits<1, false>() : c.n == 128 && o6_fits<2, false>();
}

// Whether the multi-pass FP64 solver of a larger grid runs its levels from 128^2 down on chip: the cluster's V-cycle does 33 operations per cell
// of 128^2 where the passes smooth 2.25 times the cells (256 particles of 256^2: 540 -> 395 us per V-cycle below 256^2).
bool onchip64_vcycle_supported(const Ctx& c) {
    return c.n > 128 && o6_fits<2, true>();
}

template <int C, bool V>
static void o6_launch(Ctx& c, O6Args& A, int top, int count) {
    InnerSolver<double>& s = c.s64;
    A.cc = c.cfg.coarse_scale;
    A.nu_c = c.cfg.smooth_sweeps;
    A.n = s.lv[top].n;
    for (int l = 0; l < 6 && (A.n >> l) >= 4; ++l) {
        const LevelArrays<double>& L = s.lv[top + l];
        A.lv[l] = O6Level{L.Kw, L.Ks, L.E, L.Nn, L.inv};
    }
    A.inv4 = s.binv;
    A.err = c.dev_err;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    o6_config<C, V>(cfg, attr, count, c.stream);
    check(cudaLaunchKernelEx(&cfg, k_onchip64<C, V>, A), "on-chip FP64 solve");
    ++c.pc.launches;
}

// Solves a batch into W; the counters accumulate in c.gcnt.
void solve_batch_onchip64(Ctx& c, int count, const Rhs& R, double* W) {
    InnerSolver<double>& s = c.s64;
    O6Args A{};
    A.max_outer = c.cfg.max_refine < 2 ? 2 : c.cfg.max_refine; A.maxit = c.cfg.max_iter;
    A.nu_f = c.cfg.fine_sweeps;
    A.tol2 = A.tolout2 = c.cfg.tol_outer * c.cfg.tol_outer;
    A.floor2 = 0.25 * A.tolout2;
    A.b2const = R.b2const; A.b2pp = R.b2pp;
    A.b = R.b64; A.bstride = R.stride;
    A.x = reinterpret_cast<double2*>(s.x); A.p = reinterpret_cast<double2*>(s.p[0]); A.q = reinterpret_cast<double2*>(s.q);
    A.W = W;
    A.cnt = c.gcnt;
    if (c.n == 64) o6_launch<1, false>(c, A, 0, count);
    else o6_launch<2, false>(c, A, 0, count);
}

// The V-cycle from the level of 128^2 down (r to e2 there) for the active particles.
void launch_vcycle64(Ctx& c, int level, int nact) {
    InnerSolver<double>& s = c.s64;
    O6Args A{};
    A.max_outer = 1;
    A.nu_f = c.cfg.smooth_sweeps;
    A.vr = s.lv[level].r;
    A.ve = s.lv[level].e2;
    A.list = s.list;
    A.nact = c.graph ? s.nact : nullptr;
    o6_launch<2, true>(c, A, level, nact);
}

}  // namespace smcgm
