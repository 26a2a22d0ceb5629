// The mixed-precision solve of a batch of particles on chip: one launch runs every refinement
// phase, CG iteration and V-cycle of a particle in one thread block (64^2), or in a cluster of
// 4 (128^2) or 16 (256^2) blocks that exchange edges through distributed shared memory.
//
// Why: the multi-pass solver (solver.cu) reads and writes every vector of the finest grid three
// times per CG iteration (82 bytes a cell: 4.6 TB/s at 4096 particles of 256^2), pays a launch
// for each pass of each level and waits for the host after each iteration; on 64^2 and 128^2
// grids the launches and the coarse levels' barriers are most of its time.  Here a cell's faces,
// residual and correction stay in registers for the whole solve, CG's p and the reciprocal
// diagonals in shared memory, and only the solution's three FP32 parts and x go through L2.
// Measured against it (synthesis and set-up included): 1024 solves of 64^2 4.17 -> 0.66 ms, 2048 of
// 128^2 15.7 -> 6.5 ms, 2048 of 256^2 54.9 -> 41.3 ms, 2 of 256^2 2.35 -> 0.34 ms.
//
// Layout: a block covers a strip of 64 C x 64 / C cells (C = n / 64) with 16 C x 16 / C threads, a
// 4 x 4 patch each; a thread also owns the 2 x 2 cells below its patch on the next level and the
// one cell on the level after that, so restriction and prolongation over those levels need no
// exchange, and their Galerkin faces are sums of the patch's.  Neighbours exchange the edge values
// of one colour per half-sweep; a strip's first and last thread rows also store theirs into the
// neighbouring block's guard slots (guards at the domain's walls stay zero: the wall faces only
// enter the diagonal).  Strips rather than squares: two neighbours instead of four, whole rows of
// lanes store together, and only the edge rows' warps wait for a neighbour (squares: 2048 of 256^2
// 48.7 ms).  Below that every block of a cluster holds the whole coarse problem (32^2 for 16
// blocks, 16^2 for 4) and solves it redundantly, which costs less than sharing it; the 8^2 level is
// solved with its dense inverse, formed once per solve.  A larger grid's passes use the 128^2 form for
// one V-cycle per launch, with the dense inverses formed at set-up.
//
// The V-cycle is otherwise that of solver.cu (symmetric red-black Gauss-Seidel, the same sweeps,
// Galerkin coarsening, scaled correction).  The residual after a pre-smoothing that ends with the
// black cells vanishes there, so only the red cells are restricted.
//
// What bounds it: the latency of about 30 barrier-separated phases per CG iteration (45 and 25
// remote exchanges at 256^2 and 128^2), not HBM: two blocks per SM (128 registers a
// thread, 80 to 113 KB) reach 0.53 (64^2) and 0.38 (256^2) issued instructions per scheduler cycle.
// 14 clusters of 16 fit the GPU at a time (112 of 152 SMs).
#include <cstdio>
#include "smcgm_internal.cuh"
#include "common.cuh"
#include "df32.cuh"
#include "onchip.cuh"

namespace smcgm {

constexpr int OC_T = 256;

struct OcArgs {
    int max_outer, maxit, nu_f, nu_c;
    float cc;
    float2 tol2;                 // the pair of the squared reduction per phase
    double floor2, tolout2;
    double b2const;
    const double* b2pp;
    const float *Kw, *Ks, *E, *Nn, *Kwl, *Ksl, *El, *Nl;   // faces: high and low parts
    const float2* bdf;
    size_t bstride;
    float4 *x, *wh, *wm, *wl;    // per particle n^2 floats, [block][patch row][thread]
    double* W;
    const int* badp;
    GraphCounters* cnt;
    int* err;
    // the V-cycle alone: right-hand sides, corrections, the active particles, the 8^2 level's dense inverses (`build`: form them)
    const float* vr;
    float *ve, *inv8;
    const int *list, *nact;
    int build;
};

// A block covers 64 C x 64 / C cells (a strip of rows): W x H threads, a 4 x 4 patch each.
// Shared-memory offsets (floats).
template <int C_>
struct OcMem {
    static constexpr int C = C_, CC = C * C, W = 16 * C, H = 16 / C;
    static constexpr int SZH = H * (W + 1), SZV = (H + 1) * W;   // float2 per colour of the sides W, E (H rows of W + 1) and S, N
    static constexpr int PT = W + 2, PL = (H + 2) * PT;     // pitch and size of a plane with a ring of guards
    static constexpr int P4 = 0;                            // p: 4 float4 slots
    static constexpr int INVF = P4 + 16 * OC_T;             // 1/D of the patch: 2 float4 per colour
    static constexpr int INVH = INVF + 16 * OC_T;           // float4
    static constexpr int LF = INVH + 4 * OC_T;              // C = 4: 12 faces and 4 1/D of the 32^2 level's patch
    static constexpr int SF = LF + (C == 4 ? 16 * OC_T : 0);   // C > 1: 4 faces of the 16^2 level's cell
    static constexpr int INV8 = SF + (C > 1 ? 4 * OC_T : 0);   // dense inverse of the 8^2 level, [k][row]
    static constexpr int R8 = INV8 + 4096;
    static constexpr int PART8 = R8 + 64;
    static constexpr int RED = PART8 + 256;                 // 3 slots of 8 CC warp sums (df32)
    static constexpr int THR = RED + 3 * 16 * CC;           // |r|^2 no phase need go below, |r|^2 at which the solve ends (df32)
    static constexpr int RB = THR + 4;                      // gathered right-hand side of the first local level
    static constexpr int STG = PART8;                       // C > 1: pair sums of a block's part of it, H x W / 2
    static constexpr int SIDE = RB + (C == 4 ? 1024 : C == 2 ? 256 : 0);   // 4 sides x 2 colours
    static constexpr int HP = SIDE + 8 * (SZH + SZV);       // 4 planes: cell (i, j) of each 2 x 2 patch
    static constexpr int QP = HP + 4 * PL;
    static constexpr int LP = QP + PL;                      // C = 4: as HP for the 32^2 level (16 x 16 threads)
    static constexpr int SP = LP + (C == 4 ? 4 * 324 : 0);  // C > 1: as QP for the 16^2 level
    static constexpr int TOK = SP + (C > 1 ? 324 : 0);      // C > 1: where the words of w_sync land
    static constexpr int ENDF = (TOK + 2 + 1) / 2 * 2;      // C > 1: 2 x 2 + 4 mbarriers (8 bytes each)
    static constexpr int BARS = 4 * ENDF;                   // bytes
    static constexpr int TOTAL = ENDF + (C > 1 ? 16 : 0);
    static constexpr size_t BYTES = (size_t)TOTAL * 4;
    static_assert(BYTES <= 228 * 1024 / 2 - 1024, "two blocks per SM");
    static_assert(STG % 4 == 0 && RB % 4 == 0 && SIDE % 2 == 0 && RED % 4 == 0, "vector alignment");
};

// The exchange that starts an iteration: |r|^2 and the first red edges.  True if a wait ran out in any thread
// of the block, which then leaves the loops alike (threads must not decide on sums that others did not see).
template <int C>
__device__ __forceinline__ bool rr_sync(float* sm, OcPos<OcMem<C>>& t) {
    if (C == 1) {
        __syncthreads();
        return false;
    }
    if (t.tid == 0) oc_expect(t, all_bar<OcMem<C>>(sm, OC_RR), 64 * OcMem<C>::CC);
    nb_wait(sm, t, 8 * OcMem<C>::W);
    oc_wait(t, all_bar<OcMem<C>>(sm, OC_RR), (t.par >> OC_RR) & 1);
    t.par ^= 1u << OC_RR;
    return __syncthreads_or(t.dead);
}

// The solution's parts in global memory are written: visible to the block and, for the edge rows, the neighbours' too.
// Not a cluster barrier: those have no bound, and a block whose wait ran out must meet the others at the last one
// only.  A word to either neighbour follows the block's writes instead, counted like an edge exchange.
template <int C>
__device__ __forceinline__ void w_sync(float* sm, OcPos<OcMem<C>>& t) {
    using M = OcMem<C>;
    if (C > 1 && t.nbase) __threadfence();
    __syncthreads();
    if (C > 1) {
        if (t.nbase && t.tx == 0) oc_store(t.nbase + 4 * (M::TOK + (t.lower ? 1 : 0)), 0.f, t.nbase + nb_bar(t, !t.lower));
        nb_wait(sm, t, 4);
        if (t.nbase) __threadfence();
    }
}

// ---- sums over the particle's cells: every thread of every block ends with the same bits ----
// FP32 within 256 cells (half a warp); these sums (in a cluster: the exact sums of a warp's two) are added as fixed-point numbers, 44
// bits below the largest, whose integer sums do not depend on an order.  So the sum over 65536 cells has the error of its
// 256-cell terms, as the passes' sums have (FP32 in a tile, FP64 across tiles).  Two integer additions over a warp take
// little more than the five FP32 additions by shuffle of a plain sum: a gradient call of 2048 particles of 128^2 13.90 ms with FP32
// sums throughout, 14.04 so, 14.67 with pairs of FP32 by shuffle; a move of 4096 of 256^2 83.7, 86.3, 88.0.
template <int C>
__device__ __forceinline__ void red_put(float* sm, const OcPos<OcMem<C>>& t, int slot, float v) {
    using M = OcMem<C>;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = t.tid & 31, wid = t.tid >> 5;
    float* dst = sm + M::RED + slot * 16 * M::CC + 2 * ((int)t.rank * 8 + wid);
    if (C == 1) {
        if ((lane & 15) == 0) dst[lane >> 4] = v;
        return;
    }
    float2 w;
    two_sum(v, __shfl_xor_sync(0xffffffffu, v, 16), w.x, w.y);
    if (lane < M::CC) oc_store2(oc_map(dst, (uint32_t)lane), w, oc_map(all_bar<OcMem<C>>(sm, slot), (uint32_t)lane));
}
template <int C>
__device__ __forceinline__ df32 red_get(const float* sm, const OcPos<OcMem<C>>& t, int slot) {
    using M = OcMem<C>;
    constexpr int NV = C == 4 ? 4 : 1;                       // sums per lane
    const float* s = sm + M::RED + slot * 16 * M::CC;
    const int lane = t.tid & 31;
    float2 v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k)
        v[k] = C > 1 ? reinterpret_cast<const float2*>(s)[32 * k + lane] : make_float2(lane < 16 ? s[lane] : 0.f, 0.f);
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < NV; ++k) top = max(top, __float_as_uint(v[k].x) & 0x7fffffffu);
    top = __reduce_max_sync(0xffffffffu, top);
    const int ex = max((int)(top >> 23), 24);                // sums below 2^-103 count as that
    const float up = __int_as_float((275 - ex) << 23), down = __int_as_float((ex - 21) << 23);   // to |v| < 2^22 and back
    constexpr float RINT = 12582912.f;                       // 1.5 2^23: x + RINT holds rint(x) in its last bits
    int q = 0, r = 0;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const float a = fmaf(v[k].x, up, RINT), f = fmaf(v[k].x, up, -__fsub_rn(a, RINT));   // the integer part; the rest, exact
        q += __float_as_int(a) - 0x4b400000;
        r += __float_as_int(fmaf(C > 1 ? fmaf(v[k].y, up, f) : f, 4194304.f, RINT)) - 0x4b400000;
    }
    q = __reduce_add_sync(0xffffffffu, q);                   // at most 128 of 2^22 each (r: of 0.75 2^22)
    r = __reduce_add_sync(0xffffffffu, r);
    df32 d;
    two_sum((float)(q >> 12) * 4096.f, (float)(q & 4095), d.hi, d.lo);
    two_sum(d.hi, fmaf((float)r, 1.f / 4194304.f, d.lo), d.hi, d.lo);
    d.hi *= down;
    d.lo *= down;
    if (top >= 0x7f800000u) d.hi = __int_as_float(0x7fffffff);   // infinities and NaN
    return d;
}
__host__ __device__ __forceinline__ float2 pair_of(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}
__device__ __forceinline__ bool at_most(df32 a, df32 b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }
// a / b to FP32: the remainder of a first quotient, formed exactly, corrects it.  In a field of u = 50 r.z and p.Ap are subnormal, whose
// reciprocal overflows: both are brought up first.
__device__ __forceinline__ float quotient(df32 a, df32 b) {
    const float up = fabsf(b.hi) < 0x1p-96f ? 0x1p64f : 1.f, c = b.hi * up, d = a.hi * up;
    const float inv = 1.f / c, q = d * inv;
    return fmaf((fmaf(-q, c, d) + a.lo * up) - q * (b.lo * up), inv, q);
}

// ---- the finest level: a 4 x 4 patch, e[4 j + i] of cell (i, j); red: i + j even ----
// Sides of colour col: 0 W, 1 E (rows of W + 1), 2 S, 3 N (H + 1 rows of W); the pair holds the side's two
// cells of that colour in ascending order.
template <int C>
__device__ __forceinline__ float2* side(float* sm, int s, int col) {
    using M = OcMem<C>;
    return reinterpret_cast<float2*>(sm + M::SIDE) + (s < 2 ? (s * 2 + col) * M::SZH : 4 * M::SZH + ((s - 2) * 2 + col) * M::SZV);
}

template <int C, int COL>
__device__ __forceinline__ void pub_f(float* sm, const OcPos<OcMem<C>>& t, const float (&e)[16]) {
    using M = OcMem<C>;
    const float2 s = COL == 0 ? make_float2(e[0], e[2]) : make_float2(e[1], e[3]);
    const float2 n = COL == 0 ? make_float2(e[13], e[15]) : make_float2(e[12], e[14]);
    if (C > 1 && t.nbase) {
        // to the neighbour's guard row: its north side's row 0 from below it, its south side's row H from above
        const int at = 4 * M::SZH + (t.lower ? COL * M::SZV + M::H * M::W : (2 + COL) * M::SZV);
        oc_store2(t.nbase + 4 * M::SIDE + 8 * (at + t.tx), t.lower ? s : n, t.nbase + nb_bar(t, !t.lower));
    }
    side<C>(sm, 0, COL)[t.ty * (M::W + 1) + t.tx] = COL == 0 ? make_float2(e[0], e[8]) : make_float2(e[4], e[12]);
    side<C>(sm, 1, COL)[t.ty * (M::W + 1) + t.tx + 1] = COL == 0 ? make_float2(e[7], e[15]) : make_float2(e[3], e[11]);
    side<C>(sm, 2, COL)[t.ty * M::W + t.tx] = s;
    side<C>(sm, 3, COL)[(t.ty + 1) * M::W + t.tx] = n;
}

struct HaloF { float2 w, e, s, n; };
template <int C>
__device__ __forceinline__ HaloF halo_f(float* sm, const OcPos<OcMem<C>>& t, int col) {   // the neighbours' cells of colour col
    HaloF h;
    using M = OcMem<C>;
    h.w = side<C>(sm, 1, col)[t.ty * (M::W + 1) + t.tx];
    h.e = side<C>(sm, 0, col)[t.ty * (M::W + 1) + t.tx + 1];
    h.s = side<C>(sm, 3, col)[t.ty * M::W + t.tx];
    h.n = side<C>(sm, 2, col)[(t.ty + 1) * M::W + t.tx];
    return h;
}
__device__ __forceinline__ float pick(float2 v, int k) { return k ? v.y : v.x; }

// Neighbours of cell (i, j), from the patch or the halo of the other colour.
#define OC_NB_F(i, j, e, h, w_, e_, s_, n_)                                  \
    const float w_ = (i) > 0 ? e[4 * (j) + (i) - 1] : pick(h.w, (j) >> 1);   \
    const float e_ = (i) < 3 ? e[4 * (j) + (i) + 1] : pick(h.e, (j) >> 1);   \
    const float s_ = (j) > 0 ? e[4 * (j) - 4 + (i)] : pick(h.s, (i) >> 1);   \
    const float n_ = (j) < 3 ? e[4 * (j) + 4 + (i)] : pick(h.n, (i) >> 1);

template <int C, int COL>
__device__ __forceinline__ void inv_f(const float* sm, const OcPos<OcMem<C>>& t, float (&v)[8]) {
    const float4* p = reinterpret_cast<const float4*>(sm + OcMem<C>::INVF) + 2 * COL * OC_T + t.tid;
    const float4 a = p[0], b = p[OC_T];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

template <int C, int COL>
__device__ __forceinline__ void sweep_f(float* sm, const OcPos<OcMem<C>>& t, const float (&kw)[20], const float (&ks)[20], const float (&r)[16],
                                        float (&e)[16], bool pointwise) {
    float inv[8];
    inv_f<C, COL>(sm, t, inv);
    if (pointwise) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = (j + COL) & 1; i < 4; i += 2) e[4 * j + i] = r[4 * j + i] * inv[2 * j + (i >> 1)];
        return;
    }
    const HaloF h = halo_f<C>(sm, t, 1 - COL);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = (j + COL) & 1; i < 4; i += 2) {
            OC_NB_F(i, j, e, h, ew, ee, es, en)
            const float num = fmaf(ks[4 * (j + 1) + i], en, fmaf(ks[4 * j + i], es, fmaf(kw[5 * j + i + 1], ee, fmaf(kw[5 * j + i], ew, r[4 * j + i]))));
            e[4 * j + i] = num * inv[2 * j + (i >> 1)];
        }
}

// ---- a level with a 2 x 2 patch per thread: cells 0 (0,0), 1 (1,0), 2 (0,1), 3 (1,1); red: 0 and 3 ----
struct Patch2 { float w[6], s[6]; };   // west faces [j][0..2], south faces [0..2][i]
// A thread's entry, pitch and plane size: the block's own planes (SHARED) or those of a local level.
template <int C, bool SHARED> struct OcPl {
    static constexpr int PT = SHARED ? OcMem<C>::PT : 18, PL = SHARED ? OcMem<C>::PL : 324;
    static __device__ __forceinline__ int at(const OcPos<OcMem<C>>& t) { return SHARED ? (t.ty + 1) * PT + t.tx + 1 : (t.ly + 1) * PT + t.lx + 1; }
};
template <int C, bool SHARED>
__device__ __forceinline__ void pub_h(float* pl, const OcPos<OcMem<C>>& t, int col, const float (&e)[4]) {
    using O = OcPl<C, SHARED>;
    if (SHARED && C > 1 && t.nbase) {   // cells 0, 1 (2, 3) to the block below (above), into its guard row
        using M = OcMem<C>;
        const int plane = t.lower ? (col ? 1 : 0) : (col ? 2 : 3);
        oc_store(t.nbase + 4 * (M::HP + plane * M::PL + (t.lower ? (M::H + 1) * M::PT : 0) + t.tx + 1),
                 t.lower ? (col ? e[1] : e[0]) : (col ? e[2] : e[3]), t.nbase + nb_bar(t, !t.lower));
    }
    const int at = O::at(t);
    pl[(col ? 1 : 0) * O::PL + at] = e[col ? 1 : 0];
    pl[(col ? 2 : 3) * O::PL + at] = e[col ? 2 : 3];
}
// Sum of k e over the four neighbours of the two cells of a colour (0: cells 0 and 3, 1: cells 1 and 2).
template <int C, bool SHARED>
__device__ __forceinline__ void nb_h(const float* pl, const OcPos<OcMem<C>>& t, int col, const Patch2& k, const float (&e)[4], float& a, float& b) {
    using O = OcPl<C, SHARED>;
    const float *p0 = pl + O::at(t), *p1 = p0 + O::PL, *p2 = p1 + O::PL, *p3 = p2 + O::PL;
    if (col == 0) {
        a = fmaf(k.w[0], p1[-1], fmaf(k.s[0], p2[-O::PT], fmaf(k.w[1], e[1], k.s[2] * e[2])));
        b = fmaf(k.w[5], p2[1], fmaf(k.s[5], p1[O::PT], fmaf(k.w[4], e[2], k.s[3] * e[1])));
    } else {
        a = fmaf(k.w[2], p0[1], fmaf(k.s[1], p3[-O::PT], fmaf(k.w[1], e[0], k.s[3] * e[3])));
        b = fmaf(k.w[3], p3[-1], fmaf(k.s[4], p0[O::PT], fmaf(k.w[4], e[3], k.s[2] * e[0])));
    }
}
__device__ __forceinline__ void diag_h(const Patch2& k, float (&d)[4]) {
    d[0] = (k.w[0] + k.w[1]) + (k.s[0] + k.s[2]);
    d[1] = (k.w[1] + k.w[2]) + (k.s[1] + k.s[3]);
    d[2] = (k.w[3] + k.w[4]) + (k.s[2] + k.s[4]);
    d[3] = (k.w[4] + k.w[5]) + (k.s[3] + k.s[5]);
}

// Pre-smoothing from e = 0 and the sum of the red cells' residuals (the black ones' are zero).
template <int C, bool SHARED>
__device__ __forceinline__ float pre_h(float* sm, float* pl, OcPos<OcMem<C>>& t, int nu, const Patch2& k, const float4 inv, const float (&r)[4], float (&e)[4]) {
    float a, b;
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        if (sw == 0) {
            e[0] = r[0] * inv.x;
            e[3] = r[3] * inv.w;
        } else {
            nb_h<C, SHARED>(pl, t, 0, k, e, a, b);
            e[0] = (r[0] + a) * inv.x;
            e[3] = (r[3] + b) * inv.w;
        }
        pub_h<C, SHARED>(pl, t, 0, e);
        if (SHARED) nb_sync(sm, t, 4 * OcMem<C>::W); else __syncthreads();
        nb_h<C, SHARED>(pl, t, 1, k, e, a, b);
        e[1] = (r[1] + a) * inv.y;
        e[2] = (r[2] + b) * inv.z;
        pub_h<C, SHARED>(pl, t, 1, e);
        if (SHARED) nb_sync(sm, t, 4 * OcMem<C>::W); else __syncthreads();
    }
    nb_h<C, SHARED>(pl, t, 0, k, e, a, b);
    float d[4];
    diag_h(k, d);
    return (r[0] + fmaf(-d[0], e[0], a)) + (r[3] + fmaf(-d[3], e[3], b));
}
// e already holds the corrected values; post-smoothing (black, red); the last red values are not published.
template <int C, bool SHARED>
__device__ __forceinline__ void post_h(float* sm, float* pl, OcPos<OcMem<C>>& t, int nu, const Patch2& k, const float4 inv, const float (&r)[4], float (&e)[4]) {
    float a, b;
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        pub_h<C, SHARED>(pl, t, 0, e);
        if (SHARED) nb_sync(sm, t, 4 * OcMem<C>::W); else __syncthreads();
        nb_h<C, SHARED>(pl, t, 1, k, e, a, b);
        e[1] = (r[1] + a) * inv.y;
        e[2] = (r[2] + b) * inv.z;
        pub_h<C, SHARED>(pl, t, 1, e);
        if (SHARED) nb_sync(sm, t, 4 * OcMem<C>::W); else __syncthreads();
        nb_h<C, SHARED>(pl, t, 0, k, e, a, b);
        e[0] = (r[0] + a) * inv.x;
        e[3] = (r[3] + b) * inv.w;
    }
}

// ---- a level with one cell per thread; red: tx + ty even ----
struct Cell1 { float w, e, s, n; };
template <int C, bool SHARED>
__device__ __forceinline__ void pub_q(float* pl, const OcPos<OcMem<C>>& t, float e) {
    if (SHARED && C > 1 && t.nbase) {
        using M = OcMem<C>;
        oc_store(t.nbase + 4 * (M::QP + (t.lower ? (M::H + 1) * M::PT : 0) + t.tx + 1), e, t.nbase + nb_bar(t, !t.lower));
    }
    pl[OcPl<C, SHARED>::at(t)] = e;
}
template <int C, bool SHARED>
__device__ __forceinline__ float nb_q(const float* pl, const OcPos<OcMem<C>>& t, const Cell1& k) {
    using O = OcPl<C, SHARED>;
    const float* p = pl + O::at(t);
    return fmaf(k.w, p[-1], fmaf(k.e, p[1], fmaf(k.s, p[-O::PT], k.n * p[O::PT])));
}
template <int C, bool SHARED>
__device__ __forceinline__ bool red_q(const OcPos<OcMem<C>>& t) { return ((SHARED ? t.tx + t.ty : t.lx + t.ly) & 1) == 0; }
// Pre-smoothing from e = 0; returns the residual of a red cell, 0 for a black one.
template <int C, bool SHARED>
__device__ __forceinline__ float pre_q(float* sm, float* pl, OcPos<OcMem<C>>& t, int nu, const Cell1& k, float inv, float r, float& e) {
    const bool red = red_q<C, SHARED>(t);
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        if (red) {
            e = (sw == 0 ? r : r + nb_q<C, SHARED>(pl, t, k)) * inv;
            pub_q<C, SHARED>(pl, t, e);
        }
        if (SHARED) nb_sync(sm, t, 2 * OcMem<C>::W); else __syncthreads();
        if (!red) {
            e = (r + nb_q<C, SHARED>(pl, t, k)) * inv;
            pub_q<C, SHARED>(pl, t, e);
        }
        if (SHARED) nb_sync(sm, t, 2 * OcMem<C>::W); else __syncthreads();
    }
    return red ? r + fmaf(-((k.w + k.e) + (k.s + k.n)), e, nb_q<C, SHARED>(pl, t, k)) : 0.f;
}
template <int C, bool SHARED>
__device__ __forceinline__ void post_q(float* sm, float* pl, OcPos<OcMem<C>>& t, int nu, const Cell1& k, float inv, float r, float& e) {
    const bool red = red_q<C, SHARED>(t);
#pragma unroll 1
    for (int sw = 0; sw < nu; ++sw) {
        if (red) pub_q<C, SHARED>(pl, t, e);
        if (SHARED) nb_sync(sm, t, 2 * OcMem<C>::W); else __syncthreads();
        if (!red) {
            e = (r + nb_q<C, SHARED>(pl, t, k)) * inv;
            pub_q<C, SHARED>(pl, t, e);
        }
        if (SHARED) nb_sync(sm, t, 2 * OcMem<C>::W); else __syncthreads();
        if (red) e = (r + nb_q<C, SHARED>(pl, t, k)) * inv;
    }
}

// Sum over the 2 x 2 threads that share a coarse cell (all in one warp).
__device__ __forceinline__ float quad_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

// Faces of the 2 x 2-thread coarse cell: the sums of the fine faces on its sides.
__device__ __forceinline__ Cell1 coarse_faces(const Cell1& k, int tx, int ty) {
    const Cell1 a{k.w + __shfl_xor_sync(0xffffffffu, k.w, 16), k.e + __shfl_xor_sync(0xffffffffu, k.e, 16),
                  k.s + __shfl_xor_sync(0xffffffffu, k.s, 1), k.n + __shfl_xor_sync(0xffffffffu, k.n, 1)};
    const float w1 = __shfl_xor_sync(0xffffffffu, a.w, 1), e1 = __shfl_xor_sync(0xffffffffu, a.e, 1);
    const float s1 = __shfl_xor_sync(0xffffffffu, a.s, 16), n1 = __shfl_xor_sync(0xffffffffu, a.n, 16);
    return Cell1{(tx & 1) ? w1 : a.w, (tx & 1) ? a.e : e1, (ty & 1) ? s1 : a.s, (ty & 1) ? a.n : n1};
}

// Dense inverse of the 8^2 level from its faces (each held by the four threads of its cell), by
// Gauss-Jordan elimination in registers: thread (row, quarter) holds 16 columns of a row, the
// pivot row and column go through shared memory, one barrier per step.  Stored symmetrised.
template <int C>
__device__ __forceinline__ void build_inv8(float* sm, const OcPos<OcMem<C>>& t, const Cell1& k8) {
    using M = OcMem<C>;
    float* M8 = sm + M::INV8;
    float* fa = M8;                                         // 4 x 64 faces first
    if (((t.lx | t.ly) & 1) == 0) {
        const int c = (t.ly >> 1) * 8 + (t.lx >> 1);
        fa[c] = k8.w; fa[64 + c] = k8.e; fa[128 + c] = k8.s; fa[192 + c] = k8.n;
    }
    __syncthreads();
    const int row = t.tid & 63, q = t.tid >> 6;
    float a[16];
    {
        const float w = fa[row], e = fa[64 + row], s = fa[128 + row], n = fa[192 + row];
        const int I = row & 7, J = row >> 3;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const int col = 16 * q + c;
            float v = 0.f;
            if (col == row) v = (w + e) + (s + n);
            if (I > 0 && col == row - 1) v = -w;
            if (I < 7 && col == row + 1) v = -e;
            if (J > 0 && col == row - 8) v = -s;
            if (J < 7 && col == row + 8) v = -n;
            a[c] = v;
        }
    }
    __syncthreads();
    float* buf = M8;                                        // two buffers of (row 64, column 64)
#pragma unroll 1
    for (int q0 = 0; q0 < 4; ++q0) {
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const int k = 16 * q0 + kk;
            float* rb = buf + (kk & 1) * 128;
            if (row == k) {
#pragma unroll
                for (int c = 0; c < 16; ++c) rb[16 * q + c] = a[c];
            }
            if (q == q0) rb[64 + row] = a[kk];
            __syncthreads();
            const float p = 1.f / rb[k], f = rb[64 + row];
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const float rk = rb[16 * q + c] * p;
                a[c] = row == k ? rk : fmaf(-f, rk, a[c]);
            }
            if (q == q0) a[kk] = row == k ? p : -f * p;
        }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 16; ++c) M8[(16 * q + c) * 64 + row] = a[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 16; ++c) a[c] = 0.5f * (a[c] + M8[row * 64 + 16 * q + c]);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 16; ++c) M8[(16 * q + c) * 64 + row] = a[c];
    __syncthreads();
}

// The 16^2 level (one cell per thread, its plane pl) with the dense solve of the 8^2 level below it.
template <int C, bool SHARED>
__device__ __forceinline__ void level16(float* sm, float* pl, OcPos<OcMem<C>>& t, int nu, float cc, const Cell1& k, float inv, float r, float& e) {
    using M = OcMem<C>;
    const float res = quad_sum(pre_q<C, SHARED>(sm, pl, t, nu, k, inv, r, e));
    if (((t.lx | t.ly) & 1) == 0) sm[M::R8 + (t.ly >> 1) * 8 + (t.lx >> 1)] = res;
    __syncthreads();
    {
        const int row = t.tid & 63, q = t.tid >> 6;
        const float* m = sm + M::INV8 + 16 * q * 64 + row;
        const float4* r8 = reinterpret_cast<const float4*>(sm + M::R8 + 16 * q);
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4 v = r8[c];
            a = fmaf(m[(4 * c) * 64], v.x, a);
            b = fmaf(m[(4 * c + 1) * 64], v.y, b);
            a = fmaf(m[(4 * c + 2) * 64], v.z, a);
            b = fmaf(m[(4 * c + 3) * 64], v.w, b);
        }
        sm[M::PART8 + 64 * q + row] = a + b;
    }
    __syncthreads();
    const float* p8 = sm + M::PART8 + (t.ly >> 1) * 8 + (t.lx >> 1);
    e = fmaf(cc, (p8[0] + p8[64]) + (p8[128] + p8[192]), e);
    post_q<C, SHARED>(sm, pl, t, nu, k, inv, r, e);
}

__device__ __forceinline__ Patch2 coarsen_f(const float (&kw)[20], const float (&ks)[20]) {
    Patch2 h;
#pragma unroll
    for (int J = 0; J < 2; ++J)
#pragma unroll
        for (int I = 0; I < 3; ++I) h.w[3 * J + I] = kw[5 * (2 * J) + 2 * I] + kw[5 * (2 * J + 1) + 2 * I];
#pragma unroll
    for (int J = 0; J < 3; ++J)
#pragma unroll
        for (int I = 0; I < 2; ++I) h.s[2 * J + I] = ks[4 * (2 * J) + 2 * I] + ks[4 * (2 * J) + 2 * I + 1];
    return h;
}
__device__ __forceinline__ Cell1 coarsen_h(const Patch2& h) {
    return Cell1{h.w[0] + h.w[3], h.w[2] + h.w[5], h.s[0] + h.s[1], h.s[4] + h.s[5]};
}

// ---- the solution as three FP32 parts (72 bits): no FP64 instruction, whose rate is 1/64 of FP32 ----
__device__ __forceinline__ void tri_add(float& h, float& m, float& l, float x) {
    float s, e1, u, e2;
    two_sum(h, x, s, e1);
    two_sum(m, e1, u, e2);
    const float l2 = __fadd_rn(l, e2);
    float u2;
    fast_two_sum(s, u, h, u2);
    fast_two_sum(u2, l2, m, l);
}
// The flux k (a - b) of a face as p + e: the difference to ~2^-70 |a| (hi rounded, lo the rest), p the
// rounded product of the high parts, e its error and the products with the low parts.
__device__ __forceinline__ df32 tri_flux(float kh, float kl, float ah, float am, float al, float bh, float bm, float bl) {
    float s, e, s2, e2, u, u2;
    two_sum(ah, -bh, s, e);
    two_sum(am, -bm, s2, e2);
    two_sum(s, s2, u, u2);
    const float low = __fadd_rn(__fadd_rn(u2, e), __fadd_rn(e2, __fsub_rn(al, bl)));
    df32 r;
    r.hi = __fmul_rn(kh, u);
    r.lo = fmaf(kh, low, fmaf(kl, u, fmaf(kh, u, -r.hi)));
    return r;
}
// acc += f (TwoSum of the high parts, the rest in plain FP32: a compensated sum, error ~2^-47 of the terms).
__device__ __forceinline__ void acc_add(df32& acc, float hi, float lo) {
    float s, e;
    two_sum(acc.hi, hi, s, e);
    acc.hi = s;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(e, lo));
}
// Parts outside the range of the integer form below (zeros, mostly).
__device__ __noinline__ double tri_to_double_slow(float h, float m, float l, int add) {
    return ((double)h + ((double)m + (double)l)) * exp2((double)add);
}
// (h + m + l) 2^add, rounded to FP64 with one integer conversion.
__device__ __forceinline__ double tri_to_double(float h, float m, float l, int add) {
    const int bh = __float_as_int(h), bm = __float_as_int(m), bl = __float_as_int(l);
    const int eh = (bh >> 23) & 255, em = (bm >> 23) & 255, el = (bl >> 23) & 255;
    if (eh < 64 || eh > 250) return tri_to_double_slow(h, m, l, add);
    auto mant = [](int b, int e) -> long long {
        const int v = e ? (b & 0x7fffff) | 0x800000 : 0;
        return (long long)(b < 0 ? -v : v);
    };
    long long I = mant(bh, eh) << 36;                       // unit 2^(eh - 150 - 36)
    auto shifted = [&](int b, int e) -> long long {
        const int s = 36 - (eh - e);
        const long long v = mant(b, e);
        return s >= 0 ? v << min(s, 38) : s > -40 ? v >> (-s) : 0ll;
    };
    I += shifted(bm, em) + shifted(bl, el);
    const double d = __ll2double_rn(I);
    return I ? __hiloint2double(__double2hiint(d) + ((eh - 186 + add) << 20), __double2loint(d)) : 0.0;
}

// One particle per cluster of C x C blocks, n = 64 C.  V: one V-cycle only, for the levels from n down of a larger grid's
// multi-pass solver (or, at set-up, only the dense inverse that it uses).
template <int C, bool V>
__global__ void __launch_bounds__(OC_T, 2) k_onchip(const OcArgs A) {
    using M = OcMem<C>;
    extern __shared__ __align__(16) float sm[];
    const int n = 64 * C;
    if (V && A.nact && (int)(blockIdx.x / M::CC) >= *A.nact) return;
    const int p = V && A.list ? A.list[blockIdx.x / M::CC] : (int)(blockIdx.x / M::CC);
    OcPos<OcMem<C>> t;
    oc_place(t, sm, (int)threadIdx.x % M::W, (int)threadIdx.x / M::W);
    t.lx = t.tid & 15;
    t.ly = t.tid >> 4;
    const int gx = 4 * t.tx, gy = 4 * ((int)t.rank * M::H + t.ty);
    const size_t base = (size_t)p * n * n;
    const double b2 = V ? 1.0 : A.b2pp ? A.b2pp[p] : A.b2const;
    if (!V && (!(b2 > 0.0) || (A.badp && A.badp[p]))) {             // not solved: w = 0 (the whole cluster alike)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            double2* o = reinterpret_cast<double2*>(A.W + base + (size_t)(gy + j) * n + gx);
            o[0] = o[1] = make_double2(0.0, 0.0);
        }
        return;
    }
    // the system scaled by a power of two so that |b| is in [1, 2): squares stay in range in FP32
    int sexp = -((int)((__double2hiint(b2) >> 20) & 0x7ff) - 1023 >> 1);
    sexp = max(-100, min(100, sexp));
    const float scale = __int_as_float((127 + sexp) << 23);
    if (!V && t.tid == 0) {                                          // read after the barriers of the set-up
        const double b2s = b2 * (double)scale * (double)scale;
        reinterpret_cast<float2*>(sm + M::THR)[0] = pair_of(A.floor2 * b2s);
        reinterpret_cast<float2*>(sm + M::THR)[1] = pair_of(A.tolout2 * b2s);
    }
    // guards and planes
    for (int i = M::SIDE + t.tid; i < M::ENDF; i += OC_T) sm[i] = 0.f;
    if (C > 1 && t.tid == 0) oc_init_bars<M>(sm);
    // faces of the patch: west faces 4 x 5, south faces 5 x 4
    float kw[20], ks[20];
    {
        const float *Kw = A.Kw + base, *Ks = A.Ks + base;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 v = *reinterpret_cast<const float4*>(Kw + (size_t)(gy + j) * n + gx);
            kw[5 * j] = v.x; kw[5 * j + 1] = v.y; kw[5 * j + 2] = v.z; kw[5 * j + 3] = v.w;
            kw[5 * j + 4] = gx + 4 < n ? Kw[(size_t)(gy + j) * n + gx + 4] : A.E[(size_t)p * n + gy + j];
        }
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const float4 v = gy + j < n ? *reinterpret_cast<const float4*>(Ks + (size_t)(gy + j) * n + gx)
                                        : *reinterpret_cast<const float4*>(A.Nn + (size_t)p * n + gx);
            ks[4 * j] = v.x; ks[4 * j + 1] = v.y; ks[4 * j + 2] = v.z; ks[4 * j + 3] = v.w;
        }
    }
    float4* const P4 = reinterpret_cast<float4*>(sm + M::P4) + t.tid;
    {
        float4* q = reinterpret_cast<float4*>(sm + M::INVF) + t.tid;
        float inv[2][8];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                inv[(i + j) & 1][2 * j + (i >> 1)] = 1.f / ((kw[5 * j + i] + kw[5 * j + i + 1]) + (ks[4 * j + i] + ks[4 * j + 4 + i]));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            q[(2 * c) * OC_T] = make_float4(inv[c][0], inv[c][1], inv[c][2], inv[c][3]);
            q[(2 * c + 1) * OC_T] = make_float4(inv[c][4], inv[c][5], inv[c][6], inv[c][7]);
        }
    }
    {
        const Patch2 h = coarsen_f(kw, ks);
        float d[4];
        diag_h(h, d);
        reinterpret_cast<float4*>(sm + M::INVH)[t.tid] = make_float4(1.f / d[0], 1.f / d[1], 1.f / d[2], 1.f / d[3]);
        const Cell1 k = coarsen_h(h);
        oc_sync<C>();                                       // every block of the cluster runs: its shared memory may be written
        if (C == 1) {
            build_inv8<C>(sm, t, coarse_faces(k, t.lx, t.ly));
        } else {
            // gather the next level's faces in every block (through the inverse's storage): the block's part is formed
            // where p will be, 4 values of H / 2 x W / 2 cells
            constexpr int m = C * 8, part = (M::H / 2) * (M::W / 2), all = m * m;
            float* st = sm + M::P4;
            const float2 ws = make_float2(__shfl_xor_sync(0xffffffffu, k.s, 1) + k.s, __shfl_xor_sync(0xffffffffu, k.n, 1) + k.n);
            st[t.tid] = k.w; st[OC_T + t.tid] = k.e; st[2 * OC_T + t.tid] = ws.x; st[3 * OC_T + t.tid] = ws.y;
            __syncthreads();
            float* fb = sm + M::INV8;
            for (int i = t.tid; i < 4 * part; i += OC_T) {
                const int f = i / part, c = i % part, I = c % (M::W / 2), J = c / (M::W / 2);
                const float* q = st + f * OC_T + 2 * J * M::W + 2 * I;
                const float v = f == 0 ? q[0] + q[M::W] : f == 1 ? q[1] + q[M::W + 1] : f == 2 ? q[0] : q[M::W];
                for (int d0 = 0; d0 < M::CC; ++d0) oc_push(fb + f * all + (int)t.rank * part + c, (uint32_t)d0, v, all_bar<OcMem<C>>(sm, OC_GATHER));
            }
            all_sync(sm, t, OC_GATHER, all * 16);
            Cell1 k16;
            if (C == 4) {
                float* lf = sm + M::LF + t.tid;
                Patch2 l;
#pragma unroll
                for (int J = 0; J < 2; ++J) {
                    const int c = (2 * t.ly + J) * m + 2 * t.lx;
                    l.w[3 * J] = fb[c]; l.w[3 * J + 1] = fb[c + 1]; l.w[3 * J + 2] = fb[m * m + c + 1];
                    l.s[2 * J] = fb[2 * m * m + c]; l.s[2 * J + 1] = fb[2 * m * m + c + 1];
                    if (J == 1) { l.s[4] = fb[3 * m * m + c]; l.s[5] = fb[3 * m * m + c + 1]; }
                }
                diag_h(l, d);
#pragma unroll
                for (int q = 0; q < 6; ++q) { lf[q * OC_T] = l.w[q]; lf[(6 + q) * OC_T] = l.s[q]; }
#pragma unroll
                for (int q = 0; q < 4; ++q) lf[(12 + q) * OC_T] = 1.f / d[q];
                k16 = coarsen_h(l);
            } else {
                k16 = Cell1{fb[t.tid], fb[m * m + t.tid], fb[2 * m * m + t.tid], fb[3 * m * m + t.tid]};
            }
            float* sf = sm + M::SF + t.tid;
            sf[0] = k16.w; sf[OC_T] = k16.e; sf[2 * OC_T] = k16.s; sf[3 * OC_T] = k16.n;
            const Cell1 k8 = coarse_faces(k16, t.lx, t.ly);
            __syncthreads();
            if (V && !A.build) {
                const float4* g = reinterpret_cast<const float4*>(A.inv8 + (size_t)p * 4096);
                for (int i = t.tid; i < 1024; i += OC_T) reinterpret_cast<float4*>(sm + M::INV8)[i] = g[i];
                __syncthreads();
            } else {
                build_inv8<C>(sm, t, k8);
            }
        }
    }
    if (V && A.build) {
        if (t.rank == 0)
            for (int i = t.tid; i < 4096; i += OC_T) A.inv8[(size_t)p * 4096 + i] = sm[M::INV8 + i];
        oc_leave(t, A.err);
        return;
    }
    // r = scaled b
    const float2* B = V ? nullptr : A.bdf + (size_t)p * A.bstride;
    float r[16], e[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (V) {
            const float4 v = *reinterpret_cast<const float4*>(A.vr + base + (size_t)(gy + j) * n + gx);
            r[4 * j] = v.x; r[4 * j + 1] = v.y; r[4 * j + 2] = v.z; r[4 * j + 3] = v.w;
            continue;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 v = B[(size_t)(gy + j) * n + gx + i];
            r[4 * j + i] = __fadd_rn(v.x, v.y) * scale;
        }
    }
    const size_t pb = (size_t)blockIdx.x * 4 * OC_T + t.tid;   // this thread's patch rows in x, wh, wm, wl
    int iters = 0, phases = 0, inner = 0;
    bool converged = false, wset = false, dead = false;
#pragma unroll 1
    for (int o = 0; o < A.max_outer; ++o) {
        // ---- CG on A x = r from x = 0 ----
        df32 thr{0.f, 0.f}, rz{0.f, 0.f};
        bool first = true;
        for (;;) {
            float s = 0.f;
            if (!V) {
#pragma unroll
                for (int c = 0; c < 16; ++c) s = fmaf(r[c], r[c], s);
                red_put<C>(sm, t, 0, s);
            }
            sweep_f<C, 0>(sm, t, kw, ks, r, e, true);
            pub_f<C, 0>(sm, t, e);
            if (V) {
                nb_sync(sm, t, 8 * M::W);
            } else {
                dead = rr_sync<C>(sm, t);
                if (dead) break;
                const df32 rr = red_get<C>(sm, t, 0);
                if (first) {
                    const df32 part = df_mul(df32{A.tol2.x, A.tol2.y}, rr), least{sm[M::THR], sm[M::THR + 1]};
                    thr = at_most(part, least) ? least : part;
                    if (!(rr.hi > 0.f)) break;
                    ++inner;
                } else {
                    ++iters;
                    if (at_most(rr, thr) || iters >= A.maxit || !(rr.hi == rr.hi)) break;
                }
            }
            // V-cycle: z = M r in e
#pragma unroll 1
            for (int sw = 0; sw < A.nu_f; ++sw) {
                if (sw > 0) {
                    sweep_f<C, 0>(sm, t, kw, ks, r, e, false);
                    pub_f<C, 0>(sm, t, e);
                    nb_sync(sm, t, 8 * M::W);
                }
                sweep_f<C, 1>(sm, t, kw, ks, r, e, false);
                pub_f<C, 1>(sm, t, e);
                nb_sync(sm, t, 8 * M::W);
            }
            float rh[4], eh[4];
            {
                const HaloF h = halo_f<C>(sm, t, 1);
                float res[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = j & 1; i < 4; i += 2) {
                        OC_NB_F(i, j, e, h, ew, ee, es, en)
                        const float ec = e[4 * j + i];
                        const float q = fmaf(kw[5 * j + i], ec - ew, fmaf(kw[5 * j + i + 1], ec - ee, fmaf(ks[4 * j + i], ec - es, ks[4 * j + 4 + i] * (ec - en))));
                        res[2 * (j >> 1) + (i >> 1)] += r[4 * j + i] - q;
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c) rh[c] = res[c];
            }
            const float4 invh = reinterpret_cast<const float4*>(sm + M::INVH)[t.tid];
            float rq, eq;
            {
                const Patch2 h = coarsen_f(kw, ks);
                rq = pre_h<C, true>(sm, sm + M::HP, t, A.nu_c, h, invh, rh, eh);
                const Cell1 k = coarsen_h(h);
                const float invq = 1.f / ((k.w + k.e) + (k.s + k.n));
                float* QP = sm + M::QP;
                if (C == 1) {
                    level16<C, true>(sm, QP, t, A.nu_c, A.cc, k, invq, rq, eq);
                } else {
                    // the coarse right-hand side: pair sums per thread row, then four values per thread to one block each
                    float rc = pre_q<C, true>(sm, QP, t, A.nu_c, k, invq, rq, eq);
                    rc += __shfl_xor_sync(0xffffffffu, rc, 1);
                    if ((t.tx & 1) == 0) sm[M::STG + t.ty * (M::W / 2) + (t.tx >> 1)] = rc;
                    __syncthreads();
                    constexpr int m = C * 8, part = (M::H / 2) * (M::W / 2);
                    if (t.tid < M::CC * part / 4) {
                        const int c = 4 * (t.tid % (part / 4)), J = c / (M::W / 2), I = c % (M::W / 2);
                        const float4 u = *reinterpret_cast<const float4*>(sm + M::STG + 2 * J * (M::W / 2) + I);
                        const float4 v = *reinterpret_cast<const float4*>(sm + M::STG + (2 * J + 1) * (M::W / 2) + I);
                        oc_push4(sm + M::RB + (int)t.rank * part + c, (uint32_t)(t.tid / (part / 4)),
                                 make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w), all_bar<OcMem<C>>(sm, OC_GATHER));
                    }
                    all_sync(sm, t, OC_GATHER, m * m * 4);
                    const int px = t.tx >> 1, py = (int)t.rank * (M::H / 2) + (t.ty >> 1);   // the parent on the gathered level
                    const float* sf = sm + M::SF + t.tid;
                    const Cell1 k16{sf[0], sf[OC_T], sf[2 * OC_T], sf[3 * OC_T]};
                    const float inv16 = 1.f / ((k16.w + k16.e) + (k16.s + k16.n));
                    float e16, ep;
                    if (C == 4) {
                        const float* lf = sm + M::LF + t.tid;
                        Patch2 l;
#pragma unroll
                        for (int q = 0; q < 6; ++q) { l.w[q] = lf[q * OC_T]; l.s[q] = lf[(6 + q) * OC_T]; }
                        const float4 invl = make_float4(lf[12 * OC_T], lf[13 * OC_T], lf[14 * OC_T], lf[15 * OC_T]);
                        const float* rb = sm + M::RB + 2 * t.ly * m + 2 * t.lx;
                        const float rl[4] = {rb[0], rb[1], rb[m], rb[m + 1]};
                        float el[4];
                        float* LP = sm + M::LP;
                        const float r16 = pre_h<C, false>(sm, LP, t, A.nu_c, l, invl, rl, el);
                        level16<C, false>(sm, sm + M::SP, t, A.nu_c, A.cc, k16, inv16, r16, e16);
#pragma unroll
                        for (int c = 0; c < 4; ++c) el[c] = fmaf(A.cc, e16, el[c]);
                        post_h<C, false>(sm, LP, t, A.nu_c, l, invl, rl, el);
                        pub_h<C, false>(LP, t, 0, el);
                        __syncthreads();
                        ep = LP[((px & 1) + 2 * (py & 1)) * 324 + ((py >> 1) + 1) * 18 + (px >> 1) + 1];
                    } else {
                        float* SPl = sm + M::SP;
                        level16<C, false>(sm, SPl, t, A.nu_c, A.cc, k16, inv16, sm[M::RB + t.tid], e16);
                        if (((t.lx + t.ly) & 1) == 0) SPl[(t.ly + 1) * 18 + t.lx + 1] = e16;
                        __syncthreads();
                        ep = SPl[(py + 1) * 18 + px + 1];
                    }
                    eq = fmaf(A.cc, ep, eq);
                    post_q<C, true>(sm, QP, t, A.nu_c, k, invq, rq, eq);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) eh[c] = fmaf(A.cc, eq, eh[c]);
                post_h<C, true>(sm, sm + M::HP, t, A.nu_c, h, invh, rh, eh);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) e[4 * j + i] = fmaf(A.cc, eh[2 * (j >> 1) + (i >> 1)], e[4 * j + i]);
#pragma unroll 1
            for (int sw = 0; sw < A.nu_f; ++sw) {
                pub_f<C, 0>(sm, t, e);
                nb_sync(sm, t, 8 * M::W);
                sweep_f<C, 1>(sm, t, kw, ks, r, e, false);
                pub_f<C, 1>(sm, t, e);
                nb_sync(sm, t, 8 * M::W);
                sweep_f<C, 0>(sm, t, kw, ks, r, e, false);
            }
            if (V) break;
            // beta, p = z + beta p
            s = 0.f;
#pragma unroll
            for (int c = 0; c < 16; ++c) s = fmaf(r[c], e[c], s);
            red_put<C>(sm, t, OC_RZ, s);
            all_sync(sm, t, OC_RZ, 64 * M::CC);
            const df32 rzn = red_get<C>(sm, t, 1);
            if (!first) {
                const float beta = quotient(rzn, rz);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 v = P4[j * OC_T];
                    e[4 * j] = fmaf(beta, v.x, e[4 * j]);
                    e[4 * j + 1] = fmaf(beta, v.y, e[4 * j + 1]);
                    e[4 * j + 2] = fmaf(beta, v.z, e[4 * j + 2]);
                    e[4 * j + 3] = fmaf(beta, v.w, e[4 * j + 3]);
                }
            }
            rz = rzn;
#pragma unroll
            for (int j = 0; j < 4; ++j) P4[j * OC_T] = make_float4(e[4 * j], e[4 * j + 1], e[4 * j + 2], e[4 * j + 3]);
            pub_f<C, 0>(sm, t, e);
            pub_f<C, 1>(sm, t, e);
            nb_sync(sm, t, 16 * M::W);
            // q = A p in flux form, p.q
            float q[16];
            s = 0.f;
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                const HaloF h = halo_f<C>(sm, t, 1 - col);
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = (j + col) & 1; i < 4; i += 2) {
                        OC_NB_F(i, j, e, h, ew, ee, es, en)
                        const float ec = e[4 * j + i];
                        const float v = fmaf(kw[5 * j + i], ec - ew, fmaf(kw[5 * j + i + 1], ec - ee, fmaf(ks[4 * j + i], ec - es, ks[4 * j + 4 + i] * (ec - en))));
                        q[4 * j + i] = v;
                        s = fmaf(ec, v, s);
                    }
            }
            red_put<C>(sm, t, 2, s);
            float4 xv[4];
            if (!first) {
#pragma unroll
                for (int j = 0; j < 4; ++j) xv[j] = A.x[pb + j * OC_T];
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) xv[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            all_sync(sm, t, OC_PQ, 64 * M::CC);
            const df32 pq = red_get<C>(sm, t, 2);
            const float alpha = pq.hi > 0.f ? quotient(rz, pq) : 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                xv[j].x = fmaf(alpha, e[4 * j], xv[j].x);
                xv[j].y = fmaf(alpha, e[4 * j + 1], xv[j].y);
                xv[j].z = fmaf(alpha, e[4 * j + 2], xv[j].z);
                xv[j].w = fmaf(alpha, e[4 * j + 3], xv[j].w);
                A.x[pb + j * OC_T] = xv[j];
            }
#pragma unroll
            for (int c = 0; c < 16; ++c) r[c] = fmaf(-alpha, q[c], r[c]);
            first = false;
        }
        if (V) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4*>(A.ve + base + (size_t)(gy + j) * n + gx) = make_float4(e[4 * j], e[4 * j + 1], e[4 * j + 2], e[4 * j + 3]);
            break;
        }
        if (dead) break;
        // ---- w += x; FP64-accurate residual ----
        ++phases;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const size_t at = pb + j * OC_T;
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f), m = h, l = h, x = h;
            if (wset) { h = A.wh[at]; m = A.wm[at]; l = A.wl[at]; }
            if (!first) x = A.x[at];
            tri_add(h.x, m.x, l.x, x.x);
            tri_add(h.y, m.y, l.y, x.y);
            tri_add(h.z, m.z, l.z, x.z);
            tri_add(h.w, m.w, l.w, x.w);
            A.wh[at] = h; A.wm[at] = m; A.wl[at] = l;
        }
        wset = true;
        w_sync<C>(sm, t);
        float s = 0.f;
        {
            const float *Kwl = A.Kwl + base, *Ksl = A.Ksl + base;
            const float* W3[3] = {reinterpret_cast<const float*>(A.wh), reinterpret_cast<const float*>(A.wm), reinterpret_cast<const float*>(A.wl)};
            // patch rows of the neighbouring threads (another block of the cluster at the tile's edge)
            const size_t blk = 4 * OC_T;
            const size_t pw = pb - 1, pe = pb + 1;
            const size_t ps = t.ty > 0 ? pb - M::W : pb - blk + (M::H - 1) * M::W;
            const size_t pn = t.ty < M::H - 1 ? pb + M::W : pb + blk - (M::H - 1) * M::W;
            const bool hw = gx > 0, he = gx + 4 < n, hs = gy > 0, hn = gy + 4 < n;
            float c3[3][4], f3[3][4];                           // this row, the row above or below
            df32 fs[4];
            auto row = [&](size_t at, float (&v)[3][4]) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float4 a = __ldcg(reinterpret_cast<const float4*>(W3[q]) + at);
                    v[q][0] = a.x; v[q][1] = a.y; v[q][2] = a.z; v[q][3] = a.w;
                }
            };
            auto zero = [](float (&v)[3][4]) {
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[q][i] = 0.f;
            };
            row(pb, c3);
            if (hs) row(ps + 3 * OC_T, f3); else zero(f3);
            {
                const float4 kl = *reinterpret_cast<const float4*>(Ksl + (size_t)gy * n + gx);
                const float k4[4] = {kl.x, kl.y, kl.z, kl.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    fs[i] = tri_flux(ks[i], k4[i], c3[0][i], c3[1][i], c3[2][i], f3[0][i], f3[1][i], f3[2][i]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j < 3) row(pb + (j + 1) * OC_T, f3);
                else if (hn) row(pn, f3);
                else zero(f3);
                const float4 kn = (j < 3 || hn) ? *reinterpret_cast<const float4*>(Ksl + (size_t)(gy + j + 1) * n + gx)
                                                : *reinterpret_cast<const float4*>(A.Nl + (size_t)p * n + gx);
                const float4 kv = *reinterpret_cast<const float4*>(Kwl + (size_t)(gy + j) * n + gx);
                const float ke = he ? Kwl[(size_t)(gy + j) * n + gx + 4] : A.El[(size_t)p * n + gy + j];
                const float kwl[5] = {kv.x, kv.y, kv.z, kv.w, ke}, ksl[4] = {kn.x, kn.y, kn.z, kn.w};
                float wv[3] = {0.f, 0.f, 0.f}, ev[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (hw) wv[q] = __ldcg(W3[q] + 4 * (pw + j * OC_T) + 3);
                    if (he) ev[q] = __ldcg(W3[q] + 4 * (pe + j * OC_T));
                }
                df32 fw = tri_flux(kw[5 * j], kwl[0], c3[0][0], c3[1][0], c3[2][0], wv[0], wv[1], wv[2]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int i1 = (i + 1) & 3;
                    const df32 fe = i < 3 ? tri_flux(kw[5 * j + i + 1], kwl[i + 1], c3[0][i1], c3[1][i1], c3[2][i1], c3[0][i], c3[1][i], c3[2][i])
                                          : tri_flux(kw[5 * j + 4], kwl[4], ev[0], ev[1], ev[2], c3[0][3], c3[1][3], c3[2][3]);
                    const df32 fn = tri_flux(ks[4 * j + 4 + i], ksl[i], f3[0][i], f3[1][i], f3[2][i], c3[0][i], c3[1][i], c3[2][i]);
                    const float2 bv = B[(size_t)(gy + j) * n + gx + i];
                    df32 rs{bv.x * scale, bv.y * scale};
                    acc_add(rs, -fw.hi, -fw.lo);
                    acc_add(rs, fe.hi, fe.lo);
                    acc_add(rs, -fs[i].hi, -fs[i].lo);
                    acc_add(rs, fn.hi, fn.lo);
                    const float v = __fadd_rn(rs.hi, rs.lo);
                    r[4 * j + i] = v;
                    s = fmaf(v, v, s);
                    fw = fe;
                    fs[i] = fn;
                }
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int i = 0; i < 4; ++i) c3[q][i] = f3[q][i];
            }
        }
        red_put<C>(sm, t, OC_RZ, s);
        all_sync(sm, t, OC_RZ, 64 * M::CC);
        if (C > 1 && __syncthreads_or(t.dead)) break;
        if (at_most(red_get<C>(sm, t, OC_RZ), df32{sm[M::THR + 2], sm[M::THR + 3]})) { converged = true; break; }
    }
#pragma unroll 1
    for (int j = 0; !V && j < 4; ++j) {
        const size_t at = pb + j * OC_T;
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f), m = h, l = h;
        if (wset) { h = A.wh[at]; m = A.wm[at]; l = A.wl[at]; }
        double2* o = reinterpret_cast<double2*>(A.W + base + (size_t)(gy + j) * n + gx);
        o[0] = make_double2(tri_to_double(h.x, m.x, l.x, -sexp), tri_to_double(h.y, m.y, l.y, -sexp));
        o[1] = make_double2(tri_to_double(h.z, m.z, l.z, -sexp), tri_to_double(h.w, m.w, l.w, -sexp));
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

template <int C, bool V>
static void oc_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int count, cudaStream_t st) {
    check(cudaFuncSetAttribute(k_onchip<C, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OcMem<C>::BYTES), "attr");
    if (C == 4) check(cudaFuncSetAttribute(k_onchip<C, V>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1), "attr");
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(count * C * C));
    cfg.blockDim = dim3(OC_T);
    cfg.dynamicSmemBytes = OcMem<C>::BYTES;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C * C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
}

template <int C, bool V>
static bool oc_fits() {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    oc_config<C, V>(cfg, attr, 1, nullptr);
    int nc = 0;
    if (C == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nc, k_onchip<C, V>, OC_T, OcMem<C>::BYTES) != cudaSuccess) nc = 0;
    } else if (cudaOccupancyMaxActiveClusters(&nc, k_onchip<C, V>, &cfg) != cudaSuccess) {
        nc = 0;
    }
    (void)cudaGetLastError();
    return nc > 0;
}

// Whether the context's solves run on chip: the default tile kernels and, in mixed precision (onchip64.cu: FP64), a grid of 64,
// 128 or 256 cells per side (a 512^2 strip would not fit a cluster of 16; at each of the three this is
// the faster solver from 2 particles to thousands), and clusters of that size on this device.
bool onchip_supported(const Ctx& c) {
    if (c.dim != 2 || c.cfg.tile_kernel != 0) return false;
    if (!mixed_precision(c.cfg)) return onchip64_supported(c);
    if (c.n == 64) return oc_fits<1, false>();
    if (c.n == 128) return oc_fits<2, false>();
    if (c.n == 256) return oc_fits<4, false>();
    return false;
}

// Whether the mixed-precision multi-pass solver of a larger grid (512^2) runs its levels from 128^2 down on chip: per V-cycle
// of 250 particles 126 us in five launches, which smooth 2.25 times the cells they own, and 50 in one.  Not from 256^2
// down: 14 clusters of 16 at a time would take longer (about 430 us) than its two passes and this (310).
static bool onchip32_vcycle_supported(const Ctx& c) { return c.n > 256 && oc_fits<2, true>(); }

// Whether the passes of a larger grid's solver leave the levels from 128^2 down to launch_vcycle.
bool vcycle_supported(const Ctx& c) {
    if (c.dim != 2 || c.cfg.tile_kernel != 0 || c.onchip) return false;
    return mixed_precision(c.cfg) ? onchip32_vcycle_supported(c) : onchip64_vcycle_supported(c);
}

template <int C, bool V>
static void oc_launch(Ctx& c, const OcArgs& A, int count) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    oc_config<C, V>(cfg, attr, count, c.stream);
    check(cudaLaunchKernelEx(&cfg, k_onchip<C, V>, A), "on-chip solve"); ++c.pc.launches;
}

static void solve_batch_onchip32(Ctx& c, int count, const Rhs& R, double* W) {
    InnerSolver<float>& s = c.s32;
    LevelArrays<float>& f = s.lv[0];
    OcArgs A{};
    A.max_outer = c.cfg.max_refine; A.maxit = c.cfg.max_iter; A.nu_f = c.cfg.fine_sweeps; A.nu_c = c.cfg.smooth_sweeps;
    A.cc = (float)c.cfg.coarse_scale;
    A.tol2 = pair_of(c.cfg.tol_inner * c.cfg.tol_inner);
    A.tolout2 = c.cfg.tol_outer * c.cfg.tol_outer;
    A.floor2 = 0.25 * A.tolout2;   // no phase need reduce |r| below half the final tolerance
    A.b2const = R.b2const; A.b2pp = R.b2pp;
    A.Kw = f.Kw; A.Ks = f.Ks; A.E = f.E; A.Nn = f.Nn;
    A.Kwl = c.Kwlo; A.Ksl = c.Kslo; A.El = c.Elo; A.Nl = c.Nlo;
    A.bdf = R.bdf; A.bstride = R.stride;
    A.x = reinterpret_cast<float4*>(s.x); A.wh = reinterpret_cast<float4*>(s.p[0]);
    A.wm = reinterpret_cast<float4*>(s.p[1]); A.wl = reinterpret_cast<float4*>(s.q);
    A.W = W;
    A.badp = c.lenient ? c.badp : nullptr;
    A.cnt = c.gcnt;
    A.err = c.dev_err;
    if (c.n == 64) oc_launch<1, false>(c, A, count);
    else if (c.n == 128) oc_launch<2, false>(c, A, count);
    else oc_launch<4, false>(c, A, count);
}

// The V-cycle from the level of 128^2 down (r to e2 there) for the active particles; with `build` the dense
// inverses of the 8^2 level that it uses, for the first `nact` particles.
static void vcycle32(Ctx& c, int level, int nact, bool build) {
    InnerSolver<float>& s = c.s32;
    LevelArrays<float>& f = s.lv[level];
    OcArgs A{};
    A.max_outer = 1; A.nu_f = A.nu_c = c.cfg.smooth_sweeps;
    A.cc = (float)c.cfg.coarse_scale;
    A.Kw = f.Kw; A.Ks = f.Ks; A.E = f.E; A.Nn = f.Nn;
    A.vr = f.r; A.ve = f.e2; A.inv8 = s.binv;
    A.build = build;
    if (!build) {
        A.list = s.list;
        A.nact = c.graph ? s.nact : nullptr;
    }
    A.err = c.dev_err;
    oc_launch<2, true>(c, A, nact);
}
void launch_vcycle(Ctx& c, InnerSolver<float>&, int level, int nact) { vcycle32(c, level, nact, false); }
void launch_vcycle(Ctx& c, InnerSolver<double>&, int level, int nact) { launch_vcycle64(c, level, nact); }
// At set-up, after the coarser levels: the dense inverses of the on-chip solvers' smallest level.
void launch_dense_inverses(Ctx& c, InnerSolver<double>&, int count) {
    if (c.onchip || c.vchip) launch_inv4(c, count);
}
void launch_dense_inverses(Ctx& c, InnerSolver<float>& s, int count) {
    int l = 0;
    while (s.lv[l].n > 128) ++l;
    if (c.vchip) vcycle32(c, l, count, true);
}

// Solves a batch into W; the counters accumulate in c.gcnt (OnchipCounters reads them).
void solve_batch_onchip(Ctx& c, int count, const Rhs& R, double* W) {
    const bool mixed = mixed_precision(c.cfg);
    if (c.prof) check(cudaEventRecord(c.ev0, c.stream), "event");
    if (mixed) solve_batch_onchip32(c, count, R, W);
    else solve_batch_onchip64(c, count, R, W);
    if (c.prof) {   // profiling: this kernel is the dominant one (faces in, as two parts or with 1/D and the coarser levels; w out)
        check(cudaEventRecord(c.ev1, c.stream), "event");
        check(cudaEventSynchronize(c.ev1), "event wait");
        float ms = 0.f;
        check(cudaEventElapsedTime(&ms, c.ev0, c.ev1), "event time");
        c.pc.dom_ms += ms;
        c.pc.dom_launches += 1;
        c.pc.dom_particles += count;
        c.pc.dom_bytes += (mixed ? 24.0 : 40.0) * c.n * c.n * count;
    }
}

}  // namespace smcgm
