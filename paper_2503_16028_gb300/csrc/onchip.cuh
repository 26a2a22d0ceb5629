// Exchanges between the blocks of a cluster that share a particle (the on-chip solvers): positions, remote
// stores counted by mbarriers, bounded waits.  M: the kernel's shared-memory layout (C, CC blocks, W x H threads,
// BARS: offset in bytes of its mbarriers).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace smcgm {

__device__ __forceinline__ uint32_t oc_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Barrier of the cluster (of the block when it is alone), ordering shared, distributed shared and
// global memory among its threads.
template <int C>
__device__ __forceinline__ void oc_sync() {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}
// The address of a shared-memory location of this block in block `rank` of the cluster.
__device__ __forceinline__ uint32_t oc_map(const void* p, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// Asynchronous stores into another block; the receiver's mbarrier counts their bytes, so an
// exchange needs neither a cluster barrier nor the memory fence that one implies (the fence's
// wait was the largest stall of the cluster form: 2048 solves at 256^2 took 62 ms with cluster barriers,
// 53 with these).
__device__ __forceinline__ void oc_push(void* p, uint32_t rank, float v, const void* bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(oc_map(p, rank)), "f"(v),
                 "r"(oc_map(bar, rank))
                 : "memory");
}
__device__ __forceinline__ void oc_push4(void* p, uint32_t rank, float4 v, const void* bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(oc_map(p, rank)),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(oc_map(bar, rank))
                 : "memory");
}
// The same with the addresses already those of the other block.
__device__ __forceinline__ void oc_store(uint32_t dst, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(dst), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void oc_store2(uint32_t dst, float2 v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(dst), "f"(v.x), "f"(v.y), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void oc_store(uint32_t dst, double v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(dst), "d"(v), "r"(bar) : "memory");
}

// Where a thread stands.
template <class M>
struct OcPos {
    int tid, tx, ty;         // in the block's W x H threads
    int lx, ly;              // in the threads of the local levels
    uint32_t rank;
    // Exchanges (C > 1).  Edge exchanges go pairwise between the first (last) thread row of a block and the last
    // (first) of the block below (above), through two mbarriers per side that alternate: a neighbour's edge can be
    // at most one exchange ahead, since it needs this edge's values to go on.  The all-to-all exchanges have one
    // mbarrier each: a block can be at most one all-to-all exchange ahead of any other.
    unsigned seq, par;
    bool dead;               // a wait of this thread ran out: it waits for nothing and arms no mbarrier any more
    uint32_t nbase;          // shared-memory base of the neighbouring block, for the threads of an edge row; else 0
    bool lower;              // of an edge row: the lower one (neighbour below)
};
enum OcAll { OC_RR = 0, OC_RZ = 1, OC_PQ = 2, OC_GATHER = 3 };
// Bound of a wait, in nanoseconds, after OC_POLLS tries (a build with another bound makes waits run out for a test).
#ifndef OC_WAIT_NS
#define OC_WAIT_NS 2000000000u
#endif
constexpr int OC_POLLS = 256;
// What a store under way between two blocks of a cluster takes to land, with a wide margin (it takes about a microsecond).
constexpr unsigned OC_DRAIN_NS = 200000u;

__device__ __forceinline__ unsigned oc_ns() {
    unsigned v;
    asm volatile("mov.u32 %0, %%globaltimer_lo;" : "=r"(v));
    return v;
}

// Offset (bytes) of the mbarrier of the current edge exchange in the receiving block: `below` for values that
// come from the block below it.
template <class M>
__device__ __forceinline__ int nb_bar(const OcPos<M>& t, bool below) { return M::BARS + 16 * (below ? 1 : 0) + 8 * (t.seq & 1); }
template <class M>
__device__ __forceinline__ char* all_bar(void* sm, int which) { return reinterpret_cast<char*>(sm) + M::BARS + 32 + 8 * which; }
// Arms an mbarrier for `bytes`; by the thread that also waits on it, so that none is armed twice in a phase.
template <class M>
__device__ __forceinline__ void oc_expect(const OcPos<M>& t, const void* bar, int bytes) {
    if (!t.dead)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(bytes) : "memory");
}
// Waits for a phase of an mbarrier, at most OC_WAIT_NS; the thread is dead afterwards if that ran out.
template <class M>
__device__ __forceinline__ void oc_wait(OcPos<M>& t, const void* bar, unsigned parity) {
    if (t.dead) return;
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
    uint32_t ok = 0;
    unsigned since = 0;
#pragma unroll 1
    for (int k = 0;; ++k) {
        asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}"
                     : "=r"(ok)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (ok) return;
        if (k == OC_POLLS) since = oc_ns();
        if (k > OC_POLLS && oc_ns() - since >= OC_WAIT_NS) break;
    }
    t.dead = true;
}
// The edge rows' part of an exchange: waits for the neighbour's values (`bytes` for the whole row).
template <class M>
__device__ __forceinline__ void nb_wait(void* sm, OcPos<M>& t, int bytes) {
    if (M::C > 1) {
        if (t.nbase) {
            const char* bar = reinterpret_cast<const char*>(sm) + nb_bar(t, t.lower);
            if (t.tx == 0) oc_expect(t, bar, bytes);
            oc_wait(t, bar, (t.seq >> 1) & 1);
        }
        ++t.seq;
    }
}
// After the stores of an edge exchange: the block's own are visible, and to the edge rows the neighbours'.
template <class M>
__device__ __forceinline__ void nb_sync(void* sm, OcPos<M>& t, int bytes) {
    __syncthreads();
    nb_wait(sm, t, bytes);
}
// The same for an all-to-all exchange (`bytes` from all blocks together).
template <class M>
__device__ __forceinline__ void all_sync(void* sm, OcPos<M>& t, int which, int bytes) {
    if (M::C > 1 && t.tid == 0) oc_expect(t, all_bar<M>(sm, which), bytes);
    __syncthreads();
    if (M::C > 1) {
        oc_wait(t, all_bar<M>(sm, which), (t.par >> which) & 1);
        t.par ^= 1u << which;
    }
}
// The last thing a block of a cluster does.  A block that leaves must have no store of another under way into its shared
// memory.  Every block comes here once, and between the barrier of its set-up and this one there is no other
// cluster barrier, so no block passes before all have issued their last store, whatever waits ran out where; the stores
// of an exchange that was waited for have landed, and after a wait that ran out (*err, written before the barrier)
// the first thread, which keeps its block, waits for the others to land.
template <class M>
__device__ __forceinline__ void oc_leave(const OcPos<M>& t, int* err) {
    if (M::C == 1) return;
    if (t.dead) atomicExch(err, 1);
    oc_sync<M::C>();
    if (t.tid == 0 && __ldcg(err)) {
        const unsigned since = oc_ns();
        while (oc_ns() - since < OC_DRAIN_NS) {}
    }
}
// The mbarriers of a block, initialised by one thread before the cluster's first barrier.
template <class M>
__device__ __forceinline__ void oc_init_bars(void* sm) {
    for (int k = 0; k < 8; ++k)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(reinterpret_cast<char*>(sm) + M::BARS + 8 * k)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// The thread's place: rank, row and neighbour.
template <class M>
__device__ __forceinline__ void oc_place(OcPos<M>& t, void* sm, int tx, int ty) {
    t.tid = threadIdx.x;
    t.tx = tx;
    t.ty = ty;
    t.rank = M::C == 1 ? 0u : oc_rank();
    t.seq = 0;
    t.par = 0;
    t.dead = false;
    t.nbase = 0;
    t.lower = t.ty == 0;
    if (M::C > 1) {
        if (t.ty == 0 && t.rank > 0) t.nbase = oc_map(sm, t.rank - 1);
        if (t.ty == M::H - 1 && (int)t.rank < M::CC - 1) t.nbase = oc_map(sm, t.rank + 1);
    }
}

}  // namespace smcgm
