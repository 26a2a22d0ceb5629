// The exchange helpers of the on-chip solvers (csrc/onchip.cuh) in a small kernel of their own: clusters of
// four blocks trade edge rows and sums for some rounds.  With `drop` one block leaves out one word of one edge row, as
// a lost message would: the receiver's wait runs out and it leaves after that round's sum, which the others have in
// full; their waits of the next round run out, and the kernel ends with its error flag set.  (An edge
// row, whose mbarriers no later round reaches without the receiver: the sums' one would count the next round's words.)
#include <cstdio>
#include <cuda_runtime.h>
#define OC_WAIT_NS 20000000u
#include "../paper_2503_16028_gb300/csrc/onchip.cuh"

using namespace smcgm;

struct Mem {
    static constexpr int C = 2, CC = 4, W = 32, H = 8, T = W * H;
    static constexpr int ROW = 0, SUM = 2 * W, END = SUM + CC + 4, BARS = 4 * END;   // floats; bytes
};
constexpr int ROUNDS = 16, DROP_ROUND = 5;

__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(Mem::T) k_rounds(int drop, int* done, float* total, int* err) {
    __shared__ __align__(16) float sm[Mem::END + 16];
    OcPos<Mem> t;
    oc_place(t, sm, (int)threadIdx.x % Mem::W, (int)threadIdx.x / Mem::W);
    for (int i = t.tid; i < Mem::END; i += Mem::T) sm[i] = 0.f;
    if (t.tid == 0) oc_init_bars<Mem>(sm);
    oc_sync<2>();
    int rounds = 0;
    float sum = 0.f;
    for (; rounds < ROUNDS; ++rounds) {
        const bool lost = drop && t.rank == 1 && t.lower && t.tx == 0 && rounds == DROP_ROUND;
        if (t.nbase && !lost) oc_store(t.nbase + 4 * (Mem::ROW + (t.lower ? Mem::W : 0) + t.tx), (float)(t.rank + 1), t.nbase + nb_bar(t, !t.lower));
        nb_sync(sm, t, 4 * Mem::W);
        if (t.tid < Mem::CC)
            oc_push(&sm[Mem::SUM + t.rank], (uint32_t)t.tid, (float)(t.rank + rounds), all_bar<Mem>(sm, OC_RR));
        all_sync(sm, t, OC_RR, 4 * Mem::CC);
        if (__syncthreads_or(t.dead)) break;
        for (int d = 0; d < Mem::CC; ++d) sum += sm[Mem::SUM + d];
        __syncthreads();
    }
    if (t.tid == 0) { done[blockIdx.x] = rounds; total[blockIdx.x] = sum; }
    oc_leave(t, err);
}

int main() {
    constexpr int CLUSTERS = 3, G = 4 * CLUSTERS;
    int *done, *err, h[G], e = -1;
    float *total, ht[G];
    if (cudaMalloc(&done, sizeof(h)) || cudaMalloc(&total, sizeof(ht)) || cudaMalloc(&err, sizeof(int))) return 2;
    for (int drop = 0; drop < 2; ++drop) {
        cudaMemset(err, 0, sizeof(int));
        cudaMemset(done, 0xff, sizeof(h));
        k_rounds<<<G, Mem::T>>>(drop, done, total, err);
        const cudaError_t rc = cudaDeviceSynchronize();
        cudaMemcpy(h, done, sizeof(h), cudaMemcpyDeviceToHost);
        cudaMemcpy(ht, total, sizeof(ht), cudaMemcpyDeviceToHost);
        cudaMemcpy(&e, err, sizeof(int), cudaMemcpyDeviceToHost);
        bool ok = rc == cudaSuccess && e == drop;
        for (int b = 0; b < G; ++b) {
            // sum over the rounds of (0 + 1 + 2 + 3) + 4 round
            const int r = !drop ? ROUNDS : b % 4 == 0 ? DROP_ROUND : DROP_ROUND + 1;
            ok = ok && h[b] == r && ht[b] == (float)(6 * r + 2 * r * (r - 1));
        }
        printf("drop %d: %s, error flag %d, rounds %d %d %d %d\n", drop, cudaGetErrorString(rc), e, h[0], h[1], h[2], h[3]);
        if (!ok) return 1;
    }
    printf("cluster exit ok\n");
    return 0;
}
