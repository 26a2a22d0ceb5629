// The resampling kernel when its blocks never all meet: the barrier's counter starts three short of zero, so the first
// barrier is passed at once (the count reads as huge) and the second one is never reached.  The kernel
// has to end by itself with the error flag set and no index of an earlier call left.
#include <cstdio>
#include <vector>
#define GRID_WAIT_NS 20000000u
#include "../paper_2503_16028_gb300/csrc/smc.cu"

using namespace smcgm;

int main() {
    int N = 500;                                             // two blocks, the second one in part
    double *logw, *part;
    unsigned long long *cdf, u48 = 1ull << 47;     // half a step: no index depends on how the rounded weights add up
    int *idx, *flags;                                        // flags: the barrier's counter, the error flag
    if (cudaMalloc(&logw, N * sizeof(double)) || cudaMalloc(&part, smc_partial_doubles() * sizeof(double)) ||
        cudaMalloc(&cdf, N * sizeof(*cdf)) || cudaMalloc(&idx, 512 * sizeof(int)) || cudaMalloc(&flags, 2 * sizeof(int))) return 2;
    cudaMemset(logw, 0, N * sizeof(double));
    for (int run = 0; run < 2; ++run) {
        const int start[2] = {run ? -3 : 0, 0};
        cudaMemcpy(flags, start, sizeof(start), cudaMemcpyHostToDevice);
        cudaMemset(idx, 0x11, 512 * sizeof(int));
        unsigned* bar = reinterpret_cast<unsigned*>(flags);
        int* err = flags + 1;
        void* args[] = {&N, &logw, &u48, &cdf, &idx, &part, &bar, &err};
        if (cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_resample), dim3(2), dim3(SMC_THREADS), args, 0, nullptr)) return 3;
        const cudaError_t rc = cudaDeviceSynchronize();
        std::vector<int> h(512);
        int after[2];
        cudaMemcpy(h.data(), idx, 512 * sizeof(int), cudaMemcpyDeviceToHost);
        cudaMemcpy(after, flags, sizeof(after), cudaMemcpyDeviceToHost);
        bool ok = rc == cudaSuccess && after[1] == run;
        for (int i = 0; i < 512; ++i) ok = ok && h[i] == (i >= N ? 0x11111111 : run ? -1 : i);   // equal weights: each particle once
        printf("run %d: %s, error flag %d, indices %d .. %d, %d\n", run, cudaGetErrorString(rc), after[1], h[0], h[N - 1], h[N]);
        if (!ok) return 1;
    }
    printf("resample wait ok\n");
    return 0;
}
