// The Cholesky factor's pivots over FP64's range: its reciprocal against the rounded quotient, and the factor of a matrix
// scaled by even powers of two, which is that of the matrix scaled by their roots.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#include "../paper_2503_16028_gb300/csrc/gm.cu"

using namespace smcgm;

__global__ void k_rcp(int n, const double* d, long long* worst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long long e = __double_as_longlong(rcp_newton(d[i])) - __double_as_longlong(1.0 / d[i]);
    atomicMax(reinterpret_cast<unsigned long long*>(worst), (unsigned long long)(e < 0 ? -e : e));
}

int main() {
    // reciprocals: every binary exponent of the range, the ends of each binade and pseudo-random fractions
    std::vector<double> d;
    unsigned long long x = 88172645463325252ull;
    for (int e = -1000; e < 1000; ++e)
        for (int k = 0; k < 40; ++k) {
            x ^= x << 13; x ^= x >> 7; x ^= x << 17;
            const double f = k == 0 ? 1.0 : k == 1 ? 2.0 - 0x1p-52 : k == 2 ? 1.0 + 0x1p-52 : 1.0 + (double)(x >> 12) * 0x1p-52;
            d.push_back(std::ldexp(f, e));
        }
    d.push_back(0x1p1000);
    double* dd;
    long long *dw, worst = 0;
    if (cudaMalloc(&dd, d.size() * 8) || cudaMalloc(&dw, 8)) return 2;
    cudaMemcpy(dd, d.data(), d.size() * 8, cudaMemcpyHostToDevice);
    cudaMemset(dw, 0, 8);
    k_rcp<<<((int)d.size() + 255) / 256, 256>>>((int)d.size(), dd, dw);
    if (cudaMemcpy(&worst, dw, 8, cudaMemcpyDeviceToHost)) return 3;
    printf("reciprocal: %lld ulp at most\n", worst);
    if (worst > 1) return 1;
    // factors, r = 9 (a partial panel): A = B B^T + I with entries of order one, times 2^(2 s)
    constexpr int r = 9;
    double A[r * r], L0[r * r], *cov, *L, *Lb, *ld, *w;
    int* bad;
    for (int i = 0; i < r; ++i)
        for (int j = 0; j < r; ++j) {
            A[i * r + j] = i == j;
            for (int k = 0; k < r; ++k) A[i * r + j] += std::sin(1.0 + i * 3 + k * k) * std::sin(1.0 + j * 3 + k * k);
        }
    if (cudaMalloc(&cov, sizeof(A)) || cudaMalloc(&L, sizeof(A)) || cudaMalloc(&Lb, cov_lb_doubles(1, r) * 8) || cudaMalloc(&ld, 8) || cudaMalloc(&w, 8) ||
        cudaMalloc(&bad, 4)) return 2;
    const int shifts[] = {0, 1, -40, 200, -490, -499, -505, -510, -515, -520, 499, 505};
    for (int s : shifts) {
        double S[r * r], F[r * r], logdet;
        int b = -1;
        for (int k = 0; k < r * r; ++k) S[k] = std::ldexp(A[k], 2 * s);
        cudaMemcpy(cov, S, sizeof(S), cudaMemcpyHostToDevice);
        cudaMemset(bad, 0, 4);
        k_chol<true><<<1, 256, r * (r + 1) * 8>>>(r, cov, w, L, Lb, ld, nullptr, bad);
        cudaMemcpy(F, L, sizeof(F), cudaMemcpyDeviceToHost);
        cudaMemcpy(&logdet, ld, 8, cudaMemcpyDeviceToHost);
        if (cudaMemcpy(&b, bad, 4, cudaMemcpyDeviceToHost)) return 3;
        // A's entries keep 1074 + 2 s bits when they are subnormal
        const double tol = std::fmax(1e-13, 64.0 * std::ldexp(1.0, -1074 - 2 * s));
        double err = 0.0;
        for (int k = 0; k < r * r; ++k) {
            const double v = std::ldexp(F[k], -s);
            if (s == 0) L0[k] = v;
            err = std::fmax(err, std::fabs(v - L0[k]));
            if (!(v == v)) err = INFINITY;
        }
        if (s == 0) {                                    // the base case against its own product
            for (int i = 0; i < r; ++i)
                for (int j = 0; j <= i; ++j) {
                    double p = 0.0;
                    for (int k = 0; k <= j; ++k) p += L0[i * r + k] * L0[j * r + k];
                    err = std::fmax(err, std::fabs(p - A[i * r + j]) / 10.0);
                }
        }
        printf("scale 2^%d: error %.1e, not positive %d, log det %.3f\n", 2 * s, err, b, logdet);
        if (b != 0 || !(err <= tol) || !(std::fabs(logdet) < 1e5)) return 1;
    }
    printf("factor pivots ok\n");
    return 0;
}
