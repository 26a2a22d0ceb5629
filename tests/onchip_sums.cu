// The sums over a particle's cells in the on-chip mixed-precision solver: FP32 within half a warp, exact to 2^-36 of the
// largest term beyond, the same bits in every thread of every block; NaN from NaN and infinities.
#include <cmath>
#include <cstdio>
#include <vector>
#include "../paper_2503_16028_gb300/csrc/onchip.cu"

using namespace smcgm;

template <int C>
__global__ void __launch_bounds__(OC_T, 2) k_sum(const float* v, float2* out, int* err) {
    using M = OcMem<C>;
    extern __shared__ __align__(16) float sm[];
    OcPos<M> t;
    oc_place(t, sm, (int)threadIdx.x % M::W, (int)threadIdx.x / M::W);
    if (C > 1 && t.tid == 0) oc_init_bars<M>(sm);
    oc_sync<C>();
    df32 d{0.f, 0.f};
    for (int slot = OC_RR; slot <= OC_PQ; ++slot) {          // a block may be one exchange ahead of another: a slot each
        red_put<C>(sm, t, slot, v[blockIdx.x * OC_T + t.tid]);
        all_sync(sm, t, slot, 64 * M::CC);
        const df32 e = red_get<C>(sm, t, slot);
        if (slot > OC_RR && !(e.hi == d.hi && e.lo == d.lo) && e.hi == e.hi) atomicExch(err, 2);
        d = e;
    }
    out[blockIdx.x * OC_T + t.tid] = make_float2(d.hi, d.lo);
    oc_leave(t, err);
}

static unsigned long long g_x = 88172645463325252ull;
static double uni() {
    g_x ^= g_x << 13; g_x ^= g_x >> 7; g_x ^= g_x << 17;
    return (double)(g_x >> 11) * 0x1p-53;
}

template <int C>
static int run() {
    constexpr int CC = C * C, n = CC * OC_T;
    float* dv;
    float2* dout;
    int *derr, err = -1;
    if (cudaMalloc(&dv, n * 4) || cudaMalloc(&dout, n * 8) || cudaMalloc(&derr, 4)) return 2;
    cudaMemset(derr, 0, 4);
    cudaFuncSetAttribute(k_sum<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OcMem<C>::BYTES);
    if (C == 4) cudaFuncSetAttribute(k_sum<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int kind = 0; kind < 9; ++kind) {
        std::vector<float> v(n);
        for (int i = 0; i < n; ++i) {
            const double u = uni(), w = uni();
            switch (kind) {
                case 0: v[i] = (float)(u - 0.5); break;                            // both signs
                case 1: v[i] = (float)std::exp(30.0 * u - 20.0); break;            // positive, over 13 decades
                case 2: v[i] = 1.f / 3.f; break;
                case 3: v[i] = i == n / 3 ? 1e30f : 1e-3f; break;
                case 4: v[i] = 0.f; break;
                case 5: v[i] = (float)(1e-36 * u); break;                          // below the fixed point's range in part
                case 6: v[i] = i & 32 ? -v[i - 32] * (float)(1.0 + 1e-6 * w) : (float)(1e20 * u); break;   // warps that cancel
                case 7: v[i] = i == n - 1 ? NAN : (float)u; break;
                default: v[i] = i == 0 ? INFINITY : (float)u; break;
            }
        }
        long double exact = 0.0L, top = 0.0L;
        for (int h = 0; h < n; h += 16) {
            float a[16], b[16];
            for (int l = 0; l < 16; ++l) a[l] = v[h + l];
            for (int o = 8; o > 0; o >>= 1) {
                for (int l = 0; l < 16; ++l) b[l] = a[l] + a[l ^ o];
                for (int l = 0; l < 16; ++l) a[l] = b[l];
            }
            exact += a[0];
            if (std::fabs((long double)a[0]) > top) top = std::fabs((long double)a[0]);
        }
        cudaMemcpy(dv, v.data(), n * 4, cudaMemcpyHostToDevice);
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3(CC);
        cfg.blockDim = dim3(OC_T);
        cfg.dynamicSmemBytes = OcMem<C>::BYTES;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CC; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = C > 1 ? 1 : 0;
        if (cudaLaunchKernelEx(&cfg, k_sum<C>, (const float*)dv, dout, derr)) return 3;
        std::vector<float2> out(n);
        if (cudaMemcpy(out.data(), dout, n * 8, cudaMemcpyDeviceToHost)) return 3;
        cudaMemcpy(&err, derr, 4, cudaMemcpyDeviceToHost);
        bool ok = err == 0;
        for (int i = 0; i < n; ++i) {
            if (kind >= 7) { ok = ok && std::isnan(out[i].x); continue; }
            ok = ok && out[i].x == out[0].x && out[i].y == out[0].y;
        }
        const long double e = kind >= 7 ? 0.0L : std::fabs((long double)out[0].x + (long double)out[0].y - exact);
        ok = ok && e <= 0x1p-36L * top + 1e-42L;             // 1e-42: 256 terms of half the last place at 2^-103, and denormal parts
        printf("C %d kind %d: sum %.9Lg, error %.2Lg of the largest term%s\n", C, kind, exact, top > 0 ? e / top : e, ok ? "" : "  WRONG");
        if (!ok) return 1;
    }
    return 0;
}

int main() {
    if (run<1>() || run<2>() || run<4>()) return 1;
    printf("on-chip sums ok\n");
    return 0;
}
