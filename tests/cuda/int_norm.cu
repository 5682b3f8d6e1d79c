// The error norm with integer products (err_norm2, tt_trace.cuh) against the plain one
// over the tolerances that select it, and beyond.
// Prints: evaluations that passed the checks and differ, that passed, evaluations.
#include <cstdio>

#include "tt_trace.cuh"

using namespace tt;

__global__ void k_norm(int n, double rtol, double atol, unsigned long long* out) {
    unsigned long long z0 = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 99991ull + 5;
    auto uniform = [&](double lo, double hi) {
        unsigned long long z = (z0 += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return lo + (hi - lo) * ((double)((z ^ (z >> 31)) >> 11) * 0x1p-53);
    };
    for (int i = 0; i < n; ++i) {
        const bool flat = (i & 7) == 7;         // theta and p_theta at zero
        const State y{exp(uniform(0.5, 7.0)), flat ? 0.0 : uniform(0.02, 3.1), uniform(-1.5, -0.01),
                      flat ? 0.0 : uniform(-9.0, 9.0)};
        const double f = uniform(0.9, 1.1), w = (rtol + atol) * exp(uniform(-6.0, 3.0));
        const State yn{y.r * f, y.th * f, y.pr * f, y.pth * f};
        const State e{w * uniform(-1.0, 1.0), flat ? 0.0 : w * uniform(-1.0, 1.0), w * uniform(-1.0, 1.0),
                      (i & 15) ? w * uniform(-1.0, 1.0) : 0.0};
        FpMul fm;
        IntMul im;
        im.see(yn.r);
        im.see(yn.pr);
        const double he = exp(uniform(-6.0, 5.0));
        const double p = err_norm2(y, yn, e, atol, rtol, he, fm), q = err_norm2(y, yn, e, atol, rtol, he, im);
        atomicAdd(out + 2, 1ull);
        if (!im.ok()) continue;
        atomicAdd(out + 1, 1ull);
        if (__double_as_longlong(p) != __double_as_longlong(q)) atomicAdd(out, 1ull);
    }
}

int main() {
    const double tol[][2] = {{1e-10, 1e-10}, {1e-10, 1e-15}, {1e-10, 1e-60}, {1e-10, 1e-310}, {1e-15, 1e-15},
                             {1e-27, 1e-27}, {1e-310, 1e-10}, {1e3, 1e-3},  {0x1p47, 0x1p47}, {1e-90, 1e-90},
                             {1e200, 1e200}};
    unsigned long long *dev, h[3];
    if (cudaMalloc(&dev, sizeof h) != cudaSuccess) return 1;
    for (const auto& t : tol) {
        if (cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 1;
        k_norm<<<304, 128>>>(64, t[0], t[1], dev);
        if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
        printf("%g %g %llu %llu %llu\n", t[0], t[1], h[0], h[1], h[2]);
    }
    return 0;
}
