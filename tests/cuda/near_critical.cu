// The rays of 64 drawn images that near_critical (tt_trace.cuh) picks out.
// Prints: image, picked rays, the sum of a hash of their indices.  Two builds that
// contract floating-point expressions differently must print the same.
#include <cmath>
#include <cstdio>

#include "tt_trace.cuh"

using namespace tt;

constexpr int kSide = 2048;

__global__ void k_pick(const __grid_constant__ ImageDesc d, float band, unsigned long long* out) {
    const long long n = (long long)d.nx * d.ny;
    unsigned long long count = 0, sum = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        if (!near_critical(d, q, band)) continue;
        unsigned long long z = (unsigned long long)(q + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        ++count;
        sum += z ^ (z >> 27);
    }
    atomicAdd(out, count);
    atomicAdd(out + 1, sum);
}

int main() {
    unsigned long long *dev, h[2];
    if (cudaMalloc(&dev, sizeof h) != cudaSuccess) return 1;
    for (int i = 0; i < 64; ++i) {
        ImageDesc d = {};
        const double a = i ? 0.998 * std::fmod(i * 0.6180339887, 1.0) : 0.0, th = 0.05 + 1.52 * std::fmod(i * 0.7548776662, 1.0);
        const double r = i % 3 ? 1000.0 : 100.0, half = 6.5 + i % 5;
        d.nx = d.ny = kSide;
        d.pix_count = (long long)kSide * kSide;
        d.alpha_min = -half;
        d.beta_min = -half;
        d.dalpha = d.dbeta = 2.0 * half / kSide;
        d.r_obs = r;
        d.theta_obs = th;
        d.M = 1.0;
        d.a = a;
        d.r_plus = 1.0 + std::sqrt(1.0 - a * a);
        d.r_minus = 1.0 - std::sqrt(1.0 - a * a);
        const double s = std::sin(th), c = std::cos(th), s2 = s * s, Sig = r * r + a * a * c * c;
        const double g[5] = {-(1.0 - 2.0 * r / Sig), -2.0 * a * r * s2 / Sig, Sig / (r * r - 2.0 * r + a * a), Sig,
                             (r * r + a * a + 2.0 * a * a * r * s2 / Sig) * s2};
        const double omega = -g[1] / g[4], N = std::sqrt(-g[0] + omega * omega * g[4]);
        for (int k = 0; k < 5; ++k) d.obs_g[k] = g[k];
        d.obs_omN = omega / N;
        d.obs_iN = 1.0 / N;
        d.obs_ir = 1.0 / std::sqrt(g[2]);
        d.obs_ith = 1.0 / std::sqrt(g[3]);
        d.obs_iph = 1.0 / std::sqrt(g[4]);
        d.cos2_obs = c * c;
        d.cot2_obs = c * c / s2;
        if (cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 1;
        k_pick<<<608, 256>>>(d, 0.15f, dev);
        if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
        printf("%d %llu %llx\n", i, h[0], h[1]);
    }
    return 0;
}
