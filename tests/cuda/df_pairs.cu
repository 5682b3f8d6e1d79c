// The closed-form flow with double-floats in packed pairs (tt_df.cuh) against the
// same flow one double-float at a time, bit for bit, on random states: a packed
// product contracted into a sum, or an operand swapped, changes low bits.
// Prints: states, states that differ.
#include <cstdio>

#include "tt_df.cuh"

using namespace tt;

__device__ bool same(DF a, DF b) {
    return __float_as_uint(a.hi) == __float_as_uint(b.hi) && (a.lo == b.lo || (a.lo != a.lo && b.lo != b.lo));
}

__global__ void k_pairs(int n, unsigned* out) {
    df_sincos_table(s_df_tab);
    __syncthreads();
    unsigned long long s = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 77777ull + 3;
    auto uniform = [&](double lo, double hi) {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return lo + (hi - lo) * ((double)((z ^ (z >> 31)) >> 11) * 0x1p-53);
    };
    for (int i = 0; i < n; ++i) {
        const double a = (i & 7) ? uniform(0.0, 0.998) : 0.0, rp = 1.0 + sqrt(1.0 - a * a);
        const KerrDF k = make_kerr_df(make_kerr(1.0, a));
        const RayDF R = make_ray_df(make_ray_const(a, uniform(-1.1, -0.9), uniform(-20.0, 20.0)));
        const StateDF y{df_of(i & 1 ? uniform(0.98 * rp, 6.0) : exp(uniform(0.7, 7.0))), df_of(uniform(-4.0, 8.0)),
                        df_of(uniform(-2.0, 2.0)), df_of(uniform(-10.0, 10.0))};
        StateDF f;
        DF H;
        kerr_flow_df(k, R, y, f, H);
        const FlowDF2 o = kerr_flow_pair_call(k, R, pairs(y));
        const StateDF g = halves(o.f);
        atomicAdd(out, 1u);
        if (!(same(f.r, g.r) && same(f.th, g.th) && same(f.pr, g.pr) && same(f.pth, g.pth) && same(H, o.H)))
            atomicAdd(out + 1, 1u);
    }
}

int main() {
    unsigned *dev, h[2];
    cudaMalloc(&dev, sizeof h);
    cudaMemset(dev, 0, sizeof h);
    k_pairs<<<304, 128>>>(100, dev);
    if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%u %u\n", h[0], h[1]);
    return 0;
}
