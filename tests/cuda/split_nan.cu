// FP32 step attempts of the prescribed split (step_ray32<4>, tt_trace.cuh) that end on
// the axis exactly: a ray with p_phi = 0 starts at a small theta with neighbouring
// step sizes about the one that takes it to theta = 0, where the flow is NaN though
// the new point is finite.  On either side of it the flow is smooth and a step of
// this size far inside the tolerance.
// Prints: attempts, attempts accepted, attempts that ended the ray as not finite.
#include <cstdio>

#include "tt_trace.cuh"

using namespace tt;

__global__ void k_axis(int n, unsigned* out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double a = 0.5, r = 100.0, pth = -0.5;
    ImageDesc d = {};
    d.M = 1.0;
    d.a = a;
    d.r_plus = 1.0 + sqrt(1.0 - a * a);
    d.r_minus = 1.0 - sqrt(1.0 - a * a);
    d.r_capture = 1.001 * d.r_plus;
    d.r_escape = 1000.0;
    SolverDesc sol = {};
    sol.rtol = sol.atol = 1e-8;
    sol.max_steps = 1000000;
    sol.precision = 4;
    sol.int_mul = 1;
    LaneReg L = {};
    L.d = &d;
    L.kk = make_kerr(d.M, a);
    L.c.R = make_ray_const(a, -1.0, 0.0);
    L.f32.Rf = to_float(L.c.R, d.M);
    L.f32.Mf = 1.0f;
    L.f32.a2f = (float)(a * a);
    L.f32.rpmf = (float)(d.r_plus - d.r_minus);
    L.y = State{r, 1e-4, -0.01, pth};
    // d theta / d lambda = p_theta / Sigma
    const float h0 = (float)(1e-4 * (r * r + a * a) / -pth);
    L.hf = __int_as_float(__float_as_int(h0) + k - n / 2);
    StateF unused = {};
    const int code = step_ray32<4>(L, unused, sol);
    atomicAdd(out, 1u);
    if (code == -1 && L.steps == 1) atomicAdd(out + 1, 1u);
    if (code == 4) atomicAdd(out + 2, 1u);
}

int main() {
    unsigned *dev, h[3];
    if (cudaMalloc(&dev, sizeof h) != cudaSuccess || cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 1;
    k_axis<<<2048, 128>>>(2048 * 128, dev);
    if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%u %u %u\n", h[0], h[1], h[2]);
    return 0;
}
