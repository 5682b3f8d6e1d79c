// Products on the integer pipes (tt_soft64.cuh) against FP64's, bit for bit:
//   mul    random products over 2^+-280, with factors whose low bits are zero or
//          one (ties, carries into the exponent)
//   step   step attempts of the five integrators from random states (stages inside the horizon,
//          equatorial states, huge and tiny components, NaN and infinite steps
//          among them): an attempt that passes the range checks, ok(), must
//          equal the plain one in every output
// Prints: name, mismatches, attempts that passed, attempts.
#include <cstdio>

#include "tt_trace.cuh"

using namespace tt;

struct Rng {
    unsigned long long s;
    __device__ unsigned long long next() {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    }
    __device__ double uniform(double lo, double hi) { return lo + (hi - lo) * ((double)(next() >> 11) * 0x1p-53); }
};

__device__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

__global__ void k_mul(int n, unsigned long long* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 77777ull + 5};
    for (int i = 0; i < n; ++i) {
        unsigned long long x = g.next(), y = g.next(), m = g.next();
        x = (x & 0x800fffffffffffffull) | ((743 + g.next() % 561) << 52);
        y = (y & 0x800fffffffffffffull) | ((743 + g.next() % 561) << 52);
        const int zx = m & 63, zy = (m >> 6) & 63;       // trailing zeros or ones
        if (m & 0x1000) x = x >> (zx % 53) << (zx % 53);
        if (m & 0x2000) y = y >> (zy % 53) << (zy % 53);
        if (m & 0x4000) x |= (1ull << (zx % 53)) - 1;
        if (m & 0x8000) y |= (1ull << (zy % 53)) - 1;
        const double a = __longlong_as_double((long long)x), b = __longlong_as_double((long long)y);
        if (!same(a * b, soft_mul64(a, b))) atomicAdd(out, 1ull);
        atomicAdd(out + 1, 1ull);
        atomicAdd(out + 2, 1ull);
    }
}

template <int METHOD>
__global__ void k_step(int n, unsigned long long* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 99991ull + 11 + METHOD};
    const double odd[8] = {0.0, -0.0, 1e-320, 1e-200, 1e200, 1.0 / 0.0, nan(""), -1e-40};
    ImageDesc d = {};
    for (int i = 0; i < n; ++i) {
        const int kind = (int)(g.next() % 8);
        const double a = kind == 1 ? 0.0 : g.uniform(0.0, 0.998), rp = 1.0 + sqrt(1.0 - a * a);
        const KerrK k = make_kerr(1.0, a);
        const RayConst R = make_ray_const(a, g.uniform(-1.1, -0.9), kind == 2 ? 0.0 : g.uniform(-20.0, 20.0));
        State y{kind & 1 ? g.uniform(0.9 * rp, 6.0) : exp(g.uniform(0.7, 7.0)), g.uniform(0.02, 3.1),
                g.uniform(-2.0, 2.0), g.uniform(-10.0, 10.0)};
        double h = exp(g.uniform(-12.0, 4.0));
        if (kind == 3) {                                  // the equatorial plane
            y.th = kHalfPi;
            y.pth = 0.0;
        }
        if (kind == 4) {
            double* at[5] = {&y.r, &y.th, &y.pr, &y.pth, &h};
            *at[g.next() % 5] = odd[g.next() % 8];
        }
        State k1, p, q, pk, qk, pe, qe;
        double H, s, c, pH, qH, ps, pc, qs, qc;
        flow64<0>(d, k, R, y, k1, H);
        sincos(y.th, &s, &c);
        const double tol = exp(g.uniform(-30.0, -14.0));
        FpMul fm;
        IntMul im;
        ps = qs = s;
        pc = qc = c;
        double pn = 0.0, qn = 0.0;
        if constexpr (METHOD == 4) {
            h *= 0.01;                                    // a fixed step that the iterations converge for
            verlet_step64<0>(d, k, R, y, k1, h, p, pk, pH, fm);
            verlet_step64<0>(d, k, R, y, k1, h, q, qk, qH, im);
        } else {
            if constexpr (METHOD == 3) {
                gbs_step64<0>(d, k, R, y, k1, h, p, pk, pH, pe, fm);
                gbs_step64<0>(d, k, R, y, k1, h, q, qk, qH, qe, im);
            } else {
                rk_step64<0, METHOD>(d, k, R, y, k1, h, p, pk, pH, pe, s, c, ps, pc, fm);
                rk_step64<0, METHOD>(d, k, R, y, k1, h, q, qk, qH, qe, s, c, qs, qc, im);
            }
            const double he = METHOD == 3 ? 1.0 : h;
            pn = err_norm2(y, p, pe, tol, tol, he, fm);
            qn = err_norm2(y, q, qe, tol, tol, he, im);
        }
        atomicAdd(out + 2, 1ull);
        if (!im.ok()) continue;
        atomicAdd(out + 1, 1ull);
        const bool eq = same(p.r, q.r) && same(p.th, q.th) && same(p.pr, q.pr) && same(p.pth, q.pth) &&
                        same(pk.r, qk.r) && same(pk.th, qk.th) && same(pk.pr, qk.pr) && same(pk.pth, qk.pth) &&
                        same(pH, qH) && same(ps, qs) && same(pc, qc) && same(pn, qn);
        if (!eq) atomicAdd(out, 1ull);
    }
}

int main() {
    unsigned long long *dev, h[3];
    cudaMalloc(&dev, sizeof h);
    auto report = [&](const char* name) {
        if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return false;
        printf("%s %llu %llu %llu\n", name, h[0], h[1], h[2]);
        return cudaMemset(dev, 0, sizeof h) == cudaSuccess;
    };
    cudaMemset(dev, 0, sizeof h);
    k_mul<<<304, 256>>>(500, dev);
    if (!report("mul")) return 1;
    k_step<0><<<304, 128>>>(50, dev);
    if (!report("dopri5")) return 1;
    k_step<1><<<304, 128>>>(50, dev);
    if (!report("cash_karp")) return 1;
    k_step<2><<<304, 128>>>(50, dev);
    if (!report("fehlberg")) return 1;
    k_step<3><<<304, 128>>>(10, dev);
    if (!report("gbs")) return 1;
    k_step<4><<<304, 128>>>(20, dev);
    return report("verlet") ? 0 : 1;
}
