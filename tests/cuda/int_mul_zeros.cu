// Step attempts with integer products (tt_soft64.cuh) from states whose p_phi, p_theta
// or spin is zero or tiny, and on a tabulated metric, against plain ones.
// Argument: a table's patch coefficients (tartarus_table_coefficients, raw doubles),
// its nr and nth, r_min, r_max, spin.
// Prints: name, attempts that passed the checks and differ in any output, attempts
// that passed, attempts.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "tt_trace.cuh"

using namespace tt;

__device__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
__device__ bool same(const State& a, const State& b) {
    return same(a.r, b.r) && same(a.th, b.th) && same(a.pr, b.pr) && same(a.pth, b.pth);
}

// kind 0: ordinary rays; 1: p_phi = 0; 2: p_phi ~ 1e-17 (a column alpha = 0); 3: the equatorial
// plane from rest in theta; 4: p_theta = 0 off it; 5: p_theta ~ 1e-25 in it
template <int METRIC, int METHOD>
__global__ void k_step(int n, int kind, double a, const __grid_constant__ ImageDesc d, unsigned long long* out) {
    unsigned long long z0 = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 99991ull + 17 * kind;
    auto uniform = [&](double lo, double hi) {
        unsigned long long z = (z0 += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return lo + (hi - lo) * ((double)((z ^ (z >> 31)) >> 11) * 0x1p-53);
    };
    const KerrK k = make_kerr(1.0, a);
    for (int i = 0; i < n; ++i) {
        const double pph = kind == 1 ? 0.0 : kind == 2 ? uniform(-1e-17, 1e-17) : uniform(2.0, 9.0);
        const RayConst R = make_ray_const(a, uniform(-1.1, -0.9), pph);
        State y{exp(uniform(1.8, 6.8)), uniform(0.3, 2.8), uniform(-1.2, -0.8), uniform(1.0, 5.0)};
        if (kind == 3 || kind == 5) y.th = kHalfPi;
        if (kind == 3 || kind == 4) y.pth = 0.0;
        if (kind == 5) y.pth = uniform(-1e-25, 1e-25);
        const double h = y.r * uniform(0.001, 0.1), tol = 1e-10;
        State k1, p, q, pk, qk, pe, qe;
        double H, s, c, pH, qH, ps, pc, qs, qc, pn = 0.0, qn = 0.0;
        flow64<METRIC>(d, k, R, y, k1, H);
        sincos(y.th, &s, &c);
        ps = qs = s;
        pc = qc = c;
        FpMul fm;
        IntMul im;
        if constexpr (METHOD == 3) {
            gbs_step64<METRIC>(d, k, R, y, k1, h, p, pk, pH, pe, fm);
            gbs_step64<METRIC>(d, k, R, y, k1, h, q, qk, qH, qe, im);
        } else {
            rk_step64<METRIC, METHOD>(d, k, R, y, k1, h, p, pk, pH, pe, s, c, ps, pc, fm);
            rk_step64<METRIC, METHOD>(d, k, R, y, k1, h, q, qk, qH, qe, s, c, qs, qc, im);
        }
        const double he = METHOD == 3 ? 1.0 : h;
        pn = err_norm2(y, p, pe, tol, tol, he, fm);
        qn = err_norm2(y, q, qe, tol, tol, he, im);
        atomicAdd(out + 2, 1ull);
        if (!im.ok()) continue;
        atomicAdd(out + 1, 1ull);
        if (!(same(p, q) && same(pk, qk) && same(pH, qH) && same(ps, qs) && same(pc, qc) && same(pn, qn)))
            atomicAdd(out, 1ull);
    }
}

int main(int argc, char** argv) {
    if (argc != 7) return 2;
    ImageDesc d = {};
    d.nr = atoi(argv[2]);
    d.nth = atoi(argv[3]);
    const double r_min = atof(argv[4]), r_max = atof(argv[5]), a = atof(argv[6]);
    d.kind = 1;
    d.M = 1.0;
    d.a = a;
    d.u0 = std::log(r_min);
    d.du = (std::log(r_max) - d.u0) / (d.nr - 1);
    d.dth = M_PI / (d.nth - 1);
    d.idu = 1.0 / d.du;
    d.idth = 1.0 / d.dth;
    std::vector<double> coef((size_t)(d.nr - 1) * (d.nth - 1) * kTableCoef);
    FILE* f = std::fopen(argv[1], "rb");
    if (!f || std::fread(coef.data(), sizeof(double), coef.size(), f) != coef.size()) return 3;
    std::fclose(f);
    double* table;
    unsigned long long *dev, h[3];
    if (cudaMalloc(&table, coef.size() * sizeof(double)) != cudaSuccess || cudaMalloc(&dev, sizeof h) != cudaSuccess ||
        cudaMemcpy(table, coef.data(), coef.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
        return 4;
    d.table = table;
    for (int kind = 0; kind < 6; ++kind) {
        for (int metric = 0; metric < 2; ++metric) {
            for (int gbs = 0; gbs < 2; ++gbs) {
                if (cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 5;
                const int n = gbs ? 2 : 10;
                if (metric && gbs) k_step<1, 3><<<304, 64>>>(n, kind, a, d, dev);
                else if (metric) k_step<1, 0><<<304, 64>>>(n, kind, a, d, dev);
                else if (gbs) k_step<0, 3><<<304, 64>>>(n, kind, a, d, dev);
                else k_step<0, 0><<<304, 64>>>(n, kind, a, d, dev);
                if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 6;
                printf("%s_%s_%d %llu %llu %llu\n", metric ? "table" : "kerr", gbs ? "gbs" : "dopri5", kind, h[0], h[1],
                       h[2]);
            }
        }
    }
    return 0;
}
