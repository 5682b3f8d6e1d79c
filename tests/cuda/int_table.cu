// The FP64 table path's division by a constant and cell index, and the step control's
// factor on the integer pipes, against the plain expressions, bit for bit.
// Prints: name, evaluations, evaluations that differ.
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

// spacings 2^-20 .. 2^3 (their significands at times all ones, or a power of two)
// and numerators of either sign over 2^+-40, or zero
__global__ void k_div(int n, unsigned long long* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 77777ull + 5};
    for (int i = 0; i < n; ++i) {
        double b = exp2(g.uniform(-20.0, 3.0)), a = g.uniform(-1.0, 1.0) * exp2(g.uniform(-40.0, 40.0));
        if ((i & 15) == 1) b = __longlong_as_double(__double_as_longlong(b) | 0xfffffffffffffll);
        if ((i & 15) == 2) b = __longlong_as_double(__double_as_longlong(b) & ~0xfffffffffffffll);
        if ((i & 15) == 3) a = rint(a) * b;              // quotients at, or next to, whole numbers
        if ((i & 63) == 4 || a == 0.0) a = 0.0;          // (a zero of either sign gives +0 here)
        const double q = div_by(a, b, 1.0 / b);
        atomicAdd(out, 1ull);
        if (!same(q, a / b)) atomicAdd(out + 1, 1ull);
    }
}

__global__ void k_cell(int n, unsigned long long* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 33333ull + 5};
    const double odd[] = {0.0, -0.0, 1.0, -1.0, 0.5, -1e-300, 1e-300, 0x1p20, 0x1p21, 0x1p21 - 0x1p-32, 0x1p22 + 0.5,
                          0x1p31, 1e18, -1e18, 1.0 / 0.0, -1.0 / 0.0, nan("")};
    for (int i = 0; i < n; ++i) {
        const int n_max = (i & 3) == 0 ? 0 : (i & 3) == 1 ? 1 : (int)(g.next() % 3000000u);
        double x = g.uniform(-3.0, n_max + 3.0);
        if ((i & 7) == 1) x = rint(x);
        if ((i & 7) == 2) x = __longlong_as_double(__double_as_longlong(rint(x)) + (long long)(g.next() % 3u) - 1);
        if ((i & 7) == 3) x = n_max + (double)(i % 3);
        if ((i & 7) == 4) x = odd[g.next() % (sizeof odd / sizeof *odd)];
        double f;
        const int k = table_cell(x, n_max, f);
        const int ref = min(max((int)floor(x), 0), n_max);
        atomicAdd(out, 1ull);
        // (every cell is one of the table's, whatever x is)
        if (k < 0 || k > n_max || k != ref || !same(f, (double)ref)) atomicAdd(out + 1, 1ull);
    }
}

__global__ void k_next(int n, unsigned long long* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 11111ull + 5};
    for (int i = 0; i < n; ++i) {
        const double h = exp2(g.uniform(-60.0, 100.0)), top = (i & 1) ? 1.0 : 10.0;
        double e = exp2(g.uniform(-12.0, 6.0));
        if ((i & 7) == 1) e = exp2(g.uniform(-130.0, 130.0));
        if ((i & 63) == 2) e = 0.0;
        if ((i & 63) == 3) e = 1.0 / 0.0;
        const double ref = h * fmin(top, fmax(0.2, step_factor(e)));
        atomicAdd(out, 1ull);
        if (!same(next_h(h, e, top), ref)) atomicAdd(out + 1, 1ull);
    }
}

int main() {
    unsigned long long *dev, h[2];
    if (cudaMalloc(&dev, sizeof h) != cudaSuccess) return 1;
    for (int k = 0; k < 3; ++k) {
        if (cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 1;
        if (k == 0) k_div<<<304, 256>>>(500, dev);
        if (k == 1) k_cell<<<304, 256>>>(200, dev);
        if (k == 2) k_next<<<304, 256>>>(200, dev);
        if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
        printf("%s %llu %llu\n", k == 0 ? "div_by" : k == 1 ? "table_cell" : "next_h", h[0], h[1]);
    }
    return 0;
}
