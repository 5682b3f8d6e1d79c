// float <-> double conversions on the integer pipes (tt_soft64.cuh) against the
// conversion instructions, bit for bit: random values over (and beyond) the
// floats' range, ties, zeros, subnormals, the largest floats.
// Prints: values, mismatches of int_to_double, of int_to_float where it applies,
// of float_odd.
#include <cstdio>

#include "tt_trace.cuh"

using namespace tt;

__global__ void k_convert(int n, unsigned* out) {
    unsigned long long s = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 7919ull + 1;
    auto next = [&]() {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    for (int i = 0; i < n; ++i) {
        float x = __uint_as_float((unsigned)next());               // every exponent, subnormals among them
        if (!isfinite(x)) x = (i & 1) ? 3.4028235e38f : -0.0f;
        if (i == 0) x = 0.0f;
        atomicAdd(out, 1u);
        if (__double_as_longlong((double)x) != __double_as_longlong(int_to_double(x))) atomicAdd(out + 1, 1u);
        unsigned long long b = next();
        b = (b & 0x800fffffffffffffull) | ((860 + next() % 310) << 52);     // 2^-163 .. 2^146
        if (i % 5 == 1) b &= ~0x1fffffffull;                        // a float exactly
        if (i % 5 == 2) b = (b & ~0x1fffffffull) | 0x10000000ull;   // halfway between two floats
        if (i % 5 == 3) b |= 0x000fffffe0000000ull;                 // a carry into the exponent
        if (i == 1) b = 0x8000000000000000ull;
        if (i == 2) b = 0x47efffffffffffffull;                      // rounds up to infinity
        const double y = __longlong_as_double((long long)b);
        const float f = (float)y;
        const bool odd = y != 0.0 && (fabs(y) < 0x1p-126 || fabs(y) >= 0x1p128);
        if (odd != float_odd(y)) atomicAdd(out + 3, 1u);
        if (!odd && __float_as_uint(f) != __float_as_uint(int_to_float(y))) atomicAdd(out + 2, 1u);
        if (__float_as_uint(f) != __float_as_uint(state_float(y))) atomicAdd(out + 2, 1u);
    }
}

int main() {
    unsigned *dev, h[4];
    cudaMalloc(&dev, sizeof h);
    cudaMemset(dev, 0, sizeof h);
    k_convert<<<304, 256>>>(500, dev);
    if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%u %u %u %u\n", h[0], h[1], h[2], h[3]);
    return 0;
}
