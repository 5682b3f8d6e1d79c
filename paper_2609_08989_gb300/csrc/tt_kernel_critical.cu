// tt_kernel_critical.cu -- the mixed paths' near-critical rays (closed-form Kerr),
// traced in double-float by a kernel of their own that the kernel of the other
// rays overlaps.
#include "tt_trace.cuh"

namespace tt {

// One 256-thread block per SM at 198 (FP32 pair) or 204 registers, no spills.  The kernel of the
// other rays may start once these blocks are resident (programmatic dependent
// launch): it takes the SMs as they end, so that the tail of the longest rays
// (up to ~1200 step attempts of ~6 us) runs beside it.  Fewer SMs for these rays
// (crit_stride 2, 4, 6) measured 39.1, 39.6 and 50.6 ms per 2048^2 image against
// 38.7, and 128-thread blocks, which leave room for the other kernel on every SM,
// 50.7 ms.
template <int ACC, int N>
__global__ void __launch_bounds__(256) trace_kernel_critical(const __grid_constant__ LaunchParams<N> p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    critical_loop<ACC>(p.desc, p.n_desc, p.total, p.solc, p.tune, p.queue + 1);
}

template <int N>
static cudaError_t launch_critical_n(const ImageDesc* descs, int n, long long total, const SolverDesc& sol,
                                     const LaunchShape& shape, unsigned long long* queue, cudaStream_t stream) {
    LaunchParams<N> p;
    fill_params<N>(p, descs, n, total, sol, shape, queue);
    const int grid = max(1, sm_count() / p.tune.crit_stride);
    if (sol.precision == 2) trace_kernel_critical<1, N><<<grid, 256, 0, stream>>>(p);
    else trace_kernel_critical<0, N><<<grid, 256, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_critical(const ImageDesc* descs, int n, long long total, const SolverDesc& sol,
                            const LaunchShape& shape, unsigned long long* queue, cudaStream_t stream) {
    if (n == 1) return launch_critical_n<1>(descs, n, total, sol, shape, queue, stream);
    return launch_critical_n<kMaxImagesPerLaunch>(descs, n, total, sol, shape, queue, stream);
}

}  // namespace tt
