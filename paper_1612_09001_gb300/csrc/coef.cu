// Coefficient preparation: the stacked vector of Sec. 2.2 -> the per-tap
// polynomial tables read by the forward kernels (widely-linear form, see
// dpd_internal.h) and by the adjoint input-gradient kernel (see dpd_adj.cuh).
// Also the FP64 finalisation of the coefficient gradient.
#include "dpd_device.cuh"
#include "dpd_table.cuh"

namespace dpd {

__global__ void wl_table_kernel(const float2 *h, int Bp, int Bq, int T, int B, float *__restrict__ tab,
                                float *__restrict__ adj)
{
    grid_dep_wait();
    wl_table_entry([h](int i) { return h[i]; }, threadIdx.x, Bp, Bq, T, B, tab, adj);
}

cudaError_t launch_wl_table(const float2 *h, int Bp, int Bq, int T, float *tab, float *adj_tab,
                            cudaStream_t s)
{
    const int B = Bp > Bq ? Bp : Bq;
    return launch_pdl(wl_table_kernel, dim3(1), 64, 0, s, h, Bp, Bq, T, B, tab, adj_tab);
}

// One warp per coefficient: lane t sums rows t, t + 32, ... in order (up to four
// loads in flight), then a fixed shuffle tree combines the 32 sums
// (deterministic, FP64).
constexpr int kFinalizeWarps = 8;

__global__ void __launch_bounds__(32 * kFinalizeWarps)
    adj_finalize_kernel(const float2 *partials, int rows, int K, float2 *__restrict__ gh)
{
    grid_dep_wait();
    const int i = blockIdx.x * kFinalizeWarps + (threadIdx.x >> 5), t = threadIdx.x & 31;
    if (i >= K) return;
    double re = 0.0, im = 0.0;
#pragma unroll 4
    for (int r = t; r < rows; r += 32) {
        const float2 v = partials[(size_t)r * K + i];
        re += v.x;
        im += v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (t == 0) gh[i] = make_float2((float)re, (float)im);
}

cudaError_t launch_adj_finalize(const float2 *partials, int rows, int K, float2 *gh, cudaStream_t s)
{
    return launch_pdl(adj_finalize_kernel, dim3((unsigned)((K + kFinalizeWarps - 1) / kFinalizeWarps)),
                      32 * kFinalizeWarps, 0, s, partials, rows, K, gh);
}

}  // namespace dpd
