// Coefficient preparation: the stacked vector of Sec. 2.2 -> the per-tap
// polynomial tables read by the forward kernels (widely-linear form, see
// dpd_internal.h) and by the adjoint input-gradient kernel (see dpd_adj.cuh).
// Also the FP64 finalisation of the coefficient gradient.
#include "dpd_device.cuh"
#include "dpd_internal.h"

namespace dpd {

// Coefficient k of the stacked vector as FP32 (FP64 sources are rounded to
// nearest, as the FP32 copy of an FP64 estimate is).
__device__ __forceinline__ float2 coef_f32(const float2 *h, int i) { return h[i]; }
__device__ __forceinline__ float2 coef_f32(const double2 *h, int i)
{
    return make_float2((float)h[i].x, (float)h[i].y);
}

// blockIdx.x selects a problem of a batch: coefficients hin + x * hstride,
// table tab + x * tstride (0 for a single table).
template <typename H>
__global__ void wl_table_kernel(const H *__restrict__ hin, int Bp, int Bq, int T, int B, float *__restrict__ tab,
                                float *__restrict__ adj, int hstride, int tstride)
{
    grid_dep_wait();
    hin += (size_t)blockIdx.x * hstride;
    tab += (size_t)blockIdx.x * tstride;
    auto h = [hin](int i) { return coef_f32(hin, i); };
    const int i = threadIdx.x;   // one thread per (tap k, order index m)
    if (i < T * B) {
        const int k = i / B, m = i % B;
        const float2 A = (m < Bp) ? h(m * T + k) : make_float2(0.f, 0.f);          // h_{2m+1,k}
        const float2 C = (m < Bq) ? h((Bp + m) * T + k) : make_float2(0.f, 0.f);   // hbar_{2m+1,k}
        tab[wl_index(B, k, m, 0)] = A.x + C.x;      // P0 = Re(A+C)
        tab[wl_index(B, k, m, 1)] = -(A.y - C.y);   // P1 = -Im(A-C)
        tab[wl_index(B, k, m, 2)] = A.y + C.y;      // P2 = Im(A+C)
        tab[wl_index(B, k, m, 3)] = A.x - C.x;      // P3 = Re(A-C)
        if (adj) {
            // {P0, P3} multiplies the gradient sample {c, d}, {P2, P1} its swap
            // {d, c}: conj(h) g + hbar conj(g) = {P0 c + P2 d, P3 d + P1 c}.
            float *q = adj + 4 * (k * B + m);
            q[0] = A.x + C.x;
            q[1] = A.x - C.x;
            q[2] = A.y + C.y;
            q[3] = C.y - A.y;
        }
    }
    if (i == 0) {
        const float2 c = h((Bp + Bq) * T);
        tab[4 * B * T] = c.x;
        tab[4 * B * T + 1] = c.y;
    }
}

cudaError_t launch_wl_table(const float2 *h, int Bp, int Bq, int T, float *tab, float *adj_tab,
                            cudaStream_t s)
{
    const int B = Bp > Bq ? Bp : Bq;
    return launch_pdl(wl_table_kernel<float2>, dim3(1), 64, 0, s, h, Bp, Bq, T, B, tab, adj_tab, 0, 0);
}

cudaError_t launch_wl_table_f64(const double2 *h, int Bp, int Bq, int T, float *tab, cudaStream_t s)
{
    const int B = Bp > Bq ? Bp : Bq;
    return launch_pdl(wl_table_kernel<double2>, dim3(1), 64, 0, s, h, Bp, Bq, T, B, tab, nullptr, 0, 0);
}

cudaError_t launch_wl_table_f64_many(const double2 *h, int count, int hstride, int Bp, int Bq, int T, float *tab,
                                     int tstride, cudaStream_t s)
{
    const int B = Bp > Bq ? Bp : Bq;
    return launch_pdl(wl_table_kernel<double2>, dim3((unsigned)count), 64, 0, s, h, Bp, Bq, T, B, tab, nullptr, hstride,
                      tstride);
}

// One warp per coefficient: lane t sums rows t, t + 32, ... in order (up to four
// loads in flight), then a fixed shuffle tree combines the 32 sums
// (deterministic, FP64).  blockIdx.y selects a problem of a batch (its rows and
// outputs follow the previous problem's).
constexpr int kFinalizeWarps = 8;

__global__ void __launch_bounds__(32 * kFinalizeWarps)
    adj_finalize_kernel(const float2 *__restrict__ partials, int rows, int K, float2 *__restrict__ gh,
                        double2 *__restrict__ gh64)
{
    grid_dep_wait();
    const int i = blockIdx.x * kFinalizeWarps + (threadIdx.x >> 5), t = threadIdx.x & 31;
    if (i >= K) return;
    partials += (size_t)blockIdx.y * rows * K;
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
    if (t == 0) {
        if (gh) gh[(size_t)blockIdx.y * K + i] = make_float2((float)re, (float)im);
        if (gh64) gh64[(size_t)blockIdx.y * K + i] = make_double2(re, im);
    }
}

static cudaError_t finalize(const float2 *partials, int rows, int K, int count, float2 *gh, double2 *gh64,
                            cudaStream_t s)
{
    const dim3 grid((unsigned)((K + kFinalizeWarps - 1) / kFinalizeWarps), (unsigned)count);
    return launch_pdl(adj_finalize_kernel, grid, 32 * kFinalizeWarps, 0, s, partials, rows, K, gh, gh64);
}

cudaError_t launch_adj_finalize(const float2 *partials, int rows, int K, float2 *gh, cudaStream_t s)
{
    return finalize(partials, rows, K, 1, gh, nullptr, s);
}

cudaError_t launch_adj_finalize64(const float2 *partials, int rows, int K, double2 *out, cudaStream_t s)
{
    return finalize(partials, rows, K, 1, nullptr, out, s);
}

// One partial row per problem (the batched refinement): the FP64 sum is the
// row itself, widened; one thread per coefficient instead of a 256-thread
// reduction per coefficient.
__global__ void adj_widen_kernel(const float2 *__restrict__ partials, int64_t n, double2 *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const float2 v = partials[i];
        out[i] = make_double2(v.x, v.y);
    }
}

cudaError_t launch_adj_finalize64_many(const float2 *partials, int rows, int K, int count, double2 *out,
                                       cudaStream_t s)
{
    if (rows == 1) {
        const int64_t n = (int64_t)K * count;
        adj_widen_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(partials, n, out);
        count_launch();
        return cudaGetLastError();
    }
    return finalize(partials, rows, K, count, nullptr, out, s);
}

}  // namespace dpd
