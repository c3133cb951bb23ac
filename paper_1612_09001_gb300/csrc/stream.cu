// Stream continuation for dpd_apply_stream where the plain-load forward kernel
// runs (the bulk-copy kernel takes the history itself).  A block of a continuous
// stream differs from an isolated block only in its first M outputs: the taps of
// Eq. 1 reach back into the previous block.  The forward kernel runs on the block
// with zero history; this kernel then recomputes those outputs with the saved
// history and saves the new one.
#include "dpd_device.cuh"
#include "dpd_handle.h"

namespace dpd {

__global__ void stream_head_kernel(const float *__restrict__ tab, int B, int T, const float2 *__restrict__ x,
                                   int64_t n, float2 *__restrict__ hist, float2 *__restrict__ y)
{
    const int j = threadIdx.x;   // output index; T - 1 <= kHalo - 1 < 32
    const int64_t heads = n < (int64_t)(T - 1) ? n : (int64_t)(T - 1);
    float2 out = make_float2(tab[4 * B * T], tab[4 * B * T + 1]);   // c
    if (j < heads) {
        for (int k = 0; k < T; ++k) {
            const int g = j - k;   // sample n - k, negative = previous block
            const float2 v = g >= 0 ? x[g] : hist[kHalo + g];
            const float r = v.x * v.x + v.y * v.y;
            const float4 *cf = reinterpret_cast<const float4 *>(tab) + k * B;   // {P0, P2, P1, P3} per order
            float4 p = cf[B - 1];
            for (int m = B - 2; m >= 0; --m) {
                const float4 c = cf[m];
                p.x = fmaf(p.x, r, c.x);
                p.y = fmaf(p.y, r, c.y);
                p.z = fmaf(p.z, r, c.z);
                p.w = fmaf(p.w, r, c.w);
            }
            out.x = fmaf(p.x, v.x, out.x);
            out.x = fmaf(p.z, v.y, out.x);
            out.y = fmaf(p.y, v.x, out.y);
            out.y = fmaf(p.w, v.y, out.y);
        }
    }
    // new history: position n + i of (hist ++ x), i < kHalo
    float2 nh = make_float2(0.f, 0.f);
    if (j < kHalo) {
        const int64_t src = (int64_t)j + n;
        nh = src < kHalo ? hist[src] : x[src - kHalo];
    }
    __syncwarp();   // every read of the old history precedes the writes
    if (j < heads) y[j] = out;
    if (j < kHalo) hist[j] = nh;
}

cudaError_t launch_stream_head(const float *tab, int B, int T, const float2 *x, int64_t n, float2 *hist,
                               float2 *y, cudaStream_t s)
{
    stream_head_kernel<<<1, 32, 0, s>>>(tab, B, T, x, n, hist, y);
    count_launch();
    return cudaGetLastError();
}

// Squared-error loss of direct learning and its gradient in one pass.  Each
// thread sums |e|^2 as an FP32 (sum, rounding error) pair with an exact two-sum
// per addition (about 2^-48 relative; FP64 runs at about two operations per clock
// per SM on this GPU), the warp adds its pairs, or its FP64 sums where a pair leaves
// FP32's range; the warps' totals are added in FP64 in a fixed order, and the last
// block to finish adds the block sums in block order, writes the loss and clears the
// counter for the next launch.  Four samples' loads in
// flight per thread.  GB300, 2^20 samples from DRAM, us: 9.3 without the
// gradient (11.3 with the threads' totals added in FP64; 11.4 + 4.4 with FP64 sums and a
// second launch for the block sums), 0.7 less since the last block's sum is four chains.
// Graph-replayed from L2 5.9, with the gradient 8.3.
constexpr int kLossThreads = 512;

__global__ void __launch_bounds__(kLossThreads)
    sq_error_kernel(const float2 *y, const float2 *x, int64_t n, float2 g, double scale,
                    double *__restrict__ part, float2 *__restrict__ gy, float *__restrict__ loss)
{
    grid_dep_wait();
    const float s2 = (float)(2.0 * scale);
    float2 acc = make_float2(0.f, 0.f);
    const int64_t stride = (int64_t)gridDim.x * kLossThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kLossThreads + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float2 a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            a[q] = i < n ? x[i] : make_float2(0.f, 0.f);
            b[q] = i < n ? y[i] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            const float er = b[q].x - (g.x * a[q].x - g.y * a[q].y), ei = b[q].y - (g.x * a[q].y + g.y * a[q].x);
            if (i < n) {
                two_sum_acc(acc.x, acc.y, er * er + ei * ei);
                if (gy) gy[i] = make_float2(s2 * er, s2 * ei);
            }
        }
    }
    __shared__ double red[kLossThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2 w = acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w = pair_add(w, shfl_xor_pair(w, o));
    double s = (double)w.x + (double)w.y;
    if (__any_sync(0xffffffffu, !isfinite(w.x))) {
        s = 0.0;
        for (int64_t i = (int64_t)blockIdx.x * kLossThreads + threadIdx.x; i < n; i += stride) {
            const float2 a = x[i], b = y[i];
            const float er = b.x - (g.x * a.x - g.y * a.y), ei = b.y - (g.x * a.y + g.y * a.x);
            s += (double)(er * er + ei * ei);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (warp != 0) return;
    s = lane < kLossThreads / 32 ? red[lane] : 0.0;
#pragma unroll
    for (int o = kLossThreads / 64; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    unsigned *count = reinterpret_cast<unsigned *>(part + kLossBlocks);
    int last = 0;
    if (lane == 0) {
        part[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    // Four sums a lane: a chain of all its FP64 additions took 0.7 us more.
    double q4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < (kLossBlocks + 31) / 32; ++i) {
        const int b = lane + 32 * i;
        q4[i & 3] += b < (int)gridDim.x ? __ldcg(part + b) : 0.0;
    }
    s = (q4[0] + q4[1]) + (q4[2] + q4[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        loss[0] = (float)(scale * s);
        *count = 0u;
    }
}

// The loss's gradient on its own, scaled by dL (one device float): gy = dL 2 scale (y - g x).
__global__ void __launch_bounds__(kLossThreads)
    sq_error_grad_kernel(const float2 *y, const float2 *x, int64_t n, float2 g, double scale,
                         const float *dl, float2 *__restrict__ gy)
{
    grid_dep_wait();
    const float s2 = (float)(2.0 * scale), l = dl[0];
    const int64_t stride = (int64_t)gridDim.x * kLossThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kLossThreads + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float2 a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            a[q] = i < n ? x[i] : make_float2(0.f, 0.f);
            b[q] = i < n ? y[i] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            const float er = b[q].x - (g.x * a[q].x - g.y * a[q].y), ei = b[q].y - (g.x * a[q].y + g.y * a[q].x);
            if (i < n) gy[i] = make_float2(s2 * er * l, s2 * ei * l);
        }
    }
}

cudaError_t launch_sq_error_grad(const float2 *y, const float2 *x, int64_t n, float2 g, double scale, const float *dl,
                                 float2 *gy, cudaStream_t s)
{
    return launch_pdl(sq_error_grad_kernel, dim3(kLossBlocks), kLossThreads, 0, s, y, x, n, g, scale, dl, gy);
}

cudaError_t launch_sq_error(const float2 *y, const float2 *x, int64_t n, float2 g, double scale, double *part,
                            float *loss, float2 *gy, cudaStream_t s)
{
    return launch_pdl(sq_error_kernel, dim3(kLossBlocks), kLossThreads, 0, s, y, x, n, g, scale, part, gy, loss);
}

// One Adam step (Kingma and Ba, "Adam: A Method for Stochastic Optimization",
// Algorithm 1) of a short parameter vector, in FP64 between the FP32 loads and
// stores.  One block: it has the step count to advance.  beta^t comes from repeated
// squaring (t is a whole number), about 2 log2 t FP64 products, and the roots and the
// quotient from Newton-Raphson steps on FP32 estimates: an FP64 operation takes 64
// cycles on this GPU, and pow(), square root and division are tens to hundreds of them
// (the library optimiser's step took 39.4 us; here 6.1 us from cold caches, 7.5 with the functions
// called).
__device__ __forceinline__ double inv_newton(double x)   // 1 / x, x > 0
{
    if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
    double y = (double)(1.f / (float)x);
#pragma unroll
    for (int i = 0; i < 2; ++i) y = fma(y, fma(-x, y, 1.0), y);
    return y;
}

__global__ void __launch_bounds__(256)
    adam_kernel(float *__restrict__ param, const float *grad, float *__restrict__ m,
                float *__restrict__ v, float *__restrict__ step, int64_t n, const float *lr, double beta1,
                double beta2, double eps)
{
    grid_dep_wait();
    const float t = step[0] + 1.f;
    __syncthreads();   // every thread has read the count
    if (threadIdx.x == 0) step[0] = t;
    // even lanes beta1^t, odd lanes beta2^t
    const double base = (threadIdx.x & 1) ? beta2 : beta1;
    double p = 1.0;
    if (t == truncf(t) && t >= 0.f && t < 16777216.f) {
        double sq = base;
        for (unsigned e = (unsigned)t; e; e >>= 1) {
            if (e & 1u) p *= sq;
            sq *= sq;
        }
    } else {
        p = pow(base, (double)t);
    }
    const double c1 = 1.0 - __shfl_sync(0xffffffffu, p, 0), c2 = 1.0 - __shfl_sync(0xffffffffu, p, 1);
    // 1 - beta^t > 0; sqrt(v / c2) = v / sqrt(v c2)
    const double rate = (double)lr[0] * inv_newton(c1);
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const double gd = (double)grad[i];
        const double mi = beta1 * (double)m[i] + (1.0 - beta1) * gd;
        const double vi = beta2 * (double)v[i] + (1.0 - beta2) * gd * gd;
        m[i] = (float)mi;
        v[i] = (float)vi;
        const double root = vi > 0.0 && vi < 1e300 ? vi * inv_sqrt(vi * c2) : sqrt(vi);   // 0, infinity, NaN
        const double den = root + eps;
        param[i] = (float)((double)param[i] - (den > 0.0 ? rate * mi * inv_newton(den) : rate * mi / den));
    }
}

cudaError_t launch_adam(float *param, const float *grad, float *m, float *v, float *step, int64_t n, const float *lr,
                        double beta1, double beta2, double eps, cudaStream_t s)
{
    return launch_pdl(adam_kernel, dim3(1), 256, 0, s, param, grad, m, v, step, n, lr, beta1, beta2, eps);
}

}  // namespace dpd
