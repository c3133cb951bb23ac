// FP64 side of the least-squares estimate (see dpd_gram.cuh): fixed-order
// reduction of the Gram partials, assembly of G = Psi^H Psi and g = Psi^H t, and
// the small kernels of the iterative refinement (factorisation and solves:
// chol_pair.cu).
#include "dpd_device.cuh"
#include "dpd_gram.cuh"

namespace dpd {

// Column sums over the problem's CTAs of the partial P and Q blocks (rows and
// columns < D), in FP64 and a fixed order: SPQ[i][c] for c < 2 kGramS.
constexpr int kReduceGroups = 8;   // partial groups per column, summed by separate warps

__global__ void __launch_bounds__(32 * kReduceGroups) gram_reduce_kernel(const float *__restrict__ partials, int cpp,
                                                                         int D, double *__restrict__ SPQ)
{
    // Lane l of warp g sums partials g, g + 8, g + 16, ... of entry idx in
    // FP64 (four interleaved sums), then warp 0 adds the eight group sums in
    // group order: a fixed order, with up to 19 loads in flight per thread
    // instead of one chain over all partials.
    __shared__ double grp[kReduceGroups][32];
    const int p = blockIdx.y;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int idx = blockIdx.x * 32 + lane;   // i * kGramPartCols + c
    const bool in = idx < kGramS * kGramPartCols;
    const int i = idx / kGramPartCols, c = idx % kGramPartCols, j = c % kGramS;
    double s = 0.0;
    if (in && i < D && j < D) {
        const size_t part = (size_t)kGramRows * kGramPartCols;
        const float *base = partials + (size_t)p * cpp * part + (size_t)i * kGramPartCols + c;
        double s4[4] = {0.0, 0.0, 0.0, 0.0};
        int k = g, q = 0;
        for (; k < cpp; k += kReduceGroups, q = (q + 1) & 3) s4[q] += (double)base[(size_t)k * part];
        s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    }
    grp[g][lane] = s;
    __syncthreads();
    if (g == 0 && in) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kReduceGroups; ++q) t += grp[q][lane];
        SPQ[(size_t)p * kGramS * kGramPartCols + idx] = t;
    }
}

cudaError_t launch_gram_reduce(const float *partials, int nprob, int cpp, int D, double *S, cudaStream_t s)
{
    dim3 grid((kGramS * kGramPartCols + 31) / 32, nprob);
    gram_reduce_kernel<<<grid, 32 * kReduceGroups, 0, s>>>(partials, cpp, D, S);
    count_launch();
    return cudaGetLastError();
}

// Power sums of r = |u|^2, NK = 2 B - 1 of them.  Each thread sums its powers as
// FP32 pairs (sum, rounding error) with an exact two-sum per addition: FP32
// arithmetic, about 2^-48 relative accuracy, where FP64 additions (about two per
// clock per SM on GB300) bound the kernel.  The pairs stay FP32 up to the warp's
// sum and become FP64 there (before it, if that sum leaves FP32's range).  Eight FP32 operations per sample and power bound
// it, and the block's sum costs a thread as much as 16 samples: three blocks per
// SM, four samples' loads in flight per thread.
// GB300, 2^22 samples, NK = 11: 23.5 us (64 blocks, one load at a time and an
// FP64 tree per block: 138.4).
constexpr int kMomThreads = 256;

template <int NK>
__global__ void __launch_bounds__(kMomThreads) moments_kernel(const GramProblem *__restrict__ probs, GramProblem one,
                                                              double *__restrict__ part)
{
    const GramProblem pr = probs ? probs[blockIdx.y] : one;
    float2 sum[NK];   // (sum, error)
#pragma unroll
    for (int k = 0; k < NK; ++k) sum[k] = make_float2(0.f, 0.f);
    const int64_t stride = (int64_t)gridDim.x * kMomThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kMomThreads + threadIdx.x; i0 < pr.n; i0 += 4 * stride) {
        float2 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            x[q] = i < pr.n ? pr.u[i] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float r = fmaf(x[q].x, x[q].x, x[q].y * x[q].y);
            float p = r;
#pragma unroll
            for (int k = 0; k < NK; ++k) {
                two_sum_acc(sum[k].x, sum[k].y, p);
                p *= r;
            }
        }
    }
    __shared__ double red[kMomThreads / 32][NK];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        float2 v = sum[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = pair_add(v, shfl_xor_pair(v, o));
        double d = (double)v.x + (double)v.y;
        if (__any_sync(0xffffffffu, !isfinite(v.x))) {
            d = (double)sum[k].x + (double)sum[k].y;
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        if (lane == 0) red[warp][k] = d;
    }
    __syncthreads();
    if (threadIdx.x < NK) {
        double d = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < kMomThreads / 32; ++w) d += red[w][threadIdx.x];
        part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kMomK + threadIdx.x] = d;
    }
}

// Basis of statistically orthogonal polynomials (Sec. 2.1) of a problem per block.
// Power sums mu_k: one warp per power, lane l adds blocks l, l + 32, ... in order, then a
// fixed shuffle tree.  Then one warp: the moment matrix M[a][b] = mu_{a+b+1} / n is the
// Gram matrix of the monomials |u|^{2a} u; M = L L^T (lane i holds row i) and U = L^{-T}
// (lane b solves for column b) make sum_a U[a][b] |u|^{2a} u orthonormal.  U is rounded
// to FP32 for the Gram kernels and the same values are kept in FP64 for the coefficient
// transforms.  A moment matrix that is not positive definite gives the monomials (U = I).
// FP64's latency (64 cycles) bounds it: 13 us; a kernel for the sums, two copies, two
// synchronisations and the same factorisation on the host took about 45.
__global__ void __launch_bounds__(32 * kMomK) basis_kernel(const GramProblem *probs, GramProblem one,
                                                           const double *part, int blocks, int B,
                                                           float *__restrict__ ubasis, double *__restrict__ ubasis64)
{
    __shared__ double mu[kMomK], L[kMaxB][kMaxB], rinv[kMaxB];
    grid_dep_wait();
    const int p = blockIdx.x, k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
    if (k < 2 * B - 1) {
#pragma unroll 4
        for (int b = lane; b < blocks; b += 32) s += part[((size_t)p * blocks + b) * kMomK + k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) mu[k] = s / (double)(probs ? probs[p].n : one.n);
    __syncthreads();
    if (k != 0) return;
    const int i = lane;
    double row[kMaxB];
#pragma unroll
    for (int j = 0; j < kMaxB; ++j) row[j] = i < B && j < B ? mu[i + j] : 0.0;
    bool spd = true;
#pragma unroll
    for (int j = 0; j < kMaxB; ++j)
        if (j < B && spd) {
            const double piv = __shfl_sync(0xffffffffu, row[j], j);
            spd = piv > 0.0 && isfinite(piv);
            const double r = spd ? inv_sqrt(piv) : 0.0;
            const double l = row[j] * r;
            if (i >= j && i < B) L[i][j] = l;
            if (i == j) rinv[j] = r;
#pragma unroll
            for (int q = j + 1; q < kMaxB; ++q) row[q] = fma(-l, __shfl_sync(0xffffffffu, l, q), row[q]);
        }
    __syncwarp();
    double u[kMaxB];   // column i of U
#pragma unroll
    for (int a = kMaxB - 1; a >= 0; --a) {
        u[a] = 0.0;
        if (a < B && i < B) {
            double v = a == i ? 1.0 : 0.0;
            if (spd) {
#pragma unroll
                for (int q = a + 1; q < kMaxB; ++q)
                    if (q < B) v = fma(-L[q][a], u[q], v);
                v *= rinv[a];
            }
            u[a] = v;
        }
    }
    if (i < kMaxB)
#pragma unroll
        for (int a = 0; a < kMaxB; ++a) {
            const size_t at = (size_t)p * kUSize + a * kMaxB + i;
            ubasis[at] = (float)u[a];
            ubasis64[at] = (double)(float)u[a];
        }
}

cudaError_t launch_basis(const GramProblem *probs, GramProblem one, int nprob, int64_t nmax, int B, double *part,
                         float *ubasis, double *ubasis64, cudaStream_t s)
{
    // At least a thousand samples (four per thread) a block.
    const int64_t need = (nmax + 4 * kMomThreads - 1) / (4 * kMomThreads);
    const int blocks = (int)(need < moments_blocks(nprob) ? need : moments_blocks(nprob));
    const dim3 grid((unsigned)blocks, (unsigned)nprob);
    switch (B) {
    case 1: moments_kernel<1><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    case 2: moments_kernel<3><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    case 3: moments_kernel<5><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    case 4: moments_kernel<7><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    case 5: moments_kernel<9><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    case 6: moments_kernel<11><<<grid, kMomThreads, 0, s>>>(probs, one, part); break;
    default: return cudaErrorInvalidValue;
    }
    count_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_pdl(basis_kernel, dim3((unsigned)nprob), 32 * kMomK, 0, s, probs, one, part, blocks, B, ubasis,
                      ubasis64);
}

// <x, y> for two signed distinct-column references: S = P + Q + Q^T from the
// summed blocks (P upper triangle in columns [0, kGramS), Q in [kGramS, 2 kGramS)).
__device__ __forceinline__ double dot(const double *SPQ, ColRef x, ColRef y)
{
    if (x.sign == 0 || y.sign == 0) return 0.0;
    const int i = x.d < y.d ? x.d : y.d, j = x.d < y.d ? y.d : x.d;
    const double v = SPQ[(size_t)i * kGramPartCols + j] + SPQ[(size_t)i * kGramPartCols + kGramS + j] +
                     SPQ[(size_t)j * kGramPartCols + kGramS + i];
    return x.sign * y.sign > 0 ? v : -v;
}

__global__ void gram_assemble_kernel(const double *__restrict__ Sall, int K, int Bp, int B, int T,
                                     double2 *__restrict__ G, double2 *__restrict__ g, double *__restrict__ tt,
                                     double2 *Ghost)
{
    const int p = blockIdx.y;
    const double *S = Sall + (size_t)p * kGramS * kGramPartCols;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const ColRef tre{2 * B * T + 1, 1}, tim{2 * B * T + 2, 1};
    if (idx < K * K) {
        const int a = idx / K, b = idx % K;
        ColRef ar, ai, br, bi;
        psi_column_refs(a, K, Bp, B, T, ar, ai);
        psi_column_refs(b, K, Bp, B, T, br, bi);
        const double2 v = make_double2(dot(S, ar, br) + dot(S, ai, bi), dot(S, ar, bi) - dot(S, ai, br));
        G[(size_t)p * K * K + idx] = v;
        if (Ghost && p == 0) Ghost[idx] = v;
    } else if (idx < K * K + K) {
        const int a = idx - K * K;
        ColRef ar, ai;
        psi_column_refs(a, K, Bp, B, T, ar, ai);
        if (g) g[(size_t)p * K + a] = make_double2(dot(S, ar, tre) + dot(S, ai, tim), dot(S, ar, tim) - dot(S, ai, tre));
    } else if (idx == K * K + K) {
        if (tt) tt[p] = dot(S, tre, tre) + dot(S, tim, tim);
    }
}

cudaError_t launch_gram_assemble(const double *S, int nprob, int K, int Bp, int B, int T, double2 *G, double2 *g,
                                 double *tt, double2 *Ghost, cudaStream_t s)
{
    dim3 grid((K * K + K + 1 + 255) / 256, nprob);
    gram_assemble_kernel<<<grid, 256, 0, s>>>(S, K, Bp, B, T, G, g, tt, Ghost);
    count_launch();
    return cudaGetLastError();
}

__global__ void residual_kernel(const float2 *__restrict__ t, const float2 *__restrict__ y, int64_t n,
                                float2 *__restrict__ e)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 a = t[i], b = y[i];
        e[i] = make_float2(a.x - b.x, a.y - b.y);
    }
}

cudaError_t launch_residual(const float2 *t, const float2 *y, int64_t n, float2 *e, cudaStream_t s)
{
    int64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) return cudaSuccess;
    residual_kernel<<<(unsigned)blocks, 256, 0, s>>>(t, y, n, e);
    count_launch();
    return cudaGetLastError();
}

constexpr int kNormBlocks = 1024;
static_assert(kNormBlocks <= kFwdNormSlots, "partial pairs of the statistics pass");

__global__ void sum_pairs_kernel(const double *__restrict__ part, int nb, double *__restrict__ out)
{
    __shared__ double sa[256], sb[256];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        a += part[2 * i];
        b += part[2 * i + 1];
    }
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sa[threadIdx.x] += sa[threadIdx.x + o];
            sb[threadIdx.x] += sb[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sa[0];
        out[1] = sb[0];
    }
}

// Residual and both sums of squares in one pass: e = t - y (when e is not
// null), and per block sum |e|^2 and sum |t|^2, then one fixed-order final sum
// (sum_pairs_kernel).  The squares of the FP32 samples are formed and summed
// in FP32 over the four samples of a pass, and the passes are added in FP64
// (FP64 arithmetic on this GPU is a small fraction of the FP32 rate).
__global__ void residual_norm_kernel(const float2 *__restrict__ t, const float2 *__restrict__ y, int64_t n,
                                     float2 *__restrict__ e, double *__restrict__ part)
{
    // Four samples per thread and pass (all loads issued before any use);
    // e is written only when requested.
    __shared__ double se[256], st[256];
    double a = 0.0, b = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float2 tv[4], yv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            tv[q] = i < n ? t[i] : make_float2(0.f, 0.f);
            yv[q] = i < n ? y[i] : make_float2(0.f, 0.f);
        }
        float a32 = 0.f, b32 = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 ev = make_float2(tv[q].x - yv[q].x, tv[q].y - yv[q].y);
            const int64_t i = i0 + q * stride;
            if (e && i < n) e[i] = ev;
            a32 = fmaf(ev.x, ev.x, fmaf(ev.y, ev.y, a32));
            b32 = fmaf(tv[q].x, tv[q].x, fmaf(tv[q].y, tv[q].y, b32));
        }
        a += (double)a32;
        b += (double)b32;
    }
    se[threadIdx.x] = a;
    st[threadIdx.x] = b;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            se[threadIdx.x] += se[threadIdx.x + o];
            st[threadIdx.x] += st[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = se[0];
        part[2 * blockIdx.x + 1] = st[0];
    }
}

cudaError_t launch_residual_norm(const float2 *t, const float2 *y, int64_t n, float2 *e, double *part, double *out,
                                 cudaStream_t s)
{
    residual_norm_kernel<<<kNormBlocks, 256, 0, s>>>(t, y, n, e, part);
    count_launch();
    sum_pairs_kernel<<<1, 256, 0, s>>>(part, kNormBlocks, out);
    count_launch();
    return cudaGetLastError();
}


}  // namespace dpd
