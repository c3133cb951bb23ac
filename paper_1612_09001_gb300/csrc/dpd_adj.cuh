// Adjoint of the APH DPD filter: gradients of a real loss L through y = DPD(x)
// with respect to the input samples and the coefficients, given gy = dL/dy,
// all under the convention grad = dL/dRe + j dL/dIm.
//
// With r = |x|^2, branch polynomials A_k(r) = sum_b h_{2b+1,k} r^b and
// C_k(r) = sum_b hbar_{2b+1,k} r^b (so that y_n = sum_k A_k(r_{n-k}) x_{n-k}
// + C_k(r_{n-k}) conj(x_{n-k}) + c, Eq. 1), the Wirtinger derivatives of the
// term of tap k are
//   dy/dx       = E_k(r) + G_k(r) conj(x)^2,   E = A + r A',  G = C'
//   dy/dconj(x) = F_k(r) x^2 + H_k(r),         F = A',        H = C + r C'
// and
//   gx_i = sum_k conj(dy_{i+k}/dx_i) gy_{i+k} + (dy_{i+k}/dconj(x_i)) conj(gy_{i+k})
//        = sum_k [conj(E_k) g + H_k conj(g)] + x_i^2 [conj(G_k) g + F_k conj(g)],  g = gy_{i+k}
// Each bracket is widely linear in g, so it is evaluated like the forward
// filter: four real Horner polynomials per bracket, run as two packed f32x2
// Horner chains whose results multiply the window sample {c, d} and its swap
// {d, c} (table built by wl_table_kernel, one float4 per power).
//
// The coefficient gradient is the correlation
//   gh_{(p,k)} = sum_j r_j^b conj(x_j) gy_{j+k},  gh_{(q,k)} = sum_j r_j^b x_j gy_{j+k},
//   gh_c = sum_n gy_n,
// i.e. conj(Psi)^T gy with the basis matrix Psi of Eq. 2.  Both branches come
// from two packed real correlations per (power, tap) (gh_accumulate), taken
// per thread over groups of up to five taps, reduced per CTA in a fixed order
// into a partials workspace and summed over CTAs in FP64 by
// adj_finalize_kernel.  The basis is recomputed from x: nothing from the
// forward pass is stored.
//
// Data movement.  For 16-byte aligned x and gy both gradients run as kernels
// whose warps work on their own: every warp has its share of the record's
// units and a ring of shared-memory slots that its lane 0 fills with bulk
// copies of x and gy (plus the look-ahead) completed on the warp's own
// mbarriers, so no warp waits for another one until the final reduction.
// Other alignments (and callers without an error word) use the plain-load
// kernels, which read through L1.
//
// Rounding.  The forms above and the order of the FP32 sums are fixed: training's
// first Adam step divides a gradient element by its own size plus eps, so where an
// element is nearly zero (the constant's, at the identity) its rounding becomes a
// visible part of the step.  A split of the coefficient gradient's samples over
// other threads, with gx as one FIR per power of r and the features' derivative
// after it (120 instead of 184 multiply-adds at B = T = 5), was as accurate but
// moved the outputs of the fourth step by up to 2.7e-4 on inputs whose first gradient of
// the constant is below 2e-7; in this order they stay within 2e-6.
#pragma once

#include "dpd_device.cuh"
#include "dpd_internal.h"

namespace dpd {

constexpr int kAdjV = 4;          // samples per thread and unit
constexpr int kAdjUnit = 32 * kAdjV;   // samples of a warp's work unit
constexpr int kAdjWarps = 8;      // warps per CTA of the staged gx kernel
constexpr int kAdjStages = 2;     // ring slots per warp of the staged gx kernel
// Units per slot of the staged gx kernel: with one power of r a unit has too little
// arithmetic to cover its copies.
constexpr int adj_sub(int B) { return B == 1 ? 4 : 1; }
constexpr int kAdjGhWarps = 12;   // warps per CTA of the staged gh kernel (about 165 registers per thread)
constexpr int kAdjGhStages = 2;   // ring slots per warp of the staged gh kernel
constexpr int kAdjGhSub = 4;      // units per slot of the staged gh kernel
// Measured on GB300, graph-replayed, us at 2^23 + 4097 / 2^20 samples.
// gx, P = Q = 9, M = 4 and P = Q = 7, M = 3 (CTAs per SM, slots x units): 3, 2 x 1
// 54.4 / 8.4 and 40.5 / 6.4; 2, 2 x 1 56.6 / 8.5 and 39.9 / 6.4; 2, 2 x 2 56.8 / 8.6
// and 41.2 / 6.7; 2, 4 x 1 53.7 / 8.4 and 42.4 / 6.5; 3, 3 x 1 55.0 / 8.4 and 41.5 /
// 6.6; 4 (64 registers, spills) 64.4 / 10.2 and 47.5 / 8.0.  The FMA pipe bounds the
// first (28.5 T FMA/s), traffic the second (4.97 TB/s).  With a ring shared by the CTA's
// warps and a producer warp: 53.8 / 9.3 and 41.2 / 7.4.  P = Q = 1, M = 0 at 2^22 / 2^24:
// 4 units a slot 8.6 / 62.7, 2 8.9 / 63.1, 1 17.5 / 66.8 (that ring 10.3 / 63.1).
// gh with its final sum, P = Q = 9, M = 4 and P = Q = 7, M = 3: 41.4 / 14.1 and 32.5 /
// 11.8; with a ring shared by the CTA's warps, whose slots waited for the slowest
// warp, 46.0 / 18.6 and 35.3 / 14.8.  At 2^20 the 171 tiles on 152 CTAs take two rounds
// (10.7 with the record cut evenly over the warps, a split with other sums).

// NS consecutive complex samples p[base .. base+NS-1] (zero past n).  When the
// buffer is 16-byte aligned, base is even and the rounded-up window lies inside
// the buffer, they are fetched as float4 pairs; otherwise sample by sample.
template <int NS>
__device__ __forceinline__ void adj_load_window(const float2 *__restrict__ p, int64_t base, int64_t n,
                                                bool vec, float2 (&out)[NS])
{
    constexpr int NV = (NS + 1) / 2;
    if (vec && (base & 1) == 0 && base + 2 * NV <= n) {
        const float4 *q = reinterpret_cast<const float4 *>(p + base);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            const float4 t = __ldg(q + j);
            out[2 * j] = make_float2(t.x, t.y);
            if (2 * j + 1 < NS) out[2 * j + 1] = make_float2(t.z, t.w);
        }
    } else {
#pragma unroll
        for (int j = 0; j < NS; ++j) out[j] = base + j < n ? __ldg(p + base + j) : make_float2(0.f, 0.f);
    }
}

// NS samples of a shared-memory slot from element `off`: float4 pairs when off
// is even (the slot holds the rounded-up window), else one by one.
template <int NS>
__device__ __forceinline__ void adj_slot_window(const float2 *slot, int off, float2 (&out)[NS])
{
    if ((off & 1) == 0) {
        const float4 *q = reinterpret_cast<const float4 *>(slot + off);
#pragma unroll
        for (int j = 0; j < (NS + 1) / 2; ++j) {
            const float4 t = q[j];
            out[2 * j] = make_float2(t.x, t.y);
            if (2 * j + 1 < NS) out[2 * j + 1] = make_float2(t.z, t.w);
        }
    } else {
#pragma unroll
        for (int j = 0; j < NS; ++j) out[j] = slot[off + j];
    }
}

// ---------------------------------------------------------------- warp rings
// The record is cut into units of kAdjUnit samples.  For the input gradient every
// warp of a launch takes a contiguous run of them, equal to within one unit: warp w of W takes
// units [first, first + count).  Consecutive w sit on different CTAs, so a short
// record spreads over the SMs.  (A run of 2^31 units would be 2 TB of samples.)
__device__ __forceinline__ int64_t warp_share(int64_t units, int w, int W, int &count)
{
    const int64_t q = units / W;
    const int r = (int)(units - q * W);
    count = (int)q + (w < r ? 1 : 0);
    return w * q + (w < r ? w : r);
}

// The gh kernels read the window of taps k0 .. k0 + TG - 1 with k0 <= T - 1, so
// their look-ahead reaches T + TG - 2 samples (+1 for the float4 rounding).
constexpr int kAdjGhMaxTG = 5;
constexpr int kAdjGhHalo = kMaxT + kAdjGhMaxTG - 1;
static_assert(kAdjGhHalo % 2 == 0 && kHalo % 2 == 0, "slot parts must stay 16-byte aligned");

// NS samples from element `off` of a tile whose slot holds the first `cnt` of
// the `left` samples that the record has from the tile's start (src) on.
template <int NS>
__device__ __forceinline__ void adj_slot_window_tail(const float2 *slot, int cnt, const float2 *src,
                                                     int off, int64_t left, float2 (&out)[NS])
{
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const int g = off + j;
        float2 v = make_float2(0.f, 0.f);
        if (g < cnt)
            v = slot[g];
        else if (g < left)
            v = src[g];
        out[j] = v;
    }
}

// One warp's ring over a contiguous share of the record (the input gradient):
// STAGES slots of SUB units; a slot holds x[s0, s0 + S) and, from element S on,
// gy[s0, s0 + S + HALO), S = SUB * kAdjUnit (less at the end of the warp's share
// and of the record, where only the even-length prefix that exists is copied).  Lane 0 issues the copies of tile i + STAGES once the whole
// warp has read tile i (its windows are in registers): the warp is producer and
// consumer, so the slot needs a "full" barrier only.
template <int STAGES, int SUB, int HALO>
struct AdjRing {
    static constexpr int S = SUB * kAdjUnit;
    static constexpr int kSlotElems = 2 * S + HALO;
    static constexpr size_t kBytes = (size_t)STAGES * kSlotElems * sizeof(float2);   // per warp

    const float2 *x, *gy;   // at the first sample of the warp's share
    int64_t left;           // samples of the record from there on
    float2 *slots;          // this warp's slots
    uint32_t bars;          // shared-memory address of its STAGES barriers
    int units;              // units in the share
    int tiles;              // tiles of SUB units (the last may be shorter)
    int whole;              // the first `whole` tiles lie, with their look-ahead, inside the record
    int plain;              // the first `plain` of those have SUB units

    // Share of warp w of W; returns its first sample.
    __device__ __forceinline__ int64_t init(const AdjArgs &a, int64_t total_units, int w, int W, unsigned char *mem,
                                            uint32_t bar_addr, int lane)
    {
        const int64_t s0 = warp_share(total_units, w, W, units) * kAdjUnit;
        x = a.x + s0;
        gy = a.gy + s0;
        left = a.n - s0;
        slots = reinterpret_cast<float2 *>(mem);
        bars = bar_addr;
        tiles = (units + SUB - 1) / SUB;
        const int64_t f = left >= HALO ? (left - HALO) / S : 0;
        whole = f < tiles ? (int)f : tiles;
        plain = whole < units / SUB ? whole : units / SUB;
        if (lane == 0) {
            for (int s = 0; s < STAGES; ++s) mbar_init(bars + 8u * s, 1);
            fence_barrier_init();
            for (int i = 0; i < STAGES && i < tiles; ++i) issue(i);
        }
        __syncwarp();
        return s0;
    }
    __device__ __forceinline__ int units_of(int i) const { return units - i * SUB < SUB ? units - i * SUB : SUB; }
    // Samples of x and gy that the slot of tile i holds.
    __device__ __forceinline__ void counts(int i, int &xc, int &gc) const
    {
        const int want = units_of(i) * kAdjUnit;
        xc = want;
        gc = want + HALO;
        if (i >= whole) {
            const int64_t rem = left - (int64_t)i * S;
            xc = (int)(rem < xc ? rem : (int64_t)xc) & ~1;
            gc = (int)(rem < gc ? rem : (int64_t)gc) & ~1;
        }
    }
    __device__ __forceinline__ float2 *slot(int i) const { return slots + (i % STAGES) * kSlotElems; }
    __device__ __forceinline__ void copy(int i, uint32_t xbytes, uint32_t gbytes)
    {
        const uint32_t fb = bars + 8u * (i % STAGES), dst = smem_addr(slot(i));
        mbar_arrive_expect_tx(fb, xbytes + gbytes);
        if (xbytes) bulk_copy_g2s(dst, x + (int64_t)i * S, xbytes, fb);
        if (gbytes) bulk_copy_g2s(dst + S * (uint32_t)sizeof(float2), gy + (int64_t)i * S, gbytes, fb);
    }
    __device__ __forceinline__ void issue(int i)   // lane 0
    {
        if (i < plain) {
            copy(i, S * (uint32_t)sizeof(float2), (S + HALO) * (uint32_t)sizeof(float2));
        } else {
            int xc, gc;
            counts(i, xc, gc);
            copy(i, (uint32_t)xc * (uint32_t)sizeof(float2), (uint32_t)gc * (uint32_t)sizeof(float2));
        }
    }
    // One outcome for the whole warp, whose lanes issue and reduce together.
    __device__ __forceinline__ bool wait(int i, int *status) const
    {
        return __all_sync(0xffffffffu, mbar_wait(bars + 8u * (i % STAGES), (uint32_t)((i / STAGES) & 1), status));
    }
    // The whole warp has read tile i: refill its slot.
    __device__ __forceinline__ void refill(int i, int lane)
    {
        __syncwarp();
        if (lane == 0 && i + STAGES < tiles) {
            fence_proxy_async_smem();   // the reads above precede the copy's writes
            issue(i + STAGES);
        }
    }
    // After a failed wait on tile i: let the copies in flight land.
    __device__ __forceinline__ void drain(int i, int *status) const
    {
        for (int q = i; q < i + STAGES && q < tiles; ++q) wait(q, status);
    }
    // The window of NX samples of x and NG of gy (from k0 on) of element off of tile i.
    template <int NX, int NG>
    __device__ __forceinline__ void window(int i, int off, int k0, float2 (&xs)[NX], float2 (&g)[NG]) const
    {
        const float2 *sl = slot(i);
        if (i < whole) {
            adj_slot_window<NX>(sl, off, xs);
            adj_slot_window<NG>(sl + S, off + k0, g);
        } else {
            int xc, gc;
            counts(i, xc, gc);
            const int64_t at = (int64_t)i * S;
            adj_slot_window_tail<NX>(sl, xc, x + at, off, left - at, xs);
            adj_slot_window_tail<NG>(sl + S, gc, gy + at, off + k0, left - at, g);
        }
    }
};

// Shared-memory bytes of a staged kernel: barriers, scratch (coefficient table
// or reduction rows), the rings of its warps.
template <class Ring>
__host__ __device__ constexpr size_t adj_staged_smem(int warps, int scratch_floats)
{
    return 512 + (((size_t)scratch_floats * 4 + 127) / 128) * 128 + (size_t)warps * Ring::kBytes;
}

// ---------------------------------------------------------------- input gradient
// Adjoint table passed by value (kernel parameter bank), 16-byte aligned so
// that its packed pairs can be 64-bit constant operands.
template <int B, int T>
struct alignas(16) AdjParamTab {
    float v[adj_table_floats(B, T)];
};

// gx for the V samples i0.. from their x (xs) and the gy window g (samples
// i0 .. i0 + V + T - 2).  The adjoint table of the model comes from shared
// memory (tab) or, with PARAM, from the parameter bank (ptab), whose entries
// the packed FMAs take as operands directly.
template <int B, int T, int V, bool PARAM = false>
__device__ __forceinline__ void gx_compute(const float *tab, const AdjParamTab<B, T> &ptab,
                                           const float2 (&xs)[V], const float2 (&g)[V + T - 1], float2 (&acc)[V])
{
    constexpr int QB = B, RB = B - 1;       // coefficients per Q / S polynomial
    constexpr int PER_TAP = 4 * QB + 4 * RB;
    constexpr int W = V + T - 1;
    float2 gs[W];   // window samples swapped: {d, c}
#pragma unroll
    for (int j = 0; j < W; ++j) gs[j] = make_float2(g[j].y, g[j].x);
    float ur[V], ui[V], rr[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float2 q = xs[v];
        rr[v] = fmaf(q.x, q.x, q.y * q.y);
        ur[v] = fmaf(q.x, q.x, -q.y * q.y);   // x^2
        ui[v] = 2.f * q.x * q.y;
    }
    // {Re, Im} of the gradient of each sample, and of the tap sum of the second
    // bracket (its factor x^2 does not depend on the tap, so it is applied once
    // after the tap loop).  Every tap advances all V samples together with
    // packed f32x2 FMAs (coefficient pairs adjacent in the table).
    float2 ws[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        acc[v] = make_float2(0.f, 0.f);
        ws[v] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < T; ++k) {
        // quadruple j of tap k's block: the Q quadruples, then the S ones
        auto coef = [&](int j) -> float4 {
            if constexpr (PARAM) {
                const int o = PER_TAP * k + 4 * j;
                return make_float4(ptab.v[o], ptab.v[o + 1], ptab.v[o + 2], ptab.v[o + 3]);
            } else {
                return reinterpret_cast<const float4 *>(tab + PER_TAP * k)[j];
            }
        };
        float2 pa[V], pb[V];
        {
            const float4 c4 = coef(QB - 1);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                pa[v] = make_float2(c4.x, c4.y);
                pb[v] = make_float2(c4.z, c4.w);
            }
        }
#pragma unroll
        for (int m = QB - 2; m >= 0; --m) {
            const float4 c4 = coef(m);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float2 rr2 = make_float2(rr[v], rr[v]);
                pa[v] = __ffma2_rn(pa[v], rr2, make_float2(c4.x, c4.y));
                pb[v] = __ffma2_rn(pb[v], rr2, make_float2(c4.z, c4.w));
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            acc[v] = __ffma2_rn(pa[v], g[v + k], acc[v]);    // {Q0 c, Q3 d}
            acc[v] = __ffma2_rn(pb[v], gs[v + k], acc[v]);   // {Q1 d, Q2 c}
        }
        if constexpr (RB > 0) {
            float2 sa[V], sb[V];
            {
                const float4 c4 = coef(QB + RB - 1);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    sa[v] = make_float2(c4.x, c4.y);
                    sb[v] = make_float2(c4.z, c4.w);
                }
            }
#pragma unroll
            for (int m = RB - 2; m >= 0; --m) {
                const float4 c4 = coef(QB + m);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float2 rr2 = make_float2(rr[v], rr[v]);
                    sa[v] = __ffma2_rn(sa[v], rr2, make_float2(c4.x, c4.y));
                    sb[v] = __ffma2_rn(sb[v], rr2, make_float2(c4.z, c4.w));
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                // conj(G) g + F conj(g) = {S0 c + S1 d, S2 c + S3 d}
                ws[v] = __ffma2_rn(sa[v], g[v + k], ws[v]);    // {S0 c, S3 d}
                ws[v] = __ffma2_rn(sb[v], gs[v + k], ws[v]);   // {S1 d, S2 c}
            }
        }
    }
    if constexpr (RB > 0) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            // acc += x^2 ws (complex):  {ur wr - ui wi, ur wi + ui wr}
            acc[v] = __ffma2_rn(make_float2(ur[v], ur[v]), ws[v], acc[v]);
            acc[v] = __ffma2_rn(make_float2(-ui[v], ui[v]), make_float2(ws[v].y, ws[v].x), acc[v]);
        }
    }
}

template <int V>
__device__ __forceinline__ void gx_store(float2 *__restrict__ gx, int64_t i0, int64_t n, bool vec,
                                         const float2 (&acc)[V], bool streaming)
{
    if (vec && i0 + V <= n) {
        float4 *o = reinterpret_cast<float4 *>(gx + i0);
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const float4 q = make_float4(acc[2 * j].x, acc[2 * j].y, acc[2 * j + 1].x, acc[2 * j + 1].y);
            if (streaming)
                st_stream_f4(o + j, q);
            else
                o[j] = q;
        }
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (i0 + v < n) gx[i0 + v] = acc[v];
    }
}

template <int B, int T>
__host__ __device__ constexpr int adj_tab_padded() { return ((adj_table_floats(B, T) + 3) / 4) * 4; }

// Plain-load variant (any 8-byte alignment): grid-stride over V-sample runs.
template <int B, int T, int V>
__global__ void __launch_bounds__(256) adj_gx_kernel(AdjArgs a)
{
    constexpr int W = V + T - 1;            // gy window: samples i0 .. i0 + V + T - 2
    constexpr int TABF = adj_table_floats(B, T);
    __shared__ __align__(16) float tab[adj_tab_padded<B, T>()];
    for (int i = threadIdx.x; i < TABF; i += blockDim.x) tab[i] = a.adj_tab[i];
    __syncthreads();

    static_assert(V % 2 == 0, "V samples are stored as float4 pairs");
    const bool vec_in = ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.gy)) & 15) == 0;
    const bool vec_out = (reinterpret_cast<uintptr_t>(a.gx) & 15) == 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * V;
    for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V; i0 < a.n; i0 += stride) {
        float2 xs[V], g[W], acc[V];
        adj_load_window<V>(a.x, i0, a.n, vec_in, xs);
        adj_load_window<W>(a.gy, i0, a.n, vec_in, g);
        gx_compute<B, T, V>(tab, *reinterpret_cast<const AdjParamTab<B, T> *>(tab), xs, g, acc);
        gx_store<V>(a.gx, i0, a.n, vec_out, acc, false);
    }
}

template <int B>
using GxRing = AdjRing<kAdjStages, adj_sub(B), kHalo>;

// Staged variant: CTAs of kAdjWarps independent warps (see AdjRing).  x and gy
// 16-byte aligned.
template <int B, int T, int V, bool PARAM>
__global__ void __launch_bounds__(32 * kAdjWarps, 3)
    adj_gx_tma_kernel(AdjArgs a, int64_t units, const __grid_constant__ AdjParamTab<B, T> ptab)
{
    constexpr int W = V + T - 1;
    constexpr int TABF = adj_table_floats(B, T);
    using Ring = GxRing<B>;
    constexpr int S = Ring::S;
    static_assert(T - 1 <= kHalo && V == kAdjV, "look-ahead must fit the slot");
    static_assert(kAdjWarps * kAdjStages * 8 <= 512, "barrier area");
    extern __shared__ __align__(128) unsigned char smem[];
    float *tab = reinterpret_cast<float *>(smem + 512);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    grid_dep_wait();
    Ring ring;
    const int64_t f0 = ring.init(a, units, warp * gridDim.x + blockIdx.x, kAdjWarps * gridDim.x,
                                 smem + adj_staged_smem<Ring>(warp, adj_tab_padded<B, T>()),
                                 smem_addr(smem) + 8u * kAdjStages * warp, lane);
    if constexpr (!PARAM) {
        for (int i = tid; i < TABF; i += 32 * kAdjWarps) tab[i] = a.adj_tab[i];
        __syncthreads();
    }
    const bool vec_out = (reinterpret_cast<uintptr_t>(a.gx) & 15) == 0;
    for (int i = 0; i < ring.tiles; ++i) {
        if (!ring.wait(i, a.status)) {
            ring.drain(i, a.status);
            return;
        }
        const int nu = ring.units_of(i);
#pragma unroll 1
        for (int j = 0; j < nu; ++j) {
            const int off = j * kAdjUnit + lane * V;
            float2 xs[V], g[W];
            ring.window(i, off, 0, xs, g);
            if (j == nu - 1) ring.refill(i, lane);
            float2 acc[V];
            gx_compute<B, T, V, PARAM>(tab, ptab, xs, g, acc);
            gx_store<V>(a.gx, f0 + (int64_t)i * S + off, a.n, vec_out, acc, true);
        }
    }
}

// ---------------------------------------------------------------- coefficient gradient
// Tap groups: group y owns taps [y*TG, y*TG + TG) of every branch; group 0 also
// owns the LO-leakage term.  Each CTA writes one row of partials (K complex),
// only at the indices of its group.
//
// With a_b = r^b Re x, c_b = r^b Im x and g = gy_{j+k} = c + j d, both branches
// follow from two packed correlations per (b, k):
//   X_{b,k} = sum_j {a_b, c_b}_j * {c, d},   Y_{b,k} = sum_j {a_b, c_b}_j * {d, c},
//   main  sum r^b conj(x) g = {X.x + X.y, Y.x - Y.y},
//   conj  sum r^b x g       = {X.x - X.y, Y.x + Y.y},
// so every (sample, b, tap) costs two packed f32x2 FMAs whose operands are the
// packed power {a_b, c_b} and the window sample as stored or swapped (once per
// window sample): no per-product broadcasts.  Accumulators per thread:
// [b*TG + kk] X, [B*TG + b*TG + kk] Y, last sum g (for c).
template <int B, int TG, int V>
__device__ __forceinline__ void gh_accumulate(const float2 (&xs)[V], const float2 (&g)[V + TG - 1], bool group0,
                                              float2 (&acc2)[2 * B * TG + 1])
{
    constexpr int NP = 2 * B * TG + 1;
    constexpr int NG = V + TG - 1;
    if (group0) {
#pragma unroll
        for (int v = 0; v < V; ++v)   // the gy window starts at the sample itself for group 0
            acc2[NP - 1] = __fadd2_rn(acc2[NP - 1], g[v]);
    }
    float2 gs[NG];
#pragma unroll
    for (int j = 0; j < NG; ++j) gs[j] = make_float2(g[j].y, g[j].x);
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float r = fmaf(xs[v].x, xs[v].x, xs[v].y * xs[v].y);
        float2 p = xs[v];   // {a_b, c_b}
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (b > 0) p = __fmul2_rn(p, make_float2(r, r));
#pragma unroll
            for (int kk = 0; kk < TG; ++kk) {
                acc2[b * TG + kk] = __ffma2_rn(p, g[v + kk], acc2[b * TG + kk]);
                acc2[B * TG + b * TG + kk] = __ffma2_rn(p, gs[v + kk], acc2[B * TG + b * TG + kk]);
            }
        }
    }
}

// Sum of every element of v over the 32 lanes of the warp, scattered: at each
// step a lane sends half of its elements to its partner and keeps the sums of
// the other half, so N elements take about N exchanges (a butterfly per element
// takes 5 N: 510 against 101 shuffles per warp at B = TG = 5).  Element i's sum
// ends in dst[i].
template <int N, int O>
__device__ __forceinline__ void lane_sums(const float (&v)[N], int lane, int base, int valid, float *dst)
{
    if constexpr (O == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < valid) dst[base + i] = v[i];
    } else {
        constexpr int H = (N + 1) / 2;
        const bool up = (lane & O) != 0;
        float w[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float lo = v[i], hi = i + H < N ? v[i + H < N ? i + H : 0] : 0.f;
            w[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, O);
        }
        lane_sums<H, O / 2>(w, lane, base + (up ? H : 0), up ? valid - H : (valid < H ? valid : H), dst);
    }
}

// Fixed-order reduction of the accumulators of the CTA's `nw` warps (`red`
// holds nw * NA floats), then one row of partials.
template <int B, int TG>
__device__ __forceinline__ void gh_reduce_row(const float2 (&acc2)[2 * B * TG + 1], float *red, int nw, int tid, int k0,
                                              bool group0, int T, int Bp, int Bq, float2 *row)
{
    constexpr int NP = 2 * B * TG + 1;
    constexpr int NA = 2 * NP;
    const int lane = tid & 31, warp = tid >> 5;
    float v[NA];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        v[2 * i] = acc2[i].x;
        v[2 * i + 1] = acc2[i].y;
    }
    lane_sums<NA, 16>(v, lane, 0, NA, red + warp * NA);
    __syncthreads();
    // One (b, kk) pair per thread: X and Y summed over the warps in index
    // order, then both branches.
    for (int e = tid; e <= B * TG; e += nw * 32) {
        float q[4] = {0.f, 0.f, 0.f, 0.f};
        const int i0 = e < B * TG ? 2 * e : 2 * (NP - 1), i1 = 2 * (B * TG + e);
        for (int w2 = 0; w2 < nw; ++w2) {
            const float *rw = red + w2 * NA;
            q[0] += rw[i0];
            q[1] += rw[i0 + 1];
            if (e < B * TG) {
                q[2] += rw[i1];
                q[3] += rw[i1 + 1];
            }
        }
        if (e == B * TG) {
            if (group0) row[(Bp + Bq) * T] = make_float2(q[0], q[1]);
            continue;
        }
        const int b = e / TG, kk = e % TG;
        if (k0 + kk >= T) continue;
        if (b < Bp) row[b * T + k0 + kk] = make_float2(q[0] + q[1], q[2] - q[3]);
        if (b < Bq) row[(Bp + b) * T + k0 + kk] = make_float2(q[0] - q[1], q[2] + q[3]);
    }
}

// Plain-load variant: grid (blocks, tap groups), 256 threads.
template <int B, int TG, int V>
__global__ void __launch_bounds__(256) adj_gh_kernel(AdjArgs a, int T, int Bp, int Bq, int K)
{
    constexpr int NA = 4 * B * TG + 2;
    constexpr int NP = NA / 2;
    const int k0 = blockIdx.y * TG;
    float2 acc2[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) acc2[i] = make_float2(0.f, 0.f);

    const bool vec_in = ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.gy)) & 15) == 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * V;
    for (int64_t j0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V; j0 < a.n; j0 += stride) {
        float2 xs[V], g[V + TG - 1];
        adj_load_window<V>(a.x, j0, a.n, vec_in, xs);
        adj_load_window<V + TG - 1>(a.gy, j0 + k0, a.n, vec_in, g);
        gh_accumulate<B, TG, V>(xs, g, blockIdx.y == 0, acc2);
    }
    __shared__ float red[8 * NA];
    gh_reduce_row<B, TG>(acc2, red, blockDim.x >> 5, threadIdx.x, k0, blockIdx.y == 0, T, Bp, Bq,
                                a.partials + (size_t)blockIdx.x * K);
}

// One warp's ring in the coefficient gradient.  The CTAs of a tap group take tiles of
// kAdjGhSub units per warp in turn: unit j of tile i of warp w of CTA b of G is unit
//   ((i G + b) kAdjGhSub + j) kAdjGhWarps + w
// of the record, and a lane adds its samples in that order.  A slot holds a tile: of
// each unit its x and, from element kAdjUnit on, its gy with the look-ahead (at the
// record's end the even-length prefix that exists), one bulk copy each by a lane of its
// own.  Slots and barriers as in AdjRing.
struct GhRing {
    static constexpr int kPart = 2 * kAdjUnit + kAdjGhHalo;   // elements of a unit
    static constexpr size_t kBytes = (size_t)kAdjGhStages * kAdjGhSub * kPart * sizeof(float2);   // per warp
    static_assert(2 * kAdjGhSub <= 32, "a lane per copy");

    const float2 *x, *gy;   // at the first sample of the warp's first unit
    int64_t left;           // samples of the record from there on
    int64_t step;           // samples from a tile to the next
    float2 *slots;
    uint32_t bars;
    int tiles;
    int whole;   // the first `whole` tiles lie, with their look-ahead, inside the record

    __device__ __forceinline__ void init(const AdjArgs &a, int cta, int ctas, int warp, unsigned char *mem,
                                         uint32_t bar_addr, int lane)
    {
        const int64_t s0 = ((int64_t)cta * kAdjGhSub * kAdjGhWarps + warp) * kAdjUnit;
        // Samples from a tile's first to its end with the look-ahead.
        constexpr int kReach = ((kAdjGhSub - 1) * kAdjGhWarps + 1) * kAdjUnit + kAdjGhHalo;
        x = a.x + s0;
        gy = a.gy + s0;
        left = a.n - s0;
        step = (int64_t)ctas * (kAdjGhSub * kAdjGhWarps * kAdjUnit);
        slots = reinterpret_cast<float2 *>(mem);
        bars = bar_addr;
        tiles = left > 0 ? (int)((left - 1) / step) + 1 : 0;
        whole = left >= kReach ? (int)((left - kReach) / step) + 1 : 0;
        if (lane == 0) {
            for (int s = 0; s < kAdjGhStages; ++s) mbar_init(bars + 8u * s, 1);
            fence_barrier_init();
        }
        __syncwarp();
        for (int i = 0; i < kAdjGhStages && i < tiles; ++i) issue(i, lane);
    }
    // Samples from unit j of tile i on to the end of the record.
    __device__ __forceinline__ int64_t rest(int i, int j) const
    {
        return left - i * step - j * (kAdjGhWarps * kAdjUnit);
    }
    __device__ __forceinline__ int units_of(int i) const
    {
        if (i < whole) return kAdjGhSub;
        const int64_t nu = (rest(i, 0) - 1) / (kAdjGhWarps * kAdjUnit) + 1;
        return nu < kAdjGhSub ? (int)nu : kAdjGhSub;
    }
    __device__ __forceinline__ float2 *part(int i, int j) const
    {
        return slots + ((i % kAdjGhStages) * kAdjGhSub + j) * kPart;
    }
    // Samples of x (or of gy) that the slot holds of a unit with `rem` samples to the end.
    __device__ __forceinline__ static int held(int64_t rem, bool is_gy)
    {
        const int want = is_gy ? kAdjUnit + kAdjGhHalo : kAdjUnit;
        return rem >= want ? want : rem > 0 ? (int)rem & ~1 : 0;
    }
    __device__ __forceinline__ void issue(int i, int lane)   // the whole warp
    {
        const uint32_t fb = bars + 8u * (i % kAdjGhStages);
        const int j = lane >> 1;
        const bool is_gy = lane & 1;
        uint32_t bytes = 0, all = kAdjGhSub * kPart * (uint32_t)sizeof(float2);
        if (lane < 2 * kAdjGhSub)
            bytes = (uint32_t)(i < whole ? (is_gy ? kAdjUnit + kAdjGhHalo : kAdjUnit) : held(rest(i, j), is_gy)) *
                    (uint32_t)sizeof(float2);
        if (i >= whole) all = __reduce_add_sync(0xffffffffu, bytes);
        if (lane == 0) mbar_arrive_expect_tx(fb, all);
        __syncwarp();
        if (bytes)
            bulk_copy_g2s(smem_addr(part(i, j)) + (is_gy ? kAdjUnit * (uint32_t)sizeof(float2) : 0u),
                          (is_gy ? gy : x) + i * step + j * (kAdjGhWarps * kAdjUnit), bytes, fb);
    }
    __device__ __forceinline__ bool wait(int i, int *status) const
    {
        return __all_sync(0xffffffffu, mbar_wait(bars + 8u * (i % kAdjGhStages),
                                                 (uint32_t)((i / kAdjGhStages) & 1), status));
    }
    __device__ __forceinline__ void refill(int i, int lane)   // the whole warp has read tile i
    {
        __syncwarp();
        if (i + kAdjGhStages < tiles) {
            fence_proxy_async_smem();   // the reads above precede the copies' writes
            issue(i + kAdjGhStages, lane);
        }
    }
    // After a failed wait on tile i: let the copies in flight land.
    __device__ __forceinline__ void drain(int i, int *status) const
    {
        for (int q = i; q < i + kAdjGhStages && q < tiles; ++q) wait(q, status);
    }
    // The window of NX samples of x and NG of gy (from k0 on) of element off of unit j of tile i.
    template <int NX, int NG>
    __device__ __forceinline__ void window(int i, int j, int off, int k0, float2 (&xs)[NX], float2 (&g)[NG]) const
    {
        const float2 *sl = part(i, j);
        if (i < whole) {
            adj_slot_window<NX>(sl, off, xs);
            adj_slot_window<NG>(sl + kAdjUnit, off + k0, g);
        } else {
            const int64_t rem = rest(i, j), at = i * step + j * (kAdjGhWarps * kAdjUnit);
            adj_slot_window_tail<NX>(sl, held(rem, false), x + at, off, rem, xs);
            adj_slot_window_tail<NG>(sl + kAdjUnit, held(rem, true), gy + at, off + k0, rem, g);
        }
    }
};
static_assert(GhRing::kPart % 2 == 0, "a unit's parts must stay 16-byte aligned");

// Staged variant: grid (blocks, tap groups) of CTAs of kAdjGhWarps independent
// warps (see GhRing), block x of a tap group sharing the record with the
// others of the group.  x and gy 16-byte aligned.  With 2 B TG + 1 packed
// accumulators a thread takes about 165 registers, so one CTA fits an SM.
template <int B, int TG, int V>
__device__ __forceinline__ void adj_gh_tma_body(const AdjArgs &a, int T, int Bp, int Bq, int K)
{
    constexpr int NA = 4 * B * TG + 2;
    constexpr int NP = NA / 2;
    constexpr int NG = V + TG - 1;
    static_assert(TG <= kAdjGhMaxTG && V == kAdjV, "tap group exceeds the staged look-ahead");
    static_assert(kAdjGhWarps * kAdjGhStages * 8 <= 512, "barrier area");
    extern __shared__ __align__(128) unsigned char smem[];
    float *red = reinterpret_cast<float *>(smem + 512);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k0 = blockIdx.y * TG;
    const bool group0 = blockIdx.y == 0;
    grid_dep_wait();
    GhRing ring;
    ring.init(a, blockIdx.x, gridDim.x, warp, smem + adj_staged_smem<GhRing>(warp, kAdjGhWarps * NA),
              smem_addr(smem) + 8u * kAdjGhStages * warp, lane);
    float2 acc2[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) acc2[i] = make_float2(0.f, 0.f);
    for (int i = 0; i < ring.tiles; ++i) {
        // A failed wait (error word set) ends this warp's tiles; it still joins
        // the reduction so that no warp waits for it.
        if (!ring.wait(i, a.status)) {
            ring.drain(i, a.status);
            break;
        }
        const int nu = ring.units_of(i);
#pragma unroll 1
        for (int j = 0; j < nu; ++j) {
            float2 xs[V], g[NG];
            ring.window(i, j, lane * V, k0, xs, g);
            if (j == nu - 1) ring.refill(i, lane);
            gh_accumulate<B, TG, V>(xs, g, group0, acc2);
        }
    }
    gh_reduce_row<B, TG>(acc2, red, kAdjGhWarps, tid, k0, group0, T, Bp, Bq, a.partials + (size_t)blockIdx.x * K);
}

template <int B, int TG, int V>
__global__ void __launch_bounds__(32 * kAdjGhWarps, 1)
    adj_gh_tma_kernel(AdjArgs a, int T, int Bp, int Bq, int K)
{
    adj_gh_tma_body<B, TG, V>(a, T, Bp, Bq, K);
}

// Many independent problems in one launch (the least-squares refinement of a
// batch): grid (CTAs per problem, tap groups, problems); problem z's
// arguments (x, gy, n, its own partials rows, 16-byte aligned buffers) come
// from args[z].
template <int B, int TG, int V>
__global__ void __launch_bounds__(32 * kAdjGhWarps, 1)
    adj_gh_tma_batched_kernel(const AdjArgs *args, int T, int Bp, int Bq, int K)
{
    grid_dep_wait();   // before args is read: the work list may have just been uploaded
    const AdjArgs a = args[blockIdx.z];
    adj_gh_tma_body<B, TG, V>(a, T, Bp, Bq, K);
}

// ---------------------------------------------------------------- launches
inline bool adj_staged_ok(const AdjArgs &a)
{
    return a.status != nullptr &&
           ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.gy)) & 15) == 0;
}

template <int B, int T, int V, bool PARAM>
cudaError_t launch_adj_gx_tma(const AdjArgs &a, const AdjParamTab<B, T> &ptab, int sm_count, cudaStream_t s)
{
    // The shared-memory table area is kept in both forms (it is small).
    const size_t smem = adj_staged_smem<GxRing<B>>(kAdjWarps, adj_tab_padded<B, T>());
    auto kern = adj_gx_tma_kernel<B, T, V, PARAM>;
    static SmemAttr smem_rec;
    cudaError_t attr = ensure_smem(smem_rec, (const void *)kern, smem);
    if (attr != cudaSuccess) return attr;
    static OccCache occ_rec;
    int occ = 0;
    attr = occupancy(occ_rec, (const void *)kern, 32 * kAdjWarps, smem, &occ);
    if (attr != cudaSuccess) return attr;
    if (occ < 1) occ = 1;
    const int64_t units = (a.n + kAdjUnit - 1) / kAdjUnit;
    int64_t grid = (int64_t)sm_count * occ;
    if (grid > units) grid = units;
    return launch_pdl(kern, dim3((unsigned)grid), 32 * kAdjWarps, smem, s, a, units, ptab);
}

template <int B, int T>
cudaError_t launch_adj_gx_t(const AdjArgs &a, int sm_count, cudaStream_t s)
{
    constexpr int V = kAdjV;
    if (adj_staged_ok(a)) {
        if (a.host_adj_tab) {
            AdjParamTab<B, T> ptab;
            for (int i = 0; i < adj_table_floats(B, T); ++i) ptab.v[i] = a.host_adj_tab[i];
            return launch_adj_gx_tma<B, T, V, true>(a, ptab, sm_count, s);
        }
        return launch_adj_gx_tma<B, T, V, false>(a, AdjParamTab<B, T>{}, sm_count, s);
    }
    static OccCache occ_rec;
    int occ = 0;
    const cudaError_t oe = occupancy(occ_rec, (const void *)adj_gx_kernel<B, T, V>, 256, 0, &occ);
    if (oe != cudaSuccess) return oe;
    if (occ < 1) occ = 1;
    const int64_t need = (a.n + 256 * V - 1) / (256 * V);
    int64_t grid = (int64_t)sm_count * occ;
    if (grid > need) grid = need;
    adj_gx_kernel<B, T, V><<<(unsigned)grid, 256, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int B, int TG>
cudaError_t launch_adj_gh_tg(const AdjArgs &a, int blocks, int T, int Bp, int Bq, int K, cudaStream_t s)
{
    const int groups = (T + TG - 1) / TG;
    dim3 grid((unsigned)blocks, (unsigned)groups);
    if (adj_staged_ok(a)) {
        constexpr int V = kAdjV;
        constexpr int NA = 4 * B * TG + 2;
        const size_t smem = adj_staged_smem<GhRing>(kAdjGhWarps, kAdjGhWarps * NA);
        static SmemAttr smem_rec;
        const cudaError_t attr = ensure_smem(smem_rec, (const void *)adj_gh_tma_kernel<B, TG, V>, smem);
        if (attr != cudaSuccess) return attr;
        return launch_pdl(adj_gh_tma_kernel<B, TG, V>, grid, 32 * kAdjGhWarps, smem, s, a, T, Bp, Bq, K);
    }
    adj_gh_kernel<B, TG, kAdjV><<<grid, 256, 0, s>>>(a, T, Bp, Bq, K);
    count_launch();
    return cudaGetLastError();
}

// gh: the tap-group size (1 to 5 taps per group) and the CTAs per group
// (= rows of partials, already clamped by the caller).
template <int B>
cudaError_t launch_adj_gh(const AdjArgs &a, const AdjLaunch &L, int T, int Bp, int Bq, int K, cudaStream_t s)
{
    switch (L.tap_group) {
    case 1: return launch_adj_gh_tg<B, 1>(a, L.gh_blocks, T, Bp, Bq, K, s);
    case 2: return launch_adj_gh_tg<B, 2>(a, L.gh_blocks, T, Bp, Bq, K, s);
    case 3: return launch_adj_gh_tg<B, 3>(a, L.gh_blocks, T, Bp, Bq, K, s);
    case 4: return launch_adj_gh_tg<B, 4>(a, L.gh_blocks, T, Bp, Bq, K, s);
    case 5: return launch_adj_gh_tg<B, 5>(a, L.gh_blocks, T, Bp, Bq, K, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int B, int TG>
cudaError_t launch_adj_gh_batched_tg(const AdjArgs *args, int count, int blocks, int T, int Bp, int Bq, int K,
                                     cudaStream_t s)
{
    constexpr int V = kAdjV;
    constexpr int NA = 4 * B * TG + 2;
    const size_t smem = adj_staged_smem<GhRing>(kAdjGhWarps, kAdjGhWarps * NA);
    static SmemAttr smem_rec;
    const cudaError_t attr = ensure_smem(smem_rec, (const void *)adj_gh_tma_batched_kernel<B, TG, V>, smem);
    if (attr != cudaSuccess) return attr;
    dim3 grid((unsigned)blocks, (unsigned)((T + TG - 1) / TG), (unsigned)count);
    return launch_pdl(adj_gh_tma_batched_kernel<B, TG, V>, grid, 32 * kAdjGhWarps, smem, s, args, T, Bp, Bq, K);
}

template <int B>
cudaError_t launch_adj_gh_batched(const AdjArgs *args, int count, int blocks, int tap_group, int T, int Bp, int Bq,
                                  int K, cudaStream_t s)
{
    switch (tap_group) {
    case 1: return launch_adj_gh_batched_tg<B, 1>(args, count, blocks, T, Bp, Bq, K, s);
    case 2: return launch_adj_gh_batched_tg<B, 2>(args, count, blocks, T, Bp, Bq, K, s);
    case 3: return launch_adj_gh_batched_tg<B, 3>(args, count, blocks, T, Bp, Bq, K, s);
    case 4: return launch_adj_gh_batched_tg<B, 4>(args, count, blocks, T, Bp, Bq, K, s);
    case 5: return launch_adj_gh_batched_tg<B, 5>(args, count, blocks, T, Bp, Bq, K, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int B>
cudaError_t launch_adj_gx(const AdjArgs &a, int T, int sm_count, cudaStream_t s)
{
    switch (T) {
    case 1: return launch_adj_gx_t<B, 1>(a, sm_count, s);
    case 2: return launch_adj_gx_t<B, 2>(a, sm_count, s);
    case 3: return launch_adj_gx_t<B, 3>(a, sm_count, s);
    case 4: return launch_adj_gx_t<B, 4>(a, sm_count, s);
    case 5: return launch_adj_gx_t<B, 5>(a, sm_count, s);
    case 6: return launch_adj_gx_t<B, 6>(a, sm_count, s);
    case 7: return launch_adj_gx_t<B, 7>(a, sm_count, s);
    case 8: return launch_adj_gx_t<B, 8>(a, sm_count, s);
    default: return cudaErrorInvalidValue;
    }
}

#define DPD_DEFINE_LAUNCH_ADJ(BB)                                                                  \
    template <>                                                                                    \
    cudaError_t launch_adj<BB>(const AdjArgs &a, const AdjLaunch &L, int T, int Bp, int Bq, int K, \
                               int sm_count, cudaStream_t s)                                       \
    {                                                                                              \
        if (a.gx) {                                                                                \
            cudaError_t e = launch_adj_gx<BB>(a, T, sm_count, s);                                  \
            if (e != cudaSuccess) return e;                                                        \
        }                                                                                          \
        if (a.partials) return launch_adj_gh<BB>(a, L, T, Bp, Bq, K, s);                           \
        return cudaSuccess;                                                                        \
    }                                                                                              \
    template <>                                                                                    \
    cudaError_t launch_adj_gh_many<BB>(const AdjArgs *args, int count, int blocks, int tap_group,  \
                                       int T, int Bp, int Bq, int K, cudaStream_t s)               \
    {                                                                                              \
        return launch_adj_gh_batched<BB>(args, count, blocks, tap_group, T, Bp, Bq, K, s);          \
    }

}  // namespace dpd
