// Factorisation and solves of the normal equations of the least-squares
// estimate: A = D G D = U Delta U^H (U unit lower triangular, Delta diagonal,
// D = diag(G)^{-1/2}), in FP32 pairs.
//
// FP64 runs at about two fused multiply-adds per clock per SM on GB300, FP32 at
// 128, so a value is held as an unevaluated sum hi + lo of two FP32 numbers and an
// operation on pairs costs 6 to 12 FP32 instructions.  A problem whose smallest
// pivot is not well above the pair arithmetic's error is left to the FP64 kernel
// (chol64_kernel), which every factorisation launches behind the pair kernel and
// which returns at once for all others; its factor stays in FP64, and so do the solves
// with it.
#include <type_traits>

#include "dpd_device.cuh"
#include "dpd_gram.cuh"
#include "dpd_table.cuh"

namespace dpd {

namespace {

constexpr int kCholMaxK = 2 * kMaxB * kMaxT + 1;   // 97: P = Q = 11, M = 7
constexpr int kCholWarps = 8;
constexpr int kCholThreads = 32 * kCholWarps;
constexpr int kNeedFp64 = -1;                      // info of a problem left to chol64_kernel

// Offset of row i in a lower triangle packed by rows (row i holds columns 0 .. i).
__host__ __device__ constexpr int tri_row(int i) { return i * (i + 1) / 2; }

__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float s = a + b, z = s - a;
    return make_float2(s, (a - (s - z)) + (b - z));
}

// Product of two pairs, relative error about 2^-46.
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b)
{
    const float p = __fmul_rn(a.x, b.x);
    const float e = fmaf(a.y, b.x, fmaf(a.x, b.y, fmaf(a.x, b.x, -p)));
    const float h = __fadd_rn(p, e);
    return make_float2(h, __fadd_rn(e, -__fadd_rn(h, -p)));
}

// 1 / d: the hardware's reciprocal y (within an ulp) and its correction y (e + e^2),
// e = 1 - d y exact to 2^-46.
__device__ __forceinline__ float2 pair_rcp(float2 d)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d.x));
    const float e = fmaf(-d.y, y, fmaf(-d.x, y, 1.f));
    const float c = __fmul_rn(y, fmaf(e, e, e));
    const float h = __fadd_rn(y, c);
    return make_float2(h, __fadd_rn(c, -__fadd_rn(h, -y)));
}

__device__ __forceinline__ float2 to_pair(double x)
{
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

__device__ __forceinline__ double to_double(float h, float l) { return (double)h + (double)l; }

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }   // biased
__device__ __forceinline__ double power_of_two(int e) { return __hiloint2double((e + 1023) << 20, 0); }   // |e| <= 1022

// A double whose exponent leaves both parts normal FP32 numbers, split by its bits
// (no FP64 instruction): hi is its leading 24 bits, lo the other 29 rounded to 24.
__device__ __forceinline__ bool splittable(double x)
{
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7FFu;
    return e - 920u <= 230u;
}
__device__ __forceinline__ float2 split_bits(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned sign = hi & 0x80000000u, e = (hi >> 20) & 0x7FFu;
    const float h = __uint_as_float(sign | ((e - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
    const float ulp = __uint_as_float(sign | ((e - 919u) << 23));
    return make_float2(h, (float)(lo & 0x1FFFFFFFu) * 1.862645149230957e-9f * ulp);   // 2^-29
}

}  // namespace

// One CTA of 8 warps per problem.  The columns are dealt to the warps in panels of
// four: panel P, columns 4 P .. 4 P + 3, to warp P mod 8, its element (i, k) to the
// registers of lane i mod 32: at most 24 per thread for the first n = K - 1 rows; the
// last row (K is 32 m + 1 for the largest models) is spread over the threads, element
// k on thread k.  Right-looking: for every panel each thread subtracts a_ij conj(u_kj),
// j in the panel, from its elements, a_ij the finished column and u_kj = a_kj / d_j,
// both read from shared memory (the first by lane, the second one value per warp).
// The warp that owns the next panel updates that panel first, factors it among its own
// lanes, writes it and only then updates its other columns.  The panels go through a
// ring of kCholRing slots with a full and an empty barrier each, so a warp waits for a
// panel and not for the other warps' updates: the chain of panels runs ahead of the
// bulk of the updates.  The last row's elements of a panel have a barrier of their own,
// for the warps that hold that row.
//
// Fixed-point accumulation.  A has a unit diagonal and is positive definite, so all
// elements of all trailing matrices stay within [-1, 1], and every product a_ij
// conj(u_kj) too.  An element's hi part is kept as 6 + hi, in [4, 8): one fused
// multiply-add t = C - a b rounds the product to that binade's grid of 2^-21, C - t
// is the part of it that went in, exactly, and fma(a, b, -(C - t)) the rest, which
// goes to lo with the cross terms: 6 instructions per real product where a two-sum
// takes 12.  The error of an element is about 2^-42 of the diagonal: at pivots above
// kPivotMin it is far below that of the Gram entries (2^-24 at best); smaller pivots
// go to the FP64 kernel.
//
// GB300, us, one problem / 256 problems: K = 97 72 / 140, K = 33 14.2 / 18.5 (FP64 on a
// cluster of 8 SMs 143.9 and 45.4, one CTA per problem 424.8 for 256 at K = 97; pairs
// with one column at a time 101 / 146 at K = 97).  At K = 97 the updates bound it (27
// instructions each at 0.6 per cycle and scheduler), at K = 33 the chain: a dependent
// FP32 instruction takes 4.7 cycles, and a column's update, pivot, reciprocal and scaling
// are about fifty of them; one column at a time adds a barrier and two trips through
// shared memory to each.  With the registers limited for two CTAs an SM (128, spills)
// 256 problems take 142.
constexpr float kPivotMin = 5.9604645e-8f;   // 2^-24
constexpr int kCholRing = 3;
constexpr int kCholPanel = 4;
static_assert(kCholPanel * kCholWarps == 32, "row group c holds the panels' diagonal rows of round c");

// The FP32 pairs of g s, re then im, for values that split_bits does not take.
__device__ __noinline__ float4 scaled_fp64(double2 g, double s)
{
    const float2 re = to_pair(g.x * s), im = to_pair(g.y * s);
    return make_float4(re.x, im.x, re.y, im.y);
}

__device__ __forceinline__ double equilibration(double g)   // g^{-1/2}, or 0
{
    return g > 0.0 ? inv_sqrt(g) : 0.0;
}

// NG: row groups of 32, and rounds of panels (columns 32 c + 4 warp + q).
template <int NG>
__global__ void __launch_bounds__(kCholThreads, 1)
    chol_pair_kernel(const double2 *Gall, int K, float4 *__restrict__ Uall, double *__restrict__ dall,
                     int *__restrict__ info, int *status)
{
    constexpr float kBias = 6.f;
    constexpr int R = kCholRing, PW = kCholPanel;
    __shared__ float4 raw[R][PW][32 * NG];   // a panel of the trailing matrix, {re.hi, im.hi, re.lo, im.lo}
    __shared__ float4 scl[R][PW][32 * NG];   // each column divided by its pivot
    __shared__ float4 last[R][PW];           // the last row's elements of the panel
    __shared__ float2 dinv[R][PW];           // 1 / pivots
    __shared__ int pbad[R];                  // whether a pivot is outside the pair arithmetic's reach
    __shared__ float2 dp[kCholMaxK];
    __shared__ double dd[kCholMaxK];
    __shared__ int bad;
    __shared__ uint64_t bars[3 * R];         // full, full of the last row's elements, empty
    const int p = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t full = smem_addr(bars), fullb = full + 8 * R, empty = fullb + 8 * R;
    if (tid == 0) {
        for (int s = 0; s < R; ++s) {
            mbar_init(full + 8 * s, 1);
            mbar_init(fullb + 8 * s, 1);
            mbar_init(empty + 8 * s, kCholWarps);
        }
        fence_barrier_init();
        bad = 0;
    }
    __syncthreads();
    grid_dep_wait();
    const int n = K - 1;
    const double2 *G = Gall + (size_t)p * K * K;
    float4 *U = Uall + (size_t)p * tri_row(K);

    // Every element's loads first (their bits wait in the registers of the pairs).
    float Cr[NG][NG][PW], Ci[NG][NG][PW], Lr[NG][NG][PW], Li[NG][NG][PW];   // [row group][round][column]
    float br, bi, blr, bli;   // element (n, tid)
    auto fetch = [&](bool in, int i, int k, float &cr, float &ci, float &lr, float &li) {
        const double2 g = in ? G[(size_t)i * K + k] : make_double2(0.0, 0.0);
        cr = __int_as_float(__double2loint(g.x));
        ci = __int_as_float(__double2hiint(g.x));
        lr = __int_as_float(__double2loint(g.y));
        li = __int_as_float(__double2hiint(g.y));
    };
#pragma unroll
    for (int c = 0; c < NG; ++c)
#pragma unroll
        for (int a = c; a < NG; ++a)
#pragma unroll
            for (int q = 0; q < PW; ++q) {
                const int i = 32 * a + lane, k = 32 * c + PW * warp + q;
                fetch(i < n && k <= i, i, k, Cr[a][c][q], Ci[a][c][q], Lr[a][c][q], Li[a][c][q]);
            }
    fetch(tid <= n, n, tid, br, bi, blr, bli);
    if (tid < K) {
        const double d = equilibration(G[(size_t)tid * K + tid].x);
        dd[tid] = d;
        if (splittable(d))
            dp[tid] = split_bits(d);
        else
            bad = 1;   // outside FP32's range, or not positive: the FP64 kernel decides
        dall[(size_t)p * K + tid] = d;
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) info[p] = kNeedFp64;
        return;
    }
    // Scaled, as biased elements {6 + re.hi, 6 + im.hi} and their lo parts.
    auto convert = [&](bool in, int i, int k, float &cr, float &ci, float &lr, float &li) {
        const double gx = __hiloint2double(__float_as_int(ci), __float_as_int(cr));
        const double gy = __hiloint2double(__float_as_int(li), __float_as_int(lr));
        const bool zx = (__float_as_int(ci) | __float_as_int(cr)) == 0, zy = (__float_as_int(li) | __float_as_int(lr)) == 0;
        float2 re = make_float2(0.f, 0.f), im = re;
        if (in) {
            if ((zx || splittable(gx)) && (zy || splittable(gy))) {
                const float2 sc = pair_mul(dp[i], dp[k]);
                if (!zx) re = pair_mul(split_bits(gx), sc);
                if (!zy) im = pair_mul(split_bits(gy), sc);
            } else {
                const float4 v = scaled_fp64(make_double2(gx, gy), dd[i] * dd[k]);
                re = make_float2(v.x, v.z);
                im = make_float2(v.y, v.w);
            }
        }
        cr = __fadd_rn(kBias, re.x);
        lr = __fadd_rn(__fadd_rn(re.x, -__fadd_rn(cr, -kBias)), re.y);
        ci = __fadd_rn(kBias, im.x);
        li = __fadd_rn(__fadd_rn(im.x, -__fadd_rn(ci, -kBias)), im.y);
    };
#pragma unroll
    for (int c = 0; c < NG; ++c)
#pragma unroll
        for (int a = c; a < NG; ++a)
#pragma unroll
            for (int q = 0; q < PW; ++q) {
                const int i = 32 * a + lane, k = 32 * c + PW * warp + q;
                convert(i < n && k <= i, i, k, Cr[a][c][q], Ci[a][c][q], Lr[a][c][q], Li[a][c][q]);
            }
    convert(tid <= n, n, tid, br, bi, blr, bli);

    // c -= x conj(y): x = {re.hi, im.hi, re.lo, im.lo} of a_ij, y of u_kj.
    auto mul_sub = [](float ah, float al, float bh, float bl, float &C, float &L) {
        const float t = fmaf(-ah, bh, C);
        const float q = __fadd_rn(C, -t);                // rounded product, exact
        const float r = fmaf(ah, bh, -q);                // its remainder
        L = __fadd_rn(L, -fmaf(al, bh, fmaf(ah, bl, r)));
        C = t;
    };
    auto update = [&](const float4 &x, const float4 &y, float &cr, float &ci, float &lr, float &li) {
        mul_sub(x.x, x.z, y.x, y.z, cr, lr);
        mul_sub(x.y, x.w, y.x, y.z, ci, li);
        mul_sub(x.y, x.w, y.y, y.w, cr, lr);
        mul_sub(-x.x, -x.z, y.y, y.w, ci, li);
    };
    auto value = [](float cr, float ci, float lr, float li) {
        const float2 re = two_sum(__fadd_rn(cr, -kBias), lr), im = two_sum(__fadd_rn(ci, -kBias), li);
        return make_float4(re.x, im.x, re.y, im.y);
    };
    auto scaled = [](const float4 &v, float2 s) {
        const float2 re = pair_mul(make_float2(v.x, v.z), s), im = pair_mul(make_float2(v.y, v.w), s);
        return make_float4(re.x, im.x, re.y, im.y);
    };
    auto shfl4 = [](const float4 &v, int src) {
        return make_float4(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                           __shfl_sync(0xffffffffu, v.z, src), __shfl_sync(0xffffffffu, v.w, src));
    };
    // This warp's panel of round c by the panel in slot b.
    auto panel_update = [&](auto cc, int b) {
        constexpr int c = decltype(cc)::value;
#pragma unroll
        for (int a = c; a < NG; ++a)
#pragma unroll 1
            for (int j = 0; j < PW; ++j) {
                const float4 x = raw[b][j][32 * a + lane];
                const float4 *y = &scl[b][j][32 * c + PW * warp];
#pragma unroll
                for (int q = 0; q < PW; ++q) update(x, y[q], Cr[a][c][q], Ci[a][c][q], Lr[a][c][q], Li[a][c][q]);
            }
    };
    // This warp's panel P of round c: its columns in turn, each with its pivot, as it is
    // and divided by the pivot, and U's columns.
    auto panel_factor = [&](auto cc, int P) {
        constexpr int c = decltype(cc)::value;
        const int b = P % R, j0 = PW * P, l0 = PW * warp;
        // The slot is free once every warp has read its last panel.
        if (P >= R && !mbar_wait(empty + 8 * b, (uint32_t)((P / R - 1) & 1), status)) return false;
        bool ok = true;
#pragma unroll
        for (int q = 0; q < PW; ++q)
            if (j0 + q < n) {
                float4 v[NG], u[NG];
#pragma unroll
                for (int a = c; a < NG; ++a) v[a] = value(Cr[a][c][q], Ci[a][c][q], Lr[a][c][q], Li[a][c][q]);
                const float2 d = make_float2(__shfl_sync(0xffffffffu, v[c].x, l0 + q), __shfl_sync(0xffffffffu, v[c].z, l0 + q));
                const float2 inv = pair_rcp(d);
                ok = ok && d.x > kPivotMin && d.x < 2.f;
#pragma unroll
                for (int a = c; a < NG; ++a) u[a] = scaled(v[a], inv);
#pragma unroll
                for (int r = q + 1; r < PW; ++r) {
                    const float4 y = shfl4(u[c], l0 + r);
#pragma unroll
                    for (int a = c; a < NG; ++a) update(v[a], y, Cr[a][c][r], Ci[a][c][r], Lr[a][c][r], Li[a][c][r]);
                }
#pragma unroll
                for (int a = c; a < NG; ++a) {   // rows up to the column's own and past n: never read
                    const int i = 32 * a + lane;
                    raw[b][q][i] = v[a];
                    scl[b][q][i] = u[a];
                    if (i > j0 + q && i < n) U[tri_row(i) + j0 + q] = u[a];
                }
                if (lane == l0 + q) {
                    dinv[b][q] = inv;
                    U[tri_row(j0 + q) + j0 + q] = make_float4(inv.x, 0.f, inv.y, 0.f);
                }
            }
        if (lane == 0) pbad[b] = !ok;
        __syncwarp();
        if (lane == 0) mbar_arrive(full + 8 * b);
        return true;
    };
    using std::integral_constant;

    if (warp == 0) panel_factor(integral_constant<int, 0>(), 0);
    bool failed = false;
    const int panels = (n + PW - 1) / PW;
    for (int P = 0; P < panels; ++P) {
        const int b = P % R, next = P + 1, j0 = PW * P;
        const uint32_t ph = (uint32_t)((P / R) & 1);
        if (!mbar_wait(full + 8 * b, ph, status) || pbad[b]) {   // one outcome for all warps
            failed = true;
            break;
        }
        const bool ahead = next < panels && warp == next % kCholWarps;
        if (ahead) {
            bool ok = true;
            auto advance = [&](auto cc) {
                if constexpr ((decltype(cc)::value) < NG) {
                    panel_update(cc, b);
                    ok = panel_factor(cc, next);
                }
            };
            if (next / kCholWarps == 0) advance(integral_constant<int, 0>());
            else if (next / kCholWarps == 1) advance(integral_constant<int, 1>());
            else advance(integral_constant<int, 2>());
            if (!ok) {
                failed = true;
                break;
            }
        }
        const int from = ahead ? next + 1 : next;   // first panel not yet updated
        if (warp >= from) panel_update(integral_constant<int, 0>(), b);
        if constexpr (NG > 1)
            if (kCholWarps + warp >= from) panel_update(integral_constant<int, 1>(), b);
        if constexpr (NG > 2)
            if (2 * kCholWarps + warp >= from) panel_update(integral_constant<int, 2>(), b);
        // The last row, element (n, tid), on the warps that hold unfinished elements of it.
        // The warp with the panel's own columns finishes those in turn and passes them on.
        if (32 * warp <= n && 32 * warp + 31 >= j0) {
            const bool own = warp == j0 >> 5;
            if (!own && !mbar_wait(fullb + 8 * b, ph, status)) {
                failed = true;
                break;
            }
            for (int q = 0; q < PW && j0 + q < n; ++q) {
                const int k = j0 + q;
                const float4 x = own ? shfl4(value(br, bi, blr, bli), k & 31) : last[b][q];
                const float4 u = scaled(x, dinv[b][q]);
                if (tid == k) {
                    U[tri_row(n) + k] = u;
                    last[b][q] = x;
                }
                if (tid > k && tid <= n) update(x, tid == n ? u : scl[b][q][tid], br, bi, blr, bli);   // (n, n): its own
            }
            __syncwarp();
            if (own && lane == 0) mbar_arrive(fullb + 8 * b);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + 8 * b);
    }
    if (tid == n) {
        const float4 v = value(br, bi, blr, bli);
        const float2 inv = pair_rcp(make_float2(v.x, v.z));
        U[tri_row(n) + n] = make_float4(inv.x, 0.f, inv.y, 0.f);
        info[p] = !failed && v.x > kPivotMin && v.x < 2.f ? 0 : kNeedFp64;
    }
}

// The FP64 form, one CTA per problem, for those that the pair kernel left (info =
// kNeedFp64): A = D G D in shared memory (packed lower triangle), factored in
// place (right looking) as L L^H, then U = L diag(L)^{-1} and diag(L)^{-2}.  Step j:
// thread 0 takes the pivot; the threads scale column j; the trailing update of rows
// i > j, columns j < k <= i is split into equal contiguous runs of the triangle, one
// per thread (an FP64 warp instruction costs the FP64 unit the same time however
// many lanes it has).
constexpr int kChol64Threads = 256;

__global__ void __launch_bounds__(kChol64Threads) chol64_kernel(const double2 *Gall, int K, float4 *Uall, int *wide,
                                                                double *__restrict__ dall, int *info, float4 *Uhost,
                                                                int *info_host)
{
    extern __shared__ double2 A[];   // lower triangle of K x K, packed by rows (tri_row)
    __shared__ double dsh[kCholMaxK];
    __shared__ double rinv;
    __shared__ int bad;
    grid_dep_wait();
    const int p = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    // Host copies of the first problem, whichever kernel factored it.
    auto to_host = [&](int status, int fp64) {
        if (p != 0) return;
        if (Uhost) {
#pragma unroll 8
            for (int e = tid; e < tri_row(K); e += nt) Uhost[e] = __ldcg(Uall + e);
        }
        if (info_host && tid == 0) {
            info_host[0] = status;
            info_host[1] = fp64;
        }
    };
    const int before = info[p];
    if (tid == 0) wide[p] = before == kNeedFp64;
    if (before != kNeedFp64) {
        to_host(before, 0);
        return;
    }
    const int tx = tid & 15, ty = tid >> 4, nty = nt >> 4;
    const double2 *G = Gall + (size_t)p * K * K;
    if (tid == 0) bad = 0;
    __syncthreads();
    for (int i = tid; i < K; i += nt) {
        const double gii = G[(size_t)i * K + i].x;
        dsh[i] = gii > 0.0 ? 1.0 / sqrt(gii) : 0.0;
        if (!(gii > 0.0)) atomicMax(&bad, i + 1);
    }
    __syncthreads();
    for (int i = ty; i < K; i += nty)
        for (int k = tx; k <= i; k += 16) {
            const double2 v = G[(size_t)i * K + k];
            const double sc = dsh[i] * dsh[k];
            A[tri_row(i) + k] = make_double2(v.x * sc, v.y * sc);
        }
    __syncthreads();
    for (int j = 0; j < K && !bad; ++j) {
        if (tid == 0) {
            const double piv = A[tri_row(j) + j].x;
            if (!(piv > 1e-30 && piv < 1e30)) {   // not positive definite (or numerically singular)
                bad = j + 1;
            } else {
                const double ri = inv_sqrt(piv);
                A[tri_row(j) + j] = make_double2(piv * ri, 0.0);
                rinv = ri;
            }
        }
        __syncthreads();
        if (bad) break;
        const double ri = rinv;
        for (int i = j + 1 + tid; i < K; i += nt) {
            const double2 v = A[tri_row(i) + j];
            A[tri_row(i) + j] = make_double2(v.x * ri, v.y * ri);
        }
        __syncthreads();
        {
            const int m = K - j - 1;
            const int tot = m * (m + 1) / 2;
            const int per = (tot + nt - 1) / nt;
            int e = tid * per;
            if (e < tot) {
                // row r of the triangle holding element e: r (r + 1) / 2 <= e < (r + 1) (r + 2) / 2
                int r = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                while ((r + 1) * (r + 2) / 2 <= e) ++r;
                while (r * (r + 1) / 2 > e) --r;
                int c = e - r * (r + 1) / 2;
                const int end = min(e + per, tot);
                int i = j + 1 + r, k = j + 1 + c;
                int ib = tri_row(i), kb = tri_row(k);   // packed offsets of rows i and k
                double2 a = A[ib + j];
                for (; e < end; ++e) {
                    const double2 b = A[kb + j];
                    double2 &cc = A[ib + k];
                    cc.x = fma(-a.x, b.x, fma(-a.y, b.y, cc.x));
                    cc.y = fma(-a.y, b.x, fma(a.x, b.y, cc.y));
                    if (++c > r) {   // next row of the triangle
                        c = 0;
                        ++r;
                        ++i;
                        ib += i;   // tri_row(i) = tri_row(i - 1) + i
                        k = j + 1;
                        kb = tri_row(k);
                        if (i < K) a = A[ib + j];
                    } else {
                        ++k;
                        kb += k;
                    }
                }
            }
        }
        __syncthreads();
    }
    double2 *U = reinterpret_cast<double2 *>(Uall + (size_t)p * tri_row(K));
    for (int i = ty; i < K; i += nty)
        for (int k = tx; k <= i; k += 16) {
            const double s = 1.0 / A[tri_row(k) + k].x;
            const double2 v = A[tri_row(i) + k];
            U[tri_row(i) + k] = make_double2(k < i ? v.x * s : s * s, k < i ? v.y * s : 0.0);
        }
    for (int i = tid; i < K; i += nt) dall[(size_t)p * K + i] = dsh[i];
    if (tid == 0) info[p] = bad;
    __syncthreads();   // U and every thread's read of info
    to_host(bad, 1);
}

cudaError_t launch_chol(const double2 *G, int nprob, int K, float4 *U, int *wide, double *d, int *info, float4 *Uhost,
                        int *info_host, int *status, cudaStream_t s)
{
    if (K < 2 || K > kCholMaxK) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)nprob);
    cudaError_t e = cudaErrorInvalidValue;
    switch ((K - 1 + 31) / 32) {
    case 1: e = launch_pdl(chol_pair_kernel<1>, grid, kCholThreads, 0, s, G, K, U, d, info, status); break;
    case 2: e = launch_pdl(chol_pair_kernel<2>, grid, kCholThreads, 0, s, G, K, U, d, info, status); break;
    case 3: e = launch_pdl(chol_pair_kernel<3>, grid, kCholThreads, 0, s, G, K, U, d, info, status); break;
    }
    if (e != cudaSuccess) return e;
    const size_t smem = sizeof(double2) * (size_t)tri_row(K);
    static SmemAttr smem_rec;
    e = ensure_smem(smem_rec, (const void *)chol64_kernel, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(chol64_kernel, grid, kChol64Threads, smem, s, G, K, U, wide, d, info, Uhost, info_host);
}

// One CTA per problem: x = D U^{-H} Delta^{-1} U^{-1} D rhs, in FP32 pairs.  The CTA
// stages U in shared memory and solves in blocks of 32 rows: a diagonal block is one
// warp's sequential part (element b0 + l on lane l; each step broadcasts one finished
// element and the later lanes take a complex multiply-subtract, whose latency bounds
// the solve); the update of the remaining rows is a block matrix-vector product spread
// over the CTA (8 threads per row).  GB300, K = 97, us: one problem 24.2, 256 problems 28.5
// (in FP64, four warp instructions of 64 cycles a step: 85.5 for 256).
constexpr int kSolveNB = 32;
constexpr int kSolveUnroll = 8;   // steps whose factor entries are loaded ahead

namespace {
// A complex pair as two packed halves, {re, im}.hi and {re, im}.lo, for f32x2
// instructions (half the issue slots of a chain that one warp runs alone).
struct CPair {
    float2 h, l;
};
__device__ __forceinline__ CPair cpair(const float4 &v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 quad(const CPair &v)
{
    const float2 re = two_sum(v.h.x, v.l.x), im = two_sum(v.h.y, v.l.y);
    return make_float4(re.x, im.x, re.y, im.y);
}
// a - b
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// v -= u {x, x}, u a packed pair, x a real one: the sum exact to the pair (two-sum)
__device__ __forceinline__ void mul_sub2(CPair &v, const CPair &u, float xh, float xl)
{
    const float2 X = make_float2(xh, xh), N = make_float2(-xh, -xh);
    const float2 p = __fmul2_rn(u.h, N);
    const float2 e = __ffma2_rn(u.l, X, __ffma2_rn(u.h, make_float2(xl, xl), __ffma2_rn(u.h, X, p)));
    const float2 s = __fadd2_rn(v.h, p), z = sub2(s, v.h);
    const float2 err = __fadd2_rn(sub2(v.h, sub2(s, z)), sub2(p, z));
    v.h = s;
    v.l = __fadd2_rn(v.l, sub2(err, e));
}
// v -= u x (CONJ: conj(u) x)
template <bool CONJ>
__device__ __forceinline__ void cpair_mul_sub(CPair &v, const float4 &u, const float4 &x)
{
    const CPair a = {make_float2(u.x, CONJ ? -u.y : u.y), make_float2(u.z, CONJ ? -u.w : u.w)};
    const CPair b = {make_float2(CONJ ? u.y : -u.y, u.x), make_float2(CONJ ? u.w : -u.w, u.z)};
    mul_sub2(v, a, x.x, x.z);
    mul_sub2(v, b, x.y, x.w);
}
__device__ __forceinline__ float4 shfl_cpair(const CPair &v, int src)
{
    return make_float4(__shfl_sync(0xffffffffu, v.h.x, src), __shfl_sync(0xffffffffu, v.h.y, src),
                       __shfl_sync(0xffffffffu, v.l.x, src), __shfl_sync(0xffffffffu, v.l.y, src));
}
// Sum over the 8 threads of a row, as a normalised pair.
__device__ __forceinline__ float4 row_sum(const CPair &v)
{
    float2 re = make_float2(v.h.x, v.l.x), im = make_float2(v.h.y, v.l.y);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        re = pair_add(re, shfl_xor_pair(re, o));
        im = pair_add(im, shfl_xor_pair(im, o));
    }
    return make_float4(re.x, im.x, re.y, im.y);
}
// Element j of a coefficient vector in the other basis (both branches, every tap; the
// constant unchanged), U upper triangular with rows of kMaxB:
//   MONOMIAL:  h[(a, k)] = sum_{b >= a} U[a][b] h_U[(b, k)]    (W h)
//   otherwise: g_U[(a, k)] = sum_{c <= a} U[c][a] g[(c, k)]    (W^T g, right-hand sides)
template <bool MONOMIAL>
__device__ __forceinline__ double2 basis_transform(const double2 *x, const double *U, int j, int K, int Bp, int Bq, int T)
{
    if (j == K - 1) return x[j];
    const bool conj = j >= Bp * T;
    const int base = conj ? Bp * T : 0, nb = conj ? Bq : Bp, jj = j - base, a = jj / T, k = jj % T;
    double2 v = make_double2(0.0, 0.0);
    for (int b = MONOMIAL ? a : 0; b < (MONOMIAL ? nb : a + 1); ++b) {
        const double u = MONOMIAL ? U[a * kMaxB + b] : U[b * kMaxB + a];
        v.x += u * x[base + b * T + k].x;
        v.y += u * x[base + b * T + k].y;
    }
    return v;
}
__device__ __forceinline__ float4 cpair_add(const float4 &a, const float4 &b)
{
    const float2 re = pair_add(make_float2(a.x, a.z), make_float2(b.x, b.z));
    const float2 im = pair_add(make_float2(a.y, a.w), make_float2(b.y, b.w));
    return make_float4(re.x, im.x, re.y, im.y);
}
// x <- U^{-H} Delta^{-1} U^{-1} x in FP64, one row per thread of the CTA, for the few
// problems that the FP64 kernel factored (U in shared memory, two doubles a value).
__device__ __noinline__ void solve_fp64(const double2 *U, double2 *x, int K, int tid)
{
    for (int j = 0; j < K; ++j) {
        const double2 b = x[j];
        if (tid > j && tid < K) {
            const double2 a = U[tri_row(tid) + j];
            double2 &v = x[tid];
            v.x = fma(-a.x, b.x, fma(a.y, b.y, v.x));
            v.y = fma(-a.x, b.y, fma(-a.y, b.x, v.y));
        }
        __syncthreads();
    }
    if (tid < K) {
        const double s = U[tri_row(tid) + tid].x;
        x[tid] = make_double2(x[tid].x * s, x[tid].y * s);
    }
    __syncthreads();
    for (int j = K - 1; j >= 0; --j) {
        const double2 b = x[j];
        if (tid < j) {
            const double2 a = U[tri_row(j) + tid];   // conj(a) b
            double2 &v = x[tid];
            v.x = fma(-a.x, b.x, fma(-a.y, b.y, v.x));
            v.y = fma(-a.x, b.y, fma(a.y, b.x, v.y));
        }
        __syncthreads();
    }
}
}  // namespace

__global__ void __launch_bounds__(256) chol_solve_kernel(const float4 *Uall, const int *wide, const double *dall,
                                                         const int *info, int K, SolveIo io, int *status)
{
    extern __shared__ __align__(128) float4 Us[];   // U, lower triangle packed by rows (tri_row), 1 / pivots on the diagonal
    __shared__ float4 w[kCholMaxK];
    double2 *x64 = reinterpret_cast<double2 *>(w);
    __shared__ double2 mono[kCholMaxK];      // a vector before and after a change of basis
    __shared__ float4 part[8][kCholMaxK];    // sums of rows by warp
    __shared__ uint64_t bar;
    __shared__ int top;                      // largest exponent in D rhs
    if (threadIdx.x == 0) {
        top = 0;
        mbar_init(smem_addr(&bar), 1);
        fence_barrier_init();
    }
    __syncthreads();
    grid_dep_wait();
    const int p = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int sub = tid & 7, grp = tid >> 3, ngrp = nt >> 3;   // 8 threads per row in the updates
    if (info[p] != 0) return;   // uniform over the CTA
    const bool fp64 = wide[p] != 0;
    const float4 *U = Uall + (size_t)p * tri_row(K);
    const double *d = dall + (size_t)p * K;
    const double *W = io.basis ? io.basis + (size_t)p * kUSize : nullptr;
    if (tid == 0) {   // the whole factor in one bulk copy
        mbar_arrive_expect_tx(smem_addr(&bar), (uint32_t)(tri_row(K) * sizeof(float4)));
        bulk_copy_g2s(smem_addr(Us), U, (uint32_t)(tri_row(K) * sizeof(float4)), smem_addr(&bar));
    }
    if (io.rows) {
        // Warp w adds rows w, w + 8, ..., in order, as exact pairs (about 2^-48); thread i
        // then adds the eight sums of coefficient i.
        const float2 *rows = io.rows + (size_t)p * io.nrows * K;
        CPair acc[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 8
        for (int r = warp; r < io.nrows; r += 8)
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (lane + 32 * m < K) {
                    const float2 v = rows[(size_t)r * K + lane + 32 * m];
                    two_sum_acc(acc[m].h.x, acc[m].l.x, v.x);
                    two_sum_acc(acc[m].h.y, acc[m].l.y, v.y);
                }
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (lane + 32 * m < K)
                part[warp][lane + 32 * m] = make_float4(acc[m].h.x, acc[m].h.y, acc[m].l.x, acc[m].l.y);
        __syncthreads();
        if (tid < K) {
            float4 v = part[0][tid];
#pragma unroll
            for (int q = 1; q < 8; ++q) v = cpair_add(v, part[q][tid]);
            double2 g = make_double2(to_double(v.x, v.z), to_double(v.y, v.w));
            if (!isfinite(g.x) || !isfinite(g.y)) {   // a sum outside FP32's range (or an infinite row)
                g = make_double2(0.0, 0.0);
                for (int r = 0; r < io.nrows; ++r) {
                    const float2 e = rows[(size_t)r * K + tid];
                    g = make_double2(g.x + (double)e.x, g.y + (double)e.y);
                }
            }
            mono[tid] = g;
        }
        __syncthreads();
    }
    double2 b = make_double2(0.0, 0.0);   // element tid of D rhs
    if (tid < K) {
        const double2 v = !io.rows ? io.rhs[(size_t)p * K + tid]
                          : W      ? basis_transform<false>(mono, W, tid, K, io.Bp, io.Bq, io.T)
                                   : mono[tid];
        b = make_double2(v.x * d[tid], v.y * d[tid]);
        atomicMax(&top, max(exponent(b.x), exponent(b.y)));
    }
    if (!mbar_wait(smem_addr(&bar), 0u, status)) {   // the copy lands before the CTA leaves, within the limit
        mbar_wait(smem_addr(&bar), 0u, status);
        return;
    }
    __syncthreads();
    // In pairs the right-hand side is scaled by the power of two that brings its largest
    // element to [1, 2), and the result back: exact, and no element that matters leaves
    // FP32's range on the way (a positive definite matrix with pivots above kPivotMin).
    const int shift = top >= 1 && top <= 2045 ? top - 1023 : 0;
    if (tid < K) {
        if (fp64) {
            x64[tid] = b;
        } else {
            const double s = power_of_two(-shift);
            const float2 re = to_pair(b.x * s), im = to_pair(b.y * s);
            w[tid] = make_float4(re.x, im.x, re.y, im.y);
        }
    }
    __syncthreads();
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    if (fp64) solve_fp64(reinterpret_cast<const double2 *>(Us), x64, K, tid);

    // forward: U y = D b
    for (int b0 = 0; b0 < K && !fp64; b0 += kSolveNB) {
        const int nb = min(kSolveNB, K - b0);
        if (warp == 0) {
            const bool in = lane < nb;
            CPair v = cpair(in ? w[b0 + lane] : zero);
            const float4 *row = Us + tri_row(in ? b0 + lane : b0) + b0;
            for (int i0 = 0; i0 < nb; i0 += kSolveUnroll) {
                float4 u[kSolveUnroll];
#pragma unroll
                for (int q = 0; q < kSolveUnroll; ++q) u[q] = lane > i0 + q && in ? row[i0 + q] : zero;
#pragma unroll
                for (int q = 0; q < kSolveUnroll; ++q) {
                    const float4 x = shfl_cpair(v, i0 + q);
                    CPair t = v;
                    cpair_mul_sub<false>(t, u[q], x);
                    if (lane > i0 + q) v = t;
                }
            }
            if (in) w[b0 + lane] = quad(v);
        }
        __syncthreads();
        for (int r0 = b0 + nb; r0 < K; r0 += ngrp) {   // rows below: y_r -= U[r][block] y[block]
            const int r = r0 + grp;
            CPair v = cpair(zero);
            if (r < K)
                for (int c = sub; c < nb; c += 8) cpair_mul_sub<false>(v, Us[tri_row(r) + b0 + c], w[b0 + c]);
            const float4 t = row_sum(v);
            if (r < K && sub == 0) w[r] = cpair_add(w[r], t);
        }
        __syncthreads();
    }
    if (tid < K && !fp64) {   // z = Delta^{-1} y
        const float4 q = Us[tri_row(tid) + tid], y = w[tid];
        const float2 s = make_float2(q.x, q.z);
        const float2 re = pair_mul(make_float2(y.x, y.z), s), im = pair_mul(make_float2(y.y, y.w), s);
        w[tid] = make_float4(re.x, im.x, re.y, im.y);
    }
    __syncthreads();
    // backward: U^H v = z
    for (int b0 = ((K - 1) / kSolveNB) * kSolveNB; b0 >= 0 && !fp64; b0 -= kSolveNB) {
        const int nb = min(kSolveNB, K - b0);
        if (warp == 0) {
            const bool in = lane < nb;
            CPair v = cpair(in ? w[b0 + lane] : zero);
            for (int i0 = (nb - 1) & -kSolveUnroll; i0 >= 0; i0 -= kSolveUnroll) {
                float4 u[kSolveUnroll];
#pragma unroll
                for (int q = 0; q < kSolveUnroll; ++q) {
                    const int i = i0 + q;
                    u[q] = lane < i && i < nb ? Us[tri_row(b0 + i) + b0 + lane] : zero;
                }
#pragma unroll
                for (int q = kSolveUnroll - 1; q >= 0; --q) {
                    const float4 x = shfl_cpair(v, i0 + q);
                    CPair t = v;
                    cpair_mul_sub<true>(t, u[q], x);
                    if (lane < i0 + q && i0 + q < nb) v = t;
                }
            }
            if (in) w[b0 + lane] = quad(v);
        }
        __syncthreads();
        for (int r0 = 0; r0 < b0; r0 += ngrp) {   // rows above: v_r -= sum_c conj(U[b0+c][r]) v[b0+c]
            const int r = r0 + grp;
            CPair v = cpair(zero);
            if (r < b0)
                for (int c = sub; c < nb; c += 8) cpair_mul_sub<true>(v, Us[tri_row(b0 + c) + r], w[b0 + c]);
            const float4 t = row_sum(v);
            if (r < b0 && sub == 0) w[r] = cpair_add(w[r], t);
        }
        __syncthreads();
    }
    if (tid < K) {
        const float4 v = w[tid];
        const double s = fp64 ? 1.0 : power_of_two(shift);
        double2 x = fp64 ? x64[tid] : make_double2(to_double(v.x, v.z), to_double(v.y, v.w));
        x = make_double2(x.x * d[tid] * s, x.y * d[tid] * s);
        double2 *h = io.h + (size_t)p * K + tid;
        if (io.accumulate) x = make_double2(h->x + x.x, h->y + x.y);
        *h = x;
        mono[tid] = x;
    }
    __syncthreads();
    // The monomial coefficients in FP32, and their forward table.
    float2 *hf = reinterpret_cast<float2 *>(w);
    double2 x = make_double2(0.0, 0.0);
    if (tid < K) x = W ? basis_transform<true>(mono, W, tid, K, io.Bp, io.Bq, io.T) : mono[tid];
    if (tid < K) {
        hf[tid] = make_float2((float)x.x, (float)x.y);
        io.out[(size_t)p * K + tid] = hf[tid];
    }
    __syncthreads();
    const int B = io.Bp > io.Bq ? io.Bp : io.Bq;
    wl_table_entry([hf](int i) { return hf[i]; }, tid, io.Bp, io.Bq, io.T, B, io.tab + (size_t)p * io.tstride, nullptr);
}

cudaError_t launch_chol_solve(const float4 *U, const int *wide, const double *d, const int *info, int nprob, int K,
                              const SolveIo &io, int *status, cudaStream_t s)
{
    if (K < 1 || K > kCholMaxK) return cudaErrorInvalidValue;
    const size_t smem = sizeof(float4) * (size_t)tri_row(K);
    static SmemAttr smem_rec;
    const cudaError_t e = ensure_smem(smem_rec, (const void *)chol_solve_kernel, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(chol_solve_kernel, dim3((unsigned)nprob), 256, smem, s, U, wide, d, info, K, io, status);
}

}  // namespace dpd
