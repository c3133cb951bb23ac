// libdpd C ABI, least-squares part: dpd_gram, dpd_estimate and
// dpd_estimate_batched (contracts in include/dpd.h, method in dpd_gram.cuh).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <limits>
#include <system_error>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/dpd.h"
#include "dpd_batched.cuh"
#include "dpd_gram.cuh"
#include "dpd_handle.h"

namespace {

bool aligned8(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

// Floats between the forward tables of a batch (16-byte aligned).
size_t table_stride(dpd_handle h) { return ((size_t)dpd::wl_table_floats(h->B, h->T) + 3) & ~(size_t)3; }
size_t factor_size(int K) { return (size_t)K * (K + 1) / 2; }   // values of a packed factor

// p <- `need` values in place of what it held; null, with no error pending, on failure.
template <class T>
bool grow(T *&p, size_t need)
{
    cudaFree(p);
    p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(need, 1) * sizeof(T)) == cudaSuccess) return true;
    p = nullptr;
    cudaGetLastError();
    return false;
}

// Make sure the workspace holds nprob problems with cpp Gram CTAs each at this
// precision and nsamp samples of refinement buffers.  Synchronises the device when it
// grows.  A capacity counts only once all its arrays are there: after a failure the
// next call, however small, allocates them anew.
dpd_status reserve(dpd_handle h, int nprob, int cpp, int precision, int64_t nsamp)
{
    EstimateWorkspace &w = h->est;
    const int K = h->K;
    bool ok = true;
    const size_t part = precision == dpd::kPrecFP32 ? (size_t)dpd::kGramRows * dpd::kGramPartCols
                                                    : (size_t)2 * dpd::kLagEntries;   // floats per CTA
    const size_t parts = (size_t)nprob * cpp * part;
    if (parts > w.partials_cap) {
        cudaDeviceSynchronize();
        w.partials_cap = 0;
        if (!grow(w.partials, parts)) return DPD_ERR_ALLOC;
        w.partials_cap = parts;
    }
    if (nprob > w.nprob) {
        cudaDeviceSynchronize();
        w.nprob = 0;
        const size_t np = (size_t)nprob;
        ok = ok && grow(reinterpret_cast<dpd::GramProblem *&>(w.probs), np);
        ok = ok && grow(w.S, np * dpd::kGramS * dpd::kGramPartCols) && grow(w.Clag, np * dpd::kLagEntries);
        ok = ok && grow(w.G, np * K * K) && grow(w.U, np * factor_size(K)) && grow(w.wide, np);
        ok = ok && grow(w.g, np * K) && grow(w.h64, np * K);
        ok = ok && grow(w.d, np * K) && grow(w.tt, np) && grow(w.info, np);
        ok = ok && grow(w.tab, np * table_stride(h));
        // partial pairs, the completion counter (zero)
        ok = ok && grow(w.norm_part, (size_t)2 * dpd::kFwdNormSlots + 1) &&
             cudaMemset(w.norm_part, 0, ((size_t)2 * dpd::kFwdNormSlots + 1) * sizeof(double)) == cudaSuccess;
        ok = ok && grow(w.ubasis, np * dpd::kUSize) && grow(w.ubasis64, np * dpd::kUSize);
        ok = ok && grow(w.mom_part, std::max<size_t>(np, dpd::kMomBlocks) * dpd::kMomK);
        if (!ok) return DPD_ERR_ALLOC;
        w.nprob = nprob;
    }
    if (w.hK != K || !w.h_G) {
        cudaFreeHost(w.h_G);
        cudaFreeHost(w.h_U);
        cudaFreeHost(w.h_info);
        cudaFreeHost(w.h_norm);
        w.h_G = nullptr;
        w.h_U = nullptr;
        w.h_info = nullptr;
        w.h_norm = nullptr;
        w.hK = 0;
        if (cudaMallocHost(&w.h_G, sizeof(double2) * K * K) != cudaSuccess ||
            cudaMallocHost(&w.h_U, sizeof(float4) * factor_size(K)) != cudaSuccess ||
            cudaMallocHost(&w.h_info, 2 * sizeof(int)) != cudaSuccess ||
            cudaMallocHost(&w.h_norm, 2 * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            return DPD_ERR_ALLOC;
        }
        w.hK = K;
    }
    if (!w.ev_U && cudaEventCreateWithFlags(&w.ev_U, cudaEventDisableTiming) != cudaSuccess) return DPD_ERR_CUDA;
    if (!w.ev_G && cudaEventCreateWithFlags(&w.ev_G, cudaEventDisableTiming) != cudaSuccess) return DPD_ERR_CUDA;
    if (nsamp > w.nsamp) {
        cudaDeviceSynchronize();
        w.nsamp = 0;
        ok = grow(w.y, (size_t)nsamp) && grow(w.e, (size_t)nsamp);
        if (!ok) return DPD_ERR_ALLOC;
        w.nsamp = nsamp;
    }
    return DPD_OK;
}

bool valid_precision(int p) { return p == DPD_PREC_FP32 || p == DPD_PREC_TF32X3 || p == DPD_PREC_BF16X3; }

bool ortho(dpd_handle h) { return h->est_basis == DPD_BASIS_ORTHOGONAL; }

// Basis of statistically orthogonal polynomials for the problems in w.probs, or the one
// problem *one.
dpd_status compute_basis(dpd_handle h, const dpd::GramProblem *one, int nprob, int64_t nmax, cudaStream_t s)
{
    EstimateWorkspace &w = h->est;
    return dpd::launch_basis(one ? nullptr : static_cast<const dpd::GramProblem *>(w.probs),
                             one ? *one : dpd::GramProblem{nullptr, nullptr, 0}, nprob, nmax, h->B, w.mom_part, w.ubasis,
                             w.ubasis64, s) == cudaSuccess
               ? DPD_OK
               : DPD_ERR_CUDA;
}

// Solve for problems [p0, p0 + np): right-hand sides g (w.g), or `rows` rows per problem
// of coefficient-gradient partials added to the coefficients.  Leaves the coefficients in
// w.h64, their FP32 monomial form in `out` (K per problem, of problem 0) and their forward
// tables in w.tab.
dpd_status solve(dpd_handle h, int p0, int np, const float2 *rows, int nrows, float2 *out, cudaStream_t s)
{
    EstimateWorkspace &w = h->est;
    const size_t off = (size_t)p0 * h->K;
    dpd::SolveIo io;
    io.rhs = rows ? nullptr : w.g + off;
    io.rows = rows;
    io.nrows = nrows;
    io.basis = ortho(h) ? w.ubasis64 + (size_t)p0 * dpd::kUSize : nullptr;
    io.h = w.h64 + off;
    io.accumulate = rows ? 1 : 0;
    io.out = out + off;
    io.tstride = (int)table_stride(h);
    io.tab = w.tab + p0 * table_stride(h);
    io.Bp = h->Bp;
    io.Bq = h->Bq;
    io.T = h->T;
    return dpd::launch_chol_solve(w.U + p0 * factor_size(h->K), w.wide + p0, w.d + off, w.info + p0, np, h->K, io,
                                  h->d_status, s) == cudaSuccess
               ? DPD_OK
               : DPD_ERR_CUDA;
}

int gram_cpp(dpd_handle h, int nprob, int64_t n, int precision)
{
    return dpd::gram_ctas_per_problem(precision, h->sm_count, nprob, n);
}

// Gram (+ reduction + assembly) of nprob problems described in w.probs, or of
// the single problem *one (passed by value to the kernels, no copy); G and g
// go to G_out / g_out when given, else to the workspace.  The basis is the
// handle's estimate basis, or the monomials of Eq. 2 with `monomial`.
dpd_status run_gram(dpd_handle h, int nprob, int cpp, int precision, cudaStream_t s,
                    const dpd::GramProblem *one = nullptr, double2 *G_out = nullptr, double2 *g_out = nullptr,
                    bool monomial = false, double2 *G_host = nullptr)
{
    EstimateWorkspace &w = h->est;
    dpd::GramArgs a;
    a.probs = one ? nullptr : static_cast<const dpd::GramProblem *>(w.probs);
    a.one = one ? *one : dpd::GramProblem{nullptr, nullptr, 0};
    a.nprob = nprob;
    a.cpp = cpp;
    a.Bp = h->Bp;
    a.Bq = h->Bq;
    a.T = h->T;
    a.K = h->K;
    a.partials = w.partials;
    a.status = h->d_status;
    a.ubasis = ortho(h) && !monomial ? w.ubasis : nullptr;
    double2 *G = G_out ? G_out : w.G, *g = G_out ? g_out : w.g;
    if (dpd::launch_gram(precision, a, s) != cudaSuccess) return DPD_ERR_CUDA;
    const int D = dpd::gram_distinct(h->B, h->T);
    if (precision == dpd::kPrecFP32) {
        if (dpd::launch_gram_reduce(w.partials, nprob, cpp, D, w.S, s) != cudaSuccess ||
            dpd::launch_gram_assemble(w.S, nprob, h->K, h->Bp, h->B, h->T, G, g, w.tt, G_host, s) != cudaSuccess)
            return DPD_ERR_CUDA;
    } else if (dpd::launch_gram_lag_finish(w.partials, a.probs, a.one, a.ubasis, nprob, cpp, h->K, h->Bp, h->B, h->T,
                                           nprob > 1, w.Clag, G, g, w.tt, G_host, s) != cudaSuccess) {
        return DPD_ERR_CUDA;
    }
    return DPD_OK;
}

// e = t - Psi(u) h for the current coefficients of problem p (its table in w.tab; FP32
// filter); with `norms`, only ||e||^2 and ||t||^2 into the pinned w.h_norm (e itself is not
// written).
dpd_status residual_of(dpd_handle h, int p, const float2 *u, const float2 *t, int64_t n, cudaStream_t s,
                       bool norms = false)
{
    EstimateWorkspace &w = h->est;
    dpd::FwdArgs fa;
    fa.x = u;
    fa.y = w.y;
    fa.n = n;
    fa.tab = w.tab + p * table_stride(h);
    fa.status = h->d_status;
    fa.vec_store = 1;
    fa.host_tab = nullptr;
    // Coefficients live on the device (shared-memory table): 6 samples per thread, 16
    // warps in two groups of 8, 4 stages (GB300, us per 2^22 samples at P = Q = 11, M = 7:
    // 29.3, against 41.5 at the single-stream default of 8 samples per thread); fewer than
    // eight tiles of 3,072 samples per SM go to CTAs of 4 warps (an estimate of 2^18 samples
    // at P = Q = 7, M = 3: 151.0 us against 154.3, with 86 tiles for 152 SMs).
    dpd::FwdLaunch L;
    const bool few = n < 8 * 3072 * (int64_t)h->sm_count;
    L.mode = dpd::kModePackedFma;
    L.V = 6;
    L.warps = few ? 4 : 16;
    L.group = few ? 0 : 8;
    L.stages = few ? 3 : 4;
    const bool aligned16 = ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(t)) & 15u) == 0;
    if (aligned16) {
        // The filter writes e = t - Psi(u) h itself (no separate residual
        // pass), or only sums |e|^2 and |t|^2.
        L.mode = dpd::kModePackedFma | dpd::kModeSubtract | (norms ? dpd::kModeNorms : 0);
        fa.y = w.e;
        fa.sub = t;
        fa.norms = w.norm_part;
        fa.norms_out = w.h_norm;
        return dpd::launch_fwd_any(h->B, h->T, fa, L, h->sm_count, s) == cudaSuccess ? DPD_OK : DPD_ERR_CUDA;
    }
    if ((reinterpret_cast<uintptr_t>(u) & 15u) != 0) {
        L.use_tma = 0;
        L.V = 4;
    }
    if (dpd::launch_fwd_any(h->B, h->T, fa, L, h->sm_count, s) != cudaSuccess) return DPD_ERR_CUDA;
    if (norms)
        return dpd::launch_residual_norm(t, w.y, n, nullptr, w.norm_part, w.h_norm, s) ==
                       cudaSuccess
                   ? DPD_OK
                   : DPD_ERR_CUDA;
    if (dpd::launch_residual(t, w.y, n, w.e, s) != cudaSuccess) return DPD_ERR_CUDA;
    return DPD_OK;
}

// One refinement step of problem p:  h64[p] += G^{-1} Psi^H (t - Psi h).
dpd_status refine_once(dpd_handle h, int p, const float2 *u, const float2 *t, int64_t n, float2 *out, cudaStream_t s)
{
    EstimateWorkspace &w = h->est;
    const int K = h->K;
    dpd_status st = residual_of(h, p, u, t, n, s);
    if (st != DPD_OK) return st;
    dpd::AdjArgs aa;
    aa.x = u;
    aa.gy = w.e;
    aa.n = n;
    aa.gx = nullptr;
    aa.partials = h->d_partials;
    aa.adj_tab = h->d_adj_tab;
    aa.status = h->d_status;
    dpd::AdjLaunch al = h->adj;
    const int64_t need = (n + 1023) / 1024;
    if (al.gh_blocks > need) al.gh_blocks = (int)need;
    if (al.gh_blocks > h->rows_max) al.gh_blocks = h->rows_max;
    if (al.gh_blocks < 1) al.gh_blocks = 1;
    if (dpd::launch_adj_any(h->B, aa, al, h->T, h->Bp, h->Bq, K, h->sm_count, s) != cudaSuccess) return DPD_ERR_CUDA;
    return solve(h, p, 1, h->d_partials, al.gh_blocks, out, s);   // Psi^H (t - Psi h): the sum of the rows
}

// Refinement of all problems of a batch together, each step one launch per
// kernel: the batched forward filter (6 samples per thread, 16 warps in groups of
// 8, 4 stages) into the residual buffers, e = t - Psi h, the coefficient gradients
// of all problems (a few CTAs per problem and tap group) and the batched solve.
// Needs 16-byte aligned inputs u (the bulk-copy pipelines); the caller checks that.
dpd_status refine_batched(dpd_handle h, const std::vector<dpd::GramProblem> &probs, int64_t nmax, int iters,
                          float2 *out, cudaStream_t s)
{
    EstimateWorkspace &w = h->est;
    const int K = h->K, count = (int)probs.size();
    const int64_t stride = (nmax + 1) & ~int64_t(1);   // keeps every e_p 16-byte aligned
    const int tstride = (int)table_stride(h);
    constexpr int V = 6, warps = 16, group = 8, stages = 4;
    // Two sub-blocks of 3,072 samples to an item where that leaves four items per SM
    // (256 x 2^16 at K = 97: 139 us against 147 with one).
    int64_t total = 0;
    for (const dpd::GramProblem &pr : probs) total += pr.n / (2 * warps * 32 * V);
    const int nsub = total >= 4 * (int64_t)h->sm_count ? dpd::batch_nsub(warps, group, stages, V) : 1;
    const int S = nsub * warps * 32 * V;
    // CTAs of a problem and tap group in the coefficient gradient, one per SM: the rounds
    // that the launch takes, each a share of the samples and a CTA's start and end, about
    // kCtaSamples samples' time.  A batched fit with two refinements, us, with 1, 2, 3, 4, 8
    // rows: 256 x 2^16 at K = 97 1611 1602 1607 1624 1694; 64 x 2^18 at K = 33 1101 993 1048
    // 999 1015; 16 x 2^20 at K = 51 2113 1529 1319 1232 1079.  The choice here is within 2 %
    // of the best of 1 .. 11 on these and four more.
    const int groups = (h->T + h->adj.tap_group - 1) / h->adj.tap_group;
    int rows = 1;
    int64_t best = INT64_MAX;
    for (int r = 1; r <= std::max(8, h->sm_count / (groups * count)); ++r) {
        constexpr int64_t kCtaSamples = 7000;
        const int64_t rounds = ((int64_t)groups * count * r + h->sm_count - 1) / h->sm_count;
        const int64_t cost = rounds * ((nmax + r - 1) / r + kCtaSamples);
        if (cost < best) {
            best = cost;
            rows = r;
        }
    }
    std::vector<dpd::BatchStream> st((size_t)count);
    std::vector<dpd::BatchItem> items;
    std::vector<dpd::AdjArgs> adj((size_t)count);
    for (int p = 0; p < count; ++p) {
        float2 *ep = w.e + (size_t)p * stride;
        st[p] = {probs[p].u, ep, probs[p].n, h->B, h->T, p * tstride, tstride * 4, probs[p].t};   // e = t - Psi h
        for (int64_t t = 0; t * S < probs[p].n; ++t) items.push_back({p, dpd::batch_tile(t * nsub, nsub)});
        dpd::AdjArgs &a = adj[p];
        a.x = probs[p].u;
        a.gy = ep;
        a.n = probs[p].n;
        a.gx = nullptr;
        a.adj_tab = nullptr;
        a.host_adj_tab = nullptr;
        a.status = h->d_status;
    }
    if ((size_t)count > w.bprob_cap) {
        cudaDeviceSynchronize();
        w.bprob_cap = 0;
        if (!grow(reinterpret_cast<dpd::BatchStream *&>(w.bstreams), (size_t)count) ||
            !grow(reinterpret_cast<dpd::AdjArgs *&>(w.badj), (size_t)count))
            return DPD_ERR_ALLOC;
        w.bprob_cap = (size_t)count;
    }
    if ((size_t)count * rows > w.bpart_cap) {
        cudaDeviceSynchronize();
        w.bpart_cap = 0;
        if (!grow(w.bpart, (size_t)count * rows * K)) return DPD_ERR_ALLOC;
        w.bpart_cap = (size_t)count * rows;
    }
    if (items.size() > w.bitems_cap) {
        cudaDeviceSynchronize();
        w.bitems_cap = 0;
        if (!grow(reinterpret_cast<dpd::BatchItem *&>(w.bitems), items.size())) return DPD_ERR_ALLOC;
        w.bitems_cap = items.size();
    }
    for (int p = 0; p < count; ++p) adj[p].partials = w.bpart + (size_t)p * rows * K;
    // Stream-ordered uploads from pageable memory: the runtime stages the host
    // data before each call returns (no device synchronisation), so the vectors
    // may go out of scope and the host goes on enqueuing the launches.
    if (cudaMemcpyAsync(w.bstreams, st.data(), sizeof(dpd::BatchStream) * count, cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(w.bitems, items.data(), sizeof(dpd::BatchItem) * items.size(), cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(w.badj, adj.data(), sizeof(dpd::AdjArgs) * count, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return DPD_ERR_CUDA;
    dpd::BatchArgs ba;
    ba.streams = static_cast<const dpd::BatchStream *>(w.bstreams);
    ba.items = static_cast<const dpd::BatchItem *>(w.bitems);
    ba.nitems = (int)items.size();
    ba.nstreams = count;
    ba.tabs = w.tab;
    ba.tab_floats = (int64_t)count * tstride;
    ba.status = h->d_status;
    ba.gw = group;
    ba.nsub = nsub;
    const bool small = h->B <= 5 && h->T <= 7;
    for (int it = 0; it < iters; ++it) {
        const cudaError_t fe = small ? dpd::launch_batched_57(ba, V, warps, stages, 0, h->sm_count, s)
                                     : dpd::launch_batched_68(ba, V, warps, stages, 0, h->sm_count, s);
        if (fe != cudaSuccess) return DPD_ERR_CUDA;   // the filter wrote e_p = t_p - Psi h_p
        if (dpd::launch_adj_gh_many_any(h->B, static_cast<const dpd::AdjArgs *>(w.badj), count, rows, h->adj.tap_group,
                                        h->T, h->Bp, h->Bq, K, s) != cudaSuccess)
            return DPD_ERR_CUDA;
        const dpd_status st2 = solve(h, 0, count, w.bpart, rows, out, s);
        if (st2 != DPD_OK) return st2;
    }
    return DPD_OK;
}

// Condition number of A = D G D = U Delta U^H (the equilibrated Gram matrix, D =
// diag(G)^{-1/2}) in the 2-norm: the largest eigenvalue of A (products with A
// itself, formed from G) times the largest eigenvalue of A^{-1} =
// U^{-H} Delta^{-1} U^{-1} (two triangular solves with the factor), FP64 on the
// host.  Complex vectors and matrices are kept as separate real and imaginary
// arrays, padded to an even length N with zeros, and processed two elements
// at a time with GCC vector types (portable across x86-64 and AArch64): every
// inner product is split over several vector partial sums, so no loop is one
// long chain of dependent additions.
namespace cond {

typedef double v2d __attribute__((vector_size(16)));

inline v2d ld2(const double *p) { return *reinterpret_cast<const v2d *>(p); }   // 16-byte aligned
inline void st2(double *p, v2d v) { *reinterpret_cast<v2d *>(p) = v; }
inline double hsum(v2d v) { return v[0] + v[1]; }

// Padded split storage: rows of N (even) doubles; the heap blocks of
// std::vector are 16-byte aligned (the allocator's fundamental alignment on
// x86-64 and AArch64), so every row starts on a 16-byte boundary.
struct Split {
    int rows = 0, N = 0;
    std::vector<double> re, im;
    Split(int rows_, int n) : rows(rows_), N(n), re((size_t)rows * n, 0.0), im((size_t)rows * n, 0.0) {}
    double *r(int row) { return re.data() + (size_t)row * N; }
    double *i(int row) { return im.data() + (size_t)row * N; }
    const double *r(int row) const { return re.data() + (size_t)row * N; }
    const double *i(int row) const { return im.data() + (size_t)row * N; }
};

// y = M x for the first `rows` rows of M (row-major, padded width N).  Four rows at
// a time, so every x element is loaded once per four rows.
void matvec(const Split &M, int rows, const double *xr, const double *xi, double *yr, double *yi)
{
    const int N = M.N;
    int i = 0;
    for (; i + 4 <= rows; i += 4) {
        v2d sr[4] = {}, si[4] = {};
        for (int k = 0; k < N; k += 2) {
            const v2d a = ld2(xr + k), b = ld2(xi + k);
            for (int q = 0; q < 4; ++q) {
                const v2d mr = ld2(M.r(i + q) + k), mi = ld2(M.i(i + q) + k);
                sr[q] += mr * a - mi * b;
                si[q] += mr * b + mi * a;
            }
        }
        for (int q = 0; q < 4; ++q) {
            yr[i + q] = hsum(sr[q]);
            yi[i + q] = hsum(si[q]);
        }
    }
    for (; i < rows; ++i) {
        v2d sr = {0, 0}, si = {0, 0};
        for (int k = 0; k < N; k += 2) {
            const v2d a = ld2(xr + k), b = ld2(xi + k), mr = ld2(M.r(i) + k), mi = ld2(M.i(i) + k);
            sr += mr * a - mi * b;
            si += mr * b + mi * a;
        }
        yr[i] = hsum(sr);
        yi[i] = hsum(si);
    }
}

// Products of rows i .. i + 3 of M (conjugated with CONJ) with x[from .. to), from and to
// even: every x element is loaded once per four rows.
template <bool CONJ>
void dot4(const Split &M, int i, int from, int to, const double *xr, const double *xi, double *sr, double *si)
{
    v2d ar[4] = {}, ai[4] = {};
    const double *mr[4], *mi[4];
    for (int q = 0; q < 4; ++q) {
        const int row = std::min(i + q, M.rows - 1);
        mr[q] = M.r(row);
        mi[q] = M.i(row);
    }
    for (int k = from; k < to; k += 2) {
        const v2d a = ld2(xr + k), b = ld2(xi + k);
        for (int q = 0; q < 4; ++q) {
            const v2d r = ld2(mr[q] + k), c = ld2(mi[q] + k);
            ar[q] += CONJ ? r * a + c * b : r * a - c * b;
            ai[q] += CONJ ? r * b - c * a : r * b + c * a;
        }
    }
    for (int q = 0; q < 4; ++q) {
        sr[q] = hsum(ar[q]);
        si[q] = hsum(ai[q]);
    }
}

// x <- T^{-1} x for a unit triangular T: lower (its strict part in L's rows) or, with
// CONJ, the conjugate transpose of the lower one whose transpose has its strict part in L's
// rows.  Four rows at a time: the finished elements' products, then the block's own.
template <bool CONJ>
void triangular_solve(const Split &L, double *xr, double *xi)
{
    const int K = L.rows, N = L.N, last = (K - 1) & ~3;
    for (int b = 0; b <= last; b += 4) {
        const int i = CONJ ? last - b : b, rows = std::min(4, K - i);
        double sr[4], si[4];
        dot4<CONJ>(L, i, CONJ ? i + 4 : 0, CONJ ? N : i, xr, xi, sr, si);
        for (int j = 0; j < rows; ++j) {
            const int q = CONJ ? rows - 1 - j : j;
            double re = xr[i + q] - sr[q], im = xi[i + q] - si[q];
            for (int k = CONJ ? q + 1 : 0; k < (CONJ ? rows : q); ++k) {
                const double mr = L.r(i + q)[i + k], mi = CONJ ? -L.i(i + q)[i + k] : L.i(i + q)[i + k];
                re -= mr * xr[i + k] - mi * xi[i + k];
                im -= mr * xi[i + k] + mi * xr[i + k];
            }
            xr[i + q] = re;
            xi[i + q] = im;
        }
    }
}

double2 dotc(int N, const double *a_r, const double *a_i, const double *b_r, const double *b_i)   // a^H b
{
    v2d sr[2] = {}, si[2] = {};
    int k = 0;
    for (; k + 4 <= N; k += 4)
        for (int h = 0; h < 2; ++h) {
            const v2d ar = ld2(a_r + k + 2 * h), ai = ld2(a_i + k + 2 * h), br = ld2(b_r + k + 2 * h),
                      bi = ld2(b_i + k + 2 * h);
            sr[h] += ar * br + ai * bi;
            si[h] += ar * bi - ai * br;
        }
    for (; k < N; k += 2) {
        const v2d ar = ld2(a_r + k), ai = ld2(a_i + k), br = ld2(b_r + k), bi = ld2(b_i + k);
        sr[0] += ar * br + ai * bi;
        si[0] += ar * bi - ai * br;
    }
    return make_double2(hsum(sr[0] + sr[1]), hsum(si[0] + si[1]));
}

// Largest root of the Lanczos tridiagonal by Sturm-sequence bisection,
// starting from `floor_` (the Ritz values only grow with the step count).
double ritz_max(const std::vector<double> &al, const std::vector<double> &be, double floor_)
{
    const int n = (int)al.size();
    double lo = al[0], hi = al[0];
    for (int i = 0; i < n; ++i) {
        const double r = (i > 0 ? std::fabs(be[i - 1]) : 0.0) + (i + 1 < n ? std::fabs(be[i]) : 0.0);
        lo = std::min(lo, al[i] - r);
        hi = std::max(hi, al[i] + r);
    }
    if (floor_ > lo && floor_ < hi) lo = floor_;
    auto below = [&](double x) {   // eigenvalues of the tridiagonal below x
        int c = 0;
        double dd = 1.0;
        for (int i = 0; i < n; ++i) {
            dd = al[i] - x - (i > 0 ? be[i - 1] * be[i - 1] / dd : 0.0);
            if (dd == 0.0) dd = -1e-300;
            if (dd < 0.0) ++c;
        }
        return c;
    };
    for (int it = 0; it < 200 && hi - lo > 1e-15 * std::fabs(hi); ++it) {
        const double mid = 0.5 * (lo + hi);
        if (below(mid) >= n)
            hi = mid;
        else
            lo = mid;
    }
    return 0.5 * (lo + hi);
}

// z <- (T - lam)^{-1} z for the Lanczos tridiagonal T, by elimination with partial
// pivoting (a zero pivot, lam being an eigenvalue, becomes the smallest normal number).
void tridiagonal_solve(const std::vector<double> &al, const std::vector<double> &be, double lam, std::vector<double> &z)
{
    const int n = (int)al.size();
    std::vector<double> p(n), q(n, 0.0), r(n, 0.0);   // the diagonal and the two above it
    for (int i = 0; i < n; ++i) p[i] = al[i] - lam;
    for (int i = 0; i + 1 < n; ++i) q[i] = be[i];
    auto pivot = [](double v) { return v != 0.0 ? v : std::numeric_limits<double>::min(); };
    for (int i = 0; i + 1 < n; ++i) {
        const double s = be[i];
        if (std::fabs(s) > std::fabs(p[i])) {   // rows i and i + 1 change places
            const double m = p[i] / s, above = q[i];
            p[i] = s;
            q[i] = p[i + 1];
            r[i] = q[i + 1];
            p[i + 1] = above - m * q[i];
            q[i + 1] = -m * r[i];
            std::swap(z[i], z[i + 1]);
            z[i + 1] -= m * z[i];
        } else {
            const double m = s / pivot(p[i]);
            p[i + 1] -= m * q[i];
            z[i + 1] -= m * z[i];
        }
    }
    for (int i = n - 1; i >= 0; --i) {
        double v = z[i];
        if (i + 1 < n) v -= q[i] * z[i + 1];
        if (i + 2 < n) v -= r[i] * z[i + 2];
        z[i] = v / pivot(p[i]);
    }
}

// Largest eigenvalue of the Hermitian positive definite operator `op` (w = op
// v on padded split vectors of length N, K of them significant) by Lanczos
// with full reorthogonalisation (classical Gram-Schmidt, repeated once when
// the first pass cancels more than half of the squared norm: without it, a
// vector formed after the Krylov space has converged keeps rounding-level
// components along the earlier ones, and the Ritz values of the next steps
// overshoot the spectrum), stopped once the largest Ritz value changes by
// less than 1e-12 relative over five steps (checked at steps 10, 15, ..., at
// most 40).  On these clustered spectra plain power iterations stay
// percent-level low after 100 steps; this converges to about 1e-11 in 15-40.
// `ritz`: the eigenvector's approximation (one row of N), or null.
template <class Op>
double largest(int K, int N, Op op, Split *ritz = nullptr)
{
    const int m = std::min(K, 40);
    Split Q(m + 1, N), W(1, N);
    std::vector<double> cr(m + 1), ci(m + 1), al, be;
    double *wr = W.r(0), *wi = W.i(0);
    double nv = 0;
    for (int i = 0; i < K; ++i) {
        Q.r(0)[i] = 1.0 + 0.01 * i;
        Q.i(0)[i] = 0.003 * i;
        nv += Q.r(0)[i] * Q.r(0)[i] + Q.i(0)[i] * Q.i(0)[i];
    }
    nv = std::sqrt(nv);
    for (int i = 0; i < K; ++i) {
        Q.r(0)[i] /= nv;
        Q.i(0)[i] /= nv;
    }
    double prev = -1.0, lam = 0.0;
    for (int j = 0; j < m; ++j) {
        op(Q.r(j), Q.i(j), wr, wi);
        al.push_back(dotc(N, Q.r(j), Q.i(j), wr, wi).x);
        double before = dotc(N, wr, wi, wr, wi).x;
        for (int pass = 0; pass < 2; ++pass) {
            // c = Q^H w over the j + 1 vectors so far (the rows of Q), then w -= Q^T c.
            for (int i = 0; i <= j; ++i) {
                const double2 c = dotc(N, Q.r(i), Q.i(i), wr, wi);
                cr[i] = c.x;
                ci[i] = c.y;
            }
            for (int i = 0; i <= j; ++i) {
                const v2d a = v2d{cr[i], cr[i]}, b = v2d{ci[i], ci[i]};
                const double *ur = Q.r(i), *ui = Q.i(i);
                for (int k = 0; k < N; k += 2) {
                    const v2d qr2 = ld2(ur + k), qi2 = ld2(ui + k);
                    st2(wr + k, ld2(wr + k) - (a * qr2 - b * qi2));
                    st2(wi + k, ld2(wi + k) - (a * qi2 + b * qr2));
                }
            }
            const double after = dotc(N, wr, wi, wr, wi).x;
            if (after >= 0.5 * before) break;
            before = after;
        }
        const bool check = j >= 10 && (j % 5 == 0 || j == m - 1);
        if (check || j == m - 1) {
            lam = ritz_max(al, be, prev);
            if (check && prev > 0 && std::fabs(lam - prev) <= 1e-12 * lam) break;
            prev = lam * (1.0 - 1e-15);   // bisection floor for the next check
        }
        const double bn = std::sqrt(dotc(N, wr, wi, wr, wi).x);
        if (!(bn > 1e-14 * std::fabs(al.back()))) {   // invariant subspace: its Ritz values are exact
            lam = ritz_max(al, be, prev);
            break;
        }
        be.push_back(bn);
        for (int k = 0; k < N; ++k) {
            Q.r(j + 1)[k] = wr[k] / bn;
            Q.i(j + 1)[k] = wi[k] / bn;
        }
    }
    if (ritz) {   // two steps of inverse iteration on the tridiagonal, in the Lanczos basis
        std::vector<double> z(al.size(), 1.0);
        for (int step = 0; step < 2; ++step) {
            tridiagonal_solve(al, be, lam, z);
            double top = 0.0;
            for (double v : z) top = std::max(top, std::fabs(v));
            for (double &v : z) v /= top;
        }
        for (size_t i = 0; i < z.size(); ++i)
            for (int k = 0; k < K; ++k) {
                ritz->r(0)[k] += z[i] * Q.r((int)i)[k];
                ritz->i(0)[k] += z[i] * Q.i((int)i)[k];
            }
    }
    return lam;
}

// Largest eigenvalue of D G D (D = diag(G)^{-1/2}, as the factorisation forms it).
double largest_dgd(const double2 *G, int K)
{
    const int N = (K + 1) & ~1;
    std::vector<double> d(K);
    for (int i = 0; i < K; ++i) {
        const double gii = G[(size_t)i * K + i].x;
        d[i] = gii > 0.0 ? 1.0 / std::sqrt(gii) : 0.0;
    }
    Split A(K, N);
    for (int i = 0; i < K; ++i)
        for (int k = 0; k < K; ++k) {
            A.r(i)[k] = G[(size_t)i * K + k].x * d[i] * d[k];
            A.i(i)[k] = G[(size_t)i * K + k].y * d[i] * d[k];
        }
    return largest(K, N, [&](const double *vr, const double *vi, double *wr, double *wi) {
        matvec(A, K, vr, vi, wr, wi);
    });
}

// Largest eigenvalue of (D G D)^{-1} with the packed factor of D G D = U Delta U^H
// (launch_chol; `wide`: in FP64): two triangular solves per product, by rows of U and of
// U^T.  A factor in pairs is a little off (about 2^-42 of the diagonal), and so is the
// eigenvector that Lanczos finds with it, but the value is then taken as the Rayleigh
// quotient of that vector with a product refined against G itself, whose error is that of
// the vector squared.  Of G the lower triangle, as in the factorisation: the end products
// of the tensor-core form leave the upper one up to 1e-10 off its conjugate.
double largest_inverse(const float4 *Up, bool wide, const double2 *G, int K)
{
    const int N = (K + 1) & ~1;
    Split U(K, N), Ut(K, N);
    std::vector<double> dinv(K);
    for (int i = 0; i < K; ++i) {
        const float4 *row = Up + factor_size(i);   // i (i + 1) / 2
        const double2 *row64 = reinterpret_cast<const double2 *>(row);
        for (int k = 0; k < i; ++k) {
            Ut.r(k)[i] = U.r(i)[k] = wide ? row64[k].x : (double)row[k].x + (double)row[k].z;
            Ut.i(k)[i] = U.i(i)[k] = wide ? row64[k].y : (double)row[k].y + (double)row[k].w;
        }
        dinv[i] = wide ? row64[i].x : (double)row[i].x + (double)row[i].z;
    }
    auto solve = [&](const double *vr, const double *vi, double *wr, double *wi) {
        std::copy(vr, vr + N, wr);
        std::copy(vi, vi + N, wi);
        triangular_solve<false>(U, wr, wi);
        for (int i = 0; i < K; ++i) {
            wr[i] *= dinv[i];
            wi[i] *= dinv[i];
        }
        triangular_solve<true>(Ut, wr, wi);
    };
    Split v(1, N), w(1, N), res(1, N), cor(1, N);
    const double lam = largest(K, N, solve, &v);
    solve(v.r(0), v.i(0), w.r(0), w.i(0));
    std::vector<double> d(K), xr(K), xi(K);
    for (int i = 0; i < K; ++i) {
        const double gii = G[(size_t)i * K + i].x;
        d[i] = gii > 0.0 ? 1.0 / std::sqrt(gii) : 0.0;
        xr[i] = d[i] * w.r(0)[i];
        xi[i] = d[i] * w.i(0)[i];
    }
    std::vector<double> yr(K), yi(K);   // G x
    for (int i = 0; i < K; ++i) {
        const double2 *row = G + (size_t)i * K;
        double sr = row[i].x * xr[i], si = row[i].x * xi[i];
        for (int k = 0; k < i; ++k) {
            const double2 g = row[k];
            sr += g.x * xr[k] - g.y * xi[k];
            si += g.x * xi[k] + g.y * xr[k];
            yr[k] += g.x * xr[i] + g.y * xi[i];
            yi[k] += g.x * xi[i] - g.y * xr[i];
        }
        yr[i] = sr;
        yi[i] = si;
    }
    for (int i = 0; i < K; ++i) {   // v - D G D w
        res.r(0)[i] = v.r(0)[i] - d[i] * yr[i];
        res.i(0)[i] = v.i(0)[i] - d[i] * yi[i];
    }
    solve(res.r(0), res.i(0), cor.r(0), cor.i(0));
    double num = 0.0, den = 0.0;
    for (int k = 0; k < K; ++k) {
        const double a = v.r(0)[k], b = v.i(0)[k];
        num += a * (w.r(0)[k] + cor.r(0)[k]) + b * (w.i(0)[k] + cor.i(0)[k]);
        den += a * a + b * b;
    }
    const double quotient = num / den;
    return std::isfinite(quotient) && quotient > 0.0 ? quotient : lam;
}

}  // namespace cond

dpd_status check_inputs(dpd_handle h, const void *u, const void *t, int64_t n, int precision)
{
    if (!h || n < 1 || !u || !aligned8(u) || (t && !aligned8(t))) return DPD_ERR_INVALID_ARGUMENT;
    if (!valid_precision(precision)) return DPD_ERR_INVALID_ARGUMENT;
    if (n > ((int64_t)1 << 40)) return DPD_ERR_UNSUPPORTED;
    if (dpd::gram_distinct(h->B, h->T) > dpd::kGramS) return DPD_ERR_UNSUPPORTED;
    return DPD_OK;
}

}  // namespace

void free_estimate_workspace(EstimateWorkspace &w)
{
    cudaFree(w.probs);
    cudaFree(w.partials);
    cudaFree(w.Clag);
    cudaFree(w.S);
    cudaFree(w.G);
    cudaFree(w.g);
    cudaFree(w.U);
    cudaFree(w.wide);
    cudaFree(w.h64);
    cudaFree(w.d);
    cudaFree(w.tt);
    cudaFree(w.info);
    cudaFree(w.tab);
    cudaFree(w.y);
    cudaFree(w.e);
    cudaFree(w.norm_part);
    cudaFree(w.ubasis);
    cudaFree(w.ubasis64);
    cudaFree(w.mom_part);
    cudaFree(w.bstreams);
    cudaFree(w.bitems);
    cudaFree(w.badj);
    cudaFree(w.bpart);
    cudaFreeHost(w.h_G);
    cudaFreeHost(w.h_U);
    cudaFreeHost(w.h_info);
    cudaFreeHost(w.h_norm);
    if (w.ev_U) cudaEventDestroy(w.ev_U);
    if (w.ev_G) cudaEventDestroy(w.ev_G);
    w = EstimateWorkspace();
}

extern "C" {

dpd_status dpd_set_estimate_basis(dpd_handle h, int basis)
{
    if (!h || (basis != DPD_BASIS_MONOMIAL && basis != DPD_BASIS_ORTHOGONAL)) return DPD_ERR_INVALID_ARGUMENT;
    h->est_basis = basis;
    return DPD_OK;
}

dpd_status dpd_gram(dpd_handle h, const void *u, const void *t, int64_t n, int precision, void *G, void *g,
                    double *tt, void *stream)
{
    dpd_status st = check_inputs(h, u, t, n, precision);
    if (st != DPD_OK) return st;
    if (!G || !aligned8(G) || (g && (!t || !aligned8(g)))) return DPD_ERR_INVALID_ARGUMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int cpp = gram_cpp(h, 1, n, precision);
    if ((st = reserve(h, 1, cpp, precision, 0)) != DPD_OK) return st;
    // Psi of Eq. 2 (the monomial basis, whatever the handle's estimate basis);
    // the problem travels by value in the kernel arguments.
    const dpd::GramProblem pr{static_cast<const float2 *>(u), static_cast<const float2 *>(t), n};
    if ((st = run_gram(h, 1, cpp, precision, s, &pr, static_cast<double2 *>(G), static_cast<double2 *>(g), true)) !=
        DPD_OK)
        return st;
    if (tt && t && (cudaMemcpyAsync(tt, h->est.tt, sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                    cudaStreamSynchronize(s) != cudaSuccess))
        return DPD_ERR_CUDA;
    return DPD_OK;
}

dpd_status dpd_estimate(dpd_handle h, const void *u, const void *t, int64_t n, int precision, int refine_iters,
                        void *h_out, double *stats, void *stream)
{
    dpd_status st = check_inputs(h, u, t, n, precision);
    if (st != DPD_OK) return st;
    if (!t || !h_out || !aligned8(h_out) || refine_iters < 0 || refine_iters > 100) return DPD_ERR_INVALID_ARGUMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int cpp = gram_cpp(h, 1, n, precision);
    if ((st = reserve(h, 1, cpp, precision, (refine_iters > 0 || stats) ? n : 0)) != DPD_OK) return st;
    EstimateWorkspace &w = h->est;
    const dpd::GramProblem pr{static_cast<const float2 *>(u), static_cast<const float2 *>(t), n};
    if (ortho(h) && (st = compute_basis(h, &pr, 1, n, s)) != DPD_OK) return st;
    // For the statistics the kernels write G, the factor and the sums of squares to
    // pinned host memory too (a copy in the stream would hold up the kernel behind it),
    // and the pivot status: the host condition estimate (Lanczos on D G D from G, and on
    // its inverse) runs during the factorisation and the refinement instead of after
    // them, and the solves skip a failed factorisation on the device.
    const int K = h->K;
    if ((st = run_gram(h, 1, cpp, precision, s, &pr, nullptr, nullptr, false, stats ? w.h_G : nullptr)) != DPD_OK)
        return st;
    if (stats && cudaEventRecord(w.ev_G, s) != cudaSuccess) return DPD_ERR_CUDA;
    if (dpd::launch_chol(w.G, 1, K, w.U, w.wide, w.d, w.info, stats ? w.h_U : nullptr, w.h_info, h->d_status, s) !=
            cudaSuccess ||
        cudaEventRecord(w.ev_U, s) != cudaSuccess)
        return DPD_ERR_CUDA;
    float2 *out = static_cast<float2 *>(h_out);
    if ((st = solve(h, 0, 1, nullptr, 0, out, s)) != DPD_OK) return st;
    for (int i = 0; i < refine_iters; ++i)
        if ((st = refine_once(h, 0, pr.u, pr.t, n, out, s)) != DPD_OK) return st;
    if (stats && (st = residual_of(h, 0, pr.u, pr.t, n, s, true)) != DPD_OK) return st;
    // The two Lanczos runs overlap the queued device work: the one on D G D
    // (a second host thread) as soon as G has landed, the one on the inverse
    // once the factor has.
    double lmax = 0.0, linv = 0.0;
    std::thread dgd_run;
    bool threaded = false;
    if (stats) {
        if (cudaEventSynchronize(w.ev_G) != cudaSuccess) return DPD_ERR_CUDA;
        try {
            dgd_run = std::thread([&] { lmax = cond::largest_dgd(w.h_G, K); });
            threaded = true;
        } catch (const std::system_error &) {   // no thread available: on this one, below
        }
    }
    const bool synced = cudaEventSynchronize(w.ev_U) == cudaSuccess;
    const int info = synced ? w.h_info[0] : 0;
    if (synced && stats && info == 0) linv = cond::largest_inverse(w.h_U, w.h_info[1] != 0, w.h_G, K);
    if (threaded) dgd_run.join();
    if (!synced) return DPD_ERR_CUDA;
    if (stats && !threaded) lmax = cond::largest_dgd(w.h_G, K);
    const double cond = lmax * linv;
    if (cudaStreamSynchronize(s) != cudaSuccess) return DPD_ERR_CUDA;
    if (info != 0) return DPD_ERR_NOT_SPD;
    if (stats) {
        stats[0] = cond;
        stats[1] = w.h_norm[1] > 0 ? w.h_norm[0] / w.h_norm[1] : 0.0;
    }
    return DPD_OK;
}

dpd_status dpd_estimate_batched(dpd_handle h, const void *const *u, const void *const *t, const int64_t *n,
                                int count, int precision, int refine_iters, void *h_out, int *info_out, void *stream)
{
    if (!h || count < 1 || !u || !t || !n || !h_out || !aligned8(h_out)) return DPD_ERR_INVALID_ARGUMENT;
    if (refine_iters < 0 || refine_iters > 100 || !valid_precision(precision)) return DPD_ERR_INVALID_ARGUMENT;
    if (dpd::gram_distinct(h->B, h->T) > dpd::kGramS) return DPD_ERR_UNSUPPORTED;
    std::vector<dpd::GramProblem> probs((size_t)count);
    int64_t nmax = 1;
    for (int i = 0; i < count; ++i) {
        if (n[i] < 1 || !u[i] || !t[i] || !aligned8(u[i]) || !aligned8(t[i])) return DPD_ERR_INVALID_ARGUMENT;
        probs[i] = {static_cast<const float2 *>(u[i]), static_cast<const float2 *>(t[i]), n[i]};
        nmax = std::max(nmax, n[i]);
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int cpp = gram_cpp(h, count, nmax, precision);
    // Refinement of all problems together needs 16-byte aligned inputs and one
    // residual buffer per problem; otherwise the problems are refined one by one.
    bool together = refine_iters > 0 && count > 1;
    for (int i = 0; i < count && together; ++i) together = (reinterpret_cast<uintptr_t>(u[i]) & 15u) == 0;
    const int64_t nsamp = refine_iters > 0 ? (together ? ((nmax + 1) & ~int64_t(1)) * count : nmax) : 0;
    dpd_status st = reserve(h, count, cpp, precision, nsamp);
    if (st != DPD_OK) return st;
    EstimateWorkspace &w = h->est;
    if (cudaMemcpyAsync(w.probs, probs.data(), sizeof(dpd::GramProblem) * count, cudaMemcpyHostToDevice, s) !=
        cudaSuccess)
        return DPD_ERR_CUDA;
    if (ortho(h) && (st = compute_basis(h, nullptr, count, nmax, s)) != DPD_OK) return st;
    if ((st = run_gram(h, count, cpp, precision, s)) != DPD_OK) return st;
    if (dpd::launch_chol(w.G, count, h->K, w.U, w.wide, w.d, w.info, nullptr, nullptr, h->d_status, s) != cudaSuccess)
        return DPD_ERR_CUDA;
    float2 *out = static_cast<float2 *>(h_out);
    if ((st = solve(h, 0, count, nullptr, 0, out, s)) != DPD_OK) return st;
    // The pivot status comes back here only for the refinement problem by
    // problem, which skips problems that did not factor; refined together, the
    // launches are queued behind the solve without a host round trip and the
    // status is read at the end.
    std::vector<int> info((size_t)count);
    if (!together && (cudaMemcpyAsync(info.data(), w.info, sizeof(int) * count, cudaMemcpyDeviceToHost, s) !=
                          cudaSuccess ||
                      cudaStreamSynchronize(s) != cudaSuccess))
        return DPD_ERR_CUDA;
    if (together) {   // problems that did not factor keep unspecified coefficients
        if ((st = refine_batched(h, probs, nmax, refine_iters, out, s)) != DPD_OK) return st;
    } else {
        for (int it = 0; it < refine_iters; ++it)
            for (int p = 0; p < count; ++p)
                if (info[p] == 0 && (st = refine_once(h, p, probs[p].u, probs[p].t, probs[p].n, out, s)) != DPD_OK)
                    return st;
    }
    if (together &&
        cudaMemcpyAsync(info.data(), w.info, sizeof(int) * count, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return DPD_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return DPD_ERR_CUDA;
    bool any_bad = false;
    for (int i = 0; i < count; ++i) any_bad |= info[i] != 0;
    if (info_out) std::copy(info.begin(), info.end(), info_out);
    return any_bad ? DPD_ERR_NOT_SPD : DPD_OK;
}

}  // extern "C"
