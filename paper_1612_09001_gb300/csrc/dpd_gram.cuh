// Least-squares estimation of the APH coefficients (Sec. 2.2):
//   h = (Psi^H Psi)^{-1} Psi^H t,  Psi = basis matrix of Eq. 2 built from u.
//
// Real form.  With A = [Re Psi | Re t | Im Psi | Im t] (n x (2K + 2)), every
// quantity needed is a block of A^T A:
//   Re G_ab = <Re a, Re b> + <Im a, Im b>,   Im G_ab = <Re a, Im b> - <Im a, Re b>
//   Re g_a  = <Re a, Re t> + <Im a, Im t>,   Im g_a  = <Re a, Im t> - <Im a, Re t>
//   t^H t   = <Re t, Re t> + <Im t, Im t>
// (G = Psi^H Psi, g = Psi^H t).  The conjugate branch's basis is the conjugate
// of the main branch's (Eq. 2), so Re conj(z) = Re z and Im conj(z) = -Im z:
// every real column of A is +-1 times one of D = 2 B T + 3 distinct columns
// X (B = max(Bp, Bq)), or zero (Im of the constant column):
//   d = b T + k          Re psi_b(u_{n-k})    (b < B, k < T)
//   d = B T + b T + k    Im psi_b(u_{n-k})
//   d = 2 B T            1
//   d = 2 B T + 1, + 2   Re t, Im t
// and S = X^T X (D x D, D <= 99) holds all of A^T A up to signs.
//
// S is a contraction over the n rows, run on the tensor cores.  Every distinct
// column is one of 15 signals (Re / Im psi_b, Re / Im t, the constant) read at
// a tap, so an entry of S is a lagged correlation of two signals, less the
// products that fall off the end of the record; the tensor kernel computes the
// 15 x 14 x 8 lagged correlations (the basis recomputed from u, never stored
// in global memory), as a polyphase product whose operands hold each signal
// once per sample, split into a high and a low part (BF16 or TF32), X = hi +
// lo, with hi hi + hi lo + lo hi summed in FP32 in tensor memory.  Per-CTA
// partial sums are added in FP64 in a fixed order and S is filled from them
// and the last samples of the record.  The K x K system is then equilibrated
// and factored (chol_pair.cu), and refined against the FP32 residual
// t - Psi h computed by the filter and adjoint kernels.
#pragma once

#include "dpd_internal.h"

namespace dpd {

struct GramProblem {
    const float2 *u;   // basis input (n samples)
    const float2 *t;   // target (n samples) or null
    int64_t n;
};

constexpr int kGramS = 112;             // distinct columns, padded (D <= 99); row stride of S
constexpr int kGramRows = 128;          // rows of a partial (the MMA's M)
constexpr int kGramPartCols = 2 * kGramS;   // a partial: P in columns [0, 112), Q in [112, 224)

__host__ __device__ constexpr int gram_distinct(int B, int T) { return 2 * B * T + 3; }

// Distinct column and sign of the real and imaginary parts of complex column j
// of Psi (stacking order of Sec. 2.2); sign 0 marks a zero column.
struct ColRef {
    int d, sign;
};
__host__ __device__ inline void psi_column_refs(int j, int K, int Bp, int B, int T, ColRef &re, ColRef &im)
{
    if (j == K - 1) {   // the constant column (LO leakage term c)
        re = ColRef{2 * B * T, 1};
        im = ColRef{0, 0};
        return;
    }
    const bool conj = j >= Bp * T;
    const int jj = conj ? j - Bp * T : j;
    const int b = jj / T, k = jj % T;
    re = ColRef{b * T + k, 1};
    im = ColRef{B * T + b * T + k, conj ? -1 : 1};
}

struct GramArgs {
    const GramProblem *probs;   // device array of nprob problems, or null: the one problem below
    GramProblem one;
    int nprob;
    int cpp;               // CTAs per problem (row chunks)
    int Bp, Bq, T, K;
    float *partials;       // FP32 kernel: [nprob * cpp][kGramRows][kGramPartCols] floats;
                           // tensor kernel: [nprob * cpp][kLagEntries] float pairs
    int *status;
    // Basis of the psi columns: per problem a kMaxB x kMaxB matrix U (row-major,
    // U[a][b] multiplies |u|^{2a} u in basis function b, upper triangular), or
    // null for the monomials |u|^{2b} u themselves.
    const float *ubasis;
};
constexpr int kUSize = kMaxB * kMaxB;

// Precision of the Gram contraction.
enum : int { kPrecFP32 = 0, kPrecTF32x3 = 1, kPrecBF16x3 = 2 };

cudaError_t launch_gram(int precision, const GramArgs &a, cudaStream_t s);
// S[p][i][c] (i < D, c < 2 kGramS) = sum over the problem's CTAs of the partial P and Q
// blocks, in FP64 and a fixed order (S = P + Q + Q^T is formed by the assembly).
cudaError_t launch_gram_reduce(const float *partials, int nprob, int cpp, int D, double *S, cudaStream_t s);
// Tensor-core precisions: each CTA's partial is kLagEntries lag sums C[a][b][d]
// (a < 15, b < 14, d < kMaxT), each an FP32 pair (sum, rounding error); this sums them per
// problem into C (FP64, fixed order).
// G, g and t^H t are assembled from C directly (the entries of S on the fly), into G / g
// / tt at K x K, K, 1 per problem; probs may be null for one problem passed as `one`;
// `lower`: only the lower triangle of G (what the factorisation reads).  Ghost: a copy
// of the first problem's G in mapped host memory, or null.
constexpr int kLagEntries = 15 * 14 * kMaxT;
cudaError_t launch_gram_lag_finish(const float *partials, const GramProblem *probs, GramProblem one,
                                   const float *ubasis, int nprob, int cpp, int K, int Bp, int B, int T, bool lower,
                                   double *C, double2 *G, double2 *g, double *tt, double2 *Ghost, cudaStream_t s);
// G (K x K, row-major), g (K) and t^H t per problem from S.
cudaError_t launch_gram_assemble(const double *S, int nprob, int K, int Bp, int B, int T, double2 *G, double2 *g,
                                 double *tt, double2 *Ghost, cudaStream_t s);
// Orthonormal basis U of every problem (Sec. 2.1; kUSize per problem, FP32 and the same
// values in FP64) from the power sums sum_n r_n^k, k = 1 .. 2 B - 1, of r = |u|^2: exact
// FP32 two-sum pairs within a warp, then FP64, in a fixed order (part: max(nprob,
// kMomBlocks) * kMomK doubles of scratch).  probs may be null for the one problem `one`;
// nmax: the longest problem.
constexpr int kMomK = 2 * kMaxB - 1;
constexpr int kMomBlocks = 456;   // over all problems: three per SM at 152 SMs
__host__ __device__ constexpr int moments_blocks(int nprob)   // blocks a problem gets at most
{
    return nprob < kMomBlocks ? kMomBlocks / nprob : 1;
}
cudaError_t launch_basis(const GramProblem *probs, GramProblem one, int nprob, int64_t nmax, int B, double *part,
                         float *ubasis, double *ubasis64, cudaStream_t s);
// CTAs per row chunk the launch wants for nprob problems of up to n rows.
int gram_ctas_per_problem(int precision, int sm_count, int nprob, int64_t n);
// Equilibrated factorisation of every G: D G D = U Delta U^H, D = diag(G)^{-1/2}, U
// unit lower triangular, Delta diagonal.  U per problem: K (K + 1) / 2 values packed
// by rows, with 1 / Delta on the diagonal, each an FP32 pair {re.hi, im.hi, re.lo,
// im.lo} or, with wide[p], two doubles {re, im} in the same 16 bytes; d: K per problem;
// info[p] = 0 or the failing pivot + 1.  Uhost, info_host (each may be null): copies of
// the first problem's factor, and of its status and wide flag, in mapped host memory.
cudaError_t launch_chol(const double2 *G, int nprob, int K, float4 *U, int *wide, double *d, int *info, float4 *Uhost,
                        int *info_host, int *status, cudaStream_t s);
// x = G^{-1} rhs using the factorisation (problems that did not factor are skipped).
// Every pointer: `nprob` consecutive vectors, K apart unless stated.
struct SolveIo {
    const double2 *rhs;      // right-hand sides, or null: the sums of ...
    const float2 *rows;      // ... nrows rows per problem, in the monomial basis
    int nrows;
    const double *basis;     // basis U of the system (kUSize per problem), or null: monomials
    double2 *h;              // x, or h + x with `accumulate`, in that basis
    int accumulate;
    float2 *out;             // the monomial coefficients
    float *tab;              // their forward tables, tstride floats apart
    int tstride;
    int Bp, Bq, T;
};
cudaError_t launch_chol_solve(const float4 *U, const int *wide, const double *d, const int *info, int nprob, int K,
                              const SolveIo &io, int *status, cudaStream_t s);
// e = t - y (n samples).
cudaError_t launch_residual(const float2 *t, const float2 *y, int64_t n, float2 *e, cudaStream_t s);
// e = t - y together with out[0] = sum |e|^2, out[1] = sum |t|^2 in FP64
// (part: 2 * 1024 doubles of scratch).
cudaError_t launch_residual_norm(const float2 *t, const float2 *y, int64_t n, float2 *e, double *part, double *out,
                                 cudaStream_t s);

}  // namespace dpd
