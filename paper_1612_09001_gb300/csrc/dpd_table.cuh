// Derivation of the per-tap coefficient tables (layouts in dpd_internal.h) from the
// stacked coefficient vector of Sec. 2.2, for the kernels that produce coefficients.
#pragma once

#include "dpd_internal.h"

namespace dpd {

// Thread i of a block with at least B * T threads: (tap, order) pair i; thread 0 also
// the constant.  h(j) is coefficient j; adj (the adjoint table) may be null.
template <class H>
__device__ __forceinline__ void wl_table_entry(H h, int i, int Bp, int Bq, int T, int B, float *__restrict__ tab,
                                               float *__restrict__ adj)
{
    if (i < T * B) {
        const int k = i / B, m = i % B;
        const float2 A = (m < Bp) ? h(m * T + k) : make_float2(0.f, 0.f);          // h_{2m+1,k}
        const float2 C = (m < Bq) ? h((Bp + m) * T + k) : make_float2(0.f, 0.f);   // hbar_{2m+1,k}
        tab[wl_index(B, k, m, 0)] = A.x + C.x;      // P0 = Re(A+C)
        tab[wl_index(B, k, m, 1)] = -(A.y - C.y);   // P1 = -Im(A-C)
        tab[wl_index(B, k, m, 2)] = A.y + C.y;      // P2 = Im(A+C)
        tab[wl_index(B, k, m, 3)] = A.x - C.x;      // P3 = Re(A-C)
        if (adj) {
            // Per tap: for each power m the quadruple {Q0, Q3, Q1, Q2} of the
            // bracket conj(E) g + H conj(g) = {Q0 c + Q1 d, Q2 c + Q3 d}
            // (g = c + j d), then for each m < B-1 the quadruple {S0, S3, S1, S2}
            // of conj(G) g + F conj(g): the pairs {Q0, Q3}, {Q1, Q2} multiply
            // {c, d} and {d, c} in packed f32x2 FMAs.
            float *q = adj + (4 * B + 4 * (B - 1)) * k;
            // E_m = (m+1) h_m, H_m = (m+1) hbar_m  (coefficients of r^m)
            const float s = (float)(m + 1);
            const float Er = s * A.x, Ei = s * A.y, Hr = s * C.x, Hi = s * C.y;
            q[4 * m + 0] = Er + Hr;   // Q0
            q[4 * m + 1] = Er - Hr;   // Q3
            q[4 * m + 2] = Ei + Hi;   // Q1
            q[4 * m + 3] = Hi - Ei;   // Q2
            if (m < B - 1) {
                // F_m = (m+1) h_{m+1}, G_m = (m+1) hbar_{m+1}
                const float2 A1 = (m + 1 < Bp) ? h((m + 1) * T + k) : make_float2(0.f, 0.f);
                const float2 C1 = (m + 1 < Bq) ? h((Bp + m + 1) * T + k) : make_float2(0.f, 0.f);
                const float Fr = s * A1.x, Fi = s * A1.y, Gr = s * C1.x, Gi = s * C1.y;
                float *r = q + 4 * B;
                r[4 * m + 0] = Gr + Fr;   // S0
                r[4 * m + 1] = Gr - Fr;   // S3
                r[4 * m + 2] = Gi + Fi;   // S1
                r[4 * m + 3] = Fi - Gi;   // S2
            }
        }
    }
    if (i == 0) {
        const float2 c = h((Bp + Bq) * T);
        tab[4 * B * T] = c.x;
        tab[4 * B * T + 1] = c.y;
    }
}

}  // namespace dpd
